// Batched rank-one update step of the SuperDC conquering stage on sm_103a.
//
// For every problem p of a batch (independent problems, or all nodes of one
// HSS tree level), with poles d ascending and update vector z:
//   k_deflate   -- Remark 4.1: |z_k| < tau, then the Givens scan over the
//                  survivors (in parallel but for chains of consecutive
//                  rotations); compaction into kept / deflated slots.
//   k_tiles     -- prefix of root tiles per problem (device-side, so a level
//                  can be launched without a host round trip).
//   k_secular   -- Algorithm 2 with the shifted secular equation eq. (4.13):
//                  every root iterates on its gap eta = lambda - d_K (eq. (4.17))
//                  with shifted differences (d_j - d_K) - y (eq. (4.14)); the
//                  sums are split at the root's index into the lower part psi
//                  (j <= k) and the upper part phi (j > k), eqs. (4.7)-(4.10);
//                  middle-way rational step, stopping test eq. (4.12).  Direct
//                  tiled evaluator: poles and weights staged in shared memory,
//                  one root per thread.
//   k_lowner    -- eq. (4.23) (paired ratios, shifted differences).
//   k_bnorm     -- eq. (4.27) with the shifted entries of eq. (4.28).
//   k_merge     -- new eigenvalues (eq. (4.21)) and deflated values sorted by
//                  (value, input index).
// Inputs, results and what decides their accuracy are FP64: the terms of the two
// poles next to a root, its function value and iterate, the last root, the origin's
// term of b, the factors of zhat next to the target, and everything of a problem out
// of scale.  The other terms are split into FP32 or integer parts that carry FP64's
// accuracy or more (split.cuh); only the step's model (derivatives, guess) is single
// precision.
#include "common.cuh"
#include "rank1.cuh"
#include "prof.cuh"
#include "secular.cuh"
#include "fmm.cuh"
#include "tiles.cuh"
#include <algorithm>
#include <mutex>

namespace {

constexpr int SEC_CHUNK = 1024;   // poles staged per shared-memory chunk (24 bytes each)
constexpr int LONG_M = 512;       // more poles than this: split sweeps with three-float totals (ff_close3); the
                                  // blocks of fewer leave less error than the terms.  Chosen per launch by what
                                  // the direct kernels can meet: per problem it costs what it saves
constexpr int DEFL_BIG = 128;     // problems larger than this deflate with more than one warp


// ---------------------------------------------------------------------------
// Deflation (Remark 4.1), one CTA of T threads per problem (one warp up to
// DEFL_BIG entries).  The |z| < tau mask, the adjacent Givens tests and the
// compactions run in parallel: every warp takes a contiguous segment in steps of
// 32 (ballots give the places within a step), and one sum over the warps joins
// the segments, so a pass costs one barrier instead of one scan per T entries
// (GB300, one problem of 100003 poles: 0.65 -> 0.3 ms; 64-entry problems were
// one thread each, 37 us a launch).  Only chains of consecutive rotations are
// walked sequentially.  All arithmetic is one explicitly rounded sequence (no
// fused multiply-add), so decisions and rotated values are reproducible bit for
// bit by any IEEE evaluation in the order of the plain left-to-right scan.
// ---------------------------------------------------------------------------
constexpr int DB_T = 512;         // threads per problem; 1024 when a batch has fewer problems than SMs
constexpr int WALK_CAP = 64;      // speculative steps of one chain before one thread finishes it
constexpr int ORDER_PHASES = 32;  // exchange phases on the deflated values before they are merge-sorted

// doubles ordered as integers: as <, with both zeros equal and every NaN at an end
// (a total order, so that equal keys and indexes keep a permutation)
__device__ __forceinline__ long long order_key(double v)
{
    const long long b = __double_as_longlong(v);
    return (b << 1) == 0 ? 0 : ff_ord(v);
}

// sum of cnt over the warps before this one; *total over all (every thread calls)
template <int T>
__device__ __forceinline__ int seg_base(int cnt, int *sh, int *total)
{
    const int warp = threadIdx.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[warp] = cnt;
    __syncthreads();
    int before = 0, all = 0;
    for (int w = 0; w < T / 32; w++) {
        const int v = sh[w];
        before += (w < warp) ? v : 0;
        all += v;
    }
    *total = all;
    return before;
}

template <int T>
__global__ void __launch_bounds__(T)
k_deflate(int64_t nprob, const int64_t *__restrict__ off, const double *__restrict__ d,
          const double *__restrict__ z, double sqrt_rho, double tau, double *__restrict__ wd,
          double *__restrict__ wz, int8_t *__restrict__ kept, int32_t *__restrict__ surv, R1Out o)
{
    constexpr int NWARP = T / 32;
    __shared__ int sh[NWARP];
    __shared__ int s_ng;
    __shared__ double s_w[NWARP];
    const unsigned FULL = 0xffffffffu;
    const int64_t p = blockIdx.x;
    if (p >= nprob) return;
    const int64_t b0 = off[p];
    const int m = (int)(off[p + 1] - b0);
    if ((m <= DEFL_BIG) != (T == 32)) return;       // the other launch's problem
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned below = (1u << lane) - 1u;
    const int seg = ((m + T - 1) / T) * 32;          // entries per warp, a multiple of 32
    const int beg = min(m, warp * seg), end = min(m, beg + seg);
    // A: copy, mask, survivor list
    const long long tbits = __double_as_longlong(tau);        // tau >= 0: doubles compare as their bits
    bool bad = false;
    int cnt = 0;
#pragma unroll 4
    for (int c = beg; c < end; c += 32) {
        const int i = c + lane;
        bool keep = false;
        if (i < end) {
            // (comparisons on the bits: FP64 ones are what bounds a large problem's CTA)
            const double di = d[b0 + i], z0 = z[b0 + i], zi = sqrt_rho == 1.0 ? z0 : z0 * sqrt_rho;
            bad = bad || ff_exp(di) == 0x7FF || ff_exp(zi) == 0x7FF;
            keep = !((__double_as_longlong(zi) & 0x7FFFFFFFFFFFFFFFll) < tbits);
            wd[b0 + i] = di;
            wz[b0 + i] = keep ? zi : 0.0;
            kept[b0 + i] = keep ? 1 : 0;
        }
        cnt += __popc(__ballot_sync(FULL, keep));
    }
    if (__any_sync(FULL, bad) && lane == 0) sdc_latch(o.status, SUPERDC_DEV_NONFINITE);
    int S;
    int pos = seg_base<T>(cnt, sh, &S);
#pragma unroll 4
    for (int c = beg; c < end; c += 32) {
        const int i = c + lane;
        const bool keep = i < end && kept[b0 + i] != 0;
        const unsigned mask = __ballot_sync(FULL, keep);
        if (keep) surv[b0 + pos + __popc(mask & below)] = i;
        pos += __popc(mask);
    }
    __syncthreads();
    // B: Givens scan over the survivors.  The candidate of every test is the
    // previous survivor, so a test can differ from its value on the original
    // data only right after a rotation.  First every adjacent test on the
    // original values; the positions whose test passes are the "chain heads",
    // listed in order (o.src holds the flags and o.perm the list: both are
    // written only later).  The heads are then taken T at a time: each walks its
    // chain in its own thread on the original values (rotate, re-test the next
    // pair with the rotated values, until a test fails; at most WALK_CAP
    // steps); one thread then decides in order which heads start a chain of the
    // sequential scan (a head inside or at the end of the previous chain does
    // not) and gives each chain its offset in the rotation list; finally the
    // chains write their rotations in parallel (chains are disjoint; a chain
    // longer than WALK_CAP is finished and written by that one thread).
    const int sseg = ((S + T - 1) / T) * 32, sbeg = min(S, warp * sseg), send = min(S, sbeg + sseg);
    cnt = 0;
#pragma unroll 2
    for (int c = sbeg; c < send; c += 32) {
        const int t = c + lane;
        bool hf = false;
        if (t < send && t > 0) {
            const int ia = surv[b0 + t - 1], ib = surv[b0 + t];
            const double da = wd[b0 + ia], za = wz[b0 + ia], db = wd[b0 + ib], zb = wz[b0 + ib];
            // |da - db| |za| |zb| is at least 2^el and the right-hand side less than
            // 2^(er + 4): most pairs are told apart by the exponents
            const double dd = __dsub_rn(da, db);
            const int ea = ff_exp(za) - 1023, eb = ff_exp(zb) - 1023, ed = ff_exp(dd) - 1023;
            const int el = ed + ea + eb, er = 2 * max(ea, eb) + ff_exp(tau) - 1023;
            const bool plain = min(min(ea, eb), ed) > -300 && max(max(ea, eb), ed) < 300;
            if (!(plain && el > er + 4)) {
                const double lhs = fabs(__dmul_rn(__dmul_rn(dd, za), zb));
                const double rhs = __dmul_rn(__dadd_rn(__dmul_rn(za, za), __dmul_rn(zb, zb)), tau);
                hf = lhs < rhs;
            }
        }
        if (t < send) o.src[b0 + t] = hf;
        cnt += __popc(__ballot_sync(FULL, hf));
    }
    int nheads;
    pos = seg_base<T>(cnt, sh, &nheads);
    if (tid == 0) s_ng = 0;
    if (nheads > 0) {
        __shared__ int h_pos[T], h_end[T], h_off[T];
        __shared__ int s_eprev;
        for (int c = sbeg; c < send; c += 32) {
            const int t = c + lane;
            const bool hf = t < send && o.src[b0 + t] != 0;
            const unsigned mask = __ballot_sync(FULL, hf);
            if (hf) o.perm[b0 + pos + __popc(mask & below)] = t;
            pos += __popc(mask);
        }
        // one chain from position h (candidate s_{h-1}); write = false: count
        // only.  Returns the first position whose test fails (or S), or -1 when
        // max_steps rotations were taken without reaching it.  nrot >= 0: take
        // exactly nrot rotations without testing (the chain's length is known;
        // its last, failing test would read the first entry of the next chain,
        // which that chain may be rotating at the same time).
        auto walk = [&](int h, int max_steps, bool write, int ng0, int nrot) -> int {
            int ia = surv[b0 + h - 1];
            double da = wd[b0 + ia], za = wz[b0 + ia];
            int t2 = h, k = 0;
            while (t2 < S) {
                if (nrot >= 0 && k == nrot) break;
                if (k == max_steps) return -1;
                const int ib = surv[b0 + t2];
                const double db = wd[b0 + ib], zb = wz[b0 + ib];
                const double nrm2 = __dadd_rn(__dmul_rn(za, za), __dmul_rn(zb, zb));
                if (nrot < 0) {
                    const double lhs = fabs(__dmul_rn(__dmul_rn(__dsub_rn(da, db), za), zb));
                    const double rhs = __dmul_rn(nrm2, tau);
                    if (!(lhs < rhs)) break;
                }
                const double r = __dsqrt_rn(nrm2);
                const double cc0 = __ddiv_rn(zb, r), ss0 = __ddiv_rn(za, r);
                const double cc = __dmul_rn(cc0, cc0), ss = __dmul_rn(ss0, ss0);
                const double na = __dadd_rn(__dmul_rn(cc, da), __dmul_rn(ss, db));
                const double nb = __dadd_rn(__dmul_rn(ss, da), __dmul_rn(cc, db));
                if (write) {
                    wd[b0 + ia] = na;
                    wz[b0 + ia] = 0.0;
                    kept[b0 + ia] = 0;
                    wd[b0 + ib] = nb;
                    wz[b0 + ib] = r;
                    o.giv_ab[2 * (b0 + ng0 + k)] = ia;
                    o.giv_ab[2 * (b0 + ng0 + k) + 1] = ib;
                    o.giv_cs[2 * (b0 + ng0 + k)] = cc0;
                    o.giv_cs[2 * (b0 + ng0 + k) + 1] = ss0;
                }
                ia = ib; da = nb; za = r;
                t2++;
                k++;
            }
            return t2;
        };
        if (tid == 0) s_eprev = 0;
        __syncthreads();
        for (int h0 = 0; h0 < nheads; h0 += T) {
            const int nh = min(T, nheads - h0);
            // speculative walks; a head at or before the previous chain's end is
            // not a chain start, and such a head may read rotated values, so its
            // result is only used once that has been ruled out
            if (tid < nh) {
                const int h = o.perm[b0 + h0 + tid];
                h_pos[tid] = h;
                h_end[tid] = (h <= s_eprev) ? 0 : walk(h, WALK_CAP, false, 0, -1);
            }
            __syncthreads();
            if (tid == 0) {
                int e_prev = s_eprev, ng = s_ng;
                for (int i = 0; i < nh; i++) {
                    const int h = h_pos[i];
                    if (h <= e_prev) { h_off[i] = -1; continue; }
                    int e = h_end[i];
                    if (e < 0) {                         // long chain: finished and written here
                        e = walk(h, S, true, ng, -1);
                        h_off[i] = -1;
                    } else {
                        h_off[i] = ng;
                    }
                    ng += e - h;
                    e_prev = e;
                }
                s_eprev = e_prev;
                s_ng = ng;
            }
            __syncthreads();
            if (tid < nh && h_off[tid] >= 0) walk(h_pos[tid], S, true, h_off[tid], h_end[tid] - h_pos[tid]);
            __syncthreads();
        }
    }
    __syncthreads();
    // C: compaction, kept slots in index order, then deflated slots in index order
    cnt = 0;
#pragma unroll 4
    for (int c = beg; c < end; c += 32) {
        const int i = c + lane;
        cnt += __popc(__ballot_sync(FULL, i < end && kept[b0 + i] != 0));
    }
    int mk;
    pos = seg_base<T>(cnt, sh, &mk);
    double wpart = 0.0;
#pragma unroll 4
    for (int c = beg; c < end; c += 32) {
        const int i = c + lane;
        const bool k = i < end && kept[b0 + i] != 0;
        const unsigned mask = __ballot_sync(FULL, k);
        const int before = pos + __popc(mask & below);            // kept entries before i
        if (i < end) {
            const int64_t q = b0 + (k ? before : mk + i - before);
            o.dk[q] = wd[b0 + i];
            o.src[q] = i;
            if (k) {
                const double zi = wz[b0 + i];
                o.zk[q] = zi;
                wpart = fma(zi, zi, wpart);
            }
        }
        pos += __popc(mask);
    }
    // deterministic sum of kept z^2
    for (int of = 16; of > 0; of >>= 1) wpart += __shfl_xor_sync(FULL, wpart, of);
    if (lane == 0) s_w[warp] = wpart;
    __syncthreads();
    if (tid == 0) {
        double W = 0.0;
        for (int w = 0; w < NWARP; w++) W += s_w[w];
        o.wsum[p] = W;
        o.mk[p] = mk;
        o.ngiv[p] = s_ng;
    }
    // D: deflated values sorted by (value, index).  They are in index order; only
    // a rotated value can be out of order, in a cluster by a few places, which
    // odd-even exchanges (of values strictly out of order: ties keep their order)
    // settle in as many phases.  But a rotation next to a much larger weight moves
    // its value across all entries up to the next survivor: what is not in order
    // after ORDER_PHASES is merge-sorted, a thread per entry placing it by binary
    // search in the neighbouring run, with the copies wd and surv, read for the last
    // time above, as the other buffer.  (GB300, one value moved
    // across 30000 entries, the whole step: 137 ms by exchanges alone, 7.8 by one
    // thread's insertions, 1.2 so.)
    const int nd = m - mk;
    if (nd >= 2) {
        int idle = 0;
        for (int ph = 0; idle < 2 && ph < ORDER_PHASES; ph++) {
            bool sw = false;
            for (int q = mk + (ph & 1) + 2 * tid; q + 1 < m; q += 2 * T) {
                const double v0 = o.dk[b0 + q], v1 = o.dk[b0 + q + 1];
                if (v0 > v1) {
                    const int s0 = o.src[b0 + q], s1 = o.src[b0 + q + 1];
                    o.dk[b0 + q] = v1;
                    o.dk[b0 + q + 1] = v0;
                    o.src[b0 + q] = s1;
                    o.src[b0 + q + 1] = s0;
                    sw = true;
                }
            }
            idle = __syncthreads_or(sw) ? 0 : idle + 1;
        }
        if (idle < 2) {
            double *va = o.dk + b0 + mk, *vb = wd + b0;
            int32_t *ia = o.src + b0 + mk, *ib = surv + b0;
            for (int lw = 0; lw < 31 && (1 << lw) < nd; lw++) {
                const int w = 1 << lw;
                for (int i = tid; i < nd; i += T) {
                    const int r0 = i & ~(w - 1);                       // this entry's run, and its neighbour's
                    const int q0 = min(nd, r0 ^ w), q1 = q0 + min(w, nd - q0);
                    const double v = va[i];
                    const int s = ia[i];
                    const long long k = order_key(v);
                    int lo = q0, hi = q1;
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        const long long km = order_key(va[mid]);
                        if (km < k || (km == k && ia[mid] < s)) lo = mid + 1; else hi = mid;
                    }
                    const int to = min(r0, r0 ^ w) + (i - r0) + (lo - q0);
                    vb[to] = v;
                    ib[to] = s;
                }
                __syncthreads();
                double *const tv = va;
                va = vb;
                vb = tv;
                int32_t *const ti = ia;
                ia = ib;
                ib = ti;
            }
            if (va == wd + b0)
                for (int i = tid; i < nd; i += T) {
                    o.dk[b0 + mk + i] = va[i];
                    o.src[b0 + mk + i] = ia[i];
                }
        }
    }
    __syncthreads();
    for (int s2 = mk + tid; s2 < m; s2 += T) {
        o.zk[b0 + s2] = 0.0;
        o.org[b0 + s2] = -1;
        o.eta[b0 + s2] = 0.0;
        o.dorg[b0 + s2] = o.dk[b0 + s2];
        o.vhat[b0 + s2] = 0.0;
        o.bnorm[b0 + s2] = 1.0;
        if (o.sweeps) o.sweeps[b0 + s2] = 0;
    }
}

// the two launches of a batch: problems up to DEFL_BIG entries, and larger ones
void launch_deflate(const R1Args &a, const R1Out &o, int big_t, double *wd, double *wz, int8_t *kept, int32_t *surv,
                    cudaStream_t st)
{
    k_deflate<32><<<(unsigned)a.nprob, 32, 0, st>>>(a.nprob, a.off, a.d, a.z, a.sqrt_rho, a.tau, wd, wz, kept, surv, o);
    if (a.total > DEFL_BIG) {
        auto fn = big_t == 1024 ? k_deflate<1024> : k_deflate<DB_T>;
        fn<<<(unsigned)a.nprob, big_t, 0, st>>>(a.nprob, a.off, a.d, a.z, a.sqrt_rho, a.tau, wd, wz, kept, surv, o);
    }
}

// Work units of the secular kernel: (problem, first root, end root), at most
// ubig roots each.  A unit stages its problem's poles in shared memory (all of
// them when they fit in SEC_CHUNK, else in chunks per sweep).  Units are
// ordered by decreasing problem size (largest first) so the long units start
// early, and capping the roots per unit spreads a large problem over several
// SMs, which keeps the tail of the launch short.  With last != 0 a problem's last
// root, a chain of its own, gets a unit (fourth entry 1) ahead of the others.
constexpr int SEC_UNIT_BIG = 2048;
constexpr int SORT_MAX = 8192;

__global__ void k_units(int64_t nprob, const int32_t *__restrict__ mk, const int32_t *__restrict__ fslot, int ubig,
                        int last, int4 *__restrict__ units, int *__restrict__ nunits,
                        int *__restrict__ counter)
{
    extern __shared__ unsigned long long keys[];   // SORT_MAX entries when sorting
    __shared__ int sh[32];
    const int T = blockDim.x;
    const bool sorted = nprob <= SORT_MAX;
    int64_t n2 = 1;
    if (sorted) {
        while (n2 < nprob) n2 <<= 1;
        for (int64_t i = threadIdx.x; i < n2; i += T) {
            // descending by size: key = (size << 32) | (~p) so that equal sizes keep index order
            const int mi = (i < nprob && !(fslot && fslot[i] >= 0)) ? mk[i] : 0;
            keys[i] = (i < nprob) ? (((unsigned long long)(unsigned)mi << 32) |
                                     (unsigned long long)(0xFFFFFFFFu - (unsigned)i))
                                  : 0ull;
        }
        __syncthreads();
        for (int64_t kk = 2; kk <= n2; kk <<= 1) {
            for (int64_t j = kk >> 1; j > 0; j >>= 1) {
                for (int64_t i = threadIdx.x; i < n2; i += T) {
                    int64_t ixj = i ^ j;
                    if (ixj > i) {
                        bool desc = ((i & kk) == 0);
                        unsigned long long a = keys[i], b = keys[ixj];
                        if (desc ? (a < b) : (a > b)) { keys[i] = b; keys[ixj] = a; }
                    }
                }
                __syncthreads();
            }
        }
    }
    // units per problem (in the chosen order), block-wide prefix
    int64_t per = (nprob + T - 1) / T;
    int64_t beg = min(nprob, threadIdx.x * per), end = min(nprob, beg + per);
    int cnt = 0;
    for (int64_t q = beg; q < end; q++) {
        int64_t pp = sorted ? (int64_t)(0xFFFFFFFFu - (unsigned)(keys[q] & 0xFFFFFFFFull)) : q;
        int m = (fslot && fslot[pp] >= 0) ? 0 : mk[pp];   // FMM problems: not here
        cnt += (m + ubig - 1) / ubig + (last && m >= 2 ? 1 : 0);
    }
    int all;
    int u = cta_exscan(cnt, sh, &all);
    if (threadIdx.x == 0) {
        *nunits = all;
        *counter = 0;
    }
    for (int64_t q = beg; q < end; q++) {
        int64_t pp = sorted ? (int64_t)(0xFFFFFFFFu - (unsigned)(keys[q] & 0xFFFFFFFFull)) : q;
        int m = (fslot && fslot[pp] >= 0) ? 0 : mk[pp];
        if (m <= 0) continue;
        if (last && m >= 2) units[u++] = make_int4((int)pp, m - 1, m, 1);
        for (int r = 0; r < m; r += ubig) units[u++] = make_int4((int)pp, r, min(m, r + ubig), 0);
    }
}

// One CTA of NW warps per unit, persistent over an atomic unit queue.
//
// SPLIT = false (many roots per launch, e.g. thousands of independent
// problems): each warp owns a contiguous 1/NW of the unit's roots; a lane
// whose root has converged takes the next root of the warp's range, so the
// FP64 pipe keeps working on live roots instead of waiting for the slowest
// root of a fixed group of 32.
// SPLIT = true (few large problems, e.g. the top levels of the tree): the NW
// warps share one 32-lane root range and split the poles NW ways; the partial
// sums are reduced through shared memory after every sweep and each warp
// applies the same update, so the replicated root state stays identical.
// Both keep the live roots of a warp inside a short window, so the psi/phi
// split keeps its three warp-uniform regions.
// (Without SPLIT, registers for five CTAs per SM: left to itself the compiler takes 72,
// 2048 problems of 100 to 500: 4.26 ms a step, with 96 4.07.  With SPLIT it is left to
// itself, 96 too: one batch of 16 problems 307 us, 309 with the bound, 299 with all the
// registers it wants, but then 2600 problems take 0.62 ms in this kernel instead of 0.48.)
template <int NW, bool SPLIT, bool LONG>
__global__ void __launch_bounds__(NW * 32, SPLIT ? 0 : 5)
k_secular(const int64_t *__restrict__ off, const int4 *__restrict__ units,
          const int *__restrict__ nunits, int *__restrict__ counter,
          R1Out o, double stop_c, int max_iter)
{
    // staged poles and weights: split parts (ok), or FP64 (the general form)
    __shared__ __align__(16) unsigned char stage[SEC_CHUNK * (sizeof(ff_f4) + sizeof(ff_f2))];
    ff_f4 *const fd = (ff_f4 *)stage;
    ff_f2 *const fw = (ff_f2 *)(fd + SEC_CHUNK);
    double *const sd = (double *)stage, *const sw = sd + SEC_CHUNK;
    __shared__ double red[SPLIT ? NW : 1][4][32];
    __shared__ float fred[SPLIT ? NW : 1][5][32];
    __shared__ double s_dK[SPLIT ? 32 : 1], s_y[SPLIT ? 32 : 1];
    __shared__ int s_ph[SPLIT ? 32 : 1], s_fin[SPLIT ? 32 : 1];
    __shared__ int s_unit;
    const unsigned FULL = 0xffffffffu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nu = *nunits;
    while (true) {
        __syncthreads();
        if (threadIdx.x == 0) s_unit = atomicAdd(counter, 1);
        __syncthreads();
        const int u = s_unit;
        if (u >= nu) break;
        const int4 U = units[u];
        const int64_t p = U.x;
        const int64_t b0 = off[p];
        const int m = o.mk[p];
        const double *dk = o.dk + b0, *zk = o.zk + b0;
        const double W = o.wsum[p];
        const double tol = stop_c * (double)m * SDC_EPS;
        // split FP32 sweeps where the problem's scale and the stopping test allow; its
        // last root (right of every pole, outside the fixed-point range) then runs on
        // its own
        const FfScale fs = ff_scale(dk[0], dk[m - 1], W);
        bool okt = fs.ok && !o.unshifted && m >= 2 && stop_c >= SPLIT_STOP;
        for (int j = threadIdx.x; okt && j + 1 < m; j += NW * 32) okt = ff_gap_ok(dk[j], dk[j + 1], fs.kk);
        const bool ok = __syncthreads_and(okt);
        auto last_root = [&]() {
            Root R;
            last_root_warp(dk, zk, m, W, tol, max_iter, o.status, R);
            if (lane == 0) {
                o.org[b0 + m - 1] = R.K;
                o.eta[b0 + m - 1] = R.y;
                o.dorg[b0 + m - 1] = R.dK;
                o.lamk[b0 + m - 1] = R.dK + R.y;
                if (o.sweeps) o.sweeps[b0 + m - 1] = R.nsw;
            }
        };
        if (SPLIT && U.w) {                       // the last root's unit
            if (ok && warp == 0) last_root();
            continue;
        }
        const int uend = ok ? min(U.z, m - 1) : U.z;
        const int len = uend - U.y;
        const int wbeg = SPLIT ? U.y : U.y + (int)(((int64_t)len * warp) / NW);
        const int wend = SPLIT ? uend : U.y + (int)(((int64_t)len * (warp + 1)) / NW);
        int k = wbeg + lane;
        bool act = k < wend;
        int next = wbeg + 32;
        Root R;
        R.dK = 0.0; R.y = 1.0; R.phase = 1;     // defined values for lanes that stay idle
        if (act) R.init(dk, zk, k, m, W, o.unshifted != 0);
        const bool single = (m <= SEC_CHUNK);
        auto stage_chunk = [&](int c0, int cn) {
            for (int j = threadIdx.x; j < cn; j += NW * 32) {
                const double zj = zk[c0 + j];
                if (ok) {
                    fd[j] = ff_pole(dk[c0 + j], fs);
                    fw[j] = ff_weight(zj * zj, fs.kw);
                } else {
                    sd[j] = dk[c0 + j];
                    sw[j] = zj * zj;
                }
            }
        };
        if (single) stage_chunk(0, m);
        __syncthreads();
        const bool lockstep = SPLIT || !single;
        while (lockstep ? __syncthreads_or(act) : __any_sync(FULL, act)) {
            const int kwlo = __reduce_min_sync(FULL, act ? k : 0x7fffffff);
            const int kwhi = __reduce_max_sync(FULL, act ? k : -1);
            const int kk = act ? k : kwlo;
            const bool p0 = __all_sync(FULL, !act || R.phase == 0);
            const bool any = __any_sync(FULL, act);
            Acc A = {0.0, 0.0, 0.0, 0.0};
            FfAcc S = {};
            const ff_f4 x = ff_point(R.dK, R.y, fs);
            for (int c0 = 0; c0 < m; c0 += SEC_CHUNK) {
                const int cn = min(SEC_CHUNK, m - c0);
                if (!single) {
                    __syncthreads();
                    stage_chunk(c0, cn);
                    __syncthreads();
                }
                const int j0 = SPLIT ? (int)(((int64_t)cn * warp) / NW) : 0;
                const int j1 = SPLIT ? (int)(((int64_t)cn * (warp + 1)) / NW) : cn;
                if (any) {
                    if (ok)      ff_sweep<LONG>(fd, fw, j0, j1, c0, kk, kwlo, kwhi, x, S);
                    else if (p0) sweep<false>(sd, sw, j0, j1, c0, kk, kwlo, kwhi, R.dK, R.y, A);
                    else         sweep<true>(sd, sw, j0, j1, c0, kk, kwlo, kwhi, R.dK, R.y, A);
                }
            }
            bool fin = false;
            if (SPLIT) {
                // the warps hold the same roots: warp 0 alone reduces the partial
                // sums (fixed order) and updates, the others take the new iterate
                // (an FP64 instruction costs its pipe slot in every warp that runs it)
                if (ok) {
                    float (*const fr)[32] = fred[SPLIT ? warp : 0];
                    fr[0][lane] = S.s; fr[1][lane] = S.sl; fr[2][lane] = S.psi; fr[3][lane] = S.dpsi; fr[4][lane] = S.dphi;
                } else {
                    red[SPLIT ? warp : 0][0][lane] = A.psi;
                    red[SPLIT ? warp : 0][1][lane] = A.phi;
                    red[SPLIT ? warp : 0][2][lane] = A.dpsi;
                    red[SPLIT ? warp : 0][3][lane] = A.dphi;
                }
                __syncthreads();
                if (warp == 0) {
                    Acc T = {0.0, 0.0, 0.0, 0.0};
                    if (ok) {
#pragma unroll
                        for (int w = 1; w < (SPLIT ? NW : 1); w++)
                            ff_merge(S, fred[w][0][lane], fred[w][1][lane], fred[w][2][lane], fred[w][3][lane],
                                     fred[w][4][lane]);
                    } else {
#pragma unroll
                        for (int w = 0; w < (SPLIT ? NW : 1); w++) {
                            T.psi += red[w][0][lane];
                            T.phi += red[w][1][lane];
                            T.dpsi += red[w][2][lane];
                            T.dphi += red[w][3][lane];
                        }
                    }
                    if (act) {
                        fin = ok ? R.update_split(S, 0.0, fs.kk, fs.kw, tol, max_iter, o.status)
                                 : R.update(T, tol, max_iter, o.status);
                        if (fin) {
                            o.org[b0 + k] = R.K;
                            o.eta[b0 + k] = R.y;
                            o.dorg[b0 + k] = R.dK;
                            o.lamk[b0 + k] = R.dK + R.y;
                            if (o.sweeps) o.sweeps[b0 + k] = R.nsw;
                        }
                    }
                    s_dK[SPLIT ? lane : 0] = R.dK;
                    s_y[SPLIT ? lane : 0] = R.y;
                    s_ph[SPLIT ? lane : 0] = R.phase;
                    s_fin[SPLIT ? lane : 0] = fin ? 1 : 0;
                }
                __syncthreads();
                if (warp != 0) {
                    R.dK = s_dK[SPLIT ? lane : 0];
                    R.y = s_y[SPLIT ? lane : 0];
                    R.phase = s_ph[SPLIT ? lane : 0];
                    fin = s_fin[SPLIT ? lane : 0] != 0;
                }
            } else if (act) {
                fin = ok ? R.update_split(S, 0.0, fs.kk, fs.kw, tol, max_iter, o.status)
                         : R.update(A, tol, max_iter, o.status);
                if (fin) {
                    o.org[b0 + k] = R.K;
                    o.eta[b0 + k] = R.y;
                    o.dorg[b0 + k] = R.dK;
                    o.lamk[b0 + k] = R.dK + R.y;
                    if (o.sweeps) o.sweeps[b0 + k] = R.nsw;
                }
            }
            const unsigned mask = __ballot_sync(FULL, fin);
            if (fin) {
                k = next + __popc(mask & ((1u << lane) - 1u));
                act = k < wend;
                if (act) R.init(dk, zk, k, m, W, o.unshifted != 0);
            }
            next += __popc(mask);
        }
        if (!SPLIT && ok && U.z == m && warp == NW - 1) last_root();
    }
}

// Tiles of the direct zhat and b kernels: TR targets per CTA, SW groups of TR
// threads that split the sources.  Many rows: 128 targets, one group (the staged
// sources serve four warps).  Fewer rows than two such tiles per SM: 32 targets
// and eight warps, as a thread's chain over every source, not the throughput,
// sets the time (GB300, 16 problems of 8..300: zhat 0.123 -> 0.025, b 0.127 -> 0.024 ms).
bool direct_split(int64_t rows) { return rows < (int64_t)sdc_num_sms() * 256; }

template <int SW>
__device__ __forceinline__ void grp_sync()
{
    if (SW > 1) __syncwarp();
    else __syncthreads();
}

// ---------------------------------------------------------------------------
// Loewner zhat, eq. (4.23):
//   vhat_i^2 = (lambda_{m-1} - d_i) prod_{j<i} (lambda_j - d_i)/(d_j - d_i)
//                                   prod_{i<=j<m-1} (lambda_j - d_i)/(d_{j+1} - d_i)
// with lambda_j - d_i = (d_{K_j} - d_i) + eta_j.
// ---------------------------------------------------------------------------
template <int TR, int SW>
__global__ void __launch_bounds__(TR * SW)
k_lowner(int64_t nprob, const int64_t *__restrict__ off, const int64_t *__restrict__ tile_off, R1Out o,
         const int32_t *__restrict__ fslot, unsigned long long *__restrict__ queue)
{
    __shared__ int64_t s_tile;
    __shared__ ff_w4 sd[SW][TR], sl[SW][TR];
    __shared__ FfProd part[SW > 1 ? SW : 1][2][SW > 1 ? TR : 1];
    const int tl = threadIdx.x % TR, grp = threadIdx.x / TR;
    const int64_t ntiles = tile_off[nprob];
    for (int64_t it = blockIdx.x;; it += gridDim.x) {
        int64_t tile = it;
        if (queue) {                          // tiles claimed one at a time (costs differ by m)
            __syncthreads();
            if (threadIdx.x == 0) s_tile = (int64_t)atomicAdd(queue, 1ull);
            __syncthreads();
            tile = s_tile;
        }
        if (tile >= ntiles) break;
        const int64_t p = sdc_upper_index(tile_off, nprob, tile);
        if (fslot && fslot[p] >= 0) continue;   // FMM problem
        const int64_t b0 = off[p];
        const int m = o.mk[p];
        const int i = (int)(tile - tile_off[p]) * TR + tl;
        const double *dk = o.dk + b0, *dorg = o.dorg + b0, *eta = o.eta + b0;
        const FfScale fs = ff_scale(dk[0], dk[m - 1], o.wsum[p]);
        bool okt = fs.ok && !o.unshifted && m >= 2;
        for (int j = threadIdx.x; okt && j + 1 < m; j += TR * SW) okt = ff_gap_ok(dk[j], dk[j + 1], fs.kk);
        const bool ok = __syncthreads_and(okt);
        const double di = i < m ? dk[i] : 0.0;
        double pn = 1.0, pd = 1.0;
        int ex = 0;
        if (ok) {
            // integer products (split.cuh); the two eigenvalues next to d_i and
            // the last one (outside the positions' range) in FP64
            FfProd num = {1ull << 63, 0}, den = {1ull << 63, 0};
            const ff_w4 d4 = ff_words4(ff_fixed(di, fs.kk) - fs.ref);
            const ff_u96 dw = {d4.lo, d4.mid, d4.hi};
            for (int c0 = grp * TR; c0 < m - 1; c0 += SW * TR) {
                const int cn = min(TR, m - 1 - c0), j = c0 + tl;
                grp_sync<SW>();
                if (tl < cn) {
                    sd[grp][tl] = ff_words4(ff_fixed(dk[j], fs.kk) - fs.ref);
                    sl[grp][tl] = ff_words4(ff_fixed(dorg[j], fs.kk) + ff_fixed(eta[j], fs.kk) - fs.ref);
                }
                grp_sync<SW>();
                ff_prod_sweep(sd[grp], sl[grp], cn, c0, i, dw, num, den);
            }
            if (SW > 1) {
                part[SW > 1 ? grp : 0][0][SW > 1 ? tl : 0] = num;
                part[SW > 1 ? grp : 0][1][SW > 1 ? tl : 0] = den;
                __syncthreads();
                if (grp > 0) continue;
                for (int w = 1; w < SW; w++) {
                    const FfProd a = part[SW > 1 ? w : 0][0][SW > 1 ? tl : 0], c = part[SW > 1 ? w : 0][1][SW > 1 ? tl : 0];
                    num.m = ff_mulhi(num.m, a.m);
                    den.m = ff_mulhi(den.m, c.m);
                    num.e += a.e + 64;
                    den.e += c.e + 64;
                    ff_prod_norm(num);
                    ff_prod_norm(den);
                }
            }
            if (i >= m) continue;
            lowner_edges(dk, dorg, eta, di, i, m, pn, pd, ex);
            pn *= (double)num.m;
            pd *= (double)den.m;
            ex += num.e - den.e;
        } else {
            if (i >= m || grp > 0) continue;
            // numerator and denominator products kept apart (one division per
            // entry instead of one per factor); every 8 factors both are brought
            // back to [1/2, 1) by exponent arithmetic, the exponents summed in ex
            pn = (dorg[m - 1] - di) + eta[m - 1];
            for (int j = 0; j < m - 1; j++) {
                double num = (dorg[j] - di) + eta[j];
                double den = ((j < i) ? dk[j] : dk[j + 1]) - di;
                pn *= num;
                pd *= den;
                if ((j & 7) == 7) {
                    int hn = __double2hiint(pn), hd = __double2hiint(pd);
                    int en = (hn >> 20) & 0x7FF, ed = (hd >> 20) & 0x7FF;
                    if (en != 0 && ed != 0 && en != 0x7FF && ed != 0x7FF) {
                        ex += en - ed;
                        pn = __hiloint2double((hn & 0x800FFFFF) | (1022 << 20), __double2loint(pn));
                        pd = __hiloint2double((hd & 0x800FFFFF) | (1022 << 20), __double2loint(pd));
                    }
                }
            }
        }
        double v = root_quot(pn, pd, ex);
        v = ldexp(v, ex / 2);
        if (!isfinite(v)) sdc_latch(o.status, SUPERDC_DEV_NONFINITE);
        o.vhat[b0 + i] = (o.zk[b0 + i] < 0.0) ? -v : v;
    }
}

// ---------------------------------------------------------------------------
// b_j = (sum_i vhat_i^2 / ((d_i - d_{K_j}) - eta_j)^2)^(-1/2), eq. (4.27)
// ---------------------------------------------------------------------------
template <int TR, int SW>
__global__ void __launch_bounds__(TR * SW)
k_bnorm(int64_t nprob, const int64_t *__restrict__ off, const int64_t *__restrict__ tile_off, R1Out o,
         const int32_t *__restrict__ fslot, unsigned long long *__restrict__ queue)
{
    __shared__ int64_t s_tile;
    __shared__ ff_f4 sd[SW][TR], sv[SW][TR];
    __shared__ ff_t3 part[SW > 1 ? SW : 1][SW > 1 ? TR : 1];
    __shared__ double red[TR * SW / 32];
    const int tl = threadIdx.x % TR, grp = threadIdx.x / TR;
    const int64_t ntiles = tile_off[nprob];
    for (int64_t it = blockIdx.x;; it += gridDim.x) {
        int64_t tile = it;
        if (queue) {                          // tiles claimed one at a time (costs differ by m)
            __syncthreads();
            if (threadIdx.x == 0) s_tile = (int64_t)atomicAdd(queue, 1ull);
            __syncthreads();
            tile = s_tile;
        }
        if (tile >= ntiles) break;
        const int64_t p = sdc_upper_index(tile_off, nprob, tile);
        if (fslot && fslot[p] >= 0) continue;   // FMM problem
        const int64_t b0 = off[p];
        const int m = o.mk[p];
        const int j = (int)(tile - tile_off[p]) * TR + tl;
        const double *dk = o.dk + b0, *v = o.vhat + b0;
        const FfScale fs = ff_scale(dk[0], dk[m - 1], o.wsum[p]);
        bool okt = fs.ok && !o.unshifted && m >= 2;
        for (int i = threadIdx.x; okt && i + 1 < m; i += TR * SW) okt = ff_gap_ok(dk[i], dk[i + 1], fs.kk);
        const bool ok = __syncthreads_and(okt);
        const double dK = j < m ? o.dorg[b0 + j] : 0.0, e = j < m ? o.eta[b0 + j] : 1.0;
        if (ok) {
            // three-float sums (split.cuh); the origin's term in FP64, the last
            // eigenvalue (outside the positions' range) by the whole CTA in FP64
            ff_t3 S = {0.0f, 0.0f, 0.0f};
            const int K = j < m ? o.org[b0 + j] : -1;
            const ff_f4 x = ff_point(dK, e, fs);
            const int kv = fs.kw >> 1;
            const double sc = ff_pow2(-kv);
            for (int c0 = grp * TR; c0 < m; c0 += SW * TR) {
                const int cn = min(TR, m - c0);
                grp_sync<SW>();
                if (tl < cn) {
                    const ff_t3 t = ff_split3(v[c0 + tl] * sc);
                    sd[grp][tl] = ff_pole(dk[c0 + tl], fs);
                    sv[grp][tl] = {t.a, t.b, t.c, 0.0f};
                }
                grp_sync<SW>();
                ff_sqr_sweep(sd[grp], sv[grp], cn, c0, K, x, S);
            }
            if (SW > 1) {
                part[SW > 1 ? grp : 0][SW > 1 ? tl : 0] = S;
                __syncthreads();
                if (grp == 0)
                    for (int w = 1; w < SW; w++) ff_acc3(S, part[SW > 1 ? w : 0][SW > 1 ? tl : 0]);
            }
            if (grp == 0 && j < m - 1) {
                const double r = v[K] * rcp_nr2(-e);
                o.bnorm[b0 + j] = rsqrt_any(fma(r, r, ff_join3(S) * ff_pow2(2 * (kv + fs.kk))));
            }
            if (m - 1 - (int)(tile - tile_off[p]) * TR < TR) {
                const double dl = o.dorg[b0 + m - 1], el = o.eta[b0 + m - 1];
                double s = 0.0;
                for (int i = threadIdx.x; i < m; i += TR * SW) {
                    const double vr = v[i] * rcp_nr2((dk[i] - dl) - el);
                    s = fma(vr, vr, s);
                }
                for (int sh = 16; sh > 0; sh >>= 1) s += __shfl_xor_sync(0xffffffffu, s, sh);
                if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
                __syncthreads();
                if (threadIdx.x == 0) {
                    s = 0.0;
                    for (int w = 0; w < TR * SW / 32; w++) s += red[w];
                    o.bnorm[b0 + m - 1] = rsqrt_any(s);
                }
            }
            continue;
        }
        if (j >= m || grp > 0) continue;
        double s = 0.0;
        for (int i = 0; i < m; i++) {
            double t = (dk[i] - dK) - e;
            double r = rcp_nr2(t);
            double vr = v[i] * r;
            s = fma(vr, vr, s);
        }
        o.bnorm[b0 + j] = 1.0 / sqrt(s);
    }
}

// ---------------------------------------------------------------------------
// Merge: new eigenvalue list per problem, ascending by (value, input index).
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool key_less(double v1, int s1, double v2, int s2)
{
    return v1 < v2 || (v1 == v2 && s1 < s2);
}

__global__ void k_merge(int64_t nprob, const int64_t *__restrict__ off, int64_t total, R1Out o)
{
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total;
         x += (int64_t)gridDim.x * blockDim.x) {
        if (x < off[0] || x >= off[nprob]) continue;
        const int64_t p = sdc_upper_index(off, nprob, x);
        const int64_t b0 = off[p];
        const int m = (int)(off[p + 1] - b0);
        const int mk = SDC_IDX(o.mk[p], m + 1, o.status);       // kept count in [0, m]
        const int s = (int)(x - b0);
        const double *dk = o.dk + b0, *dorg = o.dorg + b0, *eta = o.eta + b0;
        const int32_t *src = o.src + b0;
        int pos;
        double val;
        if (s < mk) {
            val = o.lamk[b0 + s];                        // eq. (4.21), d_K + eta
            // deflated slots with a smaller key
            int lo = mk, hi = m;
            while (lo < hi) {
                int mid = (lo + hi) >> 1;
                if (key_less(dk[mid], src[mid], val, src[s])) lo = mid + 1; else hi = mid;
            }
            pos = s + (lo - mk);
        } else {
            val = dk[s];
            int lo = 0, hi = mk;
            while (lo < hi) {
                int mid = (lo + hi) >> 1;
                double lm = o.lamk[b0 + mid];
                if (key_less(lm, src[mid], val, src[s])) lo = mid + 1; else hi = mid;
            }
            pos = (s - mk) + lo;
        }
        o.lam[b0 + pos] = val;
        o.perm[b0 + pos] = s;
        o.pinv[b0 + s] = pos;
    }
}

// k_units sorts in dynamic shared memory beyond the default 48 KB: raise its
// limit once per device (the attribute belongs to the device's context)
cudaError_t units_attr()
{
    static std::mutex mu;
    static bool done[64] = {false};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(mu);
    if (!done[dev]) {
        e = cudaFuncSetAttribute(k_units, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(SORT_MAX * sizeof(unsigned long long)));
        if (e != cudaSuccess) return e;
        done[dev] = true;
    }
    return cudaSuccess;
}

// Secular schedule of a batch (shared by r1_run and the allocation-free
// entry point): with many roots per CTA slot, whole problems (or 2048-root
// pieces) go to CTAs whose warps own separate root ranges; with few roots per
// slot (the top levels of a tree), units shrink so every SM gets work and the
// warps of a CTA split the poles instead of the roots.  opts.sched forces
// either mode, opts.tile_roots the unit size.
void secular_schedule(int64_t rows, int sched, int tile_roots, int slots, bool *split, int *ubig)
{
    const int64_t per = rows / slots;
    *split = (sched == 2) || (sched == 0 && per < 512);
    *ubig = SEC_UNIT_BIG / 2;
    if (*split) *ubig = (int)std::max<int64_t>(32, std::min<int64_t>(256, (per / 32) * 32));
    if (tile_roots >= 32 && tile_roots <= 4096) *ubig = (tile_roots / 32) * 32;
}

}  // namespace

cudaError_t r1_prepare() { sdc_pool(); return units_attr(); }

// ---------------------------------------------------------------------------
// Host launcher
// ---------------------------------------------------------------------------
superdc_status r1_run(const R1Args &a_in, cudaStream_t st)
{
    R1Args a = a_in;
    const int nsm = sdc_num_sms();
    double *wd = nullptr, *wz = nullptr;
    int8_t *kept = nullptr;
    int64_t *tile_off = nullptr;
    SdcScratch sc(st);
    SDC_CHECK(sc.get(&wd, a.total));
    SDC_CHECK(sc.get(&wz, a.total));
    SDC_CHECK(sc.get(&kept, a.total));
    SDC_CHECK(sc.get(&tile_off, a.nprob + 1));
    int32_t *surv = nullptr;
    SDC_CHECK(sc.get(&surv, a.total));
    SDC_CHECK(sc.get(&a.o.lamk, a.total));
    int4 *units = nullptr;
    int *ucount = nullptr;
    SDC_CHECK(sc.get(&units, 2 * a.nprob + a.total / 32 + 2));
    SDC_CHECK(sc.get(&ucount, 2));
    SDC_CHECK(units_attr());

    PROF_LAUNCH("deflate", st, launch_deflate(a, a.o, nsm > a.nprob ? 1024 : DB_T, wd, wz, kept, surv, st));
    // problems whose kept size reaches the threshold take the triangular FMM
    // path; the direct kernels below skip them
    FmmPlan fp;
    {
        const int w = a.keep ? std::min(32, a.keep_width) : 0;
        superdc_status fs = fmm_plan(fp, a.nprob, a.off, a.total, a.max_m, a.o.mk, a.o.dk, a.fmm_min_m,
                                     std::max(1, w), a.o.fmm_used, true, st);
        if (fs != SUPERDC_OK) { fmm_free(fp, st); return fs; }
    }
    const int32_t *fslot = fp.on ? fp.dv.fslot : nullptr;
    const bool dsplit = direct_split(a.rows >= 0 ? a.rows : a.total);
    PROF_LAUNCH("tiles", st, k_tiles<<<1, tiles_threads(a.nprob), 0, st>>>(a.nprob, a.o.mk, dsplit ? 32 : 128, tile_off));
    const unsigned grid = (unsigned)(nsm * 8);
    const size_t ksm = (a.nprob <= SORT_MAX) ? (size_t)SORT_MAX * sizeof(unsigned long long) : 0;
    const int slots = nsm * 6;
    bool split;
    int ubig;
    secular_schedule(a.rows >= 0 ? a.rows : a.total, a.sched, a.tile_roots, slots, &split, &ubig);
    PROF_LAUNCH("units", st, k_units<<<1, 1024, ksm, st>>>(a.nprob, a.o.mk, fslot, ubig, split ? 1 : 0, units,
                                                           ucount, ucount + 1));
    const bool lng = a.fmm_min_m <= 0 || a.fmm_min_m > LONG_M + 1;      // else the tree takes the larger ones
    const auto k_sec = split ? (lng ? k_secular<4, true, true> : k_secular<4, true, false>)
                             : (lng ? k_secular<4, false, true> : k_secular<4, false, false>);
    PROF_LAUNCH("secular", st, k_sec<<<(unsigned)slots, 128, 0, st>>>(a.off, units, ucount, ucount + 1, a.o, a.stop_c,
                                                                      a.max_iter));
    superdc_status fs = fmm_secular(fp, a.off, a.o, a.stop_c, a.max_iter, st);
    unsigned long long *tq = nullptr;          // tile queues of the direct Loewner and b kernels
    SDC_CHECK(sc.get(&tq, 2));
    SDC_CHECK(cudaMemsetAsync(tq, 0, 2 * sizeof(unsigned long long), st));
    const auto k_low = dsplit ? k_lowner<32, 8> : k_lowner<128, 1>;
    const auto k_b = dsplit ? k_bnorm<32, 8> : k_bnorm<128, 1>;
    const int dthreads = dsplit ? 256 : 128;
    PROF_LAUNCH("lowner", st, k_low<<<grid, dthreads, 0, st>>>(a.nprob, a.off, tile_off, a.o, fslot, tq));
    if (fs == SUPERDC_OK) fs = fmm_lowner(fp, a.off, a.o, st);
    PROF_LAUNCH("bnorm", st, k_b<<<grid, dthreads, 0, st>>>(a.nprob, a.off, tile_off, a.o, fslot, tq + 1));
    if (fs == SUPERDC_OK) fs = fmm_bnorm(fp, a.off, a.o, st);
    PROF_LAUNCH("merge", st, k_merge<<<(unsigned)(nsm * 8), 256, 0, st>>>(a.nprob, a.off, a.total, a.o));
    const cudaError_t le = cudaGetLastError();
    if (le != cudaSuccess) { fmm_free(fp, st); return SUPERDC_ERR_CUDA; }
    if (a.keep && fs == SUPERDC_OK) *a.keep = fp;
    else fmm_free(fp, st);
    return fs;
}

// ---------------------------------------------------------------------------
// Allocation-free variant of the batched rank-one step.
//
// Some callers cannot allocate device memory while they run: code that is
// recorded once into a CUDA graph and replayed, code on a real-time or
// latency-bound path where an allocation may block or fail, and hosts whose
// memory budget is fixed up front (a stream-ordered pool they do not own, a
// framework that has already reserved the device).  For them the scratch of
// the batched step lives in one statically sized device array that the
// library reserves when it is loaded, and the entry point below never calls
// cudaMalloc, cudaFree or any allocating routine.
//
// Limits: total entries <= SDC_NOALLOC_MAX_TOTAL, problems <= SDC_NOALLOC_MAX_PROB.
// The array is shared by every call on a device and keeps the previous call's
// contents; each call writes every scratch word before reading it (the unit
// counter is reset by k_units), so nothing has to be cleared in between.  Two
// calls whose work overlaps on the GPU (different streams, or different host
// threads on one device) race on the array: serialise them.
// ---------------------------------------------------------------------------
namespace {

constexpr int64_t NA_T = SDC_NOALLOC_MAX_TOTAL;
constexpr int64_t NA_P = SDC_NOALLOC_MAX_PROB;
constexpr size_t na_round(size_t b) { return (b + 255) & ~size_t(255); }
constexpr size_t NA_WD = 0;
constexpr size_t NA_WZ = NA_WD + na_round(NA_T * sizeof(double));
constexpr size_t NA_DORG = NA_WZ + na_round(NA_T * sizeof(double));
constexpr size_t NA_WSUM = NA_DORG + na_round(NA_T * sizeof(double));
constexpr size_t NA_TILE = NA_WSUM + na_round(NA_P * sizeof(double));
constexpr size_t NA_UNITS = NA_TILE + na_round((NA_P + 1) * sizeof(int64_t));
constexpr size_t NA_SURV = NA_UNITS + na_round((2 * NA_P + NA_T / 32 + 2) * sizeof(int4));
constexpr size_t NA_PINV = NA_SURV + na_round(NA_T * sizeof(int32_t));
constexpr size_t NA_KEPT = NA_PINV + na_round(NA_T * sizeof(int32_t));
constexpr size_t NA_UCNT = NA_KEPT + na_round(NA_T * sizeof(int8_t));
constexpr size_t NA_LAMK = NA_UCNT + na_round(2 * sizeof(int));
constexpr size_t NA_BYTES = NA_LAMK + na_round(NA_T * sizeof(double));

static __device__ __align__(256) unsigned char g_noalloc_scratch[NA_BYTES];

// Device address of g_noalloc_scratch for the current device.  In host code
// the symbol name is only a host-side stand-in, so the address is looked up
// with cudaGetSymbolAddress once per device (with that device current) and
// cached.
cudaError_t noalloc_scratch(unsigned char **ptr)
{
    static std::mutex mu;
    static unsigned char *addr[64] = {nullptr};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(mu);
    if (!addr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        addr[dev] = (unsigned char *)p;
    }
    *ptr = addr[dev];
    return cudaSuccess;
}

}  // namespace

extern "C" superdc_status superdc_secular_batched_noalloc(int64_t nprob, const int64_t *offsets, int64_t total,
                                                          const double *d, const double *z, double rho,
                                                          const superdc_opts *opts, superdc_rank1_out *out,
                                                          cudaStream_t st)
{
    superdc_opts def;
    if (!opts) { superdc_opts_default(&def); opts = &def; }
    if (nprob < 0 || total < 0 || !(rho > 0.0) || !out) return SUPERDC_ERR_ARG;
    if (!(opts->tau >= 0.0) || !(opts->stop_c > 0.0) || opts->max_iter < 1 || opts->max_iter > 10000 ||
        opts->sched < 0 || opts->sched > 2 || (opts->shifted != 0 && opts->shifted != 1))
        return SUPERDC_ERR_ARG;
    if (nprob > NA_P || total > NA_T) return SUPERDC_ERR_ARG;   // beyond the static scratch
    if (nprob == 0) return SUPERDC_OK;
    if (!offsets || !d || !z) return SUPERDC_ERR_ARG;
    if (!out->lam || !out->dk || !out->zk || !out->eta || !out->vhat || !out->bnorm || !out->org ||
        !out->src || !out->perm || !out->giv_ab || !out->giv_cs || !out->mk || !out->ngiv || !out->status)
        return SUPERDC_ERR_ARG;
    unsigned char *base = nullptr;
    SDC_CHECK(noalloc_scratch(&base));
    R1Args a;
    a.nprob = nprob; a.total = total; a.off = offsets; a.d = d; a.z = z;
    a.sqrt_rho = sqrt(rho); a.tau = opts->tau; a.stop_c = opts->stop_c; a.max_iter = opts->max_iter;
    a.tile_roots = opts->tile_roots; a.sched = opts->sched;
    a.o.lam = out->lam; a.o.dk = out->dk; a.o.zk = out->zk; a.o.eta = out->eta;
    a.o.vhat = out->vhat; a.o.bnorm = out->bnorm; a.o.org = out->org; a.o.src = out->src;
    a.o.perm = out->perm; a.o.giv_ab = out->giv_ab; a.o.giv_cs = out->giv_cs; a.o.mk = out->mk;
    a.o.ngiv = out->ngiv; a.o.sweeps = out->sweeps; a.o.status = out->status;
    a.o.unshifted = opts->shifted ? 0 : 1;
    a.o.dorg = (double *)(base + NA_DORG);
    a.o.wsum = (double *)(base + NA_WSUM);
    a.o.pinv = (int32_t *)(base + NA_PINV);
    a.o.lamk = (double *)(base + NA_LAMK);
    if (out->fmm) SDC_CHECK(cudaMemsetAsync(out->fmm, 0, (size_t)nprob * sizeof(int32_t), st));   // direct only
    double *wd = (double *)(base + NA_WD), *wz = (double *)(base + NA_WZ);
    int8_t *kept = (int8_t *)(base + NA_KEPT);
    int64_t *tile_off = (int64_t *)(base + NA_TILE);
    int32_t *surv = (int32_t *)(base + NA_SURV);
    int4 *units = (int4 *)(base + NA_UNITS);
    int *ucount = (int *)(base + NA_UCNT);
    SDC_CHECK(units_attr());
    const int nsm = sdc_num_sms();
    launch_deflate(a, a.o, DB_T, wd, wz, kept, surv, st);
    const bool dsplit = direct_split(a.total);
    k_tiles<<<1, tiles_threads(a.nprob), 0, st>>>(a.nprob, a.o.mk, dsplit ? 32 : 128, tile_off);
    const unsigned grid = (unsigned)(nsm * 8);
    const size_t ksm = (a.nprob <= SORT_MAX) ? (size_t)SORT_MAX * sizeof(unsigned long long) : 0;
    const int slots = nsm * 6;
    bool split;
    int ubig;
    secular_schedule(a.total, a.sched, a.tile_roots, slots, &split, &ubig);
    k_units<<<1, 1024, ksm, st>>>(a.nprob, a.o.mk, nullptr, ubig, split ? 1 : 0, units, ucount, ucount + 1);
    const auto k_sec = split ? k_secular<4, true, true> : k_secular<4, false, true>;
    k_sec<<<(unsigned)slots, 128, 0, st>>>(a.off, units, ucount, ucount + 1, a.o, a.stop_c, a.max_iter);
    const auto k_low = dsplit ? k_lowner<32, 8> : k_lowner<128, 1>;
    const auto k_b = dsplit ? k_bnorm<32, 8> : k_bnorm<128, 1>;
    const int dthreads = dsplit ? 256 : 128;
    k_low<<<grid, dthreads, 0, st>>>(a.nprob, a.off, tile_off, a.o, nullptr, nullptr);
    k_b<<<grid, dthreads, 0, st>>>(a.nprob, a.off, tile_off, a.o, nullptr, nullptr);
    k_merge<<<(unsigned)(nsm * 8), 256, 0, st>>>(a.nprob, a.off, a.total, a.o);
    SDC_CHECK(cudaGetLastError());
    return SUPERDC_OK;
}
