// Triangular FMM with local shifting on sm_103a (Sections 4.1.2, 4.2.2, 4.3).
//
// Geometry.  The kept poles d_0 < ... < d_{m-1} of a problem and the targets
// (roots x_k in (d_k, d_{k+1}), eigenvalues lambda_j, or the poles themselves)
// interlace (eq. (4.4)), so one index-based binary tree serves both: a leaf
// box holds B = 32 consecutive indices, so d_k and x_k of the same k
// always share a box (the paper's first design point), and every box carries the interval
// [d_{i0}, d_{i1}] of its points (the last box ends at d_{m-1}).  The index
// split adapts the boxes to clustered spectra (second design point); whether
// two boxes interact through expansions is decided geometrically: boxes S, T
// of one level are admissible when their gap is at least FMM_KAPPA times the
// larger width.  Near lists are built top-down (children of the parent's near
// list that are not admissible) and have any length (a wide box, e.g. in a
// tail of the spectrum, is close to many boxes; its narrow children are not).
// Only when the list pool is exhausted is a box marked "all near", with its
// subtree: the targets of such leaves are summed directly over every source.
// Only the last eigenvalue lambda_{m-1} lies outside the tree (to the right of
// d_{m-1}): as a target its sums run over the tree (node weights of the boxes
// far from it, direct sums over the leaf boxes next to it) or are spread over
// the leaf boxes; as a source it is added directly to every target.
//
// Expansions.  Chebyshev interpolation with FMM_P first-kind nodes per box: node
// weights W_q = sum_j w_j L_q(u_j) of the leaf boxes, parents' weights from the
// children's nodes (upward pass: k_fmm_up1 for one column, k_cm_up for blocks of
// columns, k_fmm_up for problems out of the split arithmetic's scale).  Every leaf
// box then sums the node weights of the boxes in the interaction lists (children of
// the parent's near list that are admissible) of itself and of its ancestors: at its
// own Chebyshev nodes for the one-column fields (k_fmm_far), whose coefficients are
// evaluated at the targets; at the targets themselves for blocks of columns
// (k_cm_apply).  There is no translation between boxes and no downward pass: in split
// FP32 arithmetic and on the tensor cores a node sum costs less than reading or
// forming a translation matrix.  Work is O(m P log m) for the far field plus O(m B)
// for the near field.
//
// Triangularity.  A far box lies entirely to the left or right of the target
// box in index order, so its sums go to the lower (psi, C_L w, S_L w) or the
// upper (phi, C_U w, S_U w) part; inside the near field the split is by index
// as in the direct evaluator (eq. (4.10)).
//
// Local shifting.  Near-field terms use the shifted differences of eqs.
// (4.14)/(4.28) exactly as the direct kernels; far-field terms use the plain
// positions x = d_K + y and lambda_j = d_{K_j} + eta_j (eq. (4.21)), which is
// accurate there because far points are separated by at least a box width.
//
// Because the poles and weights of a secular equation do not change during
// the iteration and every root stays inside its bracket, the far-field
// expansions on the leaf boxes' (fixed) intervals are computed once per
// problem; each sweep costs a near-field pass plus one series evaluation.
#include <algorithm>
#include <mutex>
#include "common.cuh"
#include "fmm.cuh"
#include "secular.cuh"
#include "prof.cuh"
#include "tiles.cuh"

namespace {

constexpr int P = FMM_P;
constexpr int B = 32;             // indices per leaf box
// admissibility: gap >= 0.75 x the larger width.  The nearest source then lies
// at least 2.5 half-widths from either box's centre (Bernstein ellipse
// rho >= 2.5 + sqrt(5.25) = 4.79): at 22 nodes the interpolated 1/(s-t) stays at
// the rounding floor (~1e-14 relative) and 1/(s-t)^2 within ~1e-13 over box-width
// ratios 1e-3..1e3, while index-based boxes of random spectra drop from ~4.3
// to ~3.2-3.4 near boxes per leaf (with 1.0 the box between two neighbours must
// be at least as wide as both, which a random width sequence meets a third of
// the time)
constexpr double FMM_KAPPA = 0.75;   // 3 / 4 in adm
constexpr int SPLIT_NEAR = 512 / B;   // leaf boxes with this many near boxes (512 poles) or more: CTA-split sweeps
constexpr int TAIL_X = 12;        // k_secular_fmm hands a box's last roots to the tail pass below this many busy lanes
constexpr int WMAX = 32;          // widest moment block (columns)
constexpr int NFIELD = 4;         // series per leaf box (P doubles each)

// ---------------------------------------------------------------------------
// tree shape of a problem with m kept indices: nb0 = ceil(m / B) leaf boxes,
// level l has ceil(nb0 / 2^l) boxes, the top level one box; boxes of a problem
// are stored level by level from the leaves up.
// ---------------------------------------------------------------------------
__host__ __device__ __forceinline__ int lev_nb(int nb0, int l) { return ((nb0 - 1) >> l) + 1; }

__host__ __device__ __forceinline__ int lev_count(int nb0)
{
    int L = 1;
    while (lev_nb(nb0, L - 1) > 1) L++;
    return L;
}

__host__ __device__ __forceinline__ int lev_base(int nb0, int l)
{
    int s = 0;
    for (int i = 0; i < l; i++) s += lev_nb(nb0, i);
    return s;
}

__device__ __forceinline__ bool fmm_cand(int m, int min_m) { return min_m > 0 && m >= min_m && m >= 4 * B; }

__device__ __forceinline__ void box_range(int m, int l, int b, int &i0, int &i1)
{
    const int64_t span = (int64_t)B << l;
    const int64_t a = (int64_t)b * span;
    i0 = (int)a;
    i1 = (int)std::min<int64_t>((int64_t)m, a + span);
}

__device__ __forceinline__ void box_ch(double lo, double hi, double &c, double &h)
{
    c = 0.5 * (lo + hi);
    h = 0.5 * (hi - lo);
    if (!(h > 0.0)) h = fmax(fabs(c) * 1e-15, 1e-300);
}

// on the boxes' integer intervals (60 bits of the split positions: an FP64
// comparison costs the issue slots of 64 integer ones, and the tree of a large
// problem is built by one CTA).  Good to a part in COARSE of the boxes' widths; a
// problem with narrower leaf boxes (poles graded over many orders of magnitude) or
// out of the positions' scale takes the FP64 form, for lack of which half of 40000
// poles graded over 25 decades saw each other directly: step 186 ms against 3.1
constexpr long long COARSE = 1ll << 20;
__device__ __forceinline__ bool adm(longlong2 S, longlong2 T)
{
    const long long gap = max(T.x - S.y, S.x - T.y);
    return gap > 0 && 4 * gap >= 3 * max(S.y - S.x, T.y - T.x);
}

__device__ __forceinline__ bool adm64(double loS, double hiS, double loT, double hiT)
{
    const double gap = fmax(loT - hiS, loS - hiT);
    return gap > 0.0 && gap >= FMM_KAPPA * fmax(hiS - loS, hiT - loT);
}

__device__ __forceinline__ bool adm_box(const FmmDev &pl, int64_t S, int64_t T, bool coarse)
{
    return coarse ? adm64(pl.blo[S], pl.bhi[S], pl.blo[T], pl.bhi[T]) : adm(pl.ibox[S], pl.ibox[T]);
}

// near list of a leaf box: nn >= 0 entries, or (nn < 0) every leaf box
__device__ __forceinline__ int near_len(int nn, int nb0) { return nn < 0 ? nb0 : nn; }
__device__ __forceinline__ int near_box(const FmmDev &pl, int64_t g, int nn, int i)
{
    return nn < 0 ? i : pl.near[pl.nstart[g] + i];
}
// a near box of a consumer kernel: in the checked build the list entry is
// tested against the problem's leaf box count nb0 (latched into word)
__device__ __forceinline__ int near_box_chk(const FmmDev &pl, int64_t g, int nn, int i, int nb0, int32_t *word)
{
    return SDC_IDX(near_box(pl, g, nn, i), nb0, word);
}

// Chebyshev nodes x_q = cos((2q+1) pi / 2P) and T_n(x_q) (Tx[q * P + n], by
// the three-term recurrence, one row per thread); the caller synchronises
// before the first use.  sc scales the entries n >= 1 (2: the weights of the
// moments -> node weights sums, exact, saving a multiply per term)
__device__ __forceinline__ void cheb_tables(double *xq, double *Tx, double sc = 1.0)
{
    for (int q = threadIdx.x; q < P; q += blockDim.x) {
        const double x = cospi((double)(2 * q + 1) / (2.0 * P));
        xq[q] = x;
        double t0 = 1.0, t1 = x;
        Tx[q * P] = 1.0;
        Tx[q * P + 1] = sc * x;
        for (int n = 2; n < P; n++) {
            const double t2 = 2.0 * x * t1 - t0;
            Tx[q * P + n] = sc * t2;
            t0 = t1; t1 = t2;
        }
    }
}

// Clenshaw evaluation of sum_n a_n T_n(u)
__device__ __forceinline__ double clenshaw(const double *__restrict__ a, double u)
{
    const double u2 = u + u;
    double b1 = 0.0, b2 = 0.0;
#pragma unroll 4
    for (int n = P - 1; n >= 1; n--) {
        const double b0 = fma(u2, b1, a[n] - b2);
        b2 = b1;
        b1 = b0;
    }
    return fma(u, b1, a[0] - b2);
}

// algorithmic work counter (profiling): one add per box by thread 0
__device__ __forceinline__ void fl_add(const FmmDev &pl, int64_t v)
{
    if (pl.flops && threadIdx.x == 0 && v > 0) atomicAdd(pl.flops, (unsigned long long)v);
}

// ---------------------------------------------------------------------------
// Plan: which problems take the FMM path, and the prefix of their boxes.
// ---------------------------------------------------------------------------
__global__ void k_fmm_plan(int64_t nprob, const int32_t *__restrict__ mk, int min_m, int64_t cap_boxes,
                           int64_t cap_leaves, int64_t cap_f, int64_t *__restrict__ box_base,
                           int64_t *__restrict__ leaf_base, int32_t *__restrict__ fslot,
                           int32_t *__restrict__ fprob, int32_t *__restrict__ nfmm)
{
    __shared__ int64_t sh[32];
    const int T = blockDim.x;
    const int64_t per = (nprob + T - 1) / T;
    const int64_t beg = std::min<int64_t>(nprob, (int64_t)threadIdx.x * per);
    const int64_t end = std::min<int64_t>(nprob, beg + per);
    int64_t nbx = 0, nlf = 0, nf = 0;
    for (int64_t p = beg; p < end; p++) {
        const int m = mk[p];
        if (!fmm_cand(m, min_m)) continue;
        const int nb0 = (m + B - 1) / B;
        nbx += lev_base(nb0, lev_count(nb0));
        nlf += nb0;
        nf++;
    }
    int64_t tb, tl, tf;
    int64_t ab = cta_exscan(nbx, sh, &tb), al = cta_exscan(nlf, sh, &tl);
    int af = (int)cta_exscan(nf, sh, &tf);
    const bool ok = tb <= cap_boxes && tl <= cap_leaves && tf <= cap_f;
    if (!ok) { ab = 0; al = 0; }
    if (threadIdx.x == 0) {
        box_base[nprob] = ok ? tb : 0;
        leaf_base[nprob] = ok ? tl : 0;
        *nfmm = ok ? (int)tf : 0;
    }
    for (int64_t p = beg; p < end; p++) {
        box_base[p] = ab;
        leaf_base[p] = al;
        const int m = mk[p];
        if (ok && fmm_cand(m, min_m)) {
            const int nb0 = (m + B - 1) / B;
            fslot[p] = af;
            fprob[af] = (int32_t)p;
            ab += lev_base(nb0, lev_count(nb0));
            al += nb0;
            af++;
        } else {
            fslot[p] = -1;
        }
    }
}

// Box intervals and near lists, one CTA per problem, top level first.  Near
// lists have any length; they are stored back to back in the problem's share
// of the pool (FMM_NPOOL entries per box on average).  A box whose list no
// longer fits, and its subtree, is marked "all near" (nnear = -1).  A warp takes
// a contiguous segment of a level, a lane per box; the candidates (children of
// the parent's near boxes) that are admissible are the box's interaction list,
// kept as a bit mask (the first 64), the others its near list.
// Measured (GB300, one problem of 100003 poles): 0.43 -> 0.09 ms.
__device__ __forceinline__ unsigned long long adm_mask(const FmmDev &pl, int64_t gb, int nbl, int A, int64_t pst,
                                                       int npn, int sec, bool coarse)
{
    unsigned long long mask = 0;
    const int end = min(2 * npn, 64 * sec + 64);
    if (coarse) {
        for (int c = 64 * sec; c < end; c++) {
            const int S = 2 * pl.near[pst + (c >> 1)] + (c & 1);
            if (S < nbl && S != A && adm_box(pl, gb + S, gb + A, true)) mask |= 1ull << (c & 63);
        }
        return mask;
    }
    const longlong2 T = pl.ibox[gb + A];
#pragma unroll 4
    for (int c = 64 * sec; c < end; c++) {
        const int S = 2 * pl.near[pst + (c >> 1)] + (c & 1);
        if (S < nbl && S != A && adm(pl.ibox[gb + S], T)) mask |= 1ull << (c & 63);
    }
    return mask;
}

__global__ void __launch_bounds__(1024)
k_fmm_tree(FmmDev pl, const int64_t *__restrict__ off, const int32_t *__restrict__ mk, const double *__restrict__ dk,
           double *__restrict__ blo, double *__restrict__ bhi, int32_t *__restrict__ nnear,
           int64_t *__restrict__ nstart, int32_t *__restrict__ near, int32_t *__restrict__ used)
{
    __shared__ int64_t wsum[32];
    const unsigned FULL = 0xffffffffu;
    const int T = blockDim.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t p = blockIdx.x; p < pl.nprob; p += gridDim.x) {
        if (pl.fslot[p] < 0) continue;
        const int m = mk[p];
        const double *d = dk + off[p];
        const int64_t g0 = pl.box_base[p];
        const int64_t pool_end = pl.box_base[p + 1] * FMM_NPOOL;
        const int nb0 = (m + B - 1) / B;
        const int L = lev_count(nb0);
        const FfScale fs = ff_scale(d[0], d[m - 1], 1.0);
        // intervals of every level at once
        int64_t gb = g0;
        bool narrow = !fs.ok;
        for (int l = 0; l < L; l++) {
            const int nb = lev_nb(nb0, l);
            for (int b = threadIdx.x; b < nb; b += T) {
                int i0, i1;
                box_range(m, l, b, i0, i1);
                const double lo = d[i0], hi = (i1 < m) ? d[i1] : d[m - 1];
                blo[gb + b] = lo;
                bhi[gb + b] = hi;
                longlong2 v = make_longlong2(0, 0);
                if (fs.ok) {
                    v.x = (long long)((ff_fixed(lo, fs.kk) - fs.ref) >> 34);
                    v.y = (long long)((ff_fixed(hi, fs.kk) - fs.ref) >> 34);
                    narrow = narrow || (l == 0 && b + 1 < nb && v.y - v.x < COARSE);
                }
                pl.ibox[gb + b] = v;
            }
            gb += nb;
        }
        const bool coarse = __syncthreads_or(narrow);
        if (threadIdx.x == 0) pl.coarse[p] = coarse ? 1 : 0;
        int64_t pos0 = g0 * FMM_NPOOL;                   // pool position of the level
        for (int l = L - 1; l >= 0; l--) {
            __syncthreads();
            const int nb = lev_nb(nb0, l);
            gb = g0 + lev_base(nb0, l);
            const int64_t gp0 = (l < L - 1) ? g0 + lev_base(nb0, l + 1) : 0;
            const int seg = ((nb + T - 1) / T) * 32, beg = min(nb, warp * seg), end = min(nb, beg + seg);
            // near counts (nnear holds them until the lists are placed)
            int64_t sum = 0;
            for (int c = beg; c < end; c += 32) {
                const int b = c + lane;
                int cnt = 0;
                if (b < end) {
                    unsigned long long mask = 0;
                    if (l == L - 1) cnt = 1;
                    else {
                        const int npn = nnear[gp0 + (b >> 1)];
                        if (npn < 0) cnt = -1;
                        else {
                            const int64_t pst = nstart[gp0 + (b >> 1)];
                            mask = adm_mask(pl, gb, nb, b, pst, npn, 0, coarse);
                            int far = __popcll(mask);
                            for (int sec = 1; 64 * sec < 2 * npn; sec++)
                                far += __popcll(adm_mask(pl, gb, nb, b, pst, npn, sec, coarse));
                            // a candidate beyond the level's last box is neither
                            cnt = 2 * npn - far - ((nb & 1) && near[pst + npn - 1] == (nb >> 1) ? 1 : 0);
                        }
                    }
                    nnear[gb + b] = cnt;
                    pl.amask[gb + b] = mask;
                }
                sum += max(cnt, 0);
            }
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(FULL, sum, o);
            if (lane == 0) wsum[warp] = sum;
            __syncthreads();
            int64_t pos = pos0, all = 0;
            for (int w = 0; w < T / 32; w++) {
                const int64_t v = wsum[w];
                pos += (w < warp) ? v : 0;
                all += v;
            }
            pos0 += all;
            // the lists, in box order
            for (int c = beg; c < end; c += 32) {
                const int b = c + lane;
                const int cnt = (b < end) ? nnear[gb + b] : 0;
                int x = max(cnt, 0);
                const int own = x;
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(FULL, x, o);
                    if (lane >= o) x += y;
                }
                const int64_t at = pos + x - own;
                pos += __shfl_sync(FULL, x, 31);
                if (b >= end) continue;
                nstart[gb + b] = at;
                bool fits = cnt >= 0;
                if (cnt >= 0) {
                    if (at + cnt > pool_end) {                                  // pool exhausted: all near
                        fits = false;
                        nnear[gb + b] = -1;
                        pl.amask[gb + b] = 0;
                    } else if (l == L - 1) {
                        near[at] = b;
                    } else {
                        const int64_t pst = nstart[gp0 + (b >> 1)];
                        const int npn = nnear[gp0 + (b >> 1)];
                        unsigned long long mask = pl.amask[gb + b];
                        int w = 0;
                        for (int k = 0; k < 2 * npn; k++) {
                            if (k > 0 && (k & 63) == 0) mask = adm_mask(pl, gb, nb, b, pst, npn, k >> 6, coarse);
                            const int S = 2 * near[pst + (k >> 1)] + (k & 1);
                            if (S < nb && !((mask >> (k & 63)) & 1)) near[at + w++] = S;
                        }
                    }
                }
                // leaf boxes with long near lists, for k_secular_fmm_split (in
                // any order: each box's sweeps are independent of the others)
                if (l == 0 && (!fits || cnt >= SPLIT_NEAR)) pl.split[atomicAdd(pl.nsplit, 1)] = pl.leaf_base[p] + b;
            }
        }
        if (threadIdx.x == 0 && used) used[p] = 1;
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Sources of the five sums
// ---------------------------------------------------------------------------
enum { M_SEC = 0, M_BN = 1, M_LOW = 2, M_CT = 3, M_CN = 4 };

struct SrcArgs {
    const int64_t *off;
    const int32_t *mk;
    const double *dk, *zk, *vhat, *bnorm, *dorg, *eta;
    const double *wsum;                  // one-column modes: scale of the split node weights
    const int32_t *src, *pinv;
    const double *X;
    int64_t ldx;
    int col0, nc;
#ifdef SUPERDC_CHECK
    int32_t *status;                     // index guards
#endif
    const int32_t *only;                 // the problems with only[p] != 0 (out of scale); the others
                                         // are k_fmm_up1's and k_cm_up's
};

// leaf moments and node weights of leaf box gl (box g, index Tb within its
// problem p); one thread per source (threads B.. only join the sums)
//   M_SEC: w_j = z_j^2 at d_j            M_BN: w_i = vhat_i^2 at d_i
//   M_LOW: +1 at lambda_j, -1 at d_j (j < m-1; Chebyshev differences of the pair)
//   M_CT:  vhat_i x_{src_i} at d_i       M_CN: b_j x_{pinv_j} at lambda_j (j < m-1)
constexpr int UP_ROWS = (B > 2 * P) ? B : 2 * P;   // rows of the staging arrays (sources, or 2 children x P)

template <int MODE, int WW>
__device__ __forceinline__ void leaf_moments(const FmmDev &pl, const SrcArgs &a, int64_t p, int64_t gl, int64_t g,
                                             int Tb, int nw, double (*Tt)[P + 1], double (*Wt)[WW + 1],
                                             double (*Ms)[WW + 1], const double *Tx)
{
    const int tid = threadIdx.x;
    const int64_t b0 = a.off[p];
    const int m = a.mk[p];
    double c, h;
    box_ch(pl.blo[g], pl.bhi[g], c, h);
    const int j = Tb * B + tid;
    const int jend = (MODE == M_LOW || MODE == M_CN) ? m - 1 : m;
    const bool act = tid < B && j < jend;
    __syncthreads();
    if (tid < B) {
        if (MODE == M_LOW) {
            // D_n = T_n(b) - T_n(a) with b = a + delta, by the recurrence
            // D_{n+1} = 2 delta T_n(b) + 2 a D_n - D_{n-1} (no cancellation)
            double av = 0.0, dl = 0.0;
            if (act) {
                const double ih = 1.0 / h;
                av = (a.dk[b0 + j] - c) * ih;
                dl = ((a.dorg[b0 + j] - a.dk[b0 + j]) + a.eta[b0 + j]) * ih;
            }
            const double bv = av + dl;
            double tb0 = 1.0, tb1 = bv, D0 = 0.0, D1 = dl;
            Tt[tid][0] = 0.0;
            Tt[tid][1] = D1;
            for (int n = 1; n < P - 1; n++) {
                const double D2 = 2.0 * dl * tb1 + 2.0 * av * D1 - D0;
                const double tb2 = 2.0 * bv * tb1 - tb0;
                Tt[tid][n + 1] = D2;
                D0 = D1; D1 = D2; tb0 = tb1; tb1 = tb2;
            }
            Wt[tid][0] = act ? 1.0 : 0.0;
        } else {
            double u = 0.0;
            if (act) {
                const double s = (MODE == M_CN) ? a.dorg[b0 + j] + a.eta[b0 + j] : a.dk[b0 + j];
                u = (s - c) / h;
            }
            double t0 = 1.0, t1 = u;
            Tt[tid][0] = 1.0;
            Tt[tid][1] = u;
            for (int n = 2; n < P; n++) {
                const double t2 = 2.0 * u * t1 - t0;
                Tt[tid][n] = t2;
                t0 = t1; t1 = t2;
            }
            if (MODE == M_SEC) {
                const double z = act ? a.zk[b0 + j] : 0.0;
                Wt[tid][0] = z * z;
            } else if (MODE == M_BN) {
                const double v = act ? a.vhat[b0 + j] : 0.0;
                Wt[tid][0] = v * v;
            }
        }
    }
    if (MODE == M_CT || MODE == M_CN) {
        // the columns by all warps, a lane per source
        const int js = Tb * B + (tid & 31);
        const bool in = js < jend;
        const double v = in ? (MODE == M_CT ? a.vhat[b0 + js] : a.bnorm[b0 + js]) : 0.0;
        const int64_t row = in ? b0 + SDC_IDX(MODE == M_CT ? a.src[b0 + js] : a.pinv[b0 + js], a.off[p + 1] - b0, a.status) : 0;
#pragma unroll 4
        for (int q = tid >> 5; q < nw; q += (int)blockDim.x >> 5)
            Wt[tid & 31][q] = in ? v * a.X[row + (int64_t)(a.col0 + q) * a.ldx] : 0.0;
    }
    __syncthreads();
    for (int t = tid; t < P * nw; t += blockDim.x) {
        const int n = t / nw, q = t % nw;
        double s = 0.0;
        for (int jj = 0; jj < B; jj++) s = fma(Tt[jj][n], Wt[jj][q], s);
        Ms[n][q] = s;
    }
    __syncthreads();
    for (int t = tid; t < P * nw; t += blockDim.x) {
        const int qn = t / nw, q = t % nw;
        double s = Ms[0][q];
        for (int n = 1; n < P; n++) s = fma(Tx[qn * P + n], Ms[n][q], s);     // Tx holds 2 T_n
        pl.W[(g * P + qn) * pl.ncol + q] = s * (1.0 / P);
    }
    // Chebyshev recurrence per source, moments, moments -> node weights
    const int64_t cnt = max(0, min(B, jend - Tb * B));
    fl_add(pl, cnt * ((MODE == M_LOW) ? 4 : 2) * (P - 2) + 2 * cnt * P * nw + 2 * P * P * nw);
}

// moments of box g (level l >= 1, index b) from its children's node weights:
// M_n(parent) = sum_children sum_q W_q(child) T_n(alpha x_q + beta), exact
// because T_n(alpha u + beta) has degree n < P and the children's weights
// reproduce every moment of degree < P.  The children's weights are read
// through L2 (ld.global.cg): the sibling's were written by another CTA of the
// same launch, which published them before its arrival count.
template <int WW>
__device__ __forceinline__ void m2m_box(const FmmDev &pl, int64_t p, int nb0, int l, int b, int64_t g, int nw,
                                        double (*Tv)[P + 1], double (*Wc)[WW + 1], double (*Ms)[WW + 1],
                                        const double *Tx, const double *xq)
{
    const int tid = threadIdx.x;
    double cP = 0.0, ihP = 1.0;
    if (tid < 2 * P) {                 // the threads that build Tv (uniform FP64 work costs every warp)
        double hP;
        box_ch(pl.blo[g], pl.bhi[g], cP, hP);
        ihP = rcp_nr2(hP);
    }
    const int nbc = lev_nb(nb0, l - 1);
    const int64_t gcb = pl.box_base[p] + lev_base(nb0, l - 1);
    const int nch = (2 * b + 1 < nbc) ? 2 : 1;
    __syncthreads();
    for (int t = tid; t < 2 * P; t += blockDim.x) {
        const int ci = t / P, q = t % P;
        if (ci >= nch) continue;
        const int64_t gc = gcb + 2 * b + ci;
        double cc, hc;
        box_ch(pl.blo[gc], pl.bhi[gc], cc, hc);
        const double v = fma(hc * ihP, xq[q], (cc - cP) * ihP);    // as scale and shift (see far64)
        double t0 = 1.0, t1 = v;
        Tv[t][0] = 1.0;
        Tv[t][1] = v;
        for (int n = 2; n < P; n++) {
            const double t2 = 2.0 * v * t1 - t0;
            Tv[t][n] = t2;
            t0 = t1; t1 = t2;
        }
    }
    for (int t = tid; t < 2 * P * nw; t += blockDim.x) {
        const int ci = t / (P * nw), r = t % (P * nw);
        if (ci >= nch) continue;
        const int64_t gc = gcb + 2 * b + ci;
        Wc[ci * P + r / nw][r % nw] = __ldcg(&pl.W[(gc * P + r / nw) * pl.ncol + r % nw]);
    }
    __syncthreads();
    for (int t = tid; t < P * nw; t += blockDim.x) {
        const int n = t / nw, q = t % nw;
        double s = 0.0;
        for (int ci = 0; ci < nch; ci++)
            for (int k = 0; k < P; k++) s = fma(Tv[ci * P + k][n], Wc[ci * P + k][q], s);
        Ms[n][q] = s;
    }
    __syncthreads();
    for (int t = tid; t < P * nw; t += blockDim.x) {
        const int qn = t / nw, q = t % nw;
        double s = Ms[0][q];
        for (int n = 1; n < P; n++) s = fma(Tx[qn * P + n], Ms[n][q], s);     // Tx holds 2 T_n
        pl.W[(g * P + qn) * pl.ncol + q] = s * (1.0 / P);
    }
    // children's node positions, the children's weights into moments, moments -> weights
    fl_add(pl, (int64_t)nch * 2 * P * (P - 2) + (int64_t)nch * 2 * P * P * nw + 2 * P * P * nw);
}

// The whole upward pass in one launch: the leaf boxes' moments and node
// weights (grid-stride over the leaf boxes of the FMM problems), then each
// box climbs towards its problem's top box.  A box that has finished its
// weights counts itself into its parent's arrival counter (after a device-
// scope fence); the child that arrives last computes the parent and climbs
// on, the other stops.  No CTA ever waits for another, so any grid size and
// any scheduling order are safe, and every box is computed exactly once, by
// the same arithmetic as a level-by-level pass.  The counter is reset by the
// child that consumes it, ready for the next far field built on the plan.
// Threads and staged columns of the upward pass: the one-column far fields
// (secular, b, Loewner) take 64 threads (the 2P children's nodes of a box), the
// Cauchy-like ones 256 and WMAX columns (64 columns through 20000 poles, both ways:
// 128 threads 2.56 ms, 256 2.19).
template <int MODE> constexpr bool up_wide() { return MODE == M_CT || MODE == M_CN; }
template <int MODE> constexpr int up_threads() { return up_wide<MODE>() ? 256 : 64; }
template <int MODE> constexpr int up_cols() { return up_wide<MODE>() ? WMAX : 1; }

template <int MODE>
__global__ void __launch_bounds__(up_threads<MODE>()) k_fmm_up(FmmDev pl, SrcArgs a)
{
    constexpr int WW = up_cols<MODE>();
    __shared__ double Tt[UP_ROWS][P + 1];
    __shared__ double Wt[UP_ROWS][WW + 1];
    __shared__ double Ms[P][WW + 1];
    __shared__ double Tx[P * P], xq[P];
    __shared__ int last;
    __shared__ int64_t next;
    if (a.only[pl.nprob] == 0) return;             // no problem out of scale
    cheb_tables(xq, Tx, 2.0);          // 2 T_n(x_q), n >= 1: the moments -> weights sums
    const int nw = (MODE == M_CT || MODE == M_CN) ? a.nc : 1;
    const int tid = threadIdx.x;
    const int64_t nleaf = pl.leaf_base[pl.nprob];
    for (;;) {
        // leaf boxes are claimed one at a time: a CTA that climbs takes fewer
        // (a fixed stride would pile the climbs onto the CTAs that start late)
        __syncthreads();
        if (tid == 0) {
            next = (int64_t)atomicAdd(&pl.upq[0], 1ull);
            if (next >= nleaf && atomicAdd(&pl.upq[1], 1ull) == gridDim.x - 1) {
                pl.upq[0] = 0;                 // every CTA has run past the end: reset for the next launch
                pl.upq[1] = 0;
            }
        }
        __syncthreads();
        const int64_t gl = next;
        if (gl >= nleaf) break;
        const int64_t p = sdc_upper_index(pl.leaf_base, pl.nprob, gl);
        if (pl.fslot[p] < 0 || a.only[p] == 0) continue;
        const int Tb = (int)(gl - pl.leaf_base[p]);
        const int64_t g = pl.box_base[p] + Tb;
        leaf_moments<MODE, WW>(pl, a, p, gl, g, Tb, nw, Tt, Wt, Ms, Tx);
        const int nb0 = (a.mk[p] + B - 1) / B;
        const int L = lev_count(nb0);
        // the two top levels' boxes are in no interaction list (the last root's sums
        // take them, one column)
        const int lend = up_wide<MODE>() ? L - 2 : L;
        int l = 0, b = Tb;
        while (l + 1 < lend) {
            const int bp = b >> 1;
            const int nch = (2 * bp + 1 < lev_nb(nb0, l)) ? 2 : 1;
            const int64_t gp = pl.box_base[p] + lev_base(nb0, l + 1) + bp;
            __threadfence();               // this box's weights, visible before the count
            __syncthreads();
            if (tid == 0) {
                const int old = atomicAdd(&pl.upcnt[gp], 1);
                last = (old == nch - 1);
                if (last) pl.upcnt[gp] = 0;
            }
            __syncthreads();
            if (!last) break;
            __threadfence();
            m2m_box<WW>(pl, p, nb0, l + 1, bp, gp, nw, Tt, Wt, Ms, Tx, xq);
            l++;
            b = bp;
        }
    }
}

// ---------------------------------------------------------------------------
// The upward pass of the one-column sums in split arithmetic, one warp per box:
// the weight of node q is sum_j f_j w_q / (u_j - x_q), f_j = (weight of source
// j) / sum_k w_k / (u_j - x_k) (second barycentric formula; the sources are a
// leaf's poles, or the nodes of a box's children).  First a lane per source for
// f, then a lane per node.  The secular sums (M_SEC) take blocks of 8
// with three-float totals and f by a three-float quotient: with two floats all
// through the weights' error grows with every level (against quadruple precision,
// random leaves: 3.5e-15 there, 5.6e-15 three levels up, 2e-14 in the last root of
// 60000 poles; so 1.6e-15 to 1.9e-15 on every level and 3e-15).  The dipoles of zhat (lambda_j minus d_j, nearly
// cancelling) keep FP64 at the leaves: the moments' own difference recurrence.
// Climb and counters as in k_fmm_up, which does the problems out of scale.
// Measured (GB300, 4096 problems of 32..2048 poles): 1.9 + 1.9 + 2.3 -> 1.1 + 1.1 + 1.4 ms
// (secular, b, zhat).
// ---------------------------------------------------------------------------
template <int MODE>
__global__ void __launch_bounds__(128) k_fmm_up1(FmmDev pl, SrcArgs a)
{
    __shared__ double xq[P], wq[P], Tx[(MODE == M_LOW) ? P * P : 1];
    __shared__ double Tt[(MODE == M_LOW) ? 4 : 1][(MODE == M_LOW) ? B : 1][P + 1];
    __shared__ ff_f2 sx[P], sw[P], su[4][2 * P], sf[4][2 * P];
    const unsigned FULL = 0xffffffffu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (MODE == M_LOW) cheb_tables(xq, Tx, 2.0);
    if (threadIdx.x < P) {
        const int q = threadIdx.x;
        const double w = sinpi((double)(2 * q + 1) / (2.0 * P));
        if (MODE != M_LOW) xq[q] = cospi((double)(2 * q + 1) / (2.0 * P));
        wq[q] = (q & 1) ? -w : w;
        sx[q] = ff_weight(xq[q], 0);
        sw[q] = ff_weight(wq[q], 0);
    }
    __syncthreads();
    // d = u - x, away from zero (on a node: its weight is one, the others' 2^-60)
    auto diff = [&](const ff_f2 &u, const ff_f2 &x, float &t, float &tl) {
        float s, e;
        ff_two_sum(u.x, -x.x, s, e);
        ff_fast_sum(s, ff_add(e, ff_sub(u.y, x.y)), t, tl);
        if (fabsf(t) < 0x1p-60f) { t = 0x1p-60f; tl = 0.0f; }
    };
    // f of the source in this lane
    auto factor = [&](const ff_f2 &u, const ff_f2 &w) {
        FfAcc D = {};
#pragma unroll
        for (int q = 0; q < P; q++) {
            float t, tl, p, pr;
            diff(u, sx[q], t, tl);
            ff_div(sw[q], t, tl, p, pr);
            ff_addto(D, p, pr);
            if ((q & 7) == 7) { if (MODE == M_SEC) ff_close3(D); else ff_norm(D); }
        }
        if (MODE != M_SEC) {
            ff_norm(D);
            ff_f2 f;
            ff_div(w, D.b, D.bl, f.x, f.y);
            return f;
        }
        ff_close3(D);
        const ff_t3 f = ff_mul3({w.x, w.y, 0.0f}, ff_rcp3({D.s, D.sl, D.c}));
        ff_f2 r;
        r.x = f.a;
        r.y = ff_add(f.b, f.c);
        return r;
    };
    // weight of node lane from n sources (in units of the split weights)
    auto weight = [&](int n) {
        FfAcc S = {};
        const ff_f2 x = sx[min(lane, P - 1)];
#pragma unroll 8
        for (int j = 0; j < n; j++) {
            float t, tl, p, pr;
            diff(su[warp][j], x, t, tl);
            ff_div(sf[warp][j], t, tl, p, pr);
            ff_addto(S, p, pr);
            if ((j & 7) == 7) { if (MODE == M_SEC) ff_close3(S); else ff_norm(S); }
        }
        if (MODE != M_SEC) return ((double)S.b + (double)S.bl) * wq[min(lane, P - 1)];
        ff_close3(S);
        ff_fold(S);
        return ((double)S.s + (double)S.sl) * wq[min(lane, P - 1)];
    };
    const int64_t nleaf = pl.leaf_base[pl.nprob];
    for (;;) {
        int64_t gl = 0;
        if (lane == 0) {
            gl = (int64_t)atomicAdd(&pl.upq[0], 1ull);
            if (gl >= nleaf && atomicAdd(&pl.upq[1], 1ull) == 4ull * gridDim.x - 1) {
                pl.upq[0] = 0;                 // every warp has run past the end: reset for the next launch
                pl.upq[1] = 0;
            }
        }
        gl = __shfl_sync(FULL, gl, 0);
        if (gl >= nleaf) break;
        const int64_t p = sdc_upper_index(pl.leaf_base, pl.nprob, gl);
        if (pl.fslot[p] < 0 || pl.ffbad[p]) continue;
        const int64_t b0 = a.off[p], g0 = pl.box_base[p];
        const int m = a.mk[p], nb0 = (m + B - 1) / B, L = lev_count(nb0);
        const int kw = (MODE == M_LOW) ? 0 : ff_exp(a.wsum[p]) - 1022;
        int l = 0, b = (int)(gl - pl.leaf_base[p]);
        for (;;) {
            const int64_t g = g0 + lev_base(nb0, l) + b;
            double s;                          // weight of node lane, times 2^-kw
            __syncwarp();
            if (l == 0 && MODE == M_LOW) {
                // D_n = T_n(b) - T_n(a) with b = a + delta, by the recurrence
                // D_{n+1} = 2 delta T_n(b) + 2 a D_n - D_{n-1} (no cancellation)
                double c, h, av = 0.0, dl = 0.0;
                box_ch(pl.blo[g], pl.bhi[g], c, h);
                const int j = b * B + lane;
                if (j < m - 1) {
                    const double ih = 1.0 / h;
                    av = (a.dk[b0 + j] - c) * ih;
                    dl = ((a.dorg[b0 + j] - a.dk[b0 + j]) + a.eta[b0 + j]) * ih;
                }
                const double bv = av + dl, a2 = 2.0 * av, d2 = 2.0 * dl, b2 = 2.0 * bv;
                double tb0 = 1.0, tb1 = bv, D0 = 0.0, D1 = dl;
                double *T = Tt[(MODE == M_LOW) ? warp : 0][(MODE == M_LOW) ? lane : 0];
                T[1] = D1;
                for (int n = 1; n < P - 1; n++) {
                    const double D2 = fma(d2, tb1, fma(a2, D1, -D0)), tb2 = fma(b2, tb1, -tb0);
                    T[n + 1] = D2;
                    D0 = D1; D1 = D2; tb0 = tb1; tb1 = tb2;
                }
                __syncwarp();
                double mom = 0.0;
                const int n = min(lane, P - 1);
                for (int k = 0; k < B && n > 0; k++) mom += Tt[(MODE == M_LOW) ? warp : 0][(MODE == M_LOW) ? k : 0][n];
                __syncwarp();
                Tt[(MODE == M_LOW) ? warp : 0][0][n] = mom;          // every lane has read its column
                __syncwarp();
                s = 0.0;
                for (int k = 1; k < P; k++) s = fma(Tx[n * P + k], Tt[(MODE == M_LOW) ? warp : 0][0][k], s);
                s *= 1.0 / P;
            } else if (l == 0) {
                double c, h;
                box_ch(pl.blo[g], pl.bhi[g], c, h);
                const int j = b * B + lane;
                ff_f2 u = {0.0f, 0.0f}, w = {0.0f, 0.0f};
                if (j < m) {
                    const double z = (MODE == M_SEC) ? a.zk[b0 + j] : a.vhat[b0 + j];
                    u = ff_weight((a.dk[b0 + j] - c) * rcp_nr2(h), 0);
                    w = ff_weight(z * z, kw);
                }
                su[warp][lane] = u;
                sf[warp][lane] = factor(u, w);
                __syncwarp();
                s = weight(min(B, m - b * B));
            } else {
                const int nbc = lev_nb(nb0, l - 1), nch = (2 * b + 1 < nbc) ? 2 : 1;
                const int64_t gc = g0 + lev_base(nb0, l - 1) + 2 * b;
                double cP, hP;
                box_ch(pl.blo[g], pl.bhi[g], cP, hP);
                const double ih = rcp_nr2(hP);
                for (int ci = 0; ci < nch; ci++) {
                    double cc, hc;
                    box_ch(pl.blo[gc + ci], pl.bhi[gc + ci], cc, hc);
                    const int q = min(lane, P - 1);
                    // the node as scale and shift (exact for boxes of one point)
                    const ff_f2 u = ff_weight(fma(hc * ih, xq[q], (cc - cP) * ih), 0);
                    const float2 w = __ldcg((const float2 *)&pl.nwt[(gc + ci) * P + q]);
                    const ff_f2 f = factor(u, {w.x, w.y});
                    if (lane < P) {
                        su[warp][ci * P + lane] = u;
                        sf[warp][ci * P + lane] = f;
                    }
                }
                __syncwarp();
                s = weight(nch * P);
            }
            if (lane < P) {
                pl.nwt[g * P + lane] = ff_weight(s, 0);
                if (MODE == M_SEC) pl.W[(g * P + lane) * pl.ncol] = s * ff_pow2(kw);       // k_secular_last
            }
            if (l + 1 >= L) break;
            const int bp = b >> 1, nsib = (2 * bp + 1 < lev_nb(nb0, l)) ? 2 : 1;
            const int64_t gp = g0 + lev_base(nb0, l + 1) + bp;
            __threadfence();
            __syncwarp();
            int last = 0;
            if (lane == 0) {
                last = atomicAdd(&pl.upcnt[gp], 1) == nsib - 1;
                if (last) pl.upcnt[gp] = 0;
            }
            if (!__shfl_sync(FULL, last, 0)) break;
            __threadfence();
            l++;
            b = bp;
        }
    }
}

// Kernels of the far fields (s source, t target).
enum { K_SEC = 0, K_1 = 1, K_2 = 2, K_1N = 3, K_LOG = 4 };

// ---------------------------------------------------------------------------
// Far fields of the one-column sums (secular sweeps, b, Loewner): the node
// weights of every box in the interaction lists of a leaf box and of its
// ancestors, summed at the leaf's own Chebyshev nodes, then the leaf's
// coefficients.  Against translating box by box (P^2 FP64 kernel entries per
// pair, then the fields down the tree level by level) this sums about 3.5 boxes
// per level instead of 7 per leaf in all, but by split FP32 terms (8 cycles of
// an SM per warp term against 112), reads no kernel matrices and needs no
// launch per level.  One warp per leaf box, a lane per node.
//   K_SEC: sum w/(s - t) to the left and right (psi, phi); their derivatives
//     are those of the series
//   K_2: sum w/(s - t)^2
//   K_LOG: sum w log|s - t| as its derivative sum w/(t - s) at the nodes,
//     integrated in coefficient space, plus the sum itself at the box centre
// Measured (GB300, 4096 problems of 32..2048 poles; translations, then down):
// secular 6.2 + 2.1 -> 1.4 ms, b 3.4 + 2.1 -> 1.5, Loewner 5.1 + 2.1 -> 1.5; the
// sweeps read one FP64 and three FP32 series instead of four FP64 ones, 10.1 ->
// 6.8 ms (tail pass 2.3 -> 1.4; with the mixed series below 5.2 and 0.9).  zhat's error
// falls from 5.4e-13 to 1.6e-13 (4000 poles).
// ---------------------------------------------------------------------------

// positions of every box's Chebyshev nodes as split parts
__global__ void k_fmm_nodes(FmmDev pl, const int64_t *__restrict__ off, const int32_t *__restrict__ mk,
                            const double *__restrict__ dk)
{
    __shared__ double xq[P];
    if (threadIdx.x < P) xq[threadIdx.x] = cospi((double)(2 * threadIdx.x + 1) / (2.0 * P));
    __syncthreads();
    const int64_t n = pl.box_base[pl.nprob] * P;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = t / P;
        const int64_t p = sdc_upper_index(pl.box_base, pl.nprob, g);
        if (pl.fslot[p] < 0) continue;
        const int64_t b0 = off[p];
        const FfScale s = ff_scale(dk[b0], dk[b0 + mk[p] - 1], 1.0);
        double c, h;
        box_ch(pl.blo[g], pl.bhi[g], c, h);
        pl.npos[t] = ff_point(c, h * xq[t % P], s);         // not rounded to the spacing of c
    }
}

constexpr int FAR_NW = 4;         // warps (leaf boxes) per CTA
constexpr int FAR_TAKE = 4;       // list entries taken per level and round

// Series of a leaf box in mixed precision: sum_{n < LOWN} a_n u^n (monomials, FP64)
// plus sum_{n >= LOWN} c_n T_n(u) (Chebyshev, single precision).  A box of the
// lists is at least 3/4 of the larger width away, so c_n falls as 4.8^-n
// (FMM_KAPPA): the single precision part is below 2^-27 of the sum and its rounding
// below 2^-51; the monomials' amplification, at most 2.4^n, is below that decay.  11 FP64
// instructions per evaluation instead of 43 (Clenshaw over all of them): 180
// instead of 690 cycles of the SM for a warp.
constexpr int LOWN = 12;

__device__ __forceinline__ double low_eval(const double *__restrict__ a, double u)
{
    double s = a[LOWN - 1];
#pragma unroll
    for (int n = LOWN - 2; n >= 0; n--) s = fma(s, u, a[n]);
    return s;
}

// single precision series; LO: its first LO coefficients are zero and not stored
template <int LO>
__device__ __forceinline__ float clenshawf(const float *__restrict__ a, float u)
{
    const float u2 = u + u;
    float b1 = 0.0f, b2 = 0.0f;
#pragma unroll
    for (int n = P - 1; n >= 1; n--) {
        const float b0 = fmaf(u2, b1, (n >= LO) ? a[n - LO] - b2 : -b2);
        b2 = b1;
        b1 = b0;
    }
    return fmaf(u, b1, (LO == 0) ? a[0] - b2 : -b2);
}

// M[n * LOWN + k]: coefficient of u^k in T_n
__device__ __forceinline__ void mono_table(double *M)
{
    if (threadIdx.x < LOWN) {
        const int k = threadIdx.x;
        int c0 = 0, c1 = 0;                       // coefficients of u^k in T_{n-1}, T_{n-2}
        for (int n = 0; n < LOWN; n++) {
            const int up = __shfl_up_sync((1u << LOWN) - 1u, c0, 1);
            const int c = (n == 0) ? (k == 0) : (n == 1) ? (k == 1) : 2 * (k ? up : 0) - c1;
            c1 = c0;
            c0 = c;
            M[n * LOWN + k] = (double)c;
        }
    }
}

// a leaf's series (coefficient lane in a) into the mixed form at cf, the single
// precision part times sc; one warp, t: LOWN entries of shared memory
__device__ __forceinline__ void store_series(double a, double sc, const double *M, double *t, double *__restrict__ cf)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    if (lane < LOWN) t[lane] = a;
    __syncwarp();
    if (lane < LOWN) {
        double s = 0.0;
        for (int n = 0; n < LOWN; n++) s = fma(M[n * LOWN + lane], t[n], s);
        cf[lane] = s;
    } else if (lane < P) {
        ((float *)(cf + LOWN))[lane - LOWN] = (float)(a * sc);
    }
}

// far field of a root in its leaf box gl (K_SEC's layouts): FP64 sums of a problem out of scale
__device__ __forceinline__ void far_eval(const FmmDev &pl, int64_t gl, double u, Acc &A)
{
    const double *cf = pl.coef + gl * NFIELD * P;
    A.psi += clenshaw(cf, u);
    A.phi += clenshaw(cf + P, u);
    A.dpsi += clenshaw(cf + 2 * P, u);
    A.dphi += clenshaw(cf + 3 * P, u);
}

// the same of a split sweep: single precision parts into S, the FP64 part returned
__device__ __forceinline__ double far_split(const FmmDev &pl, int64_t gl, double u, FfAcc &S)
{
    const double *cf = pl.coef + gl * NFIELD * P;
    const float *ff = (const float *)(cf + LOWN), *fd = (const float *)(cf + P);
    const float uf = ff_top(u, 0);
    ff_merge(S, clenshawf<LOWN>(ff, uf), 0.0f, clenshawf<0>(fd, uf), clenshawf<0>(fd + P, uf),
             clenshawf<0>(fd + 2 * P, uf));
    return low_eval(cf, u);
}

// ---------------------------------------------------------------------------
// Far fields of the problems out of the split arithmetic's scale, in FP64 (poles
// closer than its positions resolve): series of P coefficients per field and leaf
// box.  A CTA takes a subtree of 2^sub leaf boxes: its top box sums the interaction
// lists of itself and of every ancestor at its own nodes, the boxes below it their
// own lists, plus the parent's series at their nodes; the series of the current
// path stay in shared memory.  About 7 + 3.5 levels / 2^sub box pairs per leaf, as by
// translation level by level but in one launch (none for the one-column sums; summing every ancestor's list at
// the leaf: 3.5 per level).  Fields: K_SEC the sums w/(s-t) to the left and right,
// then w/(s-t)^2; K_2 w/(s-t)^2; K_LOG w log|s-t| as its derivative at the nodes,
// integrated in coefficient space, plus the sum itself at the box's centre; K_1 and
// K_1N nw columns w/(s-t), w/(t-s).
// Measured (GB300): step of 40000 poles, one pair of them close, 2.22 ms (2.96 with
// every list summed at the leaves, 2.57 by translations level by level, a launch per
// level); 64 columns through 20000 such poles, both directions, with k_cm_rest 6.2
// (17.0, 6.0); 124000 rows in 60 problems, 19 columns 6.6 (15.7, 7.0).
// ---------------------------------------------------------------------------
constexpr int SUB_MAX = 3;        // levels of a subtree below its top box
constexpr int F64_COLS = 32;      // widest block of columns

template <int KER> constexpr bool far_cols() { return KER == K_1 || KER == K_1N; }
template <int KER> constexpr int far_fields() { return KER == K_SEC ? 4 : far_cols<KER>() ? F64_COLS : 1; }

template <int KER> constexpr int far_threads() { return far_cols<KER>() ? 256 : 128; }

template <int KER>
__device__ __noinline__ void far64(const FmmDev &pl, const int32_t *__restrict__ mk, const int32_t *__restrict__ only,
                                   int nw, int sub, double *__restrict__ coef, int nfield, int32_t *word)
{
    constexpr bool COLS = far_cols<KER>();
    constexpr int NF = far_fields<KER>(), NT = far_threads<KER>(), PARTS = NT / P, PAIRS = COLS ? 1 : 32;
    constexpr int RMAX = (P * NF + NT - 1) / NT;
    __shared__ double xq[P], tq[P], Tx[P * P];
    __shared__ double stack[SUB_MAX + 1][NF][P];         // series of the path's boxes by level
    __shared__ double Fs[NF][P], An[P + 2], Bk[P + 1];
    __shared__ double sq[PAIRS][P], Ws[PAIRS * P][COLS ? NF : 1];
    __shared__ double K1[COLS ? P : 1][P + 1];
    __shared__ double red[COLS ? 1 : NF][COLS ? 1 : PARTS][P];
    __shared__ int s_list[32], s_nlist;
    __shared__ double s_ctr[4];
    __syncthreads();
    cheb_tables(xq, Tx);
    // columns f0 .. f0 + nf - 1 of the nw (blockIdx.y: halves)
    const int f0 = COLS ? (int)((int64_t)nw * blockIdx.y / gridDim.y) : 0;
    const int tid = threadIdx.x, nf = COLS ? (int)((int64_t)nw * (blockIdx.y + 1) / gridDim.y) - f0 : NF;
    const int64_t nleaf = pl.leaf_base[pl.nprob];
    for (int64_t t = blockIdx.x;; t += gridDim.x) {
        const int64_t w0 = t << sub;
        if (w0 >= nleaf) break;
        // the subtrees that start in this window of leaf boxes
        for (int64_t gl = w0; gl < min(nleaf, w0 + ((int64_t)1 << sub)); gl++) {
            const int64_t p = sdc_upper_index(pl.leaf_base, pl.nprob, gl);
            if (pl.fslot[p] < 0 || only[p] == 0) continue;
            const int Tb0 = (int)(gl - pl.leaf_base[p]);
            const int nb0 = (mk[p] + B - 1) / B, L = lev_count(nb0), top = min(sub, L - 1);
            if (Tb0 & ((1 << top) - 1)) continue;
            const int64_t g0 = pl.box_base[p];
            const bool coarse = pl.coarse[p] != 0;
            int npair = 0;
            for (int b = Tb0; b < min(nb0, Tb0 + (1 << top)); b++)
                for (int l = b == Tb0 ? top : __ffs(b) - 1; l >= 0; l--) {
                    const int64_t g = g0 + lev_base(nb0, l) + (b >> l);
                    const bool near_all = pl.nnear[g] < 0;               // every source directly: no far field
                    double cT, hT;
                    box_ch(pl.blo[g], pl.bhi[g], cT, hT);
                    __syncthreads();
                    if (tid < P) tq[tid] = cT + hT * xq[tid];
                    double acc[RMAX] = {};                               // COLS: entry (q, f)
                    double a1[2] = {}, a2[2] = {}, c1 = 0.0;             // else node q, by side; the centre's sum
                    const int q = tid % P, part = tid / P;
                    // the interaction lists: of this box, and of its ancestors for the subtree's top
                    for (int lv = l; lv < (near_all ? 0 : l == top ? L - 1 : l + 1); lv++) {
                        const int A = b >> lv, nbl = lev_nb(nb0, lv);
                        const int64_t gb = g0 + lev_base(nb0, lv), gP = g0 + lev_base(nb0, lv + 1) + (A >> 1);
                        const int npn = pl.nnear[gP];
                        const int64_t pst = pl.nstart[gP];
                        for (int c0 = 0; c0 < 2 * npn; c0 += 32) {
                            __syncthreads();
                            if (tid < 32) {
                                const int cd = c0 + tid;
                                int S = -1;
                                bool in = false;
                                if (cd < 2 * npn) {
                                    S = SDC_IDX(2 * pl.near[pst + (cd >> 1)] + (cd & 1), nbl + 1, word);
                                    in = S < nbl && S != A && adm_box(pl, gb + S, gb + A, coarse);
                                }
                                const unsigned bal = __ballot_sync(0xffffffffu, in);
                                if (in) s_list[__popc(bal & ((1u << tid) - 1u))] = S;
                                if (tid == 0) s_nlist = __popc(bal);
                            }
                            __syncthreads();
                            const int nlist = s_nlist;
                            npair += nlist;
                            for (int i0 = 0; i0 < nlist; i0 += PAIRS) {
                                const int cnt = min(PAIRS, nlist - i0);
                                if (i0 > 0) __syncthreads();
                                for (int e = tid; e < cnt * P; e += NT) {
                                    const int64_t gS = gb + s_list[i0 + e / P];
                                    double cS, hS;
                                    box_ch(pl.blo[gS], pl.bhi[gS], cS, hS);
                                    sq[e / P][e % P] = cS + hS * xq[e % P];
                                    if (!COLS) Ws[e][0] = pl.W[(gS * P + e % P) * pl.ncol];
                                }
                                if (COLS) {
                                    const double *Wg = pl.W + (gb + s_list[i0]) * P * pl.ncol + f0;
                                    for (int e = tid; e < P * nf; e += NT) Ws[e / nf][e % nf] = Wg[(e / nf) * pl.ncol + e % nf];
                                }
                                __syncthreads();
                                if (COLS) {
                                    for (int e = tid; e < P * P; e += NT) {
                                        const double d = sq[0][e % P] - tq[e / P];
                                        K1[e / P][e % P] = rcp_nr2(KER == K_1N ? -d : d);
                                    }
                                    __syncthreads();
#pragma unroll
                                    for (int r = 0; r < RMAX; r++) {
                                        const int e = tid + r * NT;
                                        if (e >= P * nf) break;
                                        const int eq = e / nf, ef = e % nf;
                                        double v = 0.0;
                                        for (int j = 0; j < P; j++) v = fma(K1[COLS ? eq : 0][j], Ws[j][COLS ? ef : 0], v);
                                        acc[r] += v;
                                    }
                                } else if (part < PARTS) {
                                    for (int i = 0; i < cnt; i++) {
                                        const bool left = KER != K_SEC || s_list[i0 + i] < A;
                                        double v1 = 0.0, v2 = 0.0;
                                        for (int j = part; j < P; j += PARTS) {
                                            const double r = rcp_nr2(sq[COLS ? 0 : i][j] - tq[q]);
                                            const double wr = Ws[i * P + j][0] * r;
                                            if (KER != K_2) v1 += wr;
                                            if (KER == K_SEC || KER == K_2) v2 = fma(wr, r, v2);
                                        }
                                        if (left) { a1[0] += v1; a2[0] += v2; } else { a1[1] += v1; a2[1] += v2; }
                                    }
                                }
                                if (KER == K_LOG)
                                    for (int e = tid; e < cnt * P; e += NT)
                                        c1 = fma(Ws[e][0], log(fabs(sq[COLS ? 0 : e / P][e % P] - cT)), c1);
                            }
                        }
                    }
                    // node values
                    if (COLS) {
#pragma unroll
                        for (int r = 0; r < RMAX; r++) {
                            const int e = tid + r * NT;
                            if (e < P * nf) Fs[e % nf][e / nf] = acc[r];
                        }
                    } else {
                        if (part < PARTS) {
                            const double v[4] = {KER == K_2 ? a2[0] : a1[0], a1[1], a2[0], a2[1]};
#pragma unroll
                            for (int k = 0; k < NF; k++) red[COLS ? 0 : k][COLS ? 0 : part][q] = v[k];
                        }
                        __syncthreads();
                        for (int e = tid; e < P * NF; e += NT) {
                            double v = 0.0;
                            for (int i = 0; i < PARTS; i++) v += red[COLS ? 0 : e / P][COLS ? 0 : i][e % P];
                            Fs[e / P][e % P] = v;
                        }
                    }
                    if (KER == K_LOG) {
                        // F' = -sum w/(s-t) -> antiderivative G = sum B_k T_k (k = 1..P; T_P vanishes at
                        // the nodes but not at 0), F(u) = F(centre) + h (G(u) - G(0))
                        for (int sh = 16; sh > 0; sh >>= 1) c1 += __shfl_xor_sync(0xffffffffu, c1, sh);
                        __syncthreads();
                        if (tid < P) {
                            double v = 0.0;
                            for (int j = 0; j < P; j++) v = fma(Fs[0][j], Tx[j * P + tid], v);
                            An[tid] = -v * (tid == 0 ? 1.0 / P : 2.0 / P);
                        }
                        if (tid == 0) An[P] = An[P + 1] = 0.0;
                        if ((tid & 31) == 0) s_ctr[tid >> 5] = c1;
                        __syncthreads();
                        if (tid >= 1 && tid <= P)
                            Bk[tid] = tid == 1 ? An[0] - 0.5 * An[2] : (An[tid - 1] - An[tid + 1]) * (0.5 / tid);
                        __syncthreads();
                        if (tid < P) {
                            double gq = 0.0, gz = 0.0;
                            for (int k = 1; k < P; k++) gq = fma(Bk[k], Tx[tid * P + k], gq);
                            for (int k = 2; k <= P; k += 2) gz += (k & 2) ? -Bk[k] : Bk[k];     // T_k(0)
                            Fs[0][tid] = near_all ? 0.0 : (s_ctr[0] + s_ctr[1]) + (s_ctr[2] + s_ctr[3]) + hT * (gq - gz);
                        }
                    }
                    __syncthreads();
                    // the parent's series at this box's nodes (the node as scale and shift: forming
                    // c + h x_q first would round it to the spacing of c, several percent of h on a
                    // box of one point)
                    if (l < top && !near_all) {
                        const int64_t gP = g0 + lev_base(nb0, l + 1) + (b >> (l + 1));
                        double cP, hP;
                        box_ch(pl.blo[gP], pl.bhi[gP], cP, hP);
                        const double ihP = rcp_any(hP);
                        for (int e = tid; e < P * nf; e += NT)
                            Fs[e / P][e % P] += clenshaw(stack[l + 1][e / P], fma(hT * ihP, xq[e % P], (cT - cP) * ihP));
                        __syncthreads();
                    }
                    for (int e = tid; e < P * nf; e += NT) {
                        double v = 0.0;
                        for (int j = 0; j < P; j++) v = fma(Fs[e / P][j], Tx[j * P + e % P], v);
                        v *= (e % P == 0) ? 1.0 / P : 2.0 / P;
                        stack[l][e / P][e % P] = v;
                        if (l == 0) coef[((pl.leaf_base[p] + b) * nfield + f0 + e / P) * P + e % P] = v;
                    }
                }
            // kernel entry and its products; the series per box of the subtree
            fl_add(pl, (int64_t)npair * P * P * (KER == K_SEC ? 7 : COLS ? 2 + 2 * nf : 5) +
                           (int64_t)(2 << top) * 4 * P * P * nf);
        }
    }
}

// the columns' kernel (the one-column sums': at the end of k_fmm_far)
template <int KER>
__global__ void __launch_bounds__(far_threads<KER>())
k_fmm_far64(FmmDev pl, const int32_t *__restrict__ mk, const int32_t *__restrict__ only, int nw, int sub,
            double *__restrict__ coef, int nfield, int32_t *word)
{
    if (only[pl.nprob] == 0) return;                     // no problem out of scale
    far64<KER>(pl, mk, only, nw, sub, coef, nfield, word);
}

template <int KER>
__global__ void __launch_bounds__(FAR_NW * 32, 5) k_fmm_far(FmmDev pl, const int64_t *__restrict__ off, R1Out o, int sub)
{
    __shared__ double Tx[P * P], xq[P], Mt[LOWN * LOWN];
    __shared__ float Tf[(KER == K_SEC) ? P * P : 1];
    __shared__ ff_logtab lt[(KER == K_LOG) ? 128 : 1];
    __shared__ ff_f4 sp[FAR_NW][P];
    __shared__ ff_f2 sw[FAR_NW][P];
    __shared__ int list[FAR_NW][32 * FAR_TAKE];
    __shared__ double sF[FAR_NW][P + 2];
    __shared__ float fL[FAR_NW][P], fR[FAR_NW][P];
    const unsigned FULL = 0xffffffffu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = min(lane, P - 1);
    cheb_tables(xq, Tx);
    mono_table(Mt);
    if (KER == K_LOG)
        for (int i = threadIdx.x; i < 128; i += blockDim.x) {
            const float c = ff_logc(i);
            const double v = -log((double)c);
            lt[i] = {c, (float)v, (float)(v - (double)(float)v)};
        }
    __syncthreads();
    if (KER == K_SEC)
        for (int i = threadIdx.x; i < P * P; i += blockDim.x) Tf[i] = (float)Tx[i];
    __syncthreads();
    const int64_t nleaf = pl.leaf_base[pl.nprob];
    for (int64_t gl = (int64_t)blockIdx.x * FAR_NW + warp; gl < nleaf; gl += (int64_t)gridDim.x * FAR_NW) {
        const int64_t p = sdc_upper_index(pl.leaf_base, pl.nprob, gl);
        if (pl.fslot[p] < 0 || pl.ffbad[p]) continue;        // out of scale: far64
        const int64_t b0 = off[p], g0 = pl.box_base[p];
        const int m = o.mk[p], nb0 = (m + B - 1) / B, L = lev_count(nb0);
        const int Tb = (int)(gl - pl.leaf_base[p]);
        const FfScale fs = ff_scale(o.dk[b0], o.dk[b0 + m - 1], o.wsum[p]);
        double cT, hT;
        box_ch(pl.blo[g0 + Tb], pl.bhi[g0 + Tb], cT, hT);
        const ff_f4 x = ff_point(cT, hT * xq[q], fs), xc = ff_pole(cT, fs);
        FfAcc AL = {}, AR = {}, AC = {};          // AC: K_LOG, the sum at the centre
        // lane l: the interaction list of the leaf's ancestor on level l
        int A = 0, npn = 0, sec = 0, lb = 0;
        int64_t pst = 0;
        unsigned long long mask = 0;
        if (lane < L - 1 && pl.nnear[g0 + Tb] >= 0) {
            A = Tb >> lane;
            lb = lev_base(nb0, lane);
            const int64_t gP = g0 + lev_base(nb0, lane + 1) + (A >> 1);
            npn = pl.nnear[gP];
            pst = pl.nstart[gP];
            mask = pl.amask[g0 + lb + A];
        }
        int npair = 0;
        while (__any_sync(FULL, mask != 0 || 64 * (sec + 1) < 2 * npn)) {
            if (mask == 0 && 64 * (sec + 1) < 2 * npn) {
                sec++;
                mask = adm_mask(pl, g0 + lb, lev_nb(nb0, lane), A, pst, npn, sec, false);     // coarse problems are out of scale
            }
            const int cnt = min(FAR_TAKE, __popcll(mask));
            int pos = cnt;
            for (int s = 1; s < 32; s <<= 1) {
                const int v = __shfl_up_sync(FULL, pos, s);
                if (lane >= s) pos += v;
            }
            const int total = __shfl_sync(FULL, pos, 31);
            pos -= cnt;
            __syncwarp();
            for (int i = 0; i < cnt; i++) {
                const int c = __ffsll((long long)mask) - 1;
                mask &= mask - 1;
                const int S = SDC_IDX(2 * pl.near[pst + ((64 * sec + c) >> 1)] + (c & 1), lev_nb(nb0, lane), o.status);
                list[warp][pos + i] = ((lb + S) << 1) | (S < A ? 1 : 0);
            }
            __syncwarp();
            npair += total;
            ff_f4 v = {};
            ff_f2 w = {};
            if (total > 0) {
                const int64_t t = (g0 + (list[warp][0] >> 1)) * P + q;
                v = pl.npos[t];
                w = pl.nwt[t];
            }
            for (int i = 0; i < total; i++) {
                const int e = list[warp][i];
                const bool left = e & 1;
                __syncwarp();
                if (lane < P) { sp[warp][lane] = v; sw[warp][lane] = w; }
                __syncwarp();
                const ff_f4 vq = v;
                const ff_f2 wq = w;
                if (i + 1 < total) {                         // the next pair's nodes, ahead of their use
                    const int64_t t = (g0 + (list[warp][i + 1] >> 1)) * P + q;
                    v = pl.npos[t];
                    w = pl.nwt[t];
                }
                FfAcc S = (KER == K_SEC && !left) ? AR : AL;
                // unrolled as a whole, with registers for five CTAs per SM: two nodes at a time wait
                // for their loads (zhat of 4096 problems 1.53 -> 1.41 ms, of the 90 steps of n = 131072
                // 10.6 -> 9.6)
#pragma unroll
                for (int j = 0; j < P; j++) {
                    float t, tp, tq2;
                    if (KER == K_2) ff_term2(sp[warp][j], sw[warp][j], x, t, tp);
                    else ff_term(sp[warp][j], sw[warp][j], x, t, tp, tq2);
                    ff_addto(S, t, tp);
                    if ((j & 7) == 7) ff_norm(S);
                }
                if (KER == K_SEC) ff_close3(S); else ff_close(S);
                if (KER == K_SEC && !left) AR = S; else AL = S;
                if (KER == K_LOG) {
                    // node q of the source against the centre; the box's weights sum
                    // to zero, so one exponent per box drops out
                    float t, tl2, y, yl;
                    ff_diff(vq, xc, t, tl2);
                    if (t < 0.0f) { t = -t; tl2 = -tl2; }
                    const int e0 = __shfl_sync(FULL, ff_fexp(t), 0);
                    ff_log(t, tl2, e0, lt, y, yl);
                    float pr, pe;
                    ff_two_mul(wq.x, y, pr, pe);
                    pe = ff_fma(wq.y, y, ff_fma(wq.x, yl, pe));
                    if (lane < P) ff_addto(AC, pr, pe);
                    ff_close(AC);
                }
            }
        }
        // the leaf's coefficients
        double *cf = pl.coef + gl * NFIELD * P;
        const double c1 = ff_pow2(fs.kk + fs.kw);
        const double fn = (lane == 0) ? 1.0 / P : 2.0 / P;
        auto series = [&](double F) {              // coefficient lane of the series with node values F
            __syncwarp();
            if (lane < P) sF[warp][lane] = F;
            __syncwarp();
            double a = 0.0;
            for (int j = 0; j < P; j++) a = fma(sF[warp][j], Tx[j * P + q], a);
            return a * fn;
        };
        if (KER == K_SEC) {
            // psi + phi in FP64; psi and the two derivatives in single precision,
            // scaled like the near sums (ff_collect)
            const double a = series(((double)AL.s + ((double)AL.sl + (double)AL.c) + ((double)AR.s + ((double)AR.sl + (double)AR.c))) * c1);
            if (lane < P) { fL[warp][lane] = AL.s; fR[warp][lane] = AR.s; }
            __syncwarp();
            float l = 0.0f, r = 0.0f;
            for (int j = 0; j < P; j++) {
                l = fmaf(fL[warp][j], Tf[j * P + q], l);
                r = fmaf(fR[warp][j], Tf[j * P + q], r);
            }
            l *= (float)fn;
            r *= (float)fn;
            __syncwarp();
            if (lane < P) { fL[warp][lane] = l; fR[warp][lane] = r; }
            __syncwarp();
            const float ih = (float)(1.0 / (hT * ff_pow2(fs.kk)));
            float dl = 0.0f, dr = 0.0f;
            for (int n = q + 1; n < P; n += 2) {
                dl = fmaf((float)(2 * n), fL[warp][n], dl);
                dr = fmaf((float)(2 * n), fR[warp][n], dr);
            }
            if (q == 0) { dl *= 0.5f; dr *= 0.5f; }
            if (lane < P) {
                float *ff = (float *)(cf + P);
                ff[lane] = l;
                ff[P + lane] = dl * ih;
                ff[2 * P + lane] = dr * ih;
            }
            store_series(a, ff_pow2(-(fs.kk + fs.kw)), Mt, sF[warp], cf);
        } else if (KER == K_2) {
            store_series(series((double)AL.s + (double)AL.sl), 1.0, Mt, sF[warp], cf);
        } else {
            // F' -> antiderivative G = sum B_k T_k (k = 1..P; T_P vanishes at the
            // nodes but not at 0), F(u) = F(centre) + h (G(u) - G(0))
            const double a = series(-((double)AL.s + (double)AL.sl) * ff_pow2(fs.kk));
            double c = (double)AC.s + (double)AC.sl;
            if (lane >= P) c = 0.0;
            for (int s = 16; s > 0; s >>= 1) c += __shfl_xor_sync(FULL, c, s);
            __syncwarp();
            if (lane < P + 2) sF[warp][lane] = (lane < P) ? a : 0.0;
            __syncwarp();
            double bk = 0.0;                       // lane k holds B_k
            if (lane == 1) bk = sF[warp][0] - 0.5 * sF[warp][2];
            else if (lane >= 2 && lane <= P) bk = (sF[warp][lane - 1] - sF[warp][lane + 1]) * (0.5 / lane);
            double g0s = (lane >= 2 && lane <= P && !(lane & 1)) ? ((lane & 2) ? -bk : bk) : 0.0;   // T_k(0)
            for (int s = 16; s > 0; s >>= 1) g0s += __shfl_xor_sync(FULL, g0s, s);
            const double a2 = (lane == 0) ? c - hT * g0s : hT * bk;
            store_series(a2, 1.0, Mt, sF[warp], cf);
        }
        if (pl.flops && lane == 0 && npair)
            atomicAdd(pl.flops, (unsigned long long)npair * P * (P * (KER == K_SEC ? 7 : 5) + (KER == K_LOG ? 3 : 0)) +
                                    2 * P * P);
    }
    if (pl.ffbad[pl.nprob]) far64<KER>(pl, o.mk, pl.ffbad, 1, sub, pl.coef, NFIELD, o.status);
}

// Split parts of the kept poles and weights of the FMM problems (split.cuh);
// pl.ffbad says which problems' scale, gaps or stopping test do not allow them
struct FfDev {
    const ff_f4 *d;
    const ff_f2 *w;
};

__global__ void k_ff_prep(int64_t nprob, const int64_t *__restrict__ off, int64_t total,
                          const int32_t *__restrict__ fslot, R1Out o, double stop_c, ff_f4 *__restrict__ fd,
                          ff_f2 *__restrict__ fw, int32_t *__restrict__ bad)
{
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total;
         x += (int64_t)gridDim.x * blockDim.x) {
        if (x < off[0] || x >= off[nprob]) continue;
        const int64_t p = sdc_upper_index(off, nprob, x);
        if (fslot[p] < 0) continue;
        const int64_t b0 = off[p];
        const int m = o.mk[p], j = (int)(x - b0);
        if (j >= m) continue;
        const FfScale s = ff_scale(o.dk[b0], o.dk[b0 + m - 1], o.wsum[p]);
        if (!s.ok || o.unshifted || stop_c < SPLIT_STOP || (j + 1 < m && !ff_gap_ok(o.dk[x], o.dk[x + 1], s.kk))) {
            bad[p] = 1;
            bad[nprob] = 1;
            continue;
        }
        const double z = o.zk[x];
        fd[x] = ff_pole(o.dk[x], s);
        fw[x] = ff_weight(z * z, s.kw);
    }
}

// ---------------------------------------------------------------------------
// Secular roots of the FMM problems, one warp per leaf box (its 32 roots share
// the near list).  The near boxes' poles and weights (fixed
// during the iteration) are staged in shared memory once per box; each sweep
// sums them with shifted differences and evaluates the four far-field
// expansions at x = d_K + y.  Once no root is left to hand out and fewer than
// TAIL_X lanes are busy, the box's stragglers go to k_secular_tail.  The last
// root of each problem (outside the tree) is solved by k_secular_last.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(64)
k_secular_fmm(FmmDev pl, FfDev ff, const int64_t *__restrict__ off, R1Out o, double stop_c, int max_iter,
              unsigned long long *terms)
{
    __shared__ __align__(16) unsigned char stage[2][SPLIT_NEAR * B * (sizeof(ff_f4) + sizeof(ff_f2))];
    const unsigned FULL = 0xffffffffu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    ff_f4 *const fd = (ff_f4 *)stage[warp];              // near poles: split parts, or FP64 (the general form)
    ff_f2 *const fw = (ff_f2 *)(fd + SPLIT_NEAR * B);
    double *const sd = (double *)stage[warp], *const sw = sd + SPLIT_NEAR * B;
    const int64_t nleaf = pl.leaf_base[pl.nprob];
    for (int64_t gl = (int64_t)blockIdx.x * 2 + warp; gl < nleaf; gl += (int64_t)gridDim.x * 2) {
        const int64_t p = sdc_upper_index(pl.leaf_base, pl.nprob, gl);
        if (pl.fslot[p] < 0) continue;
        const int64_t b0 = off[p];
        const int m = o.mk[p];
        const int Tb = (int)(gl - pl.leaf_base[p]);
        const int k0 = Tb * B;
        const int kend = min(k0 + B, m - 1);
        if (k0 >= kend) continue;
        const double *dk = o.dk + b0, *zk = o.zk + b0;
        const double W = o.wsum[p];
        const double tol = stop_c * (double)m * SDC_EPS;
        const int64_t g = pl.box_base[p] + Tb;
        double cT, hT;
        box_ch(pl.blo[g], pl.bhi[g], cT, hT);
        const double ihT = 1.0 / hT;
        const int nnr = pl.nnear[g];
        const int nn = near_len(nnr, (m + B - 1) / B);
        if (nnr < 0 || nnr >= SPLIT_NEAR) continue;     // long near list: k_secular_fmm_split
        const bool ok = pl.ffbad[p] == 0;
        const FfScale fs = ff_scale(dk[0], dk[m - 1], W);
        int near_terms = 0;
        __syncwarp();
        for (int i = 0; i < nn; i++) {
            const int j0 = near_box_chk(pl, g, nnr, i, (m + B - 1) / B, o.status) * B;
            const int cnt = min(B, m - j0);
            near_terms += cnt;
            for (int jj = lane; jj < cnt; jj += 32) {
                if (ok) {
                    fd[i * B + jj] = ff.d[b0 + j0 + jj];
                    fw[i * B + jj] = ff.w[b0 + j0 + jj];
                } else {
                    sd[i * B + jj] = dk[j0 + jj];
                    const double z = zk[j0 + jj];
                    sw[i * B + jj] = z * z;
                }
            }
        }
        __syncwarp();
        int k = k0 + lane;
        bool act = k < kend;
        int next = k0 + 32;
        Root R;
        R.dK = 0.0; R.y = 1.0; R.phase = 1;
        if (act) R.init(dk, zk, k, m, W, o.unshifted != 0);
        double uK = (R.dK - cT) * ihT;                  // the root's origin in the leaf's coordinate
        while (__any_sync(FULL, act)) {
            const int kwlo = __reduce_min_sync(FULL, act ? k : 0x7fffffff);
            const int kwhi = __reduce_max_sync(FULL, act ? k : -1);
            const int kk = act ? k : kwlo;
            const bool p0 = __all_sync(FULL, !act || R.phase == 0);
            const unsigned amask = __ballot_sync(FULL, act);
            if (terms && lane == 0) atomicAdd(terms, (unsigned long long)__popc(amask) * (unsigned long long)near_terms);
            Acc A = {0.0, 0.0, 0.0, 0.0};
            FfAcc S = {};
            const ff_f4 x = ff_point(R.dK, R.y, fs);
            for (int i = 0; i < nn; i++) {
                const int j0 = near_box_chk(pl, g, nnr, i, (m + B - 1) / B, o.status) * B;
                const int cnt = min(B, m - j0);
                if (ok)      ff_sweep<false>(fd + i * B, fw + i * B, 0, cnt, j0, kk, kwlo, kwhi, x, S);
                else if (p0) sweep<false>(sd + i * B, sw + i * B, 0, cnt, j0, kk, kwlo, kwhi, R.dK, R.y, A);
                else         sweep<true>(sd + i * B, sw + i * B, 0, cnt, j0, kk, kwlo, kwhi, R.dK, R.y, A);
            }
            // far field at x = d_K + y, then the step
            bool fin = false;
            const bool moved = R.phase == 0;
            if (act) {
                if (ok) {
                    const double low = far_split(pl, gl, fma(R.y, ihT, uK), S);
                    fin = R.update_split(S, low, fs.kk, fs.kw, tol, max_iter, o.status);
                } else {
                    far_eval(pl, gl, ((R.dK + R.y) - cT) * ihT, A);
                    fin = R.update(A, tol, max_iter, o.status);
                }
            }
            if (fin) {
                o.org[b0 + k] = R.K;
                o.eta[b0 + k] = R.y;
                o.dorg[b0 + k] = R.dK;
                o.lamk[b0 + k] = R.dK + R.y;
                if (o.sweeps) o.sweeps[b0 + k] = R.nsw;
            }
            const unsigned mask = __ballot_sync(FULL, fin);
            if (fin) {
                k = next + __popc(mask & ((1u << lane) - 1u));
                act = k < kend;
                if (act) R.init(dk, zk, k, m, W, o.unshifted != 0);
            }
            if (__any_sync(FULL, moved || fin)) uK = (R.dK - cT) * ihT;
            next += __popc(mask);
            // no root left to refill and fewer than TAIL_X lanes busy: the
            // stragglers go to k_secular_tail, which runs 32 of them per warp
            if (next >= kend) {
                const unsigned am = __ballot_sync(FULL, act);
                const int nact = __popc(am);
                if (nact > 0 && nact < TAIL_X) {
                    unsigned base = 0;
                    if (lane == 0) base = atomicAdd(pl.ntail, (unsigned)nact);
                    base = __shfl_sync(FULL, base, 0);
                    if (act) {
                        FmmTail tr;
                        tr.p = p; tr.k = k; tr.K = R.K; tr.phase = R.phase; tr.nsw = R.nsw;
                        tr.dK = R.dK; tr.y = R.y; tr.lo = R.lo; tr.hi = R.hi;
                        pl.tail[base + __popc(am & ((1u << lane) - 1u))] = tr;
                    }
                    break;
                }
            }
        }
    }
}

// The stragglers of k_secular_fmm: four lanes per root, each summing every
// fourth pole of each near box of the root's box (poles read through L1),
// combined by a fixed butterfly; the root's far field and update are computed
// by all four lanes alike.  The warps are persistent: a lane group whose root
// has converged claims the next straggler (ntail[1]), so lanes do not wait for
// the slowest root of a fixed batch.  A root's arithmetic does not depend on
// which group runs it.
constexpr int TAIL_LANES = 4;

__global__ void __launch_bounds__(128)
k_secular_tail(FmmDev pl, FfDev ff, const int64_t *__restrict__ off, R1Out o, double stop_c, int max_iter,
               unsigned long long *terms)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, part = lane & (TAIL_LANES - 1), lead = lane & ~(TAIL_LANES - 1);
    const unsigned n = pl.ntail[0];
    unsigned *claim = pl.ntail + 1;
    bool act = false, dry = false;
    Root R;
    R.dK = 0.0; R.y = 1.0; R.phase = 1; R.k = 0;
    int64_t b0 = 0, g = 0, gl = 0;
    int m = 1, nnr = 0, nn = 0;
    bool ok = false;
    FfScale fs = {};
    unsigned nterm = 0;
    double cT = 0.0, ihT = 1.0, tol = 0.0;
    while (true) {
        // groups without a root claim the next one (warp-wide shuffle of the claim)
        const bool need = !act && !dry;
        unsigned idx = 0;
        if (need && part == 0) idx = atomicAdd(claim, 1u);
        idx = __shfl_sync(FULL, idx, lead);
        if (need) {
            if (idx < n) {
                const FmmTail tr = pl.tail[idx];
                const int64_t p = tr.p;
                b0 = off[p];
                m = o.mk[p];
                R.init(o.dk + b0, o.zk + b0, tr.k, m, o.wsum[p], o.unshifted != 0);
                R.K = tr.K; R.phase = tr.phase; R.nsw = tr.nsw;
                R.dK = tr.dK; R.y = tr.y; R.lo = tr.lo; R.hi = tr.hi;
                const int Tb = tr.k / B;
                g = pl.box_base[p] + Tb;
                gl = pl.leaf_base[p] + Tb;
                nnr = pl.nnear[g];
                nn = near_len(nnr, (m + B - 1) / B);
                nterm = 0;
                if (part == 0)
                    for (int i = 0; i < nn; i++) nterm += min(B, m - near_box(pl, g, nnr, i) * B);
                double hT;
                box_ch(pl.blo[g], pl.bhi[g], cT, hT);
                ihT = 1.0 / hT;
                tol = stop_c * (double)m * SDC_EPS;
                ok = pl.ffbad[p] == 0;
                fs = ff_scale(o.dk[b0], o.dk[b0 + m - 1], o.wsum[p]);
                act = true;
            } else {
                dry = true;
            }
        }
        if (!__any_sync(FULL, act)) break;
        if (terms) {
            const unsigned nt = __reduce_add_sync(FULL, act ? nterm : 0u);
            if (lane == 0) atomicAdd(terms, (unsigned long long)nt);
        }
        Acc A = {0.0, 0.0, 0.0, 0.0};
        FfAcc S = {};
        if (act && ok) {
            const ff_f4 x = ff_point(R.dK, R.y, fs);
            for (int i = 0; i < nn; i++) {
                const int j0 = near_box_chk(pl, g, nnr, i, (m + B - 1) / B, o.status) * B;
                const int cnt = min(B, m - j0);
                const ff_f4 *dd = ff.d + b0 + j0;
                const ff_f2 *ww = ff.w + b0 + j0;
#pragma unroll 4
                for (int jj = part; jj < cnt; jj += TAIL_LANES) {
                    float pp, ppl, qq;
                    ff_term(dd[jj], ww[jj], x, pp, ppl, qq);
                    ff_select(S, pp, ppl, qq, j0 + jj, R.k);
                }
                ff_close(S);
            }
        } else if (act) {
            for (int i = 0; i < nn; i++) {
                const int j0 = near_box_chk(pl, g, nnr, i, (m + B - 1) / B, o.status) * B;
                const int cnt = min(B, m - j0);
                const double *dd = o.dk + b0 + j0, *zz = o.zk + b0 + j0;
                for (int jj = part; jj < cnt; jj += TAIL_LANES) {
                    const double r = rcp_nr1(shifted_t(dd[jj], R.dK, R.y));
                    const double z = zz[jj];
                    const double a = (z * z) * r;
                    if (j0 + jj <= R.k) { A.psi += a; A.dpsi = fma(a, r, A.dpsi); }
                    else                { A.phi += a; A.dphi = fma(a, r, A.dphi); }
                }
            }
        }
        // the four lanes of a root are consecutive: butterfly over lane bits 0, 1
        for (int sh = 1; sh < TAIL_LANES; sh <<= 1) {
            const float v0 = __shfl_xor_sync(FULL, S.s, sh), v1 = __shfl_xor_sync(FULL, S.sl, sh);
            const float v2 = __shfl_xor_sync(FULL, S.psi, sh), v3 = __shfl_xor_sync(FULL, S.dpsi, sh);
            ff_merge(S, v0, v1, v2, v3, __shfl_xor_sync(FULL, S.dphi, sh));
        }
        if (__any_sync(FULL, act && !ok))
            for (int sh = 1; sh < TAIL_LANES; sh <<= 1) {
                A.psi += __shfl_xor_sync(FULL, A.psi, sh);
                A.phi += __shfl_xor_sync(FULL, A.phi, sh);
                A.dpsi += __shfl_xor_sync(FULL, A.dpsi, sh);
                A.dphi += __shfl_xor_sync(FULL, A.dphi, sh);
            }
        if (act) {
            bool fin;
            if (ok) {
                const double low = far_split(pl, gl, ((R.dK + R.y) - cT) * ihT, S);
                fin = R.update_split(S, low, fs.kk, fs.kw, tol, max_iter, o.status);
            } else {
                far_eval(pl, gl, ((R.dK + R.y) - cT) * ihT, A);
                fin = R.update(A, tol, max_iter, o.status);
            }
            if (fin) {
                if (part == 0) {
                    const int k = R.k;
                    o.org[b0 + k] = R.K;
                    o.eta[b0 + k] = R.y;
                    o.dorg[b0 + k] = R.dK;
                    o.lamk[b0 + k] = R.dK + R.y;
                    if (o.sweeps) o.sweeps[b0 + k] = R.nsw;
                }
                act = false;
            }
        }
    }
}

// Leaf boxes with long near lists (SPLIT_NEAR boxes or more, or "all near"),
// one CTA of SPW warps per box: the warps hold the same 32 roots (replicated
// state), split the near boxes between them and reduce the partial sums
// through shared memory in a fixed order after every sweep; the box's roots
// run in groups of 32.
template <int SPW>
__global__ void __launch_bounds__(SPW * 32)
k_secular_fmm_split(FmmDev pl, FfDev ff, const int64_t *__restrict__ off, R1Out o, double stop_c, int max_iter,
                    unsigned long long *terms)
{
    __shared__ __align__(16) unsigned char stage[SPW][B * (sizeof(ff_f4) + sizeof(ff_f2))];
    __shared__ double red[SPW][4][32];
    __shared__ float fred[SPW][5][32];
    const unsigned FULL = 0xffffffffu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    ff_f4 *const fd = (ff_f4 *)stage[warp];
    ff_f2 *const fw = (ff_f2 *)(fd + B);
    double *const sd = (double *)stage[warp], *const sw = sd + B;
    const int nsplit = *pl.nsplit;
    for (int u = blockIdx.x; u < nsplit; u += gridDim.x) {
        const int64_t gl = pl.split[u];                  // a leaf box with a long near list
        const int64_t p = sdc_upper_index(pl.leaf_base, pl.nprob, gl);
        if (pl.fslot[p] < 0) continue;
        const int64_t b0 = off[p];
        const int m = o.mk[p];
        const int Tb = (int)(gl - pl.leaf_base[p]);
        const int64_t g = pl.box_base[p] + Tb;
        const int nnr = pl.nnear[g];
        const int nn = near_len(nnr, (m + B - 1) / B);
        const int k0b = Tb * B;
        const int kendb = min(k0b + B, m - 1);
        const double *dk = o.dk + b0, *zk = o.zk + b0;
        const double W = o.wsum[p];
        const double tol = stop_c * (double)m * SDC_EPS;
        double cT, hT;
        box_ch(pl.blo[g], pl.bhi[g], cT, hT);
        const double ihT = 1.0 / hT;
        const bool ok = pl.ffbad[p] == 0;
        const FfScale fs = ff_scale(dk[0], dk[m - 1], W);
        int near_terms = 0;
        if (terms)
            for (int i = 0; i < nn; i++) near_terms += min(B, m - near_box(pl, g, nnr, i) * B);
        for (int k0 = k0b; k0 < kendb; k0 += 32) {
            const int k = k0 + lane;
            bool act = k < kendb;
            Root R;
            R.dK = 0.0; R.y = 1.0; R.phase = 1;
            if (act) R.init(dk, zk, k, m, W, o.unshifted != 0);
            while (__syncthreads_or(act)) {
                const int kwlo = __reduce_min_sync(FULL, act ? k : 0x7fffffff);
                const int kwhi = __reduce_max_sync(FULL, act ? k : -1);
                const int kk = act ? k : kwlo;
                const bool p0 = __all_sync(FULL, !act || R.phase == 0);
                const unsigned amask = __ballot_sync(FULL, act);
                if (terms && warp == 0 && lane == 0)
                    atomicAdd(terms, (unsigned long long)__popc(amask) * (unsigned long long)near_terms);
                Acc A = {0.0, 0.0, 0.0, 0.0};
                FfAcc fa = {};
                const ff_f4 x = ff_point(R.dK, R.y, fs);
                for (int i = warp; i < nn; i += SPW) {
                    const int S = near_box_chk(pl, g, nnr, i, (m + B - 1) / B, o.status);
                    const int j0 = S * B;
                    const int cnt = min(B, m - j0);
                    __syncwarp();
                    for (int jj = lane; jj < cnt; jj += 32) {
                        if (ok) {
                            fd[jj] = ff.d[b0 + j0 + jj];
                            fw[jj] = ff.w[b0 + j0 + jj];
                        } else {
                            sd[jj] = dk[j0 + jj];
                            const double z = zk[j0 + jj];
                            sw[jj] = z * z;
                        }
                    }
                    __syncwarp();
                    if (ok)      ff_sweep(fd, fw, 0, cnt, j0, kk, kwlo, kwhi, x, fa);
                    else if (p0) sweep<false>(sd, sw, 0, cnt, j0, kk, kwlo, kwhi, R.dK, R.y, A);
                    else         sweep<true>(sd, sw, 0, cnt, j0, kk, kwlo, kwhi, R.dK, R.y, A);
                }
                const double u = ((R.dK + R.y) - cT) * ihT;
                if (!ok && warp == 0 && act) far_eval(pl, gl, u, A);
                if (ok) {
                    fred[warp][0][lane] = fa.s;
                    fred[warp][1][lane] = fa.sl;
                    fred[warp][2][lane] = fa.psi;
                    fred[warp][3][lane] = fa.dpsi;
                    fred[warp][4][lane] = fa.dphi;
                } else {
                    red[warp][0][lane] = A.psi;
                    red[warp][1][lane] = A.phi;
                    red[warp][2][lane] = A.dpsi;
                    red[warp][3][lane] = A.dphi;
                }
                __syncthreads();
                // same order in every warp
                Acc T = {0.0, 0.0, 0.0, 0.0};
                FfAcc S = {};
#pragma unroll
                for (int w = 0; w < SPW; w++) {
                    if (ok) {
                        ff_merge(S, fred[w][0][lane], fred[w][1][lane], fred[w][2][lane], fred[w][3][lane],
                                 fred[w][4][lane]);
                    } else {
                        T.psi += red[w][0][lane];
                        T.phi += red[w][1][lane];
                        T.dpsi += red[w][2][lane];
                        T.dphi += red[w][3][lane];
                    }
                }
                __syncthreads();
                int32_t *const sts = warp == 0 ? o.status : nullptr;
                bool fin = false;
                if (act && ok) {
                    const double low = far_split(pl, gl, u, S);
                    fin = R.update_split(S, low, fs.kk, fs.kw, tol, max_iter, sts);
                } else if (act) {
                    fin = R.update(T, tol, max_iter, sts);
                }
                if (fin) {
                    if (warp == 0) {
                        o.org[b0 + k] = R.K;
                        o.eta[b0 + k] = R.y;
                        o.dorg[b0 + k] = R.dK;
                        o.lamk[b0 + k] = R.dK + R.y;
                        if (o.sweeps) o.sweeps[b0 + k] = R.nsw;
                    }
                    act = false;
                }
            }
        }
    }
}

// The last root of every FMM problem (in (d_{m-1}, d_{m-1} + sum w]), one CTA
// per problem: boxes at least their own width to the left of the bracket are
// summed through their Chebyshev node weights at the plain position (far
// field), the leaf boxes next to the bracket directly with shifted
// differences; if the lists overflow, every pole directly.  Thread 0 holds
// the root state, the partial sums are reduced in a fixed order.
constexpr int SL_T = 256;

constexpr int LAST_FAR = 112;     // boxes summed through their node weights for the last root
constexpr int LAST_NEAR = 32;     // leaf boxes summed directly for it

__global__ void __launch_bounds__(SL_T)
k_secular_last(FmmDev pl, const int64_t *__restrict__ off, R1Out o, double stop_c, int max_iter,
               unsigned long long *terms)
{
    __shared__ double red[2][SL_T / 32];
    __shared__ double s_dK, s_y;
    __shared__ int s_done, s_p0;
    __shared__ double xq[P];
    __shared__ double fs[LAST_FAR * P], fw[LAST_FAR * P];      // far boxes: node positions, weights
    __shared__ int64_t s_far[LAST_FAR];
    __shared__ int s_near[LAST_NEAR], s_nfar, s_nnear, s_ok;
    const unsigned FULL = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int q = tid; q < P; q += SL_T) xq[q] = cospi((double)(2 * q + 1) / (2.0 * P));
    const int nf = *pl.nfmm;
    for (int f = blockIdx.x; f < nf; f += gridDim.x) {
        const int64_t p = pl.fprob[f];
        if (pl.fslot[p] < 0) continue;
        const int64_t b0 = off[p];
        const int m = o.mk[p];
        const double *dk = o.dk + b0, *zk = o.zk + b0;
        const double tol = stop_c * (double)m * SDC_EPS;
        Root R;
        __syncthreads();
        if (tid == 0) {
            R.init(dk, zk, m - 1, m, o.wsum[p], o.unshifted != 0);
            s_dK = R.dK; s_y = R.y; s_done = 0; s_p0 = 1;
            // every pole lies to the left of the root's bracket [d_{m-1}, d_{m-1} + W]:
            // a box at least its own width away from the bracket is summed
            // through its node weights (multipole to point), the leaf boxes
            // next to it directly; walk the tree from the top
            const int nb0 = (m + B - 1) / B;
            const int L = lev_count(nb0);
            const double tlo = dk[m - 1];
            int nfar = 0, nnear = 0, ok = 1;
            int cand[2 * LAST_NEAR], nc = 1, ncand[2 * LAST_NEAR];
            cand[0] = 0;
            for (int l = L - 1; l >= 0 && ok; l--) {
                const int64_t gb = pl.box_base[p] + lev_base(nb0, l);
                int nn2 = 0;
                for (int i = 0; i < nc && ok; i++) {
                    const int bx = cand[i];
                    const double lo = pl.blo[gb + bx], hi = pl.bhi[gb + bx];
                    if (tlo - hi >= FMM_KAPPA * (hi - lo) && hi > lo) {
                        if (nfar < LAST_FAR) s_far[nfar++] = gb + bx; else ok = 0;
                    } else if (l == 0) {
                        if (nnear < LAST_NEAR) s_near[nnear++] = bx; else ok = 0;
                    } else {
                        const int nbc = lev_nb(nb0, l - 1);
                        for (int c = 2 * bx; c <= 2 * bx + 1 && c < nbc; c++) {
                            if (nn2 < 2 * LAST_NEAR) ncand[nn2++] = c; else ok = 0;
                        }
                    }
                }
                for (int i = 0; i < nn2; i++) cand[i] = ncand[i];
                nc = nn2;
            }
            s_nfar = nfar; s_nnear = nnear; s_ok = ok;
        }
        __syncthreads();
        const bool tree = s_ok != 0;
        const int nfar = s_nfar, nnear = s_nnear;
        int64_t nterms = m;
        if (tree) {
            for (int t = tid; t < nfar * P; t += SL_T) {
                const int64_t g = s_far[t / P];
                const int q = t % P;
                double c, h;
                box_ch(pl.blo[g], pl.bhi[g], c, h);
                fs[t] = c + h * xq[q];
                fw[t] = pl.W[(g * P + q) * pl.ncol];
            }
            nterms = (int64_t)nfar * P;
            for (int i = 0; i < nnear; i++) nterms += min(B, m - s_near[i] * B);
            __syncthreads();
        }
        while (!s_done) {
            const double dK = s_dK, y = s_y;
            const bool p0 = s_p0 != 0;
            double ps = 0.0, dps = 0.0;
            if (tree) {
                // far boxes at the plain position x = d_K + y (local shifting)
                const double x = dK + y;
                for (int t = tid; t < nfar * P; t += SL_T) {
                    const double r = rcp_nr1(fs[t] - x);
                    const double a = fw[t] * r;
                    ps += a;
                    if (!p0) dps = fma(a, r, dps);
                }
                for (int i = 0; i < nnear; i++) {
                    const int j0 = s_near[i] * B, cnt = min(B, m - j0);
                    for (int jj = tid; jj < cnt; jj += SL_T) {
                        const double r = rcp_nr1(shifted_t(dk[j0 + jj], dK, y));
                        const double z = zk[j0 + jj];
                        const double a = (z * z) * r;
                        ps += a;
                        if (!p0) dps = fma(a, r, dps);
                    }
                }
            } else {
                for (int j = tid; j < m; j += SL_T) {
                    const double r = rcp_nr1(shifted_t(dk[j], dK, y));
                    const double z = zk[j];
                    const double a = (z * z) * r;
                    ps += a;
                    if (!p0) dps = fma(a, r, dps);
                }
            }
            for (int sh = 16; sh > 0; sh >>= 1) {
                ps += __shfl_down_sync(FULL, ps, sh);
                dps += __shfl_down_sync(FULL, dps, sh);
            }
            if (lane == 0) { red[0][warp] = ps; red[1][warp] = dps; }
            __syncthreads();
            if (tid == 0) {
                Acc A = {0.0, 0.0, 0.0, 0.0};
                for (int w = 0; w < SL_T / 32; w++) { A.psi += red[0][w]; A.dpsi += red[1][w]; }
                const bool fin = R.update(A, tol, max_iter, o.status);
                if (terms) atomicAdd(terms, (unsigned long long)nterms);
                s_dK = R.dK; s_y = R.y; s_p0 = (R.phase == 0); s_done = fin;
                if (fin) {
                    const int k = m - 1;
                    o.org[b0 + k] = R.K;
                    o.eta[b0 + k] = R.y;
                    o.dorg[b0 + k] = R.dK;
                    o.lamk[b0 + k] = R.dK + R.y;
                    if (o.sweeps) o.sweeps[b0 + k] = R.nsw;
                }
            }
            __syncthreads();
        }
    }
}

// running product with exponent renormalisation every 8 factors
struct Prod {
    double pn = 1.0, pd = 1.0;
    int ex = 0, cnt = 0;
    __device__ __forceinline__ void mul(double num, double den)
    {
        pn *= num;
        pd *= den;
        if ((++cnt & 7) == 0) {
            const int hn = __double2hiint(pn), hd = __double2hiint(pd);
            const int en = (hn >> 20) & 0x7FF, ed = (hd >> 20) & 0x7FF;
            if (en != 0 && ed != 0 && en != 0x7FF && ed != 0x7FF) {
                ex += en - ed;
                pn = __hiloint2double((hn & 0x800FFFFF) | (1022 << 20), __double2loint(pn));
                pd = __hiloint2double((hd & 0x800FFFFF) | (1022 << 20), __double2loint(pd));
            }
        }
    }
};

// zhat of the FMM problems, eq. (4.23) as
//   vhat_i^2 = (lambda_i - d_i) prod_{j != i} (lambda_j - d_i) / (d_j - d_i):
// near boxes and the pair j = m-1 as products of shifted differences, the far
// boxes through the logarithmic form eq. (4.25) (dipole charges +1 at
// lambda_j, -1 at d_j).  One CTA of B threads per leaf box, one target each.
__global__ void __launch_bounds__(B) k_lowner_fmm(FmmDev pl, const int64_t *__restrict__ off, R1Out o)
{
    __shared__ __align__(16) double stage[4 * B];
    double *const sd = stage, *const so = stage + B, *const se = stage + 2 * B;    // FP64 products
    ff_w4 *const wd = (ff_w4 *)stage, *const wl = wd + B;                         // integer products
    const int tid = threadIdx.x;
    const int64_t nleaf = pl.leaf_base[pl.nprob];
    for (int64_t gl = blockIdx.x; gl < nleaf; gl += gridDim.x) {
        const int64_t p = sdc_upper_index(pl.leaf_base, pl.nprob, gl);
        if (pl.fslot[p] < 0) continue;
        const int64_t b0 = off[p];
        const int m = o.mk[p];
        const int Tb = (int)(gl - pl.leaf_base[p]);
        const int64_t g = pl.box_base[p] + Tb;
        const double *dk = o.dk + b0, *dorg = o.dorg + b0, *eta = o.eta + b0;
        const int i = Tb * B + tid;
        const bool act = i < m;
        const double di = act ? dk[i] : 0.0;
        Prod pr;
        FfProd fn = {1ull << 63, 0}, fd = {1ull << 63, 0};
        const bool ok = pl.ffbad[p] == 0;
        const FfScale fs = ff_scale(dk[0], dk[m - 1], o.wsum[p]);
        const ff_w4 d4 = ff_words4(ff_fixed(di, fs.kk) - fs.ref);
        const ff_u96 dw = {d4.lo, d4.mid, d4.hi};
        if (act && !ok) {
            const double num = (dorg[m - 1] - di) + eta[m - 1];
            const double den = (i == m - 1) ? 1.0 : dk[m - 1] - di;
            pr.mul(num, den);
        }
        const int nnr = pl.nnear[g];
        const int nn = near_len(nnr, (m + B - 1) / B);
        int64_t nsrc = 0;
        for (int s = 0; s < nn; s++) {
            const int S = near_box_chk(pl, g, nnr, s, (m + B - 1) / B, o.status);
            const int j0 = S * B;
            const int cnt = min(B, (m - 1) - j0);
            nsrc += max(cnt, 0);
            __syncthreads();
            if (tid < cnt) {
                if (ok) {
                    wd[tid] = ff_words4(ff_fixed(dk[j0 + tid], fs.kk) - fs.ref);
                    wl[tid] = ff_words4(ff_fixed(dorg[j0 + tid], fs.kk) + ff_fixed(eta[j0 + tid], fs.kk) - fs.ref);
                } else {
                    sd[tid] = dk[j0 + tid];
                    so[tid] = dorg[j0 + tid];
                    se[tid] = eta[j0 + tid];
                }
            }
            __syncthreads();
            if (ok) {
                ff_prod_sweep(wd, wl, cnt, j0, i, dw, fn, fd);
            } else if (act) {
                for (int jj = 0; jj < cnt; jj++) {
                    const double num = (so[jj] - di) + se[jj];
                    const double den = (j0 + jj == i) ? 1.0 : sd[jj] - di;
                    pr.mul(num, den);
                }
            }
        }
        if (act && ok) {
            // near factors outside the integer products, then those
            lowner_edges(dk, dorg, eta, di, i, m, pr.pn, pr.pd, pr.ex);
            pr.pn *= (double)fn.m;
            pr.pd *= (double)fd.m;
            pr.ex += fn.e - fd.e;
        }
        if (act) {
            double cT, hT;
            box_ch(pl.blo[g], pl.bhi[g], cT, hT);
            const double *cf = pl.coef + gl * NFIELD * P;
            const double u = (di - cT) * rcp_any(hT);
            int ex = pr.ex;
            const double Lf = ok ? low_eval(cf, u) + (double)clenshawf<LOWN>((const float *)(cf + LOWN), ff_top(u, 0))
                                 : clenshaw(cf, u);
            double v = root_quot(pr.pn, pr.pd, ex);
            v = ldexp(v, ex / 2) * exp(0.5 * Lf);
            if (!isfinite(v)) sdc_latch(o.status, SUPERDC_DEV_NONFINITE);
            o.vhat[b0 + i] = (o.zk[b0 + i] < 0.0) ? -v : v;
        }
        // near ratios (5 each, as the direct kernel), the far field's Clenshaw sum
        const int64_t nt = max(0, min(B, m - Tb * B));
        fl_add(pl, nt * (5 * (nsrc + 1) + 2 * P + 6));
    }
}

// b of the FMM problems, eq. (4.27): near boxes with the shifted entries of
// eq. (4.28), far boxes by expansion at lambda_j = d_{K_j} + eta_j.  The last
// target j = m-1 (outside the tree) is summed directly, spread over the leaf
// boxes: each box adds up its own sources in a fixed order into lastp, and
// k_fmm_lastsum combines the boxes (so no single CTA walks all m sources).
__global__ void __launch_bounds__(B) k_bnorm_fmm(FmmDev pl, const int64_t *__restrict__ off, R1Out o)
{
    __shared__ __align__(16) double stage[4 * B];
    double *const sd = stage, *const sv = stage + B;                // FP64 sums
    ff_f4 *const fd = (ff_f4 *)stage, *const fv = fd + B;           // three-float sums
    static_assert(B == 32, "one warp per leaf box");
    const int tid = threadIdx.x;
    const int64_t nleaf = pl.leaf_base[pl.nprob];
    for (int64_t gl = blockIdx.x; gl < nleaf; gl += gridDim.x) {
        const int64_t p = sdc_upper_index(pl.leaf_base, pl.nprob, gl);
        if (pl.fslot[p] < 0) continue;
        const int64_t b0 = off[p];
        const int m = o.mk[p];
        const int Tb = (int)(gl - pl.leaf_base[p]);
        const int64_t g = pl.box_base[p] + Tb;
        const int j = Tb * B + tid;
        const bool act = j < m - 1;
        const double dK = act ? o.dorg[b0 + j] : 0.0, e = act ? o.eta[b0 + j] : 0.0;
        const bool ok = pl.ffbad[p] == 0;
        const FfScale fs = ff_scale(o.dk[b0], o.dk[b0 + m - 1], o.wsum[p]);
        double s = 0.0;
        float tail = 0.0f;                        // the far field's single precision part
        if (act) {
            double cT, hT;
            box_ch(pl.blo[g], pl.bhi[g], cT, hT);
            const double *cf = pl.coef + gl * NFIELD * P;
            const double u = ((dK + e) - cT) * rcp_any(hT);
            if (ok) {
                s = low_eval(cf, u) * ff_pow2(2 * fs.kk + fs.kw);
                tail = clenshawf<LOWN>((const float *)(cf + LOWN), ff_top(u, 0));
            } else {
                s = clenshaw(cf, u);
            }
        }
        const int kv = fs.kw >> 1;
        const int K = act ? o.org[b0 + j] : -1;
        const ff_f4 x = ff_point(dK, e, fs);
        const double sc = ok ? ff_pow2(-kv) : 1.0;
        ff_t3 s3 = {(fs.kw & 1) ? tail + tail : tail, 0.0f, 0.0f};      // in units of 2^(2 (kv + kk))
        const int nnr = pl.nnear[g];
        const int nn = near_len(nnr, (m + B - 1) / B);
        int64_t nsrc = 0;
        for (int q = 0; q < nn; q++) {
            const int S = near_box_chk(pl, g, nnr, q, (m + B - 1) / B, o.status);
            const int i0 = S * B;
            const int cnt = min(B, m - i0);
            nsrc += max(cnt, 0);
            __syncthreads();
            if (tid < cnt) {
                if (ok) {
                    const ff_t3 t = ff_split3(o.vhat[b0 + i0 + tid] * sc);
                    fd[tid] = ff_pole(o.dk[b0 + i0 + tid], fs);
                    fv[tid] = {t.a, t.b, t.c, 0.0f};
                } else {
                    sd[tid] = o.dk[b0 + i0 + tid];
                    sv[tid] = o.vhat[b0 + i0 + tid];
                }
            }
            __syncthreads();
            if (ok) {
                ff_sqr_sweep(fd, fv, cnt, i0, K, x, s3);
            } else if (act) {
                for (int ii = 0; ii < cnt; ii++) {
                    const double r = rcp_nr2((sd[ii] - dK) - e);
                    const double vr = sv[ii] * r;
                    s = fma(vr, vr, s);
                }
            }
        }
        if (act && ok) {
            const double vr = o.vhat[b0 + K] * rcp_nr2(-e);         // the origin's term
            s = fma(vr, vr, fma(ff_join3(s3), ff_pow2(2 * (kv + fs.kk)), s));
        }
        if (act) o.bnorm[b0 + j] = rsqrt_any(s);
        // this box's sources in the sum for the last target
        double t = 0.0;
        if (j < m) {
            const double r = rcp_nr2((o.dk[b0 + j] - o.dorg[b0 + m - 1]) - o.eta[b0 + m - 1]);
            const double vr = o.vhat[b0 + j] * r;
            t = vr * vr;
        }
        for (int sh = 16; sh > 0; sh >>= 1) t += __shfl_xor_sync(0xffffffffu, t, sh);
        if (tid == 0) pl.lastp[gl] = t;
        // near terms (6 each, as the direct kernel), Clenshaw, the last target's share
        const int64_t nt = max(0, min(B, (m - 1) - Tb * B)), ns = max(0, min(B, m - Tb * B));
        fl_add(pl, nt * (6 * nsrc + 2 * P + 2) + ns * 7);
    }
}

// The last eigenvalue's b from the leaf boxes' shares (lastp), one warp per FMM
// problem, in a fixed order: lane-strided partial sums, then a butterfly.
__global__ void __launch_bounds__(128) k_fmm_lastsum(FmmDev pl, const int64_t *__restrict__ off,
                                                     const int32_t *__restrict__ mk, double *__restrict__ bout)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = *pl.nfmm;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < nw;
         w += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int64_t p = pl.fprob[w];
        if (pl.fslot[p] < 0) continue;
        double a = 0.0;
        for (int64_t gl = pl.leaf_base[p] + lane; gl < pl.leaf_base[p + 1]; gl += 32) a += pl.lastp[gl];
        for (int sh = 16; sh > 0; sh >>= 1) a += __shfl_xor_sync(0xffffffffu, a, sh);
        if (lane == 0) bout[off[p] + mk[p] - 1] = 1.0 / sqrt(a);
    }
}

// ---------------------------------------------------------------------------
// Cauchy-like applications to blocks of columns on the tensor cores.
//
// Y = Qhat^T X or Qhat X is, per tile of 16 targets, a product of a kernel
// matrix and a block: sources are the poles (eigenvalues) of the near boxes, or
// every one of a problem without a tree, with the columns as they are, and the
// Chebyshev nodes of the boxes of the interaction lists of the tile's leaf and
// its ancestors with the node weights.  In FP64 that is one FMA per entry and
// column on a pipe that retires 2 per clock.  Here both operands are cut into
// seven 8-bit digits on fixed grids (Ozaki, Ogita, Oishi, Rump, Error-free
// transformations of matrix multiplication, 2012), every product of two digit
// matrices is a bf16 mma whose FP32 sums are exact integers (128 sources of
// products below 2^14, up to seven per order, stay below 2^24), and the 28
// products with i + j <= 8 carry the result to 2^-55 of the largest entry
// times the largest column value.
//   * Kernel entries come from split positions (three floats, ff_diff3,
//     ff_rcp3).  Near rows are scaled by the power of two below b_j (|v_i| for
//     Qhat X): an entry is then at most one in magnitude, as one of an
//     orthogonal matrix, and the error is that of FP64 in norm.  Far rows
//     share one power of two per tile that covers every box of the lists.
//   * The source that may be closer than the positions resolve (the origin of
//     eta_j) and the last eigenvalue (outside the positions' range) are added
//     in FP64.
//   * Problems out of the positions' scale (cm_prep) take FP64 loops.
// Digit fragments of the columns are read in mma order from global memory
// (written once per pass of 64 columns by k_cm_slice / k_cm_up).
// ---------------------------------------------------------------------------
constexpr int CM_D = 7;           // digits
constexpr int CM_NT = 8;          // column tiles of 8 per pass
constexpr int CM_TR = 64;         // targets per entry of tile_off, four CTAs of 16
constexpr int CM_TAKE = 8;        // far boxes taken per level and round
constexpr int CM_BC = F64_COLS;   // columns per pass of the FP64 loops

__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }      // -126 <= e <= 127

__device__ __forceinline__ int64_t cm_chunk(int64_t b0, int64_t p) { return (b0 >> 4) + p; }   // 16-slot chunks

// digit s (1..7) of y in [-1, 1] on the grid 2^-(8 s - 1), as bf16 bits
__device__ __forceinline__ void cm_digits(double y, unsigned short *out)
{
    long long v = __double2ll_rn(y * 36028797018963968.0);        // 2^55
#pragma unroll
    for (int s = 1; s <= CM_D; s++) {
        const int sh = 8 * (CM_D - s);
        const long long d = (s < CM_D) ? (v + (1ll << (sh - 1))) >> sh : v;
        v -= d << sh;
        out[s - 1] = (unsigned short)(__float_as_uint((float)(int)d * pow2f(1 - 8 * s)) >> 16);
    }
}

// positions and factors of the sources, and the problems out of scale
struct CmDev {
    ff_f4 *pos, *fac;            // per slot: source position, source factor (three floats)
    int32_t *bad;                // per problem, then whether any is
    int32_t *cmax;               // per (problem, column of the call): biased exponent of max |x| of the kept rows
    int64_t ccols;               // columns of the call (stride of cmax)
    uint2 *xf;                   // column digits in mma order: [chunk][tile][digit][lane]
    uint2 *wf0;                  // node weights' digits: nodes 0..15 [box][tile][digit][lane]
    unsigned *wf1;               //                       nodes 16..21
    int32_t *eb;                 // per box: exponent of its node weights over the columns' scales
    double *lastp;               // per (tile of 64, column of the pass): partial sums for the last eigenvalue
    double *coef;                // per leaf box and column: far field's series of the problems out of scale
    int cs;                      // their columns per leaf box
};

// Positions and factors of the sources; which problems are out of scale; the scale of
// every column over its problem's kept rows (a deflated row passes through unchanged,
// whatever its size).  A problem with a non-finite entry takes the FP64 loops: the
// digits of one column share the boxes' scales with the others.
template <bool TRANS>
__global__ void k_cm_prep(FactorView f, int64_t total, const double *__restrict__ X, int64_t ldx, int ncols, CmDev c)
{
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total;
         x += (int64_t)gridDim.x * blockDim.x) {
        if (x < f.off[0] || x >= f.off[f.nprob]) continue;
        const int64_t p = sdc_upper_index(f.off, f.nprob, x);
        const int64_t b0 = f.off[p];
        const int m = f.mk[p], j = (int)(x - b0);
        if (j >= m) continue;
        const double *dk = f.dk + b0;
        const FfScale s = ff_scale(dk[0], dk[m - 1], 1.0);
        const double dK = f.dorg[x];
        bool ok = s.ok && m >= 2 && (j + 1 >= m || ff_gap_ok(dk[j], dk[j + 1], s.kk)) &&
                  (dK == dk[j] || (j + 1 < m && dK == dk[j + 1]));
        const double v = TRANS ? f.vhat[x] : f.bnorm[x] * ff_pow2(s.ok ? s.kk : 0);
        const int ev = ff_exp(f.vhat[x]), eb = ff_exp(f.bnorm[x] * ff_pow2(s.ok ? s.kk : 0));
        ok = ok && ev > 923 && ev < 1113 && eb > 923 && eb < 1113;
        if (!ok) {
            c.bad[p] = 1;
            c.bad[f.nprob] = 1;
            continue;
        }
        const ff_t3 t = ff_split3(v);
        c.fac[x] = {t.a, t.b, t.c, 0.0f};
        c.pos[x] = (TRANS || j == m - 1) ? ff_pole(dk[j], s) : ff_point(dK, f.eta[x], s);
    }
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total * ncols;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t x = t % total;
        const int col = (int)(t / total);
        int64_t p = -1;
        int e = 0;
        if (x >= f.off[0] && x < f.off[f.nprob]) {
            p = sdc_upper_index(f.off, f.nprob, x);
            const int64_t b0 = f.off[p];
            if (x - b0 < f.mk[p])
                e = ff_exp(X[b0 + SDC_IDX(TRANS ? f.src[x] : f.pinv[x], f.off[p + 1] - b0, f.status) + (int64_t)col * ldx]);
        }
        // one atomic per run of lanes with the same problem and column
        const unsigned grp = __match_any_sync(__activemask(), p * ncols + col);
        const int mx = __reduce_max_sync(grp, e);
        if (p >= 0 && (int)(threadIdx.x & 31) == __ffs(grp) - 1 && mx > 0) {
            atomicMax(&c.cmax[p * c.ccols + col], mx);
            if (mx == 0x7FF) {
                c.bad[p] = 1;
                c.bad[f.nprob] = 1;
            }
        }
    }
}

// 2^-e x with |x| < 2^e for every kept row of the problem (e from the biased exponent)
__device__ __forceinline__ int cm_exp(const CmDev &c, int64_t p, int col) { return c.cmax[p * c.ccols + col] - 1022; }

// digits of the columns [col0, col0 + nc) of the kept slots; row: src (TRANS) or pinv
template <bool TRANS>
__global__ void k_cm_slice(FactorView f, int64_t nchunk_rows, const double *__restrict__ X, int64_t ldx, int col0,
                           int nc, int nt, CmDev c)
{
    // one thread per (row, column): rows in units of chunks of 16
    const int64_t n = nchunk_rows * nt * 8;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t row = t % nchunk_rows;            // chunk * 16 + k
        const int col = (int)(t / nchunk_rows);
        const int64_t ch = row >> 4;
        const int k = (int)(row & 15);
        // problem of the chunk: the last with cm_chunk(off, p) <= ch
        int64_t lo = 0, hi = f.nprob;
        while (hi - lo > 1) {
            const int64_t mid = (lo + hi) >> 1;
            if (cm_chunk(f.off[mid], mid) <= ch) lo = mid; else hi = mid;
        }
        const int64_t b0 = f.off[lo];
        const int64_t first = cm_chunk(b0, lo);
        if (ch < first) continue;
        const int j = (int)((ch - first) * 16 + k), m = f.mk[lo];
        if ((ch - first) * 16 >= m) continue;
        unsigned short dg[CM_D] = {0, 0, 0, 0, 0, 0, 0};
        if (col < nc && j < m && c.bad[lo] == 0) {
            const int64_t r = b0 + SDC_IDX(TRANS ? f.src[b0 + j] : f.pinv[b0 + j], f.off[lo + 1] - b0, f.status);
            const int e = cm_exp(c, lo, col0 + col);
            cm_digits(ldexp(X[r + (int64_t)(col0 + col) * ldx], -e), dg);
        }
        // B fragment of m16n8k16: column n = lane / 4, k = 2 (lane % 4) + {0, 1} (+ 8)
        const int lane = (col & 7) * 4 + ((k & 7) >> 1);
        unsigned short *dst = (unsigned short *)(c.xf + ((ch * nt + (col >> 3)) * CM_D) * 32 + lane);
        for (int s = 0; s < CM_D; s++) dst[(int64_t)s * 32 * 4 + ((k >> 3) << 1) + (k & 1)] = dg[s];
    }
}

__device__ __forceinline__ void cm_mma16(float (&d)[4], const uint4 &a, uint2 b)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y));
}

__device__ __forceinline__ void cm_mma8(float (&d)[4], unsigned a0, unsigned a1, unsigned b)
{
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(b));
}

// digits of an entry t (three floats, |t| <= 1) as floats on the grids 2^-(8 s - 1)
__device__ __forceinline__ void cm_cut(const ff_t3 &t, float (&d)[CM_D])
{
    float r = t.a;
#pragma unroll
    for (int s = 0; s < CM_D; s++) {
        if (s == 3) {                               // the leading part has 24 bits: bring in the next
            float e;
            ff_two_sum(r, t.b, r, e);
            d[6] = ff_add(e, t.c);
        }
        if (s == 6) r = ff_add(r, d[6]);
        const float M = 1.5f * (float)(1 << 23) * pow2f(-7 - 8 * s);
        d[s] = ff_sub(ff_add(r, M), M);
        r = ff_sub(r, d[s]);
    }
}

// two neighbouring k of a row: bf16 pair (the digits fit in 8 bits: truncation is exact)
__device__ __forceinline__ unsigned cm_pack(float lo, float hi)
{
    return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}

// exact sums of the orders i + j = 2..8 (unit entries) in two integers: hi 2^-30 + lo 2^-62
struct CmSum { long long hi, lo; };

__device__ __forceinline__ void cm_add(CmSum &v, const float (&a)[CM_D][4], int i)
{
    v.hi += ((long long)__float2int_rn(a[0][i] * 0x1p14f) << 16) + ((long long)__float2int_rn(a[1][i] * 0x1p22f) << 8) +
            __float2int_rn(a[2][i] * 0x1p30f);
    v.lo += ((long long)__float2int_rn(a[3][i] * 0x1p38f) << 24) + ((long long)__float2int_rn(a[4][i] * 0x1p46f) << 16) +
            ((long long)__float2int_rn(a[5][i] * 0x1p54f) << 8) + __float2int_rn(a[6][i] * 0x1p62f);
}

__device__ __forceinline__ double cm_value(const CmSum &v) { return fma((double)v.hi, 0x1p-30, (double)v.lo * 0x1p-62); }

__device__ __forceinline__ double cm_fold(const float (&a)[CM_D][4], int i)
{
    CmSum v = {0, 0};
    cm_add(v, a, i);
    return cm_value(v);
}

// ---------------------------------------------------------------------------
// Node weights of blocks of columns, on the tensor cores: a leaf box's weights
// are the matrix L_q(u_j) v_j (Chebyshev interpolation at the 22 nodes, times
// the source factor) times its columns, a parent's the matrix L_q of its
// children's nodes times their weights.  The matrices are formed by the second
// barycentric formula L_q(u) = (w_q / (u - x_q)) / sum_k (w_k / (u - x_k)) in
// three floats (Berrut and Trefethen, Barycentric Lagrange interpolation, 2004:
// stable for any u in the interval), cut into digits and multiplied as in
// k_cm_apply; the weights leave as the digits the next level and k_cm_apply
// read.  The climb and its arrival counters are those of k_fmm_up, which still
// does the problems out of scale.  A leaf and its parent took 33 k cycles of the
// FP64 pipe for 24 columns.  Measured (GB300, f(A) X, n = 32768, 64 columns;
// 24 columns a pass): 196 -> 59 ms, with 64 columns a pass 36.
// ---------------------------------------------------------------------------
constexpr int CU_ROWS = 32;       // matrix rows (22 nodes, zeros below)
constexpr int CU_LD = 56;         // bf16 per row: up to 48 sources, 112 bytes (no bank conflicts)

// u - x, three floats each
__device__ __forceinline__ ff_t3 ff_sub3(const ff_t3 &u, const ff_t3 &x)
{
    float s, e1, t, e2, e3;
    ff_two_sum(u.a, -x.a, s, e1);
    ff_two_sum(u.b, -x.b, t, e2);
    ff_two_sum(t, e1, t, e3);
    ff_t3 o;
    ff_two_sum(s, t, o.a, t);
    ff_fast_sum(t, ff_add(ff_sub(u.c, x.c), ff_add(e2, e3)), o.b, o.c);
    return o;
}

__device__ __forceinline__ ff_t3 ff_shfl3(const ff_t3 &v, int mask)
{
    return {__shfl_xor_sync(0xffffffffu, v.a, mask), __shfl_xor_sync(0xffffffffu, v.b, mask),
            __shfl_xor_sync(0xffffffffu, v.c, mask)};
}

// The columns k0 .. k0 + n - 1 of the digit matrices: four threads per source
// take every fourth node.  su: sources' variables, sf: their factors.
__device__ __forceinline__ void cu_matrix(const ff_t3 *su, const ff_t3 *sf, const ff_t3 *sx, const ff_t3 *sw, int k0,
                                          int n, unsigned short (*As)[CU_ROWS][CU_LD])
{
    constexpr int QN = (P + 3) / 4;
    for (int t0 = 0; t0 < n * 4; t0 += blockDim.x) {     // n a multiple of 8: whole warps
        const int t = t0 + threadIdx.x, k = t >> 2, part = t & 3;
        if (k >= n) continue;
        const ff_t3 u = su[k];
        ff_t3 wr[QN], D = {0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int i = 0; i < QN; i++) {
            const int q = min(part + 4 * i, P - 1);
            ff_t3 d = ff_sub3(u, sx[q]);
            if (fabsf(d.a) < 0x1p-60f) d = {0x1p-60f, 0.0f, 0.0f};     // on a node: L = 1 there, 2^-60 elsewhere
            wr[i] = ff_mul3(sw[q], ff_rcp3(d));
            if (part + 4 * i < P) ff_acc3(D, wr[i]);
        }
        ff_acc3(D, ff_shfl3(D, 1));
        ff_acc3(D, ff_shfl3(D, 2));
        // renormalise, then the source's factor over D
        float s, e;
        ff_fast_sum(D.a, D.b, s, e);
        D.a = s;
        ff_fast_sum(e, D.c, D.b, D.c);
        const ff_t3 f = ff_mul3(sf[k], ff_rcp3(D));
#pragma unroll
        for (int i = 0; i < QN; i++) {
            const int q = part + 4 * i;
            if (q >= P) continue;
            float dg[CM_D];
            cm_cut(ff_mul3(wr[i], f), dg);
#pragma unroll
            for (int s2 = 0; s2 < CM_D; s2++) As[s2][q][k0 + k] = (unsigned short)(__float_as_uint(dg[s2]) >> 16);
        }
    }
}

template <int NTM, bool TRANS>          // NTM: most column tiles of a pass (shared memory)
__global__ void __launch_bounds__(128) k_cm_up(FmmDev pl, FactorView f, CmDev c, int col0, int nc, int nt)
{
    __shared__ __align__(16) unsigned short As[CM_D][CU_ROWS][CU_LD];
    __shared__ __align__(16) uint2 o0[2 * CM_D * 32];        // digits of two column tiles
    __shared__ unsigned o1[2 * CM_D * 32];
    __shared__ double Ws[P][NTM * 8];
    __shared__ ff_t3 sx[P], sw[P], su[48], sf[48];
    __shared__ double xq[P];
    __shared__ int s_e, s_last;
    __shared__ int64_t s_next;
    const unsigned FULL = 0xffffffffu;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gr = lane >> 2, gc = lane & 3;
    for (int i = tid; i < CM_D * CU_ROWS * CU_LD; i += 128) ((unsigned short *)As)[i] = 0;
    if (tid < P) {
        xq[tid] = cospi((double)(2 * tid + 1) / (2.0 * P));
        sx[tid] = ff_split3(xq[tid]);
        const double w = sinpi((double)(2 * tid + 1) / (2.0 * P));
        sw[tid] = ff_split3((tid & 1) ? -w : w);
    }
    const int64_t nleaf = pl.leaf_base[pl.nprob];
    for (;;) {
        __syncthreads();
        if (tid == 0) {
            s_next = (int64_t)atomicAdd(&pl.upq[0], 1ull);
            if (s_next >= nleaf && atomicAdd(&pl.upq[1], 1ull) == gridDim.x - 1) {
                pl.upq[0] = 0;                 // every CTA has run past the end: reset for the next launch
                pl.upq[1] = 0;
            }
        }
        __syncthreads();
        const int64_t gl = s_next;
        if (gl >= nleaf) break;
        const int64_t p = sdc_upper_index(pl.leaf_base, pl.nprob, gl);
        if (pl.fslot[p] < 0 || c.bad[p]) continue;
        const int64_t b0 = f.off[p], g0 = pl.box_base[p];
        const int m = f.mk[p], nb0 = (m + B - 1) / B, L = lev_count(nb0);
        const double *dk = f.dk + b0;
        const int kk = ff_scale(dk[0], dk[m - 1], 1.0).kk;
        int l = 0, b = (int)(gl - pl.leaf_base[p]);
        for (;;) {
            const int64_t g = g0 + lev_base(nb0, l) + b;
            int nch = 0, E0 = 0;
            int64_t gc0 = 0;
            if (l == 0) {
                // sources of the leaf: variable, factor scaled to at most one
                if (warp == 0) {
                    const int j = b * B + lane, jend = TRANS ? m : m - 1;
                    double cT, hT;
                    box_ch(pl.blo[g], pl.bhi[g], cT, hT);
                    double u = 0.0;
                    ff_t3 v = {0.0f, 0.0f, 0.0f};
                    if (j < jend) {
                        u = TRANS ? (dk[j] - cT) / hT : ((f.dorg[b0 + j] - cT) + f.eta[b0 + j]) / hT;
                        const ff_f4 fc = c.fac[b0 + j];
                        v = {fc.x, fc.y, fc.z};
                    }
                    int e = v.a != 0.0f ? ff_fexp(fabsf(v.a)) + 1 : -126;
                    e = __reduce_max_sync(FULL, e);
                    const float sc = pow2f(max(-126, min(126, -e)));
                    su[lane] = ff_split3(u);
                    sf[lane] = {v.a * sc, v.b * sc, v.c * sc};
                    if (lane == 0) s_e = e - (TRANS ? 0 : kk);            // Qhat X: the factors carry 2^kk
                }
            } else {
                const int nbc = lev_nb(nb0, l - 1);
                gc0 = g0 + lev_base(nb0, l - 1) + 2 * b;
                nch = (2 * b + 1 < nbc) ? 2 : 1;
                if (warp < 2) {
                    const int ea = __ldcg(&c.eb[gc0]), eb = nch > 1 ? __ldcg(&c.eb[gc0 + 1]) : -4000;
                    const int em = max(ea, eb), ec = warp == 0 ? ea : eb;
                    if (warp < nch) {
                        double cP, hP, cc, hc;
                        box_ch(pl.blo[g], pl.bhi[g], cP, hP);
                        box_ch(pl.blo[gc0 + warp], pl.bhi[gc0 + warp], cc, hc);
                        const double ih = rcp_nr2(hP);
                        if (lane < 24) {
                            // the node as scale and shift (exact for boxes of one point)
                            su[warp * 24 + lane] = ff_split3(fma(hc * ih, xq[min(lane, P - 1)], (cc - cP) * ih));
                            const float sc = (ec < em - 120 || lane >= P) ? 0.0f : pow2f(ec - em);
                            sf[warp * 24 + lane] = {sc, 0.0f, 0.0f};
                        }
                    }
                    if (warp == 0 && lane == 0) s_e = em;
                }
            }
            __syncthreads();
            E0 = s_e;
            cu_matrix(su, sf, sx, sw, 0, l == 0 ? B : 24 * nch, As);
            __syncthreads();
            // products: (16 nodes, 8 columns) per warp
            for (int un = warp; un < 2 * nt; un += 4) {
                const int mt = un & 1, n = un >> 1;
                float acc[CM_D][4];
#pragma unroll
                for (int s = 0; s < CM_D; s++)
#pragma unroll
                    for (int i = 0; i < 4; i++) acc[s][i] = 0.0f;
                const int r0 = mt * 16 + gr;
                auto frag = [&](int s, int row, int k) {
                    return *(const unsigned *)&As[s][row][k + 2 * gc];
                };
                const int n16 = l == 0 ? 2 : nch;
                for (int st = 0; st < n16; st++) {
                    const int k0 = l == 0 ? 16 * st : 24 * st;
                    const uint2 *bf = l == 0 ? c.xf + (((cm_chunk(b0, p) + 2 * b + st) * nt + n) * CM_D) * 32 + lane
                                             : c.wf0 + (((gc0 + st) * nt + n) * CM_D) * 32 + lane;
                    if (l == 0 && b * B + 16 * st >= m) continue;
                    uint2 bb[CM_D];
                    uint4 a[CM_D];
#pragma unroll
                    for (int s = 0; s < CM_D; s++) {
                        bb[s] = __ldcg(bf + s * 32);
                        a[s] = make_uint4(frag(s, r0, k0), frag(s, r0 + 8, k0), frag(s, r0, k0 + 8),
                                          frag(s, r0 + 8, k0 + 8));
                    }
#pragma unroll
                    for (int i1 = 0; i1 < CM_D; i1++)
#pragma unroll
                        for (int j1 = 0; i1 + j1 < CM_D; j1++) cm_mma16(acc[i1 + j1], a[i1], bb[j1]);
                }
                for (int st = 0; st < nch; st++) {
                    const unsigned *bf = c.wf1 + (((gc0 + st) * nt + n) * CM_D) * 32 + lane;
                    unsigned bb[CM_D], a[CM_D][2];
#pragma unroll
                    for (int s = 0; s < CM_D; s++) {
                        bb[s] = __ldcg(bf + s * 32);
                        a[s][0] = frag(s, r0, 24 * st + 16);
                        a[s][1] = frag(s, r0 + 8, 24 * st + 16);
                    }
#pragma unroll
                    for (int i1 = 0; i1 < CM_D; i1++)
#pragma unroll
                        for (int j1 = 0; i1 + j1 < CM_D; j1++) cm_mma8(acc[i1 + j1], a[i1][0], a[i1][1], bb[j1]);
                }
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const int q = r0 + 8 * (i >> 1), col = n * 8 + 2 * gc + (i & 1);
                    if (q < P) Ws[q][col] = col < nc ? cm_fold(acc, i) : 0.0;
                }
            }
            __syncthreads();
            // the box's exponent, then its digits
            int ex = 0;
            for (int i = tid; i < P * nt * 8; i += 128) ex = max(ex, ff_exp(Ws[i / (nt * 8)][i % (nt * 8)]));
            ex = __reduce_max_sync(FULL, ex);
            if (tid == 0) s_e = 0;
            __syncthreads();
            if (lane == 0) atomicMax(&s_e, ex);
            __syncthreads();
            ex = s_e;
            const double sc = ex > 0 ? ff_pow2(1022 - ex) : 0.0;
            for (int n0 = 0; n0 < nt; n0 += 2) {
                const int nb = min(2, nt - n0);
                for (int i = tid; i < 24 * nb * 8; i += 128) {
                    const int k = i / (nb * 8), col = i % (nb * 8);
                    unsigned short dg[CM_D];
                    cm_digits(k < P ? Ws[k][n0 * 8 + col] * sc : 0.0, dg);
                    const int ln = (col & 7) * 4 + ((k & 7) >> 1), at = (col >> 3) * CM_D * 32 + ln;
                    unsigned short *dst = k < 16 ? (unsigned short *)(o0 + at) + ((k >> 3) << 1) + (k & 1)
                                                 : (unsigned short *)(o1 + at) + (k & 1);
                    const int step = k < 16 ? 32 * 4 : 32 * 2;
#pragma unroll
                    for (int s = 0; s < CM_D; s++) dst[s * step] = dg[s];
                }
                __syncthreads();
                for (int i = tid; i < nb * CM_D * 32; i += 128) {
                    c.wf0[(g * nt + n0) * CM_D * 32 + i] = o0[i];
                    c.wf1[(g * nt + n0) * CM_D * 32 + i] = o1[i];
                }
                __syncthreads();
            }
            if (tid == 0) c.eb[g] = ex > 0 ? E0 + ex - 1022 : -4000;
            if (l + 1 >= L) break;
            // the child that arrives last computes the parent (k_fmm_up)
            const int bp = b >> 1;
            const int nsib = (2 * bp + 1 < lev_nb(nb0, l)) ? 2 : 1;
            const int64_t gp = g0 + lev_base(nb0, l + 1) + bp;
            __threadfence();
            __syncthreads();
            if (tid == 0) {
                const int old = atomicAdd(&pl.upcnt[gp], 1);
                s_last = (old == nsib - 1);
                if (s_last) pl.upcnt[gp] = 0;
            }
            __syncthreads();
            if (!s_last) break;
            __threadfence();
            l++;
            b = bp;
        }
    }
}

// digits of the kernel entries of up to 32 sources (22 nodes) and 16 targets, in mma order
struct __align__(16) CmFrag { uint4 k[2][CM_D][32]; };

// The CTA's four warps form the digits of four boxes at a time (near boxes of 32
// sources, or the 22 nodes of far boxes), then multiply: warp w has the column
// tiles w % NTP + NTP i (i < TPW) of every (4 / NTP)-th box.
// What bounds it: forming a 16 x 16 block takes 800 warp instructions (three-float
// quotient and 7 digits an entry), its products 28 mma per column tile.  One warp
// per 16 targets with three tiles of its own held 255 registers: 8 warps per SM at
// 26 % of the issue slots, and every 24 columns formed the entries again.  Here a
// warp holds one or two tiles and an entry is formed once for 64 columns.
// Measured (GB300, f(A) X, n = 32768, 64 columns): 86 -> 57 ms; the
// eigendecomposition of n = 131072 (1 to 19 columns): 61 -> 58 ms.
template <int NTP, int TPW, bool TRANS>
__global__ void __launch_bounds__(128, TPW == 1 ? 4 : 3)
k_cm_apply(FmmDev pl, FactorView f, const int64_t *__restrict__ tile_off, CmDev c, const double *__restrict__ X,
           int64_t ldx, double *__restrict__ Y, int64_t ldy, int col0, int nc, int nt)
{
    constexpr int NS = 4 / NTP;                          // warps that share a column tile
    __shared__ CmFrag sA[4];
    __shared__ int2 list[32 * CM_TAKE];                  // far boxes: index, exponent of its weights
    __shared__ int lim[32 * CM_TAKE];                    // and of its largest term: weights over distance
    __shared__ int64_t s_pst[32];                        // per level: the list's start, the target's ancestor
    __shared__ int s_lb[32];
    __shared__ double s_lo[32], s_hi[32];
    __shared__ int s_total, s_ET;
    // a warp that multiplies what it formed itself needs no barrier
    auto boxes_sync = [&]() { if (NS == 4) __syncwarp(); else __syncthreads(); };
    const unsigned FULL = 0xffffffffu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gr = lane >> 2, gc = lane & 3;
    const int tl = warp % NTP, grp = warp / NTP;
    const int64_t ntiles = tile_off[f.nprob] * 4;
    for (int64_t it = blockIdx.x; it < ntiles; it += gridDim.x) {
        const int64_t tile = it >> 2;
        const int64_t p = sdc_upper_index(tile_off, f.nprob, tile);
        const int64_t b0 = f.off[p];
        const int m = f.mk[p];
        const int t0 = (int)(tile - tile_off[p]) * CM_TR + (int)(it & 3) * 16;
        const int tend = TRANS ? m - 1 : m;              // T: the last target is summed by k_cm_last
        if (t0 >= tend || c.bad[p]) continue;            // out of scale: k_cm_rest
        const bool tree = pl.fslot && pl.fslot[p] >= 0;
        const double *dk = f.dk + b0, *dorg = f.dorg + b0, *eta = f.eta + b0;
        const int nb0 = (m + B - 1) / B, Tb = t0 / B;
        const int64_t gbx = tree ? pl.box_base[p] : 0;
        const int nnr = tree ? pl.nnear[gbx + Tb] : -1;
        const int nn = near_len(nnr, nb0);               // without a tree: every box
        const int nsrc = TRANS ? m : m - 1;
        const FfScale fs = ff_scale(dk[0], dk[m - 1], 1.0);
        // the two rows of this lane: positions and the powers of two of their near entries
        ff_f4 x[2];
        float rs[2];
        double ns[2];                                    // near sums times this (2^kk by the factors of Qhat X)
        int skip[2];                                     // T: the origin's index; N: the target (skip, skip - 1)
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int r = min(t0 + gr + 8 * h, tend - 1);
            const double sc = TRANS ? f.bnorm[b0 + r] : f.vhat[b0 + r];
            x[h] = TRANS ? ff_point(dorg[r], eta[r], fs) : ff_pole(dk[r], fs);
            const int e = max(-126, min(126, ff_exp(sc) - 1023 + (TRANS ? fs.kk : 0)));
            rs[h] = pow2f(e);
            ns[h] = ff_pow2((TRANS ? fs.kk : 0) - e);
            skip[h] = TRANS ? (dorg[r] == dk[r] ? r : r + 1) : r;
        }
        float acc[TPW][CM_D][4];
        CmSum sum[TPW][4];                               // of the folds: FP64 only once per field
        double y[TPW][4];
        auto clear = [&]() {
#pragma unroll
            for (int t = 0; t < TPW; t++)
#pragma unroll
                for (int s = 0; s < CM_D; s++)
#pragma unroll
                    for (int i = 0; i < 4; i++) acc[t][s][i] = 0.0f;
        };
        auto fold = [&]() {
#pragma unroll
            for (int t = 0; t < TPW; t++)
#pragma unroll
                for (int i = 0; i < 4; i++) cm_add(sum[t][i], acc[t], i);
            clear();
        };
        // y += the sums of all warps times sc (rows gr, gr + 8), in the first group's warps
        auto collect = [&](double sc0, double sc1) {
            fold();
            if (NS > 1) {
                CmSum *red = (CmSum *)sA;
                __syncthreads();                         // every warp is done with the digits
                if (grp > 0)
#pragma unroll
                    for (int q = 0; q < 4 * TPW; q++)
                        red[(((grp - 1) * NTP + tl) * 4 * TPW + q) * 32 + lane] = sum[q >> 2][q & 3];
                __syncthreads();
                if (grp == 0)
                    for (int w = 0; w < NS - 1; w++)
#pragma unroll
                        for (int q = 0; q < 4 * TPW; q++) {
                            const CmSum v = red[((w * NTP + tl) * 4 * TPW + q) * 32 + lane];
                            sum[q >> 2][q & 3].hi += v.hi;
                            sum[q >> 2][q & 3].lo += v.lo;
                        }
            }
#pragma unroll
            for (int t = 0; t < TPW; t++)
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    if (grp == 0) y[t][i] = fma(cm_value(sum[t][i]), i < 2 ? sc0 : sc1, y[t][i]);
                    sum[t][i] = {0, 0};
                }
            __syncthreads();
        };
        // the products of the staged digits k[half] of box v with this warp's column tiles
        auto mult16 = [&](int v, int half, const uint2 *__restrict__ bf) {
            uint4 a[CM_D];
#pragma unroll
            for (int s = 0; s < CM_D; s++) a[s] = sA[v].k[half][s][lane];
#pragma unroll
            for (int t = 0; t < TPW; t++) {
                const int n = tl + NTP * t;
                if (n >= nt) break;
                uint2 b[CM_D];
#pragma unroll
                for (int s = 0; s < CM_D; s++) b[s] = bf[(n * CM_D + s) * 32 + lane];
#pragma unroll
                for (int i1 = 0; i1 < CM_D; i1++)
#pragma unroll
                    for (int j1 = 0; i1 + j1 < CM_D; j1++) cm_mma16(acc[t][i1 + j1], a[i1], b[j1]);
            }
        };
        auto mult8 = [&](int v, const unsigned *__restrict__ bf) {
            uint2 a[CM_D];
#pragma unroll
            for (int s = 0; s < CM_D; s++) a[s] = ((const uint2 *)sA[v].k[1][s])[lane];
#pragma unroll
            for (int t = 0; t < TPW; t++) {
                const int n = tl + NTP * t;
                if (n >= nt) break;
                unsigned b[CM_D];
#pragma unroll
                for (int s = 0; s < CM_D; s++) b[s] = bf[(n * CM_D + s) * 32 + lane];
#pragma unroll
                for (int i1 = 0; i1 < CM_D; i1++)
#pragma unroll
                    for (int j1 = 0; i1 + j1 < CM_D; j1++) cm_mma8(acc[t][i1 + j1], a[i1].x, a[i1].y, b[j1]);
            }
        };
        clear();
#pragma unroll
        for (int t = 0; t < TPW; t++)
#pragma unroll
            for (int i = 0; i < 4; i++) { y[t][i] = 0.0; sum[t][i] = {0, 0}; }
        __syncthreads();                                 // the previous tile's list and digits
        // ---- far field: the nodes of the interaction lists
        int far_src = 0;
        if (tree && nnr >= 0) {
            // warp 0, lane l: the list of the tile's ancestor on level l
            const int L = lev_count(nb0);
            int A = 0, npn = 0, nbl = 0, lb = 0, sec = 0;
            int64_t pst = 0;
            unsigned long long mask = 0;
            if (warp == 0 && lane < L - 1) {
                A = Tb >> lane;
                lb = lev_base(nb0, lane);
                nbl = lev_nb(nb0, lane);
                const int64_t gP = gbx + lev_base(nb0, lane + 1) + (A >> 1);
                npn = pl.nnear[gP];
                pst = pl.nstart[gP];
                mask = pl.amask[gbx + lb + A];
                s_pst[lane] = pst;
                s_lb[lane] = lb;
                s_lo[lane] = pl.blo[gbx + lb + A];
                s_hi[lane] = pl.bhi[gbx + lb + A];
            }
            for (;;) {
                // a round: warp 0 numbers the boxes, every thread looks one up; the
                // round's digits share the largest weight over distance, 2^ET
                if (warp == 0) {
                    int total = -1;
                    if (__any_sync(FULL, mask != 0 || 64 * (sec + 1) < 2 * npn)) {
                        if (mask == 0 && 64 * (sec + 1) < 2 * npn) {
                            sec++;
                            mask = adm_mask(pl, gbx + lb, nbl, A, pst, npn, sec, false);   // coarse problems are out of scale
                        }
                        const int cnt = min(CM_TAKE, __popcll(mask));
                        int pos = cnt;
                        for (int s = 1; s < 32; s <<= 1) {
                            const int v = __shfl_up_sync(FULL, pos, s);
                            if (lane >= s) pos += v;
                        }
                        total = __shfl_sync(FULL, pos, 31);
                        pos -= cnt;
                        for (int i = 0; i < cnt; i++) {
                            const int bt = __ffsll((long long)mask) - 1;
                            mask &= mask - 1;
                            list[pos + i] = make_int2(64 * sec + bt, lane);
                        }
                    }
                    if (lane == 0) { s_total = total; s_ET = -4000; }
                }
                __syncthreads();
                const int total = s_total;
                if (total < 0) break;
                for (int t = threadIdx.x; t < total; t += 128) {
                    const int2 q = list[t];
                    const int S = s_lb[q.y] + SDC_IDX(2 * pl.near[s_pst[q.y] + (q.x >> 1)] + (q.x & 1), lev_nb(nb0, q.y), f.status);
                    const int e = c.eb[gbx + S];
                    const double gap = fmax(s_lo[q.y] - pl.bhi[gbx + S], pl.blo[gbx + S] - s_hi[q.y]);
                    list[t] = make_int2(S, e);
                    lim[t] = e > -4000 ? e - (ff_exp(gap) - 1023 + fs.kk) : -8000;
                    if (e > -4000) atomicMax(&s_ET, lim[t]);
                }
                __syncthreads();
                const int ET = s_ET;
                int nsum = 0;
                far_src += total * P;
                for (int i = 0; i < total; i += 4) {
                    const int u = i + warp;
                    // else its largest term is below the last digit (the weights alone do not
                    // say so: the distances of one round differ by the spread over the gaps, 2^41)
                    if (u < total && lim[u] - ET >= -62) {
                        const float sc = TRANS ? pow2f(list[u].y - ET) : -pow2f(list[u].y - ET);
                        const ff_f4 *np = pl.npos + (gbx + list[u].x) * P;
                        // nodes 0..15, then 16..21
#pragma unroll
                        for (int kp = 0; kp < 3; kp++) {
                            const bool in = kp < 2 || gc < 3;
                            const int q0 = in ? 2 * gc + 8 * kp : 0;
                            const ff_f4 s0 = np[q0], s1 = np[q0 + 1];
                            unsigned a[2][CM_D];
#pragma unroll
                            for (int h = 0; h < 2; h++) {
                                ff_t3 w = ff_rcp3(ff_diff3(s0, x[h])), v = ff_rcp3(ff_diff3(s1, x[h]));
                                w = {w.a * sc, w.b * sc, w.c * sc};
                                v = {v.a * sc, v.b * sc, v.c * sc};
                                float d0[CM_D], d1[CM_D];
                                cm_cut(w, d0);
                                cm_cut(v, d1);
#pragma unroll
                                for (int s = 0; s < CM_D; s++) a[h][s] = in ? cm_pack(d0[s], d1[s]) : 0u;
                            }
#pragma unroll
                            for (int s = 0; s < CM_D; s++)
                                if (kp < 2) ((uint2 *)&sA[warp].k[0][s][lane])[kp] = make_uint2(a[0][s], a[1][s]);
                                else ((uint2 *)sA[warp].k[1][s])[lane] = make_uint2(a[0][s], a[1][s]);
                        }
                    }
                    boxes_sync();
                    for (int v = grp; v < 4 && i + v < total; v += NS)
                        if (lim[i + v] - ET >= -62) {
                            const int64_t at = (gbx + list[i + v].x) * nt * CM_D * 32;
                            mult16(v, 0, c.wf0 + at);
                            mult8(v, c.wf1 + at);
                        }
                    nsum += NTP;
                    if (nsum + NTP > 5) {                // 110 sources: fold before the sums leave 24 bits
                        nsum = 0;
                        fold();
                    }
                    boxes_sync();
                }
                const double sc = ET > -4000 ? ff_pow2(ET + fs.kk) : 0.0;
                collect(sc, sc);
            }
        }
        // ---- near field
        const int64_t ch0 = cm_chunk(b0, p);
        if (pl.flops && threadIdx.x == 0)
            atomicAdd(pl.flops, (unsigned long long)min(16, tend - t0) * (far_src + (int64_t)nn * B) * (3 + 2 * nc));
        int nsum = 0;
        for (int i = 0; i < nn; i += 4) {
            const int u = i + warp;
            const int kb = u < nn ? SDC_IDX(near_box(pl, gbx + Tb, nnr, u), nb0, f.status) * B : nsrc;
#pragma unroll 1
            for (int half = 0; half < 2; half++) {
                const int k0 = kb + 16 * half;
                if (k0 >= nsrc) break;
#pragma unroll
                for (int kp = 0; kp < 2; kp++) {
                    const int ka = k0 + 2 * gc + 8 * kp, kc = ka + 1;
                    const int64_t ia = b0 + min(ka, nsrc - 1), ib = b0 + min(kc, nsrc - 1);
                    const ff_f4 sa = c.pos[ia], sb = c.pos[ib], fa = c.fac[ia], fb = c.fac[ib];
                    const ff_t3 va = {fa.x, fa.y, fa.z}, vb = {fb.x, fb.y, fb.z};
                    unsigned a[2][CM_D];
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const ff_t3 ta = TRANS ? ff_diff3(sa, x[h]) : ff_diff3(x[h], sa);
                        const ff_t3 tb = TRANS ? ff_diff3(sb, x[h]) : ff_diff3(x[h], sb);
                        ff_t3 w = ff_mul3(va, ff_rcp3(ta)), v = ff_mul3(vb, ff_rcp3(tb));
                        const bool ua = ka < nsrc && (TRANS ? ka != skip[h] : (unsigned)(skip[h] - ka) > 1u);
                        const bool ub = kc < nsrc && (TRANS ? kc != skip[h] : (unsigned)(skip[h] - kc) > 1u);
                        w = {ua ? w.a * rs[h] : 0.0f, ua ? w.b * rs[h] : 0.0f, ua ? w.c * rs[h] : 0.0f};
                        v = {ub ? v.a * rs[h] : 0.0f, ub ? v.b * rs[h] : 0.0f, ub ? v.c * rs[h] : 0.0f};
                        float d0[CM_D], d1[CM_D];
                        cm_cut(w, d0);
                        cm_cut(v, d1);
#pragma unroll
                        for (int s = 0; s < CM_D; s++) a[h][s] = cm_pack(d0[s], d1[s]);
                    }
#pragma unroll
                    for (int s = 0; s < CM_D; s++)
                        ((uint2 *)&sA[warp].k[half][s][lane])[kp] = make_uint2(a[0][s], a[1][s]);
                }
            }
            boxes_sync();
            for (int v = grp; v < 4 && i + v < nn; v += NS) {
                const int kv = SDC_IDX(near_box(pl, gbx + Tb, nnr, i + v), nb0, f.status) * B;
                for (int half = 0; half < 2; half++)
                    if (kv + 16 * half < nsrc)
                        mult16(v, half, c.xf + (ch0 + (kv >> 4) + half) * nt * CM_D * 32);
            }
            nsum += NTP;
            if (nsum + NTP > 4) {                        // 128 sources
                nsum = 0;
                fold();
            }
            boxes_sync();
        }
        collect(ns[0], ns[1]);
        if (grp > 0 || tl >= nt) continue;
        // ---- FP64 terms: lane r < 16 has row r's coefficients
        // (a row of -1: no such term; 0 times another problem's row could be NaN)
        double g0 = 0.0, g1 = 0.0, g2 = 0.0;
        int64_t r0 = -1, r1 = -1, r2 = -1;
        {
            const int r = min(t0 + (lane & 15), tend - 1);
            if (TRANS) {
                const int K = dorg[r] == dk[r] ? r : r + 1;
                g0 = f.vhat[b0 + K] * rcp_nr2((dk[K] - dorg[r]) - eta[r]);
                r0 = b0 + SDC_IDX(f.src[b0 + K], f.off[p + 1] - b0, f.status);
            } else {
                if (r < m - 1) {
                    g0 = f.bnorm[b0 + r] * rcp_nr2((dk[r] - dorg[r]) - eta[r]);
                    r0 = b0 + SDC_IDX(f.pinv[b0 + r], f.off[p + 1] - b0, f.status);
                }
                if (r > 0) {
                    g1 = f.bnorm[b0 + r - 1] * rcp_nr2((dk[r] - dorg[r - 1]) - eta[r - 1]);
                    r1 = b0 + SDC_IDX(f.pinv[b0 + r - 1], f.off[p + 1] - b0, f.status);
                }
                g2 = f.bnorm[b0 + m - 1] * rcp_nr2((dk[r] - dorg[m - 1]) - eta[m - 1]);
                r2 = b0 + SDC_IDX(f.pinv[b0 + m - 1], f.off[p + 1] - b0, f.status);
            }
        }
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int src = gr + 8 * h, r = t0 + src;
            const double u0 = __shfl_sync(FULL, g0, src), u1 = __shfl_sync(FULL, g1, src), u2 = __shfl_sync(FULL, g2, src);
            const int64_t q0 = __shfl_sync(FULL, r0, src), q1 = __shfl_sync(FULL, r1, src), q2 = __shfl_sync(FULL, r2, src);
            if (r >= tend) continue;
            const double sc = TRANS ? f.bnorm[b0 + r] : f.vhat[b0 + r];
            const int64_t row = b0 + SDC_IDX(TRANS ? f.pinv[b0 + r] : f.src[b0 + r], f.off[p + 1] - b0, f.status);
#pragma unroll
            for (int t = 0; t < TPW; t++)
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    const int col = (tl + NTP * t) * 8 + 2 * gc + q;
                    if (col >= nc) continue;
                    const int cm = c.cmax[p * c.ccols + col0 + col];
                    double v = y[t][2 * h + q];
                    v = cm > 30 ? v * ff_pow2(min(cm - 1022, 1023)) * (cm > 2045 ? 2.0 : 1.0) : ldexp(v, cm - 1022);
                    const double *xc = X + (int64_t)(col0 + col) * ldx;
                    if (q0 >= 0) v = fma(u0, xc[q0], v);
                    if (!TRANS) {
                        v = fma(u2, xc[q2], v);
                        if (q1 >= 0) v = fma(u1, xc[q1], v);
                    }
                    Y[row + (int64_t)(col0 + col) * ldy] = sc * v;
                }
        }
    }
}

// What the tiles leave out, at most NC columns per launch: the deflated slots
// (identity part of the factor) and, in FP64, the problems out of the positions'
// scale: a warp per leaf box (32 targets; without a tree every box is near), near
// sources staged, far field from the box's series (far64, figures
// there).  The inner loop runs all NC columns.
template <bool TRANS, int NC>
__global__ void __launch_bounds__(128)
k_cm_rest(FmmDev pl, FactorView f, int64_t total, const int64_t *__restrict__ tile_off, CmDev c,
          const double *__restrict__ X, int64_t ldx, double *__restrict__ Y, int64_t ldy, int col0, int nc)
{
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total * nc;
         x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t slotg = x % total;
        const int64_t col = col0 + x / total;
        if (slotg < f.off[0] || slotg >= f.off[f.nprob]) continue;
        const int64_t p = sdc_upper_index(f.off, f.nprob, slotg);
        const int64_t b0 = f.off[p];
        if ((int)(slotg - b0) < f.mk[p]) continue;
        const int64_t ps = SDC_IDX(f.pinv[slotg], f.off[p + 1] - b0, f.status);
        const int64_t sr = SDC_IDX(f.src[slotg], f.off[p + 1] - b0, f.status);
        if (TRANS) Y[b0 + ps + col * ldy] = X[b0 + sr + col * ldx];
        else       Y[b0 + sr + col * ldy] = X[b0 + ps + col * ldx];
    }
    if (c.bad[f.nprob] == 0) return;
    __shared__ double sd[4][B], se[4][B], sf[4][B], sx[4][NC][B + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t nunit = tile_off[f.nprob] * (CM_TR / B);
    for (int64_t u = (int64_t)blockIdx.x * 4 + warp; u < nunit; u += (int64_t)gridDim.x * 4) {
        const int64_t tile = u / (CM_TR / B);
        const int64_t p = sdc_upper_index(tile_off, f.nprob, tile);
        if (!c.bad[p]) continue;
        const int64_t b0 = f.off[p];
        const int m = f.mk[p];
        const int Tb = (int)(tile - tile_off[p]) * (CM_TR / B) + (int)(u % (CM_TR / B));
        const int tend = TRANS ? m - 1 : m;              // T: the last target is summed by k_cm_last
        if (Tb * B >= tend) continue;
        const bool tree = pl.fslot && pl.fslot[p] >= 0;
        const double *dk = f.dk + b0, *dorg = f.dorg + b0, *eta = f.eta + b0;
        const int nb0 = (m + B - 1) / B, nsrc = TRANS ? m : m - 1;
        const int64_t gx = tree ? pl.box_base[p] + Tb : 0;
        const int nnr = tree ? pl.nnear[gx] : -1;
        const int nn = near_len(nnr, nb0);
        const int r = min(Tb * B + lane, tend - 1);
        const double a0 = TRANS ? dorg[r] : dk[r], a1 = TRANS ? eta[r] : 0.0;
        double acc[NC];
#pragma unroll
        for (int q = 0; q < NC; q++) acc[q] = 0.0;
        if (tree) {
            double cT, hT;
            box_ch(pl.blo[gx], pl.bhi[gx], cT, hT);
            const double v = ((a0 + a1) - cT) * rcp_any(hT);
            const double *cf = c.coef + (pl.leaf_base[p] + Tb) * c.cs * P;
#pragma unroll
            for (int q = 0; q < NC; q++)
                if (q < nc) acc[q] = clenshaw(cf + q * P, v);
        }
        for (int i = 0; i < nn; i++) {
            const int j0 = SDC_IDX(near_box(pl, gx, nnr, i), nb0, f.status) * B, cnt = min(B, nsrc - j0);
            __syncwarp();
            if (lane < cnt) {
                const int j = j0 + lane;
                const int64_t row = b0 + SDC_IDX(TRANS ? f.src[b0 + j] : f.pinv[b0 + j], f.off[p + 1] - b0, f.status);
                sd[warp][lane] = TRANS ? dk[j] : dorg[j];
                se[warp][lane] = TRANS ? 0.0 : eta[j];
                sf[warp][lane] = TRANS ? f.vhat[b0 + j] : f.bnorm[b0 + j];
#pragma unroll
                for (int q = 0; q < NC; q++) sx[warp][q][lane] = (q < nc) ? X[row + (int64_t)(col0 + q) * ldx] : 0.0;
            }
            __syncwarp();
#pragma unroll 2
            for (int jj = 0; jj < cnt; jj++) {
                const double t = TRANS ? (sd[warp][jj] - a0) - a1 : (a0 - sd[warp][jj]) - se[warp][jj];
                const double w = sf[warp][jj] * rcp_nr2(t);      // before x: b_j x_j could underflow
#pragma unroll
                for (int q = 0; q < NC; q++) acc[q] = fma(sx[warp][q][jj], w, acc[q]);
            }
        }
        if (!TRANS) {                                    // the last eigenvalue, outside the tree
            const double w = f.bnorm[b0 + m - 1] * rcp_nr2((a0 - dorg[m - 1]) - eta[m - 1]);
            const int64_t row = b0 + SDC_IDX(f.pinv[b0 + m - 1], f.off[p + 1] - b0, f.status);
#pragma unroll
            for (int q = 0; q < NC; q++)
                if (q < nc) acc[q] = fma(w, X[row + (int64_t)(col0 + q) * ldx], acc[q]);
        }
        if (Tb * B + lane < tend) {
            const int64_t row = b0 + SDC_IDX(TRANS ? f.pinv[b0 + r] : f.src[b0 + r], f.off[p + 1] - b0, f.status);
            const double sc = TRANS ? f.bnorm[b0 + r] : f.vhat[b0 + r];
#pragma unroll
            for (int q = 0; q < NC; q++)
                if (q < nc) Y[row + (int64_t)(col0 + q) * ldy] = sc * acc[q];
        }
    }
}

template <int NC>
void launch_rest(bool trans, const FmmDev &dv, const FactorView &f, int64_t total, const int64_t *tile_off,
                 const CmDev &c, const double *X, int64_t ldx, double *Y, int64_t ldy, int col0, int nc, unsigned g,
                 cudaStream_t st)
{
    if (trans) k_cm_rest<true, NC><<<g, 128, 0, st>>>(dv, f, total, tile_off, c, X, ldx, Y, ldy, col0, nc);
    else k_cm_rest<false, NC><<<g, 128, 0, st>>>(dv, f, total, tile_off, c, X, ldx, Y, ldy, col0, nc);
}

// Row of the last eigenvalue of Qhat^T X: the sources of one tile of 64, FP64
__global__ void __launch_bounds__(64)
k_cm_last(FactorView f, const int64_t *__restrict__ tile_off, CmDev c, const double *__restrict__ X, int64_t ldx,
          int col0, int nc)
{
    __shared__ double w[CM_TR];
    __shared__ int64_t row[CM_TR];
    const int64_t ntiles = tile_off[f.nprob];
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t p = sdc_upper_index(tile_off, f.nprob, tile);
        const int64_t b0 = f.off[p];
        const int m = f.mk[p], i = (int)(tile - tile_off[p]) * CM_TR + threadIdx.x;
        __syncthreads();
        w[threadIdx.x] = 0.0;
        row[threadIdx.x] = 0;
        if (i < m) {
            w[threadIdx.x] = f.vhat[b0 + i] * rcp_nr2((f.dk[b0 + i] - f.dorg[b0 + m - 1]) - f.eta[b0 + m - 1]);
            row[threadIdx.x] = b0 + SDC_IDX(f.src[b0 + i], f.off[p + 1] - b0, f.status);
        }
        __syncthreads();
        for (int q = threadIdx.x; q < nc; q += CM_TR) {
            double s = 0.0;
            for (int k = 0; k < CM_TR; k++)
                if (w[k] != 0.0) s = fma(w[k], X[row[k] + (int64_t)(col0 + q) * ldx], s);
            c.lastp[tile * (CM_NT * 8) + q] = s;
        }
    }
}

__global__ void __launch_bounds__(128)
k_cm_lastsum(FactorView f, const int64_t *__restrict__ tile_off, CmDev c, double *__restrict__ Y, int64_t ldy, int col0,
             int nc)
{
    const int lane = threadIdx.x & 31;
    for (int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < f.nprob * nc;
         u += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int64_t p = u / nc, b0 = f.off[p];
        const int q = (int)(u % nc), m = f.mk[p];
        if (m < 1) continue;
        double a = 0.0;
        for (int64_t t = tile_off[p] + lane; t < tile_off[p + 1]; t += 32) a += c.lastp[t * (CM_NT * 8) + q];
        for (int sh = 16; sh > 0; sh >>= 1) a += __shfl_xor_sync(0xffffffffu, a, sh);
        if (lane == 0)
            Y[b0 + SDC_IDX(f.pinv[b0 + m - 1], f.off[p + 1] - b0, f.status) + (int64_t)(col0 + q) * ldy] =
                f.bnorm[b0 + m - 1] * a;
    }
}

unsigned fmm_grid() { return (unsigned)(sdc_num_sms() * 8); }
// zhat and b: CTAs of one or two warps whose chains of FP32 operations wait on
// their own latency; 32 warps per SM
unsigned near_grid() { return (unsigned)(sdc_num_sms() * (1024 / B)); }

// As many CTAs of kernel K as the GPU holds at once (threads per CTA, static
// shared memory only), from the occupancy calculator, once per device: the
// grid of kernels whose CTAs take equal shares of the work (a second, partial
// wave would double the launch).
template <auto K>
unsigned resident_grid(int threads)
{
    static std::mutex mu;
    static int per_sm[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return (unsigned)sdc_num_sms();
    std::lock_guard<std::mutex> lk(mu);
    if (per_sm[dev] == 0) {
        int v = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, K, threads, 0) != cudaSuccess) v = 1;
        per_sm[dev] = v > 0 ? v : 1;
    }
    return (unsigned)(sdc_num_sms() * per_sm[dev]);
}

template <int MODE>
unsigned up_grid() { return resident_grid<k_fmm_up<MODE>>(up_threads<MODE>()); }

// one warp per FMM problem of k_fmm_lastsum, 4 warps per CTA
unsigned lastsum_grid(const FmmPlan &pl)
{
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((pl.cap_f + 3) / 4, (int64_t)sdc_num_sms() * 8));
}

SrcArgs src_from_r1(const int64_t *off, const R1Out &o)
{
    SrcArgs a{};
    a.off = off; a.mk = o.mk; a.dk = o.dk; a.zk = o.zk; a.vhat = o.vhat; a.bnorm = o.bnorm;
    a.dorg = o.dorg; a.eta = o.eta; a.src = o.src; a.pinv = o.pinv; a.wsum = o.wsum;
#ifdef SUPERDC_CHECK
    a.status = o.status;
#endif
    return a;
}

// Levels of far64's subtrees: of 8 leaf boxes where that leaves four subtrees to an SM
// (their lists differ in length), of 4 where it leaves one; the columns' in two halves
// where there are few.  GB300, applications of 19 columns to 124000 rows, of 64 to
// 20000, poles graded: 8 boxes 36.3 and 13.8 ms, 4 boxes 29.9 and 9.0, 2 boxes 30 and 10.7
int far64_sub(const FmmPlan &pl)
{
    const int64_t nsm = sdc_num_sms();
    return (pl.cap_leaves >> 3) >= 4 * nsm ? 3 : (pl.cap_leaves >> 2) >= nsm ? 2 : 1;
}

// far fields of the columns of the problems with only[p] != 0
template <int KER>
void launch_far64(const FmmPlan &pl, const int32_t *mk, const int32_t *only, int nw, double *coef, int nfield,
                  int32_t *word, cudaStream_t st)
{
    const int sub = far64_sub(pl);
    const int64_t units = (pl.cap_leaves >> sub) + 1;
    const unsigned g = (unsigned)std::min<int64_t>(units, resident_grid<k_fmm_far64<KER>>(far_threads<KER>()));
    const dim3 grid(g, nw > 8 && units < 2 * (int64_t)sdc_num_sms() ? 2 : 1);
    PROF_LAUNCH("fmm_far", st, k_fmm_far64<KER><<<grid, far_threads<KER>(), 0, st>>>(pl.dv, mk, only, nw, sub, coef, nfield, word));
}

// far field of a one-column sum: node weights, then every leaf's series
template <int MODE, int KER>
superdc_status far_field(const FmmPlan &pl, const int64_t *off, const R1Out &o, cudaStream_t st)
{
    const FmmDev &dv = pl.dv;
    SrcArgs a = src_from_r1(off, o);
    a.only = dv.ffbad;
    const unsigned gu = (unsigned)std::min<int64_t>((pl.cap_leaves + 3) / 4, resident_grid<k_fmm_up1<MODE>>(128));
    PROF_LAUNCH("fmm_up", st, k_fmm_up1<MODE><<<gu, 128, 0, st>>>(dv, a));
    PROF_LAUNCH("fmm_up", st, k_fmm_up<MODE><<<up_grid<MODE>(), up_threads<MODE>(), 0, st>>>(dv, a));
    const int sub = far64_sub(pl);               // (a CTA per subtree of far64, should one be out of scale)
    const int64_t want = std::max((pl.cap_leaves + FAR_NW - 1) / FAR_NW, (pl.cap_leaves >> sub) + 1);
    const unsigned g = (unsigned)std::min<int64_t>(want, resident_grid<k_fmm_far<KER>>(FAR_NW * 32));
    PROF_LAUNCH("fmm_far", st, k_fmm_far<KER><<<g, FAR_NW * 32, 0, st>>>(dv, off, o, sub));
    return SUPERDC_OK;
}

void launch_up(bool trans, const FmmDev &dv, const FactorView &f, const CmDev &c, int col0, int nc, int nt,
               cudaStream_t st)
{
    auto run = [&](auto K, unsigned g) { K<<<g, 128, 0, st>>>(dv, f, c, col0, nc, nt); };
    if (nt <= 3) {
        if (trans) run(k_cm_up<3, true>, resident_grid<k_cm_up<3, true>>(128));
        else run(k_cm_up<3, false>, resident_grid<k_cm_up<3, false>>(128));
    } else {
        if (trans) run(k_cm_up<CM_NT, true>, resident_grid<k_cm_up<CM_NT, true>>(128));
        else run(k_cm_up<CM_NT, false>, resident_grid<k_cm_up<CM_NT, false>>(128));
    }
}

template <int NTP, int TPW>
void launch_apply(bool trans, const FmmDev &dv, const FactorView &f, const int64_t *tile_off, const CmDev &c,
                  const double *X, int64_t ldx, double *Y, int64_t ldy, int col0, int nc, int nt, int64_t tiles,
                  cudaStream_t st)
{
    // four CTAs per tile of 64 rows; problems differ in size, so the CTAs are scheduled and not persistent
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>(4 * tiles, 1 << 20));
    if (trans) k_cm_apply<NTP, TPW, true><<<g, 128, 0, st>>>(dv, f, tile_off, c, X, ldx, Y, ldy, col0, nc, nt);
    else k_cm_apply<NTP, TPW, false><<<g, 128, 0, st>>>(dv, f, tile_off, c, X, ldx, Y, ldy, col0, nc, nt);
}

}  // namespace


superdc_status fmm_plan(FmmPlan &pl, int64_t nprob, const int64_t *off, int64_t total, int64_t max_m,
                        const int32_t *mk, const double *dk, int min_m, int ncol, int32_t *used, bool step,
                    cudaStream_t st)
{
    pl = FmmPlan();
    pl.total = total;
    if (nprob <= 0) return SUPERDC_OK;
    if (used) SDC_CHECK(cudaMemsetAsync(used, 0, (size_t)nprob * sizeof(int32_t), st));
    if (min_m <= 0) return SUPERDC_OK;
    const int64_t mm = (max_m >= 0) ? std::min(max_m, total) : total;
    const int eff = std::max(min_m, 4 * B);
    if (mm < eff) return SUPERDC_OK;
    const int64_t nf_cap = std::min<int64_t>(nprob, total / eff + 1);
    pl.cap_f = nf_cap;
    pl.cap_leaves = total / B + nf_cap + 1;
    pl.cap_boxes = 2 * pl.cap_leaves + nf_cap * 40;
    ncol = std::max(1, std::min(ncol, WMAX));
    FmmDev &d = pl.dv;
    d.nprob = nprob;
    d.ncol = ncol;
    auto al = [&](auto **ptr, size_t cnt) -> cudaError_t {
        cudaError_t e = sdc_alloc(ptr, cnt, st);
        if (e == cudaSuccess) pl.bufs.push_back((void *)*ptr);
        return e;
    };
    int64_t *box_base, *leaf_base;
    int32_t *fslot, *fprob, *nfmm, *nnear, *near;
    int64_t *nstart;
    double *blo, *bhi;
    SDC_CHECK(al(&box_base, nprob + 1));
    SDC_CHECK(al(&leaf_base, nprob + 1));
    SDC_CHECK(al(&fslot, nprob));
    SDC_CHECK(al(&fprob, nf_cap));
    SDC_CHECK(al(&nfmm, 1));
    SDC_CHECK(al(&blo, pl.cap_boxes));
    SDC_CHECK(al(&bhi, pl.cap_boxes));
    SDC_CHECK(al(&nnear, pl.cap_boxes));
    SDC_CHECK(al(&near, pl.cap_boxes * FMM_NPOOL));
    SDC_CHECK(al(&nstart, pl.cap_boxes));
    SDC_CHECK(al(&d.W, (size_t)pl.cap_boxes * P * ncol));
    SDC_CHECK(al(&d.npos, (size_t)pl.cap_boxes * P));
    SDC_CHECK(al(&d.amask, (size_t)pl.cap_boxes));
    SDC_CHECK(al(&d.ibox, (size_t)pl.cap_boxes));
    SDC_CHECK(al(&d.coarse, (size_t)nprob));
    if (step) {
        SDC_CHECK(al(&d.coef, (size_t)pl.cap_leaves * NFIELD * P));
        SDC_CHECK(al(&d.lastp, (size_t)pl.cap_leaves));
        SDC_CHECK(al(&d.tail, (size_t)std::max<int64_t>(1, total)));
        SDC_CHECK(al(&d.ntail, 2));
        SDC_CHECK(cudaMemsetAsync(d.ntail, 0, 2 * sizeof(unsigned int), st));
        SDC_CHECK(al(&d.nwt, (size_t)pl.cap_boxes * P));
        SDC_CHECK(al(&d.ffbad, nprob + 1));
    }
    SDC_CHECK(al(&d.upcnt, pl.cap_boxes));
    SDC_CHECK(cudaMemsetAsync(d.upcnt, 0, (size_t)pl.cap_boxes * sizeof(int32_t), st));
    SDC_CHECK(al(&d.upq, 2));
    SDC_CHECK(al(&d.split, pl.cap_leaves));
    SDC_CHECK(al(&d.nsplit, 1));
    SDC_CHECK(cudaMemsetAsync(d.upq, 0, 2 * sizeof(unsigned long long), st));
    d.cap_f = nf_cap;

    d.flops = prof_counter("fmm_flops");
    d.box_base = box_base; d.leaf_base = leaf_base; d.fslot = fslot; d.fprob = fprob; d.nfmm = nfmm;
    d.blo = blo; d.bhi = bhi; d.nnear = nnear; d.near = near; d.nstart = nstart;
    PROF_LAUNCH("fmm_plan", st, k_fmm_plan<<<1, tiles_threads(nprob), 0, st>>>(nprob, mk, min_m, pl.cap_boxes, pl.cap_leaves,
                                                               pl.cap_f, box_base, leaf_base, fslot, fprob, nfmm));
    // one CTA per problem; a batch of fewer problems than SMs (the top tree
    // levels) gives each tree 1024 threads instead of 256
    const unsigned gt = (unsigned)std::min<int64_t>(nprob, (int64_t)sdc_num_sms() * 4);
    const int tt = (nprob < sdc_num_sms()) ? 1024 : 256;
    SDC_CHECK(cudaMemsetAsync(d.nsplit, 0, sizeof(int32_t), st));
    PROF_LAUNCH("fmm_tree", st, k_fmm_tree<<<gt, tt, 0, st>>>(d, off, mk, dk, blo, bhi, nnear, nstart, near, used));
    {
        auto gr = [&](int64_t n) {
            return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)sdc_num_sms() * 8));
        };
        PROF_LAUNCH("fmm_plan", st, k_fmm_nodes<<<gr(pl.cap_boxes * P), 256, 0, st>>>(d, off, mk, dk));
    }
    SDC_CHECK(cudaGetLastError());
    pl.on = true;
    return SUPERDC_OK;
}

void fmm_free(FmmPlan &pl, cudaStream_t st)
{
    for (void *p : pl.bufs) cudaFreeAsync(p, st);
    pl.bufs.clear();
    pl.on = false;
}

superdc_status fmm_secular(const FmmPlan &pl, const int64_t *off, const R1Out &o, double stop_c, int max_iter,
                           cudaStream_t st)
{
    if (!pl.on) return SUPERDC_OK;
    const unsigned gl = (unsigned)std::max<int64_t>(1, std::min<int64_t>(pl.cap_f, (int64_t)sdc_num_sms() * 2));
    ff_f4 *fd = nullptr;
    ff_f2 *fw = nullptr;
    SdcScratch sc(st);
    SDC_CHECK(sc.get(&fd, (size_t)pl.total));
    SDC_CHECK(sc.get(&fw, (size_t)pl.total));
    SDC_CHECK(cudaMemsetAsync(pl.dv.ffbad, 0, (size_t)(pl.dv.nprob + 1) * sizeof(int32_t), st));
    const unsigned gp = (unsigned)std::max<int64_t>(1, std::min<int64_t>((pl.total + 255) / 256,
                                                                         (int64_t)sdc_num_sms() * 8));
    PROF_LAUNCH("fmm_secular", st, k_ff_prep<<<gp, 256, 0, st>>>(pl.dv.nprob, off, pl.total, pl.dv.fslot, o, stop_c, fd, fw,
                                                                 pl.dv.ffbad));
    const FfDev ff = {fd, fw};
    far_field<M_SEC, K_SEC>(pl, off, o, st);
    unsigned long long *terms = prof_counter("fmm_secular_terms");
    unsigned long long *lterms = prof_counter("fmm_secular_last_terms");
    PROF_LAUNCH("fmm_secular_last", st, k_secular_last<<<gl, SL_T, 0, st>>>(pl.dv, off, o, stop_c, max_iter,
                                                                             lterms));
    PROF_LAUNCH("fmm_secular", st, k_secular_fmm<<<fmm_grid(), 64, 0, st>>>(pl.dv, ff, off, o, stop_c, max_iter,
                                                                             terms));
    PROF_LAUNCH("fmm_secular", st, k_secular_tail<<<(unsigned)(sdc_num_sms() * 4), 128, 0, st>>>(
                                       pl.dv, ff, off, o, stop_c, max_iter, terms));
    PROF_LAUNCH("fmm_secular", st, (k_secular_fmm_split<8><<<fmm_grid(), 256, 0, st>>>(pl.dv, ff, off, o, stop_c,
                                                                                      max_iter, terms)));
    SDC_CHECK(cudaGetLastError());
    return SUPERDC_OK;
}

superdc_status fmm_lowner(const FmmPlan &pl, const int64_t *off, const R1Out &o, cudaStream_t st)
{
    if (!pl.on) return SUPERDC_OK;
    far_field<M_LOW, K_LOG>(pl, off, o, st);
    PROF_LAUNCH("fmm_lowner", st, k_lowner_fmm<<<near_grid(), B, 0, st>>>(pl.dv, off, o));
    SDC_CHECK(cudaGetLastError());
    return SUPERDC_OK;
}

superdc_status fmm_bnorm(const FmmPlan &pl, const int64_t *off, const R1Out &o, cudaStream_t st)
{
    if (!pl.on) return SUPERDC_OK;
    far_field<M_BN, K_2>(pl, off, o, st);
    PROF_LAUNCH("fmm_bnorm", st, k_bnorm_fmm<<<near_grid(), B, 0, st>>>(pl.dv, off, o));
    PROF_LAUNCH("fmm_bnorm", st, k_fmm_lastsum<<<lastsum_grid(pl), 128, 0, st>>>(pl.dv, off, o.mk, o.bnorm));
    SDC_CHECK(cudaGetLastError());
    return SUPERDC_OK;
}

superdc_status fmm_columns(const FmmPlan &pl, const FactorView &f, int64_t total, const int64_t *tile_off,
                       const double *X, int64_t ldx, double *Y, int64_t ldy, int ncols, bool trans, cudaStream_t st)
{
    const int ntmax = std::min(CM_NT, (ncols + 7) / 8);
    const int64_t chunks = total / 16 + f.nprob + 1, tiles = total / CM_TR + f.nprob + 1;
    SdcScratch sc(st);
    CmDev c{};
    c.ccols = ncols;
    SDC_CHECK(sc.get(&c.pos, (size_t)total));
    SDC_CHECK(sc.get(&c.fac, (size_t)total));
    const size_t nflag = (size_t)f.nprob + 1 + (size_t)f.nprob * ncols;
    SDC_CHECK(sc.get(&c.bad, nflag));
    c.cmax = c.bad + f.nprob + 1;
    SDC_CHECK(sc.get(&c.xf, (size_t)chunks * ntmax * CM_D * 32));
    if (trans) SDC_CHECK(sc.get(&c.lastp, (size_t)tiles * CM_NT * 8));
    if (pl.on) {
        SDC_CHECK(sc.get(&c.wf0, (size_t)pl.cap_boxes * ntmax * CM_D * 32));
        SDC_CHECK(sc.get(&c.wf1, (size_t)pl.cap_boxes * ntmax * CM_D * 32));
        SDC_CHECK(sc.get(&c.eb, (size_t)pl.cap_boxes));
        // the digits are read for the last time before the FP64 loops write their series:
        // cs columns of P doubles in the digits' place of a box
        c.coef = (double *)c.wf0;
        c.cs = CM_D * 32 / P * ntmax;
        static_assert(CM_D * 32 / P >= 8 && sizeof(uint2) == sizeof(double), "a tile's series fit its digits");
    }
    SDC_CHECK(cudaMemsetAsync(c.bad, 0, nflag * sizeof(int32_t), st));
    auto gr = [&](int64_t n) {
        return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)sdc_num_sms() * 8));
    };
    const int64_t rows = chunks * 16;
    if (trans) PROF_LAUNCH("cauchy", st, k_cm_prep<true><<<gr(total * ncols), 256, 0, st>>>(f, total, X, ldx, ncols, c));
    else PROF_LAUNCH("cauchy", st, k_cm_prep<false><<<gr(total * ncols), 256, 0, st>>>(f, total, X, ldx, ncols, c));
    FmmDev dv = pl.dv;
    if (!pl.on) dv = FmmDev{};
    int32_t *word = nullptr;                             // of the index guards (checked build)
#ifdef SUPERDC_CHECK
    word = f.status;
#endif
    for (int c0 = 0; c0 < ncols; c0 += CM_NT * 8) {
        const int nc = std::min(CM_NT * 8, ncols - c0), nt = (nc + 7) / 8;
        if (trans) PROF_LAUNCH("cauchy", st, k_cm_slice<true><<<gr(rows * nt * 8), 256, 0, st>>>(f, rows, X, ldx, c0, nc, nt, c));
        else PROF_LAUNCH("cauchy", st, k_cm_slice<false><<<gr(rows * nt * 8), 256, 0, st>>>(f, rows, X, ldx, c0, nc, nt, c));
        if (pl.on) PROF_LAUNCH("fmm_up", st, launch_up(trans, dv, f, c, c0, nc, nt, st));
        auto fn = (nt == 1) ? launch_apply<1, 1> : (nt == 2) ? launch_apply<2, 1> : (nt <= 4) ? launch_apply<4, 1>
                                                                                              : launch_apply<4, 2>;
        PROF_LAUNCH("cauchy", st, fn(trans, dv, f, tile_off, c, X, ldx, Y, ldy, c0, nc, nt, tiles, st));
        if (trans) {
            PROF_LAUNCH("cauchy", st, k_cm_last<<<(unsigned)std::min<int64_t>(tiles, (int64_t)sdc_num_sms() * 16), 64, 0,
                                                 st>>>(f, tile_off, c, X, ldx, c0, nc));
            PROF_LAUNCH("cauchy", st, k_cm_lastsum<<<gr(f.nprob * nc * 32), 128, 0, st>>>(f, tile_off, c, Y, ldy, c0, nc));
        }
    }
    for (int c0 = 0; c0 < ncols; c0 += CM_BC) {
        const int nc = std::min(CM_BC, ncols - c0);
        if (pl.on) {
            // node weights in FP64 of the problems out of scale (nothing to do as a rule)
            SrcArgs a{};
            a.off = f.off; a.mk = f.mk; a.dk = f.dk; a.vhat = f.vhat; a.bnorm = f.bnorm; a.dorg = f.dorg; a.eta = f.eta;
            a.src = f.src; a.pinv = f.pinv; a.X = X; a.ldx = ldx; a.col0 = c0; a.nc = nc; a.only = c.bad;
#ifdef SUPERDC_CHECK
            a.status = word;
#endif
            if (trans) PROF_LAUNCH("fmm_up", st, k_fmm_up<M_CT><<<up_grid<M_CT>(), up_threads<M_CT>(), 0, st>>>(dv, a));
            else PROF_LAUNCH("fmm_up", st, k_fmm_up<M_CN><<<up_grid<M_CN>(), up_threads<M_CN>(), 0, st>>>(dv, a));
            if (trans) launch_far64<K_1>(pl, f.mk, c.bad, nc, c.coef, c.cs, word, st);
            else launch_far64<K_1N>(pl, f.mk, c.bad, nc, c.coef, c.cs, word, st);
        }
        auto fn = nc <= 2 ? launch_rest<2> : nc <= 4 ? launch_rest<4> : nc <= 8 ? launch_rest<8> : nc <= 12 ? launch_rest<12>
                : nc <= 16 ? launch_rest<16> : nc <= 20 ? launch_rest<20> : nc <= 24 ? launch_rest<24> : launch_rest<CM_BC>;
        PROF_LAUNCH("deflcopy", st, fn(trans, dv, f, total, tile_off, c, X, ldx, Y, ldy, c0, nc, gr(total * nc), st));
    }
    SDC_CHECK(cudaGetLastError());
    return SUPERDC_OK;
}
