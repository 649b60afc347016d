// Adjoint of the batched rank-one step (reverse mode through the secular roots).
//
// Forward, per problem: M = diag(d) + rho z z^T  ->  new eigenvalues lambda
// (sorted) and, for caller columns X, Y = Qhat^T X with
// Qhat = G^T [C (+) I] Pi^T (rotations G, Cauchy-like block C of eq. (4.26)
// on the kept set, identity on the deflated set, sort Pi).
// Given cotangents lambda_bar (merged order) and Ybar, this computes
// d_bar, z_bar (input order) and X_bar = Qhat Ybar.
//
// Kept block (implicit-function theorem on the secular equation, i.e. the
// eigen-adjoint of M_k = diag(d_k) + z_k z_k^T = C Lambda C^T):
//   Mbar = C E C^T,  E = diag(lambda_bar) + sym(F o (Y Ybar^T)),
//   F_kl = 1/(lambda_l - lambda_k) (k != l);  d_bar = diag(Mbar), z_bar = 2 Mbar z.
// With C^T z = -b (Loewner's zhat makes sum_i zhat_i^2/(d_i - lambda_k) = -1),
//   u_k = -lambda_bar_k b_k - 1/2 sum_c (y_kc P_kc - ybar_kc R_kc),
//   P_kc = sum_{l!=k} b_l ybar_lc/(lambda_l - lambda_k), R_kc = sum_{l!=k} b_l y_lc/(lambda_l - lambda_k),
//   z_bar_i = 2 (C u)_i = 2 vhat_i sum_k b_k u_k / (d_i - lambda_k),
// and, by partial fractions 1/((d-l_k)(d-l_l)) = [1/(d-l_k) - 1/(d-l_l)]/(l_k - l_l),
//   d_bar_i = vhat_i^2 sum_k [h_k/(d_i - lambda_k)^2 + g_k/(d_i - lambda_k)],
//   h_k = b_k^2 lambda_bar_k,  g_k = sum_c (beta_kc Delta_kc - alpha_kc Gamma_kc),
//   alpha_kc = b_k y_kc, beta_kc = b_k ybar_kc,
//   Gamma_kc = sum_{l!=k} beta_lc/(lambda_k - lambda_l)^2, Delta_kc = sum_{l!=k} alpha_lc/(lambda_k - lambda_l)^2.
// Every difference is taken in shifted form: d_i - lambda_k = (d_i - d_{K_k}) - eta_k
// (eq. (4.28)) and lambda_k - lambda_l = (d_{K_k} - d_{K_l}) + (eta_k - eta_l).
// Deflation: the rotations are treated as fixed linear maps (their dependence
// on z is of the order of tau); deflated eigenvalues are the rotated poles.
// Eigenvalue pairs with |lambda_k - lambda_l| <= 1e-10 max(|lambda_k|, |lambda_l|)
// are treated as one eigenspace (no coupling term): eigenvector losses are not
// differentiable there, and losses invariant within the eigenspace are exact.
#include <algorithm>
#include <cuda_runtime.h>
#include "common.cuh"
#include "cauchy.cuh"
#include "fmm.cuh"
#include "prof.cuh"
#include "tiles.cuh"
#include "secular.cuh"

namespace {

constexpr int BW_C = 8;      // columns per pass of the lambda-lambda kernel
constexpr int BW_T = 32;     // targets per CTA (one per lane)
constexpr int BW_W = 8;      // warps per CTA; they split the sources
constexpr int BW_S = 32;     // sources staged per warp

// pinv from perm, d_K from org (inputs are the public forward outputs)
__global__ void k_prep(int64_t nprob, const int64_t *__restrict__ off, int64_t total, const int32_t *__restrict__ mk,
                       const int32_t *__restrict__ perm, const int32_t *__restrict__ org, const double *__restrict__ dk,
                       int32_t *__restrict__ pinv, double *__restrict__ dorg)
{
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total; x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = sdc_upper_index(off, nprob, x);
        const int64_t b0 = off[p];
        const int pos = (int)(x - b0);
        pinv[b0 + perm[x]] = pos;
        const int s = (int)(x - b0);
        dorg[x] = (s < mk[p]) ? dk[b0 + org[x]] : dk[x];
    }
}

// Per kept root k, columns [c0, c0 + nc): u_k and g_k from the four sums P, R,
// Gamma, Delta of every column, each added up in the order of the sources.  (One
// factor per pair, s_kl = sum_c (ybar_kc alpha_lc - y_kc beta_lc), takes half of
// the operations and cancels before it divides, but its g differs from these sums
// by their own rounding, up to 1e-9 of the result at close pairs.)
// A CTA takes 32 targets: its eight warps form the reciprocals of 32 sources at a
// time, then every warp carries one or two sums pairs (P, Gamma or R, Delta of a
// column) through them, so a pair costs 10 + 4 nc FP64 operations, a chain 2 or 4
// per source, and every column count pays for its own columns only (a thread
// with all sums of 8 columns, 128 targets per CTA, left most SMs idle below 20000
// rows).  Measured (GB300, n = 4096 tree adjoint, 7 columns on average, 36 steps):
// 104.7 -> 17.8 ms; k_bw_dz 19.3 -> 3.5 ms.
template <int NU>                       // sum pairs per warp
__global__ void __launch_bounds__(BW_W * 32)
k_bw_lamlam(int64_t nprob, const int64_t *__restrict__ off, const int64_t *__restrict__ tile_off,
            const int32_t *__restrict__ mk, const double *__restrict__ dorg, const double *__restrict__ eta,
            const double *__restrict__ bnorm, const int32_t *__restrict__ pinv,
            const double *__restrict__ Y, int64_t ld, const double *__restrict__ Ybar, int64_t ldb, int c0, int nc,
            double *__restrict__ u, double *__restrict__ g)
{
    __shared__ double sK[BW_S], sE[BW_S], sV[2 * BW_C][BW_S], sR[2][BW_S][BW_T];
    __shared__ double red[2][2 * BW_C][BW_T];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t ntiles = tile_off[nprob];
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t p = sdc_upper_index(tile_off, nprob, tile);
        const int64_t b0 = off[p];
        const int m = mk[p];
        const int k = (int)(tile - tile_off[p]) * BW_T + lane;
        const bool act = k < m;
        const double dKk = act ? dorg[b0 + k] : 0.0, ek = act ? eta[b0 + k] : 0.0;
        // exponent of the largest |lambda|: differences above 2^-32 of it are not degenerate
        const double lmax = fmax(fabs(dorg[b0] + eta[b0]), fabs(dorg[b0 + m - 1] + eta[b0 + m - 1]));
        const int emin = ((__double2hiint(lmax) >> 20) & 0x7FF) + 1 - 32;
        double s1[NU], s2[NU];
#pragma unroll
        for (int i = 0; i < NU; i++) s1[i] = s2[i] = 0.0;
        for (int l0 = 0; l0 < m; l0 += BW_S) {
            const int cn = min(BW_S, m - l0);
            __syncthreads();
            if (lane < cn) {
                const int64_t s = b0 + l0 + lane;
                const double bl = bnorm[s];
                const int64_t row = b0 + pinv[s];
                if (warp == 0) { sK[lane] = dorg[s]; sE[lane] = eta[s]; }
                for (int c = warp; c < nc; c += BW_W) {
                    sV[2 * c][lane] = bl * Ybar[row + ldb * (c0 + c)];
                    sV[2 * c + 1][lane] = bl * Y[row + ld * (c0 + c)];
                }
            }
            __syncthreads();
#pragma unroll
            for (int i = 0; i < BW_S / BW_W; i++) {
                const int ll = warp * (BW_S / BW_W) + i;
                if (ll >= cn) break;
                const double dl = (dKk - sK[ll]) + (ek - sE[ll]);     // lambda_k - lambda_l
                bool use = l0 + ll != k;
                // numerically degenerate pairs form one eigenspace: no coupling
                if (((__double2hiint(dl) >> 20) & 0x7FF) < emin)
                    use = use && fabs(dl) > 1e-10 * fmax(fabs(dKk + ek), fabs(sK[ll] + sE[ll]));
                const double r = use ? rcp_rn(dl) : 0.0;
                sR[0][ll][lane] = r;
                sR[1][ll][lane] = r * r;
            }
            __syncthreads();
#pragma unroll
            for (int i = 0; i < NU; i++) {
                const int q = warp + BW_W * i;
                if (q >= 2 * nc) break;
                double a = s1[i], b = s2[i];
#pragma unroll 4
                for (int ll = 0; ll < cn; ll++) {
                    const double v = sV[q][ll];
                    a = fma(-v, sR[0][ll][lane], a);     // sum beta_l/(lambda_l - lambda_k), or of alpha_l
                    b = fma(v, sR[1][ll][lane], b);
                }
                s1[i] = a;
                s2[i] = b;
            }
        }
#pragma unroll
        for (int i = 0; i < NU; i++)
            if (warp + BW_W * i < 2 * nc) {
                red[0][warp + BW_W * i][lane] = s1[i];
                red[1][warp + BW_W * i][lane] = s2[i];
            }
        __syncthreads();
        if (warp == 0 && act) {
            const double bk = bnorm[b0 + k];
            const int64_t row = b0 + pinv[b0 + k];
            double uu = 0.0, gg = 0.0;
            for (int c = 0; c < nc; c++) {
                const double y = Y[row + ld * (c0 + c)], yb = Ybar[row + ldb * (c0 + c)];
                uu += -0.5 * (y * red[0][2 * c][lane] - yb * red[0][2 * c + 1][lane]);
                gg += (bk * yb) * red[1][2 * c + 1][lane] - (bk * y) * red[1][2 * c][lane];
            }
            u[b0 + k] += uu;
            g[b0 + k] += gg;
        }
    }
}

// d_bar_i, z_bar_i of the kept rows; targets and warps as above
__global__ void __launch_bounds__(BW_W * 32)
k_bw_dz(int64_t nprob, const int64_t *__restrict__ off, const int64_t *__restrict__ tile_off,
        const int32_t *__restrict__ mk, const double *__restrict__ dk, const double *__restrict__ dorg,
        const double *__restrict__ eta, const double *__restrict__ vhat, const double *__restrict__ bnorm,
        const int32_t *__restrict__ pinv, const double *__restrict__ lam_bar, const double *__restrict__ u,
        const double *__restrict__ g, double *__restrict__ dbar_s, double *__restrict__ zbar_s)
{
    __shared__ double sK[BW_W][BW_S], sE[BW_W][BW_S], sH[BW_W][BW_S], sG[BW_W][BW_S], sU[BW_W][BW_S];
    __shared__ double red[2][BW_W][BW_T];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t ntiles = tile_off[nprob];
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t p = sdc_upper_index(tile_off, nprob, tile);
        const int64_t b0 = off[p];
        const int m = mk[p];
        const int i = (int)(tile - tile_off[p]) * BW_T + lane;
        const bool act = i < m;
        const double di = act ? dk[b0 + i] : 0.0;
        double a1 = 0.0, a2 = 0.0;
        for (int k0 = warp * BW_S; k0 < m; k0 += BW_W * BW_S) {
            const int cn = min(BW_S, m - k0);
            __syncwarp();
            if (lane < cn) {
                const int64_t s = b0 + k0 + lane;
                const double bk = bnorm[s];
                const double lb = lam_bar ? lam_bar[b0 + pinv[s]] : 0.0;
                sK[warp][lane] = dorg[s];
                sE[warp][lane] = eta[s];
                sH[warp][lane] = bk * bk * lb;
                sG[warp][lane] = g[s];
                sU[warp][lane] = bk * (u[s] - lb * bk);
            }
            __syncwarp();
            if (act) {
#pragma unroll 2
                for (int kk = 0; kk < cn; kk++) {
                    const double r = rcp_nr2((di - sK[warp][kk]) - sE[warp][kk]);
                    a1 = fma(fma(sH[warp][kk], r, sG[warp][kk]), r, a1);
                    a2 = fma(sU[warp][kk], r, a2);
                }
            }
        }
        red[0][warp][lane] = a1;
        red[1][warp][lane] = a2;
        __syncthreads();
        if (warp == 0 && act) {
            double s1 = 0.0, s2 = 0.0;
            for (int w = 0; w < BW_W; w++) { s1 += red[0][w][lane]; s2 += red[1][w][lane]; }
            const double v = vhat[b0 + i];
            dbar_s[b0 + i] = v * v * s1;
            zbar_s[b0 + i] = 2.0 * v * s2;
        }
        __syncthreads();
    }
}

// scatter to input order, deflated eigenvalues, rho scaling (one thread per slot)
__global__ void k_bw_scatter(int64_t nprob, const int64_t *__restrict__ off, int64_t total,
                             const int32_t *__restrict__ mk, const int32_t *__restrict__ src,
                             const int32_t *__restrict__ pinv, const double *__restrict__ lam_bar,
                             const double *__restrict__ dbar_s, const double *__restrict__ zbar_s, double sqrt_rho,
                             double *__restrict__ dbar, double *__restrict__ zbar)
{
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total; x += (int64_t)gridDim.x * blockDim.x) {
        if (x < off[0] || x >= off[nprob]) continue;
        const int64_t p = sdc_upper_index(off, nprob, x);
        const int64_t b0 = off[p], in = b0 + src[x];
        const bool kept = (int)(x - b0) < mk[p];
        dbar[in] = kept ? dbar_s[x] : (lam_bar ? lam_bar[b0 + pinv[x]] : 0.0);
        zbar[in] = kept ? zbar_s[x] * sqrt_rho : 0.0;
    }
}

// the rotations in reverse: chains touch disjoint entries (k_givens), so one
// thread per chain walks it from its end
__global__ void k_bw_rotate(int64_t nprob, const int64_t *__restrict__ off, int64_t total,
                            const int32_t *__restrict__ ngiv, const int32_t *__restrict__ giv_ab,
                            const double *__restrict__ giv_cs, double *__restrict__ dbar, double *__restrict__ zbar)
{
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total; x += (int64_t)gridDim.x * blockDim.x) {
        if (x < off[0] || x >= off[nprob]) continue;
        const int64_t p = sdc_upper_index(off, nprob, x);
        const int64_t b0 = off[p];
        const int t0 = (int)(x - b0), ng = ngiv[p];
        if (t0 >= ng) continue;
        const int32_t *ab = giv_ab + 2 * b0;
        const double *cs = giv_cs + 2 * b0;
        if (t0 + 1 < ng && ab[2 * (t0 + 1)] == ab[2 * t0 + 1]) continue;       // not a chain end
        for (int t = t0; t >= 0; t--) {
            if (t < t0 && ab[2 * (t + 1)] != ab[2 * t + 1]) break;
            const int a = ab[2 * t], bb = ab[2 * t + 1];
            const double c = cs[2 * t], s = cs[2 * t + 1];
            const double da = dbar[b0 + a], db = dbar[b0 + bb];
            dbar[b0 + a] = c * c * da + s * s * db;
            dbar[b0 + bb] = s * s * da + c * c * db;
            const double za = zbar[b0 + a], zb = zbar[b0 + bb];
            zbar[b0 + a] = c * za + s * zb;
            zbar[b0 + bb] = -s * za + c * zb;
        }
    }
}

}  // namespace

// Adjoint of one batched rank-one step given its factor view (pinv and d_K
// available).  X: the columns the step transformed (input order, read only),
// Ybar: cotangent of Qhat^T X (merged order); lam_bar may be NULL.
superdc_status r1_backward_fv(const FactorView &f, int64_t total, const double *lam_bar, int ncols,
                              const double *X, int64_t ldx, const double *Ybar, int64_t ldy, double *d_bar,
                              double *z_bar, double *X_bar, int64_t ldxb, double sqrt_rho, cudaStream_t st)
{
    const int nsm = sdc_num_sms();
    double *u = nullptr, *g = nullptr, *dbs = nullptr, *zbs = nullptr, *Y = nullptr, *Xw = nullptr;
    int64_t *tile_off = nullptr;
    SdcScratch sc(st);
    SDC_CHECK(sc.get(&u, total));
    SDC_CHECK(sc.get(&g, total));
    SDC_CHECK(sc.get(&dbs, total));
    SDC_CHECK(sc.get(&zbs, total));
    SDC_CHECK(sc.get(&tile_off, f.nprob + 1));
    SDC_CHECK(cudaMemsetAsync(u, 0, total * sizeof(double), st));
    SDC_CHECK(cudaMemsetAsync(g, 0, total * sizeof(double), st));
    k_tiles<<<1, tiles_threads(f.nprob), 0, st>>>(f.nprob, f.mk, BW_T, tile_off);
    superdc_status s = SUPERDC_OK;
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(total / BW_T + f.nprob, (int64_t)nsm * 8));
    if (ncols > 0) {
        // Y = Qhat^T X is recomputed (the rotations act on a copy of X)
        SDC_CHECK(sc.get(&Y, (size_t)total * ncols));
        SDC_CHECK(sc.get(&Xw, (size_t)total * ncols));
        SDC_CHECK(cudaMemcpy2DAsync(Xw, total * sizeof(double), X, ldx * sizeof(double), total * sizeof(double),
                                    ncols, cudaMemcpyDeviceToDevice, st));
        s = cauchy_apply_T(f, total, Xw, total, Y, total, ncols, st);
        if (s == SUPERDC_OK) s = cauchy_apply_N(f, total, Ybar, ldy, X_bar, ldxb, ncols, st);
        for (int c0 = 0; c0 < ncols && s == SUPERDC_OK; c0 += BW_C) {
            const int nc = std::min(BW_C, ncols - c0);
            auto fn = 2 * nc <= BW_W ? k_bw_lamlam<1> : k_bw_lamlam<2 * BW_C / BW_W>;
            PROF_LAUNCH("bw_lamlam", st, fn<<<grid, BW_W * 32, 0, st>>>(
                f.nprob, f.off, tile_off, f.mk, f.dorg, f.eta, f.bnorm, f.pinv, Y, total, Ybar, ldy, c0, nc, u, g));
        }
    }
    PROF_LAUNCH("bw_dz", st, k_bw_dz<<<grid, BW_W * 32, 0, st>>>(
        f.nprob, f.off, tile_off, f.mk, f.dk, f.dorg, f.eta, f.vhat, f.bnorm, f.pinv, lam_bar, u, g, dbs, zbs));
    const unsigned gr = (unsigned)std::max<int64_t>(1, std::min<int64_t>((total + 255) / 256, (int64_t)nsm * 8));
    k_bw_scatter<<<gr, 256, 0, st>>>(f.nprob, f.off, total, f.mk, f.src, f.pinv, lam_bar, dbs, zbs, sqrt_rho, d_bar,
                                     z_bar);
    k_bw_rotate<<<gr, 256, 0, st>>>(f.nprob, f.off, total, f.ngiv, f.giv_ab, f.giv_cs, d_bar, z_bar);
    cudaError_t e = cudaGetLastError();
    if (s != SUPERDC_OK) return s;
    return e == cudaSuccess ? SUPERDC_OK : SUPERDC_ERR_CUDA;
}

extern "C" superdc_status superdc_secular_batched_backward(
    int64_t nprob, const int64_t *offsets, int64_t total, double rho, const superdc_rank1_out *fwd,
    const double *lam_bar, int64_t ncols, const double *X, int64_t ldx, const double *Ybar, int64_t ldy,
    double *d_bar, double *z_bar, double *X_bar, int64_t ldxb, cudaStream_t st)
{
    if (nprob < 0 || total < 0 || !(rho > 0.0) || !fwd || ncols < 0 || ncols > 4096) return SUPERDC_ERR_ARG;
    if (nprob == 0 || total == 0) return SUPERDC_OK;
    if (!offsets || !d_bar || !z_bar || !fwd->dk || !fwd->eta || !fwd->vhat || !fwd->bnorm || !fwd->org ||
        !fwd->src || !fwd->perm || !fwd->giv_ab || !fwd->giv_cs || !fwd->mk || !fwd->ngiv)
        return SUPERDC_ERR_ARG;
    if (ncols > 0 && (!X || !Ybar || !X_bar || ldx < total || ldy < total || ldxb < total)) return SUPERDC_ERR_ARG;
    const int nsm = sdc_num_sms();
    int32_t *pinv = nullptr;
    double *dorg = nullptr;
    SdcScratch sc(st);
    SDC_CHECK(sc.get(&pinv, total));
    SDC_CHECK(sc.get(&dorg, total));
    k_prep<<<(unsigned)(nsm * 8), 256, 0, st>>>(nprob, offsets, total, fwd->mk, fwd->perm, fwd->org, fwd->dk, pinv,
                                                 dorg);
    FactorView f;
    f.nprob = nprob; f.off = offsets; f.mk = fwd->mk; f.ngiv = fwd->ngiv; f.dk = fwd->dk; f.eta = fwd->eta;
    f.dorg = dorg; f.vhat = fwd->vhat; f.bnorm = fwd->bnorm; f.src = fwd->src; f.perm = fwd->perm; f.pinv = pinv;
    f.giv_ab = fwd->giv_ab; f.giv_cs = fwd->giv_cs;
#ifdef SUPERDC_CHECK
    f.status = fwd->status;
#endif
    return r1_backward_fv(f, total, lam_bar, (int)ncols, X, ldx, Ybar, ldy, d_bar, z_bar, X_bar, ldxb, sqrt(rho), st);
}

extern "C" superdc_status superdc_rank1_apply(int64_t nprob, const int64_t *offsets, int64_t total,
                                              const superdc_rank1_out *fwd, int32_t trans, int64_t ncols,
                                              const double *X, int64_t ldx, double *Y, int64_t ldy,
                                              const superdc_opts *opts, cudaStream_t st)
{
    superdc_opts def;
    if (!opts) { superdc_opts_default(&def); opts = &def; }
    if (nprob < 0 || total < 0 || !fwd || ncols < 0 || (trans != 0 && trans != 1)) return SUPERDC_ERR_ARG;
    if (nprob == 0 || total == 0 || ncols == 0) return SUPERDC_OK;
    if (!offsets || !X || !Y || ldx < total || ldy < total || !fwd->dk || !fwd->eta || !fwd->vhat ||
        !fwd->bnorm || !fwd->org || !fwd->src || !fwd->perm || !fwd->giv_ab || !fwd->giv_cs || !fwd->mk ||
        !fwd->ngiv)
        return SUPERDC_ERR_ARG;
    const int nsm = sdc_num_sms();
    int32_t *pinv = nullptr;
    double *dorg = nullptr, *Xw = nullptr;
    SdcScratch sc(st);
    SDC_CHECK(sc.get(&pinv, total));
    SDC_CHECK(sc.get(&dorg, total));
    k_prep<<<(unsigned)(nsm * 8), 256, 0, st>>>(nprob, offsets, total, fwd->mk, fwd->perm, fwd->org, fwd->dk, pinv,
                                                 dorg);
    FactorView f;
    f.nprob = nprob; f.off = offsets; f.mk = fwd->mk; f.ngiv = fwd->ngiv; f.dk = fwd->dk; f.eta = fwd->eta;
    f.dorg = dorg; f.vhat = fwd->vhat; f.bnorm = fwd->bnorm; f.src = fwd->src; f.perm = fwd->perm; f.pinv = pinv;
    f.giv_ab = fwd->giv_ab; f.giv_cs = fwd->giv_cs;
#ifdef SUPERDC_CHECK
    f.status = fwd->status;
#endif
    f.fmm_min_m = fmm_resolve_rows(opts->fmm_min_m, total);
    superdc_status s;
    if (trans) {
        SDC_CHECK(sc.get(&Xw, (size_t)total * ncols));
        SDC_CHECK(cudaMemcpy2DAsync(Xw, total * sizeof(double), X, ldx * sizeof(double), total * sizeof(double),
                                    ncols, cudaMemcpyDeviceToDevice, st));
        s = cauchy_apply_T(f, total, Xw, total, Y, ldy, (int)ncols, st);
    } else {
        s = cauchy_apply_N(f, total, X, ldx, Y, ldy, (int)ncols, st);
    }
    cudaError_t e = cudaGetLastError();
    if (s != SUPERDC_OK) return s;
    return e == cudaSuccess ? SUPERDC_OK : SUPERDC_ERR_CUDA;
}
