// Application of one batched rank-one factor to a block of columns:
// Transpose (conquering stage, Algorithm 3; superdcmv with transpose,
// Algorithm 4):   y_j = b_j sum_i vhat_i x_i / ((d_i - d_{K_j}) - eta_j)
// Forward (superdcmv without transpose):
//                 y_i = vhat_i sum_j b_j x_j / ((d_i - d_{K_j}) - eta_j)
// with the shifted differences of eq. (4.28).  The rotations, the deflated
// slots and the order of the calls are here; the kept rows' products run on
// the tensor cores (fmm_columns, k_cm_apply).
#include "common.cuh"
#include <algorithm>
#include "cauchy.cuh"
#include "fmm.cuh"
#include "prof.cuh"
#include "tiles.cuh"

namespace {

constexpr int TR = 64;    // kept rows per tile of the application kernels

// rotations of the deflation, in scan order (forward) or reversed with the
// transposed rotation (inverse).  The rotation list is a sequence of chains
// (rotation k + 1 continues rotation k when its first index is the second
// index of k); different chains touch disjoint entries, so one thread per
// (chain, column) applies its chain in order (reversed for the inverse).
__global__ void k_givens(FactorView f, int64_t total, double *X, int64_t ldx, int ncols, int inverse)
{
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total * ncols;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t x = t % total;
        const int col = (int)(t / total);
        if (x < f.off[0] || x >= f.off[f.nprob]) continue;
        const int64_t p = sdc_upper_index(f.off, f.nprob, x);
        const int64_t b0 = f.off[p];
        const int g = (int)(x - b0);
        const int ng = f.ngiv[p];
        if (g >= ng) continue;
        const int32_t *ab = f.giv_ab + 2 * b0;
        const double *cs = f.giv_cs + 2 * b0;
        double *xv = X + b0 + (int64_t)col * ldx;
        if (!inverse) {
            if (g > 0 && ab[2 * g] == ab[2 * (g - 1) + 1]) continue;      // not a chain start
            for (int k = g; k < ng; k++) {
                if (k > g && ab[2 * k] != ab[2 * (k - 1) + 1]) break;
                const int a = ab[2 * k], b = ab[2 * k + 1];
                const double c = cs[2 * k], s = cs[2 * k + 1];
                const double xa = xv[a], xb = xv[b];
                xv[a] = c * xa - s * xb;
                xv[b] = s * xa + c * xb;
            }
        } else {
            if (g + 1 < ng && ab[2 * (g + 1)] == ab[2 * g + 1]) continue;  // not a chain end
            for (int k = g; k >= 0; k--) {
                if (k < g && ab[2 * (k + 1)] != ab[2 * k + 1]) break;
                const int a = ab[2 * k], b = ab[2 * k + 1];
                const double c = cs[2 * k], s = cs[2 * k + 1];
                const double xa = xv[a], xb = xv[b];
                xv[a] = c * xa + s * xb;
                xv[b] = -s * xa + c * xb;
            }
        }
    }
}

superdc_status run(const FactorView &f, int64_t total, double *Xmut, const double *X, int64_t ldx, double *Y,
                   int64_t ldy, int ncols, bool trans, cudaStream_t st, const FmmPlan *shared)
{
    if (ncols <= 0 || total <= 0) return SUPERDC_OK;
    const int nsm = sdc_num_sms();
    int64_t *tile_off = nullptr;
    SdcScratch sc(st);
    SDC_CHECK(sc.get(&tile_off, f.nprob + 1));
    k_tiles<<<1, tiles_threads(f.nprob), 0, st>>>(f.nprob, f.mk, TR, tile_off);
    const int gthreads = 128;
    if (trans)
        PROF_LAUNCH("givens", st, k_givens<<<(unsigned)(nsm * 8), gthreads, 0, st>>>(f, total, Xmut, ldx, ncols, 0));
    // problems whose kept size reaches the threshold have a box tree: the plan
    // of this factor's rank-one step when one was kept, else a new one
    FmmPlan fp;
    const int w = std::min(32, ncols);
    const bool use_shared = shared && shared->on && shared->dv.ncol >= w;
    if (!use_shared) {
        superdc_status fs = fmm_plan(fp, f.nprob, f.off, total, f.max_m, f.mk, f.dk, f.fmm_min_m, w, nullptr, false,
                                     st);
        if (fs != SUPERDC_OK) { fmm_free(fp, st); return fs; }
    }
    const superdc_status fs = fmm_columns(use_shared ? *shared : fp, f, total, tile_off, X, ldx, Y, ldy, ncols, trans, st);
    if (!trans)
        PROF_LAUNCH("givens", st, k_givens<<<(unsigned)(nsm * 8), gthreads, 0, st>>>(f, total, Y, ldy, ncols, 1));
    const cudaError_t le = cudaGetLastError();
    fmm_free(fp, st);
    if (le != cudaSuccess) return SUPERDC_ERR_CUDA;
    return fs;
}

}  // namespace

superdc_status cauchy_apply_T(const FactorView &f, int64_t total, double *X, int64_t ldx, double *Y, int64_t ldy,
                              int ncols, cudaStream_t st, const FmmPlan *plan)
{
    return run(f, total, X, X, ldx, Y, ldy, ncols, true, st, plan);
}

superdc_status cauchy_apply_N(const FactorView &f, int64_t total, const double *X, int64_t ldx, double *Y,
                              int64_t ldy, int ncols, cudaStream_t st)
{
    return run(f, total, nullptr, X, ldx, Y, ldy, ncols, false, st, nullptr);
}
