// Triangular FMM with leaf boxes of 32 indices: the entry points of fmm.cuh.
#define FMM_BOX 32
#define FMM_NS fmm_b32
#include "fmm_impl.cuh"

superdc_status fmm_plan(FmmPlan &pl, int64_t nprob, const int64_t *off, int64_t total, int64_t max_m,
                        const int32_t *mk, const double *dk, int min_m, int ncol, int32_t *used, bool step,
                        cudaStream_t st)
{
    return fmm_b32::plan(pl, nprob, off, total, max_m, mk, dk, min_m, ncol, used, step, st);
}

void fmm_free(FmmPlan &pl, cudaStream_t st) { fmm_b32::free_plan(pl, st); }

superdc_status fmm_secular(const FmmPlan &pl, const int64_t *off, const R1Out &o, double stop_c, int max_iter,
                           cudaStream_t st)
{
    return fmm_b32::secular(pl, off, o, stop_c, max_iter, st);
}

superdc_status fmm_lowner(const FmmPlan &pl, const int64_t *off, const R1Out &o, cudaStream_t st)
{
    return fmm_b32::lowner(pl, off, o, st);
}

superdc_status fmm_bnorm(const FmmPlan &pl, const int64_t *off, const R1Out &o, cudaStream_t st)
{
    return fmm_b32::bnorm(pl, off, o, st);
}

superdc_status fmm_columns(const FmmPlan &pl, const FactorView &f, int64_t total, const int64_t *tile_off,
                           const double *X, int64_t ldx, double *Y, int64_t ldy, int ncols, bool trans,
                           cudaStream_t st)
{
    return fmm_b32::columns(pl, f, total, tile_off, X, ldx, Y, ldy, ncols, trans, st);
}
