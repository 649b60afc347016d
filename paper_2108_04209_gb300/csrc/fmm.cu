// Library defaults of the FMM threshold.
#include "fmm.cuh"

// measured on GB300 (python -m paper_2108_04209_gb300.crossover: batches of
// equal-size rank-one problems, whole step, direct / FMM): at m = 512 1.52 / 1.45
// ms for 256 problems and 4.66 / 3.68 for 1024, at m = 768 2.80 / 1.94 and
// 9.6 / 5.3, at 1024 4.5 / 2.6 and 16.4 / 7.7, at 2048 21.7 / 4.4 (256).  The
// autotuner refines it per batch.
int fmm_default_min_m() { return 512; }

// Below 128 rows per SM (19456), where neither path fills the GPU: step, direct /
// FMM, 16 problems of 512 0.44 / 0.80 ms, of 768 0.56 / 0.92, of 1024 0.67 /
// 0.97, of 1536 1.07 / 1.13, of 2048 1.62 / 1.15; one problem of 1536 0.82 /
// 0.98, of 2048 1.00 / 0.82; the applications (1 to 64 columns) cross between 1024
// and 2048 as well.  Above the line: 64 problems of 768 1.63 / 1.11, of 1024 2.20
// / 1.24, functions of a factor of 32768 rows to 64 columns 4 ms slower with 1536.  An eigendecomposition of n = 512 (leaf 32, rank 4)
// 6.4 -> 5.4 ms.  Steps called directly keep 512 at any number of rows: which problems
// took the tree is one of their results (superdc_rank1_out.fmm).
int fmm_few_rows_min_m() { return 1536; }
