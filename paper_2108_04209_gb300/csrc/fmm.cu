// Library default of the FMM threshold.
#include "fmm.cuh"

// measured on GB300 (python -m paper_2108_04209_gb300.crossover: batches of
// equal-size rank-one problems, whole step direct vs FMM): at m = 256 few
// problems keep enough poles for the tree and the direct path is 10 % faster;
// at m = 512 the FMM step is 1.4x faster (4096 problems), at 1024 2.6x, at
// 2048 7x; in the n = 131072 eigendecomposition (256 problems of 512 on that
// level) the threshold 512 beats 1024 and 256.  The autotuner refines it per
// batch.
int fmm_default_min_m() { return 512; }
