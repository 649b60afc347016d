// The triangular FMM's translation unit (entry points of fmm.cuh, leaf boxes of 32).
#include "fmm_impl.cuh"
