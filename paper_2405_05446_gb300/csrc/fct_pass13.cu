// FFT lengths of the direct solve, part 13 of 16 (fct_pass.cuh).
#include "fct_pass.cuh"

GDGS_FCT_SLICE(13)
