// Compile-time line length 768: apply passes of fft_passes.cuh (see there).
#include "fft_passes.cuh"
#define RVE_NL 768
#include "fft_inst_ct.cuh"
