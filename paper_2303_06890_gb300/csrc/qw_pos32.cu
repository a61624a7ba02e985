/* qw_pos32.cu -- the positional layout's kernels for complex64 amplitudes. */
#include "qw_pos.cuh"

QW_POS_INSTANTIATE(32, float2)
