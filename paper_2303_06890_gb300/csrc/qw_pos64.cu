/* qw_pos64.cu -- the positional layout's kernels for complex128 amplitudes. */
#include "qw_pos.cuh"

QW_POS_INSTANTIATE(64, double2)
