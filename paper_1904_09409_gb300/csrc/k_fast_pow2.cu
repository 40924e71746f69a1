// The fixed-length kernels of the powers of two and 3 x 2^a up to 1536.
#include "fast_kernels.cuh"

FT_FAST_POW2(FT_FAST_INSTANTIATE)

FT_DEBUG_READER(ft_debug_read_fast_pow2)
