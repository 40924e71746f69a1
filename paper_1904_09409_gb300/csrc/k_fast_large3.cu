// The fixed-length kernels of lengths 2^a 3^b from 2304 to 3888.
#include "fast_kernels.cuh"

FT_FAST_LARGE3(FT_FAST_INSTANTIATE)

FT_DEBUG_READER(ft_debug_read_fast_large3)
