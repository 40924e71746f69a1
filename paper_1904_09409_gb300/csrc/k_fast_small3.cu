// The fixed-length kernels of lengths 2^a 3^b from 72 to 576.
#include "fast_kernels.cuh"

FT_FAST_SMALL3(FT_FAST_INSTANTIATE)

FT_DEBUG_READER(ft_debug_read_fast_small3)
