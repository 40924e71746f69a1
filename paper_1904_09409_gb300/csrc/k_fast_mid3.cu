// The fixed-length kernels of lengths 2^a 3^b from 648 to 1944.
#include "fast_kernels.cuh"

FT_FAST_MID3(FT_FAST_INSTANTIATE)

FT_DEBUG_READER(ft_debug_read_fast_mid3)
