// Launchers of the fixed-length kernels for one length each (defined in
// fast_kernels.cuh, instantiated in the units k_fast_*.cu), and the lengths of
// each unit.
#pragma once

#include "fft_fast.cuh"

#define FT_FAST_POW2(X) X(64) X(128) X(256) X(512) X(1024) X(2048) X(4096) X(8192) X(192) X(384) X(768) X(1536)
#define FT_FAST_SMALL3(X) X(72) X(96) X(108) X(144) X(162) X(216) X(288) X(324) X(432) X(486) X(576)
#define FT_FAST_MID3(X) X(648) X(864) X(972) X(1152) X(1296) X(1458) X(1728) X(1944)
#define FT_FAST_LARGE3(X) X(2304) X(2592) X(2916) X(3072) X(3456) X(3888)
#define FT_FAST_LENGTHS(X) FT_FAST_POW2(X) FT_FAST_SMALL3(X) FT_FAST_MID3(X) FT_FAST_LARGE3(X)

// arguments as for the launch_*_fast functions of fft_fast.cuh (stw: the
// length's per-pass twiddles)
template <int N>
cudaError_t go_r2c(const float* in, int rows_in, int ncols, int in_pitch, size_t in_img, int row0,
                          const float2* stw, float2* out, int out_pitch, size_t out_img, float es, float ms,
                          int batch, cudaStream_t st, bool pdl, bool follows_peak, unsigned* err, long long wait);
template <int N>
cudaError_t go_r2c_loss(const float* map, const float* target, int ncols, const float2* stw, float2* out,
                               int out_pitch, size_t out_img, float es, float ms, float scale, float gscale,
                               float* partial, int batch, cudaStream_t st, bool pdl, unsigned* err, long long wait);
template <int N>
cudaError_t go_c2r(const float2* in, int ncols, int in_pitch, size_t in_img, const float2* stw,
                          float mid, float* out, int row0, int rows_out, int out_pitch, size_t out_img,
                          float os, unsigned* tmax, int batch, cudaStream_t st, bool pdl, unsigned* err,
                          long long wait);
template <int N>
cudaError_t go_rows(float2* ws, int W, int Hp, int L, int interp, const float2* stw, int batch,
                           cudaStream_t st, bool pdl, unsigned* err, long long wait);
template <int N>
cudaError_t go_rows_adj(float2* ws, int W, int Hp, int L, int interp, const float2* stw, int batch,
                               cudaStream_t st, bool pdl, LossSum ls);
