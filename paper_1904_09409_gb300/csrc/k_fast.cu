// The fixed-length column and row kernels by length (see fast_kernels.cuh): the
// launch_*_fast functions of fft_fast.cuh.
#include "fast_launch.cuh"

unsigned ft_debug_read_fast_pow2();
unsigned ft_debug_read_fast_small3();
unsigned ft_debug_read_fast_mid3();
unsigned ft_debug_read_fast_large3();
unsigned ft_debug_read_fast() {
    return ft_debug_read_fast_pow2() | ft_debug_read_fast_small3() | ft_debug_read_fast_mid3() |
           ft_debug_read_fast_large3();
}

cudaError_t launch_col_r2c_fast(const float* in, int rows_in, int ncols, int in_pitch, size_t in_img,
                                int row0, const FftLen& f, float2* out, int out_pitch, size_t out_img,
                                float end_scale, float mid_scale, int batch, cudaStream_t st, bool pdl,
                                bool follows_peak, unsigned* err, long long wait) {
    switch (f.N) {
#define X(n) case n: return go_r2c<n>(in, rows_in, ncols, in_pitch, in_img, row0, f.stw, out, out_pitch, \
                                      out_img, end_scale, mid_scale, batch, st, pdl, follows_peak, err, wait);
        FT_FAST_LENGTHS(X)
#undef X
    }
    return cudaErrorNotSupported;
}

int col_r2c_loss_blocks(const FftLen& f, int ncols) {
    switch (f.N) {
#define X(n) case n: return (ncols + 2 * fs_Bcol(n) - 1) / (2 * fs_Bcol(n));
        FT_FAST_LENGTHS(X)
#undef X
    }
    return 0;
}

cudaError_t launch_col_r2c_loss_fast(const float* map, const float* target, int ncols, const FftLen& f,
                                     float2* out, int out_pitch, size_t out_img, float end_scale, float mid_scale,
                                     float scale, float gscale, float* partial, int batch, cudaStream_t st,
                                     bool pdl, unsigned* err, long long wait) {
    if (ncols & 1) return cudaErrorInvalidValue;
    switch (f.N) {
#define X(n) case n: return go_r2c_loss<n>(map, target, ncols, f.stw, out, out_pitch, out_img, end_scale, mid_scale, \
                                           scale, gscale, partial, batch, st, pdl, err, wait);
        FT_FAST_LENGTHS(X)
#undef X
    }
    return cudaErrorNotSupported;
}

cudaError_t launch_col_c2r_fast(const float2* in, int ncols, int in_pitch, size_t in_img,
                                const FftLen& f, float mid_scale, float* out, int row0, int rows_out,
                                int out_pitch, size_t out_img, float out_scale, int batch,
                                cudaStream_t st, unsigned* tmax, bool pdl, unsigned* err, long long wait) {
    if (tmax && (row0 != 0 || rows_out != f.N)) return cudaErrorInvalidValue;
    switch (f.N) {
#define X(n) case n: return go_c2r<n>(in, ncols, in_pitch, in_img, f.stw, mid_scale, out, row0, rows_out, \
                                      out_pitch, out_img, out_scale, tmax, batch, st, pdl, err, wait);
        FT_FAST_LENGTHS(X)
#undef X
    }
    return cudaErrorNotSupported;
}

bool c2r_tile_shape(int N, int* rows, int* cols, int* bands) {
    if (!c2r_tiles(N)) return false;
    switch (N) {
#define X(n) case n: *rows = c2r_tile_rows(n); *cols = 2 * fs_Bc2r(n); *bands = c2r_tile_bands(n); return true;
        FT_FAST_LENGTHS(X)
#undef X
    }
    return false;
}

cudaError_t launch_nvmt_rows_fast(float2* ws, int W, int Hp, int L, int interp, const FftLen& fx,
                                  int batch, cudaStream_t st, bool pdl, unsigned* err, long long wait) {
    if (((uintptr_t)ws & 15) || (W & 1) || wait < 0) return cudaErrorInvalidValue;   // bulk-copy alignment
    switch (fx.N) {
#define X(n) case n: return go_rows<n>(ws, W, Hp, L, interp, fx.stw, batch, st, pdl, err, wait);
        FT_FAST_LENGTHS(X)
#undef X
    }
    return cudaErrorNotSupported;
}

cudaError_t launch_nvmt_rows_adjoint_fast(float2* ws, int W, int Hp, int L, int interp,
                                          const FftLen& fx, int batch, cudaStream_t st, bool pdl, LossSum ls) {
    switch (fx.N) {
#define X(n) case n: return go_rows_adj<n>(ws, W, Hp, L, interp, fx.stw, batch, st, pdl, ls);
        FT_FAST_LENGTHS(X)
#undef X
    }
    return cudaErrorNotSupported;
}
