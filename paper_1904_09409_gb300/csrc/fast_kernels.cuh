// Fixed-length versions of the column and row kernels over a uniform batch
// (see k_cols.cu and k_rows.cu for what each step computes): one block of
// fast_blocks.cuh per CUDA block, the image index in blockIdx.y.  The units
// k_fast_*.cu instantiate the launchers (fast_launch.cuh) for a group of lengths
// each, so that the groups compile in parallel; k_fast.cu chooses by length.
#pragma once

#include <string.h>

#include <atomic>

#include "fast_blocks.cuh"
#include "fast_launch.cuh"

// tma_nb > 0: the image columns are staged by tma_nb tensor copies of tma_h
// rows (tmap describes the launch's images), else read from global memory.
// follows_peak: the predecessor on the stream is the peak pass of the previous
// batch of ft_detect_batches, which has waited for its own step 4 and touches
// only the maps, the tile maxima and the peak records: this kernel reads its
// images and writes the spectrum workspace without waiting for it, and only its
// last block waits for that pass before exiting, so that the completion of this
// grid (which the next kernels wait for) implies the completion of the pass.
template <int N>
__global__ void __launch_bounds__(fs_T(N) * fs_Bcol(N), fs_minblocks(N, fs_T(N) * fs_Bcol(N)))
k_col_r2c_fast(const float* __restrict__ in, int rows_in, int ncols, int in_pitch, size_t in_img,
               int row0, const float2* __restrict__ stw, float2* __restrict__ out, int out_pitch,
               size_t out_img, float end_scale, float mid_scale, const __grid_constant__ CUtensorMap tmap,
               int tma_h, int tma_nb, unsigned* __restrict__ err, long long wait, int pf, int follows_peak) {
    extern __shared__ __align__(128) float2 sm[];
    pdl_trigger_large();
    if (!follows_peak) pdl_wait();
    const float* src = in + (size_t)blockIdx.y * in_img;
    float2* dst = out + (size_t)blockIdx.y * out_img;
    if (tma_nb > 0) {
        const int nxt = blockIdx.y * gridDim.x + blockIdx.x + pf;
        const int pimg = pf > 0 && nxt < gridDim.x * gridDim.y ? nxt / gridDim.x : -1;
        r2c_block<N, fs_Bcol(N), true>(src, rows_in, ncols, in_pitch, row0, stw, dst, out_pitch, end_scale,
                                       mid_scale, blockIdx.x, sm, &tmap, tma_h, tma_nb, blockIdx.y, err, wait,
                                       nxt - pimg * gridDim.x, pimg);
    }
    else
        r2c_block<N, fs_Bcol(N)>(src, rows_in, ncols, in_pitch, row0, stw, dst, out_pitch, end_scale, mid_scale,
                                 blockIdx.x, sm);
    if (follows_peak && blockIdx.x == gridDim.x - 1 && blockIdx.y == gridDim.y - 1) pdl_wait();
}

// tma_nb > 0: the Hermitian half is staged by tma_nb tensor copies of tma_h rows
// (tmap describes the launch's half spectra), else by cp.async
template <int N>
__global__ void __launch_bounds__(fs_T(N) * fs_Bc2r(N), fs_minblocks(N, fs_T(N) * fs_Bc2r(N)))
k_col_c2r_fast(const float2* __restrict__ in, int ncols, int in_pitch, size_t in_img,
               const float2* __restrict__ stw, float mid_scale, float* __restrict__ out, int row0,
               int rows_out, int out_pitch, size_t out_img, float out_scale, unsigned* __restrict__ tmax,
               const __grid_constant__ CUtensorMap tmap, int tma_h, int tma_nb, unsigned* __restrict__ err,
               long long wait, int pf) {
    extern __shared__ __align__(128) float2 sm[];
    pdl_trigger_large();
    pdl_wait();
    constexpr int bands = c2r_tile_bands(N);
    const float2* src = in + (size_t)blockIdx.y * in_img;
    float* dst = out + (size_t)blockIdx.y * out_img;
    unsigned* tm = tmax ? tmax + (size_t)blockIdx.y * bands * gridDim.x : nullptr;
    if (tma_nb > 0) {
        const int nxt = blockIdx.y * gridDim.x + blockIdx.x + pf;
        const int pimg = pf > 0 && nxt < gridDim.x * gridDim.y ? nxt / gridDim.x : -1;
        c2r_block<N, fs_Bc2r(N), true>(src, ncols, in_pitch, stw, mid_scale, dst, row0, rows_out, out_pitch,
                                       out_scale, tm, gridDim.x, blockIdx.x, sm, &tmap, tma_h, tma_nb, blockIdx.y,
                                       err, wait, nxt - pimg * gridDim.x, pimg);
    }
    else
        c2r_block<N, fs_Bc2r(N)>(src, ncols, in_pitch, stw, mid_scale, dst, row0, rows_out, out_pitch, out_scale,
                                 tm, gridDim.x, blockIdx.x, sm);
}

// The adjoint of step 4 fed straight from the loss of the gradient workload:
// the input column pair is not a stored gradient map but
//     g = 2 r scale sign(P) gscale,   r = |P| scale - T
// computed from the map P and the target T as the columns are loaded (the loss
// gradient of k_loss.cu), while every thread adds r^2 of its samples (FP32,
// compensated) and the block writes one partial of the image's loss.  Each map
// cell is loaded by exactly one thread, so the partials of an image's blocks
// add up to its sum of r^2 (within a block by a fixed shuffle tree); the next
// kernel adds them (LossSum: a launch of its own took 6 us, and counting the blocks
// so that the last one adds them 15 us of 166 per 64 x 1024^2, the fence's wait).  With
// tma_nb > 0 the map columns arrive by tensor copies into the exchange buffer
// (pmap, waited for with the bound `wait`; bit 3 of *err when it runs out, and
// the block returns without writing); the map and target (tmapt) boxes
// of the block pf blocks later are prefetched into L2.  Everything after the
// load is r2c_finish.
template <int N>
__global__ void __launch_bounds__(fs_T(N) * fs_Bcol(N), fs_minblocks(N, fs_T(N) * fs_Bcol(N)))
k_col_r2c_loss_fast(const float* __restrict__ map, const float* __restrict__ target, int ncols, size_t img_cells,
                    const float2* __restrict__ stw, float2* __restrict__ out, int out_pitch, size_t out_img,
                    float end_scale, float mid_scale, float scale, float gscale, float* __restrict__ partial,
                    const __grid_constant__ CUtensorMap pmap, const __grid_constant__ CUtensorMap tmapt, int tma_h,
                    int tma_nb, unsigned* __restrict__ err, long long wait, int pf) {
    constexpr int B = fs_Bcol(N), E = fs_E(N), NT = fs_T(N) * fs_Bcol(N), NW = (NT + 31) / 32;
    constexpr int R0 = fs_radix(N, 0), G0 = E / R0;
    using F = FastFft<N, -1, B>;
    extern __shared__ __align__(128) float2 sm[];
    __shared__ float red[NW];
    const int f = threadIdx.x % B;
    const int t = threadIdx.x / B;
    const int c = blockIdx.x * 2 * B + 2 * f;
    const bool colok = c < ncols;
    const float* P = map + (size_t)blockIdx.y * img_cells + c;
    const float* Tg = target + (size_t)blockIdx.y * img_cells + c;
    const float* stg = reinterpret_cast<const float*>(sm);   // [>= N][2B] map values
    __shared__ uint64_t mbar;
    const uint32_t mb = smem_u32(&mbar);
    float2 v[E];
    pdl_trigger_large();
    pdl_wait();
    float* part = partial + (size_t)blockIdx.y * gridDim.x + blockIdx.x;
    if (tma_nb > 0) {
        // the block's map columns by tensor copies into the exchange buffer; their
        // latency hides that of the target values, which come straight from global
        // memory to registers (prefetched into L2 like the map by the block pf blocks
        // before).  A second round of copies for the target, after the map had gone to
        // registers, took 49.5 us per 16 Mpx of 512^2 and 167 us per 64 x 1024^2, this 44
        // and 161
        if (threadIdx.x == 0) {
            mbar_init(mb, 1);
            mbar_arrive_expect_tx(mb, (uint32_t)(tma_nb * tma_h * 2 * B * sizeof(float)));
            for (int k = 0; k < tma_nb; ++k)
                tma_load_3d(reinterpret_cast<float*>(sm) + k * tma_h * 2 * B, &pmap, blockIdx.x * 2 * B, k * tma_h,
                            blockIdx.y, mb);
            const int nxt = blockIdx.y * gridDim.x + blockIdx.x + pf;
            if (pf > 0 && nxt < gridDim.x * gridDim.y) {
                const int pimg = nxt / gridDim.x, pbx = nxt - pimg * gridDim.x;
                for (int k = 0; k < tma_nb; ++k) {
                    tma_prefetch_3d(&pmap, pbx * 2 * B, k * tma_h, pimg);
                    tma_prefetch_3d(&tmapt, pbx * 2 * B, k * tma_h, pimg);
                }
            }
        }
    } else if (colok) {
        // the same overlap where the tensor copies don't apply (2B columns or an image
        // row no multiple of 16 bytes): every thread copies its own pairs and waits for
        // them alone (16 Mpx of 486^2: 83.0 us with the map read in the loop below, 54.8 so)
        static_assert(N * B <= F::SLOTS, "the map columns fit the exchange buffer");
#pragma unroll
        for (int m = 0; m < G0; ++m)
#pragma unroll
            for (int q = 0; q < R0; ++q) {
                const int row = F::template in_pos<0>(t, m, q);
                if (FT_IN(row, N, FT_DBG_R2C_LOAD) && FT_IN(c + 1, ncols, FT_DBG_R2C_LOAD) &&
                    FT_IN(row * B + f, F::SLOTS, FT_DBG_FFT_SLOT))
                    cp_async8(reinterpret_cast<float*>(sm) + row * 2 * B + 2 * f, P + (size_t)row * ncols);
            }
    }
#pragma unroll
    for (int m = 0; m < G0; ++m)
#pragma unroll
        for (int q = 0; q < R0; ++q)
            v[m * R0 + q] = colok && FT_IN(c + 1, ncols, FT_DBG_R2C_LOAD)
                                ? __ldg(reinterpret_cast<const float2*>(
                                      Tg + (size_t)F::template in_pos<0>(t, m, q) * ncols))
                                : make_float2(0.f, 0.f);
    if (tma_nb > 0) {
        __syncthreads();                               // the mbarrier is initialised
        const bool ok = mbar_wait(mb, 0, wait);
        if (__syncthreads_or(!ok)) {
            if (threadIdx.x == 0 && err) atomicOr(err, 8u);
            mbar_wait(mb, 0);                          // the copies in flight land first
            if (threadIdx.x == 0) *part = __int_as_float(0x7fc00000);   // NaN: the loss is incomplete
            return;
        }
    } else {
        cp_async_wait_all();
    }

    // compensated sums of r^2, one per column of the pair (two chains of dependent adds)
    float acc2[2] = {0.f, 0.f}, comp2[2] = {0.f, 0.f};
    auto add = [&](int i, float y) {
        const float z = y - comp2[i];
        const float s2 = acc2[i] + z;
        comp2[i] = (s2 - acc2[i]) - z;
        acc2[i] = s2;
    };
#pragma unroll
    for (int m = 0; m < G0; ++m)
#pragma unroll
        for (int q = 0; q < R0; ++q) {
            const int row = F::template in_pos<0>(t, m, q);
            float2 g = make_float2(0.f, 0.f);
            if (colok) {
                const float2 p = *reinterpret_cast<const float2*>(stg + row * 2 * B + 2 * f);
                const float2 tt = v[m * R0 + q];
                const float r0 = fabsf(p.x) * scale - tt.x, r1 = fabsf(p.y) * scale - tt.y;
                add(0, r0 * r0);
                add(1, r1 * r1);
                const float s0 = p.x > 0.f ? 1.f : (p.x < 0.f ? -1.f : 0.f);
                const float s1 = p.y > 0.f ? 1.f : (p.y < 0.f ? -1.f : 0.f);
                g = make_float2(2.f * r0 * scale * s0 * gscale, 2.f * r1 * scale * s1 * gscale);
            }
            v[m * R0 + q] = g;
        }
    const float comp = comp2[0] + comp2[1];
    float acc = acc2[0] + acc2[1] - (comp == comp ? comp : 0.f);   // NaN once a sum overflows
    // the block's partial: a fixed shuffle tree per warp, then over the warps (the
    // last warp may be partial; lane 0's sum takes nothing from lanes it lacks)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int lanes = min(32, NT - 32 * warp);
    const unsigned mask = 0xffffffffu >> (32 - lanes);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float x = __shfl_xor_sync(mask, acc, o);
        acc += (lane ^ o) < lanes ? x : 0.f;
    }
    if (lane == 0) red[warp] = acc;
    __syncthreads();                                   // also: the staged map is no longer read
    if (warp == 0) {
        float x = lane < NW ? red[lane] : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) *part = x;
    }
    r2c_finish<N, fs_Bcol(N)>(v, sm, t, f, stw, colok, out + (size_t)blockIdx.y * out_img + c, out_pitch, end_scale,
                              mid_scale);
}

// 64 threads per block at most lengths and at most 64 registers (fs_minblocks: 72 to 112
// where a thread holds 18 to 36 samples), so that 16 blocks share a multiprocessor
template <int N, int INTERP>
__global__ void __launch_bounds__(fs_T(N) * fs_Brow(N), fs_minblocks(N, fs_T(N) * fs_Brow(N)))
k_nvmt_rows_fast(float2* __restrict__ ws, int W, int Hp, int L, const float2* __restrict__ stw,
                 unsigned* __restrict__ err, long long wait) {
    extern __shared__ __align__(128) float2 sm[];
    pdl_trigger_large();
    pdl_wait();
    // images in reverse order: the first blocks read the half spectra step 1
    // wrote last (still in L2), and step 4, in forward order, starts on the
    // rows written here last (per 64 x 1024^2: steps 2-3 103.2 -> 100.3 us,
    // step 4 115.4 -> 112.5 us)
    rows_block<N, INTERP, fs_Brow(N), true>(ws + (size_t)(gridDim.y - 1 - blockIdx.y) * L * N, W, Hp, L, stw,
                                            blockIdx.x, sm, err, wait);
}

template <int N, int INTERP>
__global__ void __launch_bounds__(fs_T(N) * fs_Brow(N), fs_minblocks(N, fs_T(N) * fs_Brow(N)))
k_nvmt_rows_adjoint_fast(float2* __restrict__ ws, int W, int Hp, int L, const float2* __restrict__ stw, LossSum ls) {
    pdl_trigger_large();
    pdl_wait();
    if (ls.loss && blockIdx.x == gridDim.x - 1) loss_sum_block(ls, blockIdx.y);
    constexpr int B = fs_Brow(N), E = fs_E(N), T = N / E;
    constexpr int R0 = fs_radix(N, 0), G0 = E / R0;
    constexpr int RL = fs_radix(N, fs_nst(N) - 1), GL = E / RL;
    using F = FastFft<N, -1, 1, true>;                 // the row length's seed table
    extern __shared__ float2 smrows[];
    const int f = threadIdx.x / T;                     // T consecutive threads per row
    const int t = threadIdx.x % T;
    float2* sm = smrows + f * F::SLOTS;
    const int l = blockIdx.x * B + f;
    // images in reverse order, as in k_nvmt_rows_fast (L2 reuse with the column
    // kernels before and after, which run in forward order)
    float2* row = ws + (size_t)(gridDim.y - 1 - blockIdx.y) * L * N + (size_t)l * N;

    float2 v[E];
#pragma unroll
    for (int m = 0; m < G0; ++m)
#pragma unroll
        for (int q = 0; q < R0; ++q)
            v[m * R0 + q] = l < L && FT_IN((fs_rotate<N, R0>(F::template in_pos<0>(t, m, q), q)), N, FT_DBG_NVMT_ADJ)
                                ? row[fs_rotate<N, R0>(F::template in_pos<0>(t, m, q), q)]
                                : make_float2(0.f, 0.f);
    F::template run<0>(v, sm, t, 0, stw);
    // gV[x'] = (-1)^{i + N/2} z[i], i = x' + N/2, z the transform of (-1)^s g[s]: the
    // signs are the rotations of the transform's input and output by N/2
    const int st = spos(t);
#pragma unroll
    for (int m = 0; m < GL; ++m)
#pragma unroll
        for (int q = 0; q < RL; ++q) {
            const int c = F::out_pos(0, m, q);
            const int o = RL % 2 == 0 ? spos_plus(t, st, q < RL / 2 ? c + N / 2 : c - N / 2)
                                      : spos(fs_rotate<N, RL>(t + c, q));
            if (FT_IN(o, F::SLOTS, FT_DBG_FFT_SLOT)) sm[o] = v[m * RL + q];
        }
    __syncthreads();
    if (l >= L) return;
    // Column x receives, for each tap d, from the sample x' with floor(x' H' / (2 l)) =
    // u = x - W/2 - d (at most one, since H' >= 2 l): x' = ceil(u 2 l / H'), with
    // x' H' - u 2 l = k (0 <= k < H'); such an x' exists iff k < 2 l, and its fraction is
    // k / (2 l).  A thread takes two adjacent columns, whose taps share all but one of
    // their u: ND + 1 pairs (x', k) instead of 2 ND, stepped exactly from one pair of
    // columns to the next (k, an integer below 8192, in FP32: no conversion for the
    // fraction).  The kernel is bound by these instructions: 16 Mpx of 1024^2 took 35.1 us
    // (linear) and 53.1 (cubic) with one column and integer steps per pass, 29.3 and 38.0
    // so.
    constexpr int DLO = INTERP == FT_INTERP_LINEAR ? 0 : -1;
    constexpr int DHI = INTERP == FT_INTERP_LINEAR ? 1 : 2;
    constexpr int ND = DHI - DLO + 1;
    const int den = 2 * l;
    const float inv = 1.f / (float)den;
    const float hpf = (float)Hp, denf = (float)den;
    const int sA = 2 * T * den / Hp;
    const float sB = (float)(2 * T * den - sA * Hp);
    int xp[ND + 1];
    float k[ND + 1];
    {
        const int num = (2 * t + 1 - (W >> 1) - DLO) * den + Hp - 1;
        xp[0] = floor_div(num, Hp);
        k[0] = (float)(Hp - 1 - (num - xp[0] * Hp));
    }
#pragma unroll
    for (int j = 1; j <= ND; ++j) {                    // u one less: k grows by 2 l <= H'
        xp[j] = xp[j - 1];
        k[j] = k[j - 1] + denf;
        if (k[j] >= hpf) { k[j] -= hpf; xp[j] -= 1; }
    }
    for (int x = 2 * t; x < W; x += 2 * T) {
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);  // columns x, x + 1
        if (l >= 1) {
#pragma unroll
            for (int j = 0; j <= ND; ++j) {
                if (k[j] < denf && xp[j] >= -N / 2 && xp[j] < N / 2 && FT_IN(xp[j] + N / 2, N, FT_DBG_NVMT_ADJ)) {
                    const float fr = k[j] * inv;
                    float w[ND];
                    if constexpr (INTERP == FT_INTERP_LINEAR) {
                        w[0] = 1.f - fr;
                        w[1] = fr;
                    } else {
                        keys_weights(fr, w);           // those the unrolled j uses are computed
                    }
                    const float2 g = sm[spos(xp[j] + N / 2)];
                    if (j >= 1) {
                        acc.x = fmaf(w[j - 1], g.x, acc.x);
                        acc.y = fmaf(w[j - 1], g.y, acc.y);
                    }
                    if (j < ND) {
                        acc.z = fmaf(w[j], g.x, acc.z);
                        acc.w = fmaf(w[j], g.y, acc.w);
                    }
                }
                xp[j] += sA;
                k[j] -= sB;
                if (k[j] < 0.f) { k[j] += hpf; xp[j] += 1; }
            }
        }
        if (!FT_IN(x, N, FT_DBG_ROW_STORE)) continue;
        if (x + 1 < W) *reinterpret_cast<float4*>(row + x) = acc;
        else row[x] = make_float2(acc.x, acc.y);
    }
}

// cuTensorMapEncodeTiled through the runtime's driver entry points (no link to
// the driver library); null when unavailable
typedef CUresult (*encode_tiled_fn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                    const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                    CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static encode_tiled_fn encode_tiled() {
    static encode_tiled_fn fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (encode_tiled_fn)f;
    }
    return fn;
}

// Tensor copies of step 1's image columns: the N expanded rows of 2B columns in
// nb boxes of h <= 256 rows (each box 128-byte aligned in shared memory), within
// the exchange buffer; false when that does not fit, B < 2 (a box row of 16
// bytes at least), the images are not laid out in 16-byte multiples or the map
// cannot be encoded (the first pass then reads global memory directly).
template <int N>
static bool r2c_tma_map(const float* in, int rows_in, int ncols, int in_pitch, size_t in_img, int batch,
                        CUtensorMap* map, int* h, int* nb) {
    constexpr int B = fs_Bcol(N);
    const encode_tiled_fn enc = encode_tiled();
    if (!enc || B < 2 || ((uintptr_t)in & 15) || (in_pitch & 3) || (in_img & 3) || ncols < 1 || rows_in < 1)
        return false;
    const int step = B >= 16 ? 1 : 16 / B;             // h 2B 4 bytes a multiple of 128
    int n = (N + 255) / 256, hh = 0;
    for (;; ++n) {
        hh = (N + n - 1) / n;
        hh = (hh + step - 1) / step * step;
        if (hh <= 256) break;
    }
    if ((size_t)n * hh * 2 * B * sizeof(float) > (size_t)FastFft<N, -1, B>::SLOTS * sizeof(float2)) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)ncols, (cuuint64_t)rows_in, (cuuint64_t)batch};
    const cuuint64_t strides[2] = {(cuuint64_t)in_pitch * sizeof(float), (cuuint64_t)in_img * sizeof(float)};
    const cuuint32_t box[3] = {(cuuint32_t)(2 * B), (cuuint32_t)hh, 1u};
    const cuuint32_t estr[3] = {1u, 1u, 1u};
    if (enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(in), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return false;
    *h = hh;
    *nb = n;
    return true;
}

// the distance, in blocks, of the column kernels' L2 prefetch: half of the
// blocks of kernel k (threads, sm bytes of dynamic shared memory) resident on
// the whole GPU at once (0 when it cannot be determined).  Measured per
// 64 x 1024^2 step (pipelined): 2 waves 345 us, 1 wave 320, 1/2 317, 1/4 316,
// 1/8 320, none 327.
// It depends only on the kernel and the device, and the occupancy query is a large
// part of a small launch's host time, so each launcher keeps it per device (cache:
// the launcher's own words, 0: unknown, else distance + 1; any thread may fill them).
#define FT_PF_DEVICES 16
template <typename K>
static int prefetch_distance(std::atomic<int>* cache, K k, int threads, size_t sm) {
    int dev = 0, per = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (dev < FT_PF_DEVICES) {
        const int c = cache[dev].load(std::memory_order_relaxed);
        if (c) return c - 1;
    }
    if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, threads, sm) != cudaSuccess)
        return 0;
    const int d = per * nsm / 2;
    if (dev < FT_PF_DEVICES) cache[dev].store(d + 1, std::memory_order_relaxed);
    return d;
}

// dynamic shared memory above the 48 KB that every kernel may use needs the
// kernel's consent
template <typename K>
static cudaError_t allow_smem(K k, size_t sm) {
    return sm > 48 * 1024 ? cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) : cudaSuccess;
}

template <int N>
cudaError_t go_r2c(const float* in, int rows_in, int ncols, int in_pitch, size_t in_img, int row0,
                          const float2* stw, float2* out, int out_pitch, size_t out_img, float es, float ms,
                          int batch, cudaStream_t st, bool pdl, bool follows_peak, unsigned* err, long long wait) {
    constexpr int B = fs_Bcol(N);
    const size_t sm = (size_t)FastFft<N, -1, B>::SLOTS * sizeof(float2);
    cudaError_t e = allow_smem(k_col_r2c_fast<N>, sm);
    if (e != cudaSuccess) return e;
    CUtensorMap map;
    memset(&map, 0, sizeof(map));
    int h = 0, nb = 0;
    if (!err || wait < 0 || !r2c_tma_map<N>(in, rows_in, ncols, in_pitch, in_img, batch, &map, &h, &nb)) nb = 0;
    dim3 grid((ncols + 2 * B - 1) / (2 * B), batch);
    static std::atomic<int> pfc[FT_PF_DEVICES];
    const int pf = prefetch_distance(pfc, k_col_r2c_fast<N>, fs_T(N) * B, sm);
    return launch_maybe_pdl(k_col_r2c_fast<N>, grid, dim3(fs_T(N) * B), sm, st, pdl, in, rows_in, ncols, in_pitch,
                            in_img, row0, stw, out, out_pitch, out_img, es, ms, map, h, nb, err, wait, pf,
                            (pdl && follows_peak) ? 1 : 0);
}

template <int N>
cudaError_t go_r2c_loss(const float* map, const float* target, int ncols, const float2* stw, float2* out,
                               int out_pitch, size_t out_img, float es, float ms, float scale, float gscale,
                               float* partial, int batch, cudaStream_t st, bool pdl, unsigned* err, long long wait) {
    constexpr int B = fs_Bcol(N);
    const size_t sm = (size_t)FastFft<N, -1, B>::SLOTS * sizeof(float2);
    cudaError_t e = allow_smem(k_col_r2c_loss_fast<N>, sm);
    if (e != cudaSuccess) return e;
    CUtensorMap pm, tm;
    memset(&pm, 0, sizeof(pm));
    memset(&tm, 0, sizeof(tm));
    const size_t cells = (size_t)N * ncols;
    int h = 0, nb = 0, h2 = 0, nb2 = 0;
    if (!err || wait < 0 || !r2c_tma_map<N>(map, N, ncols, ncols, cells, batch, &pm, &h, &nb) ||
        !r2c_tma_map<N>(target, N, ncols, ncols, cells, batch, &tm, &h2, &nb2))
        nb = 0;
    dim3 grid((ncols + 2 * B - 1) / (2 * B), batch);
    static std::atomic<int> pfc[FT_PF_DEVICES];
    const int pf = prefetch_distance(pfc, k_col_r2c_loss_fast<N>, fs_T(N) * B, sm);
    return launch_maybe_pdl(k_col_r2c_loss_fast<N>, grid, dim3(fs_T(N) * B), sm, st, pdl, map, target, ncols, cells,
                            stw, out, out_pitch, out_img, es, ms, scale, gscale, partial, pm, tm, h, nb, err, wait, pf);
}

// Tensor copies of step 4's staging: the N/2 + 1 Hermitian rows in nb boxes of
// h <= 256 rows, h B a multiple of 8 (each box starts on a 128-byte boundary of
// shared memory), all within the block's exchange buffer; false when that does
// not fit, the input is not 16-byte aligned or the map cannot be encoded (the
// kernel then stages with cp.async).
template <int N>
static bool c2r_tma_map(const float2* in, int in_pitch, size_t in_img, int batch, CUtensorMap* map, int* h, int* nb) {
    constexpr int B = fs_Bc2r(N), rows = N / 2 + 1;
    const encode_tiled_fn enc = encode_tiled();
    if (!enc || ((uintptr_t)in & 15) || (in_pitch & 1) || (in_img & 1)) return false;
    const int step = B >= 8 ? 1 : 8 / B;
    int n = (rows + 255) / 256, hh = 0;
    for (;; ++n) {
        hh = (rows + n - 1) / n;
        hh = (hh + step - 1) / step * step;
        if (hh <= 256) break;
    }
    if ((size_t)n * hh * 2 * B > (size_t)FastFft<N, +1, B>::SLOTS) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)in_pitch, (cuuint64_t)rows, (cuuint64_t)batch};
    const cuuint64_t strides[2] = {(cuuint64_t)in_pitch * sizeof(float2), (cuuint64_t)in_img * sizeof(float2)};
    const cuuint32_t box[3] = {(cuuint32_t)(2 * B), (cuuint32_t)hh, 1u};
    const cuuint32_t estr[3] = {1u, 1u, 1u};
    if (enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 3, const_cast<float2*>(in), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return false;
    *h = hh;
    *nb = n;
    return true;
}

template <int N>
cudaError_t go_c2r(const float2* in, int ncols, int in_pitch, size_t in_img, const float2* stw,
                          float mid, float* out, int row0, int rows_out, int out_pitch, size_t out_img,
                          float os, unsigned* tmax, int batch, cudaStream_t st, bool pdl, unsigned* err,
                          long long wait) {
    constexpr int B = fs_Bc2r(N);
    const size_t sm = (size_t)FastFft<N, +1, B>::SLOTS * sizeof(float2);
    cudaError_t e = allow_smem(k_col_c2r_fast<N>, sm);
    if (e != cudaSuccess) return e;
    CUtensorMap map;
    memset(&map, 0, sizeof(map));
    int h = 0, nb = 0;
    if (!err || wait < 0 || !c2r_tma_map<N>(in, in_pitch, in_img, batch, &map, &h, &nb)) nb = 0;
    dim3 grid((ncols + 2 * B - 1) / (2 * B), batch);
    static std::atomic<int> pfc[FT_PF_DEVICES];
    const int pf = prefetch_distance(pfc, k_col_c2r_fast<N>, fs_T(N) * B, sm);
    return launch_maybe_pdl(k_col_c2r_fast<N>, grid, dim3(fs_T(N) * B), sm, st, pdl, in, ncols, in_pitch, in_img, stw,
                            mid, out, row0, rows_out, out_pitch, out_img, os, tmax, map, h, nb, err, wait, pf);
}

template <int N, int INTERP>
static cudaError_t go_rows_i(float2* ws, int W, int Hp, int L, const float2* stw, int batch, cudaStream_t st,
                             bool pdl, unsigned* err, long long wait) {
    constexpr int B = fs_Brow(N);
    const size_t slots = FastFft<N, +1, B>::SLOTS, rows = (size_t)srow_pitch(W, INTERP) * B;
    const size_t sm = (slots > rows ? slots : rows) * sizeof(float2);
    cudaError_t e = allow_smem(k_nvmt_rows_fast<N, INTERP>, sm);
    if (e != cudaSuccess) return e;
    dim3 grid((L + B - 1) / B, batch);
    return launch_maybe_pdl(k_nvmt_rows_fast<N, INTERP>, grid, dim3(fs_T(N) * B), sm, st, pdl, ws, W, Hp, L, stw,
                            err, wait);
}

template <int N>
cudaError_t go_rows(float2* ws, int W, int Hp, int L, int interp, const float2* stw, int batch,
                           cudaStream_t st, bool pdl, unsigned* err, long long wait) {
    return interp == FT_INTERP_LINEAR ? go_rows_i<N, FT_INTERP_LINEAR>(ws, W, Hp, L, stw, batch, st, pdl, err, wait)
                                      : go_rows_i<N, FT_INTERP_CUBIC>(ws, W, Hp, L, stw, batch, st, pdl, err, wait);
}

template <int N, int INTERP>
static cudaError_t go_rows_adj_i(float2* ws, int W, int Hp, int L, const float2* stw, int batch, cudaStream_t st,
                                 bool pdl, LossSum ls) {
    constexpr int B = fs_Brow(N);
    const size_t sm = (size_t)FastFft<N, -1, B>::SLOTS * sizeof(float2);
    cudaError_t e = allow_smem(k_nvmt_rows_adjoint_fast<N, INTERP>, sm);
    if (e != cudaSuccess) return e;
    dim3 grid((L + B - 1) / B, batch);
    return launch_maybe_pdl(k_nvmt_rows_adjoint_fast<N, INTERP>, grid, dim3(fs_T(N) * B), sm, st, pdl, ws, W, Hp, L,
                            stw, ls);
}

template <int N>
cudaError_t go_rows_adj(float2* ws, int W, int Hp, int L, int interp, const float2* stw, int batch, cudaStream_t st,
                        bool pdl, LossSum ls) {
    return interp == FT_INTERP_LINEAR ? go_rows_adj_i<N, FT_INTERP_LINEAR>(ws, W, Hp, L, stw, batch, st, pdl, ls)
                                      : go_rows_adj_i<N, FT_INTERP_CUBIC>(ws, W, Hp, L, stw, batch, st, pdl, ls);
}

// the launchers of length n
#define FT_FAST_INSTANTIATE(n) \
    template cudaError_t go_r2c<n>(const float* in, int rows_in, int ncols, int in_pitch, size_t in_img, int row0, const float2* stw, float2* out, int out_pitch, size_t out_img, float es, float ms, int batch, cudaStream_t st, bool pdl, bool follows_peak, unsigned* err, long long wait); \
    template cudaError_t go_r2c_loss<n>(const float* map, const float* target, int ncols, const float2* stw, float2* out, int out_pitch, size_t out_img, float es, float ms, float scale, float gscale, float* partial, int batch, cudaStream_t st, bool pdl, unsigned* err, long long wait); \
    template cudaError_t go_c2r<n>(const float2* in, int ncols, int in_pitch, size_t in_img, const float2* stw, float mid, float* out, int row0, int rows_out, int out_pitch, size_t out_img, float os, unsigned* tmax, int batch, cudaStream_t st, bool pdl, unsigned* err, long long wait); \
    template cudaError_t go_rows<n>(float2* ws, int W, int Hp, int L, int interp, const float2* stw, int batch, cudaStream_t st, bool pdl, unsigned* err, long long wait); \
    template cudaError_t go_rows_adj<n>(float2* ws, int W, int Hp, int L, int interp, const float2* stw, int batch, cudaStream_t st, bool pdl, LossSum ls);
