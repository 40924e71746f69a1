// The band-limited (chirp-z) NVMT of Sec. IV fused with step 3, on the
// register-resident FFT of fft_fast.cuh: the same chain as k_fourier.cu (see
// there for the derivation),
//     row F (W) --F_W^- --> Fh --pre-chirp, 1/W--> y (M) --F_M^- --x Hc--> --F_M^+-->
//     z --post-chirp, 1/M, support mask, (-1)^k--> V (S) --F_S^+--> G, (-1)^(s+S/2)
// for W = S and M = 2W where both lengths have a compile-time schedule.
//
// A length-M transform has G = fs_T(M) / fs_T(W) times the threads of a length-W
// one (2 for the powers of two), so a block of B fs_T(M) threads takes G B rows:
// the transforms of length W and S run on all G B rows at once, the two of length
// M on B rows at a time in G rounds, and every thread has work in every pass.
// (One round of B rows per block, half of the threads idle in the passes of length
// W and S, took 124 us per 16 x 1024^2, this form 103, with
// the centring factors as rotations and constant shared-memory offsets.)  Between the transforms the rows live
// in a second shared buffer; the exchanges go through the first.  Rows are
// numbered l batch + image, so consecutive rows share the chirp tables of row l
// (pre-chirp W + 1 entries, post-chirp S, chirp spectrum M), which are read from
// memory about once per call, and blocks are full whatever the batch.  The kernel
// is bound by issue and latency at 16 warps per multiprocessor (four transforms
// in a row keep about 170 registers live unbounded; 128 leave at most a few words
// spilled at most widths, 72 to 140 bytes at 576 and 972 and 140 forward, 256 adjoint at
// 1536), so what counts is the number of passes and table loads per row.  Its
// blocks are too large to share a multiprocessor with waiting ones of step 4, so it
// does not trigger early (1024x512, two images: 30.0 us per forward, now 22.0).
#include "fft_fast.cuh"

template <int W>
struct FrShape {
    static constexpr int M = 2 * W, TM = fs_T(M), TW = fs_T(W);
    // rows per round: about 128 threads, or 256 where 128 / TM rows would leave most of
    // a warp empty
    static constexpr int B = TM >= 128 ? 1 : 128 / TM * TM >= 112 ? 128 / TM : 256 / TM;
    static constexpr int G = TM / TW;                          // rounds
    static constexpr int NR = G * B;                           // rows per block
    static constexpr int NT = TM * B;
    // resident blocks of NT threads per multiprocessor the registers are sized for
    static constexpr int MINB = 512 / NT > 0 ? 512 / NT : 1;
    static_assert(G >= 1 && G * TW == TM, "the rows of a block keep every thread busy");
    static constexpr int SX_W = FastFft<W, -1, NR>::SLOTS, SX_M = FastFft<M, -1, B>::SLOTS;
    static constexpr int SX = SX_M > SX_W ? SX_M : SX_W;       // exchange slots
    static constexpr int SLOTS = SX + SX_W;                    // and the rows between the transforms
};

// row of the block's sample index: its frequency l, image and first element
struct FrRow {
    int l;
    bool ok;                // a row of the launch (l = 0, the DC row, included)
    float2* p;
};
__device__ __forceinline__ FrRow fr_row(float2* ws, int r, int L, int batch, int S) {
    FrRow o;
    o.l = r / batch;
    o.ok = o.l < L;
    o.p = ws + ((size_t)(r - o.l * batch) * L + o.l) * S;
    return o;
}

// a copy of a thread index that the compiler takes for a new value: each transform
// of the chain computes its shared-memory addresses from its own copy, so that
// those of one transform are not kept in registers through the others
__device__ __forceinline__ int fr_fresh(int t) {
    asm volatile("" : "+r"(t));
    return t;
}

// the samples k = x' + S/2 of row l inside the support, x' H' / (2 l) in
// [-W/2, W/2 - 1]: lo <= k <= hi
__device__ __forceinline__ void fr_support(int l, int Hp, int W, int S, int& lo, int& hi) {
    lo = ceil_div(-(W / 2) * 2 * l, Hp) + S / 2;
    hi = floor_div((W / 2 - 1) * 2 * l, Hp) + S / 2;
}

template <int W>
__global__ void __launch_bounds__(FrShape<W>::NT, FrShape<W>::MINB)
k_nvmt_rows_fourier_fast(float2* __restrict__ ws, int Hp, int L, int batch, const float2* __restrict__ stw_w,
                         const float2* __restrict__ stw_m, const float2* __restrict__ stw_s,
                         const float2* __restrict__ chirp_u, const float2* __restrict__ chirp_x,
                         const float2* __restrict__ hc) {
    using Sh = FrShape<W>;
    constexpr int M = Sh::M, S = W, B = Sh::B, NR = Sh::NR;
    constexpr int EW = fs_E(W), EM = fs_E(M);
    using FW = FastFft<W, -1, 1, true>;
    using FMf = FastFft<M, -1, 1, true>;
    using FMi = FastFft<M, +1, 1, true>;
    using FS = FastFft<S, +1, 1, true>;
    constexpr int R0W = fs_radix(W, 0), G0W = EW / R0W, RLW = fs_radix(W, fs_nst(W) - 1), GLW = EW / RLW;
    constexpr int R0M = fs_radix(M, 0), G0M = EM / R0M, RLM = fs_radix(M, fs_nst(M) - 1), GLM = EM / RLM;
    static_assert(R0W % 2 == 0 && R0M % 2 == 0, "halves of a row are whole elements of the first pass");
    extern __shared__ __align__(16) float2 sm[];
    float2* rows = sm + Sh::SX;                        // [spos(k)][NR]
    pdl_wait();

    // T consecutive threads per transform, each transform in an exchange buffer of its own
    const int fr = threadIdx.x / Sh::TW, tr0 = threadIdx.x % Sh::TW;
    float2* smr = sm + fr * FW::SLOTS;
    float2* rowr = rows + fr * FW::SLOTS;
    const FrRow rw = fr_row(ws, blockIdx.x * NR + fr, L, batch, S);
    // ---- F_W^- of the block's rows
    {
        const int tr = fr_fresh(tr0);
        float2 v[EW];
#pragma unroll
        for (int m = 0; m < G0W; ++m)
#pragma unroll
            for (int q = 0; q < R0W; ++q)
                v[m * R0W + q] = rw.ok && FT_IN((fs_rotate<W, R0W>(FW::template in_pos<0>(tr, m, q), q)), W, FT_DBG_CHIRP)
                                     ? __ldcg(rw.p + fs_rotate<W, R0W>(FW::template in_pos<0>(tr, m, q), q))
                                     : make_float2(0.f, 0.f);
        FW::template run<0>(v, smr, tr, 0, stw_w);
#pragma unroll
        for (int m = 0; m < GLW; ++m)
#pragma unroll
            for (int q = 0; q < RLW; ++q) {
                const int o = spos_plus(tr, spos(tr), FW::out_pos(0, m, q));
                if (FT_IN(o, FW::SLOTS, FT_DBG_CHIRP)) rowr[o] = v[m * RLW + q];
            }
    }
    __syncthreads();

    const int f = threadIdx.x / Sh::TM, t0 = threadIdx.x % Sh::TM;
    float2* smf = sm + f * FMf::SLOTS;
#pragma unroll 1
    for (int g = 0; g < Sh::G; ++g) {
        const int fg = g * B + f;
        float2* rowg = rows + fg * FW::SLOTS;
        const FrRow rm = fr_row(ws, blockIdx.x * NR + fg, L, batch, S);
        const int t = fr_fresh(t0), st = spos(t);
        const int l = rm.ok ? rm.l : 0;                // the tables' row; rows past the end are not stored
        // ---- y[i] = Fh[u mod W] (halved at u = +-W/2) x pre-chirp, u = i - W/2 (i <= W),
        // 0 beyond: only element q = R0M / 2 of thread 0 (i = W) of the upper half
        float2 v[EM];
        {
            const float2* cu = chirp_u + (size_t)l * (W + 1);
#pragma unroll
            for (int m = 0; m < G0M; ++m)
#pragma unroll
                for (int q = 0; q < R0M; ++q) {
                    constexpr bool quarters = R0M % 4 == 0;        // i < W/2 is decided by q
                    float2 y = make_float2(0.f, 0.f);
                    if (q < R0M / 2 || (q == R0M / 2 && m == 0 && t == 0)) {
                        const int i = FMf::template in_pos<0>(t, m, q);
                        const int c = FMf::template in_pos<0>(0, m, q);
                        int slot;
                        if (quarters)
                            slot = spos_plus(t, st, q < R0M / 4 ? c + W / 2 : c - W / 2);
                        else
                            slot = spos(i < W / 2 ? i + W / 2 : i - W / 2);
                        float2 a = FT_IN(slot, FW::SLOTS, FT_DBG_CHIRP) ? rowg[slot] : make_float2(0.f, 0.f);
                        if (m == 0 && (q == 0 || q == R0M / 2) && t == 0) a = cscale(a, 0.5f);
                        y = cmul(a, __ldg(cu + i));
                    }
                    v[m * R0M + q] = y;
                }
        }
        // ---- F_M^-, times the chirp spectrum, back to the input order, F_M^+
        FMf::template run<0>(v, smf, t, 0, stw_m);
        {
            const float2* hl = hc + (size_t)l * M;
#pragma unroll
            for (int m = 0; m < GLM; ++m)
#pragma unroll
                for (int q = 0; q < RLM; ++q) {
                    const int k = FMf::out_pos(t, m, q);
                    const int o = spos_plus(t, st, FMf::out_pos(0, m, q));
                    if (FT_IN(k, M, FT_DBG_CHIRP) && FT_IN(o, FMf::SLOTS, FT_DBG_FFT_SLOT))
                        smf[o] = cmul(v[m * RLM + q], __ldg(hl + k));
                }
        }
        __syncthreads();
        const int ti = fr_fresh(t0), sti = spos(ti);
#pragma unroll
        for (int m = 0; m < G0M; ++m)
#pragma unroll
            for (int q = 0; q < R0M; ++q) {
                const int o = spos_plus(ti, sti, FMi::template in_pos<0>(0, m, q));
                v[m * R0M + q] = FT_IN(o, FMi::SLOTS, FT_DBG_FFT_SLOT) ? smf[o] : make_float2(0.f, 0.f);
            }
        __syncthreads();
        FMi::template run<0>(v, smf, ti, 0, stw_m);
        // ---- V[k] = z[k] / (W M) x post-chirp inside the support, for k < S = M / 2 (the
        // lower half of the last pass's elements), stored rotated by S/2; the DC row is zero
        {
            const float2* cx = chirp_x + (size_t)l * S;
            const float sc = 1.f / ((float)M * (float)W);
            int lo, hi;
            fr_support(l, Hp, W, S, lo, hi);
            if (l == 0) hi = -1;
#pragma unroll
            for (int m = 0; m < GLM; ++m)
#pragma unroll
                for (int q = 0; q < RLM; ++q) {
                    const int k = FMi::out_pos(ti, m, q);
                    if (RLM % 2 == 0 ? q < RLM / 2 : k < S) {
                        float2 r = make_float2(0.f, 0.f);
                        if (k >= lo && k <= hi) r = cscale(cmul(v[m * RLM + q], __ldg(cx + k)), sc);
                        int slot;
                        if (RLM % 4 == 0)                          // k < S/2 is decided by q
                            slot = spos_plus(ti, sti, FMi::out_pos(0, m, q) + (q < RLM / 4 ? S / 2 : -S / 2));
                        else
                            slot = spos(k < S / 2 ? k + S / 2 : k - S / 2);
                        if (FT_IN(slot, FW::SLOTS, FT_DBG_CHIRP)) rowg[slot] = r;
                    }
                }
        }
    }
    __syncthreads();

    // ---- step 3: F_S^+ of the block's rows.  The centring factors (-1)^k of V and
    // (-1)^(s + S/2) of G are the rotations by S/2 of its input and output
    {
        const int tr = fr_fresh(tr0), str = spos(tr);
        float2 v[EW];
#pragma unroll
        for (int m = 0; m < G0W; ++m)
#pragma unroll
            for (int q = 0; q < R0W; ++q) {
                const int o = spos_plus(tr, str, FS::template in_pos<0>(0, m, q));
                v[m * R0W + q] = FT_IN(o, FW::SLOTS, FT_DBG_CHIRP) ? rowr[o] : make_float2(0.f, 0.f);
            }
        FS::template run<0>(v, smr, tr, 0, stw_s);
        if (rw.ok) {
#pragma unroll
            for (int m = 0; m < GLW; ++m)
#pragma unroll
                for (int q = 0; q < RLW; ++q) {
                    const int o = fs_rotate<S, RLW>(FS::out_pos(tr, m, q), q);
                    if (FT_IN(o, S, FT_DBG_CHIRP)) rw.p[o] = v[m * RLW + q];
                }
        }
    }
}

// Transpose of the above (see k_nvmt_rows_fourier_adj in k_fourier.cu): with
// O the output sign, D_x the post-chirp / 1/M / mask / (-1)^k, D_h the chirp
// spectrum, D_u the pre-chirp and P the re-indexing u mod W with its weights,
//     gF = F_W^+ P^T conj(D_u) F_M^+ conj(D_h) F_M^- conj(D_x) F_S^- O gG.
// conj(D_u) is applied as F_M^+ ends, and P^T stores entry i = u + W/2 at u mod
// W; the two Nyquist entries i = 0 and i = W share index W/2, so the second goes
// to a slot of its own and is added when F_W^+ reads index W/2.
template <int W>
__global__ void __launch_bounds__(FrShape<W>::NT, FrShape<W>::MINB)
k_nvmt_rows_fourier_adj_fast(float2* __restrict__ ws, int Hp, int L, int batch, const float2* __restrict__ stw_w,
                             const float2* __restrict__ stw_m, const float2* __restrict__ stw_s,
                             const float2* __restrict__ chirp_u, const float2* __restrict__ chirp_x,
                             const float2* __restrict__ hc) {
    using Sh = FrShape<W>;
    constexpr int M = Sh::M, S = W, B = Sh::B, NR = Sh::NR;
    constexpr int EW = fs_E(W), EM = fs_E(M);
    using FS = FastFft<S, -1, 1, true>;
    using FMf = FastFft<M, -1, 1, true>;
    using FMi = FastFft<M, +1, 1, true>;
    using FW = FastFft<W, +1, 1, true>;
    constexpr int R0W = fs_radix(W, 0), G0W = EW / R0W, RLW = fs_radix(W, fs_nst(W) - 1), GLW = EW / RLW;
    constexpr int R0M = fs_radix(M, 0), G0M = EM / R0M, RLM = fs_radix(M, fs_nst(M) - 1), GLM = EM / RLM;
    extern __shared__ __align__(16) float2 sm[];
    float2* rows = sm + Sh::SX;
    __shared__ float2 nyq[NR];
    pdl_wait();

    // T consecutive threads per transform, each transform in an exchange buffer of its own
    const int fr = threadIdx.x / Sh::TW, tr0 = threadIdx.x % Sh::TW;
    float2* smr = sm + fr * FW::SLOTS;
    float2* rowr = rows + fr * FW::SLOTS;
    const FrRow rw = fr_row(ws, blockIdx.x * NR + fr, L, batch, S);
    // ---- O, F_S^-, (-1)^k: rotations by S/2 of the input and the output
    {
        const int tr = fr_fresh(tr0);
        float2 v[EW];
#pragma unroll
        for (int m = 0; m < G0W; ++m)
#pragma unroll
            for (int q = 0; q < R0W; ++q)
                v[m * R0W + q] = rw.ok && FT_IN((fs_rotate<S, R0W>(FS::template in_pos<0>(tr, m, q), q)), S, FT_DBG_CHIRP)
                                     ? __ldcg(rw.p + fs_rotate<S, R0W>(FS::template in_pos<0>(tr, m, q), q))
                                     : make_float2(0.f, 0.f);
        FS::template run<0>(v, smr, tr, 0, stw_s);
#pragma unroll
        for (int m = 0; m < GLW; ++m)
#pragma unroll
            for (int q = 0; q < RLW; ++q) {
                const int c = FS::out_pos(0, m, q);
                const int slot = RLW % 2 == 0 ? spos_plus(tr, spos(tr), q < RLW / 2 ? c + S / 2 : c - S / 2)
                                              : spos(fs_rotate<S, RLW>(tr + c, q));
                if (FT_IN(slot, FS::SLOTS, FT_DBG_CHIRP)) rowr[slot] = v[m * RLW + q];
            }
    }
    __syncthreads();

    const int f = threadIdx.x / Sh::TM, t0 = threadIdx.x % Sh::TM;
    float2* smf = sm + f * FMf::SLOTS;
#pragma unroll 1
    for (int g = 0; g < Sh::G; ++g) {
        const int fg = g * B + f;
        float2* rowg = rows + fg * FW::SLOTS;
        const FrRow rm = fr_row(ws, blockIdx.x * NR + fg, L, batch, S);
        const int t = fr_fresh(t0), st = spos(t);
        const int l = rm.ok ? rm.l : 0;
        // ---- conj(D_x) on k < S = M / 2, zero beyond and for the DC row, F_M^-
        float2 v[EM];
        {
            const float2* cx = chirp_x + (size_t)l * S;
            const float sc = 1.f / ((float)M * (float)W);
            int lo, hi;
            fr_support(l, Hp, W, S, lo, hi);
            if (l == 0) hi = -1;
#pragma unroll
            for (int m = 0; m < G0M; ++m)
#pragma unroll
                for (int q = 0; q < R0M; ++q) {
                    float2 r = make_float2(0.f, 0.f);
                    if (q < R0M / 2) {
                        const int k = FMf::template in_pos<0>(t, m, q);
                        if (k >= lo && k <= hi) {
                            const float2 c = __ldg(cx + k);
                            const int o = spos_plus(t, st, FMf::template in_pos<0>(0, m, q));
                            const float2 a = FT_IN(o, FS::SLOTS, FT_DBG_CHIRP) ? rowg[o] : make_float2(0.f, 0.f);
                            r = cscale(cmul(a, make_float2(c.x, -c.y)), sc);
                        }
                    }
                    v[m * R0M + q] = r;
                }
        }
        FMf::template run<0>(v, smf, t, 0, stw_m);
        {
            const float2* hl = hc + (size_t)l * M;
#pragma unroll
            for (int m = 0; m < GLM; ++m)
#pragma unroll
                for (int q = 0; q < RLM; ++q) {
                    const int k = FMf::out_pos(t, m, q);
                    const float2 h = __ldg(hl + k);
                    const int o = spos_plus(t, st, FMf::out_pos(0, m, q));
                    if (FT_IN(k, M, FT_DBG_CHIRP) && FT_IN(o, FMf::SLOTS, FT_DBG_FFT_SLOT))
                        smf[o] = cmul(v[m * RLM + q], make_float2(h.x, -h.y));
                }
        }
        __syncthreads();
        const int ti = fr_fresh(t0), sti = spos(ti);
#pragma unroll
        for (int m = 0; m < G0M; ++m)
#pragma unroll
            for (int q = 0; q < R0M; ++q) {
                const int o = spos_plus(ti, sti, FMi::template in_pos<0>(0, m, q));
                v[m * R0M + q] = FT_IN(o, FMi::SLOTS, FT_DBG_FFT_SLOT) ? smf[o] : make_float2(0.f, 0.f);
            }
        __syncthreads();
        FMi::template run<0>(v, smf, ti, 0, stw_m);
        // ---- conj(D_u) and P^T on the entries i = u + W/2 <= W (halved at u = +-W/2)
        {
            const float2* cu = chirp_u + (size_t)l * (W + 1);
#pragma unroll
            for (int m = 0; m < GLM; ++m)
#pragma unroll
                for (int q = 0; q < RLM; ++q) {
                    const int i = FMi::out_pos(ti, m, q);
                    if (RLM % 2 == 0 ? (q < RLM / 2 || (q == RLM / 2 && m == 0 && ti == 0)) : i <= W) {
                        const float2 c = __ldg(cu + i);
                        float2 r = cmul(v[m * RLM + q], make_float2(c.x, -c.y));
                        if (i == 0 || i == W) r = cscale(r, 0.5f);
                        if (i == W)
                            nyq[fg] = r;
                        else if (FT_IN(spos(i < W / 2 ? i + W / 2 : i - W / 2), FW::SLOTS, FT_DBG_CHIRP))
                            rowg[spos(i < W / 2 ? i + W / 2 : i - W / 2)] = r;
                    }
                }
        }
    }
    __syncthreads();

    // ---- F_W^+ (the DC row's gradient is zero: its V is); the weight (-1)^u is a
    // rotation of the result by W/2
    {
        const int tr = fr_fresh(tr0), str = spos(tr);
        float2 v[EW];
#pragma unroll
        for (int m = 0; m < G0W; ++m)
#pragma unroll
            for (int q = 0; q < R0W; ++q) {
                const int o = spos_plus(tr, str, FW::template in_pos<0>(0, m, q));
                float2 a = FT_IN(o, FW::SLOTS, FT_DBG_CHIRP) ? rowr[o] : make_float2(0.f, 0.f);
                if (FW::template in_pos<0>(tr, m, q) == W / 2) a = cadd(a, nyq[fr]);
                v[m * R0W + q] = a;
            }
        FW::template run<0>(v, smr, tr, 0, stw_w);
        if (rw.ok) {
#pragma unroll
            for (int m = 0; m < GLW; ++m)
#pragma unroll
                for (int q = 0; q < RLW; ++q) {
                    const int o = fs_rotate<W, RLW>(FW::out_pos(tr, m, q), q);
                    if (FT_IN(o, W, FT_DBG_CHIRP)) rw.p[o] = v[m * RLW + q];
                }
        }
    }
}

FT_DEBUG_READER(ft_debug_read_fourier_fast)

// ------------------------------------------------------------------ dispatch
#define FR_FAST_LENGTHS(X) \
    X(128) X(144) X(162) X(192) X(216) X(256) X(288) X(324) X(384) X(432) X(486) X(512) X(576) X(648) X(768) X(864) \
    X(972) X(1024) X(1152) X(1536) X(2048)

bool fourier_fast_ok(int W, int M, int S) {
    if (W != S || M != 2 * W) return false;
    switch (W) {
#define X(n) case n:
        FR_FAST_LENGTHS(X)
#undef X
        return true;
    }
    return false;
}

template <int N>
static cudaError_t go_fourier(bool adj, float2* ws, int Hp, int L, int batch, const float2* stw_w,
                              const float2* stw_m, const float2* stw_s, const float2* cu, const float2* cx,
                              const float2* hc, cudaStream_t st, bool pdl) {
    using Sh = FrShape<N>;
    const size_t sm = (size_t)Sh::SLOTS * sizeof(float2);
    const auto k = adj ? k_nvmt_rows_fourier_adj_fast<N> : k_nvmt_rows_fourier_fast<N>;
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    const unsigned blocks = ((unsigned)L * (unsigned)batch + Sh::NR - 1) / Sh::NR;
    return launch_maybe_pdl(k, dim3(blocks), dim3(Sh::NT), sm, st, pdl, ws, Hp, L, batch, stw_w, stw_m, stw_s, cu, cx,
                            hc);
}

cudaError_t launch_nvmt_rows_fourier_fast(bool adjoint, float2* ws, int W, int S, int Hp, int L, const FftLen& fw,
                                          const FftLen& fm, const FftLen& fs, const float2* chirp_u,
                                          const float2* chirp_x, const float2* hc, int batch, cudaStream_t st,
                                          bool pdl) {
    if (!fourier_fast_ok(W, fm.N, S) || !fw.stw || !fm.stw || !fs.stw) return cudaErrorNotSupported;
    switch (W) {
#define X(n) \
    case n: return go_fourier<n>(adjoint, ws, Hp, L, batch, fw.stw, fm.stw, fs.stw, chirp_u, chirp_x, hc, st, pdl);
        FR_FAST_LENGTHS(X)
#undef X
    }
    return cudaErrorNotSupported;
}
