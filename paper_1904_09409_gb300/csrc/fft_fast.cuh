// Register-resident Stockham FFT with compile-time schedules.
//
// For the lengths below every thread of a transform holds E elements (16 for the
// powers of two, 8 at 64; 12, 18, 24 or 36 when N has a factor 3) in registers; a transform of length N uses T = N / E
// threads, and a block runs B transforms side by side (transform f's sample n
// lives at smem[spos(n) * B + f]).  A pass with radix R and P = product of the
// earlier radices does, for butterfly i in [0, N/R) with k = i mod P:
//     inputs x[i + q N/R] * w^{q k N/(P R)},  q < R   (w = exp(SIGN 2 pi i / N))
//     radix-R DFT in registers
//     outputs y[(i - k) R + k + q P]
// so the result comes out in natural order (self-sorting).  Each pass costs one
// shared-memory round trip; the first pass loads and the last pass stores
// through caller code, which lets the column and row kernels read and write
// global memory directly.  All index arithmetic is by compile-time constants.
//
// Twiddles come from a per-length table (FP64 values rounded to FP32, built on
// the host): for pass s >= 1, row k of a full table holds w_k^q, q = 1 .. R-1,
// w_k = exp(-2 pi i k / (P R)); row k of a seed table holds only some of these
// powers and a thread builds the others as products (at most three for radix 16: a
// few FP32 roundings).  Entries are stored in pairs that load as float4.  A
// radix-16 group reads 8 float4 of a full row against 2 of a seed
// row and 11 complex products: the row kernels (steps 2-3, scattered rows k
// per lane) run faster on seed tables (103 against 112 us per 64 x 1024^2),
// the column kernels on full ones (step 4: 121 against 128 us).
#pragma once

#include "ft_internal.cuh"

// Schedules: E samples per thread and the radices of the passes (each divides
// E).  Powers of two hold 16 samples (radix 16, 8, 4, 2 passes); lengths with
// factors of 3 take the E whose divisors give few passes: 12 (radices 12, 6, 4,
// 3, 2), 18 (18, 9, 6, 3, 2), 24 (24, 12, 8, 6) or 36 (18, 12).  Steps 1 / 2-3 / 4 of
// 16 Mpx in square images, us, against the generic shared-memory kernels: 486^2
// 38 / 38 / 32 (113 / 187 / 89), 1152^2 36 / 37 / 34 (109 / 132 / 86), 1944^2
// 43 / 35 / 36 (127 / 191 / 104), 3456^2 51 / 36 / 46 (199 / 182 / 162).  Where two
// schedules compete the choice is measured too: 1152 as 12 12 8 with E = 24
// against 12 12 4 2 with E = 12 36 / 37 / 34 (44 / 35 / 42), 2304 as 24 12 8 against
// 12 12 4 4 40 / 30 / 41 (55 / 35 / 53), 576 as 24 24 against 12 12 4 30 / 35 / 28
// (35 / 35 / 37); but 288 as 12 12 2 against 24 12 29 / 38 / 28 (29 / 47 / 27), and
// 1296 as 6 6 6 6 with E = 12 against 12 12 9 with E = 36, which spills, the same
// forward and a faster adjoint (50 against 58).  2592 and 3888 hold 36 all the same
// (step 1 of 2592 spills 252 bytes, step 4 and the loss kernel about 140): forward and
// backward of two 2592^2 images 99 and 105 us (generic 374 and 363), of one 3888^2 125
// and 131 (476 and 454); schedules with fewer samples there were not compared.  192, 384, 768 and 1536 start with
// radix 12 and save a pass against radix 4 passes and a last radix 3 (384^2 40 / 42 /
// 34 -> 37 / 35 / 32, 1536^2 51 / 41 / 49 -> 47 / 40 / 45).  The shortest, against the
// generic kernels: 64^2 26 / 31 / 26 (65 / 141 / 54; as 16 4 with E = 16 26 / 37 / 24),
// 72^2 33 / 35 / 37 (90 / 144 / 78), 96^2 26 / 35 / 29 (67 / 138 / 56; as 12 4 2 32 / 37 /
// 33), 108^2 28 / 35 / 31 (85 / 142 / 74; as 12 3 3 33 / 43 / 34).
struct FsSched {
    int N, E, nst, r[6];
};
__host__ __device__ constexpr FsSched fs_sched(int N) {
    switch (N) {
        case 64: return {64, 8, 2, {8, 8}};
        case 72: return {72, 12, 2, {12, 6}};
        case 96: return {96, 24, 2, {24, 4}};
        case 108: return {108, 18, 2, {18, 6}};
        case 128: return {128, 16, 2, {16, 8}};
        case 144: return {144, 12, 2, {12, 12}};
        case 162: return {162, 18, 2, {18, 9}};
        case 192: return {192, 12, 3, {12, 4, 4}};
        case 216: return {216, 12, 3, {12, 6, 3}};
        case 256: return {256, 16, 2, {16, 16}};
        case 288: return {288, 12, 3, {12, 12, 2}};
        case 324: return {324, 18, 2, {18, 18}};
        case 384: return {384, 12, 4, {12, 4, 4, 2}};
        case 432: return {432, 12, 3, {12, 12, 3}};
        case 486: return {486, 18, 3, {18, 9, 3}};
        case 512: return {512, 16, 3, {16, 8, 4}};
        case 576: return {576, 24, 2, {24, 24}};
        case 648: return {648, 18, 3, {18, 18, 2}};
        case 768: return {768, 12, 4, {12, 4, 4, 4}};
        case 864: return {864, 12, 3, {12, 12, 6}};
        case 972: return {972, 18, 3, {18, 18, 3}};
        case 1024: return {1024, 16, 3, {16, 16, 4}};
        case 1152: return {1152, 24, 3, {12, 12, 8}};
        case 1296: return {1296, 12, 4, {6, 6, 6, 6}};
        case 1458: return {1458, 18, 3, {18, 9, 9}};
        case 1536: return {1536, 12, 5, {12, 4, 4, 4, 2}};
        case 1728: return {1728, 12, 3, {12, 12, 12}};
        case 1944: return {1944, 18, 3, {18, 18, 6}};
        case 2048: return {2048, 16, 3, {16, 16, 8}};
        case 2304: return {2304, 24, 3, {24, 12, 8}};
        case 2592: return {2592, 36, 3, {18, 12, 12}};
        case 2916: return {2916, 18, 3, {18, 18, 9}};
        case 3072: return {3072, 24, 4, {8, 8, 8, 6}};
        case 3456: return {3456, 24, 3, {24, 12, 12}};
        case 3888: return {3888, 36, 3, {18, 18, 12}};
        case 4096: return {4096, 16, 3, {16, 16, 16}};
        case 8192: return {8192, 16, 4, {16, 16, 16, 2}};
    }
    return {0, 1, 0, {0}};
}
__host__ __device__ constexpr bool fs_has(int N) { return fs_sched(N).N != 0; }
__host__ __device__ constexpr int fs_E(int N) { return fs_sched(N).E; }
__host__ __device__ constexpr int fs_T(int N) { return N / fs_E(N); }
__host__ __device__ constexpr int fs_nst(int N) { return fs_sched(N).nst; }
__host__ __device__ constexpr int fs_radix(int N, int s) { return fs_sched(N).r[s]; }
__host__ __device__ constexpr int fs_P(int N, int s) {
    int p = 1;
    for (int j = 0; j < s; ++j) p *= fs_radix(N, j);
    return p;
}
// entries of a table row: a full table holds the powers 1 .. R - 1, a seed table
// of radix 12 and above the powers 1, 2, 4, 8, ..., below that 1 .. b and the
// multiples of b (b = 3 for R = 3, 6, 9, 2 for R = 4, else 4), as many float4
// but with every other power one product of two entries
__host__ __device__ constexpr int fs_seedbase(int R) { return R == 3 || R == 6 || R == 9 ? 3 : R == 4 ? 2 : 4; }
__host__ __device__ constexpr int fs_nent(int R, bool seed) {
    if (!seed) return R - 1;
    const int b = fs_seedbase(R);
    if (R < 12) return R <= b ? R - 1 : b + (R - 1) / b - 1;
    int n = 0;
    while ((1 << n) < R) ++n;
    return n;
}
// the exponent of entry j, and the float4 (pairs of entries) a row takes
__host__ __device__ constexpr int fs_entexp(int R, bool seed, int j) {
    const int b = fs_seedbase(R);
    return !seed ? j + 1 : R >= 12 ? 1 << j : j < b ? j + 1 : (j - b + 2) * b;
}
__host__ __device__ constexpr int fs_pairs(int R, bool seed) { return (fs_nent(R, seed) + 1) / 2; }
// float4 index of pair h of row k of a pass with P rows: by rows (the pairs of a
// row adjacent), or by pairs (those of successive rows adjacent) in the seed
// tables of the row kernels, whose warps hold up to 32 rows, and in the full
// tables of the long column lengths, whose warps hold 8 to 16: a load then
// touches one or two lines instead of one per row (steps 1 and 4 of four 4096^2
// images 180 / 178 -> 169 / 162 us, 8192 in 16 Mpx 72 / 70 -> 62 / 60; equal
// within noise at 1024 and below, with 4 rows per warp or fewer)
__host__ __device__ constexpr bool fs_bypairs(int N, bool seed) { return seed || N > 1024; }
__host__ __device__ constexpr int fs_pairpos(int N, int R, int P, bool seed, int h, int k) {
    return fs_bypairs(N, seed) ? h * P + k : k * fs_pairs(R, seed) + h;
}
__host__ __device__ constexpr int fs_twoff(int N, int s, bool seed) {
    int o = 0;
    for (int j = 1; j < s; ++j) o += fs_P(N, j) * 2 * fs_pairs(fs_radix(N, j), seed);
    return o;
}
__host__ __device__ constexpr int fs_twsize(int N, bool seed) { return fs_twoff(N, fs_nst(N), seed); }
// transforms per block for the column R2C kernels (512 threads, 256 up to length
// 512: 32 x 512^2 steps 1 and its transpose 27.1 -> 24.2 us; for N >= 4096,
// 1024 threads so that a block still reads 4 column pairs = 32-byte row
// segments), the column C2R kernel (256 threads, at least 4 column pairs, so
// 512 threads for N = 1536, 2048; for N = 1024 512 threads, 8 column pairs:
// 98 us per 64 x 1024^2 against 109 with 256, and the peak pass is faster on the
// 16 x 16 tiles that gives) and the row kernels (64 threads, T consecutive ones per
// row, so that a warp reads and writes consecutive samples: 64 x 1024^2 84 us, with
// 128 threads 86, with 256 97; 16 Mpx of 256^2 23 us, with 128 threads and the rows
// interleaved over the lanes 34, of 128^2 27 against 57)
//
// The lengths with radices 6 to 24 (fs_wide) hold more than 64 registers' worth of
// samples per thread (E = 18, 24, 36) or more temporaries (E = 12): fs_resident
// threads share a multiprocessor (72, 80 or 112 registers each), and a column
// block takes 8 column pairs (64-byte image rows) where at most 512 threads then
// transform them, else 4 (16 or 32 where it would fall below 200 threads).
// Measured as above: 16 pairs instead of 8 at 324 32 / 31 against 30 / 28 (steps 1 /
// 4), at 648 46 / 43 against 35 / 31; 8 instead of 4 at 864 47 / 46 against 36 / 34;
// 2 instead of 4 at 2304 and above slower or equal.
__host__ __device__ constexpr int fs_clampB(int v, int hi) { return v < 1 ? 1 : (v > hi ? hi : v); }
__host__ __device__ constexpr bool fs_wide(int N) { return N % 3 == 0 && N != 192 && N != 384 && N != 768 && N != 1536; }
__host__ __device__ constexpr int fs_resident(int N) {
    return !fs_wide(N) || fs_E(N) == 12 ? 1024 : fs_E(N) == 18 ? 864 : fs_E(N) == 24 ? 768 : 576;
}
__host__ __device__ constexpr int fs_minblocks(int N, int threads) {
    return fs_resident(N) / threads > 0 ? fs_resident(N) / threads : 1;
}
__host__ __device__ constexpr int fs_Bwide(int N) {
    return fs_T(N) * 32 <= 288 ? 32 : fs_T(N) * 16 <= 192 ? 16 : fs_T(N) * 8 <= 512 ? 8 : 4;
}
__host__ __device__ constexpr int fs_Bcol(int N) {
    return fs_wide(N) ? fs_Bwide(N) : fs_T(N) >= 256 ? 1024 / fs_T(N) : fs_clampB((N <= 512 ? 256 : 512) / fs_T(N), 32);
}
__host__ __device__ constexpr int fs_Bc2r(int N) {
    return fs_wide(N) ? fs_Bwide(N)
         : fs_T(N) >= 256 ? 1024 / fs_T(N)
                          : fs_clampB(N == 1024 ? 512 / fs_T(N) : (256 / fs_T(N) < 4 ? 4 : 256 / fs_T(N)), 32);
}
// rows per block of the row kernels: 64 threads for the powers of two and 3 x 2^a up
// to 1536 (one row from length 1024 on), and for the other lengths, whose T is no
// multiple of a warp, the count that fills its last warp best with at most 144
__host__ __device__ constexpr int fs_Brow(int N) {
    if (!fs_wide(N)) return fs_clampB(64 / fs_T(N), 16);
    int best = 1, num = 0, den = 1;
    for (int b = 1; b == 1 || b * fs_T(N) <= 144; ++b) {
        const int used = b * fs_T(N), alloc = (used + 31) / 32 * 32;
        if (used >= 48 && used * den > num * alloc) {
            best = b;
            num = used;
            den = alloc;
        }
    }
    return best;
}
// padded shared-memory slot of sample n (one spare slot every 16 samples
// spreads the strided stores of the first pass over the banks)
__host__ __device__ constexpr int spos(int n) { return n + (n >> 4); }
__host__ __device__ constexpr int fs_slots(int N) { return spos(N - 1) + 1; }
// the slot of sample n + c, given sn = spos(n): for a constant c that is a
// multiple of 16 a constant distance, which becomes the access's immediate offset
__device__ __forceinline__ int spos_plus(int n, int sn, int c) { return (c & 15) == 0 ? sn + c + (c >> 4) : spos(n + c); }
// position pos of element q of a pass with radix R, rotated by half the length
template <int N, int R>
__device__ __forceinline__ int fs_rotate(int pos, int q) {
    return (R % 2 == 0 ? q < R / 2 : pos < N / 2) ? pos + N / 2 : pos - N / 2;
}

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async8(void* smem_dst, const void* gmem_src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(smem_dst)),
                 "l"(gmem_src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

template <int SIGN>
__device__ __forceinline__ float2 tw_sign(float2 w) { return SIGN > 0 ? make_float2(w.x, -w.y) : w; }

// w[q] = w_k^q (conjugated for SIGN > 0), q = 1 .. R-1, from row k of the table wp
// of a pass: the entries are read, the powers a seed table lacks are products of
// two earlier ones
template <int N, int R, int P, int SIGN, bool SEED>
__device__ __forceinline__ void tw_powers(const float4* __restrict__ wp, int k, float2 (&w)[R]) {
    constexpr int NE = fs_nent(R, SEED), SB = fs_seedbase(R);
    wp += fs_pairpos(N, R, P, SEED, 0, k);
#pragma unroll
    for (int h = 0; h < fs_pairs(R, SEED); ++h) {
        const float4 a = __ldg(wp + fs_pairpos(N, R, P, SEED, h, 0));
        w[fs_entexp(R, SEED, 2 * h)] = tw_sign<SIGN>(make_float2(a.x, a.y));
        if (2 * h + 1 < NE) w[fs_entexp(R, SEED, 2 * h + 1)] = tw_sign<SIGN>(make_float2(a.z, a.w));
    }
    if constexpr (SEED && R < 12) {
#pragma unroll
        for (int q = SB + 1; q < R; ++q)
            if (q % SB != 0) w[q] = cmul(w[q - q % SB], w[q % SB]);
    } else if constexpr (SEED) {
#pragma unroll
        for (int b = 2; b < R; b *= 2)
#pragma unroll
            for (int q = b + 1; q < 2 * b && q < R; ++q) w[q] = cmul(w[q - b], w[b]);
    }
}

// radix 9 as 3 x 3 with the internal twiddles exp(SIGN 2 pi i m / 9)
template <int SIGN>
struct Dft<9, SIGN> {
    __device__ __forceinline__ static void run(float2* u) {
        const float c1 = 0.76604444311897803520f, s1 = 0.64278760968653932632f;    // 2 pi / 9
        const float c2 = 0.17364817766693034885f, s2 = 0.98480775301220805937f;    // 4 pi / 9
        const float c4 = -0.93969262078590838405f, s4 = 0.34202014332566873304f;   // 8 pi / 9
        float2 a[3][3];
#pragma unroll
        for (int n2 = 0; n2 < 3; ++n2) {
            float2 t[3] = {u[n2], u[3 + n2], u[6 + n2]};
            Dft<3, SIGN>::run(t);
#pragma unroll
            for (int k1 = 0; k1 < 3; ++k1) a[n2][k1] = t[k1];
        }
        a[1][1] = cmul(a[1][1], make_float2(c1, SIGN * s1));
        a[1][2] = cmul(a[1][2], make_float2(c2, SIGN * s2));
        a[2][1] = cmul(a[2][1], make_float2(c2, SIGN * s2));
        a[2][2] = cmul(a[2][2], make_float2(c4, SIGN * s4));
#pragma unroll
        for (int k1 = 0; k1 < 3; ++k1) {
            float2 t[3] = {a[0][k1], a[1][k1], a[2][k1]};
            Dft<3, SIGN>::run(t);
#pragma unroll
            for (int k2 = 0; k2 < 3; ++k2) u[k1 + 3 * k2] = t[k2];
        }
    }
};

// radix A B with A, B coprime by the prime-factor map: with n = (B a + A b) mod
// A B and k = the residue pair (k mod A, k mod B), exp(2 pi i n k / (A B)) splits
// into exp(2 pi i a k / A) exp(2 pi i b k / B), so no internal twiddles are needed
template <int A, int B, int SIGN>
struct DftCoprime {
    __device__ __forceinline__ static void run(float2* u) {
        float2 x[A][B];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            float2 t[A];
#pragma unroll
            for (int a = 0; a < A; ++a) t[a] = u[(B * a + A * b) % (A * B)];
            Dft<A, SIGN>::run(t);
#pragma unroll
            for (int a = 0; a < A; ++a) x[a][b] = t[a];
        }
#pragma unroll
        for (int a = 0; a < A; ++a) Dft<B, SIGN>::run(x[a]);
#pragma unroll
        for (int k = 0; k < A * B; ++k) u[k] = x[k % A][k % B];
    }
};
template <int SIGN> struct Dft<6, SIGN> : DftCoprime<2, 3, SIGN> {};
template <int SIGN> struct Dft<12, SIGN> : DftCoprime<4, 3, SIGN> {};
template <int SIGN> struct Dft<18, SIGN> : DftCoprime<2, 9, SIGN> {};
template <int SIGN> struct Dft<24, SIGN> : DftCoprime<8, 3, SIGN> {};

// radix-16 as 4 x 4 with the internal twiddles exp(SIGN 2 pi i m / 16)
template <int SIGN>
struct Dft<16, SIGN> {
    __device__ __forceinline__ static void run(float2* u) {
        const float c1 = 0.92387953251128675613f;   // cos(pi/8)
        const float s1 = 0.38268343236508977173f;   // sin(pi/8)
        const float r = 0.70710678118654752440f;    // sqrt(2)/2
        float2 a[4][4];
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) {
            float2 t[4] = {u[n2], u[4 + n2], u[8 + n2], u[12 + n2]};
            Dft<4, SIGN>::run(t);
#pragma unroll
            for (int k1 = 0; k1 < 4; ++k1) a[n2][k1] = t[k1];
        }
        const float2 w1 = make_float2(c1, SIGN * s1), w2 = make_float2(r, SIGN * r);
        const float2 w3 = make_float2(s1, SIGN * c1), w6 = make_float2(-r, SIGN * r);
        const float2 w9 = make_float2(-c1, -SIGN * s1);
        a[1][1] = cmul(a[1][1], w1);
        a[1][2] = cmul(a[1][2], w2);
        a[1][3] = cmul(a[1][3], w3);
        a[2][1] = cmul(a[2][1], w2);
        a[2][2] = cmul_si<SIGN>(a[2][2]);
        a[2][3] = cmul(a[2][3], w6);
        a[3][1] = cmul(a[3][1], w3);
        a[3][2] = cmul(a[3][2], w6);
        a[3][3] = cmul(a[3][3], w9);
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            float2 t[4] = {a[0][k1], a[1][k1], a[2][k1], a[3][k1]};
            Dft<4, SIGN>::run(t);
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) u[k1 + 4 * k2] = t[k2];
        }
    }
};

// SEED: the twiddle table is a seed table (the row kernels' tables), else full
template <int N, int SIGN, int B, bool SEED = false>
struct FastFft {
    static constexpr int E = fs_E(N);
    static constexpr int T = N / E;
    static constexpr int NS = fs_nst(N);
    static constexpr int SLOTS = fs_slots(N) * B;      // float2 slots of shared memory

    // sample index of element (m, q) of pass s for thread t of a transform
    template <int s>
    __device__ __forceinline__ static int in_pos(int t, int m, int q) {
        return t + m * T + q * (N / fs_radix(N, s));
    }
    // sample index of output element (m, q) of the last pass
    __device__ __forceinline__ static int out_pos(int t, int m, int q) {
        return t + m * T + q * (N / fs_radix(N, NS - 1));
    }

    template <int s>
    __device__ __forceinline__ static void compute(float2 (&v)[E], int t, const float2* __restrict__ stw) {
        constexpr int R = fs_radix(N, s), P = fs_P(N, s), G = E / R;
#pragma unroll
        for (int m = 0; m < G; ++m) {
            if constexpr (P > 1) {
                const int k = (t + m * T) % P;
                float2 w[R];
                tw_powers<N, R, P, SIGN, SEED>(reinterpret_cast<const float4*>(stw + fs_twoff(N, s, SEED)), k, w);
#pragma unroll
                for (int q = 1; q < R; ++q) v[m * R + q] = cmul(v[m * R + q], w[q]);
            }
            Dft<R, SIGN>::run(&v[m * R]);
        }
    }

    template <int s>
    __device__ __forceinline__ static void store(const float2 (&v)[E], float2* sm, int t, int f) {
        constexpr int R = fs_radix(N, s), P = fs_P(N, s), G = E / R;
#pragma unroll
        for (int m = 0; m < G; ++m) {
            const int i = t + m * T;
            const int k = i % P;
            const int j = (i - k) * R + k, sj = spos(j);
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const int o = spos_plus(j, sj, q * P) * B + f;
                if (FT_IN(o, SLOTS, FT_DBG_FFT_SLOT)) sm[o] = v[m * R + q];
            }
        }
    }

    template <int s>
    __device__ __forceinline__ static void load(float2 (&v)[E], const float2* sm, int t, int f) {
        constexpr int R = fs_radix(N, s), G = E / R;
        const int st = spos(t);
#pragma unroll
        for (int m = 0; m < G; ++m)
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const int k = spos_plus(t, st, in_pos<s>(0, m, q)) * B + f;
                v[m * R + q] = FT_IN(k, SLOTS, FT_DBG_FFT_SLOT) ? sm[k] : make_float2(0.f, 0.f);
            }
    }

    // The barriers of run<s> for the threads of a block that hold no transform of
    // this length (a block whose stages use transforms of different lengths).
    template <int s>
    __device__ __forceinline__ static void idle() {
        if constexpr (s + 1 < NS) {
            __syncthreads();
            __syncthreads();
            idle<s + 1>();
        }
    }

    // Passes s .. NS-1.  On entry v holds the inputs of pass s in (m, q) order;
    // on return it holds the outputs of the last pass, element (m, q) being the
    // sample out_pos(t, m, q).  Every thread of the block must call it; it leaves
    // shared memory free to reuse (the last barrier follows the last read).
    template <int s>
    __device__ __forceinline__ static void run(float2 (&v)[E], float2* sm, int t, int f,
                                               const float2* __restrict__ stw) {
        compute<s>(v, t, stw);
        if constexpr (s + 1 < NS) {
            store<s>(v, sm, t, f);
            __syncthreads();
            load<s + 1>(v, sm, t, f);
            __syncthreads();
            run<s + 1>(v, sm, t, f, stw);
        }
    }
};

// launchers of the fixed-length kernels (k_fast.cu); they return
// cudaErrorNotSupported when N has no schedule

// (pdl: launched with programmatic stream serialisation, the blocks waiting for
// the predecessor before they read or write; follows_peak (with pdl): the
// predecessor is the peak pass of the previous batch of ft_detect_batches, not
// waited for (see k_col_r2c_fast); err, wait: with err given, the image columns
// are staged through tensor copies whose bounded waits set bit 3 of *err when
// they run out)
cudaError_t launch_col_r2c_fast(const float* in, int rows_in, int ncols, int in_pitch, size_t in_img,
                                int row0, const FftLen& f, float2* out, int out_pitch, size_t out_img,
                                float end_scale, float mid_scale, int batch, cudaStream_t st, bool pdl = false,
                                bool follows_peak = false, unsigned* err = nullptr,
                                long long wait = FT_WAIT_CYCLES);
// the adjoint of step 4 with the input gradient computed from the map and the
// target of the gradient workload (k_col_r2c_loss_fast); partial gets
// col_r2c_loss_blocks() floats per image
int col_r2c_loss_blocks(const FftLen& f, int ncols);
// (err, wait: with err given, the map columns are staged through tensor copies
// whose bounded waits set bit 3 of *err when they run out)
cudaError_t launch_col_r2c_loss_fast(const float* map, const float* target, int ncols, const FftLen& f,
                                     float2* out, int out_pitch, size_t out_img, float end_scale, float mid_scale,
                                     float scale, float gscale, float* partial, int batch, cudaStream_t st,
                                     bool pdl, unsigned* err = nullptr, long long wait = FT_WAIT_CYCLES);
// tmax (may be NULL; only with row0 = 0 and rows_out = N): the maxima of |out| per
// tile of c2r_tile_shape rows x columns, [batch][ceil(N / rows)][ceil(ncols / cols)] as
// float bits
// (err, wait: with err given, the staging goes through tensor copies whose
// bounded waits set bit 2 of *err when they run out; without, cp.async)
cudaError_t launch_col_c2r_fast(const float2* in, int ncols, int in_pitch, size_t in_img,
                                const FftLen& f, float mid_scale, float* out, int row0, int rows_out,
                                int out_pitch, size_t out_img, float out_scale, int batch,
                                cudaStream_t st, unsigned* tmax = nullptr, bool pdl = false,
                                unsigned* err = nullptr, long long wait = FT_WAIT_CYCLES);
// tiles of the tile maxima of launch_col_c2r_fast for length N: rows x cols
// cells, bands = N / rows tiles per column block; false without a schedule.
// A tile is 256 cells: 128 / B rows of one column block of 2B columns (the last
// band of a length that the rows do not divide is ragged).
// Maps of fewer than 128 rows have none: ft_detect keeps ft_forward and ft_peaks there,
// whose tiles are 16 x 16 instead of 4 x 64 (detection, us, with tiles from step 4 /
// from a pass of their own: 96x486 x 8 30.6 / 27.9, 96^2 x 64 30.2 / 26.9, 64^2 x 64
// 19.9 / 21.1, 108x4096 x 16 49.4 / 53.6).
__host__ __device__ constexpr bool c2r_tiles(int N) { return N >= 128; }
__host__ __device__ constexpr int c2r_tile_rows(int N) { return 128 / fs_Bc2r(N); }
__host__ __device__ constexpr int c2r_tile_bands(int N) { return (N + c2r_tile_rows(N) - 1) / c2r_tile_rows(N); }
bool c2r_tile_shape(int N, int* rows, int* cols, int* bands);
// (err: bit 1 set when a bulk-copy wait ran out after `wait` SM cycles)
cudaError_t launch_nvmt_rows_fast(float2* ws, int W, int Hp, int L, int interp, const FftLen& fx,
                                  int batch, cudaStream_t st, bool pdl, unsigned* err, long long wait);
cudaError_t launch_nvmt_rows_adjoint_fast(float2* ws, int W, int Hp, int L, int interp,
                                          const FftLen& fx, int batch, cudaStream_t st, bool pdl, LossSum ls);
