// Peak detection of Sec. 4.4 from tile maxima of |P|, spread over the whole GPU
// (k_peak_sparse.cu runs one block per image): the same detected list.
//
// A peak inside tile j never exceeds the tile's maximum M[j].  A tile whose
// maximum is strictly larger than those of its 8 neighbours in the tile grid
// (wrapped) holds a peak of value M[j]: of its cells of that value the one with
// the smallest linear index precedes every cell around it, inside and outside the
// tile.  So the top_k-th largest maximum among such tiles bounds the top_k-th peak
// from below, and it is known before any cell of the map is read:
//   k_peak_bound  every tile against its 8 neighbours, the strict maxima appended
//                 to a list per image; the last block of an image to finish takes
//                 a 13-bit histogram of the list (exponent and 5 mantissa bits)
//                 and the lower edge of the bin that holds the top_k-th value,
//                 at most 3 % below it, becomes the bound (the threshold when
//                 there are fewer than top_k);
//   k_peak_scan   the tiles whose maximum reaches the bound, one per warp, tested
//                 cell by cell exactly as k_peak_sparse does (TileTester) and
//                 their strict local maxima at or above the bound appended to a
//                 list per image; the last block of an image selects and sorts its
//                 best top_k.  A list that overflows its PM_CAP keys (noise with fewer
//                 strict tile maxima than a large top_k: the bound is then the
//                 threshold) is dropped and that block runs the one-block pass on
//                 the image instead.
// Every key of the dense list lies in a tile that is tested and is at or above the
// bound, so the list is the same.
//
// What bounds the one-block pass is its serial chain on one multiprocessor:
// selecting among the tiles, then batches of 32 tiles, over 20 at 4096^2 with
// top_k = 100 (618 us for two images); the per-tile key pass reads every cell of
// the map instead (four images 109 + 31 us).  Here the tiles to test, about 1000 per
// such image, fill the GPU once.  Four images then take 62 us instead of 140 with top_k = 100, 44 instead of 104 with 8.
//
// The blocks of an image count themselves on a per-image word and the last one
// works on what the others wrote (fence, then atomic); no block waits for another.
// The words are zero before the first call and the last block to use one clears
// it, so calls follow each other without a memset.
#include <algorithm>

#include "peak_sparse_block.cuh"

#define PM_CAP 65536        // keys per image of the candidate list, or all that a map can have
#define PM_BINS 8192        // |P| bits >> 18 (no sign bit): exponent (8) and 5 mantissa bits
#define PM_THREADS 1024

struct PmState {            // per image, zero between calls
    int nloc, done1;        // strict tile maxima listed, blocks of k_peak_bound finished
    int ncand, done2;       // candidates listed, blocks of k_peak_scan finished
    unsigned bound;         // float bits of the bound (k_peak_bound -> k_peak_scan)
    int pad[3];
};

size_t peak_multi_state_bytes(int batch) { return (size_t)batch * sizeof(PmState); }

static size_t pm_loc_cap(int ntiles) { return (size_t)ntiles / 4 + 1; }
// a quarter of the cells at most are strict local maxima (a 2 x 2 block holds one)
static int pm_cap(int Hp, int S) { return (int)std::min((size_t)PM_CAP, (size_t)Hp * S / 4); }
size_t peak_multi_scratch_bytes(int Hp, int S, int ntiles, int batch) {
    return (size_t)batch * (pm_cap(Hp, S) * sizeof(u64) + pm_loc_cap(ntiles) * sizeof(unsigned));
}

__global__ void __launch_bounds__(PM_THREADS)
k_peak_bound(const unsigned* __restrict__ tmax, int nty, int ntx, int K, float thr, unsigned* __restrict__ loc,
             int loc_cap, PmState* __restrict__ state) {
    __shared__ unsigned hist[PM_BINS];
    __shared__ int last, nlist;
    pdl_wait();
    pdl_trigger();
    const int img = blockIdx.y, ntiles = nty * ntx;
    const unsigned* tm = tmax + (size_t)img * ntiles;
    unsigned* list = loc + (size_t)img * loc_cap;
    PmState* st = state + img;
    const int i = blockIdx.x * PM_THREADS + threadIdx.x;
    bool is = false;
    unsigned v = 0u;
    if (i < ntiles) {
        // a maximum of |P| has no sign bit; what a step 4 whose wait ran out left
        // unwritten may have one, and would fall outside the histogram's bins
        v = tm[i] & 0x7fffffffu;
        if (__uint_as_float(v) >= thr) {
            const int ty = i / ntx, tx = i - ty * ntx;
            const int up = (ty == 0 ? nty - 1 : ty - 1) * ntx, dn = (ty == nty - 1 ? 0 : ty + 1) * ntx, mid = ty * ntx;
            const int lf = tx == 0 ? ntx - 1 : tx - 1, rt = tx == ntx - 1 ? 0 : tx + 1;
            const unsigned a = max(max(tm[up + lf], tm[up + tx]), tm[up + rt]);
            const unsigned b = max(max(tm[dn + lf], tm[dn + tx]), tm[dn + rt]);
            is = v > max(max(a, b), max(tm[mid + lf], tm[mid + rt]));
        }
    }
    const unsigned bal = __ballot_sync(0xffffffffu, is);
    if (bal) {
        const int lane = threadIdx.x & 31;
        int pos = 0;
        if (lane == 0) pos = atomicAdd(&st->nloc, __popc(bal));
        pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(bal & ((1u << lane) - 1u));
        if (is && pos < loc_cap) list[pos] = v;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(&st->done1, 1) == (int)gridDim.x - 1;
        if (last) {
            __threadfence();
            nlist = min(atomicExch(&st->nloc, 0), loc_cap);
            st->done1 = 0;
        }
    }
    __syncthreads();
    if (!last) return;
    // the last block of the image: the bin of the K-th largest listed maximum
    const int n = nlist;
    unsigned bits = 0u;
    if (n >= K) {
        for (int b = threadIdx.x; b < PM_BINS; b += PM_THREADS) hist[b] = 0u;
        __syncthreads();
        for (int j = threadIdx.x; j < n; j += PM_THREADS) {
            const unsigned b = __ldcg(list + j) >> 18;
            if (FT_IN(b, PM_BINS, FT_DBG_PEAK_LIST)) atomicAdd(&hist[b], 1u);
        }
        __syncthreads();
        // thread t owns bins PM_BINS - 1 - 8 t - (0 .. 7), descending; an inclusive scan of
        // the owned counts finds the thread whose bins pass K
        constexpr int OWN = PM_BINS / PM_THREADS;
        const int top = PM_BINS - 1 - OWN * threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        unsigned own = 0u;
#pragma unroll
        for (int b = 0; b < OWN; ++b) own += hist[top - b];
        unsigned incl = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        __shared__ unsigned wsum[PM_THREADS / 32];
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        unsigned before = 0u;
        for (int w = 0; w < warp; ++w) before += wsum[w];
        incl += before;
        if (incl >= (unsigned)K && incl - own < (unsigned)K) {     // exactly one thread
            unsigned cum = incl - own;
            int b = top;
            for (int k = 0; k < OWN; ++k, --b) {
                cum += hist[b];
                if (cum >= (unsigned)K) break;
            }
            st->bound = (unsigned)b << 18;
        }
    } else if (threadIdx.x == 0) {
        st->bound = bits;
    }
}

__global__ void __launch_bounds__(PM_THREADS)
k_peak_scan(const float* __restrict__ map, const unsigned* __restrict__ tmax, int Hp, int S, int TH, int logTW,
            int nty, int ntx, int K, float thr, u64* __restrict__ cands, int cap, PmState* __restrict__ state,
            ft_peak* __restrict__ out, int32_t* __restrict__ count) {
    extern __shared__ __align__(16) unsigned char spsm[];
    __shared__ SparseShared sh;
    __shared__ int last;
    pdl_wait();
    pdl_trigger();
    const int img = blockIdx.y, ntiles = nty * ntx;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const float* m = map + (size_t)img * Hp * S;
    const unsigned* tm = tmax + (size_t)img * ntiles;
    u64* cand = cands + (size_t)img * cap;
    PmState* st = state + img;
    const float bound = fmaxf(thr, __uint_as_float(st->bound));
    float* stg = reinterpret_cast<float*>(spsm) + (size_t)warp * (TH + 2) * ((1 << logTW) + 8);
    int* list = reinterpret_cast<int*>(sh.st.hist);                // tiles of one round, at most the block's threads
    static_assert(sizeof(sh.st.hist) >= 256 * sizeof(int), "a round lists at most 256 tiles");
    const TileTester tester(m, Hp, S, TH, logTW, ntx, stg, lane);
    // tiles blockIdx.x + gridDim.x j: neighbouring tiles, which are bright together,
    // go to different blocks; 256 of them per round
    for (int j0 = 0; blockIdx.x + (size_t)gridDim.x * j0 < (size_t)ntiles; j0 += 256) {
        if (threadIdx.x == 0) sh.nlist = 0;
        __syncthreads();
        if (threadIdx.x < 256) {
            const long long t = blockIdx.x + (long long)gridDim.x * (j0 + threadIdx.x);
            bool w = false;
            if (t < ntiles) {
                const float x = __uint_as_float(tm[t]);
                w = x >= thr && x >= bound;
            }
            const unsigned bal = __ballot_sync(0xffffffffu, w);
            int pos = 0;
            if (lane == 0 && bal) pos = atomicAdd(&sh.nlist, __popc(bal));
            pos = __shfl_sync(0xffffffffu, pos, 0);
            pos += __popc(bal & ((1u << lane) - 1u));
            if (w && FT_IN(pos, 256, FT_DBG_PEAK_LIST)) list[pos] = (int)t;
        }
        __syncthreads();
        const int nl = sh.nlist;
        for (int j = warp; j < nl; j += nw) {
            unsigned long long mask;
            const unsigned best = tester.test(list[j], bound, mask);
            if (best) tester.append(list[j], bound, mask, cand, &st->ncand, cap);
            __syncwarp();
        }
        __syncthreads();
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(&st->done2, 1) == (int)gridDim.x - 1;
        if (last) {
            __threadfence();
            sh.ncand = atomicExch(&st->ncand, 0);
            st->done2 = 0;
        }
    }
    __syncthreads();
    if (!last) return;
    const int n = sh.ncand;
    if (n > cap) {
        __syncthreads();
        peak_sparse_block(m, tm, Hp, S, TH, logTW, nty, ntx, K, thr, out + (size_t)img * K, count + img, spsm, sh);
        return;
    }
    // the best min(K, n) keys, sorted: through shared memory when they fit the
    // staging area (the usual case), radix selection, then a bitonic sort
    const size_t stage = (size_t)nw * (TH + 2) * ((1 << logTW) + 8) * sizeof(float);
    u64* keep = reinterpret_cast<u64*>(spsm + ((stage + 15) & ~(size_t)15));   // next_pow2(K) keys
    const u64* keys = cand;
    if ((size_t)n * sizeof(u64) <= stage) {
        u64* k2 = reinterpret_cast<u64*>(spsm);
        for (int i = threadIdx.x; i < n; i += blockDim.x) k2[i] = __ldcg(cand + i);
        keys = k2;
        __syncthreads();
    }
    cta_select(keys, n, K, sh.st);
    if (threadIdx.x == 0) sh.st.count = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const u64 key = keys[i];
        if (selected(key, sh.st)) {
            const int o = atomicAdd(&sh.st.count, 1);
            if (FT_IN(o, K, FT_DBG_PEAK_LIST)) keep[o] = key;
        }
    }
    __syncthreads();
    const int cnt = sh.st.count, Kp = next_pow2(max(cnt, 1));
    for (int i = threadIdx.x; i < Kp; i += blockDim.x)
        if (i >= cnt) keep[i] = 0ull;
    __syncthreads();
    bitonic_desc(keep, Kp);
    write_peaks(keep, cnt, K, Hp, S, out, count, img);
}

FT_DEBUG_READER(ft_debug_read_peak_multi)

cudaError_t launch_peak_multi(const float* map, const unsigned* tmax, int Hp, int S, int tile_rows, int tile_cols,
                              int batch, int top_k, float threshold, void* scratch, void* state, ft_peak* out,
                              int32_t* count, cudaStream_t st, bool pdl) {
    int logTW = 0;
    while ((1 << logTW) < tile_cols) ++logTW;
    const int nty = (Hp + tile_rows - 1) / tile_rows, ntx = (S + tile_cols - 1) / tile_cols, ntiles = nty * ntx;
    const int nw = sparse_warps(tile_rows, tile_cols, top_k);
    if (nw == 0) return cudaErrorInvalidValue;
    u64* cands = static_cast<u64*>(scratch);
    const int cap = pm_cap(Hp, S);
    unsigned* loc = reinterpret_cast<unsigned*>(cands + (size_t)batch * cap);
    PmState* ps = static_cast<PmState*>(state);
    cudaError_t e = launch_maybe_pdl(k_peak_bound, dim3((ntiles + PM_THREADS - 1) / PM_THREADS, batch),
                                     dim3(PM_THREADS), 0, st, pdl, tmax, nty, ntx, top_k, threshold, loc,
                                     (int)pm_loc_cap(ntiles), ps);
    if (e != cudaSuccess) return e;
    const size_t sm = sparse_smem(tile_rows, tile_cols, top_k, nw, ntiles);
    e = cudaFuncSetAttribute(k_peak_scan, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    // 256 tiles per block: one round of listing
    return launch_maybe_pdl(k_peak_scan, dim3((ntiles + 255) / 256, batch), dim3(nw * 32), sm, st, pdl, map, tmax, Hp,
                            S, tile_rows, logTW, nty, ntx, top_k, threshold, cands, cap, ps, out, count);
}
