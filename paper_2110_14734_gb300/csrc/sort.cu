// The long radix sort's kernels (see prims.cuh) and the entry the stages use.
#include "internal.h"
#include "prims.cuh"

#include <algorithm>

namespace pd {

__global__ void __launch_bounds__(RS_THREADS) k_radix_counts(const uint64_t* __restrict__ keys, int64_t n, int first,
                                                             int passes, unsigned long long* __restrict__ hist) {
    __shared__ uint32_t h[RS_MAXPASS][256];
    for (int p = 0; p < passes; p++) h[p][threadIdx.x] = 0;
    __syncthreads();
    const int64_t step = (int64_t)gridDim.x * RS_THREADS;
    for (int64_t i = (int64_t)blockIdx.x * RS_THREADS + threadIdx.x; i < n; i += step) {
        const uint64_t k = keys[i] >> (8 * first);
        for (int p = 0; p < passes; p++) atomicAdd(&h[p][(uint32_t)(k >> (8 * p)) & 0xffu], 1u);
    }
    __syncthreads();
    for (int p = 0; p < passes; p++)
        if (h[p][threadIdx.x]) atomicAdd(&hist[256 * p + threadIdx.x], (unsigned long long)h[p][threadIdx.x]);
}

// Keys with digit d among the first n.
__device__ __noinline__ unsigned long long count_digit(const uint64_t* __restrict__ keys, int64_t n, int shift,
                                                       uint32_t d) {
    unsigned long long c = 0;
    for (int64_t i = 0; i < n; i++) c += ((uint32_t)(keys[i] >> shift) & 0xffu) == d;
    return c;
}

__global__ void __launch_bounds__(RS_THREADS) k_radix_pass(const uint64_t* __restrict__ kin,
                                                           const uint32_t* __restrict__ vin,
                                                           uint64_t* __restrict__ kout, uint32_t* __restrict__ vout,
                                                           int64_t n, int shift,
                                                           const unsigned long long* __restrict__ hist,
                                                           unsigned long long* ticket, volatile unsigned long long* state,
                                                           int polls) {
    __shared__ uint32_t cnt[RS_WARPS][256];
    __shared__ uint64_t skey[RS_TILE];
    __shared__ int64_t base[256];  // of a digit: output index less index in the tile's order
    __shared__ uint32_t first[256];
    __shared__ int64_t s_tile;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t below = (1u << lane) - 1u;
    if (tid == 0) s_tile = (int64_t)atomicAdd(ticket, 1ull);
#pragma unroll
    for (int q = 0; q < RS_WARPS; q++) cnt[q][tid] = 0;
    __syncthreads();
    const int64_t tile = s_tile, t0 = tile * RS_TILE;
    const int m = (int)min((int64_t)RS_TILE, n - t0);
    const int i0 = w * 32 * RS_ITEMS + lane;
    uint64_t k[RS_ITEMS];
    uint32_t at[RS_ITEMS];
#pragma unroll
    for (int q = 0; q < RS_ITEMS; q++) k[q] = i0 + 32 * q < m ? kin[t0 + i0 + 32 * q] : ~0ull;
#pragma unroll
    for (int q = 0; q < RS_ITEMS; q++) {
        const bool in = i0 + 32 * q < m;  // past the end: no count
        const uint32_t d = (uint32_t)(k[q] >> shift) & 0xffu;
        const uint32_t peers = same_digit(d) & __ballot_sync(0xffffffffu, in);
        const uint32_t seen = cnt[w][d];
        __syncwarp();
        if (in && (peers & below) == 0) cnt[w][d] = seen + __popc(peers);
        __syncwarp();
        at[q] = seen + __popc(peers & below);
    }
    __syncthreads();
    uint32_t c = 0;
#pragma unroll
    for (int q = 0; q < RS_WARPS; q++) {
        const uint32_t t = cnt[q][tid];
        cnt[q][tid] = c;
        c += t;
    }
    state[256 * tile + tid] = (tile == 0 ? 2ull : 1ull) << 62 | c;
    uint32_t tot;
    const uint32_t ex = block_excl_scan<uint32_t>(c, &tot);
    unsigned long long all;
    const unsigned long long hx = block_excl_scan<unsigned long long>(hist[tid], &all);
    // eight tiles back at a time: when all tiles run at once, most of them have
    // only their own counts out yet (condensation of 2,000,000 points: 0.731 ms one
    // by one, 0.714 so)
    unsigned long long before = 0;
    int64_t rest = 0;  // keys before the tiles that answered, all of whose digits are to be counted
    bool open = tile > 0;
    for (int64_t t = tile - 1; open; t -= RS_BACK) {
        unsigned long long v[RS_BACK];
#pragma unroll
        for (int j = 0; j < RS_BACK; j++) v[j] = t >= j ? state[256 * (t - j) + tid] : 2ull << 62;
#pragma unroll
        for (int j = 0; j < RS_BACK; j++) {
            if (!open) continue;
            for (int q = 0; v[j] >> 62 == 0 && q < polls; q++) v[j] = state[256 * (t - j) + tid];
            if (v[j] >> 62 == 0) rest = (t - j + 1) * RS_TILE;  // and the search ends
            before += v[j] & RS_VALUE;
            open = v[j] >> 62 == 1;
        }
    }
    if (rest > 0) before += count_digit(kin, rest, shift, tid);
    if (tile > 0) state[256 * tile + tid] = 2ull << 62 | (before + c);
    first[tid] = ex;
    base[tid] = (int64_t)(hx + before) - (int64_t)ex;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < RS_ITEMS; q++)
        if (i0 + 32 * q < m) {
            const uint32_t d = (uint32_t)(k[q] >> shift) & 0xffu;
            at[q] += first[d] + cnt[w][d];
            skey[at[q]] = k[q];
        }
    __syncthreads();
    uint32_t out[RS_ITEMS];  // with values n < 2^32
#pragma unroll
    for (int q = 0; q < RS_ITEMS; q++) {
        const int i = tid + q * RS_THREADS;
        if (i < m) {
            const uint64_t key = skey[i];
            const int64_t o = base[(uint32_t)(key >> shift) & 0xffu] + i;
            kout[o] = key;
            out[q] = (uint32_t)o;
        }
    }
    if (vin) {
        uint32_t* sval = (uint32_t*)skey;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < RS_ITEMS; q++)
            if (i0 + 32 * q < m) sval[at[q]] = vin[t0 + i0 + 32 * q];
        __syncthreads();
#pragma unroll
        for (int q = 0; q < RS_ITEMS; q++) {
            const int i = tid + q * RS_THREADS;
            if (i < m) vout[out[q]] = sval[i];
        }
    }
}

__global__ void __launch_bounds__(CS_THREADS) k_sort_small(uint64_t* __restrict__ keys, uint32_t* __restrict__ vals,
                                                           int n, int bits) {
    extern __shared__ __align__(16) unsigned char sort_dyn[];
    CtaSort& s = *(CtaSort*)sort_dyn;
    const int base = (threadIdx.x >> 5) * 32 * CS_ITEMS + (threadIdx.x & 31);
    uint64_t k[CS_ITEMS];
    uint32_t v[CS_ITEMS];
#pragma unroll
    for (int q = 0; q < CS_ITEMS; q++) {
        const int i = base + 32 * q;
        k[q] = i < n ? keys[i] : ~0ull;
        v[q] = i < n && vals ? vals[i] : 0u;
    }
    cta_sort(s, k, v, bits);
#pragma unroll
    for (int q = 0; q < CS_ITEMS; q++) {
        const int i = base + 32 * q;
        if (i < n) {
            keys[i] = k[q];
            if (vals) vals[i] = v[q];
        }
    }
}

// Above these sizes a block's sort (1,024 threads on one SM) takes longer than
// the long sort's launches.
pd_status sort_u64(Ctx* c, uint64_t*& keys, uint64_t*& keys_alt, uint32_t*& vals, uint32_t*& vals_alt, int64_t n,
                   int bits, cudaStream_t st, int polls) {
    if (n <= 1 || bits <= 0) return PD_OK;
    if (n <= CS_MAX) {
        static std::atomic<uint64_t> done{0};
        PD_TRY(smem_limit(c, done, (const void*)k_sort_small, sizeof(CtaSort)));
        k_sort_small<<<1, CS_THREADS, sizeof(CtaSort), st>>>(keys, vals, (int)n, bits); pd::count_launch();
        PD_TRY_CUDA(c, cudaGetLastError());
        return PD_OK;
    }
    const int passes = radix_passes(bits);
    const int64_t tiles = radix_tiles(n);
    // short of memory (a quarter of what other scratch may take: it stays beside the
    // stages that follow): one pass's worth, counted and cleared before each
    int sets = beyond_cap(c, 4 * 8 * radix_words(n, passes)) ? 1 : passes;
    unsigned long long* w = bufT<unsigned long long>(c, B_RS_COUNTS, radix_words(n, sets));
    if (!w && sets > 1) {
        c->err.clear();
        sets = 1;
        w = bufT<unsigned long long>(c, B_RS_COUNTS, radix_words(n, sets));
    }
    if (!w) return PD_ENOMEM;
    unsigned long long *hist = w, *state = w + 256 * sets, *ticket = state + 256 * tiles * sets;
    const unsigned count_grid = (unsigned)std::min<int64_t>(tiles, 4 * std::max(c->sm_count, 1));
    for (int p = 0; p < passes; p++) {
        const int q = p % sets;
        if (q == 0) {
            PD_TRY_CUDA(c, cudaMemsetAsync(w, 0, sizeof(unsigned long long) * radix_words(n, sets), st));
            k_radix_counts<<<count_grid, RS_THREADS, 0, st>>>(keys, n, p, sets, hist); pd::count_launch();
        }
        k_radix_pass<<<(unsigned)tiles, RS_THREADS, 0, st>>>(keys, vals, keys_alt, vals ? vals_alt : nullptr, n, 8 * p,
                                                            hist + 256 * q, ticket + q, state + 256 * tiles * q,
                                                            polls); pd::count_launch();
        std::swap(keys, keys_alt);
        std::swap(vals, vals_alt);
    }
    PD_TRY_CUDA(c, cudaGetLastError());
    return PD_OK;
}

}  // namespace pd
