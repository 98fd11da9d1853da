// Primitives written for this library: exclusive scan (reduce, scan of tile
// sums, scan of tiles) and a stable LSD radix sort.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace pd {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

template <typename T>
PD_D T warp_incl_scan(T v) {
    int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

template <typename T>
PD_D T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Exclusive scan of one value per thread over the block; returns the block
// total through *total (all threads).  blockDim.x must be a multiple of 32.
template <typename T>
PD_D T block_excl_scan(T v, T* total) {
    __shared__ T wsum[33];
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T inc = warp_incl_scan(v);
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    if (w == 0) {
        T s = lane < nw ? wsum[lane] : T(0);
        T si = warp_incl_scan(s);
        if (lane < nw) wsum[lane] = si - s;
        if (lane == nw - 1) wsum[32] = si;
    }
    __syncthreads();
    T res = inc - v + wsum[w];
    *total = wsum[32];
    __syncthreads();
    return res;
}

template <typename T>
__global__ void k_tile_sum(const T* __restrict__ in, int64_t n, T* __restrict__ part) {
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    T s = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
        int64_t i = base + (int64_t)j * SCAN_THREADS + threadIdx.x;
        if (i < n) s += in[i];
    }
    s = warp_sum(s);
    __shared__ T ws[SCAN_THREADS / 32];
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        T t = 0;
        for (int w = 0; w < SCAN_THREADS / 32; w++) t += ws[w];
        part[blockIdx.x] = t;
    }
}

// One block of 1024 threads scans all tile sums in place (exclusive).
template <typename T>
__global__ void k_scan_partials(T* part, int64_t nb, T* total) {
    T carry = 0;
    for (int64_t base = 0; base < nb; base += blockDim.x) {
        int64_t i = base + threadIdx.x;
        T v = i < nb ? part[i] : T(0);
        T tot;
        T ex = block_excl_scan(v, &tot);
        if (i < nb) part[i] = ex + carry;
        carry += tot;
    }
    if (threadIdx.x == 0 && total) *total = carry;
}

template <typename T>
__global__ void k_tile_scan(const T* in, T* out, int64_t n, const T* __restrict__ part) {
    __shared__ T tile[SCAN_TILE];
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
        int64_t i = base + (int64_t)j * SCAN_THREADS + threadIdx.x;
        tile[j * SCAN_THREADS + threadIdx.x] = i < n ? in[i] : T(0);
    }
    __syncthreads();
    T loc[SCAN_ITEMS];
    T s = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
        loc[j] = tile[threadIdx.x * SCAN_ITEMS + j];
        s += loc[j];
    }
    T tot;
    T ex = block_excl_scan(s, &tot) + part[blockIdx.x];
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
        tile[threadIdx.x * SCAN_ITEMS + j] = ex;
        ex += loc[j];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
        int64_t i = base + (int64_t)j * SCAN_THREADS + threadIdx.x;
        if (i < n) out[i] = tile[j * SCAN_THREADS + threadIdx.x];
    }
}

inline int64_t scan_tiles(int64_t n) { return (n + SCAN_TILE - 1) / SCAN_TILE; }

// One block of 1024 threads scans in[0..n) into out (exclusive; in == out
// allowed: every element is read before the barrier that precedes its
// write), 4 consecutive elements a thread per step.  For short arrays, where
// the three-launch scan is all launch overhead.
constexpr int64_t SCAN_SMALL_MAX = int64_t(1) << 14;
template <typename T>
__global__ void __launch_bounds__(1024) k_scan_small(const T* in, T* out, int64_t n, T* total) {
    T carry = 0;
    for (int64_t base = 0; base < n; base += 4 * (int64_t)blockDim.x) {
        const int64_t i0 = base + 4 * (int64_t)threadIdx.x;
        T v[4];
        T s = 0;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            v[j] = i0 + j < n ? in[i0 + j] : T(0);
            s += v[j];
        }
        T tot;
        T ex = block_excl_scan(s, &tot) + carry;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            if (i0 + j < n) out[i0 + j] = ex;
            ex += v[j];
        }
        carry += tot;
    }
    if (threadIdx.x == 0 && total) *total = carry;
}

// out[i] = sum of in[0..i-1]; in == out allowed.  part: scan_tiles(n) + 1
// elements of scratch; *total_dev (device, may be NULL) gets the sum.
template <typename T>
cudaError_t exclusive_scan(const T* in, T* out, int64_t n, T* part, T* total_dev, cudaStream_t st) {
    if (n <= 0) {
        if (total_dev) return cudaMemsetAsync(total_dev, 0, sizeof(T), st);
        return cudaSuccess;
    }
    if (n <= SCAN_SMALL_MAX) {
        k_scan_small<T><<<1, 1024, 0, st>>>(in, out, n, total_dev); pd::count_launch();
        return cudaGetLastError();
    }
    int64_t nb = scan_tiles(n);
    k_tile_sum<T><<<(unsigned)nb, SCAN_THREADS, 0, st>>>(in, n, part); pd::count_launch();
    k_scan_partials<T><<<1, 1024, 0, st>>>(part, nb, total_dev); pd::count_launch();
    k_tile_scan<T><<<(unsigned)nb, SCAN_THREADS, 0, st>>>(in, out, n, part); pd::count_launch();
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// LSD radix sort, 8-bit digits
// ---------------------------------------------------------------------------
//
// Long arrays: one read for the digit counts of every pass, then one launch per
// pass.  A tile ranks its keys in registers, takes each digit's offset from the
// tiles before it by decoupled look-back (Merrill & Garland: a tile first
// publishes its own counts, then their running sum; tile numbers are tickets, so
// the tiles looked back at have started), orders the keys in shared memory and
// writes them in runs.  Should a tile looked back at not have published after the
// bounded wait, its digits and all before it are counted from the keys, which this
// pass only reads: the sort never waits without end and never ends unsorted.  A
// pass moves each key once in and once out; what bounds it is the ranking and the
// look-back's latency: 2,000,000 64-bit keys 26 us a pass
// (5 at the copy rate), two tiles an SM at a time.
//
// Short arrays (at most CS_MAX): one block sorts in shared memory, one launch for
// all passes.

// Lanes of the warp whose 8-bit digit is this lane's: eight ballots, independent
// of each other, where one __match_any_sync makes every lane wait for a pass over
// the distinct values (a sorting pass over 2,000,000 keys: 36 -> 26 us).
PD_D uint32_t same_digit(uint32_t d) {
    uint32_t p = 0xffffffffu;
#pragma unroll
    for (int b = 0; b < 8; b++) {
        const uint32_t bit = d >> b & 1u;
        p &= __ballot_sync(0xffffffffu, bit) ^ (bit - 1u);
    }
    return p;
}

constexpr int RS_THREADS = 256;
constexpr int RS_ITEMS = 16;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_MAXPASS = 8;
constexpr uint64_t RS_VALUE = (1ull << 62) - 1;  // of a state word: flag << 62 | value
constexpr int RS_BACK = 8;                                // tiles looked back at a time

inline int64_t radix_tiles(int64_t n) { return (n + RS_TILE - 1) / RS_TILE; }
inline int radix_passes(int bits) { return (bits + 7) / 8; }
// Words of scratch of `passes` passes: their counts, states (rows of 2 KB, aligned to
// lines) and tickets.
inline int64_t radix_words(int64_t n, int passes) { return passes * (256 + 256 * radix_tiles(n) + 1); }

// Digit counts of the passes first .. first + passes - 1.
__global__ void __launch_bounds__(RS_THREADS) k_radix_counts(const uint64_t* __restrict__ keys, int64_t n, int first,
                                                             int passes, unsigned long long* __restrict__ hist);
// One pass; vin / vout may be null.  polls: bound of a look-back wait.
__global__ void __launch_bounds__(RS_THREADS) k_radix_pass(const uint64_t* __restrict__ kin,
                                                           const uint32_t* __restrict__ vin,
                                                           uint64_t* __restrict__ kout, uint32_t* __restrict__ vout,
                                                           int64_t n, int shift,
                                                           const unsigned long long* __restrict__ hist,
                                                           unsigned long long* ticket, volatile unsigned long long* state,
                                                           int polls);

// ---- sort of one block of CS_THREADS threads

constexpr int CS_THREADS = 1024;
constexpr int CS_ITEMS = 8;
constexpr int CS_MAX = CS_THREADS * CS_ITEMS;
constexpr int CS_WARPS = CS_THREADS / 32;

struct CtaSort {
    uint64_t key[CS_MAX];
    uint32_t val[CS_MAX];
    uint32_t cnt[CS_WARPS][256];
    uint32_t part[4][256];
    uint32_t wsum[8];
};

// Stable sort of the block's items by the low `bits` bits of their keys.  Thread
// t of warp w holds items w * 32 * CS_ITEMS + 32 q + lane; past the end the
// keys are all ones.  The result is in k / v and in s.key / s.val.
PD_D void cta_sort(CtaSort& s, uint64_t (&k)[CS_ITEMS], uint32_t (&v)[CS_ITEMS], int bits) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t below = (1u << lane) - 1u;
    const int base = w * 32 * CS_ITEMS + lane;
    for (int shift = 0; shift < bits; shift += 8) {
        for (int q = tid; q < CS_WARPS * 256; q += CS_THREADS) (&s.cnt[0][0])[q] = 0;
        __syncthreads();
        uint32_t rank[CS_ITEMS];
#pragma unroll
        for (int q = 0; q < CS_ITEMS; q++) {
            const uint32_t d = (uint32_t)(k[q] >> shift) & 0xffu;
            const uint32_t peers = same_digit(d);
            const uint32_t seen = s.cnt[w][d];
            __syncwarp();
            if ((peers & below) == 0) s.cnt[w][d] = seen + __popc(peers);
            __syncwarp();
            rank[q] = seen + __popc(peers & below);
        }
        __syncthreads();
        // per digit: an exclusive sum over the warps (four threads, eight warps each), then over the digits
        {
            const int d = tid & 255, g = tid >> 8;
            uint32_t c[8], t = 0;
#pragma unroll
            for (int q = 0; q < 8; q++) c[q] = s.cnt[8 * g + q][d];
#pragma unroll
            for (int q = 0; q < 8; q++) t += c[q];
            s.part[g][d] = t;
            __syncthreads();
            uint32_t at = 0, tot = 0;
#pragma unroll
            for (int q = 0; q < 4; q++) {
                at += q < g ? s.part[q][d] : 0u;
                tot += s.part[q][d];
            }
            uint32_t inc = tot;
            if (g == 0) {
                inc = warp_incl_scan(tot);
                if (lane == 31) s.wsum[w] = inc;
            }
            __syncthreads();
            if (g == 0) {
                uint32_t o = inc - tot;
                for (int q = 0; q < w; q++) o += s.wsum[q];
                s.part[0][d] = o;  // (the four sums have been read)
            }
            __syncthreads();
            at += s.part[0][d];
#pragma unroll
            for (int q = 0; q < 8; q++) {
                s.cnt[8 * g + q][d] = at;
                at += c[q];
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < CS_ITEMS; q++) {
            const uint32_t at = s.cnt[w][(uint32_t)(k[q] >> shift) & 0xffu] + rank[q];
            s.key[at] = k[q];
            s.val[at] = v[q];
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < CS_ITEMS; q++) {
            k[q] = s.key[base + 32 * q];
            v[q] = s.val[base + 32 * q];
        }
    }
    if (bits <= 0) {
#pragma unroll
        for (int q = 0; q < CS_ITEMS; q++) {
            s.key[base + 32 * q] = k[q];
            s.val[base + 32 * q] = v[q];
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// small helpers
// ---------------------------------------------------------------------------

__global__ void k_fill_i64(int64_t* p, int64_t n, int64_t v);
__global__ void k_fill_i32(int32_t* p, int64_t n, int32_t v);

inline unsigned grid_for(int64_t n, int threads) {
    int64_t g = (n + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > 2147483647LL) g = 2147483647LL;
    return (unsigned)g;
}

}  // namespace pd
