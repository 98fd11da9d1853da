// Quantisation, 0-condensation, RWMD (Algorithm 1) and delta-condensation
// (Algorithm 2) on the device.
#include "internal.h"
#include "prims.cuh"

#include <algorithm>
#include <cmath>

namespace pd {

// small-scalar slots in B_SMALL (int64)
enum : int {
    S_MNX = 0, S_MXX, S_MNY, S_MXY, S_FA, S_FB, S_ERR, S_NA, S_M, S_L0, S_L1,
    S_CMNX, S_CMXX, S_CMNY, S_CMXY, S_N, S_NMNX, S_NMXX, S_NMNY, S_NMXY, S_COUNT = 32
};

__global__ void k_init_small(int64_t* s) {
    int i = threadIdx.x;
    if (i < S_COUNT) {
        int64_t v = 0;
        if (i == S_MNX || i == S_MNY || i == S_CMNX || i == S_CMNY || i == S_NMNX || i == S_NMNY) v = INT64_MAX;
        if (i == S_MXX || i == S_MXY || i == S_CMXX || i == S_CMXY || i == S_NMXX || i == S_NMXY) v = INT64_MIN;
        s[i] = v;
    }
}

// Sums and extremes over all blocks end in atomics on a handful of words.  One set
// of them per warp serialises (2,000,000 points: 201 microseconds for k_quantize,
// 160 for k_cells), so the kernels that need them run few blocks that stride over
// the data, and each block adds one set.
constexpr int BOX_THREADS = 256;
static unsigned box_grid(const Ctx* c, int64_t n) {
    return (unsigned)std::min<int64_t>(grid_for(n, BOX_THREADS), 4 * std::max(c->sm_count, 1));
}

// Block extremes b = (min x, max x, min y, max y) into at[0 .. 3] (min, max, min, max).
PD_D void box_to(int32_t (&b)[4], int64_t* at) {
    __shared__ int32_t s[4][BOX_THREADS / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        b[q] = q & 1 ? __reduce_max_sync(0xffffffffu, b[q]) : __reduce_min_sync(0xffffffffu, b[q]);
        if (lane == 0) s[q][w] = b[q];
    }
    __syncthreads();
    if (w != 0) return;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        const int32_t v = s[q][lane & (BOX_THREADS / 32 - 1)];
        b[q] = q & 1 ? __reduce_max_sync(0xffffffffu, v) : __reduce_min_sync(0xffffffffu, v);
    }
    if (lane == 0 && b[0] <= b[1]) {
        atomicMin((long long*)&at[0], (long long)b[0]);
        atomicMax((long long*)&at[1], (long long)b[1]);
        atomicMin((long long*)&at[2], (long long)b[2]);
        atomicMax((long long*)&at[3], (long long)b[3]);
    }
}

// a1: X = rint(b 2^k), Y = rint(d 2^k) of one point; false (X = Y = 0) when
// non-finite or |X|, |Y| >= 2^29.
PD_D bool quantize_point(const void* __restrict__ p, int64_t j, int dt, int k, int32_t* X, int32_t* Y) {
    int64_t qx = 0, qy = 0;
    bool ok = true;
    if (dt == PD_F32) {
        const float2 v = ((const float2*)p)[j];
        if (k <= 127) {
            // a power of two scales a float exactly (2^k >= 1: nothing is lost below; above, infinity
            // is rejected): single precision gives what double would, which has a 64th of its rate
            const float s = __int_as_float((127 + k) << 23), rb = rintf(v.x * s), rd = rintf(v.y * s);
            ok = fabsf(rb) < (float)COORD_LIMIT && fabsf(rd) < (float)COORD_LIMIT;  // false for a NaN
            if (ok) {
                qx = (int64_t)(int32_t)rb;
                qy = (int64_t)(int32_t)rd;
            }
        } else {
            const double s = ldexp(1.0, k), rb = rint((double)v.x * s), rd = rint((double)v.y * s);
            ok = fabs(rb) < (double)COORD_LIMIT && fabs(rd) < (double)COORD_LIMIT;
            if (ok) {
                qx = (int64_t)rb;
                qy = (int64_t)rd;
            }
        }
    } else {
        const uchar2 v = ((const uchar2*)p)[j];
        qx = (int64_t)v.x << k;
        qy = (int64_t)v.y << k;
        ok = qx < COORD_LIMIT && qy < COORD_LIMIT;
    }
    *X = (int32_t)qx;
    *Y = (int32_t)qy;
    return ok;
}

// Quantises all points: keep unless X == Y; track min/max and the masses of A
// and B; count the rejected ones.
__global__ void __launch_bounds__(BOX_THREADS) k_quantize(const void* __restrict__ a, int64_t na, int dta,
                                                          const void* __restrict__ b, int64_t nb, int dtb, int k,
                                                          int32_t* __restrict__ X, int32_t* __restrict__ Y,
                                                          uint8_t* __restrict__ keep, int64_t* __restrict__ sm) {
    const int64_t n = na + nb, step = (int64_t)gridDim.x * BOX_THREADS;
    int32_t box[4] = {INT32_MAX, INT32_MIN, INT32_MAX, INT32_MIN};
    uint32_t c[3] = {0, 0, 0};  // kept of A, of B, rejected
    for (int64_t i = (int64_t)blockIdx.x * BOX_THREADS + threadIdx.x; i < n; i += step) {
        const bool isB = i >= na;
        int32_t qx, qy;
        const bool bad = !quantize_point(isB ? b : a, isB ? i - na : i, isB ? dtb : dta, k, &qx, &qy);
        const bool kp = !bad && qx != qy;
        X[i] = qx;
        Y[i] = qy;
        keep[i] = (uint8_t)kp;
        if (kp) {
            box[0] = min(box[0], qx);
            box[1] = max(box[1], qx);
            box[2] = min(box[2], qy);
            box[3] = max(box[3], qy);
        }
        c[0] += kp && !isB;
        c[1] += kp && isB;
        c[2] += bad;
    }
    __shared__ uint32_t s_c[3];
    if (threadIdx.x < 3) s_c[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 3; q++) {
        c[q] = __reduce_add_sync(0xffffffffu, c[q]);
        if ((threadIdx.x & 31) == 0 && c[q]) atomicAdd(&s_c[q], c[q]);
    }
    __syncthreads();
    if (threadIdx.x < 3 && s_c[threadIdx.x]) {
        const int slot[3] = {S_FA, S_FB, S_ERR};
        atomicAdd((unsigned long long*)&sm[slot[threadIdx.x]], (unsigned long long)s_c[threadIdx.x]);
    }
    box_to(box, &sm[S_MNX]);
}

// Sort key: diagram bit, then X, then Y (lexicographic); dropped points get
// the all-ones key so that they sort last.
__global__ void k_point_keys(const int32_t* __restrict__ X, const int32_t* __restrict__ Y,
                             const uint8_t* __restrict__ keep, int64_t na, int64_t n, const int64_t* __restrict__ sm,
                             int bx, int by, uint64_t* __restrict__ key) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint64_t sent = (bx + by + 2 >= 64) ? ~0ull : ((1ull << (bx + by + 2)) - 1);
    if (!keep[i]) {
        key[i] = sent;
        return;
    }
    uint64_t isB = i >= na;
    key[i] = (isB << (bx + by)) | ((uint64_t)(X[i] - sm[S_MNX]) << by) | (uint64_t)(Y[i] - sm[S_MNY]);
}

__global__ void k_run_flags(const uint64_t* __restrict__ key, int64_t n, uint64_t sent, int64_t* __restrict__ flag) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint64_t k = key[i];
    flag[i] = (k != sent && (i == 0 || key[i - 1] != k)) ? 1 : 0;
}

// Node j of the 0-condensation starts at sorted position start[j].
__global__ void k_hat_compact(const uint64_t* __restrict__ key, int64_t n, uint64_t sent,
                              const int64_t* __restrict__ idx, const int64_t* __restrict__ sm, int bx, int by,
                              int32_t* __restrict__ HX, int32_t* __restrict__ HY, int64_t* __restrict__ start,
                              int64_t* __restrict__ nA) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint64_t k = key[i];
    if (k == sent || (i > 0 && key[i - 1] == k)) return;
    int64_t j = idx[i];
    uint64_t ymask = (by >= 64) ? ~0ull : ((1ull << by) - 1);
    uint64_t xmask = (bx >= 64) ? ~0ull : ((1ull << bx) - 1);
    HX[j] = (int32_t)((int64_t)((k >> by) & xmask) + sm[S_MNX]);
    HY[j] = (int32_t)((int64_t)(k & ymask) + sm[S_MNY]);
    start[j] = i;
    // A's nodes come first: B's first node says how many there are
    if ((k >> (bx + by)) & 1ull && (i == 0 || !((key[i - 1] >> (bx + by)) & 1ull))) *nA = j;
}

__global__ void k_hat_counts(const int64_t* __restrict__ start, int64_t M, int64_t nvalid, int64_t* __restrict__ cnt) {
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= M) return;
    int64_t e = (j + 1 < M) ? start[j + 1] : nvalid;
    cnt[j] = e - start[j];
}

// ---- short inputs: a whole stage in one block, one launch -----------------
//
// At a few thousand points a stage is all launches (18 for the 0-condensation,
// 35 for the delta-condensation, of 2 to 3 microseconds each, and a host round
// trip in the middle for the key's width).  One block of 1,024 threads holds up
// to CS_MAX points in registers, sorts them in shared memory and writes the
// results; widths stay on the device.  out (host memory): the stage's scalars.
// Measured for two diagrams of 2,000 points: pd_rwmd_lower_bound (with
// k_rwmd_small) 240 -> 87 us, the two condensations together 0.53 -> 0.08 ms.

struct CtaStage {
    CtaSort sort;
    int32_t ext[4][CS_WARPS];
    uint32_t count[4];
};

// Extremes of the block's x and y (min x, max x, min y, max y) in every thread;
// values beyond the items are passed as the neutral ones.
PD_D void cta_box(CtaStage& s, int32_t (&b)[4]) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        b[q] = q & 1 ? __reduce_max_sync(0xffffffffu, b[q]) : __reduce_min_sync(0xffffffffu, b[q]);
        if (lane == 0) s.ext[q][w] = b[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; q++)
        b[q] = q & 1 ? __reduce_max_sync(0xffffffffu, s.ext[q][lane]) : __reduce_min_sync(0xffffffffu, s.ext[q][lane]);
    __syncthreads();
}

PD_D int dev_bits_for(uint32_t v) { return 32 - __clz((int)v); }  // 0 for 0

__global__ void __launch_bounds__(CS_THREADS) k_condense0_small(const void* __restrict__ a, int na, int dta,
                                                                const void* __restrict__ b, int nb, int dtb, int k,
                                                                int32_t* __restrict__ HX, int32_t* __restrict__ HY,
                                                                int64_t* __restrict__ cnt, int64_t* __restrict__ sm,
                                                                int64_t* out) {
    extern __shared__ __align__(16) unsigned char cond_dyn[];
    CtaStage& s = *(CtaStage*)cond_dyn;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, n = na + nb;
    const int base = w * 32 * CS_ITEMS + lane;
    if (tid < 4) s.count[tid] = 0;
    if (tid < S_COUNT) sm[tid] = 0;  // what the next stages add to
    int32_t box[4] = {INT32_MAX, INT32_MIN, INT32_MAX, INT32_MIN}, x[CS_ITEMS], y[CS_ITEMS];
    uint32_t keep = 0, fa = 0, fb = 0, bad = 0;
#pragma unroll
    for (int q = 0; q < CS_ITEMS; q++) {
        const int i = base + 32 * q;
        x[q] = y[q] = 0;
        if (i < n) {
            const bool isB = i >= na;
            if (!quantize_point(isB ? b : a, isB ? i - na : i, isB ? dtb : dta, k, &x[q], &y[q])) {
                bad++;
            } else if (x[q] != y[q]) {
                keep |= 1u << q;
                fa += !isB;
                fb += isB;
                box[0] = min(box[0], x[q]);
                box[1] = max(box[1], x[q]);
                box[2] = min(box[2], y[q]);
                box[3] = max(box[3], y[q]);
            }
        }
    }
    cta_box(s, box);
    fa = __reduce_add_sync(0xffffffffu, fa);
    fb = __reduce_add_sync(0xffffffffu, fb);
    bad = __reduce_add_sync(0xffffffffu, bad);
    if (lane == 0) {
        atomicAdd(&s.count[0], fa);
        atomicAdd(&s.count[1], fb);
        atomicAdd(&s.count[2], bad);
    }
    __syncthreads();
    const int nv = (int)(s.count[0] + s.count[1]);
    if (s.count[2] || nv == 0) {
        if (tid == 0) {
            out[S_ERR] = s.count[2];
            out[S_FA] = out[S_FB] = out[S_M] = out[S_NA] = 0;
        }
        return;
    }
    // diagram bit, then X, then Y; dropped points keep the all-ones key
    const int bx = dev_bits_for((uint32_t)(box[1] - box[0])), by = dev_bits_for((uint32_t)(box[3] - box[2]));
    uint64_t key[CS_ITEMS];
    uint32_t none[CS_ITEMS];
#pragma unroll
    for (int q = 0; q < CS_ITEMS; q++) {
        const uint64_t isB = base + 32 * q >= na;
        key[q] = keep >> q & 1u ? isB << (bx + by) | (uint64_t)(uint32_t)(x[q] - box[0]) << by | (uint32_t)(y[q] - box[2])
                                : ~0ull;
        none[q] = 0;
    }
    cta_sort(s.sort, key, none, bx + by + 2);
    // runs: a thread's items are CS_ITEMS consecutive positions now
    uint32_t heads = 0;
    const int p0 = tid * CS_ITEMS;
#pragma unroll
    for (int q = 0; q < CS_ITEMS; q++) {
        const int i = p0 + q;
        if (i < nv && (i == 0 || s.sort.key[i - 1] != s.sort.key[i])) heads |= 1u << q;
    }
    uint32_t M;
    uint32_t j = block_excl_scan<uint32_t>(__popc(heads), &M);
    uint32_t* start = s.sort.val;  // first position of every node
    uint32_t inA = 0;
    for (uint32_t h = heads; h; h &= h - 1, j++) {
        const int i = p0 + __ffs(h) - 1;
        const uint64_t kk = s.sort.key[i];
        HX[j] = (int32_t)((kk >> by) & ((1ull << bx) - 1)) + box[0];
        HY[j] = (int32_t)(kk & ((1ull << by) - 1)) + box[2];
        start[j] = (uint32_t)i;
        inA += (kk >> (bx + by) & 1ull) == 0;
    }
    inA = __reduce_add_sync(0xffffffffu, inA);
    if (lane == 0) atomicAdd(&s.count[3], inA);
    __syncthreads();
    for (uint32_t q = tid; q < M; q += CS_THREADS) cnt[q] = (int64_t)((q + 1 < M ? start[q + 1] : (uint32_t)nv) - start[q]);
    if (tid == 0) {
        out[S_ERR] = 0;
        out[S_FA] = s.count[0];
        out[S_FB] = s.count[1];
        out[S_M] = M;
        out[S_NA] = s.count[3];
    }
}

pd_status stage_condense0(Ctx* c, const DevDiag& A, const DevDiag& B, int k, Hats* out, cudaStream_t st) {
    int64_t n = A.n + B.n;
    int64_t* sm = bufT<int64_t>(c, B_SMALL, 64);
    if (!sm) return PD_ENOMEM;
    out->nA = out->nB = out->FA = out->FB = 0;
    out->X = bufT<int32_t>(c, B_HAT_X, n);
    out->Y = bufT<int32_t>(c, B_HAT_Y, n);
    out->cnt = bufT<int64_t>(c, B_HAT_C, n);
    if (!out->X || !out->Y || !out->cnt) return PD_ENOMEM;
    if (n == 0) return PD_OK;
    if (n <= CS_MAX) {
        int64_t* h = c->h_small;
        static std::atomic<uint64_t> done{0};
        PD_TRY(smem_limit(c, done, (const void*)k_condense0_small, sizeof(CtaStage)));
        k_condense0_small<<<1, CS_THREADS, sizeof(CtaStage), st>>>(A.bd, (int)A.n, A.dtype, B.bd, (int)B.n, B.dtype, k,
                                                                   out->X, out->Y, out->cnt, sm, h); pd::count_launch();
        PD_TRY_CUDA(c, cudaGetLastError());
        PD_TRY_CUDA(c, cudaStreamSynchronize(st));
        if (h[S_ERR]) return fail(c, PD_EINVAL, "diagram has a non-finite coordinate or |coordinate| * 2^k >= 2^29");
        out->FA = h[S_FA];
        out->FB = h[S_FB];
        out->nA = h[S_NA];
        out->nB = h[S_M] - h[S_NA];
        return PD_OK;
    }
    k_init_small<<<1, 64, 0, st>>>(sm); pd::count_launch();
    int32_t* X = bufT<int32_t>(c, B_QX, n);
    int32_t* Y = bufT<int32_t>(c, B_QY, n);
    uint8_t* keep = bufT<uint8_t>(c, B_FLAG, n);
    uint64_t* key = bufT<uint64_t>(c, B_QKEY, n);
    uint64_t* key2 = bufT<uint64_t>(c, B_QKEY2, n);
    int64_t* flag = bufT<int64_t>(c, B_IDX, n);
    int64_t* start = bufT<int64_t>(c, B_QVAL, n);
    if (!X || !Y || !keep || !key || !key2 || !flag || !start) return PD_ENOMEM;
    k_quantize<<<box_grid(c, n), BOX_THREADS, 0, st>>>(A.bd, A.n, A.dtype, B.bd, B.n, B.dtype, k, X, Y, keep, sm); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    PD_TRY_CUDA(c, cudaMemcpyAsync(c->h_small, sm, sizeof(int64_t) * S_COUNT, cudaMemcpyDeviceToHost, st));
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));
    int64_t* h = c->h_small;
    if (h[S_ERR]) return fail(c, PD_EINVAL, "diagram has a non-finite coordinate or |coordinate| * 2^k >= 2^29");
    out->FA = h[S_FA];
    out->FB = h[S_FB];
    int64_t nvalid = h[S_FA] + h[S_FB];
    if (nvalid == 0) return PD_OK;
    int bx = bits_for((uint64_t)(h[S_MXX] - h[S_MNX])), by = bits_for((uint64_t)(h[S_MXY] - h[S_MNY]));
    int kb = bx + by + 2;
    uint64_t sent = (kb >= 64) ? ~0ull : ((1ull << kb) - 1);
    k_point_keys<<<grid_for(n, 256), 256, 0, st>>>(X, Y, keep, A.n, n, sm, bx, by, key); pd::count_launch();
    uint32_t *none = nullptr, *none2 = nullptr;
    PD_TRY(sort_u64(c, key, key2, none, none2, n, kb, st));
    k_run_flags<<<grid_for(n, 256), 256, 0, st>>>(key, n, sent, flag); pd::count_launch();
    PD_TRY(scan_i64(c, flag, flag, n, sm + S_M, st));
    k_hat_compact<<<grid_for(n, 256), 256, 0, st>>>(key, n, sent, flag, sm, bx, by, out->X, out->Y, start,
                                                      sm + S_NA); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    PD_TRY_CUDA(c, cudaMemcpyAsync(c->h_small, sm, sizeof(int64_t) * S_COUNT, cudaMemcpyDeviceToHost, st));
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));
    int64_t M = h[S_M];
    out->nA = out->FB > 0 ? h[S_NA] : M;
    out->nB = M - out->nA;
    k_hat_counts<<<grid_for(M, 256), 256, 0, st>>>(start, M, nvalid, out->cnt); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    return PD_OK;
}

// ---------------------------------------------------------------------------
// RWMD (Algorithm 1, with the diagonal option of the relaxed flow)
// ---------------------------------------------------------------------------

constexpr int RW_THREADS = 256;
constexpr int RW_TILE = 2048;

// Exact minimum squared distance from every node of one side to the nodes of
// the other side; blockIdx.y splits the other side, blockIdx.z = direction.
__global__ void __launch_bounds__(RW_THREADS) k_rwmd_min(const int32_t* __restrict__ X, const int32_t* __restrict__ Y,
                                                         int64_t nA, int64_t nB, int64_t chunk,
                                                         unsigned long long* __restrict__ mind2) {
    __shared__ int2 q[RW_TILE];
    int dir = blockIdx.z;
    int64_t pbase = dir == 0 ? 0 : nA, np = dir == 0 ? nA : nB;
    int64_t qbase = dir == 0 ? nA : 0, nq = dir == 0 ? nB : nA;
    int64_t u = (int64_t)blockIdx.x * RW_THREADS + threadIdx.x;
    int64_t q0 = (int64_t)blockIdx.y * chunk, q1 = min(nq, q0 + chunk);
    if ((int64_t)blockIdx.x * RW_THREADS >= np || q0 >= q1) return;
    int32_t ux = 0, uy = 0;
    if (u < np) {
        ux = X[pbase + u];
        uy = Y[pbase + u];
    }
    unsigned long long best = ~0ull;
    for (int64_t t0 = q0; t0 < q1; t0 += RW_TILE) {
        int tn = (int)min((int64_t)RW_TILE, q1 - t0);
        __syncthreads();
        for (int j = threadIdx.x; j < tn; j += RW_THREADS) q[j] = make_int2(X[qbase + t0 + j], Y[qbase + t0 + j]);
        __syncthreads();
        for (int j = 0; j < tn; j++) {
            int2 v = q[j];
            long long dx = (long long)(ux - v.x), dy = (long long)(uy - v.y);
            unsigned long long d2 = (unsigned long long)(dx * dx) + (unsigned long long)(dy * dy);
            best = d2 < best ? d2 : best;
        }
    }
    if (u < np) atomicMin(&mind2[pbase + u], best);
}

__global__ void __launch_bounds__(BOX_THREADS) k_rwmd_sum(const int32_t* __restrict__ X, const int32_t* __restrict__ Y,
                                                          const int64_t* __restrict__ cnt, int64_t nA, int64_t n,
                                                          const unsigned long long* __restrict__ mind2, DiagCost dc,
                                                          int64_t* __restrict__ L) {
    __shared__ unsigned long long s[2][BOX_THREADS / 32];
    unsigned long long va = 0, vb = 0;
    for (int64_t i = (int64_t)blockIdx.x * BOX_THREADS + threadIdx.x; i < n; i += (int64_t)gridDim.x * BOX_THREADS) {
        int64_t c = cost_make(X[i], Y[i], dc);
        const unsigned long long m = mind2[i];
        if (m != ~0ull) {
            const int64_t cn = (int64_t)ceil_sqrt_u64(m);
            c = cn < c ? cn : c;
        }
        (i < nA ? va : vb) += (unsigned long long)(c * cnt[i]);
    }
    va = warp_sum(va);
    vb = warp_sum(vb);
    if ((threadIdx.x & 31) == 0) {
        s[0][threadIdx.x >> 5] = va;
        s[1][threadIdx.x >> 5] = vb;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        unsigned long long v = 0;
        for (int q = 0; q < BOX_THREADS / 32; q++) v += s[threadIdx.x][q];
        if (v) atomicAdd((unsigned long long*)&L[threadIdx.x], v);
    }
}

// ---- short sides: minima and sums in one launch -----------------------------
// A block takes 32 nodes (a lane each); its eight warps scan an eighth of the
// other side each, every node of it read by a whole warp at once.
__global__ void __launch_bounds__(RW_THREADS) k_rwmd_small(const int32_t* __restrict__ X, const int32_t* __restrict__ Y,
                                                           const int64_t* __restrict__ cnt, int nA, int nB, int blocksA,
                                                           DiagCost dc, int64_t* __restrict__ L) {
    __shared__ unsigned long long m[RW_THREADS / 32][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const bool a = (int)blockIdx.x < blocksA;
    const int first = 32 * ((int)blockIdx.x - (a ? 0 : blocksA)) + lane, np = a ? nA : nB, nq = a ? nB : nA;
    const int u = (a ? 0 : nA) + first;
    const int32_t *qx = X + (a ? nA : 0), *qy = Y + (a ? nA : 0);
    int32_t ux = 0, uy = 0;
    if (first < np) {
        ux = X[u];
        uy = Y[u];
    }
    unsigned long long best = ~0ull;
    const int per = (nq + RW_THREADS / 32 - 1) / (RW_THREADS / 32), q1 = min(nq, (w + 1) * per);
#pragma unroll 4
    for (int q = w * per; q < q1; q++) {
        const long long dx = (long long)(ux - qx[q]), dy = (long long)(uy - qy[q]);
        const unsigned long long d2 = (unsigned long long)(dx * dx) + (unsigned long long)(dy * dy);
        best = d2 < best ? d2 : best;
    }
    m[w][lane] = best;
    __syncthreads();
    if (w != 0) return;
    unsigned long long v = 0;
    if (first < np) {
#pragma unroll
        for (int q = 1; q < RW_THREADS / 32; q++) best = m[q][lane] < best ? m[q][lane] : best;
        int64_t c = cost_make(ux, uy, dc);
        if (best != ~0ull) {
            const int64_t cn = (int64_t)ceil_sqrt_u64(best);
            c = cn < c ? cn : c;
        }
        v = (unsigned long long)(c * cnt[u]);
    }
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0 && v) atomicAdd((unsigned long long*)&L[a ? 0 : 1], v);
}

// One launch instead of three up to here: the scan of a side by one warp's share
// (nq / 8 nodes) is then no longer than the launches saved.
constexpr int64_t RW_SMALL = 8192;

// ---- the same minima through a uniform grid over each side ----------------
// Large sides make the all-pairs scan quadratic (about 10^12 distance
// evaluations at a million nodes a side).  Each side's nodes are bucketed into a
// grid (a counting sort by cell), and every node of the other side searches
// growing squares of cells around its own cell.  After a square of half side K every
// node not yet seen lies beyond one of its sides that are not the grid's border, so
// its distance is at least LB, the distance from the query to the nearest such side.  The
// search stops when LB^2 >= the best squared distance found (the minimum is
// exact), or when LB >= the query's diagonal cost c_make: every unseen node then
// costs at least c_make, the relaxed flow takes min(c(u, nearest), c_make) either
// way, and the stored value min(best, c_make^2) gives the same term.  A query that
// has not stopped at half side RW_KMAX (a far outlier) keeps its best as an upper
// bound and is finished by the all-pairs scan over the other side.
//
// A square grows to what the best distance or the diagonal cost leaves open, by a
// quarter while nothing is found; its new cells are one stretch of nodes a row above
// and below and two a row beside, so that empty space costs a few loads a row and
// RW_KMAX reaches as far as 24 rings of cells of half a node did.
//
// Bound by the distances evaluated and by the gathers of cells.  Diagrams crowd
// near the diagonal, so cells of two nodes on average hold dozens where most
// nodes are: the grid has RW_CELLS cells a node instead.  Queries run in the
// order of their own side's cells, so the lanes of a warp search the same cells.
// pd_rwmd_lower_bound, a side: 1,000,000 nodes (mixture) 3.31 ms with half a cell a
// node, queries by coordinate and single rings, 0.75 so; 100,000 nodes in 40 clusters,
// the other side's elsewhere, 3.2 and 3.2 (8.3 where only single rings, 24 of them,
// reached across 8 cells a node); 300,000 in three clusters on both sides 30 and 25.

constexpr int RW_KMAX = 96;
constexpr int64_t RW_CELLS = 8;
constexpr uint32_t RW_CROWD = 64;  // nodes of a cell that is searched before its neighbours
constexpr int64_t RW_GRID_MIN = int64_t(1) << 28;  // nA * nB from which the grid is used

struct RwGrid {
    int64_t x0, y0, h;  // origin and cell side (quanta)
    int32_t gw, gh;     // cells per axis
    int64_t base;       // first cell of this grid in the shared cell arrays
};

// box[4 s ..] = min x, max x, min y, max y of side s (blockIdx.y).
__global__ void k_rw_box_init(int64_t* box) {
    if (threadIdx.x < 8) box[threadIdx.x] = (threadIdx.x & 1) ? INT64_MIN : INT64_MAX;
}
__global__ void __launch_bounds__(BOX_THREADS) k_rw_box(const int32_t* __restrict__ X, const int32_t* __restrict__ Y,
                                                        int64_t nA, int64_t n, int64_t* __restrict__ box) {
    const int64_t i0 = blockIdx.y ? nA : 0, i1 = blockIdx.y ? n : nA;
    int32_t b[4] = {INT32_MAX, INT32_MIN, INT32_MAX, INT32_MIN};
    for (int64_t i = i0 + (int64_t)blockIdx.x * BOX_THREADS + threadIdx.x; i < i1; i += (int64_t)gridDim.x * BOX_THREADS) {
        b[0] = min(b[0], X[i]);
        b[1] = max(b[1], X[i]);
        b[2] = min(b[2], Y[i]);
        b[3] = max(b[3], Y[i]);
    }
    box_to(b, box + 4 * blockIdx.y);
}

PD_D int32_t rw_cell_axis(int64_t v, int64_t o, int64_t h, int32_t g) {
    if (v < o) return 0;
    const int64_t c = (v - o) / h;
    return c >= g ? g - 1 : (int32_t)c;
}

PD_D uint32_t rw_cell(const RwGrid& g, int32_t x, int32_t y) {
    return (uint32_t)(g.base + (int64_t)rw_cell_axis(y, g.y0, g.h, g.gh) * g.gw + rw_cell_axis(x, g.x0, g.h, g.gw));
}

// Node i of side s goes into grid s (its cell's count).
__global__ void k_rw_hist(const int32_t* __restrict__ X, const int32_t* __restrict__ Y, int64_t nA, int64_t n,
                          RwGrid g0, RwGrid g1, uint32_t* __restrict__ cnt) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) atomicAdd(&cnt[rw_cell(i < nA ? g0 : g1, X[i], Y[i])], 1u);
}

// Nodes placed by cell (order inside a cell is arbitrary: only minima are read),
// with their index.  cur: the cells' starts, moved to their ends.
__global__ void k_rw_scatter(const int32_t* __restrict__ X, const int32_t* __restrict__ Y, int64_t nA, int64_t n,
                             RwGrid g0, RwGrid g1, uint32_t* __restrict__ cur, int2* __restrict__ pts,
                             uint32_t* __restrict__ id) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int2 p = make_int2(X[i], Y[i]);
    const uint32_t k = atomicAdd(&cur[rw_cell(i < nA ? g0 : g1, p.x, p.y)], 1u);
    pts[k] = p;
    id[k] = (uint32_t)i;
}

// Search of the q-th placed node in the other side's grid; see above.  end:
// the cells' ends (a cell starts where the one before it ends).  Unfinished queries
// are listed: side A's from list[0], side B's from list[nA], their counts in nl[0],
// nl[1].
__global__ void k_rw_query(int64_t nA, int64_t n, RwGrid g0, RwGrid g1, const uint32_t* __restrict__ end,
                           const int2* __restrict__ pts, const uint32_t* __restrict__ id, DiagCost dc,
                           unsigned long long* __restrict__ mind2, int32_t* __restrict__ list, int* __restrict__ nl) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const bool sa = q < nA;  // A's grid comes first, and its nodes
    const RwGrid& g = sa ? g1 : g0;
    const int2 u = pts[q];
    const int64_t cm = cost_make(u.x, u.y, dc);
    const int32_t cx = rw_cell_axis(u.x, g.x0, g.h, g.gw), cy = rw_cell_axis(u.y, g.y0, g.h, g.gh);
    unsigned long long best = ~0ull;
    // cells x0 .. x1 of row y hold one stretch of nodes
    auto row = [&](int32_t y, int32_t x0, int32_t x1) {
        const int64_t c = g.base + (int64_t)y * g.gw;
        const uint32_t k1 = end[c + x1];
        for (uint32_t k = c + x0 > 0 ? end[c + x0 - 1] : 0u; k < k1; k++) {
            const int2 v = pts[k];
            const int32_t dx = u.x - v.x, dy = u.y - v.y;  // below 2^30: products of 32 bits
            const unsigned long long d2 = (unsigned long long)((int64_t)dx * dx) + (unsigned long long)((int64_t)dy * dy);
            best = d2 < best ? d2 : best;
        }
    };
    int state = 0;          // 0 searching, 1 exact, 2 stopped by the diagonal cost
    int32_t done = -1;      // half side of the square of cells that is searched
    auto widen = [&](int32_t K) {
        const int32_t xlo = max(cx - K, 0), xhi = min(cx + K, g.gw - 1);
        for (int32_t y = max(cy - K, 0); y <= min(cy + K, g.gh - 1); y++) {
            if (abs(y - cy) > done) {
                row(y, xlo, xhi);
            } else {
                if (cx - done > xlo) row(y, xlo, cx - done - 1);
                if (cx + done < xhi) row(y, cx + done + 1, xhi);
            }
        }
        done = K;
        // distance to the nearest side of the searched square beyond which nodes may remain
        const int64_t ux = u.x, uy = u.y;
        int64_t lb = INT64_MAX;
        if (cx - K > 0) lb = min(lb, ux - (g.x0 + (int64_t)(cx - K) * g.h));
        if (cx + K < g.gw - 1) lb = min(lb, g.x0 + (int64_t)(cx + K + 1) * g.h - ux);
        if (cy - K > 0) lb = min(lb, uy - (g.y0 + (int64_t)(cy - K) * g.h));
        if (cy + K < g.gh - 1) lb = min(lb, g.y0 + (int64_t)(cy + K + 1) * g.h - uy);
        if (lb == INT64_MAX) {
            state = 1;  // the whole grid is searched
        } else {
            lb = lb < 0 ? 0 : lb;
            if ((unsigned long long)lb * (unsigned long long)lb >= best) state = 1;
            else if (lb >= cm) state = 2;
        }
    };
    // a crowded cell by itself first: its neighbours are as crowded, and mostly not needed
    const int64_t own = g.base + (int64_t)cy * g.gw + cx;
    if (end[own] - (own > 0 ? end[own - 1] : 0u) > RW_CROWD) widen(0);
    if (state == 0) widen(1);
    while (state == 0 && done < RW_KMAX) {
        // as far as the best so far and the diagonal leave open, by a quarter while nothing is found
        const float cells = 1.f / (float)g.h;
        const int32_t open = (int32_t)((float)cm * cells);
        const int32_t K = best == ~0ull ? min(done + max(1, done / 4), open) : min((int32_t)(sqrtf((float)best) * cells), open);
        widen(min(max(K, done + 1), RW_KMAX));
    }
    if (state == 2) {
        const unsigned long long c2 = (unsigned long long)cm * (unsigned long long)cm;
        best = c2 < best ? c2 : best;
    }
    const uint32_t i = id[q];
    mind2[i] = best;
    if (state == 0) {
        const int k = atomicAdd(&nl[sa ? 0 : 1], 1);
        list[(sa ? 0 : nA) + k] = (int32_t)(sa ? i : i - nA);
    }
}

// The all-pairs scan for listed queries only (indices within their side);
// blockIdx.z = direction, blockIdx.y splits the other side.
__global__ void __launch_bounds__(RW_THREADS) k_rwmd_min_list(const int32_t* __restrict__ X,
                                                              const int32_t* __restrict__ Y, int64_t nA, int64_t nB,
                                                              const int32_t* __restrict__ list, int nlA, int nlB,
                                                              int64_t chunk, unsigned long long* __restrict__ mind2) {
    __shared__ int2 q[RW_TILE];
    const int dir = blockIdx.z;
    const int64_t pbase = dir == 0 ? 0 : nA, np = dir == 0 ? nlA : nlB;
    const int64_t qbase = dir == 0 ? nA : 0, nq = dir == 0 ? nB : nA;
    const int64_t t = (int64_t)blockIdx.x * RW_THREADS + threadIdx.x;
    const int64_t q0 = (int64_t)blockIdx.y * chunk, q1 = min(nq, q0 + chunk);
    if ((int64_t)blockIdx.x * RW_THREADS >= np || q0 >= q1) return;
    int64_t u = -1;
    int32_t ux = 0, uy = 0;
    if (t < np) {
        u = pbase + list[pbase + t];
        ux = X[u];
        uy = Y[u];
    }
    unsigned long long best = ~0ull;
    for (int64_t t0 = q0; t0 < q1; t0 += RW_TILE) {
        const int tn = (int)min((int64_t)RW_TILE, q1 - t0);
        __syncthreads();
        for (int j = threadIdx.x; j < tn; j += RW_THREADS) q[j] = make_int2(X[qbase + t0 + j], Y[qbase + t0 + j]);
        __syncthreads();
        for (int j = 0; j < tn; j++) {
            const int2 v = q[j];
            const long long dx = (long long)(ux - v.x), dy = (long long)(uy - v.y);
            const unsigned long long d2 = (unsigned long long)(dx * dx) + (unsigned long long)(dy * dy);
            best = d2 < best ? d2 : best;
        }
    }
    if (u >= 0) atomicMin(&mind2[u], best);
}

__global__ void k_fill_u64(unsigned long long* p, int64_t n, unsigned long long v) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = v;
}

// Grid geometry of one side with box b (xmin, xmax, ymin, ymax) and n nodes:
// about `pair` cells for two nodes, at most twice as many and 64.
static RwGrid rw_grid(const int64_t* b, int64_t n, int64_t base, int64_t pair) {
    RwGrid g{};
    const int64_t W = b[1] - b[0], H = b[3] - b[2];
    const int64_t want = std::min<int64_t>(std::max<int64_t>(pair * n / 2, 1), int64_t(1) << 29);  // both grids below 2^32 cells
    const double cells = (double)want;
    int64_t hs = (int64_t)ceil(sqrt((double)(W + 1) * (double)(H + 1) / cells));
    hs = std::max<int64_t>(hs, 1);
    for (;;) {
        const int64_t gw = W / hs + 1, gh = H / hs + 1;
        if (gw * gh <= 2 * want + 64) {
            g.gw = (int32_t)gw;
            g.gh = (int32_t)gh;
            break;
        }
        hs *= 2;
    }
    g.x0 = b[0];
    g.y0 = b[2];
    g.h = hs;
    g.base = base;
    return g;
}

// Exact minima of both directions through the grids (see k_rw_query), the
// queries that it did not finish completed by the all-pairs scan.
static pd_status rwmd_grid(Ctx* c, const Hats& h, DiagCost dc, unsigned long long* mind2, int64_t chunk, int64_t gy,
                           cudaStream_t st) {
    const int64_t n = h.nA + h.nB;
    int64_t* box = bufT<int64_t>(c, B_RW_BOX, 8);
    int* nl = bufT<int>(c, B_RW_NL, 2);
    if (!box || !nl) return PD_ENOMEM;
    k_rw_box_init<<<1, 32, 0, st>>>(box); pd::count_launch();
    k_rw_box<<<dim3(box_grid(c, std::max(h.nA, h.nB)), 2), BOX_THREADS, 0, st>>>(h.X, h.Y, h.nA, n, box); pd::count_launch();
    int64_t hb[8];
    PD_TRY_CUDA(c, cudaMemcpyAsync(hb, box, sizeof(hb), cudaMemcpyDeviceToHost, st));
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));
    RwGrid g0, g1;
    int64_t cells = 0;
    uint32_t* cell = nullptr;
    int2* pts = bufT<int2>(c, B_RW_PTS, n);
    uint32_t* id = bufT<uint32_t>(c, B_RW_CUR, n);
    int32_t* list = bufT<int32_t>(c, B_RW_LIST, n);
    if (!pts || !id || !list) return PD_ENOMEM;
    for (int64_t pair = 2 * RW_CELLS; pair > 0; pair /= 4) {  // fewer cells if memory is short
        g0 = rw_grid(hb, h.nA, 0, pair);
        g1 = rw_grid(hb + 4, h.nB, (int64_t)g0.gw * g0.gh, pair);
        cells = g1.base + (int64_t)g1.gw * g1.gh;
        if (pair > 1 && beyond_cap(c, 4 * cells)) continue;
        cell = bufT<uint32_t>(c, B_RW_START, cells);
        if (cell) break;
        if (pair / 4 > 0) c->err.clear();
    }
    uint32_t* part = bufT<uint32_t>(c, B_SCAN_PART, scan_tiles(cells) + 1);
    if (!cell || !part) return PD_ENOMEM;
    PD_TRY_CUDA(c, cudaMemsetAsync(cell, 0, sizeof(uint32_t) * cells, st));
    PD_TRY_CUDA(c, cudaMemsetAsync(nl, 0, 2 * sizeof(int), st));
    k_rw_hist<<<grid_for(n, 256), 256, 0, st>>>(h.X, h.Y, h.nA, n, g0, g1, cell); pd::count_launch();
    PD_TRY_CUDA(c, exclusive_scan<uint32_t>(cell, cell, cells, part, nullptr, st));
    k_rw_scatter<<<grid_for(n, 256), 256, 0, st>>>(h.X, h.Y, h.nA, n, g0, g1, cell, pts, id); pd::count_launch();
    k_rw_query<<<grid_for(n, 128), 128, 0, st>>>(h.nA, n, g0, g1, cell, pts, id, dc, mind2, list, nl); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    int hn[2];
    PD_TRY_CUDA(c, cudaMemcpyAsync(hn, nl, sizeof(hn), cudaMemcpyDeviceToHost, st));
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));
    if (hn[0] + hn[1] > 0) {
        const int64_t gx = (std::max(hn[0], hn[1]) + RW_THREADS - 1) / RW_THREADS;
        k_rwmd_min_list<<<dim3((unsigned)gx, (unsigned)gy, 2), RW_THREADS, 0, st>>>(h.X, h.Y, h.nA, h.nB, list, hn[0],
                                                                                    hn[1], chunk, mind2); pd::count_launch();
        PD_TRY_CUDA(c, cudaGetLastError());
    }
    return PD_OK;
}

pd_status stage_rwmd(Ctx* c, const Hats& h, int64_t L[3], DiagCost dc, cudaStream_t st) {
    int64_t n = h.nA + h.nB;
    int64_t* sm = bufT<int64_t>(c, B_SMALL, 64);
    unsigned long long* mind2 = bufT<unsigned long long>(c, B_QKEY2, n);
    if (!sm || !mind2) return PD_ENOMEM;
    PD_TRY_CUDA(c, cudaMemsetAsync(sm + S_L0, 0, 2 * sizeof(int64_t), st));
    if (n > 0 && n <= RW_SMALL) {
        const int ba = (int)((h.nA + 31) / 32), bb = (int)((h.nB + 31) / 32);
        k_rwmd_small<<<ba + bb, RW_THREADS, 0, st>>>(h.X, h.Y, h.cnt, (int)h.nA, (int)h.nB, ba, dc, sm + S_L0); pd::count_launch();
        PD_TRY_CUDA(c, cudaGetLastError());
    } else if (n > 0) {
        k_fill_u64<<<grid_for(n, 256), 256, 0, st>>>(mind2, n, ~0ull); pd::count_launch();
        int64_t npmax = h.nA > h.nB ? h.nA : h.nB;
        int64_t gx = (npmax + RW_THREADS - 1) / RW_THREADS;
        int64_t want = 4LL * (c->sm_count > 0 ? c->sm_count : 152);
        int64_t gy = (want + gx - 1) / gx;
        int64_t nqmax = npmax;
        int64_t chunk = (nqmax + gy - 1) / gy;
        if (chunk < 256) chunk = 256;
        gy = (nqmax + chunk - 1) / chunk;
        if (gy < 1) gy = 1;
        if (h.nA > 0 && h.nB > 0 && h.nA * h.nB >= RW_GRID_MIN) {
            PD_TRY(rwmd_grid(c, h, dc, mind2, chunk, gy, st));
        } else if (gx > 0 && h.nA > 0 && h.nB > 0) {
            k_rwmd_min<<<dim3((unsigned)gx, (unsigned)gy, 2), RW_THREADS, 0, st>>>(h.X, h.Y, h.nA, h.nB, chunk, mind2); pd::count_launch();
        }
        k_rwmd_sum<<<box_grid(c, n), BOX_THREADS, 0, st>>>(h.X, h.Y, h.cnt, h.nA, n, mind2, dc, sm + S_L0); pd::count_launch();
        PD_TRY_CUDA(c, cudaGetLastError());
    }
    PD_TRY_CUDA(c, cudaMemcpyAsync(c->h_small, sm, sizeof(int64_t) * S_COUNT, cudaMemcpyDeviceToHost, st));
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));
    L[0] = c->h_small[S_L0];
    L[1] = c->h_small[S_L1];
    L[2] = L[0] > L[1] ? L[0] : L[1];
    return PD_OK;
}

// ---------------------------------------------------------------------------
// delta-condensation (Algorithm 2) and Morton order
// ---------------------------------------------------------------------------

__global__ void __launch_bounds__(BOX_THREADS) k_cells(const int32_t* __restrict__ X, const int32_t* __restrict__ Y,
                                                       int64_t n, int64_t G, int32_t* __restrict__ CX,
                                                       int32_t* __restrict__ CY, int64_t* __restrict__ sm) {
    int32_t box[4] = {INT32_MAX, INT32_MIN, INT32_MAX, INT32_MIN};
    for (int64_t i = (int64_t)blockIdx.x * BOX_THREADS + threadIdx.x; i < n; i += (int64_t)gridDim.x * BOX_THREADS) {
        const int32_t cx = (int32_t)floor_div(2 * (int64_t)X[i] + G, 2 * G);  // nearest lattice point, ties up
        const int32_t cy = (int32_t)floor_div(2 * (int64_t)Y[i] + G, 2 * G);  // |cell| <= 2^29
        CX[i] = cx;
        CY[i] = cy;
        box[0] = min(box[0], cx);
        box[1] = max(box[1], cx);
        box[2] = min(box[2], cy);
        box[3] = max(box[3], cy);
    }
    box_to(box, &sm[S_CMNX]);
}

__global__ void k_cell_keys(const int32_t* __restrict__ CX, const int32_t* __restrict__ CY, int64_t n,
                            const int64_t* __restrict__ sm, int bcy, uint64_t* __restrict__ key,
                            uint32_t* __restrict__ val) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    key[i] = ((uint64_t)(CX[i] - sm[S_CMNX]) << bcy) | (uint64_t)(CY[i] - sm[S_CMNY]);
    val[i] = (uint32_t)i;
}

// One node per distinct cell: place it at G * cell + shift(seed, cell).
__global__ void __launch_bounds__(BOX_THREADS) k_cell_place(const uint64_t* __restrict__ key, int64_t n,
                                                            const int64_t* __restrict__ idx,
                                                            const int64_t* __restrict__ sm, int bcy, int64_t G,
                                                            int64_t P, uint64_t seed, int32_t* __restrict__ NX,
                                                            int32_t* __restrict__ NY, int64_t* __restrict__ CA,
                                                            int64_t* __restrict__ CB, int64_t* __restrict__ smw) {
    int32_t box[4] = {INT32_MAX, INT32_MIN, INT32_MAX, INT32_MIN};
    bool bad = false;
    const uint64_t ymask = bcy >= 64 ? ~0ull : ((1ull << bcy) - 1);
    const int64_t mnx = sm[S_CMNX], mny = sm[S_CMNY];
    for (int64_t i = (int64_t)blockIdx.x * BOX_THREADS + threadIdx.x; i < n; i += (int64_t)gridDim.x * BOX_THREADS) {
        const uint64_t k = key[i];
        if (i > 0 && key[i - 1] == k) continue;
        const int64_t cx = (int64_t)(k >> bcy) + mnx, cy = (int64_t)(k & ymask) + mny;
        int64_t dx, dy;
        cell_shift(seed, cx, cy, P, &dx, &dy);
        const int64_t x = G * cx + dx, y = G * cy + dy, lim = int64_t(1) << 30;
        bad |= x <= -lim || x >= lim || y <= -lim || y >= lim;
        const int64_t j = idx[i];
        NX[j] = (int32_t)x;
        NY[j] = (int32_t)y;
        CA[j] = CB[j] = 0;
        box[0] = min(box[0], (int32_t)x);
        box[1] = max(box[1], (int32_t)x);
        box[2] = min(box[2], (int32_t)y);
        box[3] = max(box[3], (int32_t)y);
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicAdd((unsigned long long*)&smw[S_ERR], 1ull);
    box_to(box, &smw[S_NMNX]);
}

// Aggregate the multiplicities of the nodes snapped into each cell.
__global__ void k_cell_accum(const uint64_t* __restrict__ key, const uint32_t* __restrict__ val, int64_t n,
                             const int64_t* __restrict__ idx, const int64_t* __restrict__ cnt, int64_t nA,
                             int64_t* __restrict__ CA, int64_t* __restrict__ CB) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int64_t j = idx[i] + ((i == 0 || key[i - 1] != key[i]) ? 1 : 0) - 1;
    const uint32_t v = val[i];
    atomicAdd((unsigned long long*)((int64_t)v < nA ? &CA[j] : &CB[j]), (unsigned long long)cnt[v]);
}

__global__ void k_morton_keys(const int32_t* __restrict__ NX, const int32_t* __restrict__ NY, int64_t N,
                              const int64_t* __restrict__ sm, uint64_t* __restrict__ key, uint32_t* __restrict__ val) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    key[i] = morton2((uint32_t)(NX[i] - sm[S_NMNX]), (uint32_t)(NY[i] - sm[S_NMNY]));
    val[i] = (uint32_t)i;
}

__global__ void k_node_gather(const uint64_t* __restrict__ key, const uint32_t* __restrict__ val, int64_t N,
                              const int32_t* __restrict__ NX, const int32_t* __restrict__ NY,
                              const int64_t* __restrict__ CA, const int64_t* __restrict__ CB, int32_t* __restrict__ OX,
                              int32_t* __restrict__ OY, int64_t* __restrict__ OA, int64_t* __restrict__ OB,
                              uint64_t* __restrict__ OC) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const uint32_t v = val[i];
    OX[i] = NX[v];
    OY[i] = NY[v];
    OA[i] = CA[v];
    OB[i] = CB[v];
    OC[i] = key[i];
}

// The whole stage for at most CS_MAX 0-condensed nodes (see k_condense0_small).
__global__ void __launch_bounds__(CS_THREADS) k_condense_delta_small(
    const int32_t* __restrict__ HX, const int32_t* __restrict__ HY, const int64_t* __restrict__ cnt, int nA, int n,
    int64_t G, int64_t P, uint64_t seed, int32_t* __restrict__ NX, int32_t* __restrict__ NY, int64_t* __restrict__ CA,
    int64_t* __restrict__ CB, int32_t* __restrict__ OX, int32_t* __restrict__ OY, int64_t* __restrict__ OA,
    int64_t* __restrict__ OB, uint64_t* __restrict__ OC, int64_t* out) {
    extern __shared__ __align__(16) unsigned char cond_dyn[];
    CtaStage& s = *(CtaStage*)cond_dyn;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int base = w * 32 * CS_ITEMS + lane, p0 = tid * CS_ITEMS;
    if (tid == 0) s.count[0] = 0;
    int32_t box[4] = {INT32_MAX, INT32_MIN, INT32_MAX, INT32_MIN};
    uint64_t key[CS_ITEMS];
    uint32_t val[CS_ITEMS];
    int32_t cx[CS_ITEMS], cy[CS_ITEMS];  // |cell| <= 2^29: 32 bits
#pragma unroll
    for (int q = 0; q < CS_ITEMS; q++) {
        const int i = base + 32 * q;
        cx[q] = cy[q] = 0;
        if (i < n) {
            cx[q] = (int32_t)floor_div(2 * (int64_t)HX[i] + G, 2 * G);  // nearest lattice point, ties up
            cy[q] = (int32_t)floor_div(2 * (int64_t)HY[i] + G, 2 * G);
            box[0] = min(box[0], cx[q]);
            box[1] = max(box[1], cx[q]);
            box[2] = min(box[2], cy[q]);
            box[3] = max(box[3], cy[q]);
        }
    }
    cta_box(s, box);
    const int bcx = dev_bits_for((uint32_t)(box[1] - box[0])), bcy = dev_bits_for((uint32_t)(box[3] - box[2]));
#pragma unroll
    for (int q = 0; q < CS_ITEMS; q++) {
        const int i = base + 32 * q;
        key[q] = i < n ? (uint64_t)(uint32_t)(cx[q] - box[0]) << bcy | (uint32_t)(cy[q] - box[2]) : ~0ull;
        val[q] = (uint32_t)i;
    }
    cta_sort(s.sort, key, val, bcx + bcy);
    // one node per distinct cell, at G * cell + shift(seed, cell)
    uint32_t heads = 0;
#pragma unroll
    for (int q = 0; q < CS_ITEMS; q++) {
        const int i = p0 + q;
        if (i < n && (i == 0 || s.sort.key[i - 1] != s.sort.key[i])) heads |= 1u << q;
    }
    uint32_t N;
    const uint32_t j0 = block_excl_scan<uint32_t>(__popc(heads), &N);
    int32_t nb[4] = {INT32_MAX, INT32_MIN, INT32_MAX, INT32_MIN};
    uint32_t bad = 0, j = j0;
    for (uint32_t h = heads; h; h &= h - 1, j++) {
        const uint64_t kk = s.sort.key[p0 + __ffs(h) - 1];
        const int64_t ccx = (int64_t)(kk >> bcy) + box[0], ccy = (int64_t)(kk & ((1ull << bcy) - 1)) + box[2];
        int64_t dx, dy;
        cell_shift(seed, ccx, ccy, P, &dx, &dy);
        const int64_t X = G * ccx + dx, Y = G * ccy + dy, lim = int64_t(1) << 30;
        bad |= X <= -lim || X >= lim || Y <= -lim || Y >= lim;
        NX[j] = (int32_t)X;
        NY[j] = (int32_t)Y;
        CA[j] = CB[j] = 0;
        nb[0] = min(nb[0], (int32_t)X);
        nb[1] = max(nb[1], (int32_t)X);
        nb[2] = min(nb[2], (int32_t)Y);
        nb[3] = max(nb[3], (int32_t)Y);
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) s.count[0] = 1;
    cta_box(s, nb);  // (and every CA, CB is zero)
    if (s.count[0]) {
        if (tid == 0) out[S_ERR] = 1;
        return;
    }
    // multiplicities of the nodes snapped into each cell
    j = j0;
#pragma unroll
    for (int q = 0; q < CS_ITEMS; q++) {
        const int i = p0 + q;
        if (i < n) {
            j += heads >> q & 1u;
            const uint32_t v = s.sort.val[i];
            atomicAdd((unsigned long long*)((int)v < nA ? &CA[j - 1] : &CB[j - 1]), (unsigned long long)cnt[v]);
        }
    }
    __syncthreads();
    // Morton order
#pragma unroll
    for (int q = 0; q < CS_ITEMS; q++) {
        const int i = base + 32 * q;
        key[q] = i < (int)N ? morton2((uint32_t)NX[i] - (uint32_t)nb[0], (uint32_t)NY[i] - (uint32_t)nb[2]) : ~0ull;
        val[q] = (uint32_t)i;
    }
    const int bm = dev_bits_for(max((uint32_t)nb[1] - (uint32_t)nb[0], (uint32_t)nb[3] - (uint32_t)nb[2]));
    __syncthreads();
    cta_sort(s.sort, key, val, 2 * bm);
#pragma unroll
    for (int q = 0; q < CS_ITEMS; q++) {
        const int i = base + 32 * q;
        if (i < (int)N) {
            const uint32_t v = val[q];
            OX[i] = NX[v];
            OY[i] = NY[v];
            OA[i] = __ldcg(&CA[v]);  // summed by atomics: not through L1
            OB[i] = __ldcg(&CB[v]);
            OC[i] = key[q];
        }
    }
    if (tid == 0) {
        out[S_ERR] = 0;
        out[S_N] = N;
    }
}

pd_status stage_condense_delta(Ctx* c, const Hats& hats, int64_t G, int64_t P, uint64_t seed, pd_nodes* out,
                               cudaStream_t st) {
    const Hats& h = hats;
    int64_t n = h.nA + h.nB;
    out->n_nodes = 0;
    out->X = bufT<int32_t>(c, B_NX, n);
    out->Y = bufT<int32_t>(c, B_NY, n);
    out->cntA = bufT<int64_t>(c, B_NCA, n);
    out->cntB = bufT<int64_t>(c, B_NCB, n);
    out->morton = bufT<uint64_t>(c, B_NCODE, n);
    int64_t* sm = bufT<int64_t>(c, B_SMALL, 64);
    if (!out->X || !out->Y || !out->cntA || !out->cntB || !out->morton || !sm) return PD_ENOMEM;
    if (n == 0) return PD_OK;
    if (n <= CS_MAX) {
        int32_t* NX = bufT<int32_t>(c, B_QX, n);
        int32_t* NY = bufT<int32_t>(c, B_QY, n);
        int64_t* CA = bufT<int64_t>(c, B_CA, n);
        int64_t* CB = bufT<int64_t>(c, B_CB, n);
        if (!NX || !NY || !CA || !CB) return PD_ENOMEM;
        int64_t* hs = c->h_small;
        static std::atomic<uint64_t> done{0};
        PD_TRY(smem_limit(c, done, (const void*)k_condense_delta_small, sizeof(CtaStage)));
        k_condense_delta_small<<<1, CS_THREADS, sizeof(CtaStage), st>>>(hats.X, hats.Y, hats.cnt, (int)hats.nA, (int)n, G, P,
                                                                        seed, NX, NY, CA, CB, out->X, out->Y, out->cntA,
                                                                        out->cntB, out->morton, hs); pd::count_launch();
        PD_TRY_CUDA(c, cudaGetLastError());
        PD_TRY_CUDA(c, cudaStreamSynchronize(st));
        if (hs[S_ERR]) return fail(c, PD_EINVAL, "condensed node coordinate outside (-2^30, 2^30)");
        out->n_nodes = hs[S_N];
        return PD_OK;
    }
    int32_t* CX = bufT<int32_t>(c, B_CX, n);
    int32_t* CY = bufT<int32_t>(c, B_CY, n);
    uint64_t* key = bufT<uint64_t>(c, B_CKEY, n);
    uint64_t* key2 = bufT<uint64_t>(c, B_CKEY2, n);
    uint32_t* val = bufT<uint32_t>(c, B_CVAL, n);
    uint32_t* val2 = bufT<uint32_t>(c, B_CVAL2, n);
    int64_t* idx = bufT<int64_t>(c, B_CIDX, n);
    int32_t* NX = bufT<int32_t>(c, B_QX, n);
    int32_t* NY = bufT<int32_t>(c, B_QY, n);
    int64_t* CA = bufT<int64_t>(c, B_CA, n);
    int64_t* CB = bufT<int64_t>(c, B_CB, n);
    if (!CX || !CY || !key || !key2 || !val || !val2 || !idx || !NX || !NY || !CA || !CB) return PD_ENOMEM;
    k_init_small<<<1, 64, 0, st>>>(sm); pd::count_launch();
    k_cells<<<box_grid(c, n), BOX_THREADS, 0, st>>>(h.X, h.Y, n, G, CX, CY, sm); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    PD_TRY_CUDA(c, cudaMemcpyAsync(c->h_small, sm, sizeof(int64_t) * S_COUNT, cudaMemcpyDeviceToHost, st));
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));
    int64_t* hs = c->h_small;
    int bcx = bits_for((uint64_t)(hs[S_CMXX] - hs[S_CMNX])), bcy = bits_for((uint64_t)(hs[S_CMXY] - hs[S_CMNY]));
    k_cell_keys<<<grid_for(n, 256), 256, 0, st>>>(CX, CY, n, sm, bcy, key, val); pd::count_launch();
    PD_TRY(sort_u64(c, key, key2, val, val2, n, bcx + bcy, st));
    k_run_flags<<<grid_for(n, 256), 256, 0, st>>>(key, n, ~0ull, idx); pd::count_launch();
    PD_TRY(scan_i64(c, idx, idx, n, sm + S_N, st));
    k_cell_place<<<box_grid(c, n), BOX_THREADS, 0, st>>>(key, n, idx, sm, bcy, G, P, seed, NX, NY, CA, CB, sm); pd::count_launch();
    k_cell_accum<<<grid_for(n, 256), 256, 0, st>>>(key, val, n, idx, h.cnt, h.nA, CA, CB); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    PD_TRY_CUDA(c, cudaMemcpyAsync(c->h_small, sm, sizeof(int64_t) * S_COUNT, cudaMemcpyDeviceToHost, st));
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));
    if (hs[S_ERR]) return fail(c, PD_EINVAL, "condensed node coordinate outside (-2^30, 2^30)");
    int64_t N = hs[S_N];
    int bm = bits_for((uint64_t)(hs[S_NMXX] - hs[S_NMNX]));
    int bm2 = bits_for((uint64_t)(hs[S_NMXY] - hs[S_NMNY]));
    if (bm2 > bm) bm = bm2;
    k_morton_keys<<<grid_for(N, 256), 256, 0, st>>>(NX, NY, N, sm, key, val); pd::count_launch();
    PD_TRY(sort_u64(c, key, key2, val, val2, N, 2 * bm, st));
    k_node_gather<<<grid_for(N, 256), 256, 0, st>>>(key, val, N, NX, NY, CA, CB, out->X, out->Y, out->cntA,
                                                      out->cntB, out->morton); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    out->n_nodes = N;
    return PD_OK;
}

}  // namespace pd
