// The potential predictor of the warm start: per transportation node, 68
// features -> 128 -> 128 -> 1 (ReLU), weights stored in bf16 with float32
// master copies for the optimiser, every product accumulated in float32.
// Forward, backward and Adam are this file's kernels; the predictor and its
// training are not part of the paper (its solver always starts cold).
//
// Features of a node at (X, Y) of a pair whose condensed nodes span the box
// [x0, x0 + ext] x [y0, y0 + ext]:
//   0, 1   (X - x0) / ext, (Y - y0) / ext
//   2, 3   log(1 + cntA), log(1 + cntB)
//   4..67  an 8 x 8 window of a 64 x 64 grid over the box around the node's
//          grid cell (offsets -4..3 on each axis): per cell the signed supply
//          sum(cntA - cntB) of the nodes in it, as sign * log(1 + |sum|)
//   68     half the gap between the coarse optimum's two c-transform
//          envelopes at the node, over the coarse cell Gc (at most 16)
//   69     +1 for a source, -1 for a sink
//   70, 71 offset of the node from its coarse lattice point, over Gc
//          (in [-1/2, 1/2]); 68, 70, 71 are 0 without a coarse solve
// Target / output: the correction from the coarse solve's potential to the
// optimal one (each less its mean over the largest component of the optimal
// simplex tree), over Gc (the box's side without a coarse solve); nodes
// outside that component are left out of the loss.
#include <math.h>

#include <algorithm>
#include <chrono>
#include <cstring>
#include <memory>
#include <new>
#include <vector>

#include <cuda_bf16.h>

#include "mlp.cuh"

namespace pd {

// ---------------------------------------------------------------------------
// features
// ---------------------------------------------------------------------------

__global__ void k_box(const int32_t* __restrict__ X, const int32_t* __restrict__ Y, int64_t N,
                      long long* __restrict__ box) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    long long mnx = LLONG_MAX, mny = LLONG_MAX, mxx = LLONG_MIN, mxy = LLONG_MIN;
    if (i < N) {
        mnx = mxx = X[i];
        mny = mxy = Y[i];
    }
    for (int o = 16; o > 0; o >>= 1) {
        mnx = min(mnx, __shfl_xor_sync(0xffffffffu, mnx, o));
        mny = min(mny, __shfl_xor_sync(0xffffffffu, mny, o));
        mxx = max(mxx, __shfl_xor_sync(0xffffffffu, mxx, o));
        mxy = max(mxy, __shfl_xor_sync(0xffffffffu, mxy, o));
    }
    if ((threadIdx.x & 31) == 0 && mxx != LLONG_MIN) {
        atomicMin(&box[0], mnx);
        atomicMin(&box[1], mny);
        atomicMax(&box[2], mxx);
        atomicMax(&box[3], mxy);
    }
}

PD_D int grid_cell(int32_t v, long long v0, long long ext) {
    long long g = ((long long)v - v0) * WS_GRID / (ext + 1);
    return (int)(g < 0 ? 0 : (g >= WS_GRID ? WS_GRID - 1 : g));
}

__global__ void k_grid(const int32_t* __restrict__ X, const int32_t* __restrict__ Y,
                       const int64_t* __restrict__ cntA, const int64_t* __restrict__ cntB, int64_t N,
                       const long long* __restrict__ box, float* __restrict__ grid) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const long long ext = max(box[2] - box[0], box[3] - box[1]);
    const int gx = grid_cell(X[i], box[0], ext), gy = grid_cell(Y[i], box[1], ext);
    atomicAdd(&grid[gx * WS_GRID + gy], (float)(cntA[i] - cntB[i]));
}

// Features of the transportation nodes: sources S, sinks T (condensed node
// ids); rows nS + nT (the diagonal node) get no row.
__global__ void k_features(const int32_t* __restrict__ X, const int32_t* __restrict__ Y,
                           const int64_t* __restrict__ cntA, const int64_t* __restrict__ cntB,
                           const int32_t* __restrict__ S, const int32_t* __restrict__ T, int64_t nS, int64_t nT,
                           const long long* __restrict__ box, const float* __restrict__ grid,
                           const double* __restrict__ gap, int64_t Gc, __nv_bfloat16* __restrict__ F) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nS + nT) return;
    const int32_t u = r < nS ? S[r] : T[r - nS];
    const long long ext = max(max(box[2] - box[0], box[3] - box[1]), 1LL);
    __nv_bfloat16* f = F + r * WS_IN;
    f[0] = __float2bfloat16((float)((double)((long long)X[u] - box[0]) / (double)ext));
    f[1] = __float2bfloat16((float)((double)((long long)Y[u] - box[1]) / (double)ext));
    f[2] = __float2bfloat16(log1pf((float)cntA[u]));
    f[3] = __float2bfloat16(log1pf((float)cntB[u]));
    const int gx = grid_cell(X[u], box[0], ext), gy = grid_cell(Y[u], box[1], ext);
    for (int dx = 0; dx < 8; dx++)
        for (int dy = 0; dy < 8; dy++) {
            const int cx = gx + dx - 4, cy = gy + dy - 4;
            float v = 0.f;
            if (cx >= 0 && cx < WS_GRID && cy >= 0 && cy < WS_GRID) v = grid[cx * WS_GRID + cy];
            f[4 + dx * 8 + dy] = __float2bfloat16(v < 0.f ? -log1pf(-v) : log1pf(v));
        }
    float g = 0.f, ox = 0.f, oy = 0.f;
    if (Gc > 0) {
        g = gap ? (float)fmin(gap[r] / (double)Gc, 16.0) : 0.f;
        // the coarse lattice point of Algorithm 2's snapping: floor((2X + Gc) / (2 Gc)) Gc
        const int64_t cx = floor_div(2 * (int64_t)X[u] + Gc, 2 * Gc), cy = floor_div(2 * (int64_t)Y[u] + Gc, 2 * Gc);
        ox = (float)((double)((int64_t)X[u] - cx * Gc) / (double)Gc);
        oy = (float)((double)((int64_t)Y[u] - cy * Gc) / (double)Gc);
    }
    f[68] = __float2bfloat16(g);
    f[69] = __float2bfloat16(r < nS ? 1.f : -1.f);
    f[70] = __float2bfloat16(ox);
    f[71] = __float2bfloat16(oy);
}

// The child of the root above node v in the solved tree (its component).
PD_D int32_t tree_component(const int32_t* __restrict__ parent, int32_t v, int32_t root, int32_t limit) {
    for (int32_t k = 0; k < limit; k++) {
        const int32_t p = parent[v];
        if (p == root || p < 0) return v;
        v = p;
    }
    return -1;
}

// Component (child of the root) of every transportation node in the solved
// tree, and the component sizes.
__global__ void k_components(const int32_t* __restrict__ parent, int64_t n, int32_t root, int32_t* __restrict__ comp,
                             int32_t* __restrict__ size) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int32_t c = tree_component(parent, (int32_t)r, root, root + 1);
    comp[r] = c;
    if (c >= 0) atomicAdd(&size[c], 1);
}

__global__ void k_component_sum(const int64_t* __restrict__ pi, const int32_t* __restrict__ comp, int64_t n,
                                int32_t anchor, unsigned long long* __restrict__ sum) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < n && comp[r] == anchor) atomicAdd(sum, (unsigned long long)pi[r]);  // two's complement sum
}

// Targets: (pi(node) - mean pi of the largest component) / ext for the nodes
// of the largest component of the optimal tree (mask 1).  The other
// components hang from the root by artificial arcs, which fix their
// potentials only up to an offset of their own; a common offset does not
// matter to the start (only differences enter reduced costs).
// Target of row r: its optimal potential minus the anchor component's mean,
// less the same for the base potentials (a coarse solve's) when given, over
// `scale` (the coarse cell; the node box's side when 0); rows outside the
// anchor component are masked out.
__global__ void k_targets(const int64_t* __restrict__ pi, const int32_t* __restrict__ comp, int64_t n,
                          int32_t anchor, double mean, const double* __restrict__ base, double base_mean,
                          const long long* __restrict__ box, int64_t scale, float* __restrict__ t,
                          float* __restrict__ mask) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const long long ext = scale > 0 ? (long long)scale : max(max(box[2] - box[0], box[3] - box[1]), 1LL);
    const bool ok = comp[r] == anchor;
    const double b = base ? base[r] - base_mean : 0.0;
    t[r] = ok ? (float)(((double)pi[r] - mean - b) / (double)ext) : 0.f;
    mask[r] = ok ? 1.f : 0.f;
}

// Potentials from the distance to the diagonal: +d(u) for a source, -d(v)
// for a sink, 0 for the diagonal node, so that the reduced cost of an arc is
// c(u, v) - d(u) - d(v) <= 0: minus the saving of sending u to v instead of
// both to the diagonal.
__global__ void k_diag_potentials(const int32_t* __restrict__ X, const int32_t* __restrict__ Y,
                                  const int32_t* __restrict__ S, const int32_t* __restrict__ T, int64_t nS, int64_t nT,
                                  float* __restrict__ p, DiagCost dc) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r > nS + nT) return;
    if (r == nS + nT) {
        p[r] = 0.f;
        return;
    }
    const int32_t u = r < nS ? S[r] : T[r - nS];
    const float d = (float)cost_make(X[u], Y[u], dc);
    p[r] = r < nS ? d : -d;
}

pd_status ws_diag_potentials(Ctx* c, const pd_nodes& nodes, const W1Prep& w, std::vector<float>* p, cudaStream_t st) {
    const int64_t n = w.nS + w.nT;
    float* dp = bufT<float>(c, B_WS_PS, n + 1);
    if (!dp) return PD_ENOMEM;
    k_diag_potentials<<<grid_for(n + 1, 256), 256, 0, st>>>(nodes.X, nodes.Y, w.S, w.T, w.nS, w.nT, dp, w.dc); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    p->resize((size_t)(n + 1));
    PD_TRY_CUDA(c, cudaMemcpyAsync(p->data(), dp, sizeof(float) * (n + 1), cudaMemcpyDeviceToHost, st));
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));
    return PD_OK;
}

// ---------------------------------------------------------------------------
// the network: tiles of WS_TILE rows, one block of WS_THREADS threads each
// ---------------------------------------------------------------------------
//
// 25,728 multiply-adds a row forward, twice that backward, in float32 (weights
// bf16): the CUDA cores' work, so what matters is multiply-adds per shared-memory
// load and enough blocks.  Activations lie transposed, [unit][row], so that one
// 16-byte load gives a unit for four rows: a thread computes 4 rows x 2 units
// of a layer (8 multiply-adds per two loads) and 8 x 8 of the 128 x 128 weight
// gradients (256 per 16 loads), the latter in registers over all tiles of its
// block.  16 rows a tile: the 2,048 rows of a training step fill 128 SMs.  With 32
// rows, one unit a thread, gradients summed in shared memory and the features
// rounded on the host, pd_ws_grad took 335 microseconds on 2,048 rows and
// pd_ws_forward 207; now 115 and 59, copies included.

struct MlpW {
    const __nv_bfloat16* W1;  // [WS_IN][WS_H]
    const float* b1;          // [WS_H]
    const __nv_bfloat16* W2;  // [WS_H][WS_H]
    const float* b2;
    const __nv_bfloat16* w3;  // [WS_H]
    const float* b3;          // [1]
};

constexpr int WS_THREADS = 256;
// Floats between units, for 16-byte loads: no conflicts in the products, two ways where
// they are stored; the gradients' lanes lie 8 and 4 units apart, eight and four ways.
constexpr int WS_LD = WS_TILE + 4;

// Thread t: rows 4 (t / 64) .. + 3, units 2 (t % 64) and the next.
struct MlpTile {
    float x[WS_IN][WS_LD];
    float h1[WS_H][WS_LD];    // then delta1
    float h2[WS_H][WS_LD];    // delta2
    float out[2][WS_TILE];    // the output's two half sums, then delta3 in out[0]
    float sums[4][3][WS_H];   // per group of rows: gradients of b1, b2, w3
    float loss[3];            // gradient of b3, loss, mask
};

PD_D void tile_load(MlpTile& s, const __nv_bfloat16* __restrict__ F, int64_t r0, int nrow) {
    for (int t = threadIdx.x; t < WS_TILE * WS_IN; t += WS_THREADS) {
        const int r = t / WS_IN, k = t - r * WS_IN;
        s.x[k][r] = r < nrow ? __bfloat162float(F[(r0 + r) * WS_IN + k]) : 0.f;
    }
}

// acc[row][unit] += sum over K of in[k][rows] w[k][units] (w: rows of WS_H bf16)
template <int K>
PD_D void tile_product(const float (*in)[WS_LD], const __nv_bfloat16* __restrict__ w, int row, int unit,
                       float (&acc)[4][2]) {
#pragma unroll 8
    for (int k = 0; k < K; k++) {
        const float4 v = *(const float4*)&in[k][row];
        const float2 f = __bfloat1622float2(*(const __nv_bfloat162*)(w + k * WS_H + unit));
        acc[0][0] = fmaf(v.x, f.x, acc[0][0]);
        acc[0][1] = fmaf(v.x, f.y, acc[0][1]);
        acc[1][0] = fmaf(v.y, f.x, acc[1][0]);
        acc[1][1] = fmaf(v.y, f.y, acc[1][1]);
        acc[2][0] = fmaf(v.z, f.x, acc[2][0]);
        acc[2][1] = fmaf(v.z, f.y, acc[2][1]);
        acc[3][0] = fmaf(v.w, f.x, acc[3][0]);
        acc[3][1] = fmaf(v.w, f.y, acc[3][1]);
    }
}

// x -> h1 (kept), h2 (registers), out[0] + out[1].  Ends with a barrier.
PD_D void tile_forward(MlpTile& s, const MlpW& w, float (&h2)[4][2]) {
    const int tid = threadIdx.x, unit = 2 * (tid & 63), row = 4 * (tid >> 6);
    float a[4][2] = {};
    tile_product<WS_IN>(s.x, w.W1, row, unit, a);
#pragma unroll
    for (int c = 0; c < 2; c++) {
        const float b = w.b1[unit + c];
        *(float4*)&s.h1[unit + c][row] = make_float4(fmaxf(a[0][c] + b, 0.f), fmaxf(a[1][c] + b, 0.f),
                                                     fmaxf(a[2][c] + b, 0.f), fmaxf(a[3][c] + b, 0.f));
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; r++) h2[r][0] = h2[r][1] = 0.f;
    tile_product<WS_H>(s.h1, w.W2, row, unit, h2);
    float o[4];
    const float2 w3 = __bfloat1622float2(*(const __nv_bfloat162*)(w.w3 + unit));
#pragma unroll
    for (int r = 0; r < 4; r++) {
        h2[r][0] = fmaxf(h2[r][0] + w.b2[unit], 0.f);
        h2[r][1] = fmaxf(h2[r][1] + w.b2[unit + 1], 0.f);
        o[r] = fmaf(h2[r][0], w3.x, h2[r][1] * w3.y);
        for (int q = 16; q > 0; q >>= 1) o[r] += __shfl_xor_sync(0xffffffffu, o[r], q);
    }
    if ((tid & 31) == 0)
#pragma unroll
        for (int r = 0; r < 4; r++) s.out[(tid >> 5) & 1][row + r] = o[r];
    __syncthreads();
}

__global__ void __launch_bounds__(WS_THREADS) k_mlp_forward(MlpW w, const __nv_bfloat16* __restrict__ F, int64_t n,
                                                            float* __restrict__ y) {
    __shared__ __align__(16) MlpTile s;
    for (int64_t r0 = (int64_t)blockIdx.x * WS_TILE; r0 < n; r0 += (int64_t)gridDim.x * WS_TILE) {
        const int nrow = (int)min((int64_t)WS_TILE, n - r0);
        __syncthreads();
        tile_load(s, F, r0, nrow);
        __syncthreads();
        float h2[4][2];
        tile_forward(s, w, h2);
        if (threadIdx.x < nrow) y[r0 + threadIdx.x] = s.out[0][threadIdx.x] + s.out[1][threadIdx.x] + w.b3[0];
    }
}

// Loss sum(mask * (y - t)^2) / sum(mask) and its gradients; every block sums
// its tiles' gradients into its own row of `part` (WS_NPARAMS floats + 2:
// loss sum, mask sum), reduced afterwards in a fixed order.
__global__ void __launch_bounds__(WS_THREADS) k_mlp_backward(MlpW w, const __nv_bfloat16* __restrict__ F,
                                                             const float* __restrict__ tgt,
                                                             const float* __restrict__ mask, int64_t n, float inv_norm,
                                                             float* __restrict__ part) {
    extern __shared__ __align__(16) unsigned char mlp_dyn[];
    MlpTile& s = *(MlpTile*)mlp_dyn;
    __nv_bfloat16* wt = (__nv_bfloat16*)(&s + 1);  // W2 transposed: [unit of layer 2][unit of layer 1]
    const int tid = threadIdx.x, unit = 2 * (tid & 63), row = 4 * (tid >> 6);
    const int k2 = 8 * (tid >> 4), j2 = 8 * (tid & 15);  // this thread's 8 x 8 of W2's gradient
    const int k1 = 9 * (tid >> 5), j1 = 4 * (tid & 31);  // ... and 9 x 4 of W1's
    for (int t = tid; t < WS_H * WS_H; t += WS_THREADS) wt[(t & (WS_H - 1)) * WS_H + (t >> 7)] = w.W2[t];
    float g2[8][8] = {}, g1[9][4] = {}, gb1[2] = {}, gb2[2] = {}, gw3[2] = {}, gl[3] = {};
    const float2 w3 = __bfloat1622float2(*(const __nv_bfloat162*)(w.w3 + unit));
    for (int64_t r0 = (int64_t)blockIdx.x * WS_TILE; r0 < n; r0 += (int64_t)gridDim.x * WS_TILE) {
        const int nrow = (int)min((int64_t)WS_TILE, n - r0);
        __syncthreads();
        tile_load(s, F, r0, nrow);
        __syncthreads();
        float h2[4][2];
        tile_forward(s, w, h2);
        // delta3 = 2 mask (y - t) / norm; rows past the end have none
        float d3 = 0.f;
        if (tid < nrow) {
            const float e = s.out[0][tid] + s.out[1][tid] + w.b3[0] - tgt[r0 + tid], mk = mask[r0 + tid];
            d3 = 2.f * mk * e * inv_norm;
            gl[0] += d3;
            gl[1] += mk * e * e;
            gl[2] += mk;
        }
        __syncthreads();
        if (tid < WS_TILE) s.out[0][tid] = d3;
        __syncthreads();
        // delta2 = delta3 w3 relu'(h2)
        {
            const float4 d = *(const float4*)&s.out[0][row];
            const float dr[4] = {d.x, d.y, d.z, d.w};
            float d2[2][4];
#pragma unroll
            for (int r = 0; r < 4; r++) {
                gw3[0] = fmaf(h2[r][0], dr[r], gw3[0]);
                gw3[1] = fmaf(h2[r][1], dr[r], gw3[1]);
                d2[0][r] = h2[r][0] > 0.f ? dr[r] * w3.x : 0.f;
                d2[1][r] = h2[r][1] > 0.f ? dr[r] * w3.y : 0.f;
                gb2[0] += d2[0][r];
                gb2[1] += d2[1][r];
            }
#pragma unroll
            for (int c = 0; c < 2; c++)
                *(float4*)&s.h2[unit + c][row] = make_float4(d2[c][0], d2[c][1], d2[c][2], d2[c][3]);
        }
        __syncthreads();
        // delta1 = (delta2 W2^T) relu'(h1), and W2's gradient from the h1 it replaces
        float d1[4][2] = {};
        tile_product<WS_H>(s.h2, wt, row, unit, d1);
#pragma unroll
        for (int r = 0; r < WS_TILE; r += 4) {
            float4 b[8];
#pragma unroll
            for (int q = 0; q < 8; q++) b[q] = *(const float4*)&s.h2[j2 + q][r];
#pragma unroll
            for (int p = 0; p < 8; p++) {
                const float4 a = *(const float4*)&s.h1[k2 + p][r];
#pragma unroll
                for (int q = 0; q < 8; q++)
                    g2[p][q] = fmaf(a.x, b[q].x, fmaf(a.y, b[q].y, fmaf(a.z, b[q].z, fmaf(a.w, b[q].w, g2[p][q]))));
            }
        }
#pragma unroll
        for (int c = 0; c < 2; c++) {
            const float4 h = *(const float4*)&s.h1[unit + c][row];
            d1[0][c] = h.x > 0.f ? d1[0][c] : 0.f;
            d1[1][c] = h.y > 0.f ? d1[1][c] : 0.f;
            d1[2][c] = h.z > 0.f ? d1[2][c] : 0.f;
            d1[3][c] = h.w > 0.f ? d1[3][c] : 0.f;
            gb1[c] += (d1[0][c] + d1[1][c]) + (d1[2][c] + d1[3][c]);
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < 2; c++)
            *(float4*)&s.h1[unit + c][row] = make_float4(d1[0][c], d1[1][c], d1[2][c], d1[3][c]);
        __syncthreads();
#pragma unroll
        for (int r = 0; r < WS_TILE; r += 4) {
            float4 b[4];
#pragma unroll
            for (int q = 0; q < 4; q++) b[q] = *(const float4*)&s.h1[j1 + q][r];
#pragma unroll
            for (int p = 0; p < 9; p++) {
                const float4 a = *(const float4*)&s.x[k1 + p][r];
#pragma unroll
                for (int q = 0; q < 4; q++)
                    g1[p][q] = fmaf(a.x, b[q].x, fmaf(a.y, b[q].y, fmaf(a.z, b[q].z, fmaf(a.w, b[q].w, g1[p][q]))));
            }
        }
    }
    // layout of a gradient row: W1, b1, W2, b2, w3, b3, then loss sum, mask sum
    float* out = part + (int64_t)blockIdx.x * WS_PART;
#pragma unroll
    for (int p = 0; p < 9; p++)
#pragma unroll
        for (int q = 0; q < 4; q++) out[WS_OFF_W1 + (k1 + p) * WS_H + j1 + q] = g1[p][q];
#pragma unroll
    for (int p = 0; p < 8; p++)
#pragma unroll
        for (int q = 0; q < 8; q++) out[WS_OFF_W2 + (k2 + p) * WS_H + j2 + q] = g2[p][q];
#pragma unroll
    for (int c = 0; c < 2; c++) {
        s.sums[tid >> 6][0][unit + c] = gb1[c];
        s.sums[tid >> 6][1][unit + c] = gb2[c];
        s.sums[tid >> 6][2][unit + c] = gw3[c];
    }
    if (tid < 32)
#pragma unroll
        for (int q = 0; q < 3; q++) {
            for (int o = 16; o > 0; o >>= 1) gl[q] += __shfl_xor_sync(0xffffffffu, gl[q], o);
            if (tid == 0) s.loss[q] = gl[q];
        }
    __syncthreads();
    for (int t = tid; t < 3 * WS_H; t += WS_THREADS) {
        const int q = t / WS_H, j = t - q * WS_H;
        out[(q == 0 ? WS_OFF_B1 : q == 1 ? WS_OFF_B2 : WS_OFF_W3) + j] =
            (s.sums[0][q][j] + s.sums[1][q][j]) + (s.sums[2][q][j] + s.sums[3][q][j]);
    }
    if (tid == 0) {
        out[WS_OFF_B3] = s.loss[0];
        out[WS_NPARAMS] = s.loss[1];
        out[WS_NPARAMS + 1] = s.loss[2];
    }
}

// Sum of the blocks' rows, in pairs of pairs: the rounding error of 128 rows is
// that of 7 additions and not of 127 (2,048 rows against 64 bits, six seeds: relative
// error 0.5 .. 1.6e-7; 1.7 .. 2.3e-7 one after the other; 110 and 112 us a call).
// A warp takes 32 columns of every eighth row.
constexpr int RP_GROUPS = 8, RP_ROWS = 32;
constexpr int WS_BLOCKS = RP_GROUPS * RP_ROWS;  // rows at most
__global__ void __launch_bounds__(32 * RP_GROUPS) k_reduce_parts(const float* __restrict__ part, int nb,
                                                                 float* __restrict__ g) {
    __shared__ float s[RP_GROUPS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, t = blockIdx.x * 32 + lane;
    float v[RP_ROWS];
#pragma unroll
    for (int q = 0; q < RP_ROWS; q++) {
        const int b = q * RP_GROUPS + w;
        v[q] = b < nb && t < WS_PART ? part[(int64_t)b * WS_PART + t] : 0.f;
    }
#pragma unroll
    for (int half = RP_ROWS / 2; half > 0; half /= 2)
#pragma unroll
        for (int q = 0; q < half; q++) v[q] += v[q + half];
    s[w][lane] = v[0];
    for (int half = RP_GROUPS / 2; half > 0; half /= 2) {
        __syncthreads();
        if (w < half) s[w][lane] += s[w + half][lane];
    }
    if (w == 0 && t < WS_PART) g[t] = s[0][lane];
}

// Adam on the float32 master weights; bf16 copies of the weight matrices.
__global__ void k_adam(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ g, float lr, float b1, float b2, float eps, float c1, float c2,
                       __nv_bfloat16* __restrict__ wb) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= WS_NPARAMS) return;
    const float gt = g[t];
    const float mt = b1 * m[t] + (1.f - b1) * gt;
    const float vt = b2 * v[t] + (1.f - b2) * gt * gt;
    m[t] = mt;
    v[t] = vt;
    const float pt = p[t] - lr * (mt / c1) / (sqrtf(vt / c2) + eps);
    p[t] = pt;
    wb[t] = __float2bfloat16(pt);
}

__global__ void k_to_bf16(const float* __restrict__ p, __nv_bfloat16* __restrict__ wb) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < WS_NPARAMS) wb[t] = __float2bfloat16(p[t]);
}

// Rows idx[0..n) of the data set (features, targets, mask) into a batch.
__global__ void k_gather_rows(const __nv_bfloat16* __restrict__ F, const float* __restrict__ T,
                              const float* __restrict__ M, const int32_t* __restrict__ idx, int64_t n,
                              __nv_bfloat16* __restrict__ Fo, float* __restrict__ To, float* __restrict__ Mo) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * WS_IN) return;
    const int64_t r = t / WS_IN, k = t - r * WS_IN;
    const int64_t src = idx[r];
    Fo[t] = F[src * WS_IN + k];
    if (k == 0) {
        To[r] = T[src];
        Mo[r] = M[src];
    }
}

// Outputs in cost units: times the coarse cell (scale > 0) or the box's side.
__global__ void k_scale_out(const float* __restrict__ y, int64_t n, const long long* __restrict__ box,
                            int64_t scale, float* __restrict__ p) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r > n) return;
    const long long ext = scale > 0 ? (long long)scale : max(max(box[2] - box[0], box[3] - box[1]), 1LL);
    p[r] = r < n ? y[r] * (float)ext : 0.f;  // row n: the diagonal node, potential 0
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

static Ctx* owner(Ctx* c) { return c->mlp_owner ? c->mlp_owner : c; }

static MlpW weights_of(Ctx* c) {
    c = owner(c);
    const __nv_bfloat16* wb = (const __nv_bfloat16*)c->ptr[B_MLP_WB];
    const float* p = (const float*)c->ptr[B_MLP_P];
    // biases are read in float32 from the master copy; matrices in bf16
    return MlpW{wb + WS_OFF_W1, p + WS_OFF_B1, wb + WS_OFF_W2, p + WS_OFF_B2, wb + WS_OFF_W3, p + WS_OFF_B3};
}

static size_t backward_smem() { return sizeof(MlpTile) + sizeof(__nv_bfloat16) * WS_H * WS_H; }

// Parameters: allocated and initialised once per context (hidden layers
// He-uniform from a SplitMix64 stream of `seed`, output layer and biases 0).
pd_status mlp_init(Ctx* c, uint64_t seed, bool force, cudaStream_t st) {
    if (c->mlp_ready && !force) return PD_OK;
    float* p = bufT<float>(c, B_MLP_P, WS_NPARAMS);
    float* m = bufT<float>(c, B_MLP_M, WS_NPARAMS);
    float* v = bufT<float>(c, B_MLP_V, WS_NPARAMS);
    __nv_bfloat16* wb = bufT<__nv_bfloat16>(c, B_MLP_WB, WS_NPARAMS);
    if (!p || !m || !v || !wb) return PD_ENOMEM;
    std::vector<float> h(WS_NPARAMS, 0.f);
    uint64_t z = seed;
    auto unif = [&]() {
        z += 0x9E3779B97F4A7C15ull;
        uint64_t x = z;
        x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
        x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
        x ^= x >> 31;
        return (double)(x >> 11) * (1.0 / 9007199254740992.0) * 2.0 - 1.0;
    };
    const double a1 = std::sqrt(6.0 / WS_IN), a2 = std::sqrt(6.0 / WS_H);
    for (int t = 0; t < WS_IN * WS_H; t++) h[WS_OFF_W1 + t] = (float)(a1 * unif());
    for (int t = 0; t < WS_H * WS_H; t++) h[WS_OFF_W2 + t] = (float)(a2 * unif());
    // the output layer starts at 0: the untrained network predicts no
    // correction, so the start is the coarse solve's until training moves it
    PD_TRY(mlp_set(c, h.data(), st));
    c->mlp_steps = 0;
    return PD_OK;
}

pd_status mlp_set(Ctx* c, const float* host, cudaStream_t st) {
    float* p = bufT<float>(c, B_MLP_P, WS_NPARAMS);
    float* m = bufT<float>(c, B_MLP_M, WS_NPARAMS);
    float* v = bufT<float>(c, B_MLP_V, WS_NPARAMS);
    __nv_bfloat16* wb = bufT<__nv_bfloat16>(c, B_MLP_WB, WS_NPARAMS);
    if (!p || !m || !v || !wb) return PD_ENOMEM;
    PD_TRY_CUDA(c, cudaMemcpyAsync(p, host, sizeof(float) * WS_NPARAMS, cudaMemcpyHostToDevice, st));
    PD_TRY_CUDA(c, cudaMemsetAsync(m, 0, sizeof(float) * WS_NPARAMS, st));
    PD_TRY_CUDA(c, cudaMemsetAsync(v, 0, sizeof(float) * WS_NPARAMS, st));
    k_to_bf16<<<grid_for(WS_NPARAMS, 256), 256, 0, st>>>(p, wb); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));
    c->mlp_ready = true;
    c->mlp_steps = 0;
    return PD_OK;
}

pd_status mlp_get(Ctx* c, float* host, cudaStream_t st) {
    if (!c->mlp_ready) return fail(c, PD_EINVAL, "the warm-start network has no parameters yet");
    PD_TRY_CUDA(c, cudaMemcpyAsync(host, c->ptr[B_MLP_P], sizeof(float) * WS_NPARAMS, cudaMemcpyDeviceToHost, st));
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));
    return PD_OK;
}

pd_status mlp_forward(Ctx* c, const __nv_bfloat16* F, int64_t n, float* y, cudaStream_t st) {
    if (!owner(c)->mlp_ready) return fail(c, PD_EINVAL, "the warm-start network has no parameters yet");
    if (n <= 0) return PD_OK;
    const int64_t tiles = (n + WS_TILE - 1) / WS_TILE;
    const int grid = (int)std::min<int64_t>(tiles, 4 * std::max(c->sm_count, 1));
    k_mlp_forward<<<grid, WS_THREADS, 0, st>>>(weights_of(c), F, n, y); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    return PD_OK;
}

// Rows of partial gradients, one per block of k_mlp_backward: fewer if memory is short.
static float* mlp_parts(Ctx* c, int64_t n, int* nb) {
    const int64_t tiles = std::max<int64_t>((n + WS_TILE - 1) / WS_TILE, 1);
    *nb = (int)std::min<int64_t>(tiles, std::min(std::max(c->sm_count, 1), WS_BLOCKS));
    if (beyond_cap(c, (int64_t)*nb * WS_PART * sizeof(float))) *nb = (*nb + 1) / 2;  // leaves room for what follows
    for (;; *nb /= 2) {
        float* part = bufT<float>(c, B_MLP_PART, (int64_t)*nb * WS_PART);
        if (part || *nb == 1) return part;
        c->err.clear();
    }
}

// Loss and gradients of rows [0, n) into g (device, WS_PART floats: the
// WS_NPARAMS gradients, loss sum, mask sum).
pd_status mlp_grad(Ctx* c, const __nv_bfloat16* F, const float* t, const float* mask, int64_t n, float inv_norm,
                   float* g, cudaStream_t st) {
    if (!c->mlp_ready) return fail(c, PD_EINVAL, "the warm-start network has no parameters yet");
    int nb;
    float* part = mlp_parts(c, n, &nb);
    if (!part) return PD_ENOMEM;
    const size_t smem = backward_smem();
    static std::atomic<uint64_t> done{0};
    PD_TRY(smem_limit(c, done, (const void*)k_mlp_backward, smem));
    k_mlp_backward<<<nb, WS_THREADS, smem, st>>>(weights_of(c), F, t, mask, n, inv_norm, part); pd::count_launch();
    k_reduce_parts<<<grid_for(WS_PART, 32), 32 * RP_GROUPS, 0, st>>>(part, nb, g); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    return PD_OK;
}

pd_status mlp_adam(Ctx* c, const float* g, float lr, cudaStream_t st) {
    c->mlp_steps++;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - std::pow(b1, (float)c->mlp_steps), c2 = 1.f - std::pow(b2, (float)c->mlp_steps);
    k_adam<<<grid_for(WS_NPARAMS, 256), 256, 0, st>>>((float*)c->ptr[B_MLP_P], (float*)c->ptr[B_MLP_M],
                                                       (float*)c->ptr[B_MLP_V], g, lr, b1, b2, 1e-8f, c1, c2,
                                                       (__nv_bfloat16*)c->ptr[B_MLP_WB]); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    return PD_OK;
}

pd_status mlp_gather_rows(Ctx* c, const int32_t* idx, int64_t n, __nv_bfloat16** F, float** T, float** M,
                          cudaStream_t st) {
    __nv_bfloat16* Fo = bufT<__nv_bfloat16>(c, B_WS_BF, std::max<int64_t>(n, 1) * WS_IN);
    float* To = bufT<float>(c, B_WS_BT, std::max<int64_t>(n, 1));
    float* Mo = bufT<float>(c, B_WS_BM, std::max<int64_t>(n, 1));
    if (!Fo || !To || !Mo) return PD_ENOMEM;
    if (n > 0) {
        k_gather_rows<<<grid_for(n * WS_IN, 256), 256, 0, st>>>((const __nv_bfloat16*)c->ptr[B_WS_DF],
                                                                 (const float*)c->ptr[B_WS_DT],
                                                                 (const float*)c->ptr[B_WS_DM], idx, n, Fo, To, Mo); pd::count_launch();
        PD_TRY_CUDA(c, cudaGetLastError());
    }
    *F = Fo;
    *T = To;
    *M = Mo;
    return PD_OK;
}

// Master parameters to the snapshot (restore false) or back from it, with
// the bf16 copies and the optimiser state left as they are.
pd_status mlp_snapshot(Ctx* c, bool restore, cudaStream_t st) {
    float* p = (float*)c->ptr[B_MLP_P];
    float* b = bufT<float>(c, B_MLP_BEST, WS_NPARAMS);
    if (!p || !b) return PD_ENOMEM;
    PD_TRY_CUDA(c, cudaMemcpyAsync(restore ? p : b, restore ? b : p, sizeof(float) * WS_NPARAMS,
                                   cudaMemcpyDeviceToDevice, st));
    if (restore) {
        k_to_bf16<<<grid_for(WS_NPARAMS, 256), 256, 0, st>>>(p, (__nv_bfloat16*)c->ptr[B_MLP_WB]); pd::count_launch();
        PD_TRY_CUDA(c, cudaGetLastError());
    }
    return PD_OK;
}

// Mean squared error (over the masked rows) of data-set rows [r0, r1).
pd_status mlp_loss(Ctx* c, int64_t r0, int64_t r1, double* loss, cudaStream_t st) {
    float* g = bufT<float>(c, B_MLP_G, WS_PART);
    if (!g) return PD_ENOMEM;
    const __nv_bfloat16* F = (const __nv_bfloat16*)c->ptr[B_WS_DF];
    const float* T = (const float*)c->ptr[B_WS_DT];
    const float* M = (const float*)c->ptr[B_WS_DM];
    double ls = 0.0, ms = 0.0;
    for (int64_t a = r0; a < r1; a += 2048) {
        const int64_t nb = std::min<int64_t>(2048, r1 - a);
        PD_TRY(mlp_grad(c, F + a * WS_IN, T + a, M + a, nb, 1.f, g, st));
        float lm[2];
        PD_TRY_CUDA(c, cudaMemcpyAsync(lm, g + WS_NPARAMS, sizeof(lm), cudaMemcpyDeviceToHost, st));
        PD_TRY_CUDA(c, cudaStreamSynchronize(st));
        ls += lm[0];
        ms += lm[1];
    }
    *loss = ms > 0.0 ? ls / ms : 0.0;
    return PD_OK;
}

// Features of a prepared transportation instance (rows: its sources then its
// sinks), written to F (device, (nS + nT) x WS_IN bf16); box (device, 4).
pd_status ws_features(Ctx* c, const pd_nodes& nodes, const W1Prep& w, __nv_bfloat16* F, long long* box,
                      cudaStream_t st) {
    const int64_t N = nodes.n_nodes;
    float* grid = bufT<float>(c, B_WS_GRID, WS_GRID * WS_GRID);
    if (!grid) return PD_ENOMEM;
    const long long init[4] = {LLONG_MAX, LLONG_MAX, LLONG_MIN, LLONG_MIN};
    std::memcpy(c->h_small + 24, init, sizeof(init));
    PD_TRY_CUDA(c, cudaMemcpyAsync(box, c->h_small + 24, sizeof(init), cudaMemcpyHostToDevice, st));
    PD_TRY_CUDA(c, cudaMemsetAsync(grid, 0, sizeof(float) * WS_GRID * WS_GRID, st));
    if (N > 0) {
        k_box<<<grid_for(N, 256), 256, 0, st>>>(nodes.X, nodes.Y, N, box); pd::count_launch();
        k_grid<<<grid_for(N, 256), 256, 0, st>>>(nodes.X, nodes.Y, nodes.cntA, nodes.cntB, N, box, grid); pd::count_launch();
    }
    // the coarse solve's envelope gaps and cell, when one ran on this context for this instance
    const int64_t Gc = c->last_coarse_cell;
    const double* gap = Gc > 0 ? (const double*)c->ptr[B_CO_GAP] : nullptr;
    if (w.nS + w.nT > 0)
        k_features<<<grid_for(w.nS + w.nT, 128), 128, 0, st>>>(nodes.X, nodes.Y, nodes.cntA, nodes.cntB, w.S, w.T,
                                                                w.nS, w.nT, box, grid, gap, Gc, F); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));  // h_small + 24 is reused
    return PD_OK;
}

// Predicted potentials (host, nS + nT + 1 floats, cost units, the diagonal
// node last at 0) of a prepared transportation instance.
pd_status ws_predict(Ctx* c, const pd_nodes& nodes, const W1Prep& w, std::vector<float>* p, cudaStream_t st) {
    const int64_t n = w.nS + w.nT;
    __nv_bfloat16* F = bufT<__nv_bfloat16>(c, B_WS_FEAT, std::max<int64_t>(n, 1) * WS_IN);
    float* y = bufT<float>(c, B_WS_Y, n + 1);
    float* ps = bufT<float>(c, B_WS_PS, n + 1);
    long long* box = bufT<long long>(c, B_WS_BOX, 4);
    if (!F || !y || !ps || !box) return PD_ENOMEM;
    PD_TRY(ws_features(c, nodes, w, F, box, st));
    PD_TRY(mlp_forward(c, F, n, y, st));
    k_scale_out<<<grid_for(n + 1, 256), 256, 0, st>>>(y, n, box, c->last_coarse_cell, ps); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    p->resize((size_t)(n + 1));
    PD_TRY_CUDA(c, cudaMemcpyAsync(p->data(), ps, sizeof(float) * (n + 1), cudaMemcpyDeviceToHost, st));
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));
    return PD_OK;
}

// Training rows of one solved pair appended to the context's data set: the
// instance's features and the targets from the solved record r.
pd_status ws_collect(Ctx* c, const pd_nodes& nodes, const W1Prep& w, const NSInst& r,
                     const std::vector<double>* base, cudaStream_t st) {
    const int64_t n = w.nS + w.nT;
    if (n <= 0) return PD_OK;
    const int64_t have = c->ws_rows;
    if (have + n > c->ws_cap) return fail(c, PD_ECAPACITY, "training rows exceed the reserved data set");
    __nv_bfloat16* F = (__nv_bfloat16*)c->ptr[B_WS_DF];
    float* T = (float*)c->ptr[B_WS_DT];
    float* M = (float*)c->ptr[B_WS_DM];
    if (!F || !T || !M) return fail(c, PD_EINVAL, "no training data set reserved");
    long long* box = bufT<long long>(c, B_WS_BOX, 4);
    if (!box) return PD_ENOMEM;
    PD_TRY(ws_features(c, nodes, w, F + have * WS_IN, box, st));
    const int32_t root = (int32_t)(w.nt);  // the simplex root follows the transportation nodes
    int32_t* comp = bufT<int32_t>(c, B_WS_COMP, n);
    int32_t* csize = bufT<int32_t>(c, B_WS_CSIZE, root + 1);
    unsigned long long* sum = bufT<unsigned long long>(c, B_WS_CSUM, 1);
    if (!comp || !csize || !sum) return PD_ENOMEM;
    PD_TRY_CUDA(c, cudaMemsetAsync(csize, 0, sizeof(int32_t) * (root + 1), st));
    PD_TRY_CUDA(c, cudaMemsetAsync(sum, 0, sizeof(unsigned long long), st));
    k_components<<<grid_for(n, 256), 256, 0, st>>>(r.parent, n, root, comp, csize); pd::count_launch();
    std::vector<int32_t> hs((size_t)(root + 1));
    PD_TRY_CUDA(c, cudaMemcpyAsync(hs.data(), csize, sizeof(int32_t) * (root + 1), cudaMemcpyDeviceToHost, st));
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));
    const int32_t anchor = (int32_t)(std::max_element(hs.begin(), hs.end()) - hs.begin());
    k_component_sum<<<grid_for(n, 256), 256, 0, st>>>(r.pi, comp, n, anchor, sum); pd::count_launch();
    unsigned long long hsum = 0;
    PD_TRY_CUDA(c, cudaMemcpyAsync(&hsum, sum, sizeof(hsum), cudaMemcpyDeviceToHost, st));
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));
    const double mean = (double)(int64_t)hsum / (double)std::max(hs[(size_t)anchor], 1);
    // base potentials: the network learns the correction to them
    double* db = nullptr;
    double bmean = 0.0;
    if (base && (int64_t)base->size() >= n) {
        std::vector<int32_t> hc((size_t)n);
        PD_TRY_CUDA(c, cudaMemcpyAsync(hc.data(), comp, sizeof(int32_t) * n, cudaMemcpyDeviceToHost, st));
        PD_TRY_CUDA(c, cudaStreamSynchronize(st));
        int64_t cnt = 0;
        for (int64_t v = 0; v < n; v++)
            if (hc[(size_t)v] == anchor) {
                bmean += (*base)[(size_t)v];
                cnt++;
            }
        bmean = cnt ? bmean / (double)cnt : 0.0;
        db = bufT<double>(c, B_CO_P2, n);
        if (!db) return PD_ENOMEM;
        PD_TRY_CUDA(c, cudaMemcpyAsync(db, base->data(), sizeof(double) * n, cudaMemcpyHostToDevice, st));
    }
    k_targets<<<grid_for(n, 256), 256, 0, st>>>(r.pi, comp, n, anchor, mean, db, bmean, box,
                                                db ? c->last_coarse_cell : 0, T + have, M + have); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));  // the base copy's host memory belongs to the caller
    c->ws_rows = have + n;
    return PD_OK;
}

}  // namespace pd

// ---------------------------------------------------------------------------
// C ABI of the network
// ---------------------------------------------------------------------------

using namespace pd;

static_assert(PD_WS_NPARAMS == WS_NPARAMS && PD_WS_NFEAT == WS_IN, "warm-start layout differs from the header");

extern "C" pd_status pd_ws_get_params(pd_ctx* cx, float* params) {
    Ctx* c = cx;
    if (!c || !params) return PD_EINVAL;
    c->err.clear();
    if (cudaSetDevice(c->device) != cudaSuccess) return cuda_fail(c, cudaGetLastError(), "cudaSetDevice");
    return mlp_get(c, params, 0);
}

extern "C" pd_status pd_ws_set_params(pd_ctx* cx, const float* params) {
    Ctx* c = cx;
    if (!c || !params) return PD_EINVAL;
    c->err.clear();
    if (cudaSetDevice(c->device) != cudaSuccess) return cuda_fail(c, cudaGetLastError(), "cudaSetDevice");
    return mlp_set(c, params, 0);
}

__global__ void k_rows_to_bf16(const float4* __restrict__ x, int64_t n4, uint2* __restrict__ y) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n4) return;
    const float4 v = x[i];
    const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    y[i] = make_uint2(*(const uint32_t*)&a, *(const uint32_t*)&b);
}

// Host feature rows -> bf16 device rows in B_WS_IN: copied as they are and
// rounded on the device (2,048 rows: rounding on the host took longer than the
// copy and the network together), on the host where memory is short.  Called after
// everything else that the call needs has its memory.
static pd_status upload_rows(Ctx* c, const float* feats, int64_t n, __nv_bfloat16** out, cudaStream_t st) {
    static_assert(WS_IN % 4 == 0, "whole 16-byte steps");
    const int64_t m = n * WS_IN;
    __nv_bfloat16* F = bufT<__nv_bfloat16>(c, B_WS_IN, std::max<int64_t>(m, 1));
    if (!F) return PD_ENOMEM;
    *out = F;
    float* raw = beyond_cap(c, sizeof(float) * m) ? nullptr : bufT<float>(c, B_WS_RAW, m);
    if (!raw) {
        c->err.clear();
        const std::unique_ptr<__nv_bfloat16[]> hb(new (std::nothrow) __nv_bfloat16[m]);
        if (!hb) return fail(c, PD_ENOMEM, "no host memory for the features");
        for (int64_t t = 0; t < m; t++) hb[t] = __float2bfloat16(feats[t]);
        PD_TRY_CUDA(c, cudaMemcpyAsync(F, hb.get(), sizeof(__nv_bfloat16) * m, cudaMemcpyHostToDevice, st));
        PD_TRY_CUDA(c, cudaStreamSynchronize(st));  // hb is freed on return
        return PD_OK;
    }
    PD_TRY_CUDA(c, cudaMemcpyAsync(raw, feats, sizeof(float) * m, cudaMemcpyHostToDevice, st));
    k_rows_to_bf16<<<grid_for(m / 4, 256), 256, 0, st>>>((const float4*)raw, m / 4, (uint2*)F); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    return PD_OK;
}

extern "C" pd_status pd_ws_forward(pd_ctx* cx, const float* feats, int64_t n, float* y, void* stream) {
    Ctx* c = cx;
    if (!c || n < 0 || (n > 0 && (!feats || !y))) return PD_EINVAL;
    c->err.clear();
    if (cudaSetDevice(c->device) != cudaSuccess) return cuda_fail(c, cudaGetLastError(), "cudaSetDevice");
    cudaStream_t st = (cudaStream_t)stream;
    if (n == 0) return PD_OK;
    __nv_bfloat16* F;
    float* dy = bufT<float>(c, B_WS_Y, n);
    if (!dy) return PD_ENOMEM;
    PD_TRY(upload_rows(c, feats, n, &F, st));
    PD_TRY(mlp_forward(c, F, n, dy, st));
    PD_TRY_CUDA(c, cudaMemcpyAsync(y, dy, sizeof(float) * n, cudaMemcpyDeviceToHost, st));
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));
    return PD_OK;
}

extern "C" pd_status pd_ws_grad(pd_ctx* cx, const float* feats, const float* target, const float* mask, int64_t n,
                                float* grad, float* loss, void* stream) {
    Ctx* c = cx;
    if (!c || n <= 0 || !feats || !target || !grad) return PD_EINVAL;
    c->err.clear();
    if (cudaSetDevice(c->device) != cudaSuccess) return cuda_fail(c, cudaGetLastError(), "cudaSetDevice");
    cudaStream_t st = (cudaStream_t)stream;
    __nv_bfloat16* F = bufT<__nv_bfloat16>(c, B_WS_IN, n * WS_IN);
    float* dt = bufT<float>(c, B_WS_TIN, n);
    float* dm = bufT<float>(c, B_WS_MIN, n);
    float* g = bufT<float>(c, B_MLP_G, WS_PART);
    int nb;
    if (!F || !dt || !dm || !g || !mlp_parts(c, n, &nb)) return PD_ENOMEM;
    PD_TRY(upload_rows(c, feats, n, &F, st));
    std::vector<float> ones;
    if (!mask) {
        ones.assign((size_t)n, 1.f);
        mask = ones.data();
    }
    PD_TRY_CUDA(c, cudaMemcpyAsync(dt, target, sizeof(float) * n, cudaMemcpyHostToDevice, st));
    PD_TRY_CUDA(c, cudaMemcpyAsync(dm, mask, sizeof(float) * n, cudaMemcpyHostToDevice, st));
    PD_TRY(mlp_grad(c, F, dt, dm, n, 1.f / (float)n, g, st));
    const std::unique_ptr<float[]> hg(new (std::nothrow) float[WS_PART]);
    if (!hg) return fail(c, PD_ENOMEM, "no host memory for the gradient");
    PD_TRY_CUDA(c, cudaMemcpyAsync(hg.get(), g, sizeof(float) * WS_PART, cudaMemcpyDeviceToHost, st));
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));
    std::memcpy(grad, hg.get(), sizeof(float) * WS_NPARAMS);
    if (loss) *loss = hg[WS_NPARAMS] / (float)n;
    return PD_OK;
}

static const char WS_MAGIC[8] = {'P', 'D', 'W', 'S', '0', '0', '0', '1'};

extern "C" pd_status pd_ws_save(pd_ctx* cx, const char* path) {
    Ctx* c = cx;
    if (!c || !path) return PD_EINVAL;
    c->err.clear();
    if (cudaSetDevice(c->device) != cudaSuccess) return cuda_fail(c, cudaGetLastError(), "cudaSetDevice");
    std::vector<float> p(WS_NPARAMS);
    PD_TRY(mlp_get(c, p.data(), 0));
    FILE* f = fopen(path, "wb");
    if (!f) return fail(c, PD_EINVAL, std::string("cannot open ") + path);
    const int64_t n = WS_NPARAMS;
    bool ok = fwrite(WS_MAGIC, 1, 8, f) == 8 && fwrite(&n, sizeof(n), 1, f) == 1 &&
              fwrite(p.data(), sizeof(float), p.size(), f) == p.size();
    ok = (fclose(f) == 0) && ok;
    return ok ? PD_OK : fail(c, PD_EINVAL, std::string("cannot write ") + path);
}

extern "C" pd_status pd_ws_load(pd_ctx* cx, const char* path) {
    Ctx* c = cx;
    if (!c || !path) return PD_EINVAL;
    c->err.clear();
    if (cudaSetDevice(c->device) != cudaSuccess) return cuda_fail(c, cudaGetLastError(), "cudaSetDevice");
    FILE* f = fopen(path, "rb");
    if (!f) return fail(c, PD_EINVAL, std::string("cannot open ") + path);
    char magic[8];
    int64_t n = 0;
    std::vector<float> p(WS_NPARAMS);
    bool ok = fread(magic, 1, 8, f) == 8 && std::memcmp(magic, WS_MAGIC, 8) == 0 && fread(&n, sizeof(n), 1, f) == 1 &&
              n == WS_NPARAMS && fread(p.data(), sizeof(float), p.size(), f) == p.size();
    fclose(f);
    if (!ok) return fail(c, PD_EINVAL, std::string("not a warm-start parameter file: ") + path);
    return mlp_set(c, p.data(), 0);
}
