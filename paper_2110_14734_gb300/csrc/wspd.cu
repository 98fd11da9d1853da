// Hierarchical tree (binary radix tree over Morton order), s-WSPD biarcs
// (Algorithms 6-8, pairs walked depth first), diagonal arcs
// (Algorithm 9) and the CSR network.
#include "internal.h"
#include "netsimplex.cuh"
#include "prims.cuh"

#include <algorithm>

namespace pd {

// ---------------------------------------------------------------------------
// radix tree (Karras 2012) and bottom-up bounding boxes
// ---------------------------------------------------------------------------

PD_D int code_delta(const uint64_t* __restrict__ code, int64_t N, int64_t i, int64_t j) {
    if (j < 0 || j >= N) return -1;
    return __clzll((long long)(code[i] ^ code[j]));
}

// Internal node i covers [lo, hi] with i at one end; its split is the last
// index below the highest bit where the range's codes differ.  Children:
// c >= 0 internal c, c < 0 leaf ~c.
__global__ void k_karras(const uint64_t* __restrict__ code, int64_t N, int32_t* __restrict__ left,
                         int32_t* __restrict__ right, int32_t* __restrict__ par_int, int32_t* __restrict__ par_leaf,
                         int32_t* __restrict__ visit) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N - 1) return;
    visit[i] = 0;
    int d = (code_delta(code, N, i, i + 1) - code_delta(code, N, i, i - 1)) > 0 ? 1 : -1;
    int dmin = code_delta(code, N, i, i - d);
    int64_t lmax = 2;
    while (code_delta(code, N, i, i + lmax * d) > dmin) lmax <<= 1;
    int64_t l = 0;
    for (int64_t t = lmax >> 1; t >= 1; t >>= 1)
        if (code_delta(code, N, i, i + (l + t) * d) > dmin) l += t;
    int64_t j = i + l * d;
    int dnode = code_delta(code, N, i, j);
    int64_t s = 0, t = l;
    do {
        t = (t + 1) >> 1;
        if (code_delta(code, N, i, i + (s + t) * d) > dnode) s += t;
    } while (t > 1);
    int64_t gamma = i + s * d + (d < 0 ? -1 : 0);
    int64_t lo = i < j ? i : j, hi = i < j ? j : i;
    if (lo == gamma) {
        left[i] = ~(int32_t)gamma;
        par_leaf[gamma] = (int32_t)i;
    } else {
        left[i] = (int32_t)gamma;
        par_int[gamma] = (int32_t)i;
    }
    if (hi == gamma + 1) {
        right[i] = ~(int32_t)(gamma + 1);
        par_leaf[gamma + 1] = (int32_t)i;
    } else {
        right[i] = (int32_t)(gamma + 1);
        par_int[gamma + 1] = (int32_t)i;
    }
    if (i == 0) par_int[0] = -1;
}

// Each leaf climbs; the second child to arrive at a node computes the node's
// tight box, leftmost member (min X, then min Y) and leaf count from its two
// children.
__global__ void k_bbox(int64_t N, const int32_t* __restrict__ X, const int32_t* __restrict__ Y,
                       const int32_t* __restrict__ left, const int32_t* __restrict__ right,
                       const int32_t* __restrict__ par_int, const int32_t* __restrict__ par_leaf, int4* bb,
                       int32_t* rep, int32_t* leaves, int32_t* visit) {
    int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= N) return;
    int32_t cur = par_leaf[l];
    for (int depth = 0; cur >= 0 && depth < 130; depth++) {  // a radix tree over 64-bit codes is < 65 deep
        __threadfence();
        if (atomicAdd(&visit[cur], 1) == 0) return;
        int4 b[2];
        int32_t r[2], n[2];
        int32_t ch[2] = {left[cur], right[cur]};
        for (int q = 0; q < 2; q++) {
            int32_t c = ch[q];
            if (c < 0) {
                int32_t p = ~c;
                b[q] = make_int4(X[p], X[p], Y[p], Y[p]);
                r[q] = p;
                n[q] = 1;
            } else {
                n[q] = __ldcg(&leaves[c]);
                b[q] = __ldcg(&bb[c]);
                r[q] = __ldcg(&rep[c]);
            }
        }
        int4 u = make_int4(min(b[0].x, b[1].x), max(b[0].y, b[1].y), min(b[0].z, b[1].z), max(b[0].w, b[1].w));
        int32_t rr = (X[r[1]] < X[r[0]] || (X[r[1]] == X[r[0]] && Y[r[1]] < Y[r[0]])) ? r[1] : r[0];
        __stcg(&bb[cur], u);
        __stcg(&rep[cur], rr);
        __stcg(&leaves[cur], n[0] + n[1]);
        cur = par_int[cur];
    }
}

// ---------------------------------------------------------------------------
// separation test, and membership of one arc in the s-WSPD (certificate)
// ---------------------------------------------------------------------------

struct TNode {
    int32_t mnx, mxx, mny, mxy, rep, l, r;
};

PD_D TNode load_tnode(int32_t ref, const int32_t* __restrict__ X, const int32_t* __restrict__ Y,
                      const int4* __restrict__ bb, const int32_t* __restrict__ rep, const int32_t* __restrict__ left,
                      const int32_t* __restrict__ right) {
    TNode t;
    if (ref < 0) {
        int32_t p = ~ref;
        t.mnx = t.mxx = X[p];
        t.mny = t.mxy = Y[p];
        t.rep = p;
        t.l = t.r = 0;
    } else {
        int4 b = bb[ref];
        t.mnx = b.x;
        t.mxx = b.y;
        t.mny = b.z;
        t.mxy = b.w;
        t.rep = rep[ref];
        t.l = left[ref];
        t.r = right[ref];
    }
    return t;
}

// s-well-separated with circumscribed circles of the tight boxes and the
// larger radius for both: in doubled coordinates |C_u - C_v| >= (s+2) D,
// D the larger box diagonal; exact in 128-bit integers.
PD_D bool well_separated(const TNode& a, const TNode& b, int64_t s) {
    int64_t dx = ((int64_t)a.mnx + a.mxx) - ((int64_t)b.mnx + b.mxx);
    int64_t dy = ((int64_t)a.mny + a.mxy) - ((int64_t)b.mny + b.mxy);
    uint64_t ax = (uint64_t)(dx < 0 ? -dx : dx), ay = (uint64_t)(dy < 0 ? -dy : dy);
    unsigned __int128 D2 = (unsigned __int128)ax * ax + (unsigned __int128)ay * ay;
    uint64_t awx = (uint64_t)((int64_t)a.mxx - a.mnx), awy = (uint64_t)((int64_t)a.mxy - a.mny);
    uint64_t bwx = (uint64_t)((int64_t)b.mxx - b.mnx), bwy = (uint64_t)((int64_t)b.mxy - b.mny);
    uint64_t ra = awx * awx + awy * awy, rb = bwx * bwx + bwy * bwy;
    uint64_t R2 = ra > rb ? ra : rb;
    uint64_t k = (uint64_t)(s + 2) * (uint64_t)(s + 2);
    return D2 >= (unsigned __int128)k * R2;
}

PD_D int64_t max_side(const TNode& a) {
    int64_t wx = (int64_t)a.mxx - a.mnx, wy = (int64_t)a.mxy - a.mny;
    return wx > wy ? wx : wy;
}

// Is (a, b), a < b two leaves (Morton ranks), one of the biarcs of the
// s-WSPD?  The pairs of the decomposition partition all leaf pairs, so (a, b)
// lies in exactly one of them: start at the pair of children of the lowest
// common ancestor and follow the same split rule as k_ws_walk (larger box
// side, ties split the second node), always into the child holding a
// (resp. b), until the pair is well separated.  (a, b) is an arc iff a and b
// are the representatives of that pair.  A walk longer than any tree path
// answers false, which the certificate treats as a failure (never as proof).
PD_D bool ws_arc_exists(int32_t a, int32_t b, int64_t N, const int32_t* __restrict__ X,
                        const int32_t* __restrict__ Y, const int4* __restrict__ bb, const int32_t* __restrict__ rep,
                        const int32_t* __restrict__ left, const int32_t* __restrict__ right, int64_t s) {
    if (N < 2 || a >= b || a < 0 || b >= N) return false;
    int32_t z = 0;  // the root covers [0, N - 1]
    int32_t sp = 0;
    int depth = 0;
    for (; depth < 130; depth++) {
        const int32_t lc = left[z], rc = right[z];
        sp = lc >= 0 ? lc : ~lc;  // left child covers [lo, sp], right child [sp + 1, hi]
        if (b <= sp) {
            if (lc < 0) return false;
            z = lc;
        } else if (a > sp) {
            if (rc < 0) return false;
            z = rc;
        } else {
            break;
        }
    }
    if (depth >= 130) return false;
    int32_t P = left[z], Q = right[z];
    for (int it = 0; it < 260; it++) {
        const TNode tp = load_tnode(P, X, Y, bb, rep, left, right);
        const TNode tq = load_tnode(Q, X, Y, bb, rep, left, right);
        if (well_separated(tp, tq, s)) return tp.rep == a && tq.rep == b;
        if (max_side(tp) > max_side(tq)) {
            if (P < 0) return false;
            const int32_t c = tp.l >= 0 ? tp.l : ~tp.l;
            P = a <= c ? tp.l : tp.r;
        } else {
            if (Q < 0) return false;
            const int32_t c = tq.l >= 0 ? tq.l : ~tq.l;
            Q = b <= c ? tq.l : tq.r;
        }
    }
    return false;
}

// Certificate of a transportation optimum against the sparse network: every
// source -> sink pair that carries flow on its direct route must be a WSPD
// biarc (found by ws_arc_exists); routes through the diagonal use arcs that
// always exist.  out[0] = pairs missing, out[1] = total flow over the arcs of
// the sparse network that the flow uses (rounding slack).
__global__ void k_certify_tree(const NSInst* __restrict__ I, const int32_t* __restrict__ S,
                               const int32_t* __restrict__ T, int64_t nS, int64_t ld, WsTree tr, int64_t s,
                               DiagCost dc, unsigned long long* __restrict__ out) {
    int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= I->n) return;
    int64_t a = I->pred[v], f = I->flow[v];
    if (a >= I->m || f <= 0) return;
    int64_t mst = nS * ld;
    if (a >= mst) {  // arc of the diagonal node: one arc of the sparse network
        atomicAdd(&out[1], (unsigned long long)f);
        return;
    }
    int64_t i = a / ld, j = a - i * ld;
    int32_t u = S[i], w = T[j];
    int64_t d = cost_l2(tr.X[u], tr.Y[u], tr.X[w], tr.Y[w]);
    int64_t g = cost_make(tr.X[u], tr.Y[u], dc) + cost_make(tr.X[w], tr.Y[w], dc);
    if (g <= d) {  // through the diagonal node: u -> diag -> w, both arcs exist
        atomicAdd(&out[1], (unsigned long long)(2 * f));
        return;
    }
    const int32_t lo = u < w ? u : w, hi = u < w ? w : u;
    if (!ws_arc_exists(lo, hi, tr.N, tr.X, tr.Y, tr.bb, tr.rep, tr.left, tr.right, s)) atomicAdd(&out[0], 1ull);
    atomicAdd(&out[1], (unsigned long long)f);
}

__global__ void k_certify_batch(const CertJob* __restrict__ jobs, unsigned long long* __restrict__ out) {
    const CertJob J = jobs[blockIdx.y];
    const NSInst* I = J.inst;
    unsigned long long* o = out + 2 * (int64_t)blockIdx.y;
    const int64_t mst = J.nS * J.ld;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < I->n; v += (int64_t)gridDim.x * blockDim.x) {
        const int64_t a = I->pred[v], f = I->flow[v];
        if (a >= I->m || f <= 0) continue;
        if (a >= mst) {
            atomicAdd(&o[1], (unsigned long long)f);
            continue;
        }
        const int64_t i = a / J.ld, j = a - i * J.ld;
        const int32_t u = J.S[i], w = J.T[j];
        const WsTree& tr = J.tree;
        const int64_t d = cost_l2(tr.X[u], tr.Y[u], tr.X[w], tr.Y[w]);
        const int64_t g = cost_make(tr.X[u], tr.Y[u], J.dc) + cost_make(tr.X[w], tr.Y[w], J.dc);
        if (g <= d) {
            atomicAdd(&o[1], (unsigned long long)(2 * f));
            continue;
        }
        const int32_t lo = u < w ? u : w, hi = u < w ? w : u;
        if (!ws_arc_exists(lo, hi, tr.N, tr.X, tr.Y, tr.bb, tr.rep, tr.left, tr.right, J.s)) atomicAdd(&o[0], 1ull);
        atomicAdd(&o[1], (unsigned long long)f);
    }
}

// ---------------------------------------------------------------------------
// enumeration: warps walk the pair tree depth first
// ---------------------------------------------------------------------------
//
// The recursion tests as many pairs as the decomposition has, twice over (at
// 2 M nodes and s = 167: 21 G separated pairs and as many split ones), and a pair
// needs only its two nodes.  So what bounds it is the gather of node records
// and the instructions of a test, as long as what waits to be visited never
// leaves the SM: every warp keeps it in a stack in shared memory and visits the
// 32 topmost pairs at a time.  These descend from one pair a few levels up, so
// the 32 lanes touch about a dozen different nodes.
//
// The records.  An internal node's 32 bytes: doubled centre, separation
// threshold (s + 2)^2 diagonal^2, larger side, children, and the representative
// (when pairs are stored) or the leaves below it (when they are counted).  A
// leaf needs its coordinates only, and a pair of leaves nothing: it is always
// separated, and is counted where it would be pushed.
//
// Lattices.  Nodes snapped to a grid have no small boxes.  Below a pair of
// nodes whose farthest points are closer than the smallest box's threshold, only
// pairs of leaves can be separated: as many as the product of the leaf counts.
// Where that reaches over more than a sixteenth of the nodes' extent, counting
// stops there (8,205 lattice nodes, s = 327: 0.58 -> 0.18 ms; mixture points take no
// notice of the test).
//
// Balance.  Initial pairs (one per internal node) differ by many orders of
// magnitude in the pairs below them, so a warp that has walked `budget` steps
// on its chunk hands what is left on its stack to the next launch, where other
// warps take it up.  Once the room for these is half full, only every eighth
// time: used up early, it would leave the largest stacks to single warps
// (mixture points, counts: 50,000 + 50,000 at eps 0.01 167 -> 17 ms, 100,000 + 100,000
// at 0.02 773 -> 30, 250,000 + 250,000 at 0.05 706 -> 51).
//
// Measured (pd_w1_sparsify_count's WSPD stage, mixture points, s = 167): 1,000,000
// + 1,000,000 points 493 -> 161 ms, 100,000 + 100,000 23 -> 7.2 ms, against
// level-by-level frontiers in global memory (689 GB of DRAM traffic a call, and
// 128-bit products per test).  Entries of two pairs, a node and its partner's
// children, were slower (269 ms).

struct __align__(32) WsRec {
    int32_t cx, cy;  // doubled centre
    uint64_t thr;    // least doubled squared distance that separates (saturated)
    uint32_t side;   // larger box side
    int32_t l, r;    // children
    int32_t last;    // representative, or leaves (see above)
};

// Also the leaves' doubled coordinates, and over all internal nodes ext[0] = ~
// the least threshold and ext[1] = the largest side (maxima; both start at 0).
// last: the leaf counts or the representatives.
__global__ void k_ws_records(int64_t M, const int4* __restrict__ bb, const int32_t* __restrict__ last,
                             const int32_t* __restrict__ left, const int32_t* __restrict__ right,
                             const int32_t* __restrict__ X, const int32_t* __restrict__ Y, int64_t s,
                             WsRec* __restrict__ rec, int2* __restrict__ leaf, int2* __restrict__ F,
                             unsigned long long* __restrict__ ext) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long inv = 0, side = 0;
    if (i <= M) leaf[i] = make_int2(2 * X[i], 2 * Y[i]);  // |coordinate| < 2^30: no overflow
    if (i < M) {
        const int4 b = bb[i];
        const uint64_t wx = (uint64_t)((int64_t)b.y - b.x), wy = (uint64_t)((int64_t)b.w - b.z);
        const uint64_t k = (uint64_t)(s + 2) * (uint64_t)(s + 2);
        const unsigned __int128 t = (unsigned __int128)k * (wx * wx + wy * wy);
        WsRec q;
        q.cx = b.x + b.y;
        q.cy = b.z + b.w;
        q.thr = (t >> 64) != 0 ? ~0ull : (uint64_t)t;
        q.side = (uint32_t)(wx > wy ? wx : wy);
        q.l = left[i];
        q.r = right[i];
        q.last = last[i];
        rec[i] = q;
        F[i] = make_int2(q.l, q.r);  // the first pairs: every internal node's children
        inv = ~q.thr;
        side = q.side;
    }
    __shared__ unsigned long long part[2][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int pass = 0; pass < 2; pass++) {
        for (int o = 16; o > 0; o >>= 1) {
            inv = max(inv, __shfl_xor_sync(0xffffffffu, inv, o));
            side = max(side, __shfl_xor_sync(0xffffffffu, side, o));
        }
        if (pass == 1) break;
        if (lane == 0) {
            part[0][wid] = inv;
            part[1][wid] = side;
        }
        __syncthreads();
        if (wid > 0) return;
        inv = lane < (int)(blockDim.x >> 5) ? part[0][lane] : 0ull;
        side = lane < (int)(blockDim.x >> 5) ? part[1][lane] : 0ull;
    }
    if (lane == 0) {
        atomicMax(&ext[0], inv);
        atomicMax(&ext[1], side);
    }
}

PD_D WsRec ws_load(int32_t ref, const WsRec* __restrict__ rec, const int2* __restrict__ leaf, bool counts) {
    WsRec q;
    if (ref < 0) {
        const int2 p = __ldg(leaf + ~ref);
        q.cx = p.x;
        q.cy = p.y;
        q.thr = 0;
        q.side = 0;
        q.l = q.r = 0;
        q.last = counts ? 1 : ~ref;
    } else {
        uint32_t w0, w1, w2, w3, w4, w5, w6, w7;
        asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
            : "=r"(w0), "=r"(w1), "=r"(w2), "=r"(w3), "=r"(w4), "=r"(w5), "=r"(w6), "=r"(w7)
            : "l"(rec + ref));
        q.cx = (int32_t)w0;
        q.cy = (int32_t)w1;
        q.thr = (uint64_t)w3 << 32 | w2;
        q.side = w4;
        q.l = (int32_t)w5;
        q.r = (int32_t)w6;
        q.last = (int32_t)w7;
    }
    return q;
}

// well_separated on records: doubled squared distance >= both thresholds.  The
// distance's 64 bits overflow only for coordinates near the limit; then the
// 128-bit test decides.
PD_D bool ws_far(const WsRec& a, const WsRec& b, int32_t ra, int32_t rb, int64_t s, const WsTree& tr) {
    const uint32_t dx = a.cx > b.cx ? (uint32_t)a.cx - (uint32_t)b.cx : (uint32_t)b.cx - (uint32_t)a.cx;
    const uint32_t dy = a.cy > b.cy ? (uint32_t)a.cy - (uint32_t)b.cy : (uint32_t)b.cy - (uint32_t)a.cy;
    const uint64_t x2 = (uint64_t)dx * dx, d2 = x2 + (uint64_t)dy * dy;
    if (d2 < x2)
        return well_separated(load_tnode(ra, tr.X, tr.Y, tr.bb, tr.rep, tr.left, tr.right),
                              load_tnode(rb, tr.X, tr.Y, tr.bb, tr.rep, tr.left, tr.right), s);
    return d2 >= a.thr && d2 >= b.thr;
}

constexpr int WS_WARPS = 8;      // per block
constexpr int WS_OUT = 256;      // separated pairs a warp gathers before it stores them
constexpr int WS_STACK = 736;    // pairs a warp's stack holds
constexpr int WS_MARGIN = 200;   // above WS_STACK - WS_MARGIN pairs it visits one at a time: a path is
                                 // at most 2 * 65 splits long (78 + 78 on the split tree), each net +1

// lv[0] += separated pairs, lv[1] = pairs offered to the next launch (the first
// cap of them are in Fn), lv[2] = initial pairs taken; ext as in k_ws_records.
// STORE: both arcs of every separated pair to arcs (room for `room` pairs), at
// slots from lv[0], which counts all pairs.  counted: the records hold leaf counts.
template <bool STORE>
__global__ void __launch_bounds__(32 * WS_WARPS) k_ws_walk(const int2* __restrict__ F, int64_t nf, int chunk,
                                                           const WsRec* __restrict__ rec,
                                                           const int2* __restrict__ leaf, WsTree tr, int64_t s,
                                                           int64_t budget, int2* __restrict__ Fn,
                                                           unsigned long long cap, int hb, uint64_t* __restrict__ arcs,
                                                           unsigned long long room,
                                                           unsigned long long* __restrict__ lv,
                                                           const unsigned long long* __restrict__ ext, int counted) {
    __shared__ int2 stack_[WS_WARPS][WS_STACK];
    extern __shared__ int2 out_[];  // STORE: separated pairs on their way out, WS_OUT a warp
    int2* const ow = out_ + (threadIdx.x >> 5) * WS_OUT;
    int on_out = 0;
    const int lane = threadIdx.x & 31;
    int2* const st = stack_[threadIdx.x >> 5];
    const unsigned below = (1u << lane) - 1u;
    unsigned long long count = 0;
    // lattices (sides below 2^28: nothing overflows)
    const uint64_t least = ~ext[0], widest = ext[1];
    const bool lattice = !STORE && counted && widest < (1u << 28) && least >= widest * widest / 64;
    // the buffered pairs' arcs, at slots taken with one atomic; past `room` they are only counted
    auto flush = [&]() {
        __syncwarp();
        unsigned long long at = 0;
        if (lane == 0) at = atomicAdd(&lv[0], (unsigned long long)on_out);
        at = __shfl_sync(0xffffffffu, at, 0);
        for (int q = lane; q < on_out && at + q < room; q += 32) {
            const int2 a = ow[q];
            ulonglong2 w;
            w.x = (uint64_t)a.x << hb | (uint64_t)a.y;
            w.y = (uint64_t)a.y << hb | (uint64_t)a.x;
            *(ulonglong2*)(arcs + 2 * (at + q)) = w;
        }
        on_out = 0;
        __syncwarp();
    };
    // up to three separated pairs of a lane, by their representatives
    auto emit = [&](bool on0, int2 a0, bool on1, int2 a1, bool on2, int2 a2) {
        if constexpr (STORE) {
            const unsigned m0 = __ballot_sync(0xffffffffu, on0), m1 = __ballot_sync(0xffffffffu, on1),
                           m2 = __ballot_sync(0xffffffffu, on2);
            const int c0 = __popc(m0), c1 = __popc(m1), c2 = __popc(m2);
            if (on0) ow[on_out + __popc(m0 & below)] = a0;
            if (on1) ow[on_out + c0 + __popc(m1 & below)] = a1;
            if (on2) ow[on_out + c0 + c1 + __popc(m2 & below)] = a2;
            on_out += c0 + c1 + c2;
            if (on_out > WS_OUT - 96) flush();
        } else {
            count += (unsigned)on0 + (unsigned)on1 + (unsigned)on2;
        }
    };
    int h = 0;  // height of the stack
    int64_t steps = 0;
    int tight = 0;  // budgets used up while the room was more than half full: every eighth hands on
    for (;;) {
        int2 p = make_int2(0, 0);
        bool on;
        if (h == 0) {
            unsigned long long at = 0;
            if (lane == 0) at = atomicAdd(&lv[2], (unsigned long long)chunk);
            at = __shfl_sync(0xffffffffu, at, 0);
            if (at >= (unsigned long long)nf) break;
            on = lane < chunk && at + lane < (unsigned long long)nf;
            if (on) p = F[at + lane];
            const bool leaves = on && p.x < 0 && p.y < 0;
            emit(leaves, make_int2(~p.x, ~p.y), false, p, false, p);
            on = on && !leaves;
            steps = 0;
        } else {
            const int take = h > WS_STACK - WS_MARGIN ? 1 : min(h, 32);
            h -= take;
            on = lane < take;
            if (on) p = st[h + lane];
            __syncwarp();
        }
        int2 c0 = make_int2(-1, -1), c1 = make_int2(-1, -1);
        bool far = false;
        WsRec u{}, v{};
        if (on) {
            u = ws_load(p.x, rec, leaf, !STORE);
            v = ws_load(p.y, rec, leaf, !STORE);
            far = ws_far(u, v, p.x, p.y, s, tr);
            if (!far) {
                // split the node with the larger box side, ties split the second
                const bool su = u.side > v.side;
                c0 = su ? make_int2(u.l, p.y) : make_int2(p.x, v.l);
                c1 = su ? make_int2(u.r, p.y) : make_int2(p.x, v.r);
            }
        }
        bool open = on && !far;
        if constexpr (!STORE) {
            if (lattice && open) {  // only pairs of leaves separated below this one?
                const uint64_t w = (uint64_t)u.side + v.side;
                const uint64_t x = (uint64_t)abs(u.cx - v.cx) + w, y = (uint64_t)abs(u.cy - v.cy) + w;
                if (x * x + y * y < least) {
                    open = false;
                    count += (unsigned long long)u.last * (unsigned long long)v.last;
                }
            }
        }
        const bool l0 = open && (c0.x & c0.y) < 0, l1 = open && (c1.x & c1.y) < 0;  // two leaves
        emit(far, make_int2(u.last, v.last), l0, make_int2(~c0.x, ~c0.y), l1, make_int2(~c1.x, ~c1.y));
        const bool p0 = open && !l0, p1 = open && !l1;
        const unsigned m0 = __ballot_sync(0xffffffffu, p0), m1 = __ballot_sync(0xffffffffu, p1);
        const int at = h + __popc(m0 & below) + __popc(m1 & below);
        if (p0) st[at] = c0;
        if (p1) st[at + p0] = c1;
        h += __popc(m0) + __popc(m1);
        __syncwarp();
        if (++steps > budget && h > 0) {
            // to the next launch, as far as it still has room
            unsigned long long at2 = cap;
            if (lane == 0) {
                const unsigned long long used = *(volatile unsigned long long*)&lv[1];
                if (used < cap && (used < cap / 2 || (++tight & 7) == 0)) at2 = atomicAdd(&lv[1], (unsigned long long)h);
            }
            at2 = __shfl_sync(0xffffffffu, at2, 0);
            const int give = at2 >= cap ? 0 : (int)min((unsigned long long)h, cap - at2);
            for (int q = lane; q < give; q += 32) Fn[at2 + q] = st[h - give + q];
            h -= give;
            steps = 0;
            __syncwarp();
        }
    }
    if constexpr (STORE) {
        if (on_out > 0) flush();
    } else {
        for (int o = 16; o > 0; o >>= 1) count += __shfl_xor_sync(0xffffffffu, count, o);
        if (lane == 0 && count) atomicAdd(&lv[0], count);
    }
}

// Diagonal arcs: u -> ā if u holds A mass, b̄ -> u if u holds B mass, and
// b̄ -> ā; absent arcs become the all-ones key, which sorts last.
__global__ void k_diag_arcs(int64_t N, const int64_t* __restrict__ cntA, const int64_t* __restrict__ cntB, int hb,
                            uint64_t sent, uint64_t* __restrict__ arcs, unsigned long long* __restrict__ counts) {
    int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (u > N) return;
    if (u == N) {
        arcs[2 * N] = ((uint64_t)(N + 1) << hb) | (uint64_t)N;
        return;
    }
    bool a = cntA[u] > 0, b = cntB[u] > 0;
    arcs[2 * u] = a ? (((uint64_t)u << hb) | (uint64_t)N) : sent;
    arcs[2 * u + 1] = b ? (((uint64_t)(N + 1) << hb) | (uint64_t)u) : sent;
    unsigned ma = __ballot_sync(__activemask(), a), mb = __ballot_sync(__activemask(), b);
    if ((threadIdx.x & 31) == (__ffs(__activemask()) - 1)) {
        atomicAdd(&counts[0], (unsigned long long)__popc(ma));
        atomicAdd(&counts[1], (unsigned long long)__popc(mb));
    }
}

// row_ptr from arc keys sorted by (tail, head).
__global__ void k_row_ptr(const uint64_t* __restrict__ key, int64_t m, int hb, int64_t nrows,
                          int64_t* __restrict__ row_ptr) {
    int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= m) return;
    int64_t t = (int64_t)(key[a] >> hb);
    int64_t tp = a == 0 ? -1 : (int64_t)(key[a - 1] >> hb);
    for (int64_t r = tp + 1; r <= t; r++) row_ptr[r] = a;
    if (a == m - 1)
        for (int64_t r = t + 1; r <= nrows; r++) row_ptr[r] = m;
}

__global__ void k_head_cost(const uint64_t* __restrict__ key, int64_t m, int hb, int64_t N,
                            const int32_t* __restrict__ X, const int32_t* __restrict__ Y, int32_t* __restrict__ head,
                            int64_t* __restrict__ cost, DiagCost dc) {
    int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= m) return;
    uint64_t k = key[a];
    int64_t t = (int64_t)(k >> hb), h = (int64_t)(k & ((1ull << hb) - 1));
    head[a] = (int32_t)h;
    int64_t c = 0;
    if (t < N && h < N)
        c = cost_l2(X[t], Y[t], X[h], Y[h]);
    else if (t < N && h == N)
        c = cost_make(X[t], Y[t], dc);
    else if (t == N + 1 && h < N)
        c = cost_make(X[h], Y[h], dc);
    cost[a] = c;
}

__global__ void k_supply(int64_t N, const int64_t* __restrict__ cntA, const int64_t* __restrict__ cntB, int64_t FA,
                         int64_t FB, int64_t* __restrict__ sup) {
    int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (u < N) sup[u] = cntA[u] - cntB[u];
    if (u == N) sup[N] = -FA;
    if (u == N + 1) sup[N + 1] = FB;
}

// Nodes that hold A mass, B mass, and both masses (out[0 .. 3]), in one pass.
__global__ void k_diag_counts(int64_t N, const int64_t* __restrict__ cntA, const int64_t* __restrict__ cntB,
                              unsigned long long* __restrict__ out) {
    const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned long long a = u < N ? (unsigned long long)cntA[u] : 0ull, b = u < N ? (unsigned long long)cntB[u] : 0ull;
    const unsigned ma = __ballot_sync(0xffffffffu, a > 0), mb = __ballot_sync(0xffffffffu, b > 0);
    const unsigned long long sa = warp_sum(a), sb = warp_sum(b);
    if ((threadIdx.x & 31) == 0) {
        if (ma) {
            atomicAdd(&out[0], (unsigned long long)__popc(ma));
            atomicAdd(&out[2], sa);
        }
        if (mb) {
            atomicAdd(&out[1], (unsigned long long)__popc(mb));
            atomicAdd(&out[3], sb);
        }
    }
}

__global__ void k_mass(int64_t N, const int64_t* __restrict__ cntA, const int64_t* __restrict__ cntB,
                       unsigned long long* __restrict__ out) {
    int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long a = 0, b = 0;
    if (u < N) {
        a = (unsigned long long)cntA[u];
        b = (unsigned long long)cntB[u];
    }
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (a) atomicAdd(&out[2], a);
        if (b) atomicAdd(&out[3], b);
    }
}

__global__ void k_check_nodes(const uint64_t* __restrict__ code, const int32_t* __restrict__ X,
                              const int32_t* __restrict__ Y, const int64_t* __restrict__ cntA,
                              const int64_t* __restrict__ cntB, int64_t N, unsigned long long* __restrict__ bad) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int32_t lim = 1 << 30;
    bool b = (i + 1 < N && !(code[i] < code[i + 1])) || X[i] <= -lim || X[i] >= lim || Y[i] <= -lim || Y[i] >= lim ||
             cntA[i] < 0 || cntB[i] < 0;
    if (b) atomicAdd(bad, 1ull);
}

pd_status validate_nodes(Ctx* c, const pd_nodes& nodes, cudaStream_t st) {
    int64_t N = nodes.n_nodes;
    if (N <= 0) return PD_OK;
    unsigned long long* sm = bufT<unsigned long long>(c, B_SMALL, 64);
    if (!sm) return PD_ENOMEM;
    PD_TRY_CUDA(c, cudaMemsetAsync(sm, 0, sizeof(unsigned long long), st));
    k_check_nodes<<<grid_for(N, 256), 256, 0, st>>>(nodes.morton, nodes.X, nodes.Y, nodes.cntA, nodes.cntB, N, sm); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    PD_TRY_CUDA(c, cudaMemcpyAsync(c->h_small, sm, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));
    if (c->h_small[0])
        return fail(c, PD_EINVAL,
                    "nodes need strictly increasing Morton codes, |X|,|Y| < 2^30 and non-negative multiplicities");
    return PD_OK;
}

__global__ void k_merge_diag(const int64_t* __restrict__ rp, const int64_t* __restrict__ sup, int64_t N, int64_t m,
                             int64_t* __restrict__ mrp, int64_t* __restrict__ msup) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i <= N) mrp[i] = rp[i];
    if (i == N + 1) mrp[N + 1] = m - 1;
    if (i < N) msup[i] = sup[i];
    if (i == N) msup[N] = sup[N] + sup[N + 1];
}

// Network of nodes 0..N-1 plus one diagonal node N: rows 0..N-1 unchanged
// (their arcs to ā now point to N), row N = b̄'s row without its last arc
// b̄ -> ā (ā = N is the largest head of b̄'s row and ā's own row is empty).
pd_status merge_diagonal(Ctx* c, const pd_network& net, int64_t N, pd_network* out, cudaStream_t st) {
    int64_t* mrp = bufT<int64_t>(c, B_M_ROWPTR, N + 2);
    int64_t* msup = bufT<int64_t>(c, B_M_SUPPLY, N + 1);
    if (!mrp || !msup) return PD_ENOMEM;
    k_merge_diag<<<grid_for(N + 2, 256), 256, 0, st>>>(net.row_ptr, net.supply, N, net.n_arcs, mrp, msup); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    out->n_nodes = N + 1;
    out->n_arcs = net.n_arcs - 1;
    out->row_ptr = mrp;
    out->head = net.head;
    out->cost = net.cost;
    out->supply = msup;
    return PD_OK;
}

// The walk's device words: 0 .. 2 lv, 3 .. 4 ext, 5 .. 8 k_diag_counts (all cleared before k_ws_records).
constexpr int WS_WORDS = 9;
static unsigned long long* ws_words(Ctx* c) { return bufT<unsigned long long>(c, B_SMALL, 64) + 12; }

// All launches of the walk over the tree's pairs (see k_ws_walk): *pairs =
// separated pairs; arcs (may be null): where their arcs go.  The walk's words end
// up in h_small.
static pd_status ws_walk(Ctx* c, const WsTree& tr, const WsRec* rec, const int2* leaf, int64_t s, int hb, bool counted,
                         uint64_t* arcs, int64_t room, int64_t* pairs, cudaStream_t st) {
    unsigned long long* lv = ws_words(c);
    const int blocks = 4 * std::max(c->sm_count, 1);  // the stacks of four blocks fit an SM
    const int64_t warps = (int64_t)blocks * WS_WARPS;
    // room for handed-on pairs: the more, the better the balance; less will do
    constexpr int64_t least = 256;
    int64_t cap = std::min<int64_t>(int64_t(1) << 27, std::max<int64_t>(int64_t(1) << 16, 64 * (tr.N - 1)));  // even
    while (cap > least && beyond_cap(c, 2 * sizeof(int2) * cap)) cap = cap / 8 * 2;
    int2* out[2];
    static std::atomic<uint64_t> done{0};
    if (arcs) PD_TRY(smem_limit(c, done, (const void*)k_ws_walk<true>, sizeof(int2) * WS_WARPS * WS_OUT));
    for (;; cap = cap / 8 * 2) {
        out[0] = bufT<int2>(c, B_F1, cap);
        out[1] = out[0] ? bufT<int2>(c, B_WSOFF, cap) : nullptr;
        if (out[0] && out[1]) break;
        if (cap <= least) return PD_ENOMEM;
        c->err.clear();
    }
    const int2* F = (const int2*)c->ptr[B_F0];
    int64_t nf = tr.N - 1, total = 0;
    // short first launches spread the few large pairs, later ones finish
    // Steps a warp spends on a chunk.  Many chunks: longer, so that the handed-on
    // pairs fit (2 M nodes: 165 ms with 512, 166 with 128, the room used up and
    // 3,700 ms with 48).  Few: shorter (8,271 lattice nodes: 0.55 ms with 48, 0.66
    // with 128, 0.90 with 512).
    const int64_t budget = tr.N > (int64_t(1) << 20) ? 512 : 64;
    for (int64_t round = 0; nf > 0; round++) {
        const int chunk = (int)std::min<int64_t>(32, std::max<int64_t>(1, nf / warps));
        if (round > 0)
            PD_TRY_CUDA(c, cudaMemsetAsync(lv + (arcs ? 1 : 0), 0, (arcs ? 2 : 3) * sizeof(unsigned long long), st));
        const unsigned grid = (unsigned)std::min<int64_t>(blocks, ((nf + chunk - 1) / chunk + WS_WARPS - 1) / WS_WARPS);
        if (arcs) {
            k_ws_walk<true><<<grid, 32 * WS_WARPS, sizeof(int2) * WS_WARPS * WS_OUT, st>>>(
                F, nf, chunk, rec, leaf, tr, s, budget, out[round & 1], (unsigned long long)cap, hb, arcs,
                (unsigned long long)room, lv, lv + 3, 0); pd::count_launch();
        } else {
            k_ws_walk<false><<<grid, 32 * WS_WARPS, 0, st>>>(F, nf, chunk, rec, leaf, tr, s, budget, out[round & 1],
                                                             (unsigned long long)cap, hb, nullptr, 0, lv, lv + 3,
                                                             counted ? 1 : 0); pd::count_launch();
        }
        PD_TRY_CUDA(c, cudaGetLastError());
        PD_TRY_CUDA(c, cudaMemcpyAsync(c->h_small, lv, WS_WORDS * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
        PD_TRY_CUDA(c, cudaStreamSynchronize(st));
        total = arcs ? c->h_small[0] : total + c->h_small[0];  // with arcs, lv[0] runs on as their slot counter
        nf = std::min<int64_t>(c->h_small[1], cap);
        F = out[round & 1];
    }
    *pairs = total;
    return PD_OK;
}

pd_status stage_network(Ctx* c, const pd_nodes& nodes, int64_t s, pd_network* out, float* ms_tree,
                        float* ms_wspd, float* ms_csr, cudaStream_t st, bool count_only, WsTree* tree,
                        const WsTree* given, DiagCost dc) {
    int64_t N = nodes.n_nodes;
    if (N >= (int64_t(1) << 31) - 4) return fail(c, PD_ECAPACITY, "more than 2^31 - 4 condensed nodes");
    if (s < 1) return fail(c, PD_EINVAL, "WSPD parameter s must be >= 1");
    cudaEvent_t* ev;
    PD_TRY(ctx_events(c, EV_NETWORK, 4, &ev));
    PD_TRY_CUDA(c, cudaEventRecord(ev[0], st));
    int64_t M = N > 1 ? N - 1 : 1;
    unsigned long long* cnts = bufT<unsigned long long>(c, B_SMALL, 64);
    if (!cnts) return PD_ENOMEM;
    const int32_t *left, *right, *rep, *leaves = nullptr;  // (a given tree comes without its leaf counts)
    const int4* bb;
    if (given) {
        if (given->N != N || given->X != nodes.X || given->Y != nodes.Y)
            return fail(c, PD_EINVAL, "the given tree is not over these nodes");
        left = given->left;
        right = given->right;
        bb = given->bb;
        rep = given->rep;
    } else {
        int32_t* l = bufT<int32_t>(c, B_T_LEFT, M);
        int32_t* r = bufT<int32_t>(c, B_T_RIGHT, M);
        int4* b = bufT<int4>(c, B_T_BB, M);
        int32_t* rp = bufT<int32_t>(c, B_T_REP, M);
        int32_t* par_int = bufT<int32_t>(c, B_T_PARENT, M);
        int32_t* par_leaf = bufT<int32_t>(c, B_T_LPARENT, N);
        int32_t* visit = bufT<int32_t>(c, B_T_VISIT, M);
        int32_t* lc = bufT<int32_t>(c, B_T_LEAVES, M);
        if (!l || !r || !b || !rp || !lc || !par_int || !par_leaf || !visit) return PD_ENOMEM;
        left = l;
        right = r;
        bb = b;
        rep = rp;
        leaves = lc;
        if (N >= 2) {
            k_karras<<<grid_for(N - 1, 256), 256, 0, st>>>(nodes.morton, N, l, r, par_int, par_leaf, visit); pd::count_launch();
            k_bbox<<<grid_for(N, 256), 256, 0, st>>>(N, nodes.X, nodes.Y, l, r, par_int, par_leaf, b, rp, lc, visit); pd::count_launch();
            PD_TRY_CUDA(c, cudaGetLastError());
        }
    }
    PD_TRY_CUDA(c, cudaEventRecord(ev[1], st));
    if (tree) *tree = WsTree{N, nodes.X, nodes.Y, left, right, bb, rep};

    int hb = bits_for((uint64_t)(N + 2));
    int kb = 2 * hb;
    uint64_t sent = (kb >= 64) ? ~0ull : ((1ull << kb) - 1);
    // the pairs of the WSPD: counted, then (unless only the count is wanted) stored
    const WsTree tr{N, nodes.X, nodes.Y, left, right, bb, rep};
    int64_t narcs = 0;
    uint64_t* arcs = nullptr;
    int64_t* h = c->h_small;
    if (N >= 2) {
        WsRec* rec = bufT<WsRec>(c, B_WSFLAG, N - 1);
        int2* F = bufT<int2>(c, B_F0, N - 1);
        if (!rec || !F) return PD_ENOMEM;
        int2* leaf = bufT<int2>(c, B_T_LEAFXY, N);
        if (!leaf) return PD_ENOMEM;
        unsigned long long* words = ws_words(c);
        PD_TRY_CUDA(c, cudaMemsetAsync(words, 0, WS_WORDS * sizeof(unsigned long long), st));
        k_ws_records<<<grid_for(N, 256), 256, 0, st>>>(N - 1, bb, count_only && leaves ? leaves : rep, left, right, nodes.X,
                                                       nodes.Y, s, rec, leaf, F, words + 3); pd::count_launch();
        PD_TRY_CUDA(c, cudaGetLastError());
        int64_t pairs = 0;
        if (count_only) {
            k_diag_counts<<<grid_for(N, 256), 256, 0, st>>>(N, nodes.cntA, nodes.cntB, words + 5); pd::count_launch();
            PD_TRY(ws_walk(c, tr, rec, leaf, s, hb, leaves != nullptr, nullptr, 0, &pairs, st));
        } else {
            // stored into the buffer the context has (64 arcs a node the first time);
            // if they are more, the walk has counted them and the second one stores them
            int64_t room = 0;
            for (int pass = 0; pass < 2; pass++) {
                const int64_t keys = 2 * (pass ? pairs : 32 * N) + 2 * N + 1;
                const bool guess = pass == 0 && !beyond_cap(c, 8 * keys);
                arcs = guess || pass ? bufT<uint64_t>(c, B_ARCKEY, keys) : nullptr;
                if (!arcs && pass == 0) {  // no room for a guess: counted first
                    c->err.clear();
                    PD_TRY(ws_walk(c, tr, rec, leaf, s, hb, false, nullptr, 0, &pairs, st));
                    continue;
                }
                if (!arcs) return PD_ENOMEM;
                room = ((int64_t)(c->bytes[B_ARCKEY] / sizeof(uint64_t)) - (2 * N + 1)) / 2;
                if (pass) PD_TRY_CUDA(c, cudaMemsetAsync(words, 0, 3 * sizeof(unsigned long long), st));
                PD_TRY(ws_walk(c, tr, rec, leaf, s, hb, false, arcs, room, &pairs, st));
                if (pairs <= room) break;
            }
            if (pairs > room) return fail(c, PD_ECUDA, "the WSPD's pairs changed between two walks");
        }
        narcs = 2 * pairs;
    }
    PD_TRY_CUDA(c, cudaEventRecord(ev[2], st));
    if (count_only) {
        // only the counts: arcs of the WSPD and (already here, unless there was nothing to walk) the diagonal's
        if (N < 2) {
            PD_TRY_CUDA(c, cudaMemsetAsync(cnts, 0, 4 * sizeof(unsigned long long), st));
            k_diag_counts<<<grid_for(N, 256), 256, 0, st>>>(N, nodes.cntA, nodes.cntB, cnts); pd::count_launch();
            PD_TRY_CUDA(c, cudaGetLastError());
            PD_TRY_CUDA(c, cudaMemcpyAsync(h + 5, cnts, 2 * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
        }
        PD_TRY_CUDA(c, cudaEventRecord(ev[3], st));
        PD_TRY_CUDA(c, cudaEventSynchronize(ev[3]));
        *out = pd_network{N + 2, narcs + h[5] + h[6] + 1, nullptr, nullptr, nullptr, nullptr};
        if (ms_tree) cudaEventElapsedTime(ms_tree, ev[0], ev[1]);
        if (ms_wspd) cudaEventElapsedTime(ms_wspd, ev[1], ev[2]);
        if (ms_csr) cudaEventElapsedTime(ms_csr, ev[2], ev[3]);
        return PD_OK;
    }
    if (!arcs) {
        arcs = bufT<uint64_t>(c, B_ARCKEY, 2 * N + 1);
        if (!arcs) return PD_ENOMEM;
    }
    // diagonal arcs + masses
    PD_TRY_CUDA(c, cudaMemsetAsync(cnts, 0, 8 * sizeof(unsigned long long), st));
    k_diag_arcs<<<grid_for(N + 1, 256), 256, 0, st>>>(N, nodes.cntA, nodes.cntB, hb, sent, arcs + narcs, cnts); pd::count_launch();
    k_mass<<<grid_for(N, 256), 256, 0, st>>>(N, nodes.cntA, nodes.cntB, cnts); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    PD_TRY_CUDA(c, cudaMemcpyAsync(h, cnts, 4 * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    int64_t ntot = narcs + 2 * N + 1;
    uint64_t* alt = bufT<uint64_t>(c, B_ARCKEY2, ntot);
    if (!alt) return PD_ENOMEM;
    uint32_t *none = nullptr, *none2 = nullptr;
    PD_TRY(sort_u64(c, arcs, alt, none, none2, ntot, kb, st));
    PD_TRY_CUDA(c, cudaStreamSynchronize(st));
    int64_t na = h[0], nb = h[1], FA = h[2], FB = h[3];
    int64_t m = narcs + na + nb + 1;
    int64_t nrows = N + 2;
    out->n_nodes = nrows;
    out->n_arcs = m;
    out->row_ptr = bufT<int64_t>(c, B_ROWPTR, nrows + 1);
    out->head = bufT<int32_t>(c, B_HEAD, m);
    out->cost = bufT<int64_t>(c, B_COST, m);
    out->supply = bufT<int64_t>(c, B_SUPPLY, nrows);
    if (!out->row_ptr || !out->head || !out->cost || !out->supply) return PD_ENOMEM;
    k_row_ptr<<<grid_for(m, 256), 256, 0, st>>>(arcs, m, hb, nrows, out->row_ptr); pd::count_launch();
    k_head_cost<<<grid_for(m, 256), 256, 0, st>>>(arcs, m, hb, N, nodes.X, nodes.Y, out->head, out->cost, dc); pd::count_launch();
    k_supply<<<grid_for(N + 2, 256), 256, 0, st>>>(N, nodes.cntA, nodes.cntB, FA, FB, out->supply); pd::count_launch();
    PD_TRY_CUDA(c, cudaGetLastError());
    PD_TRY_CUDA(c, cudaEventRecord(ev[3], st));
    PD_TRY_CUDA(c, cudaEventSynchronize(ev[3]));
    if (ms_tree) cudaEventElapsedTime(ms_tree, ev[0], ev[1]);
    if (ms_wspd) cudaEventElapsedTime(ms_wspd, ev[1], ev[2]);
    if (ms_csr) cudaEventElapsedTime(ms_csr, ev[2], ev[3]);
    return PD_OK;
}

}  // namespace pd
