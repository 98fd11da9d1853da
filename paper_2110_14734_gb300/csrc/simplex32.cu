// The network simplex of netsimplex.cu for instances whose potentials fit 32
// bits: the same method (block search pricing, strongly feasible tree, explicit
// preorder), one CTA of 512 threads per instance, laid out for the latency of a
// pivot.  netsimplex.cu keeps the 64-bit kernel for every other instance.
//
// What bounds it: a chain of dependent pivots (about 70,000 for a pair of
// 100,000 lower-star points), each a handful of barriers, of dependent
// shared-memory round trips and of instructions that every warp issues; neither
// DRAM nor an arithmetic unit.  Fewer warps issue fewer of them: 512 threads.
//
// Per pivot:
//   price   A block of arcs, copied to shared memory by one bulk copy; eight
//           consecutive arcs of a matrix row per thread and step.  Warps 1 ..
//           price the next block while warp 0 pivots, on the potentials from
//           before that pivot; each thread's best arc is priced again after it,
//           so the entering arc's reduced cost is exact.
//   scan    The preorder keeps, by position, node and end of its subtree in one
//           word (end in the high half), so "the node at position x <= p has p
//           in its subtree" is one unsigned comparison of that word.  A warp
//           reads 128 positions at a time, a lane every 32nd of them.  Nodes above exactly one end of the
//           entering arc are the two half-cycles; they are collected unordered.
//   pivot   One warp: ratio test (positions order a path, so neither the
//           minimum nor its tie rule needs the path in order), flows and
//           subtree ends of the path, and the cut part (from the entering arc's
//           end up to the leaving arc, five nodes on average) sorted.
//   move    One thread per cut node re-roots it; all threads gather the new
//           preorder of the moved range (the cut nodes' sizes are the output
//           offsets of the re-rooted segments), shift the potentials of the cut
//           subtree, and write the range back.  The subtree goes to the start
//           or the end of its new parent's, whichever moves less.
//
// Measured against the 64-bit kernel on the same instances: one pair of 100,000
// lower-star points from a cold start 983 -> 278 ms (11.0 -> 3.6 us a pivot),
// 2,000 uniform points 105 -> 26 ms, an arc list of 1.9 M arcs 206 -> 58 ms.  256
// or 1024 threads were slower (409 and 332 ms where 512 took 308).
//
// 32 bits: |potential| <= 2^28 is kept by a running bound (every pivot shifts a
// subtree by |reduced cost|; the exact maximum is taken again when the bound is
// reached), costs are at most 2^25, so no sum overflows.  An instance that
// would leave the range, or that ends with flow on an artificial arc although
// `big` was not above every path's cost, reports S32_REDO and goes on in the
// 64-bit kernel, from the tree it has.  Artificial arcs leave the problem when they leave the
// tree: they are never priced.
#include <mutex>
#include <type_traits>

#include "internal.h"
#include "netsimplex.cuh"

namespace pd {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int S32_THREADS = 512;
constexpr int S32_HALF_THREADS = 256;         // layout 4
constexpr int S32_HITS = 1024;                // path nodes listed in shared memory
constexpr int S32_PATH = 1024;                // cut nodes listed in shared memory
constexpr int S32_MOVE = 16;                  // moved positions held in registers, per thread
constexpr int32_t S32_LIMIT = 1 << 28;        // |potential|

extern __shared__ __align__(16) unsigned char s32_dyn[];

struct Shared {
    NSInst inst;           // the record being solved
    int64_t pivots, degen, scanned;
    uint64_t t0;
    int32_t key[2][32];    // per-warp pricing minima, double-buffered
    uint32_t ends[2][32];  // tail << 16 | head of each warp's winner
    int32_t arc[2][32];    // its arc id (arc lists)
    uint64_t mbar;         // arrival of the staged block
    int32_t hits;          // path nodes listed
    int32_t late, status, maxpi;
    // the pivot's move, from the pivot warp
    int32_t k, S, dpi, delta, lo, hi, ins, shift;
    unsigned long long obj, art;
    uint16_t list[S32_HITS];
    uint32_t cut[S32_PATH];  // the cut path: position | subtree size << 16, deepest first
};
PD_D Shared& shared() { return *(Shared*)s32_dyn; }  // at the start of the dynamic shared memory

// Dynamic shared memory of a layout: 1 holds every node array (20 B a node), 2
// all but flow and pred (12 B), 3 only the preorder, positions and parents (8 B).
// 4 is 1 for half an SM: a smaller stage and half the threads, so that two
// instances share an SM and one's instructions fill the other's waits (a lone
// CTA issues in 31 % of the cycles).
// The arrays lie at fixed offsets for the layout's capacity, so that no
// register holds them.
// Beside them lies the pricing block's stage.
PD_HD constexpr int32_t s32_capacity(int layout) {
    return layout == 1 ? 7824 : layout == 2 ? 13040 : layout == 3 ? 23664 : S32_HALF_NODES;
}
template <int LAY>
struct Layout {
    static constexpr uint32_t N = s32_capacity(LAY), W2 = 2 * N, W4 = 4 * N;
    static constexpr bool FLOWS = LAY != 2 && LAY != 3, PIS = LAY != 3;  // what shared memory holds
    static constexpr int THREADS = LAY == 4 ? S32_HALF_THREADS : S32_THREADS, WARPS = THREADS / 32;
    static constexpr int PRICERS = THREADS - 32;  // warps 1 .. price, warp 0 pivots
    static constexpr uint32_t STAGE = LAY >= 3 ? 32768 : 65536;  // bytes of a pricing block
    static constexpr uint32_t stage = (sizeof(Shared) + 15) & ~15u, ord = stage + STAGE, pos = ord + W4, par = pos + W2;
    static constexpr uint32_t fu = par + W2, pred = fu + (FLOWS ? W4 : 0);
    // the sinks' potentials pi[nS ..] start on a 16-byte boundary (up to three
    // words of shift), and padding columns are read past the last node
    static constexpr uint32_t pi = pred + (FLOWS ? W4 : 0), total = pi + (PIS ? W4 + 64 : 0);
    static_assert(N % 16 == 0 && total + 16 <= (LAY == 4 ? 113 : 227) * 1024, "the layout does not fit an SM");
};

// Steps of a pricing block of `block` arcs (STEP: a step's arcs): a whole number of
// the pricing threads, at most the stage.
template <int LAY, int STEP>
PD_HD constexpr int32_t block_steps(int64_t block) {
    constexpr int P = Layout<LAY>::PRICERS;
    constexpr int64_t most = (int32_t)(Layout<LAY>::STAGE / 32) / P;
    const int64_t k = (block + STEP * P / 2) / (STEP * P);
    const int32_t m = (int32_t)(k < most ? k : most);
    return P * (m > 1 ? m : 1);
}

template <int LAY>
struct Nodes {
    using L = Layout<LAY>;
    uint32_t shift;  // 4 * ((-nS) mod 4)
    int32_t* gpi;
    uint32_t* gfu;
    int32_t* gpred;
    PD_D int32_t& pi(int32_t v) const {
        if constexpr (L::PIS) return *(int32_t*)(s32_dyn + L::pi + shift + 4 * v);
        else return gpi[v];
    }
    // the same by byte offset: pi(v) is at pi0() + 4 v
    PD_D uint32_t pi0() const { return L::PIS ? L::pi + shift : 0u; }
    PD_D int32_t pi_at(uint32_t off) const {
        if constexpr (L::PIS) return *(const int32_t*)(s32_dyn + off);
        else return *(const int32_t*)((const char*)gpi + off);
    }
    PD_D int4 pi4_at(uint32_t off) const {
        if constexpr (L::PIS) return *(const int4*)(s32_dyn + off);
        else return *(const int4*)((const char*)gpi + off);
    }
    PD_D uint32_t& fu(int32_t v) const {
        if constexpr (L::FLOWS) return *(uint32_t*)(s32_dyn + L::fu + 4 * v);
        else return gfu[v];
    }
    PD_D int32_t& pred(int32_t v) const {
        if constexpr (L::FLOWS) return *(int32_t*)(s32_dyn + L::pred + 4 * v);
        else return gpred[v];
    }
    // position x: node | end of its subtree << 16
    PD_D uint32_t& ord(int32_t x) const { return *(uint32_t*)(s32_dyn + L::ord + 4 * x); }
    PD_D uint16_t& pos(int32_t v) const { return *(uint16_t*)(s32_dyn + L::pos + 2 * v); }
    PD_D uint16_t& par(int32_t v) const { return *(uint16_t*)(s32_dyn + L::par + 2 * v); }
};

PD_D uint64_t s32_now() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// ---- the stage: bulk copies counted by an mbarrier in shared memory
PD_D uint32_t s32_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
PD_D void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
PD_D void bulk_prefetch(const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
// Waits for a phase of the mbarrier; gives up (false) after two seconds.
PD_D bool stage_wait(uint32_t bar, uint32_t parity) {
    uint64_t t0 = 0;
    for (int tries = 0;; tries++) {
        uint32_t ok;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if (tries == 64) t0 = s32_now();
        if (tries > 64 && (tries & 63) == 0 && s32_now() - t0 > 2000000000ull) return false;
    }
}

// The new order's word at offset o of the re-rooted segment, which starts at ins.
template <int LAY>
PD_D uint32_t moved(const Nodes<LAY>& T, const uint32_t* cut, int32_t k, int32_t S, int32_t ins, int32_t o,
                    int32_t dpi) {
    int32_t a = 0, b = k;  // the first cut node whose old subtree holds more than o nodes
    while (a < b) {
        const int32_t mid = (a + b) >> 1;
        if (o < (int32_t)(cut[mid] >> 16)) b = mid;
        else a = mid + 1;
    }
    const int32_t px = (int32_t)(cut[a] & 0xffffu);
    int32_t src = px + o, size = -1;
    if (a == 0) {
        if (o == 0) size = S;
    } else {
        const uint32_t c = cut[a - 1];
        const int32_t below = (int32_t)(c >> 16);
        if (o - below < (int32_t)(c & 0xffffu) - px) src -= below;
        if (o == below) size = S - below;
    }
    const uint32_t w = T.ord(src);
    const int32_t v = (int32_t)(w & 0xffffu);
    if (size < 0) size = (int32_t)(w >> 16) - src;
    T.pi(v) += dpi;
    return (uint32_t)v | (uint32_t)(ins + o + size) << 16;
}

// The new order of [a0, a0 + len), every node shift positions from where it was
// (at most NR of them per thread, in registers), and of the re-rooted segment
// (one per thread).
template <int LAY, int NR>
PD_D void shift_and_insert(const Nodes<LAY>& T, int32_t a0, int32_t len, int32_t shift, int32_t k, int32_t S,
                           int32_t ins, int32_t dpi) {
    const int tid = threadIdx.x;
    const uint32_t turn = (uint32_t)-shift << 16;  // a shifted node's end moves with it
    uint32_t w[NR], wm = 0;
#pragma unroll
    for (int q = 0; q < NR; q++)
        if (tid + q * Layout<LAY>::THREADS < len) w[q] = T.ord(a0 + tid + q * Layout<LAY>::THREADS + shift) + turn;
    if (tid < S) wm = moved<LAY>(T, shared().cut, k, S, ins, tid, dpi);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NR; q++)
        if (tid + q * Layout<LAY>::THREADS < len) {
            const int32_t x = a0 + tid + q * Layout<LAY>::THREADS;
            T.ord(x) = w[q];
            T.pos((int32_t)(w[q] & 0xffffu)) = (uint16_t)x;
        }
    if (tid < S) {
        T.ord(ins + tid) = wm;
        T.pos((int32_t)(wm & 0xffffu)) = (uint16_t)(ins + tid);
    }
}

// A wide move (more of the cut subtree than a position per thread) is gathered
// into the stage, or global scratch where that is too small, before it is
// written back.
template <int LAY>
PD_D bool wide_move(const Shared& s) {
    return s.S > Layout<LAY>::THREADS || s.hi - s.lo - s.S > S32_MOVE * Layout<LAY>::THREADS || s.k >= S32_PATH;
}

// Moves the cut subtree (parameters in shared memory); ends without a barrier
// (the next reader of the order passes the pricing barrier first).
template <int LAY>
PD_D void rehang(const Nodes<LAY>& T, bool wide, const uint32_t* gcut, uint32_t* tmp) {
    Shared& s = shared();
    const int tid = threadIdx.x;
    const int32_t k = s.k, S = s.S, dpi = s.dpi, lo = s.lo, hi = s.hi, ins = s.ins, shift = s.shift;
    // the shifted nodes fill [a0, a0 + len), beside the re-rooted segment
    const int32_t a0 = shift < 0 ? ins + S : lo, len = hi - lo - S;
    if (!wide) {
        if (len <= 2 * Layout<LAY>::THREADS) shift_and_insert<LAY, 2>(T, a0, len, shift, k, S, ins, dpi);
        else if (len <= 5 * Layout<LAY>::THREADS) shift_and_insert<LAY, 5>(T, a0, len, shift, k, S, ins, dpi);
        else shift_and_insert<LAY, S32_MOVE>(T, a0, len, shift, k, S, ins, dpi);
    } else {
        const uint32_t turn = (uint32_t)-shift << 16;
        if (hi - lo <= (int32_t)(Layout<LAY>::STAGE / 4)) tmp = (uint32_t*)(s32_dyn + Layout<LAY>::stage) - lo;
        for (int32_t x = a0 + tid; x < a0 + len; x += Layout<LAY>::THREADS) tmp[x] = T.ord(x + shift) + turn;
        for (int32_t o = tid; o < S; o += Layout<LAY>::THREADS)
            tmp[ins + o] = moved<LAY>(T, k < S32_PATH ? s.cut : gcut, k, S, ins, o, dpi);
        __syncthreads();
        for (int32_t x = lo + tid; x < hi; x += Layout<LAY>::THREADS) {
            const uint32_t w = tmp[x];
            T.ord(x) = w;
            T.pos((int32_t)(w & 0xffffu)) = (uint16_t)x;
        }
    }
}

// What the pivot warp starts from.  pl <= ph: positions of the entering arc's
// ends; nodes at positions up to pl are on pl's side of the cycle, the others on
// ph's; low_i: pl is the tail's.
struct Enter {
    int32_t pl, ph, rc, ent;
    bool low_i;
};

// Flow word w of a path node after a change by f along the cycle.
PD_D uint32_t pushed(uint32_t w, bool on_i, uint32_t f) { return (w >> 31 != 0) == on_i ? w - f : w + f; }

// The ratio test's key of a path node: flows against the cycle (up on i's side,
// down on j's) block it; ties go to j's side, nearest the apex, then to i's side,
// nearest i.
PD_D void block_key(uint32_t w, int32_t x, bool on_i, uint32_t& bf, uint32_t& bt) {
    if ((w >> 31 != 0) == on_i) {
        const uint32_t f = w & 0x7fffffffu, tie = on_i ? 0x1ffffu - (uint32_t)x : (uint32_t)x;
        if (f < bf || (f == bf && tie < bt)) {
            bf = f;
            bt = tie;
        }
    }
}

// The move of the cut subtree [L0, L0 + S): to the start or the end of the part
// of its new parent (position pr, end er), whichever shifts fewer positions.
PD_D void set_move(const Enter& e, bool side_i, int32_t n, int32_t S, int32_t L0, uint32_t mf, int32_t pr, int32_t er) {
    Shared& s = shared();
    s.k = n - 1;
    s.S = S;
    s.delta = (int32_t)mf;
    s.dpi = side_i ? e.rc : -e.rc;  // makes the entering arc's reduced cost 0
    const bool left = pr < L0 && (er <= L0 || L0 - (pr + 1) <= er - (L0 + S));
    const int32_t q = left ? (er <= L0 ? er : pr + 1) : (pr < L0 ? er : pr + 1);
    s.lo = left ? q : L0;
    s.hi = left ? L0 + S : q;
    s.ins = left ? q : q - S;
    s.shift = left ? -S : S;
}

// The pivot warp's part: the ratio test over the listed path nodes, their flows
// and subtree ends, the cut path re-rooted and listed, the move.  Up to 32 NE
// path nodes, held in registers.  false: no arc blocks the cycle.
template <int LAY, int NE>
PD_D bool pivot(const Nodes<LAY>& T, const Enter& en, int32_t hits) {
    Shared& s = shared();
    const int lane = threadIdx.x & 31;
    int32_t x[NE];
    uint32_t o[NE], w[NE];
    bool on_i[NE], ok[NE];
    const uint32_t wl = T.ord(en.pl), wh = T.ord(en.ph);
#pragma unroll
    for (int e = 0; e < NE; e++) {
        ok[e] = lane + 32 * e < hits;
        x[e] = ok[e] ? (int32_t)s.list[lane + 32 * e] : 0;
    }
#pragma unroll
    for (int e = 0; e < NE; e++) o[e] = T.ord(x[e]);
    uint32_t bf = 0xffffffffu, bt = 0xffffffffu;
#pragma unroll
    for (int e = 0; e < NE; e++) w[e] = T.fu((int32_t)(o[e] & 0xffffu));
#pragma unroll
    for (int e = 0; e < NE; e++) {
        on_i[e] = (x[e] <= en.pl) == en.low_i;
        if (ok[e]) block_key(w[e], x[e], on_i[e], bf, bt);
    }
    const uint32_t mf = __reduce_min_sync(FULL, bf);
    if (mf == 0xffffffffu) return false;
    const uint32_t mt = __reduce_min_sync(FULL, bf == mf ? bt : 0xffffffffu);
    const bool side_i = mt >= 0x10000u, cut_low = side_i == en.low_i;
    const int32_t L0 = (int32_t)(side_i ? 0x1ffffu - mt : mt);
    const int32_t S = (int32_t)(T.ord(L0) >> 16) - L0;
    const uint32_t wr = cut_low ? wh : wl;  // the other end: the subtree's new parent
    const int32_t xq = cut_low ? en.pl : en.ph;
    bool cut[NE];
    int32_t up[NE], pred[NE];
#pragma unroll
    for (int e = 0; e < NE; e++) {
        const bool same = on_i[e] == side_i;
        const int32_t v = (int32_t)(o[e] & 0xffffu);
        cut[e] = ok[e] && same && x[e] >= L0;
        w[e] = pushed(w[e], on_i[e], mf);
        up[e] = pred[e] = 0;
        if (cut[e]) {
            up[e] = T.par(v);
            pred[e] = T.pred(v);
        } else if (ok[e]) {
            if (mf) T.fu(v) = w[e];
            // the cut subtree leaves the chain above it and joins the other end's
            T.ord(x[e]) = same ? o[e] - ((uint32_t)S << 16) : o[e] + ((uint32_t)S << 16);
        }
    }
    __syncwarp();
    // re-rooting: a cut node's parent hangs from it by the arc between them
    int32_t n = 0, rank[NE];
    uint32_t bal[NE];
#pragma unroll
    for (int e = 0; e < NE; e++) {
        const int32_t v = (int32_t)(o[e] & 0xffffu);
        if (cut[e] && x[e] != L0) {
            T.par(up[e]) = (uint16_t)v;
            T.pred(up[e]) = pred[e];
            T.fu(up[e]) = w[e] ^ 0x80000000u;
        }
        if (cut[e] && x[e] == xq) {
            T.par(v) = (uint16_t)(wr & 0xffffu);
            T.pred(v) = en.ent;
            T.fu(v) = mf | (side_i ? 0x80000000u : 0u);  // the entering arc runs i -> j
        }
        bal[e] = __ballot_sync(FULL, cut[e]);
        n += __popc(bal[e]);
        rank[e] = 0;
    }
#pragma unroll
    for (int f = 0; f < NE; f++)
        for (uint32_t b = bal[f]; b; b &= b - 1) {
            const int32_t y = __shfl_sync(FULL, x[f], __ffs(b) - 1);
#pragma unroll
            for (int e = 0; e < NE; e++) rank[e] += y > x[e];
        }
#pragma unroll
    for (int e = 0; e < NE; e++)
        if (cut[e]) s.cut[rank[e]] = (uint32_t)x[e] | ((o[e] >> 16) - (uint32_t)x[e]) << 16;
    if (lane == 0) set_move(en, side_i, n, S, L0, mf, cut_low ? en.ph : en.pl, (int32_t)(wr >> 16));
    return true;
}

// The same for any number of path nodes (lists in shared, then global memory).
template <int LAY>
PD_D bool pivot_long(const Nodes<LAY>& T, const Enter& en, int32_t hits, int32_t* glist, uint32_t* gcut) {
    Shared& s = shared();
    const int lane = threadIdx.x & 31;
    auto entry = [&](int32_t t) -> int32_t { return t < S32_HITS ? (int32_t)s.list[t] : glist[t]; };
    uint32_t bf = 0xffffffffu, bt = 0xffffffffu;
    for (int32_t t = lane; t < hits; t += 32) {
        const int32_t x = entry(t);
        block_key(T.fu((int32_t)(T.ord(x) & 0xffffu)), x, (x <= en.pl) == en.low_i, bf, bt);
    }
    const uint32_t mf = __reduce_min_sync(FULL, bf);
    if (mf == 0xffffffffu) return false;
    const uint32_t mt = __reduce_min_sync(FULL, bf == mf ? bt : 0xffffffffu);
    const bool side_i = mt >= 0x10000u, cut_low = side_i == en.low_i;
    const int32_t L0 = (int32_t)(side_i ? 0x1ffffu - mt : mt);
    const int32_t S = (int32_t)(T.ord(L0) >> 16) - L0;
    const int32_t pr = cut_low ? en.ph : en.pl, xq = cut_low ? en.pl : en.ph;
    const uint32_t wr = T.ord(pr);
    __syncwarp();
    int32_t n = 0;
    for (int32_t b = 0; b < hits; b += 32) {
        bool on_cut = false;
        if (b + lane < hits) {
            const int32_t x = entry(b + lane);
            const bool on_i = (x <= en.pl) == en.low_i, same = on_i == side_i;
            const uint32_t o = T.ord(x);
            const int32_t v = (int32_t)(o & 0xffffu);
            if (mf) T.fu(v) = pushed(T.fu(v), on_i, mf);
            on_cut = same && x >= L0;
            if (!on_cut) T.ord(x) = same ? o - ((uint32_t)S << 16) : o + ((uint32_t)S << 16);
        }
        n += __popc(__ballot_sync(FULL, on_cut));
    }
    __syncwarp();
    // the cut path from its deepest node up, by one lane; then re-rooted from the
    // top down, 32 nodes at a time, each from the one below it
    uint32_t* cut = n <= S32_PATH ? s.cut : gcut;
    if (lane == 0) {
        int32_t x = xq;
        for (int32_t t = 0; t < n; t++) {
            const uint32_t o = T.ord(x);
            cut[t] = (uint32_t)x | ((o >> 16) - (uint32_t)x) << 16;
            if (t + 1 < n) x = T.pos(T.par((int32_t)(o & 0xffffu)));
        }
    }
    __syncwarp();
    auto node = [&](int32_t t) -> int32_t { return (int32_t)(T.ord((int32_t)(cut[t] & 0xffffu)) & 0xffffu); };
    for (int32_t b = n - 1; b >= 0; b -= 32) {
        const int32_t t = b - lane;
        int32_t v = 0, below = 0, pred = 0;
        uint32_t w = 0;
        if (t >= 0) {
            v = node(t);
            if (t > 0) {
                below = node(t - 1);
                pred = T.pred(below);
                w = T.fu(below) ^ 0x80000000u;
            } else {
                below = (int32_t)(wr & 0xffffu);
                pred = en.ent;
                w = mf | (side_i ? 0x80000000u : 0u);
            }
        }
        __syncwarp();
        if (t >= 0) {
            T.par(v) = (uint16_t)below;
            T.pred(v) = pred;
            T.fu(v) = w;
        }
        __syncwarp();
    }
    if (lane == 0) set_move(en, side_i, n, S, L0, mf, pr, (int32_t)(wr >> 16));
    return true;
}

// IMPL: the arcs are a cost matrix (then a few explicit ones); otherwise an arc list.
template <int LAY, bool IMPL>
PD_D void s32_body(NSInst& G) {
    Shared& s = shared();
    const NSInst& I = s.inst;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int32_t n = I.n, root = n, N1 = n + 1;
    Nodes<LAY> T;
    T.shift = 4u * (uint32_t)(-(int32_t)I.nS & 3);
    T.gpi = (int32_t*)I.pi + (-(int32_t)I.nS & 3);
    T.gfu = (uint32_t*)I.flow;
    T.gpred = I.pred;
    constexpr int STEP = IMPL ? 8 : 4;     // arcs of a thread's step
    constexpr int MAXIT = (s32_capacity(LAY) - 1) / (128 * Layout<LAY>::WARPS) + 1;  // scan rounds
    static_assert(4 * MAXIT <= 64, "a thread's scan mask");

    // ---- initial tree ------------------------------------------------------
    const int32_t big = (int32_t)I.big;
    int32_t worst = 0;  // largest |potential|
    if (tid == 0) {
        s.status = 0;
        s.late = 0;
        s.maxpi = 0;
        s.hits = 0;
        s.pivots = s.degen = s.scanned = 0;
        s.t0 = s32_now();
    }
    if (I.init_tree) {
        // the 64-bit potentials share the memory of the 32-bit ones of layout 3: all are read first
        for (int32_t v = tid; v < N1; v += Layout<LAY>::THREADS) {
            const int64_t p = G.pi[v];
            worst = max(worst, p > S32_LIMIT || p < -S32_LIMIT ? S32_LIMIT + 1 : (int32_t)(p < 0 ? -p : p));
            I.tmp[v] = (int32_t)p;
        }
        __syncthreads();
        for (int32_t v = tid; v < N1; v += Layout<LAY>::THREADS) {
            const uint32_t f = (uint32_t)G.flow[v] | (G.up[v] ? 0x80000000u : 0u);
            const int32_t x = G.pos[v];
            T.pi(v) = I.tmp[v];
            T.pred(v) = G.pred[v];
            T.fu(v) = f;
            T.par(v) = (uint16_t)G.parent[v];
            T.pos(v) = (uint16_t)x;
            T.ord(x) = (uint32_t)v | (uint32_t)(x + G.size[v]) << 16;
        }
    } else {
        for (int32_t v = tid; v < n; v += Layout<LAY>::THREADS) {
            const int64_t b = I.supply[v];
            const int32_t ca = I.art ? big + (int32_t)I.art[v] : big;
            T.pi(v) = b >= 0 ? ca : -ca;
            T.pred(v) = (int32_t)(I.m + v);
            T.fu(v) = (uint32_t)(b >= 0 ? b : -b) | (b >= 0 ? 0x80000000u : 0u);
            T.par(v) = (uint16_t)root;
            T.pos(v) = (uint16_t)(1 + v);
            T.ord(1 + v) = (uint32_t)v | (uint32_t)(2 + v) << 16;
            worst = max(worst, ca);
        }
        if (tid == 0) {
            T.pi(root) = 0;
            T.pred(root) = -1;
            T.fu(root) = 0;
            T.par(root) = 0xffff;
            T.pos(root) = 0;
            T.ord(0) = (uint32_t)root | (uint32_t)N1 << 16;
        }
    }
    if (tid < 8) T.pi(N1 + tid) = 0;  // read by padding columns
    __syncthreads();
    worst = __reduce_max_sync(FULL, worst);
    if (lane == 0) atomicMax(&s.maxpi, worst);
    __syncthreads();
    int32_t bound = s.maxpi;
    if (bound > S32_LIMIT) {
        if (tid == 0) G.status = S32_REDO;
        return;
    }

    // Arcs in steps; the matrix first.  The explicit arcs of a matrix instance are
    // blocks of their own, read in place.
    const int32_t QI = IMPL ? (int32_t)(I.mst / STEP) : (int32_t)((I.m + 3) >> 2);  // staged steps
    const int32_t Q = IMPL ? QI + (int32_t)((I.m - I.mst + 3) >> 2) : QI;
    const int32_t B = block_steps<LAY, STEP>(I.block);
    const int pt = tid - 32;  // this pricing thread
    const int32_t nS = (int32_t)I.nS, ldq = IMPL ? (int32_t)(I.ld / STEP) : 1;
    // row and sinks' potentials of a step, as byte offsets
    const uint32_t pb = T.pi0(), row_end = pb + 4u * (uint32_t)nS + 32u * (uint32_t)ldq;
    const uint32_t step_i = 4u * (uint32_t)(Layout<LAY>::PRICERS / ldq), step_j = 32u * (uint32_t)(Layout<LAY>::PRICERS % ldq);
    const uint32_t oi_0 = pb + 4u * (uint32_t)(max(pt, 0) / ldq);
    const uint32_t oj_0 = pb + 4u * (uint32_t)nS + 32u * (uint32_t)(max(pt, 0) % ldq);
    uint32_t oi = oi_0, oj = oj_0;  // of step next + pt
    int32_t next = 0;               // first step of the next block
    int buf = 0;
    uint32_t parity = 0;
    const uint32_t bar = s32_addr(&s.mbar);
    const unsigned char* stage = s32_dyn + Layout<LAY>::stage;
    // one thread, once after each priced block: block `next` into the stage, the one after it into L2
    auto fetch = [&]() {
        const int32_t steps = min(B, QI - next);
        if (steps <= 0) return;
        const char* c = (const char*)(IMPL ? I.cmat : I.cost);
        constexpr int32_t W = 4 * STEP;  // bytes of a step's costs
        const uint32_t bytes = (uint32_t)(steps * W);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(IMPL ? bytes : 2 * bytes)
                     : "memory");
        bulk_copy(s32_addr(stage), c + (int64_t)next * W, bytes, bar);
        if constexpr (!IMPL) bulk_copy(s32_addr(stage) + Layout<LAY>::STAGE / 2, (const char*)I.th + (int64_t)next * W, bytes, bar);
        const int32_t after = min(B, QI - next - steps);
        if (after > 0) {
            bulk_prefetch(c + (int64_t)(next + steps) * W, (uint32_t)(after * W));
            if constexpr (!IMPL) bulk_prefetch((const char*)I.th + (int64_t)(next + steps) * W, (uint32_t)(after * W));
        }
    };
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        fetch();
    }
    __syncthreads();

    // The pricing threads price block `next`: each keeps its most negative arc
    // (reduced cost, cost, offsets of its ends' potentials).
    int32_t best = 0, cost = 0, arc = 0, steps = 0;
    uint32_t bi = 0, bj = 0;
    auto price = [&]() {
        const int32_t qa = next, qe = min(qa + B, qa < QI ? QI : Q);
        steps = qe - qa;
        next = qe >= Q ? 0 : qe;
        best = 0;
        bi = bj = pb;
        if (wid > 0) {
            auto four = [&](int32_t a, const int4& cc, const int4& tt) {  // listed arcs
                const uint32_t t4[4] = {(uint32_t)tt.x, (uint32_t)tt.y, (uint32_t)tt.z, (uint32_t)tt.w};
                const int32_t c4[4] = {cc.x, cc.y, cc.z, cc.w};
#pragma unroll
                for (int e = 0; e < 4; e++) {
                    const uint32_t t = pb + 4u * (t4[e] >> 16), h = pb + 4u * (t4[e] & 0xffffu);
                    const int32_t r = c4[e] + T.pi_at(h) - T.pi_at(t);
                    if (r < best) {
                        best = r;
                        bi = t;
                        bj = h;
                        arc = 4 * a + e;
                    }
                }
            };
            if (qa < QI) {
                if (!stage_wait(bar, parity)) s.status = 4;
                parity ^= 1;
                if constexpr (IMPL) {
                    // 16-byte halves in an order that keeps a warp off bank conflicts
                    const uint32_t h = (uint32_t)(lane & 4) << 2;
                    const unsigned char* at = stage + 32 * pt + h;
                    const unsigned char* const end = stage + 32 * steps;
#pragma unroll 1
                    for (; at < end; at += 32 * Layout<LAY>::PRICERS) {
                        const int4 c0 = *(const int4*)at, c1 = *(const int4*)(at + 16 - 2 * (int)h);
                        const int4 p0 = T.pi4_at(oj + h), p1 = T.pi4_at(oj + 16u - h);
                        const int32_t r0 = c0.x + p0.x, r1 = c0.y + p0.y, r2 = c0.z + p0.z, r3 = c0.w + p0.w,
                                      r4 = c1.x + p1.x, r5 = c1.y + p1.y, r6 = c1.z + p1.z, r7 = c1.w + p1.w;
                        const int32_t ma = min(__vimin3_s32(r0, r1, r2), r3), mb = min(__vimin3_s32(r4, r5, r6), r7);
                        const int32_t r = min(ma, mb) - T.pi_at(oi);
                        if (r < best) {
                            best = r;
                            bi = oi;
                            bj = oj + (ma <= mb ? h + (r0 == ma ? 0u : r1 == ma ? 4u : r2 == ma ? 8u : 12u)
                                                : 16u - h + (r4 == mb ? 0u : r5 == mb ? 4u : r6 == mb ? 8u : 12u));
                        }
                        oi += step_i;
                        oj += step_j;
                        if (oj >= row_end) {
                            oj -= 32u * (uint32_t)ldq;
                            oi += 4u;
                        }
                    }
                } else {
#pragma unroll 1
                    for (int32_t a = pt; a < steps; a += Layout<LAY>::PRICERS)
                        four(qa + a, *(const int4*)(stage + 16 * a), *(const int4*)(stage + Layout<LAY>::STAGE / 2 + 16 * a));
                }
            } else {  // (matrix instances)
#pragma unroll 1
                for (int32_t a = qa - QI + pt; a < qe - QI; a += Layout<LAY>::PRICERS)
                    four(a, __ldcg((const int4*)I.cost + a), __ldcg((const int4*)I.th + a));
            }
            cost = best + T.pi_at(bi) - T.pi_at(bj);
            if (tid == 32) s.scanned += (int64_t)steps * (qa < QI ? STEP : 4);
        }
        if (next == 0) {
            oi = oi_0;
            oj = oj_0;
        }
    };

    // A block priced while the pivot warp works sees the potentials from before
    // that pivot's move (stale): each thread's arc is then priced again, and if
    // none is left the block proves nothing.  Optimal: all arcs priced without a
    // negative one and without a pivot in between (clean).
    bool stale = false;
    int32_t clean = 0;
    if (Q > 0) price();
    for (;;) {
        // ---- the entering arc --------------------------------------------------
        const int32_t wmin = __reduce_min_sync(FULL, best);
        const uint32_t mine = (bi - pb) << 14 | (bj - pb) >> 2;  // tail << 16 | head
        const uint32_t cand = wmin < 0 && best == wmin ? mine : 0xffffffffu;
        const uint32_t wends = __reduce_min_sync(FULL, cand);
        if (lane == 0) {
            s.key[buf][wid] = wmin;
            s.ends[buf][wid] = wends;
        }
        if (!IMPL && wmin < 0 && cand == wends) s.arc[buf][wid] = arc;
        __syncthreads();
        if (tid == 0 && !stale && Q > 0) fetch();
        const int32_t k2 = s.key[buf][lane & (Layout<LAY>::WARPS - 1)];
        const uint32_t e2 = s.ends[buf][lane & (Layout<LAY>::WARPS - 1)];
        const int32_t rc = __reduce_min_sync(FULL, k2);
        if (rc >= 0) {
            buf ^= 1;
            if (!stale) clean += steps;
            if (clean >= Q || s.status) break;  // no arc with a negative reduced cost: optimal
            stale = false;
            price();
            continue;
        }
        const uint32_t c2 = k2 == rc ? e2 : 0xffffffffu;
        const uint32_t ends = __reduce_min_sync(FULL, c2);
        const int32_t ei = (int32_t)(ends >> 16), ej = (int32_t)(ends & 0xffffu);
        int32_t ent = 0;
        if constexpr (!IMPL) ent = s.arc[buf][__ffs(__ballot_sync(FULL, c2 == ends)) - 1];
        buf ^= 1;
        clean = 0;
        if (s.late | s.status) {
            if (tid == 0 && s.late) s.status = 2;
            break;
        }
        if (bound > S32_LIMIT + rc) {
            // the running bound is used up: take the exact maximum (pi[0..n])
            __syncthreads();
            if (tid == 0) s.maxpi = 0;
            __syncthreads();
            int32_t w = 0;
            for (int32_t v = tid; v < N1; v += Layout<LAY>::THREADS) w = max(w, abs(T.pi(v)));
            w = __reduce_max_sync(FULL, w);
            if (lane == 0) atomicMax(&s.maxpi, w);
            __syncthreads();
            bound = s.maxpi;
            if (bound > S32_LIMIT + rc) {
                if (tid == 0) s.status = S32_REDO;
                break;
            }
        }
        bound -= rc;

        // ---- scan: the nodes above exactly one end of the entering arc --------
        const int32_t pI = T.pos(ei), pJ = T.pos(ej);
        const bool low_i = pI < pJ;
        const int32_t pl = low_i ? pI : pJ, ph = low_i ? pJ : pI;
        {
            // up to pl: pl < end <= ph; in (pl, ph]: end > ph; both as w - A < R
            const uint32_t A1 = (uint32_t)(pl + 1) << 16, R1 = (uint32_t)(ph - pl) << 16;
            const uint32_t A2 = (uint32_t)(ph + 1) << 16, R2 = 0u - A2;
            // neighbours in the order go to different lanes: a path's nodes are often next to each other
            using Mask = std::conditional_t<(MAXIT <= 8), uint32_t, uint64_t>;
            Mask m = 0;
            int32_t x = 128 * wid + lane;
#pragma unroll
            for (int it = 0; it < MAXIT; it++, x += 128 * Layout<LAY>::WARPS) {
                const int32_t xb = 128 * wid + it * 128 * Layout<LAY>::WARPS;
                if (xb > ph) break;
                uint32_t w[4];
#pragma unroll
                for (int e = 0; e < 4; e++) w[e] = T.ord(x + 32 * e);  // past the last node: not looked at, x > ph
                if (xb + 127 <= pl || (xb > pl && xb + 127 <= ph)) {
                    const uint32_t A = xb > pl ? A2 : A1, R = xb > pl ? R2 : R1;
#pragma unroll
                    for (int e = 0; e < 4; e++)
                        if (w[e] - A < R) m |= Mask(1) << (4 * it + e);
                } else {
#pragma unroll
                    for (int e = 0; e < 4; e++)
                        if (x + 32 * e <= pl ? w[e] - A1 < R1 : x + 32 * e <= ph && w[e] - A2 < R2)
                            m |= Mask(1) << (4 * it + e);
                }
            }
            if (m) {
                int32_t at = atomicAdd(&s.hits, __popcll(m));
                for (; m; m &= m - 1, at++) {
                    const int b = __ffsll((long long)m) - 1;
                    const int32_t y = 128 * (wid + Layout<LAY>::WARPS * (b >> 2)) + 32 * (b & 3) + lane;
                    if (at < S32_HITS) s.list[at] = (uint16_t)y;
                    else I.path[at] = y;
                }
            }
        }
        __syncthreads();

        // ---- pivot --------------------------------------------------------------
        if (wid == 0) {
            Enter en{pl, ph, rc, ent, low_i};
            if constexpr (IMPL) {  // the entering arc's id follows from its ends
                const int32_t D = nS + (int32_t)I.nT;
                en.ent = ei < nS && ej < D ? ei * (int32_t)I.ld + (ej - nS)
                                           : (int32_t)I.mst + (ei == D ? ej - nS : ei);
            }
            const int32_t hits = s.hits;
            const bool ok = hits <= 32    ? pivot<LAY, 1>(T, en, hits)
                            : hits <= 64  ? pivot<LAY, 2>(T, en, hits)
                            : hits <= 128 ? pivot<LAY, 4>(T, en, hits)
                                          : pivot_long<LAY>(T, en, hits, I.path, (uint32_t*)I.seg);
            if (!ok && lane == 0) s.status = 3;
        }
        price();  // (warps 1 ..)
        if (tid == 32) {
            // pivot cap and wall-clock limit (looked at every 128 pivots) take effect at the next pivot
            const int64_t p = ++s.pivots;
            if (p >= I.max_pivots || ((p & 127) == 0 && s32_now() - s.t0 > I.time_limit_ns)) s.late = 1;
        }
        __syncthreads();
        const bool wide = wide_move<LAY>(s);
        if (tid == 0) {
            if (!wide) fetch();
            s.hits = 0;
            s.degen += s.delta == 0;
        }
        if (s.status == 3) {  // no arc blocks the cycle
            if (tid == 0 && wide) fetch();
            break;
        }
        rehang<LAY>(T, wide, (const uint32_t*)I.seg, (uint32_t*)I.tmp);
        if (wide) {  // the stage is free again
            __syncthreads();
            if (tid == 0) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                fetch();
            }
        }
        best = min(0, cost - T.pi_at(bi) + T.pi_at(bj));
        stale = true;
    }

    // ---- result ---------------------------------------------------------------
    // a block is on its way unless the matrix's explicit arcs are next
    if (wid > 0 && next < QI) stage_wait(bar, parity);
    __syncthreads();
    if (tid == 0) asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
    if (tid == 0) {
        s.obj = 0;
        s.art = 0;
    }
    for (int32_t v = tid; v < N1; v += Layout<LAY>::THREADS) I.tmp[v] = T.pi(v);
    __syncthreads();
    unsigned long long obj = 0, art = 0;
    for (int32_t v = tid; v < N1; v += Layout<LAY>::THREADS) {
        const uint32_t w = T.fu(v);
        const int32_t a = T.pred(v), f = (int32_t)(w & 0x7fffffffu);
        if (v < n) {
            if (a >= I.m) art += f != 0;
            else if (f > 0) obj += (unsigned long long)(a < I.mst ? I.cmat[a] : I.cost[a - I.mst]) * (unsigned long long)f;
        }
        const int32_t x = T.pos(v), p = T.par(v);
        G.pi[v] = I.tmp[v];
        G.pred[v] = a;
        G.flow[v] = f;
        G.up[v] = (uint8_t)(w >> 31);
        G.parent[v] = p == 0xffff ? -1 : p;
        G.size[v] = (int32_t)(T.ord(x) >> 16) - x;
        G.pos[v] = x;
    }
    atomicAdd(&s.obj, obj);
    atomicAdd(&s.art, art);
    __syncthreads();
    if (tid == 0) {
        G.pivots = s.pivots;
        G.degenerate = s.degen;
        G.scanned = s.scanned;
        G.opt = (int64_t)s.obj;
        G.status = s.status ? s.status : !s.art ? 0 : I.big_safe ? 1 : S32_REDO;
    }
}

// Persistent over `count` instances of one layout and arc form (a kernel of its
// own per variant: several bodies in one kernel spill).
template <int LAY, bool IMPL>
__global__ void __launch_bounds__(Layout<LAY>::THREADS, LAY == 4 ? 2 : 1) k_simplex32(NSInst* insts, const int32_t* __restrict__ order,
                                                             int32_t count, int32_t* __restrict__ next) {
    __shared__ int32_t s_k;
    for (;;) {
        if (threadIdx.x == 0) s_k = atomicAdd(next, 1);
        __syncthreads();
        const int32_t k = s_k;
        __syncthreads();
        if (k >= count) break;
        if (threadIdx.x == 0) shared().inst = insts[order[k]];
        __syncthreads();
        s32_body<LAY, IMPL>(insts[order[k]]);
        __syncthreads();
    }
}

size_t smem_bytes(int layout) {
    return layout == 1 ? Layout<1>::total : layout == 2 ? Layout<2>::total : layout == 3 ? Layout<3>::total : Layout<4>::total;
}

using Kernel = void (*)(NSInst*, const int32_t*, int32_t, int32_t*);
const Kernel kernels[S32_CLASSES] = {k_simplex32<1, false>, k_simplex32<1, true>, k_simplex32<2, false>,
                                     k_simplex32<2, true>,  k_simplex32<3, false>, k_simplex32<3, true>,
                                     k_simplex32<4, true>};

}  // namespace

int s32_class(const NSInst& h) { return h.lay32 ? 2 * (h.lay32 - 1) + (h.mst > 0 ? 1 : 0) : -1; }

template <int LAY>
static int64_t block_arcs(bool matrix, int64_t block) {
    return matrix ? 8 * (int64_t)block_steps<LAY, 8>(block) : 4 * (int64_t)block_steps<LAY, 4>(block);
}

int64_t s32_block(int cls, int64_t block) {
    if (cls == S32_HALF) return block_arcs<4>(true, block);
    const bool matrix = cls & 1;
    return cls / 2 == 0 ? block_arcs<1>(matrix, block) : cls / 2 == 1 ? block_arcs<2>(matrix, block) : block_arcs<3>(matrix, block);
}

void s32_launch(int cls, int grid, NSInst* insts, const int32_t* order, int32_t count, int32_t* next,
                cudaStream_t st) {
    kernels[cls]<<<grid, cls == S32_HALF ? S32_HALF_THREADS : S32_THREADS, smem_bytes(cls / 2 + 1), st>>>(insts, order, count, next);
}

int s32_layout(int64_t N1) {
    for (int layout = 1; layout <= 3; layout++)
        if (N1 <= s32_capacity(layout)) return layout;
    return 0;
}

cudaError_t s32_kernel_setup() {
    static std::mutex mu;
    static bool done[256] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 256) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> g(mu);
    if (done[dev]) return cudaSuccess;
    for (int q = 0; q < S32_CLASSES; q++) {
        e = cudaFuncSetAttribute(kernels[q], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem_bytes(q / 2 + 1));
        if (e != cudaSuccess) return e;
    }
    done[dev] = true;
    return cudaSuccess;
}

}  // namespace pd
