// Instance record of the single-CTA network simplex kernel (netsimplex.cu).
#pragma once
#include <stddef.h>
#include <stdint.h>

#include "internal.h"

namespace pd {

constexpr int NS_THREADS = 1024;

struct NSInst {
    int32_t n;         // real nodes (root = n)
    int64_t m;         // real arcs
    // arcs a < mst = nS * ld are implicit: tail a / ld, head nS + a % ld, cost
    // cmat[a]; columns nT <= j < ld pad a row to a multiple of eight (cost
    // NS_PAD_COST, never chosen).  Arcs mst <= a < m are explicit: ends from
    // th (tail << 16 | head) when given, else tail/head, cost[a - mst]; th and
    // cost are readable up to a multiple of four arcs
    int64_t mst;
    int64_t nT;
    int64_t nS;
    int64_t ld;
    const int32_t* cmat;
    const uint32_t* th;
    const int32_t* tail;
    const int32_t* head;
    const int32_t* cost;
    const int64_t* supply;
    const int64_t* art;  // n or null: the artificial arc of node i costs big + art[i] (art[i] >= 0; null = 0)
    int64_t* pi;       // n + 1
    int32_t* parent;   // n + 1
    int32_t* pred;     // n + 1 (arc id; artificial arc of node i is m + i; m + n < 2^31)
    int32_t* flow;     // n + 1: flow on the pred arc (total supply < 2^31; bit 31 = up while solving in global mode)
    uint8_t* up;       // n + 1: pred arc points from the node to its parent
    int32_t* ord;      // n + 1 preorder
    int32_t* pos;      // n + 1
    int32_t* size;     // n + 1
    int32_t* tmp;      // n + 1 scratch (re-hang buffer of the global layout)
    int32_t* path;     // 2 (n + 1) scratch: the two half-cycles past the shared-memory part
    int32_t* seg;      // 3 * (2n + 3) scratch: segment start, length, output offset
    int64_t block;     // pricing block (arcs)
    int64_t big;       // cost of the artificial arcs
    int64_t big64;     // ... that the 64-bit kernel takes when it solves the instance again: more than any path cost
    int32_t lay32;     // k_simplex32's layout (1 .. 3; ns_plan may launch 1 as 4, on half an SM); 0: k_netsimplex's
    int32_t big_safe;  // 1: `big` proves infeasibility when artificial flow remains
    int32_t smem_nodes; // node arrays: 1 all in shared memory, 2 all but pred / flow, 3 the 16-bit ones, 0 global
    int32_t walk;      // shared-memory layout: longest half-cycle side followed by the two-lane walk (longer: the scan)
    int32_t init_tree;  // 1: pi, pred, parent, flow, up, ord, pos, size hold a strongly feasible start
    int32_t pad1;
    int64_t scanned;   // result: arcs priced
    int64_t max_pivots;
    uint64_t time_limit_ns;
    // results
    int64_t opt;
    int64_t pivots;    // (k_simplex32 leaves -1 when it has no tree to go on from)
    int64_t degenerate;
    int32_t status;    // 0 ok, 1 infeasible, 2 pivot cap / time, 3 unbounded, 4 path too long, S32_REDO
    int32_t pad;
};

constexpr int32_t NS_PAD_COST = 1 << 30;  // cost of a matrix row's padding columns
constexpr int64_t S32_MAX_COST = int64_t(1) << 25;  // k_simplex32: largest arc cost ...
constexpr int64_t S32_MAX_BIG = int64_t(1) << 26;   // ... and artificial cost
constexpr int32_t S32_REDO = 5;  // status: k_netsimplex has to solve the instance

// The simplex on 32-bit potentials (simplex32.cu), for records with lay32 > 0:
// a kernel per class (layout and arc form), persistent like k_netsimplex, one
// CTA per SM, two of S32_HALF (which ns_plan puts matrices of layout 1 into).
constexpr int S32_CLASSES = 7;
constexpr int S32_MATRIX = 1;             // matrices of layout 1
constexpr int S32_HALF = 6;               // matrices on half an SM
constexpr int32_t S32_HALF_NODES = 3712;  // nodes with the root that half an SM holds
constexpr int32_t S32_SMALL_NODES = 1280; // ... up to which half the threads are the better choice anyway
int s32_class(const NSInst& h);  // -1: not a 32-bit instance
int s32_layout(int64_t N1);      // the smallest layout that holds N1 nodes (0: none)
int64_t s32_block(int cls, int64_t block);  // arcs that a class prices at a time for a block of `block` arcs
inline int s32_grid(int cls, int count, int sm_count) {
    const int most = (cls == S32_HALF ? 2 : 1) * (sm_count > 1 ? sm_count : 1);
    return count < most ? count : most;
}
void s32_launch(int cls, int grid, NSInst* insts, const int32_t* order, int32_t count, int32_t* next,
                cudaStream_t st);
cudaError_t s32_kernel_setup();  // as ns_kernel_setup
// Ends of CSR arcs packed as tail << 16 | head and their costs in 32 bits, in
// chunks of NS_CHUNK arcs, the last one padded, chunk c at place c * stride mod
// their number; bad += costs outside [0, 2^31), *cmax = the largest.  n < 65535.
//
// Neighbouring rows belong to neighbouring nodes, and so do the arcs of a pricing
// block if they stay in order.  Spread out, every block samples the whole network.
// What that does to the pivots depends on the network (in order / spread, s each):
// mixtures of 5,000 + 5,000 points (5.0 M arcs) 0.39 / 0.12, 9,000 + 9,000 (5.1 M)
// 0.88 / 0.37; Gaussians of 5,000 + 5,000 (5.9 M) 0.23 / 0.27, 10,000 + 10,000 (39 M)
// 2.5 / 2.8, 14,500 + 14,500 (7.5 M) 1.4 / 2.1; a mixture of 1.9 M arcs 0.098 / 0.102.
// So spread from NS_SPREAD_ARCS on, where what is gained is the larger part, but only
// up to the nodes of k_simplex32: beyond them longer cycles cost too much (Gaussians
// of 24,432 nodes and 5.0 M arcs 2.9 / 5.0, 32,714 and 8.0 M 16.5 / 52.9).  Rows of a cost
// matrix stay in order too: 100,000 lower-star points 278 ms, spread 291 (path nodes
// a pivot 51, spread 79); 20,000: 119 and 113; 2,000 uniform points: 25.7 and 25.1.
constexpr int64_t NS_CHUNK = 64;
constexpr int64_t NS_SPREAD_ARCS = int64_t(1) << 22;
PD_HD int64_t ns_chunks(int64_t m) { return (m + NS_CHUNK - 1) / NS_CHUNK; }
__global__ void k_arc_pack(const int64_t* __restrict__ rp, const int32_t* __restrict__ hd,
                           const int64_t* __restrict__ cost, int64_t n, int64_t m, int64_t stride,
                           uint32_t* __restrict__ th, int32_t* __restrict__ c32, unsigned long long* __restrict__ bad,
                           unsigned long long* __restrict__ cmax);
// The stride of the chunks of m arcs between `nodes` nodes: 1, or (see above) about the
// golden ratio of their number and coprime to it.
inline int64_t ns_chunk_stride(int64_t nodes, int64_t m) {
    const int64_t n = ns_chunks(m);
    if (m < NS_SPREAD_ARCS || s32_layout(nodes + 1) == 0) return 1;
    int64_t s = (int64_t)(0.6180339887498949 * (double)n);
    for (;; s++) {
        int64_t a = n, b = s;
        while (b) {
            const int64_t t = a % b;
            a = b;
            b = t;
        }
        if (a == 1) return s;
    }
}

// Persistent over `count` instance records taken in `order` (next = a zeroed
// device counter); results are written back into the records.
__global__ void k_netsimplex(NSInst* insts, const int32_t* __restrict__ order, int32_t count,
                             int32_t* __restrict__ next);
// Dynamic shared memory of N1 nodes in shared-memory layout 1, 2 or 3.
size_t ns_smem_bytes(int64_t N1, int layout);
// Raises the kernel's dynamic shared memory limit on the current device once,
// to the most any instance can use (thread-safe; never lowers it).
cudaError_t ns_kernel_setup();
// The layout N1 nodes get beside the kernel's static shared memory
// (max_optin: the device's opt-in limit per CTA): 1 all node arrays in shared
// memory, 2 all but pred and the packed flow, 3 only the four 16-bit arrays,
// 0 none (global memory).
int ns_smem_layout(int64_t N1, int max_optin);
__global__ void k_i64_to_i32_cost(const int64_t* __restrict__ c, int64_t m, int32_t* __restrict__ o,
                                  unsigned long long* __restrict__ bad);
__global__ void k_abs_sum(const int64_t* __restrict__ s, int64_t n, unsigned long long* __restrict__ out);
__global__ void k_check_network(const int64_t* __restrict__ rp, const int32_t* __restrict__ hd, int64_t n, int64_t m,
                                unsigned long long* __restrict__ bad);

// An instance ready to launch (buffers of the context that prepared it).
struct NSPrep {
    NSInst h{};
    bool ready = false;  // false: nothing to solve
};

// The transportation form of one W1 network, prepared for the simplex.
struct W1Prep {
    NSPrep ns;           // ns.ready false: solve the sparse network instead
    DiagCost dc{1, 0, 0};  // creation / destruction costs of the diagonal node's routes
    const int32_t* S = nullptr;
    const int32_t* T = nullptr;
    int64_t nS = 0, nT = 0, ld = 0, nt = 0;
};

// The arcs of an instance (see NSInst).
struct NSArcs {
    int64_t m = 0, mst = 0, nS = 0, nT = 1, ld = 1;
    const int32_t* cmat = nullptr;
    const uint32_t* th = nullptr;
    const int32_t* tail = nullptr;
    const int32_t* head = nullptr;
    const int32_t* cost = nullptr;
    bool complete = false;  // every supply node has an arc to every demand node
    int64_t supply_bound = -1;  // of the sum of |supplies| (-1: not known, it is summed)
};
pd_status ns_prepare_arcs(Ctx* c, int32_t n, const NSArcs& a, const int64_t* supply, int64_t cmax, const pd_opts& o,
                          NSPrep* p, cudaStream_t st);
// Runs `count` prepared instances (one CTA each): h -> device records d ->
// results r (host), synchronising the stream.
pd_status ns_run(Ctx* c, const NSInst* h, int count, NSInst* d, NSInst* r, cudaStream_t st);
// What pd_autotune tells apart: the size class floor(log2(arcs + nodes)) and the form,
// which is the kernel with its layout and whether the arcs are a matrix.
constexpr int TUNE_FORMS = 8;
int tune_class(int64_t M);
inline int tune_form(const NSInst& h) { return 2 * h.lay32 + (h.mst > 0 ? 1 : 0); }
inline int tune_key(int cls, int form) { return cls * TUNE_FORMS + form; }
const Ctx::Tuned* tuned(const Ctx* c, const NSInst& h);  // null: none, the defaults apply
// The kernel an instance goes to, its layout and its artificial costs.
int64_t ns_default_block(const NSInst& h);
void ns_choose_kernel(NSInst* h, int64_t cmax, bool complete, bool smem, int max_optin);
pd_status ns_status(Ctx* c, const NSInst& r);
pd_status ns_prepare_w1(Ctx* c, const pd_nodes& nodes, int64_t n_arcs, int64_t massA, int64_t massB, const pd_opts& o,
                        W1Prep* w, cudaStream_t st);
// Certificate (on the WSPD tree of s) and fallback after the launch; d_res =
// the device record of the solved instance, r = its host copy.  merged ==
// nullptr: no fallback here -- out->method = -1 tells the caller to solve the
// sparse network itself.
pd_status ns_finish_w1(Ctx* c, const WsTree& tr, int64_t s, const pd_network* merged, const pd_opts& o,
                       const W1Prep& w, const NSInst* d_res, const NSInst& r, SolveStats* out, cudaStream_t st);
__global__ void k_certify_tree(const NSInst* __restrict__ I, const int32_t* __restrict__ S,
                               const int32_t* __restrict__ T, int64_t nS, int64_t ld, WsTree tr, int64_t s,
                               DiagCost dc, unsigned long long* __restrict__ out);

// One pair's certificate in a batched launch: its solved record, its
// transportation lists and its WSPD tree.
struct CertJob {
    const NSInst* inst;  // device record (set by ns_run_wave from rec)
    int64_t rec;         // index of the pair's record in the wave
    const int32_t* S;
    const int32_t* T;
    int64_t nS, ld, s;
    WsTree tree;
    DiagCost dc;
};
// k_certify_tree for every job: blockIdx.y = job, out[2 job .. 2 job + 1].
__global__ void k_certify_batch(const CertJob* __restrict__ jobs, unsigned long long* __restrict__ out);

// One wave of a batch as a CUDA graph: upload of the records, the persistent
// simplex over all of them, every pair's certificate, download of records and
// certificate counts.  Captured once per configuration, replayed per wave.
pd_status ns_run_wave(Ctx* c, const NSInst* h, int count, const CertJob* jobs, NSInst* r,
                      unsigned long long* cert, cudaStream_t st);

}  // namespace pd
