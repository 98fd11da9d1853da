// Autotuner of the network simplex's launch parameters (no counterpart in the
// paper, whose block search uses a block of sqrt(arcs)): the pricing block,
// which trades pricing work per pivot against the quality of the entering
// arc, and, in the 64-bit kernel, the walk limit, below which the two half-cycles
// of a pivot are followed by two lanes instead of scanned by the whole CTA.  The
// best values depend on the instance's size, on the kernel that takes it and on the
// GPU, so they are measured: the transportation instances of sample pairs are solved
// once per candidate (block, walk) that makes a difference to their kernel, each
// launch timed by CUDA events, and the fastest is kept per size class
// (floor(log2(arcs + nodes))) and form (kernel, layout, matrix or list) in the
// context -- every later solve of that class and form whose pd_opts.ns_block is 0
// (ns_walk -1) uses it -- and in an optional cache file, one line per (GPU name, SM
// count, form, class): "name sms f<form> class block walk".
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <fstream>
#include <map>
#include <string>
#include <vector>

#include "internal.h"
#include "netsimplex.cuh"

using namespace pd;

namespace {

const int64_t kBlocks[] = {4096, 8192, 16384, 32768};
const int32_t kWalks[] = {0, 8, 32};
constexpr int kDefaultWalk = 0;
using Choices = std::map<int, Ctx::Tuned>;  // by tune_key

std::string device_key(int device, int sms) {
    cudaDeviceProp p;
    std::string name = "gpu";
    if (cudaGetDeviceProperties(&p, device) == cudaSuccess) name = p.name;
    else cudaGetLastError();
    for (char& ch : name)
        if (ch == ' ' || ch == '\t' || ch == '\n') ch = '_';
    return name + " " + std::to_string(sms);
}

// The cache file's choices for this GPU, and the lines of other GPUs.  Lines of
// this GPU that are not of the form above say nothing about the kernel they were
// measured on and are left out.
void read_cache(const char* path, const std::string& key, Choices* mine, std::vector<std::string>* others) {
    if (!path) return;
    std::ifstream f(path);
    for (std::string line; std::getline(f, line);) {
        char name[256];
        int sms = 0, form = 0, cls = 0, walk = 0, end = 0;
        long long blk = 0;
        if (sscanf(line.c_str(), "%255s %d", name, &sms) != 2) continue;
        if (std::string(name) + " " + std::to_string(sms) != key) {
            others->push_back(line);
        } else if (sscanf(line.c_str(), "%255s %d f%d %d %lld %d %n", name, &sms, &form, &cls, &blk, &walk, &end) == 6 &&
                   line.c_str()[end] == 0 && form >= 0 && form < TUNE_FORMS && cls >= 0 && cls < 64 && blk > 0 && walk >= 0) {
            (*mine)[tune_key(cls, form)] = Ctx::Tuned{(int64_t)blk, walk};
        }
    }
}

// Other GPUs' lines stay, this GPU's are replaced.
bool write_cache(const char* path, const std::string& key, const Choices& mine, const std::vector<std::string>& others) {
    FILE* f = fopen(path, "w");
    if (!f) return false;
    for (auto& l : others) fprintf(f, "%s\n", l.c_str());
    for (auto& e : mine)
        fprintf(f, "%s f%d %d %lld %d\n", key.c_str(), e.first % TUNE_FORMS, e.first / TUNE_FORMS,
                (long long)e.second.block, e.second.walk);
    return fclose(f) == 0;
}

// Whether candidate (b, w) is none of those before it to the kernel of h: only
// k_netsimplex walks, and k_simplex32 cuts blocks to its stage.
bool differs(const NSInst& h, int b, int w) {
    if (!h.lay32) return true;
    if (w > 0) return false;
    const int cls = s32_class(h);
    auto same = [&](int k) { return s32_block(k, kBlocks[b]) == s32_block(k, kBlocks[b - 1]); };
    return b == 0 || !same(cls) || (cls == S32_MATRIX && h.n < S32_HALF_NODES && !same(S32_HALF));
}

}  // namespace

namespace pd {

int tune_class(int64_t M) { return M > 0 ? (int)floor(log2((double)M)) : 0; }

const Ctx::Tuned* tuned(const Ctx* c, const NSInst& h) {
    const Ctx* o = c->parent ? c->parent : c;
    auto it = o->tuned.find(tune_key(tune_class(h.m + h.n), tune_form(h)));
    return it == o->tuned.end() ? nullptr : &it->second;
}

}  // namespace pd

extern "C" pd_status pd_autotune(pd_ctx* cx, const pd_diagram* A, const pd_diagram* B, int64_t count, double eps,
                                 const pd_opts* opts, const char* cache_path, pd_tune_result* out, void* stream) {
    Ctx* c = cx;
    if (!c || !out || count < 0 || (count > 0 && (!A || !B))) return PD_EINVAL;
    c->err.clear();
    pd_opts o;
    pd_opts_default(&o);
    if (opts) o = *opts;
    if (!(eps > 0.0) && o.s_override <= 0) return fail(c, PD_EINVAL, "eps must be > 0 (or set s_override)");
    if (o.solver == 1) return fail(c, PD_EINVAL, "the tuner times the network simplex");
    o.warm_start = 0;
    if (cudaSetDevice(c->device) != cudaSuccess) return cuda_fail(c, cudaGetLastError(), "cudaSetDevice");
    cudaStream_t st = (cudaStream_t)stream;
    pd_tune_result r;
    memset(&r, 0, sizeof(r));
    r.size_class = -1;
    const std::string key = device_key(c->device, c->sm_count);
    Choices cached;
    std::vector<std::string> others;
    read_cache(cache_path, key, &cached, &others);
    NSInst* d = bufT<NSInst>(c, B_NS_INST, 1);
    if (!d) return PD_ENOMEM;
    const int NB = (int)(sizeof(kBlocks) / sizeof(kBlocks[0])), NW = (int)(sizeof(kWalks) / sizeof(kWalks[0]));
    // per size class and form: total device time of every candidate over the pairs timed
    std::map<int, std::vector<double>> total;
    std::map<int, double> dflt;
    int first = -1;  // the first pair's
    for (int64_t i = 0; i < count; i++) {
        Front f;
        PD_TRY(front_half(c, A[i], B[i], eps, o, &f, st, true));
        W1Prep w;
        PD_TRY(ns_prepare_w1(c, f.nodes, f.net.n_arcs, f.h.FA, f.h.FB, o, &w, st));
        if (!w.ns.ready) continue;
        const int64_t M = w.ns.h.m + w.ns.h.n;
        const int what = tune_key(tune_class(M), tune_form(w.ns.h));
        if (first < 0) {
            first = what;
            r.size_class = tune_class(M);
        }
        if (cached.count(what)) {
            c->tuned[what] = cached.at(what);
            continue;
        }
        std::vector<double>& t = total[what];
        t.resize((size_t)(NB * NW), 0.0);
        int64_t opt = -1;
        for (int q = 0; q <= NB * NW; q++) {  // the candidates, then the defaults
            NSInst h = w.ns.h;
            if (q < NB * NW) {
                h.block = kBlocks[q / NW];
                h.walk = kWalks[q % NW];
                if (h.block > 4 * M || !differs(h, q / NW, q % NW)) continue;
            } else {
                h.block = ns_default_block(h);
                h.walk = kDefaultWalk;
            }
            NSInst res{};
            c->last_ns_ms = 0.f;
            PD_TRY(ns_run(c, &h, 1, d, &res, st));
            PD_TRY(ns_status(c, res));
            if (opt >= 0 && res.opt != opt) return fail(c, PD_ECUDA, "tuner: the optimum changed with the parameters");
            opt = res.opt;
            if (q < NB * NW) t[(size_t)q] += c->last_ns_ms;
            else dflt[what] += c->last_ns_ms;
        }
        r.pairs++;
    }
    Choices mine = cached;
    for (auto& e : total) {
        size_t best = 0;
        for (size_t q = 1; q < e.second.size(); q++)
            if (e.second[q] > 0.0 && (e.second[best] <= 0.0 || e.second[q] < e.second[best])) best = q;
        c->tuned[e.first] = mine[e.first] = Ctx::Tuned{kBlocks[best / NW], kWalks[best % NW]};
        if (e.first == first) {
            r.best_ms = (float)e.second[best];
            r.default_ms = (float)dflt[e.first];
        }
    }
    r.candidates = NB * NW;
    r.from_cache = (first >= 0 && total.count(first) == 0) ? 1 : 0;
    if (first >= 0) {
        r.ns_block = c->tuned[first].block;
        r.ns_walk = c->tuned[first].walk;
    }
    if (cache_path && !total.empty() && !write_cache(cache_path, key, mine, others))
        return fail(c, PD_EINVAL, std::string("cannot write the tuning cache ") + cache_path);
    *out = r;
    return PD_OK;
}

extern "C" pd_status pd_tuned_block(const pd_ctx* cx, int64_t arcs_and_nodes, int64_t* block_out) {
    if (!cx || !block_out) return PD_EINVAL;
    const Ctx* o = cx->parent ? cx->parent : cx;
    *block_out = 0;
    for (int form : {3, 5, 7, 1, 2, 4, 6, 0}) {  // matrices before lists, 32-bit kernel before 64-bit
        auto it = o->tuned.find(tune_key(tune_class(arcs_and_nodes), form));
        if (it == o->tuned.end()) continue;
        *block_out = it->second.block;
        break;
    }
    return PD_OK;
}
