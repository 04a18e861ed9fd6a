// Many independent inverse problems advanced together (C ABI smc_batch_*).
//
// Each problem is its own handle (own hierarchy, K, data, particles). A batch evaluation takes,
// per problem, a level and a device array of particles, and runs: the tensor-core KL synthesis of
// every mixed-precision problem, then ONE persistent solve launch per level size, whose blocks pull
// (problem, particle) items across all problems of that size from a device counter. The whole
// sequence is captured once into a CUDA graph and replayed while the problems, levels, counts and
// pointers stay the same (the signature); a new signature rebuilds the argument tables and the graph.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "batch.h"
#include "handle.h"
#include "internal.h"
#include "smc_device.h"

namespace mls2mc {

long long launch_count();

bool Forks::ready() {
    for (int i = 0; i < kMax; ++i) {
        if (!s[i] && cudaStreamCreateWithFlags(&s[i], cudaStreamNonBlocking) != cudaSuccess) return false;
        if (!end[i] && cudaEventCreateWithFlags(&end[i], cudaEventDisableTiming) != cudaSuccess) return false;
    }
    return start || cudaEventCreateWithFlags(&start, cudaEventDisableTiming) == cudaSuccess;
}

cudaError_t Forks::fork(int n, cudaStream_t st) {
    cudaError_t e = cudaEventRecord(start, st);
    for (int i = 0; i < n && e == cudaSuccess; ++i) e = cudaStreamWaitEvent(s[i], start, 0);
    return e;
}

cudaError_t Forks::join(int n, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < n && e == cudaSuccess; ++i) {
        e = cudaEventRecord(end[i], s[i]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(st, end[i], 0);
    }
    return e;
}

Forks::~Forks() {
    for (int i = 0; i < kMax; ++i) {
        if (s[i]) cudaStreamDestroy(s[i]);
        if (end[i]) cudaEventDestroy(end[i]);
    }
    if (start) cudaEventDestroy(start);
}

// A small problem's split and contraction are a few microseconds each on a few SMs, and a batch has many. One
// launch splits for all of them, and in a graph the contractions are parallel branches: 64 problems of 16 .. 256
// particles 825 us an evaluation with everything in one line, 672 us. Launched eagerly they stay on the
// caller's stream: there the host's launches set the pace.
int synth_many(const std::vector<SynthReq>& reqs, Forks* forks, cudaStream_t st, std::string* err) {
    std::vector<SplitTask> tasks;
    for (const SynthReq& r : reqs) {
        if (kl_groups(r.h->K) > 1) continue;
        const int rc = r.h->synth_reserve(r.level, r.n);
        if (rc != SMC_OK) {
            *err = r.h->last_error;
            return rc;
        }
        tasks.push_back({r.theta, r.h->synth_theta_buf, r.n, r.h->K, kl_split_total(r.h->K)});
    }
    cudaError_t e = theta_split_multi_launch(tasks, st);
    const int nf = forks && reqs.size() > 1 ? std::min<int>(Forks::kMax, (int)reqs.size()) : 0;
    if (e == cudaSuccess && nf) e = forks->fork(nf, st);
    int rc = SMC_OK;
    for (size_t i = 0; i < reqs.size() && rc == SMC_OK && e == cudaSuccess; ++i) {
        const SynthReq& r = reqs[i];
        rc = r.h->synth_kappa(r.level, r.n, r.theta, nf ? forks->s[i % nf] : st, kl_groups(r.h->K) > 1);
        if (rc != SMC_OK) *err = r.h->last_error;
    }
    if (e == cudaSuccess && nf) e = forks->join(nf, st);   // also after a failure: a capture must be able to end
    if (rc == SMC_OK && e != cudaSuccess) {
        *err = std::string("batched synthesis: ") + cudaGetErrorString(e);
        rc = SMC_ECUDA;
    }
    return rc;
}

namespace {

// enqueue the whole batch evaluation on st (syntheses, counter resets, persistent launches); forks: st is captured
int enqueue(Batch* b, const int* level, const int* n, const double* const* theta, Forks* forks, cudaStream_t st) {
    std::vector<SynthReq> reqs;
    for (size_t p = 0; p < b->h.size(); ++p)
        if (n[p] > 0 && b->h[p]->precision == SMC_MIXED) reqs.push_back({b->h[p], level[p], n[p], theta[p]});
    const int rc = synth_many(reqs, forks, st, &b->last_error);
    if (rc != SMC_OK) return rc;
    cudaError_t e = cudaMemsetAsync(b->d_counters, 0, sizeof(int) * b->groups.size(), st);
    for (size_t g = 0; g < b->groups.size() && e == cudaSuccess; ++g) {
        const auto& G = b->groups[g];
        if (fem_tile_form(G.N, G.precision, false))   // the form single solves default to
            e = fem_tile_multi_launch(G.N, G.d_args, G.d_offsets, G.d_item_group, G.total, b->big_scratch,
                                      b->d_counters + g, st);
        else if (G.N >= 128)
            e = fem_eval_global_multi_launch(G.N, G.d_args, G.d_offsets, G.d_item_group, G.total, b->big_scratch,
                                             fem_global_blocks(G.N), b->d_counters + g, st);
        else
            e = fem_eval_persistent_launch(G.N, G.precision, G.T, G.d_args, G.d_offsets, G.d_item_group, G.total,
                                           b->d_counters + g, st);
    }
    return e == cudaSuccess ? SMC_OK : SMC_ECUDA;
}

}  // namespace

}  // namespace mls2mc

using namespace mls2mc;

extern "C" {

int smc_batch_create(int n, smc_handle* const* handles, smc_batch** out) {
    if (!out || n < 1 || !handles) return SMC_EINVAL;
    *out = nullptr;
    Batch* b = new Batch();
    for (int i = 0; i < n; ++i) {
        Handle* h = reinterpret_cast<Handle*>(handles[i]);
        // the persistent multi-problem forms solve the Dirichlet problem only
        if (!h || h->forward_kind != SMC_FWD_FEM || h->flow_cell ||
            std::find(b->h.begin(), b->h.end(), h) != b->h.end()) {
            delete b;
            return SMC_EINVAL;
        }
        b->h.push_back(h);
    }
    *out = reinterpret_cast<smc_batch*>(b);
    return SMC_OK;
}

void smc_batch_destroy(smc_batch* bb) { delete reinterpret_cast<Batch*>(bb); }

const char* smc_batch_last_error(const smc_batch* bb) {
    return bb ? reinterpret_cast<const Batch*>(bb)->last_error.c_str() : "null batch";
}

int smc_batch_eval(smc_batch* bb, const int* level, const int* n, const double* const* theta, double* const* phi,
                   int* const* iters, void* stream, int use_graph) {
    if (!bb || !level || !n || !theta || !phi) return SMC_EINVAL;
    Batch* b = reinterpret_cast<Batch*>(bb);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (use_graph && !st) {
        b->last_error = "graph capture needs a non-default stream";
        return SMC_EINVAL;
    }
    const size_t P = b->h.size();
    std::vector<long long> sig;
    for (size_t p = 0; p < P; ++p) {
        Handle* h = b->h[p];
        if (level[p] < 0 || level[p] >= (int)h->levels.size() || n[p] < 0 || (n[p] > 0 && (!theta[p] || !phi[p]))) {
            b->last_error = "bad level, count or pointer for problem " + std::to_string(p);
            return SMC_EINVAL;
        }
        sig.insert(sig.end(), {(long long)level[p], (long long)n[p], (long long)(uintptr_t)theta[p],
                               (long long)(uintptr_t)phi[p], (long long)(uintptr_t)(iters ? iters[p] : nullptr)});
    }
    if (sig != b->signature) {
        b->free_groups();
        // one eager pass per problem first, so every buffer the syntheses need exists before capture
        for (size_t p = 0; p < P; ++p) {
            Handle* h = b->h[p];
            if (n[p] <= 0) continue;
            int rc = h->ensure_scratch(n[p]);
            if (rc == SMC_OK && h->precision == SMC_MIXED) rc = h->synth_kappa(level[p], n[p], theta[p], st);
            if (rc != SMC_OK) {
                b->last_error = h->last_error;
                return rc;
            }
        }
        std::map<std::pair<int, int>, size_t> gidx;
        for (size_t p = 0; p < P; ++p) {
            Handle* h = b->h[p];
            if (n[p] <= 0) continue;
            const Level& L = h->levels[level[p]];
            auto key = std::make_pair(L.N, h->precision);
            if (!gidx.count(key)) {
                gidx[key] = b->groups.size();
                Batch::Group G;
                G.N = L.N;
                G.precision = h->precision;
                G.T = h->block_size(L.N);
                b->groups.push_back(G);
            }
            Batch::Group& G = b->groups[gidx[key]];
            FemArgs a = h->fem_args(level[p], n[p], theta[p], nullptr, phi[p], iters ? iters[p] : h->scratch_iters);
            a.kappa = h->precision == SMC_MIXED ? h->synth_kappa_buf : nullptr;
            G.offsets.push_back(G.total);
            G.args.push_back(a);
            G.total += n[p];
        }
        cudaError_t e = cudaMalloc((void**)&b->d_counters, sizeof(int) * std::max<size_t>(1, b->groups.size()));
        size_t big_need = 0;   // one scratch for all groups: they run one after another
        for (auto& G : b->groups) big_need = std::max(big_need, fem_multi_scratch(G.N, G.precision));
        if (e == cudaSuccess && big_need) e = cudaMalloc((void**)&b->big_scratch, big_need * sizeof(float));
        for (auto& G : b->groups) {
            if (e == cudaSuccess) e = cudaMalloc((void**)&G.d_args, sizeof(FemArgs) * G.args.size());
            if (e == cudaSuccess) e = cudaMalloc((void**)&G.d_offsets, sizeof(int) * G.offsets.size());
            if (e == cudaSuccess)
                e = cudaMemcpy(G.d_args, G.args.data(), sizeof(FemArgs) * G.args.size(), cudaMemcpyHostToDevice);
            if (e == cudaSuccess)
                e = cudaMemcpy(G.d_offsets, G.offsets.data(), sizeof(int) * G.offsets.size(), cudaMemcpyHostToDevice);
            std::vector<int> ig((size_t)std::max(G.total, 1), 0);
            for (size_t q = 0; q < G.offsets.size(); ++q) {
                const int end = q + 1 < G.offsets.size() ? G.offsets[q + 1] : G.total;
                for (int i = G.offsets[q]; i < end; ++i) ig[(size_t)i] = (int)q;
            }
            if (e == cudaSuccess) e = cudaMalloc((void**)&G.d_item_group, sizeof(int) * ig.size());
            if (e == cudaSuccess)
                e = cudaMemcpy(G.d_item_group, ig.data(), sizeof(int) * ig.size(), cudaMemcpyHostToDevice);
        }
        if (e != cudaSuccess) {
            b->last_error = cudaGetErrorString(e);
            b->free_groups();
            return SMC_ENOMEM;
        }
        b->signature = sig;
    }
    if (!use_graph) return enqueue(b, level, n, theta, nullptr, st);
    if (!b->exec) {
        const long long k0 = launch_count();
        Forks* forks = b->forks.ready() ? &b->forks : nullptr;
        cudaError_t e = cudaStreamBeginCapture(st, cudaStreamCaptureModeRelaxed);
        if (e != cudaSuccess) {
            b->last_error = cudaGetErrorString(e);
            return SMC_ECUDA;
        }
        const int rc = enqueue(b, level, n, theta, forks, st);
        e = cudaStreamEndCapture(st, &b->graph);
        if (rc != SMC_OK || e != cudaSuccess) {
            b->last_error = "graph capture failed";
            if (b->graph) cudaGraphDestroy(b->graph);
            b->graph = nullptr;
            return rc != SMC_OK ? rc : SMC_ECUDA;
        }
        e = cudaGraphInstantiate(&b->exec, b->graph, 0);
        if (e != cudaSuccess) {
            b->last_error = cudaGetErrorString(e);
            return SMC_ECUDA;
        }
        b->graph_kernels = launch_count() - k0;
        count_launches(-b->graph_kernels);   // counted when the graph runs, not when it is captured
    }
    cudaError_t e = cudaGraphLaunch(b->exec, st);
    if (e != cudaSuccess) {
        b->last_error = cudaGetErrorString(e);
        return SMC_ECUDA;
    }
    count_launches(b->graph_kernels);
    return SMC_OK;
}

}  // extern "C"
