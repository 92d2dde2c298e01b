// Internal entry points of the join algorithms (device-resident columns).
#pragma once

#include <memory>
#include <vector>

#include "jn_common.cuh"

namespace jnx {

enum RunMode { MODE_COUNT = 0, MODE_AGG = 1, MODE_EMIT = 2 };

// One table with every column already in device memory.
template <typename K>
struct Cols {
    const K* key;
    const K* key2;
    const int32_t* pay;  // NULL = row index
    int64_t n;
    bool host = false;   // columns read in place from page-locked host memory
};

// Where the pairs of an emitting run go (see jn.h's output convention).
struct OutPlan {
    jn_pair** user_out = nullptr;
    uint64_t capacity = 0;
    uint64_t* n_out = nullptr;
    jn_pair* dev = nullptr;      // device buffer the kernels write
    bool host_copy = false;      // caller buffer is host memory, filled by a copy
    bool lib_alloc = false;      // library allocated the result
    bool mapped = false;         // caller buffer is page-locked host memory written in place
    bool copied = false;         // the run already copied the pairs to the caller's host buffer
    bool admitted = false;       // the limit and the hook have let the run pass: they are asked once
    bool no_memory = false;      // the output's allocation failed
};

// Sizes the output for `m` pairs (allocating or checking the caller buffer).
jn_status out_prepare(jn_ctx* c, Scratch& s, uint64_t m, OutPlan& plan);
// The same for a run that keeps its pairs in scratch: where the output finds no
// memory beside them, give_up() releases them (true: it had some) and the
// allocation is tried once more; the run then writes its pairs in a second pass.
template <typename F>
jn_status out_prepare_or(jn_ctx* c, Scratch& s, uint64_t m, OutPlan& plan, F give_up) {
    const jn_status st = out_prepare(c, s, m, plan);
    if (st != JN_ERR_OOM || !plan.no_memory || !give_up()) return st;
    c->err.clear();
    JN_CUDA(c, cudaStreamSynchronize(c->stream));  // the released memory can take another shape
    return out_prepare(c, s, m, plan);
}
// Copies to a host buffer when needed and publishes the result.
jn_status out_finish(jn_ctx* c, uint64_t m, OutPlan& plan);

struct RunResult {
    uint64_t count = 0;
    uint64_t checksum = 0;
};

// R rows one hash-join work item holds in shared memory, by key type.
int hash_cap(int32_t key_type);

template <typename K>
jn_status run_hash(jn_ctx* c, const Cols<K>& R, const Cols<K>& S, int mode, OutPlan* plan,
                   RunResult* res, bool sort_merge = false);

// The direct join (jn_direct.cuh), when it suits the tables and the tuning:
// *taken false = nothing was done, the partitioned join is to run (*repeats:
// because the build keys have several rows).
template <typename K>
jn_status run_direct(jn_ctx* c, const Cols<K>& R, const Cols<K>& S, int mode, OutPlan* plan, RunResult* res,
                     bool* taken, bool* repeats);

// A batch of joins run as one: prepare() (all passes up to the exact
// counts) fills total and the per-join offsets; emit() writes the pairs to
// out[0 .. total).  The object owns the batch's scratch between the two.
struct BatchRun {
    uint64_t total = 0;
    std::vector<uint64_t> offsets;  // joins + 1 offsets inside this run's pairs
    virtual ~BatchRun() {}
    virtual jn_status emit(jn_ctx* c, jn_pair* out) = 0;
};

template <typename K>
jn_status batch_hash_prepare(jn_ctx* c, int n, const Cols<K>* Rs, const Cols<K>* Ss, std::unique_ptr<BatchRun>* run);

// The same without partitioning (jn_direct.cuh), for the joins it takes;
// count_only: the run is never asked to emit.  *run stays empty where the
// partitioned batch is the better one.
bool batch_direct_takes(const jn_ctx* c, int64_t nr, int64_t ns);
template <typename K>
jn_status batch_direct_prepare(jn_ctx* c, int n, const Cols<K>* Rs, const Cols<K>* Ss, bool count_only,
                               std::unique_ptr<BatchRun>* run);

template <typename K>
jn_status batch_band_prepare(jn_ctx* c, int m, const Cols<K>* Rs, const Cols<K>* Ss, const int* ops,
                             const int64_t* bands, std::unique_ptr<BatchRun>* run);

// Band joins without partitioning (k_band.cu), for the joins it takes.  A
// join that turns out to have too many candidates is `stopped`: it has no
// pairs here and is left to the partitioned join.  JN_ERR_OOM: nothing ran.
struct BandDirect : BatchRun {
    std::vector<char> stopped;
    uint64_t checksum = 0;    // aggregate
    uint64_t candidates = 0;  // rows compared
    uint64_t buckets = 0, tiles = 0;
};
bool band_direct_takes(const jn_ctx* c, int64_t nr, int64_t ns);
template <typename K>
jn_status band_direct_prepare(jn_ctx* c, int n, const Cols<K>* Rs, const Cols<K>* Ss, const int* ops,
                              const int64_t* bands, int mode, std::unique_ptr<BandDirect>* run);

// Captures a sequence of launches on the context's private stream and replays
// it as a CUDA graph on the context's stream (or runs it directly when graphs
// are off).  The caller's stream may be the legacy default stream, which
// cannot itself be captured.
struct GraphPhase {
    jn_ctx* c;
    bool on;
    cudaStream_t user = nullptr;
    cudaGraph_t g = nullptr;
    cudaGraphExec_t x = nullptr;
    GraphPhase(jn_ctx* ctx, bool graphs) : c(ctx), on(graphs) {}
    ~GraphPhase();
    jn_status begin();
    jn_status end_and_run();
    void abort();
};

template <typename K>
jn_status run_nlj(jn_ctx* c, const Cols<K>& R, const Cols<K>& S, const jn_pred& pred, int mode,
                  OutPlan* plan, RunResult* res);

template <typename K>
jn_status run_theta(jn_ctx* c, const Cols<K>& R, const Cols<K>& S, int op, int64_t band, int mode,
                    OutPlan* plan, RunResult* res);

}  // namespace jnx
