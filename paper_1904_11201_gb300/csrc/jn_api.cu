// extern "C" entry points of libjn: argument checks, host-column staging,
// dispatch on key type, and the output convention of jn.h.
#include <string.h>

#include <vector>

#include "jn_algos.h"

namespace jnx {

// Admission by exact bytes: the count is known, nothing is allocated yet.
static jn_status admit(jn_ctx* c, uint64_t m, uint64_t out_bytes, OutPlan& plan) {
    if (c->mem_limit && out_bytes + c->scratch_bytes > c->mem_limit) {
        *plan.n_out = m;
        return fail(c, JN_ERR_OOM, "the exact result and the scratch held exceed the memory limit");
    }
    if (c->admit) {
        const jn_status st = c->admit(c->admit_user, out_bytes, c->scratch_bytes);
        if (st != JN_OK) {
            *plan.n_out = m;
            return fail(c, st, "the admission hook refused the run");
        }
    }
    return JN_OK;
}

jn_status out_prepare(jn_ctx* c, Scratch& s, uint64_t m, OutPlan& plan) {
    jn_pair* user = *plan.user_out;
    plan.host_copy = false;
    plan.lib_alloc = false;
    const jn_pair* mapped =
        user && (c->tune.host_io & 2) ? static_cast<const jn_pair*>(host_mapped(user)) : nullptr;
    plan.no_memory = false;
    if (!plan.admitted) {
        const bool dev_out =
            user != nullptr && (m == 0 || m > plan.capacity || mapped || is_device_pointer(user));
        JN_TRY(admit(c, m, dev_out ? 0 : m * sizeof(jn_pair), plan));
        plan.admitted = true;
    }
    if (user == nullptr) {
        plan.lib_alloc = true;
        plan.dev = nullptr;
        if (m > 0) {
            void* p = nullptr;
            const jn_status st = dalloc(c, &p, m * sizeof(jn_pair));
            plan.no_memory = st == JN_ERR_OOM;
            if (st != JN_OK) return st;
            plan.dev = static_cast<jn_pair*>(p);
        }
        return JN_OK;
    }
    if (m > plan.capacity) {
        *plan.n_out = m;
        return fail(c, JN_ERR_CAPACITY, "output buffer holds fewer pairs than the result");
    }
    // the kernels store a pair as one 8-byte word: a caller buffer off an
    // 8-byte boundary is filled by a copy from an aligned scratch buffer
    const bool aligned = ((uintptr_t)user & 7) == 0;
    if (m == 0 || (aligned && is_device_pointer(user))) {
        plan.dev = user;
        return JN_OK;
    }
    if (mapped && aligned) {  // page-locked host memory: the kernels write the pairs in place
        plan.dev = const_cast<jn_pair*>(mapped);
        plan.mapped = true;
        return JN_OK;
    }
    plan.host_copy = true;
    const jn_status st = s.get(&plan.dev, m);
    plan.no_memory = st == JN_ERR_OOM;
    return st;
}

jn_status out_finish(jn_ctx* c, uint64_t m, OutPlan& plan) {
    if (plan.mapped && m > 0) JN_CUDA(c, cudaStreamSynchronize(c->stream));  // pairs visible to the host
    if (plan.host_copy && m > 0) {
        if (!plan.copied)
            JN_CUDA(c, cudaMemcpyAsync(*plan.user_out, plan.dev, m * sizeof(jn_pair), cudaMemcpyDefault,
                                       c->stream));
        JN_CUDA(c, cudaStreamSynchronize(c->stream));
    }
    if (plan.lib_alloc) *plan.user_out = plan.dev;
    *plan.n_out = m;
    return JN_OK;
}

static jn_status check_table(jn_ctx* c, const jn_table* t, const char* name, bool need_key2) {
    if (!t) return fail(c, JN_ERR_INVALID, std::string(name) + ": NULL table");
    if (t->key_type != JN_KEY_I32 && t->key_type != JN_KEY_I64)
        return fail(c, JN_ERR_INVALID, std::string(name) + ": key_type must be JN_KEY_I32 or JN_KEY_I64");
    if (t->n < 0 || t->n > INT32_MAX)
        return fail(c, JN_ERR_INVALID, std::string(name) + ": row count out of range");
    if (t->reserved != 0) return fail(c, JN_ERR_INVALID, std::string(name) + ": reserved must be 0");
    if (t->n > 0 && t->key == nullptr) return fail(c, JN_ERR_INVALID, std::string(name) + ": NULL key");
    if (need_key2 && t->n > 0 && t->key2 == nullptr)
        return fail(c, JN_ERR_INVALID, std::string(name) + ": key2 required");
    return JN_OK;
}

static bool valid_op(int op) { return op >= JN_EQ && op <= JN_ANY; }

// Host columns of one run: device scratch for each, filled on the copy
// stream (key columns first, then second columns and payloads), with one
// event when the keys have landed and one when everything has.
struct HostCopies {
    jn_ctx* c;
    struct Job {
        void* dst;
        const void* src;
        size_t bytes;
        bool key;
        bool first;  // a column of the first table staged
    };
    std::vector<Job> jobs;
    bool first_table = true;  // stage() calls of the first table come first
    explicit HostCopies(jn_ctx* ctx) : c(ctx) {}
    ~HostCopies() {
        // the run's stream-ordered frees of the scratch come after every copy
        if (c->copied_all) cudaStreamWaitEvent(c->stream, c->copied_all, 0);
        if (c->copied_keys) cudaEventDestroy(c->copied_keys);
        if (c->copied_r) cudaEventDestroy(c->copied_r);
        if (c->copied_all) cudaEventDestroy(c->copied_all);
        c->copied_keys = c->copied_r = c->copied_all = nullptr;
    }
    // a device column as it is, or scratch that a later copy fills
    jn_status column(Scratch& s, const void* p, size_t bytes, bool key, const void** dp) {
        if (p == nullptr || bytes == 0 || is_device_pointer(p)) {
            *dp = p;
            return JN_OK;
        }
        uint8_t* d = nullptr;
        JN_TRY(s.get(&d, bytes));
        jobs.push_back(Job{d, p, bytes, key, first_table});
        *dp = d;
        return JN_OK;
    }
    jn_status start() {
        if (jobs.empty()) return JN_OK;
        if (!c->copy_stream) JN_CUDA(c, cudaStreamCreateWithFlags(&c->copy_stream, cudaStreamNonBlocking));
        cudaEvent_t ready;  // the scratch allocations (stream-ordered on the run's stream) come first
        JN_CUDA(c, cudaEventCreateWithFlags(&ready, cudaEventDisableTiming));
        cudaEventRecord(ready, c->stream);
        cudaStreamWaitEvent(c->copy_stream, ready, 0);
        cudaEventDestroy(ready);
        JN_CUDA(c, cudaEventCreateWithFlags(&c->copied_keys, cudaEventDisableTiming));
        JN_CUDA(c, cudaEventCreateWithFlags(&c->copied_r, cudaEventDisableTiming));
        JN_CUDA(c, cudaEventCreateWithFlags(&c->copied_all, cudaEventDisableTiming));
        // keys of both tables, then the rest of the first table, then the rest
        cudaEvent_t marks[3] = {c->copied_keys, c->copied_r, c->copied_all};
        for (int pass = 0; pass < 3; pass++) {
            for (const Job& j : jobs)
                if (pass == 0 ? j.key : (!j.key && j.first == (pass == 1)))
                    JN_CUDA(c, cudaMemcpyAsync(j.dst, j.src, j.bytes, cudaMemcpyHostToDevice, c->copy_stream));
            JN_CUDA(c, cudaEventRecord(marks[pass], c->copy_stream));
        }
        return JN_OK;
    }
};

template <typename K>
static jn_status stage(jn_ctx* c, Scratch& s, HostCopies& hc, const jn_table* t, bool use_key2, Cols<K>* out,
                       bool in_place = false) {
    const size_t kb = (size_t)t->n * sizeof(K);
    const void *k = nullptr, *k2 = nullptr, *p = nullptr;
    // a path that reads each column in a couple of streaming passes reads
    // page-locked host columns in place instead of copying them first
    const void* mk = in_place ? host_mapped(t->key) : nullptr;
    const void* mp = in_place && t->payload ? host_mapped(t->payload) : nullptr;
    out->host = mk && (mp || !t->payload) && !(use_key2 && t->key2);
    if (out->host) {
        k = mk;
        p = mp;
    } else {
        JN_TRY(hc.column(s, t->key, kb, true, &k));
        if (use_key2 && t->key2) JN_TRY(hc.column(s, t->key2, kb, false, &k2));
        if (t->payload) JN_TRY(hc.column(s, t->payload, (size_t)t->n * 4, false, &p));
    }
    out->key = static_cast<const K*>(k);
    out->key2 = static_cast<const K*>(k2);
    out->pay = static_cast<const int32_t*>(p);
    out->n = t->n;
    return JN_OK;
}

template <typename K>
static jn_status dispatch(jn_ctx* c, int algo, const jn_table* R, const jn_table* S, const jn_pred& pr,
                          int mode, OutPlan* plan, RunResult* res) {
    Scratch s(c);
    HostCopies hc(c);
    Cols<K> r, q;
    const bool equi = algo == JN_ALGO_HASH || algo == JN_ALGO_SORT;
    const bool use2 = !equi;
    // the equi joins sample a column, then read it in two streaming passes
    const bool in_place = equi && (c->tune.host_io & 1);
    JN_TRY(stage<K>(c, s, hc, R, use2, &r, in_place));
    hc.first_table = false;
    JN_TRY(stage<K>(c, s, hc, S, use2, &q, in_place));
    JN_TRY(hc.start());
    if (!equi) JN_TRY(wait_copies(c, true));  // the equi joins wait per phase
    switch (algo) {
        case JN_ALGO_HASH: return run_hash<K>(c, r, q, mode, plan, res);
        case JN_ALGO_SORT: return run_hash<K>(c, r, q, mode, plan, res, true);
        case JN_ALGO_NLJ: return run_nlj<K>(c, r, q, pr, mode, plan, res);
        case JN_ALGO_THETA: return run_theta<K>(c, r, q, pr.op_a, pr.band, mode, plan, res);
    }
    return fail(c, JN_ERR_INVALID, "unknown algorithm");
}

static jn_status run(jn_ctx* c, int algo, const jn_table* R, const jn_table* S, const jn_pred* pred,
                     int mode, jn_pair** out, uint64_t capacity, uint64_t* n_out, uint64_t* count,
                     uint64_t* checksum) {
    if (!c) return JN_ERR_INVALID;
    c->err.clear();
    jn_pred pr;
    pr.op_a = JN_EQ;
    pr.op_k = JN_ANY;
    pr.band = -1;
    if (pred) pr = *pred;
    if (!valid_op(pr.op_a) || !valid_op(pr.op_k)) return fail(c, JN_ERR_INVALID, "unknown predicate op");
    if (algo == JN_ALGO_HASH || algo == JN_ALGO_SORT) {
        const bool second = pred && (pr.band >= 0 || pr.op_k != JN_ANY);
        if (pr.op_a != JN_EQ || second)
            return fail(c, JN_ERR_UNSUPPORTED, "the hash and sort-merge joins take the equality predicate only");
    }
    const bool need2 = algo == JN_ALGO_THETA && pr.band >= 0;
    JN_TRY(check_table(c, R, "R", need2));
    JN_TRY(check_table(c, S, "S", need2));
    if (R->key_type != S->key_type) return fail(c, JN_ERR_INVALID, "R and S key types differ");
    if (mode == MODE_EMIT && (!out || !n_out)) return fail(c, JN_ERR_INVALID, "NULL output pointer");
    if (mode != MODE_EMIT && !count) return fail(c, JN_ERR_INVALID, "NULL count pointer");
    JN_CUDA(c, cudaSetDevice(c->device));
    c->info = jn_run_info();
    const uint64_t l0 = c->launches_total;
    OutPlan plan;
    plan.user_out = out;
    plan.capacity = capacity;
    plan.n_out = n_out;
    RunResult res;
    jn_status st = (R->key_type == JN_KEY_I32)
                       ? dispatch<int32_t>(c, algo, R, S, pr, mode, &plan, &res)
                       : dispatch<int64_t>(c, algo, R, S, pr, mode, &plan, &res);
    c->info.kernel_launches = c->launches_total - l0;
    if (st != JN_OK) return st;
    if (count) *count = res.count;
    if (checksum) *checksum = res.checksum;
    return JN_OK;
}

// direct: joins may run without partitioning; *direct then tells whether one did.
template <typename K>
static jn_status batch_parts(jn_ctx* c, int count, const jn_join* joins, jn_pair** out, uint64_t capacity,
                             uint64_t* n_out, uint64_t* first, uint64_t* pairs, bool count_only, bool* direct) {
    Scratch s(c);
    // the batch's parts: equi-joins with a table small enough to stay in L2
    // and the others, band joins likewise; each part runs as one
    constexpr int PARTS = 4;
    std::vector<int> part[PARTS];
    for (int i = 0; i < count; i++) {
        const int64_t nr = joins[i].R.n, ns = joins[i].S.n;
        part[joins[i].band >= 0 ? (*direct && band_direct_takes(c, nr, ns) ? 2 : 3)
                                : *direct && batch_direct_takes(c, nr, ns) ? 0 : 1]
            .push_back(i);
    }
    *direct = !part[0].empty() || !part[2].empty();
    std::vector<Cols<K>> cr[PARTS], cs[PARTS];
    std::vector<int> bops[PARTS];
    std::vector<int64_t> bbands[PARTS];
    HostCopies hc(c);
    for (int k = 0; k < PARTS; k++) {
        cr[k].resize(part[k].size());
        cs[k].resize(part[k].size());
        for (size_t j = 0; j < part[k].size(); j++) {
            const jn_join& x = joins[part[k][j]];
            JN_TRY(stage<K>(c, s, hc, &x.R, k >= 2, &cr[k][j]));
            JN_TRY(stage<K>(c, s, hc, &x.S, k >= 2, &cs[k][j]));
            bops[k].push_back(x.op);
            bbands[k].push_back(x.band);
        }
    }
    JN_TRY(hc.start());
    JN_TRY(wait_copies(c, true));
    // every join is counted before the single output allocation
    std::unique_ptr<BatchRun> run[PARTS];
    auto move_join = [&](int from, int to, size_t j) {
        part[to].push_back(part[from][j]);
        cr[to].push_back(cr[from][j]);
        cs[to].push_back(cs[from][j]);
        bops[to].push_back(bops[from][j]);
        bbands[to].push_back(bbands[from][j]);
    };
    if (!part[0].empty()) {
        const jn_status st =
            batch_direct_prepare<K>(c, (int)part[0].size(), cr[0].data(), cs[0].data(), count_only, &run[0]);
        if (st == JN_ERR_OOM || (st == JN_OK && !run[0])) {
            // a device too full for the tables and the pairs' room, or joins
            // that run better so: all of them partitioned
            c->err.clear();
            for (size_t j = 0; j < part[0].size(); j++) move_join(0, 1, j);
            part[0].clear();
        } else if (st != JN_OK) {
            return st;
        }
    }
    if (!part[1].empty())
        JN_TRY(batch_hash_prepare<K>(c, (int)part[1].size(), cr[1].data(), cs[1].data(), &run[1]));
    std::vector<char> moved(part[2].size(), 0);  // band joins left to the partitioned join
    if (!part[2].empty()) {
        std::unique_ptr<BandDirect> direct;
        const jn_status st =
            band_direct_prepare<K>(c, (int)part[2].size(), cr[2].data(), cs[2].data(), bops[2].data(),
                                   bbands[2].data(), count_only ? MODE_COUNT : MODE_EMIT, &direct);
        if (st != JN_OK && st != JN_ERR_OOM) return st;
        c->err.clear();
        if (st == JN_OK) {
            moved = direct->stopped;
            c->info.partitions += direct->buckets;
            c->info.work_items += direct->tiles;
            run[2] = std::move(direct);
        } else {
            moved.assign(part[2].size(), 1);
        }
        for (size_t j = 0; j < part[2].size(); j++)
            if (moved[j]) move_join(2, 3, j);
    }
    if (!part[3].empty())
        JN_TRY(batch_band_prepare<K>(c, (int)part[3].size(), cr[3].data(), cs[3].data(), bops[3].data(),
                                     bbands[3].data(), &run[3]));
    uint64_t total = 0;
    for (int k = 0; k < PARTS; k++) total += run[k] ? run[k]->total : 0;
    auto publish = [&] {
        uint64_t at = 0;
        for (int k = 0; k < PARTS; k++) {
            for (size_t j = 0; j < part[k].size(); j++) {
                if (k == 2 && moved[j]) continue;
                first[part[k][j]] = at + run[k]->offsets[j];
                pairs[part[k][j]] = run[k]->offsets[j + 1] - run[k]->offsets[j];
            }
            at += run[k] ? run[k]->total : 0;
        }
    };
    if (count_only) {
        publish();
        *n_out = total;
        c->info.result = total;
        return JN_OK;
    }
    OutPlan plan;
    plan.user_out = out;
    plan.capacity = capacity;
    plan.n_out = n_out;
    JN_TRY(out_prepare(c, s, total, plan));
    if (plan.host_copy && !is_device_pointer(*out))
        return fail(c, JN_ERR_INVALID, "batch outputs must be device memory");
    uint64_t at = 0;
    for (int k = 0; k < PARTS; k++) {
        if (!run[k]) continue;
        const jn_status st = run[k]->emit(c, plan.dev + at);
        if (st != JN_OK) {
            if (plan.lib_alloc) dfree(c, plan.dev);
            return st;
        }
        at += run[k]->total;
    }
    publish();
    JN_TRY(out_finish(c, total, plan));
    uint64_t dummy;
    uint64_t* d_small;
    JN_TRY(s.get(&d_small, 1));
    JN_TRY(read_back(c, d_small, &dummy, 0));  // reports a device wait that ran out
    c->info.result = total;
    return JN_OK;
}

template <typename K>
static jn_status batch_typed(jn_ctx* c, int count, const jn_join* joins, jn_pair** out, uint64_t capacity,
                             uint64_t* n_out, uint64_t* first, uint64_t* pairs, bool count_only) {
    bool direct = true;
    const jn_status st =
        batch_parts<K>(c, count, joins, out, capacity, n_out, first, pairs, count_only, &direct);
    if (st != JN_ERR_OOM || !direct) return st;
    // tables, indexes and kept pairs left too little of the device for the
    // other joins or the output: every join partitioned, which keeps nothing
    // (direct joins are not taken under a limit or a hook, so neither refused)
    c->err.clear();
    c->info = jn_run_info();
    JN_CUDA(c, cudaStreamSynchronize(c->stream));  // the released memory can take another shape
    direct = false;
    return batch_parts<K>(c, count, joins, out, capacity, n_out, first, pairs, count_only, &direct);
}

}  // namespace jnx

using namespace jnx;

extern "C" {

jn_status jn_count(jn_ctx* ctx, int32_t algo, const jn_table* R, const jn_table* S, const jn_pred* pred,
                   uint64_t* count) {
    return run(ctx, algo, R, S, pred, MODE_COUNT, nullptr, 0, nullptr, count, nullptr);
}

jn_status jn_aggregate(jn_ctx* ctx, int32_t algo, const jn_table* R, const jn_table* S,
                       const jn_pred* pred, uint64_t* count, uint64_t* checksum) {
    return run(ctx, algo, R, S, pred, MODE_AGG, nullptr, 0, nullptr, count, checksum);
}

jn_status jn_nested_loop(jn_ctx* ctx, const jn_table* R, const jn_table* S, const jn_pred* pred,
                         jn_pair** out, uint64_t capacity, uint64_t* n_out) {
    return run(ctx, JN_ALGO_NLJ, R, S, pred, MODE_EMIT, out, capacity, n_out, nullptr, nullptr);
}

jn_status jn_hash(jn_ctx* ctx, const jn_table* R, const jn_table* S, jn_pair** out, uint64_t capacity,
                  uint64_t* n_out) {
    return run(ctx, JN_ALGO_HASH, R, S, nullptr, MODE_EMIT, out, capacity, n_out, nullptr, nullptr);
}

jn_status jn_sort_merge(jn_ctx* ctx, const jn_table* R, const jn_table* S, jn_pair** out, uint64_t capacity,
                        uint64_t* n_out) {
    return run(ctx, JN_ALGO_SORT, R, S, nullptr, MODE_EMIT, out, capacity, n_out, nullptr, nullptr);
}

static jn_status batch_entry(jn_ctx* ctx, int32_t count, const jn_join* joins, jn_pair** out, uint64_t capacity,
                             uint64_t* n_out, uint64_t* first, uint64_t* pairs, bool count_only) {
    if (!ctx) return JN_ERR_INVALID;
    ctx->err.clear();
    if (count < 0 || (count > 0 && (!joins || !first || !pairs)) || !out || !n_out)
        return fail(ctx, JN_ERR_INVALID, "jn_batch: bad arguments");
    if (count == 0) {
        *n_out = 0;
        return JN_OK;
    }
    const int32_t kt = joins[0].R.key_type;
    for (int i = 0; i < count; i++) {
        const jn_join& j = joins[i];
        const bool band = j.band >= 0;
        JN_TRY(check_table(ctx, &j.R, "R", band));
        JN_TRY(check_table(ctx, &j.S, "S", band));
        if (j.R.key_type != kt || j.S.key_type != kt)
            return fail(ctx, JN_ERR_INVALID, "jn_batch: all tables of a batch share one key type");
        if (j.reserved != 0 || !valid_op(j.op)) return fail(ctx, JN_ERR_INVALID, "jn_batch: bad join");
        if (!band && j.op != JN_EQ)
            return fail(ctx, JN_ERR_UNSUPPORTED, "jn_batch: a join without a band must be an equi-join");
    }
    JN_CUDA(ctx, cudaSetDevice(ctx->device));
    ctx->info = jn_run_info();
    const uint64_t l0 = ctx->launches_total;
    jn_status st = kt == JN_KEY_I32
                       ? batch_typed<int32_t>(ctx, count, joins, out, capacity, n_out, first, pairs, count_only)
                       : batch_typed<int64_t>(ctx, count, joins, out, capacity, n_out, first, pairs, count_only);
    ctx->info.kernel_launches = ctx->launches_total - l0;
    return st;
}

jn_status jn_batch(jn_ctx* ctx, int32_t count, const jn_join* joins, jn_pair** out, uint64_t capacity,
                   uint64_t* n_out, uint64_t* first, uint64_t* pairs) {
    return batch_entry(ctx, count, joins, out, capacity, n_out, first, pairs, false);
}

jn_status jn_batch_count(jn_ctx* ctx, int32_t count, const jn_join* joins, uint64_t* pairs, uint64_t* total) {
    if (!ctx) return JN_ERR_INVALID;
    if (count > 0 && !pairs) return fail(ctx, JN_ERR_INVALID, "jn_batch_count: NULL pairs");
    std::vector<uint64_t> first(count > 0 ? count : 1);
    jn_pair* none = nullptr;
    uint64_t n = 0;
    const jn_status st = batch_entry(ctx, count, joins, &none, 0, &n, first.data(), pairs, true);
    if (st == JN_OK && total) *total = n;
    return st;
}

jn_status jn_theta(jn_ctx* ctx, const jn_table* R, const jn_table* S, int32_t op, int64_t band,
                   jn_pair** out, uint64_t capacity, uint64_t* n_out) {
    jn_pred p;
    p.op_a = op;
    p.op_k = JN_ANY;
    p.band = band;
    return run(ctx, JN_ALGO_THETA, R, S, &p, MODE_EMIT, out, capacity, n_out, nullptr, nullptr);
}

}  // extern "C"
