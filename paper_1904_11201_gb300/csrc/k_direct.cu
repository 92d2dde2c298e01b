// Direct equi join of two tables (jn_direct.cuh): build on the smaller one,
// probe with the other, one pass that counts and writes the pairs to scratch,
// the exact output allocation, one copy.
#include <algorithm>

#include "jn_direct.cuh"

namespace jnx {

// Pairs past which an emitting run is left to the partitioned join: many
// times the rows, so frequent keys carry it, whose cross products that join
// writes as dense tiles spread over the whole device.
static uint64_t direct_most_pairs(uint64_t rows) { return 8 * rows + (1u << 20); }

template <typename K, int MODE>
static jn_status direct_mode(jn_ctx* c, const Cols<K>& R, const Cols<K>& S, OutPlan* plan, RunResult* res,
                             bool* taken) {
    const bool swap = S.n < R.n;
    const Cols<K>&B = swap ? S : R, &P = swap ? R : S;
    const uint64_t nb = (uint64_t)B.n, np = (uint64_t)P.n;
    const DirectLayout<K, MODE> lay(nb);
    const size_t head = sizeof(DirectSmall);
    static_assert(sizeof(DirectSmall) % 32 == 0, "buckets follow the counters, 32-byte aligned");
    const DirectStage sg(np);
    uint32_t segs = MODE == MODE_EMIT ? sg.segs : 1;
    uint64_t cap = MODE == MODE_EMIT ? sg.cap : 0;
    if (c->mem_limit || c->admit) {
        // a run admitted by its bytes holds no more scratch here than the
        // partitioned join would (two copies of the rows of both tables)
        const uint64_t most = 2 * (sizeof(K) == 4 ? 8 : 16) * (nb + np);
        if (head + lay.bytes() + segs * cap * sizeof(jn_pair) > most) cap = 0;
        if (head + lay.bytes() > most) return JN_OK;
    }
    Scratch s(c);
    unsigned char* mem = nullptr;
    jn_pair* staged = nullptr;
    if (s.get(&mem, head + lay.bytes()) != JN_OK) {
        c->err.clear();  // a device too full for the table takes the partitioned path
        return JN_OK;
    }
    Scratch ss(c);
    if (cap && ss.get(&staged, segs * cap) != JN_OK) {
        c->err.clear();
        cap = 0;
    }
    DirectSmall* small = reinterpret_cast<DirectSmall*>(mem);
    JN_TRY(zero(c, mem, head + lay.zeroed()));
    DirectTab<K, MODE> t;
    JN_TRY(wait_copies(c, true));
    JN_TRY((direct_build<K, MODE>(c, B, swap ? 1 : 0, lay, mem + head, small, &t)));
    auto kp = k_direct_probe<K, MODE>;
    int per = 0;
    JN_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kp, DJ_T, 0));
    const uint64_t tiles = ceil_div(np, DJ_T * DJ_U);
    const dim3 g((unsigned)std::min<uint64_t>(tiles, (uint64_t)std::max(per, 1) * c->num_sms));
    JN_TRY(launch(c, K_DIRECT_PROBE, kp, g, dim3(DJ_T), 0, P.key, P.pay, P.n, t, swap ? 1 : 0, small, staged, segs,
                  (unsigned long long)cap));
    DirectResult r;
    JN_TRY(direct_result(c, small, segs, cap, &r));
    const uint64_t total = r.total;
    const bool done = r.fits;
    if (MODE == MODE_EMIT && !done && total > direct_most_pairs(nb + np)) return JN_OK;
    *taken = true;
    jn_run_info& info = c->info;
    res->count = total;
    res->checksum = r.chk;
    info.result = total;
    info.r_survivors = (uint64_t)R.n;
    info.s_survivors = (uint64_t)S.n;
    info.partitions = 1;
    info.work_items = tiles;
    info.hash_path = 3;
    info.cartesian_bound = nb * np;
    if (MODE != MODE_EMIT) return JN_OK;
    // a table no longer needed, or the scratch the pairs did not fit
    (done ? s : ss).release();
    JN_TRY(out_prepare(c, ss, total, *plan));
    if (total && done && plan->host_copy && segs == 1) {
        // straight to the caller's buffer
        JN_CUDA(c, cudaMemcpyAsync(*plan->user_out, staged, total * sizeof(jn_pair), cudaMemcpyDefault, c->stream));
        plan->copied = true;
    } else if (total && done) {
        JN_TRY((direct_gather<uint64_t, 1>(c, K_DIRECT_PROBE, staged, segs, cap, r, plan->dev)));
    } else if (total) {
        JN_TRY(zero(c, &small->lines[0].total, 8));
        JN_TRY(launch(c, K_DIRECT_PROBE, kp, g, dim3(DJ_T), 0, P.key, P.pay, P.n, t, swap ? 1 : 0, small, plan->dev,
                      1u, (unsigned long long)total));
        JN_CUDA(c, cudaStreamSynchronize(c->stream));  // this pass reads the caller's columns
    }
    return out_finish(c, total, *plan);
}

template <typename K>
jn_status run_direct(jn_ctx* c, const Cols<K>& R, const Cols<K>& S, int mode, OutPlan* plan, RunResult* res,
                     bool* taken) {
    *taken = false;
    const uint64_t nb = (uint64_t)std::min(R.n, S.n);
    if (nb == 0 || nb > DJ_MAX || !direct_allowed(c) || R.host || S.host) return JN_OK;
    if (mode == MODE_EMIT) return direct_mode<K, MODE_EMIT>(c, R, S, plan, res, taken);
    if (mode == MODE_AGG) return direct_mode<K, MODE_AGG>(c, R, S, plan, res, taken);
    return direct_mode<K, MODE_COUNT>(c, R, S, plan, res, taken);
}

template jn_status run_direct<int32_t>(jn_ctx*, const Cols<int32_t>&, const Cols<int32_t>&, int, OutPlan*, RunResult*,
                                       bool*);
template jn_status run_direct<int64_t>(jn_ctx*, const Cols<int64_t>&, const Cols<int64_t>&, int, OutPlan*, RunResult*,
                                       bool*);

}  // namespace jnx
