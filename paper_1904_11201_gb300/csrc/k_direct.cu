// Direct equi join of two tables (jn_direct.cuh): build on the smaller one,
// probe with the other, one pass that counts and writes the pairs to scratch,
// the exact output allocation, one copy.
#include <algorithm>
#include <vector>

#include "jn_direct.cuh"
#include "jn_partition.cuh"

namespace jnx {

template <typename K, int MODE>
static jn_status direct_mode(jn_ctx* c, const Cols<K>& R, const Cols<K>& S, OutPlan* plan, RunResult* res,
                             bool* taken, bool* repeats) {
    const bool swap = S.n < R.n;
    const Cols<K>&B = swap ? S : R, &P = swap ? R : S;
    const uint64_t nb = (uint64_t)B.n, np = (uint64_t)P.n;
    const DirectLayout<K, MODE> lay(nb);
    const size_t head = sizeof(DirectSmall);
    static_assert(sizeof(DirectSmall) % 32 == 0, "buckets follow the counters, 32-byte aligned");
    const DirectStage sg(np, DJ_ROOM), less(np, DJ_ROOM_LEAST);
    uint32_t segs = MODE == MODE_EMIT ? sg.segs : 1;
    uint64_t cap = MODE == MODE_EMIT ? sg.cap : 0;
    // kept pairs, and the long runs among them
    auto keep_bytes = [&](uint64_t pairs) { return pairs * sizeof(jn_pair) + (pairs / DJ_LONG + 1) * sizeof(LongRun); };
    if (c->mem_limit || c->admit) {
        // a run admitted by its bytes holds no more scratch here than the
        // partitioned join would (two copies of the rows of both tables)
        const uint64_t most = 2 * (sizeof(K) == 4 ? 8 : 16) * (nb + np);
        if (head + lay.bytes() + keep_bytes(segs * cap) > most) cap = std::min(cap, less.cap);
        if (head + lay.bytes() + keep_bytes(segs * cap) > most) cap = 0;
        if (head + lay.bytes() > most) return JN_OK;
    }
    Scratch s(c);
    unsigned char* mem = nullptr;
    jn_pair* staged = nullptr;
    // Pairs written, 8-byte slots: past 2^21 build rows the table and the runs of
    // repeated keys leave L2, and with two rows a key the partitioned join is the
    // faster one (2^22 x 2^24 rows, two a key: 0.81 ms there, 0.91 here; four 1.0
    // and 1.46; 1.6 rows a key are equal).
    const bool look = sizeof(K) == 4 && MODE == MODE_EMIT && nb > (1u << 21);
    const size_t db = look ? dup_bytes<K>(1) : 0;
    if (s.get(&mem, head + db + lay.bytes()) != JN_OK) {
        c->err.clear();  // a device too full for the table takes the partitioned path
        return JN_OK;
    }
    Scratch ss(c);
    LongRun* longs = nullptr;
    unsigned char* kept = nullptr;
    if (cap && ss.get(&kept, keep_bytes(segs * cap)) != JN_OK) {
        c->err.clear();
        cap = 0;
    }
    if (cap) {
        staged = reinterpret_cast<jn_pair*>(kept);
        longs = reinterpret_cast<LongRun*>(kept + segs * cap * sizeof(jn_pair));
    }
    DirectSmall* small = reinterpret_cast<DirectSmall*>(mem);
    JN_TRY(zero(c, mem, head + db + (look ? 0 : lay.zeroed())));
    DirectTab<K, MODE> t;
    JN_TRY(wait_copies(c, true));
    DupCount* dup = nullptr;
    if (look) {
        dup = reinterpret_cast<DupCount*>(mem + head);
        DupTables<K> tabs{};
        tabs.add(B.key, B.n);
        JN_TRY(dup_sample<K>(c, tabs, dup));
        JN_TRY(launch(c, K_MEMSET, k_direct_zero, dim3(8 * (unsigned)c->num_sms), dim3(256), 0,
                      reinterpret_cast<uint4*>(mem + head + db), (uint64_t)(lay.zeroed() / 16), (const DupCount*)dup));
    }
    JN_TRY((direct_build<K, MODE>(c, B, swap ? 1 : 0, lay, mem + head + db, small, &t, dup)));
    auto kp = k_direct_probe<K, MODE>;
    int per = 0;
    JN_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kp, DJ_T, 0));
    const uint64_t tiles = ceil_div(np, DJ_T * DJ_U);
    const dim3 g((unsigned)std::min<uint64_t>(tiles, (uint64_t)std::max(per, 1) * c->num_sms));
    JN_TRY(launch(c, K_DIRECT_PROBE, kp, g, dim3(DJ_T), 0, P.key, P.pay, P.n, t, swap ? 1 : 0, small, staged, segs,
                  (unsigned long long)cap, longs, (const DupCount*)dup));
    DirectResult r;
    JN_TRY(direct_result(c, small, segs, cap, &r));
    if (r.left) {
        *repeats = true;
        return JN_OK;
    }
    const uint64_t total = r.total;
    const bool done = r.fits;
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
    if (done && r.longs) JN_TRY(direct_long(c, longs, &small->lines[0].longs));
    // a table no longer needed, or the scratch the pairs did not fit
    (done ? s : ss).release();
    const jn_status st = out_prepare(c, ss, total, *plan);
    if (st == JN_ERR_OOM && plan->no_memory) {
        // no memory for the output beside the table or the kept pairs: the
        // partitioned join, which can do with less
        c->err.clear();
        *taken = false;
        ss.release();
        s.release();
        JN_CUDA(c, cudaStreamSynchronize(c->stream));  // the released memory can take another shape
        return JN_OK;
    }
    if (st != JN_OK) return st;
    if (total && done && plan->host_copy && segs == 1) {
        // straight to the caller's buffer
        JN_CUDA(c, cudaMemcpyAsync(*plan->user_out, staged, total * sizeof(jn_pair), cudaMemcpyDefault, c->stream));
        plan->copied = true;
    } else if (total && done) {
        JN_TRY((direct_gather<uint64_t, 1>(c, K_DIRECT_PROBE, staged, segs, cap, r, plan->dev)));
    } else if (total) {
        longs = nullptr;  // a run admitted by its bytes takes no more scratch
        if (r.dup && !c->mem_limit && !c->admit && ss.get(&longs, total / DJ_LONG + 1) != JN_OK) c->err.clear();
        JN_TRY(zero(c, &small->lines[0].total, 8));
        JN_TRY(zero(c, &small->lines[0].longs, 4));
        JN_TRY(launch(c, K_DIRECT_PROBE, kp, g, dim3(DJ_T), 0, P.key, P.pay, P.n, t, swap ? 1 : 0, small, plan->dev,
                      1u, (unsigned long long)total, longs, (const DupCount*)nullptr));
        if (longs) JN_TRY(direct_long(c, longs, &small->lines[0].longs));
        JN_CUDA(c, cudaStreamSynchronize(c->stream));  // this pass reads the caller's columns
    }
    return out_finish(c, total, *plan);
}

template <typename K>
jn_status run_direct(jn_ctx* c, const Cols<K>& R, const Cols<K>& S, int mode, OutPlan* plan, RunResult* res,
                     bool* taken, bool* repeats) {
    *taken = *repeats = false;
    const uint64_t nb = (uint64_t)std::min(R.n, S.n);
    if (nb == 0 || nb > DJ_MAX || !direct_allowed(c) || R.host || S.host) return JN_OK;
    if (mode == MODE_EMIT) return direct_mode<K, MODE_EMIT>(c, R, S, plan, res, taken, repeats);
    if (mode == MODE_AGG) return direct_mode<K, MODE_AGG>(c, R, S, plan, res, taken, repeats);
    return direct_mode<K, MODE_COUNT>(c, R, S, plan, res, taken, repeats);
}

template jn_status run_direct<int32_t>(jn_ctx*, const Cols<int32_t>&, const Cols<int32_t>&, int, OutPlan*, RunResult*,
                                       bool*, bool*);
template jn_status run_direct<int64_t>(jn_ctx*, const Cols<int64_t>&, const Cols<int64_t>&, int, OutPlan*, RunResult*,
                                       bool*, bool*);

// ------------------------------------------------------------------ batch --
// Equi-joins of a batch by the same method, all of them in every launch: each
// join has its own table, its own line of counters and its own room for its
// pairs, and the blocks take tiles of DB_ROWS rows of all joins in turn (join
// by join, so the tables in use at a time stay in L2).
constexpr int DB_ROWS = 4096;
constexpr uint64_t DB_ROOM = 1ull << 30;  // pairs of room for a whole batch at most (8 GB)

template <typename K>
struct DirectJoin {
    const K* bkey;  // build side: the smaller table
    const int32_t* bpay;
    const K* pkey;
    const int32_t* ppay;
    int64_t bn, pn;
    uint64_t bucket0;  // first bucket of the table
    uint64_t row0;     // build rows of the joins before this one
    uint64_t stage0;   // where its room begins, in pairs
    uint64_t cap;      // and how many it holds
    uint32_t nb;       // buckets (and one for key 0)
    int32_t swap;      // the build side is S
};

// Tile t of n joins' build (or probe) tables: its join and first row.
__device__ __forceinline__ int db_tile(const uint64_t* __restrict__ prefix, int n, uint64_t t, int64_t* row) {
    const int j = find_segment(prefix, n, t);
    *row = (int64_t)(t - prefix[j]) * DB_ROWS;
    return j;
}

template <typename K, int MODE>
struct DirectBatch {
    const DirectJoin<K>* joins;
    const uint64_t* btiles;  // n + 1 tile offsets of the build tables, and of the probe tables
    const uint64_t* ptiles;
    int n;
    typename DirectSlot<K, MODE>::T* slots;
    uint32_t* counts;
    uint2* where;
    int32_t* runs;
    DirectLine* lines;
    LongRun* longs;  // long runs of all joins, counted in lines[0]
    __device__ __forceinline__ DirectTab<K, MODE> table(const DirectJoin<K>& d, int j) const {
        using DS = DirectSlot<K, MODE>;
        DirectTab<K, MODE> t;
        t.slots = slots + d.bucket0 * DS::B;
        t.nb = d.nb;
        t.counts = counts + d.bucket0 * DS::B;
        t.sums = nullptr;
        t.runs = runs + d.row0 * (DS::COUNTS_ASIDE ? 2 : 1);
        t.dup = &lines[j].dup;
        return t;
    }
};

template <typename K, int MODE>
__global__ void __launch_bounds__(DJ_T)
k_batch_insert(DirectBatch<K, MODE> b) {
    const uint64_t tiles = b.btiles[b.n];
    for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        int64_t row;
        const int j = db_tile(b.btiles, b.n, t, &row);
        const DirectJoin<K> d = b.joins[j];
        dj_insert_rows<K, MODE>(d.bkey, d.bpay, row, min(d.bn, row + DB_ROWS), DJ_T, b.table(d, j), d.swap,
                                b.where + d.row0, b.lines + j);
    }
}

// step 0: the runs of keys with several rows, 1: their payloads.
template <typename K>
__global__ void __launch_bounds__(DJ_T)
k_batch_runs(DirectBatch<K, MODE_EMIT> b, int step) {
    const uint64_t tiles = b.btiles[b.n];
    for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        int64_t row;
        const int j = db_tile(b.btiles, b.n, t, &row);
        if (!b.lines[j].dup) continue;
        const DirectJoin<K> d = b.joins[j];
        const int64_t end = min(d.bn, row + DB_ROWS);
        if (step == 0)
            dj_runs_rows<K>(row, end, DJ_T, b.table(d, j), b.where + d.row0, b.lines + j);
        else
            dj_place_rows<K>(d.bpay, row, end, DJ_T, b.table(d, j), b.where + d.row0, b.lines + j);
    }
}

// Emit, first pass (off == NULL): join j's pairs to its room at `out`.
// Second pass: the joins whose pairs passed their room, to out + off[j].
template <typename K, int MODE>
__global__ void __launch_bounds__(DJ_T, JN_DJ_MINB)
k_batch_probe(DirectBatch<K, MODE> b, jn_pair* __restrict__ out, const uint64_t* __restrict__ off) {
    using Out = WarpOut<2>;
    __shared__ int2 s_buf[MODE == MODE_EMIT ? DJ_T / 32 : 1][MODE == MODE_EMIT ? Out::ROOM : 1];
    const uint64_t tiles = b.ptiles[b.n];
    for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        int64_t row;
        const int j = db_tile(b.ptiles, b.n, t, &row);
        const DirectJoin<K> d = b.joins[j];
        uint64_t at = d.stage0, cap = d.cap;
        unsigned long long* cursor = &b.lines[j].total;
        if (MODE == MODE_EMIT && off) {
            at = off[j];
            cap = off[j + 1] - at;
            if (cap <= d.cap) continue;  // already written
            cursor = &b.lines[j].chk;    // the first pass's total stays
        }
        Out wo{MODE == MODE_EMIT ? s_buf[threadIdx.x >> 5] : nullptr, cursor, reinterpret_cast<int2*>(out + at), cap, 0,
               b.longs, &b.lines[0].longs};
        unsigned long long acc = 0, csum = 0;
        dj_probe_rows<K, MODE>(d.pkey, d.ppay, row, min(d.pn, row + DB_ROWS), DJ_T * DJ_U, b.table(d, j), d.swap, wo,
                               acc, csum);
        if (MODE == MODE_EMIT)
            wo.flush();
        else
            warp_add_to(cursor, acc);
    }
}

// The pairs of the joins that fit their room, to their place in the output:
// DB_ROWS pairs of one join per block and round.
__global__ void __launch_bounds__(256)
k_batch_gather(const uint64_t* __restrict__ staged, const uint64_t* __restrict__ stage0,
               const uint64_t* __restrict__ off, const uint64_t* __restrict__ chunks, int n, uint64_t* __restrict__ out) {
    const uint64_t total = chunks[n];
    for (uint64_t c = blockIdx.x; c < total; c += gridDim.x) {
        const int j = find_segment(chunks, n, c);
        const uint64_t q0 = (c - chunks[j]) * DB_ROWS;
        const uint64_t m = min((uint64_t)DB_ROWS, off[j + 1] - off[j] - q0);
        const uint64_t* src = staged + stage0[j] + q0;
        uint64_t* dst = out + off[j] + q0;
        for (uint64_t e = threadIdx.x; e < m; e += 256) dst[e] = __ldcs(src + e);
    }
}

template <typename K, int MODE>
struct DirectBatchRun : BatchRun {
    std::unique_ptr<Scratch> s;
    int n = 0;
    DirectBatch<K, MODE> b{};
    std::vector<DirectJoin<K>> joins;
    jn_pair* staged = nullptr;
    uint64_t btiles = 0, ptiles = 0;
    bool fits = true;
    std::vector<uint64_t> words;  // emit: stage0, chunk offsets

    dim3 grid(jn_ctx* c, const void* fn, uint64_t tiles) const {
        int per = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, DJ_T, 0) != cudaSuccess) {
            cudaGetLastError();
            per = 1;
        }
        return dim3((unsigned)std::min<uint64_t>(std::max<uint64_t>(tiles, 1), (uint64_t)std::max(per, 1) * c->num_sms));
    }

    jn_status prepare(jn_ctx* c, const Cols<K>* Rs, const Cols<K>* Ss) {
        using DS = DirectSlot<K, MODE>;
        s.reset(new Scratch(c));
        joins.resize(n);
        std::vector<uint64_t> bt(n + 1, 0), pt(n + 1, 0);
        uint64_t buckets = 0, rows = 0, stage = 0;
        for (int i = 0; i < n; i++) {
            const bool swap = Ss[i].n < Rs[i].n;
            const Cols<K>&B = swap ? Ss[i] : Rs[i], &P = swap ? Rs[i] : Ss[i];
            const bool live = B.n > 0;
            DirectJoin<K>& d = joins[i];
            d = DirectJoin<K>{B.key, B.pay, P.key, P.pay, B.n, live ? P.n : 0, buckets, rows, stage, 0, 0, swap ? 1 : 0};
            if (live) d.nb = dj_buckets<K, MODE>((uint64_t)B.n);
            if (live && MODE == MODE_EMIT) d.cap = (uint64_t)P.n + (uint64_t)P.n / 4 + 1024;
            buckets += live ? d.nb + 1 : 0;
            rows += (uint64_t)B.n;
            stage += d.cap;
            bt[i + 1] = bt[i] + ceil_div((uint64_t)d.bn, DB_ROWS);
            pt[i + 1] = pt[i] + ceil_div((uint64_t)d.pn, DB_ROWS);
        }
        btiles = bt[n];
        ptiles = pt[n];
        if (stage > DB_ROOM) {  // no room kept: the first pass counts, the second writes
            for (DirectJoin<K>& d : joins) d.stage0 = d.cap = 0;
            stage = 0;
        }
        DirectJoin<K>* d_joins;
        uint64_t *d_bt, *d_pt;
        unsigned char* zeroed;
        const size_t lines = sizeof(DirectLine) * n;
        const size_t slots = buckets * 32, counts = DS::COUNTS_ASIDE ? buckets * DS::B * 4 : 0;
        JN_TRY(s->get(&d_joins, (size_t)n));
        JN_TRY(s->get(&d_bt, (size_t)n + 1));
        JN_TRY(s->get(&d_pt, (size_t)n + 1));
        JN_TRY(s->get(&zeroed, lines + slots + counts));
        if (MODE == MODE_EMIT) {
            JN_TRY(s->get(&b.where, rows));
            JN_TRY(s->get(&b.runs, rows * (DS::COUNTS_ASIDE ? 2 : 1)));
            JN_TRY(s->get(&staged, stage));
            if (stage) JN_TRY(s->get(&b.longs, stage / DJ_LONG + 1));
        }
        b.joins = d_joins;
        b.btiles = d_bt;
        b.ptiles = d_pt;
        b.n = n;
        b.lines = reinterpret_cast<DirectLine*>(zeroed);
        b.slots = reinterpret_cast<typename DS::T*>(zeroed + lines);  // lines are 128 bytes: aligned to a bucket
        b.counts = reinterpret_cast<uint32_t*>(zeroed + lines + slots);
        JN_CUDA(c, cudaMemcpyAsync(d_joins, joins.data(), sizeof(DirectJoin<K>) * n, cudaMemcpyHostToDevice, c->stream));
        JN_CUDA(c, cudaMemcpyAsync(d_bt, bt.data(), 8 * (n + 1), cudaMemcpyHostToDevice, c->stream));
        JN_CUDA(c, cudaMemcpyAsync(d_pt, pt.data(), 8 * (n + 1), cudaMemcpyHostToDevice, c->stream));
        JN_CUDA(c, cudaStreamSynchronize(c->stream));  // the host vectors go out of scope below
        GraphPhase gp(c, c->tune.graphs != 0 && !c->profiling);
        JN_TRY(gp.begin());
        jn_status st = JN_OK;
        do {
            if ((st = zero(c, zeroed, lines + slots + counts)) != JN_OK) break;
            auto ki = k_batch_insert<K, MODE>;
            if ((st = launch(c, K_DIRECT_BUILD, ki, grid(c, (const void*)ki, btiles), dim3(DJ_T), 0, b)) != JN_OK) break;
            if constexpr (MODE == MODE_EMIT) {
                auto kr = k_batch_runs<K>;
                const dim3 g = grid(c, (const void*)kr, btiles);
                if ((st = launch(c, K_DIRECT_BUILD, kr, g, dim3(DJ_T), 0, b, 0)) != JN_OK) break;
                if ((st = launch(c, K_DIRECT_BUILD, kr, g, dim3(DJ_T), 0, b, 1)) != JN_OK) break;
            }
            auto kp = k_batch_probe<K, MODE>;
            if ((st = launch(c, K_DIRECT_PROBE, kp, grid(c, (const void*)kp, ptiles), dim3(DJ_T), 0, b, staged,
                             (const uint64_t*)nullptr)) != JN_OK)
                break;
            if (b.longs) st = direct_long(c, b.longs, &b.lines[0].longs);
        } while (0);
        if (st != JN_OK) {
            gp.abort();
            return st;
        }
        JN_TRY(gp.end_and_run());
        std::vector<uint64_t> tot(n);
        JN_CUDA(c, cudaMemcpy2DAsync(tot.data(), 8, b.lines, sizeof(DirectLine), 8, n, cudaMemcpyDeviceToHost, c->stream));
        JN_CUDA(c, cudaStreamSynchronize(c->stream));
        offsets.assign((size_t)n + 1, 0);
        for (int i = 0; i < n; i++) {
            offsets[i + 1] = offsets[i] + tot[i];
            fits &= tot[i] <= joins[i].cap;
        }
        total = offsets[n];
        return JN_OK;
    }

    jn_status emit(jn_ctx* c, jn_pair* out) override {
        if (total == 0) return JN_OK;
        if constexpr (MODE == MODE_EMIT) {
            // chunks of the joins whose pairs are in their room
            words.assign(2 * (size_t)n + 1, 0);
            uint64_t* chunks = words.data() + n;
            for (int i = 0; i < n; i++) {
                const uint64_t m = offsets[i + 1] - offsets[i];
                words[i] = joins[i].stage0;
                chunks[i + 1] = chunks[i] + (m <= joins[i].cap ? ceil_div(m, DB_ROWS) : 0);
            }
            uint64_t *d_words, *d_off;
            JN_TRY(s->get(&d_words, words.size()));
            JN_TRY(s->get(&d_off, offsets.size()));
            JN_CUDA(c, cudaMemcpyAsync(d_words, words.data(), 8 * words.size(), cudaMemcpyHostToDevice, c->stream));
            JN_CUDA(c, cudaMemcpyAsync(d_off, offsets.data(), 8 * offsets.size(), cudaMemcpyHostToDevice, c->stream));
            JN_TRY(launch(c, K_DIRECT_PROBE, k_batch_gather,
                          dim3((unsigned)std::min<uint64_t>(std::max<uint64_t>(chunks[n], 1), 8 * (uint64_t)c->num_sms)),
                          dim3(256), 0, reinterpret_cast<const uint64_t*>(staged), (const uint64_t*)d_words,
                          (const uint64_t*)d_off, (const uint64_t*)(d_words + n), n, reinterpret_cast<uint64_t*>(out)));
            if (!fits) {
                auto kp = k_batch_probe<K, MODE>;
                b.longs = nullptr;
                if (s->get(&b.longs, total / DJ_LONG + 1) != JN_OK) c->err.clear();
                JN_TRY(zero(c, &b.lines[0].longs, 4));
                JN_TRY(launch(c, K_DIRECT_PROBE, kp, grid(c, (const void*)kp, ptiles), dim3(DJ_T), 0, b, out,
                              (const uint64_t*)d_off));
                if (b.longs) JN_TRY(direct_long(c, b.longs, &b.lines[0].longs));
            }
        }
        return JN_OK;
    }
};

bool batch_direct_takes(const jn_ctx* c, int64_t nr, int64_t ns) {
    return direct_allowed(c) && c->tune.part_rows == 0 && !c->mem_limit && !c->admit &&
           (uint64_t)std::min(nr, ns) <= DJ_MAX;
}

template <typename K>
jn_status batch_direct_prepare(jn_ctx* c, int n, const Cols<K>* Rs, const Cols<K>* Ss, bool count_only,
                               std::unique_ptr<BatchRun>* run) {
    auto go = [&](auto* r) -> jn_status {
        std::unique_ptr<BatchRun> own(r);
        r->n = n;
        const jn_status st = r->prepare(c, Rs, Ss);
        if (st != JN_OK) return st;
        c->info.partitions += (uint64_t)n;
        c->info.work_items += r->ptiles;
        *run = std::move(own);
        return JN_OK;
    };
    if (count_only) return go(new DirectBatchRun<K, MODE_COUNT>());
    return go(new DirectBatchRun<K, MODE_EMIT>());
}

template jn_status batch_direct_prepare<int32_t>(jn_ctx*, int, const Cols<int32_t>*, const Cols<int32_t>*, bool,
                                                 std::unique_ptr<BatchRun>*);
template jn_status batch_direct_prepare<int64_t>(jn_ctx*, int, const Cols<int64_t>*, const Cols<int64_t>*, bool,
                                                 std::unique_ptr<BatchRun>*);

}  // namespace jnx
