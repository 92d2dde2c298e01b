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
    DupHead* dup = nullptr;
    if (look) {
        dup = reinterpret_cast<DupHead*>(mem + head);
        DupTables<K> tabs{};
        tabs.add(B.key, B.n);
        DupRule rule;
        rule.ratio = 1.8f;
        rule.once[0] = 0;
        rule.again[0] = 1;
        JN_TRY(dup_sample<K>(c, tabs, rule, dup));
        JN_TRY(launch(c, K_MEMSET, k_direct_zero, dim3(8 * (unsigned)c->num_sms), dim3(256), 0,
                      reinterpret_cast<uint4*>(mem + head + db), (uint64_t)(lay.zeroed() / 16), (const DupHead*)dup));
    }
    JN_TRY((direct_build<K, MODE>(c, B, swap ? 1 : 0, lay, mem + head + db, small, &t, dup)));
    auto kp = k_direct_probe<K, MODE>;
    int per = 0;
    JN_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kp, DJ_T, 0));
    const uint64_t tiles = ceil_div(np, DJ_T * DJ_U);
    const dim3 g((unsigned)std::min<uint64_t>(tiles, (uint64_t)std::max(per, 1) * c->num_sms));
    JN_TRY(launch(c, K_DIRECT_PROBE, kp, g, dim3(DJ_T), 0, P.key, P.pay, P.n, t, swap ? 1 : 0, small, staged, segs,
                  (unsigned long long)cap, longs, (const DupHead*)dup));
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
                      1u, (unsigned long long)total, longs, (const DupHead*)nullptr));
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
// by join, so the tables in use at a time stay in L2: the resident blocks' 1216
// tiles are 1.2e6 rows.  With tiles of 4096 rows they were 5e6, the rows of
// nineteen joins of 2^18, whose tables are 180 MB, and a batch of few joins had
// too few tiles: 48 joins of 2^18 x 2^18 1.13 ms then, 0.95 now; 16 of 30000 x
// 30000 rows with 100 rows a key 0.56 and 0.30).
constexpr int DB_ROWS = 1024;
constexpr int DB_CHUNK = 4096;              // pairs copied per block and round
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
    const DupHead* dup;  // the sample's verdict, or NULL
    __device__ __forceinline__ bool left() const { return dj_left(dup); }
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
k_batch_zero(const __grid_constant__ DirectBatch<K, MODE> b, uint4* __restrict__ p, uint64_t n) {
    if (!b.left()) dj_zero(p, n);
}

template <typename K, int MODE>
__global__ void __launch_bounds__(DJ_T)
k_batch_insert(const __grid_constant__ DirectBatch<K, MODE> b) {
    if (b.left()) return;
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
k_batch_runs(const __grid_constant__ DirectBatch<K, MODE_EMIT> b, int step) {
    if (b.left()) return;
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
k_batch_probe(const __grid_constant__ DirectBatch<K, MODE> b, jn_pair* __restrict__ out, const uint64_t* __restrict__ off) {
    using Out = WarpOut<2>;
    __shared__ int2 s_buf[MODE == MODE_EMIT ? DJ_T / 32 : 1][MODE == MODE_EMIT ? Out::ROOM : 1];
    if (b.left()) {
        if (blockIdx.x == 0 && threadIdx.x == 0) b.lines[0].left = 1;
        return;
    }
    const uint64_t tiles = b.ptiles[b.n];
    int held = -1;  // the join whose pairs or count the warp holds
    Out wo{MODE == MODE_EMIT ? s_buf[threadIdx.x >> 5] : nullptr, nullptr, nullptr, 0, 0, b.longs, &b.lines[0].longs};
    unsigned long long acc = 0, csum = 0;
    auto put = [&] {
        if (held < 0) return;
        if (MODE == MODE_EMIT)
            wo.flush();
        else
            warp_add_to(wo.cursor, acc);
        acc = 0;
    };
    for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        int64_t row;
        const int j = db_tile(b.ptiles, b.n, t, &row);
        const DirectJoin<K> d = b.joins[j];
        if (MODE == MODE_EMIT && off && off[j + 1] - off[j] <= d.cap) continue;  // already written
        if (j != held) {
            put();
            held = j;
            if (MODE == MODE_EMIT && off) {
                wo.out = reinterpret_cast<int2*>(out + off[j]);
                wo.cap = off[j + 1] - off[j];
                wo.cursor = &b.lines[j].chk;  // the first pass's total stays
            } else {
                wo.out = reinterpret_cast<int2*>(out + d.stage0);
                wo.cap = d.cap;
                wo.cursor = &b.lines[j].total;
            }
        }
        dj_probe_rows<K, MODE>(d.pkey, d.ppay, row, min(d.pn, row + DB_ROWS), DJ_T * DJ_U, b.table(d, j), d.swap, wo,
                               acc, csum);
    }
    put();
}

// The pairs of the joins that fit their room, to their place in the output:
// DB_CHUNK pairs of one join per block and round.
__global__ void __launch_bounds__(256)
k_batch_gather(const uint64_t* __restrict__ staged, const uint64_t* __restrict__ stage0,
               const uint64_t* __restrict__ off, const uint64_t* __restrict__ chunks, int n, uint64_t* __restrict__ out) {
    const uint64_t total = chunks[n];
    for (uint64_t c = blockIdx.x; c < total; c += gridDim.x) {
        const int j = find_segment(chunks, n, c);
        const uint64_t q0 = (c - chunks[j]) * DB_CHUNK;
        const uint64_t m = min((uint64_t)DB_CHUNK, off[j + 1] - off[j] - q0);
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
    std::vector<uint64_t> bt, pt;  // tile offsets; like joins, kept for the copies to the device
    jn_pair* staged = nullptr;
    uint64_t btiles = 0, ptiles = 0;
    bool fits = true;
    bool left = false;   // the rule's verdict: nothing was done
    uint32_t longs = 0;  // parts of long runs among the kept pairs
    std::vector<uint64_t> words;  // emit: stage0, chunk offsets

    dim3 grid(jn_ctx* c, const void* fn, uint64_t tiles) const {
        int per = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, DJ_T, 0) != cudaSuccess) {
            cudaGetLastError();
            per = 1;
        }
        return dim3((unsigned)std::min<uint64_t>(std::max<uint64_t>(tiles, 1), (uint64_t)std::max(per, 1) * c->num_sms));
    }

    // Whether the batch's equi-joins go to the partitioned batch after all, all of
    // them: the sum of what they take here beyond what they take there, with the
    // largest build sides' repeated keys from a sample, against what a second set
    // of launches and the sets' own small terms take.  False: not to be asked.
    // us per 2^20 rows on GB300, build + probe rows, from batches of joins of 2^14
    // to 2^20 build rows: int32 keys 62 + 13 here, 90 + 28 with repeated keys,
    // 29 a row partitioned; int64 keys 58 + 14, 75 + 33 and 46.  Joins of up to
    // 8192 rows are not looked at: launches and latency bound both.
    bool ask(const Cols<K>* Rs, const Cols<K>* Ss, DupTables<K>* tabs, DupRule* r) {
        constexpr bool W = sizeof(K) == 8;
        constexpr int64_t SMALL = 8192, LOOK = 1 << 16;  // a part of a table shows repeats too
        std::vector<int> large;
        double worst = 0, least = 0, all = 0, seen = 0;
        auto rows = [&](int i, double* bn, double* pn) {
            *bn = (double)std::min(Rs[i].n, Ss[i].n) / (1 << 20);
            *pn = (double)std::max(Rs[i].n, Ss[i].n) / (1 << 20);
        };
        auto loss = [&](int i, bool again) {
            double bn, pn;
            rows(i, &bn, &pn);
            return again ? (W ? 75 : 90) * bn + (W ? 33 : 28) * pn - (W ? 46 : 29) * (bn + pn)
                         : (W ? 58 : 62) * bn + (W ? 14 : 13) * pn - (W ? 46 : 29) * (bn + pn);
        };
        r->most = 110;
        for (int i = 0; i < n; i++) {
            if (std::min(Rs[i].n, Ss[i].n) > SMALL)
                large.push_back(i);
            else
                r->base += (float)loss(i, false);
        }
        for (int i : large) {
            worst += std::max(loss(i, true), loss(i, false));
            least += std::min(loss(i, true), loss(i, false));
        }
        if (worst + r->base <= r->most) return false;
        if (least + r->base > r->most) {  // whatever the keys are
            left = true;
            return false;
        }
        std::sort(large.begin(), large.end(),
                  [&](int x, int y) { return std::min(Rs[x].n, Ss[x].n) > std::min(Rs[y].n, Ss[y].n); });
        for (size_t k = 0; k < large.size(); k++) {
            double bn, pn;
            rows(large[k], &bn, &pn);
            all += bn;
            if (k >= DUP_MANY) continue;
            seen += bn;
            const Cols<K>& B = Ss[large[k]].n < Rs[large[k]].n ? Ss[large[k]] : Rs[large[k]];
            tabs->add(B.key, std::min(B.n, LOOK));
            r->once[k] = (float)loss(large[k], false);
            r->again[k] = (float)loss(large[k], true);
        }
        for (int k = 0; k < tabs->n; k++) {  // the ones looked at stand for the rest
            r->once[k] *= (float)(all / seen);
            r->again[k] *= (float)(all / seen);
        }
        return true;
    }

    jn_status prepare(jn_ctx* c, const Cols<K>* Rs, const Cols<K>* Ss) {
        using DS = DirectSlot<K, MODE>;
        DupTables<K> tabs{};
        DupRule rule;
        const bool asked = MODE == MODE_EMIT && ask(Rs, Ss, &tabs, &rule);
        if (left) return JN_OK;
        s.reset(new Scratch(c));
        joins.resize(n);
        bt.assign((size_t)n + 1, 0);
        pt.assign((size_t)n + 1, 0);
        uint64_t buckets = 0, rows = 0, stage = 0, probed = 0;
        for (int i = 0; i < n; i++) probed += (uint64_t)std::max(Rs[i].n, Ss[i].n);
        const uint32_t quarters = probed > DB_ROOM / DJ_ROOM * 4 ? DJ_ROOM_LEAST : DJ_ROOM;
        for (int i = 0; i < n; i++) {
            const bool swap = Ss[i].n < Rs[i].n;
            const Cols<K>&B = swap ? Ss[i] : Rs[i], &P = swap ? Rs[i] : Ss[i];
            const bool live = B.n > 0;
            DirectJoin<K>& d = joins[i];
            d = DirectJoin<K>{B.key, B.pay, P.key, P.pay, B.n, live ? P.n : 0, buckets, rows, stage, 0, 0, swap ? 1 : 0};
            if (live) d.nb = dj_buckets<K, MODE>((uint64_t)B.n);
            if (live && MODE == MODE_EMIT) d.cap = DirectStage((uint64_t)P.n, quarters).room();
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
        // counters and sample (128 and 256 bytes' multiples), then the tables
        const size_t db = asked ? dup_bytes<K>(tabs.n) : 0, tables = (slots + counts + 15) & ~(size_t)15;
        JN_TRY(s->get(&zeroed, lines + db + tables));
        DupHead* const dup = asked ? reinterpret_cast<DupHead*>(zeroed + lines) : nullptr;
        b.dup = dup;
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
        b.slots = reinterpret_cast<typename DS::T*>(zeroed + lines + db);  // aligned to a bucket
        b.counts = reinterpret_cast<uint32_t*>(zeroed + lines + db + slots);
        JN_CUDA(c, cudaMemcpyAsync(d_joins, joins.data(), sizeof(DirectJoin<K>) * n, cudaMemcpyHostToDevice, c->stream));
        JN_CUDA(c, cudaMemcpyAsync(d_bt, bt.data(), 8 * (n + 1), cudaMemcpyHostToDevice, c->stream));
        JN_CUDA(c, cudaMemcpyAsync(d_pt, pt.data(), 8 * (n + 1), cudaMemcpyHostToDevice, c->stream));
        GraphPhase gp(c, c->tune.graphs != 0 && !c->profiling);
        JN_TRY(gp.begin());
        jn_status st = JN_OK;
        do {
            if ((st = zero(c, zeroed, lines + db + (dup ? 0 : tables))) != JN_OK) break;
            if (dup) {
                if ((st = dup_sample<K>(c, tabs, rule, dup)) != JN_OK) break;
                if ((st = launch(c, K_MEMSET, k_batch_zero<K, MODE>, dim3(8 * (unsigned)c->num_sms), dim3(DJ_T), 0, b,
                                 reinterpret_cast<uint4*>(zeroed + lines + db), (uint64_t)(tables / 16))) != JN_OK)
                    break;
            }
            auto ki = k_batch_insert<K, MODE>;
            if ((st = launch(c, K_DIRECT_BUILD, ki, grid(c, (const void*)ki, btiles), dim3(DJ_T), 0, b)) != JN_OK) break;
            if constexpr (MODE == MODE_EMIT) {
                auto kr = k_batch_runs<K>;
                const dim3 g = grid(c, (const void*)kr, btiles);
                if ((st = launch(c, K_DIRECT_BUILD, kr, g, dim3(DJ_T), 0, b, 0)) != JN_OK) break;
                if ((st = launch(c, K_DIRECT_BUILD, kr, g, dim3(DJ_T), 0, b, 1)) != JN_OK) break;
            }
            auto kp = k_batch_probe<K, MODE>;
            st = launch(c, K_DIRECT_PROBE, kp, grid(c, (const void*)kp, ptiles), dim3(DJ_T), 0, b, staged,
                        (const uint64_t*)nullptr);
        } while (0);
        if (st != JN_OK) {
            gp.abort();
            return st;
        }
        JN_TRY(gp.end_and_run());
        constexpr int LW = DJ_LINE_WORDS;
        std::vector<uint64_t> tot((size_t)LW * n);
        JN_CUDA(c, cudaMemcpy2DAsync(tot.data(), 8 * LW, b.lines, sizeof(DirectLine), 8 * LW, n, cudaMemcpyDeviceToHost,
                                     c->stream));
        JN_CUDA(c, cudaStreamSynchronize(c->stream));
        longs = (uint32_t)(tot[4] >> 32);
        left = (tot[5] & 0xffffffffu) != 0;
        if (left) return JN_OK;
        b.dup = nullptr;  // a second pass does not ask again
        offsets.assign((size_t)n + 1, 0);
        for (int i = 0; i < n; i++) {
            offsets[i + 1] = offsets[i] + tot[(size_t)LW * i];
            fits &= tot[(size_t)LW * i] <= joins[i].cap;
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
                chunks[i + 1] = chunks[i] + (m <= joins[i].cap ? ceil_div(m, DB_CHUNK) : 0);
            }
            uint64_t *d_words, *d_off;
            JN_TRY(s->get(&d_words, words.size()));
            JN_TRY(s->get(&d_off, offsets.size()));
            JN_CUDA(c, cudaMemcpyAsync(d_words, words.data(), 8 * words.size(), cudaMemcpyHostToDevice, c->stream));
            JN_CUDA(c, cudaMemcpyAsync(d_off, offsets.data(), 8 * offsets.size(), cudaMemcpyHostToDevice, c->stream));
            if (b.longs && longs) JN_TRY(direct_long(c, b.longs, &b.lines[0].longs));
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
        if (st != JN_OK || r->left) return st;
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
