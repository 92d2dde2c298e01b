// Star join: a centre table R with two join columns (fk1 = key, fk2 = key2)
// against two dimension tables, S1 on fk1 and S2 on fk2.  Sec. 6 leaves
// multi-table joins to future work; this is the two-table method applied
// twice, as a left-deep plan:
//   1. J1 = R (fk1, row index) joined with S1 by the partitioned hash join;
//   2. the fk2 of every J1 pair's R row is gathered into a key column T1;
//   3. J2 = T1 (row index = J1 index) joined with S2 by the same hash join;
//   4. every J2 pair (j, s2) becomes the triple (R payload of J1[j], J1[j].s, s2).
// Both joins keep their exact count pass, so J1, J2 and the triples are each
// allocated once at their exact size.
//
// Dimensions whose hash tables stay in L2 (jn_direct.cuh) are joined in one
// pass instead: every row of R is looked up in both tables and writes its
// triples, in R's order and with no intermediate pairs.
#include <string.h>

#include "jn_algos.h"
#include "jn_direct.cuh"

namespace jnx {

constexpr int ST_ILP = 4;  // gathers in flight per thread

// t1key[i] = fk2[J1[i].r]: the second join column of each first-join pair's R
// row.  A block covers 256 * ST_ILP consecutive pairs; each thread issues its
// ST_ILP random reads of fk2 before it stores any (the reads are independent).
template <typename K>
__global__ void __launch_bounds__(256)
k_star_keys(const jn_pair* __restrict__ j1, uint64_t m1, const K* __restrict__ fk2, K* __restrict__ t1key) {
    const uint64_t base = (uint64_t)blockIdx.x * (256 * ST_ILP) + threadIdx.x;
    int32_t r[ST_ILP];
#pragma unroll
    for (int u = 0; u < ST_ILP; u++) {
        const uint64_t i = base + (uint64_t)u * 256;
        r[u] = i < m1 ? j1[i].r : -1;
    }
    K v[ST_ILP];
#pragma unroll
    for (int u = 0; u < ST_ILP; u++) v[u] = r[u] >= 0 ? fk2[r[u]] : K(0);
#pragma unroll
    for (int u = 0; u < ST_ILP; u++) {
        const uint64_t i = base + (uint64_t)u * 256;
        if (i < m1) t1key[i] = v[u];
    }
}

// out[i] = (R payload of J1[J2[i].r] (its row index when rpay is NULL),
// J1[J2[i].r].s, J2[i].s), with ST_ILP independent gather chains per thread.
__global__ void __launch_bounds__(256)
k_star_emit(const jn_pair* __restrict__ j1, const jn_pair* __restrict__ j2, uint64_t m2,
            const int32_t* __restrict__ rpay, jn_triple* __restrict__ out) {
    const uint64_t base = (uint64_t)blockIdx.x * (256 * ST_ILP) + threadIdx.x;
    jn_pair b[ST_ILP], a[ST_ILP];
#pragma unroll
    for (int u = 0; u < ST_ILP; u++) {
        const uint64_t i = base + (uint64_t)u * 256;
        b[u] = i < m2 ? j2[i] : jn_pair{-1, 0};
    }
#pragma unroll
    for (int u = 0; u < ST_ILP; u++) a[u] = b[u].r >= 0 ? j1[b[u].r] : jn_pair{-1, 0};
    int32_t p[ST_ILP];
#pragma unroll
    for (int u = 0; u < ST_ILP; u++) p[u] = (rpay && a[u].r >= 0) ? rpay[a[u].r] : a[u].r;
#pragma unroll
    for (int u = 0; u < ST_ILP; u++) {
        const uint64_t i = base + (uint64_t)u * 256;
        if (i < m2) {
            jn_triple t;
            t.r = p[u];
            t.s1 = a[u].s;
            t.s2 = b[u].s;
            out[i] = t;
        }
    }
}

// One pass over R: rows of fk1 in T1 and of fk2 in T2 give m1 * m2 triples.
// The counters get the triples and the pairs of the first join (the left-deep
// plan's intermediate).  Emit: in WarpOut's manner and segments, as
// k_direct_probe, so the 12-byte triples leave as whole lines.
#ifndef JN_SJ_MINB
#define JN_SJ_MINB 6
#endif
constexpr int SJ_U = 1;  // rows a thread looks up at once, in two tables each

template <typename K, int MODE>
__global__ void __launch_bounds__(DJ_T, JN_SJ_MINB)
k_star_probe(const K* __restrict__ fk1, const K* __restrict__ fk2, const int32_t* __restrict__ pay, int64_t n,
             DirectTab<K, MODE> t1, DirectTab<K, MODE> t2, DirectSmall* __restrict__ small, int32_t* __restrict__ out,
             uint32_t segs, unsigned long long cap) {
    constexpr int U = SJ_U, TILE = DJ_T * U;
    using Out = WarpOut<3>;
    __shared__ int32_t s_buf[MODE == MODE_EMIT ? DJ_T / 32 : 1][MODE == MODE_EMIT ? 3 * Out::ROOM : 1];
    const int lane = threadIdx.x & 31;
    const uint32_t seg = blockIdx.x % segs;
    out += 3 * seg * cap;
    Out wo{MODE == MODE_EMIT ? s_buf[threadIdx.x >> 5] : nullptr, &small->lines[seg].total, out, cap, 0};
    const bool dup1 = MODE == MODE_EMIT && *t1.dup != 0, dup2 = MODE == MODE_EMIT && *t2.dup != 0;
    unsigned long long acc = 0, acc1 = 0;
    for (int64_t r0 = (int64_t)blockIdx.x * TILE; r0 < n; r0 += (int64_t)gridDim.x * TILE) {
        K k1[U], k2[U];
        bool valid[U];
        uint32_t m1[U], m2[U], v1[U], v2[U];
        unsigned long long m[U], none[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int64_t i = r0 + u * DJ_T + threadIdx.x;
            valid[u] = i < n;
            k1[u] = valid[u] ? __ldcs(fk1 + i) : K(0);
            k2[u] = valid[u] ? __ldcs(fk2 + i) : K(0);
        }
        dj_lookup<K, MODE, U>(t1, dup1, k1, valid, m1, v1, none);
        dj_lookup<K, MODE, U>(t2, dup2, k2, valid, m2, v2, none);
#pragma unroll
        for (int u = 0; u < U; u++) {
            m[u] = (unsigned long long)m1[u] * m2[u];
            acc1 += m1[u];
            acc += m[u];
        }
        if constexpr (MODE == MODE_EMIT) {
            int32_t pp[U];
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int64_t i = r0 + u * DJ_T + threadIdx.x;
                pp[u] = m[u] ? (pay ? __ldcs(pay + i) : (int32_t)i) : 0;
            }
#pragma unroll
            for (int u = 0; u < U; u++) {
                if (!__any_sync(0xffffffffu, m[u] > 1)) {  // at most one triple per row
                    unsigned any;
                    int32_t* q = wo.slot(m[u] != 0, &any);
                    if (m[u]) {
                        q[0] = pp[u];
                        q[1] = dj_single<K>(dup1, 1) ? (int32_t)v1[u] : t1.runs[v1[u]];
                        q[2] = dj_single<K>(dup2, 1) ? (int32_t)v2[u] : t2.runs[v2[u]];
                    }
                    wo.check();
                    continue;
                }
                const unsigned have = __ballot_sync(0xffffffffu, m[u] != 0);
                const unsigned long long incl = warp_incl_scan(m[u]);
                unsigned long long at;
                if (!wo.reserve(__shfl_sync(0xffffffffu, incl, 31), &at)) continue;
                const unsigned long long mine = at + (incl - m[u]);
                for (unsigned lanes = have; lanes; lanes &= lanes - 1) {
                    const int src = __ffs(lanes) - 1;
                    const unsigned long long lm = __shfl_sync(0xffffffffu, m[u], src);
                    const unsigned long long o = 3 * __shfl_sync(0xffffffffu, mine, src);
                    const uint32_t a1 = __shfl_sync(0xffffffffu, m1[u], src), a2 = __shfl_sync(0xffffffffu, m2[u], src);
                    const uint32_t b1 = __shfl_sync(0xffffffffu, v1[u], src), b2 = __shfl_sync(0xffffffffu, v2[u], src);
                    const int32_t p = __shfl_sync(0xffffffffu, pp[u], src);
                    for (unsigned long long e = lane; e < lm; e += 32) {
                        const uint32_t e1 = (uint32_t)(e / a2), e2 = (uint32_t)(e - (unsigned long long)e1 * a2);
                        out[o + 3 * e] = p;
                        out[o + 3 * e + 1] = dj_single<K>(dup1, a1) ? (int32_t)b1 : t1.runs[b1 + e1];
                        out[o + 3 * e + 2] = dj_single<K>(dup2, a2) ? (int32_t)b2 : t2.runs[b2 + e2];
                    }
                }
            }
        }
    }
    if (MODE == MODE_EMIT)
        wo.flush();
    __shared__ unsigned long long tmp[33];
    acc1 = block_sum(acc1, tmp);
    if (MODE != MODE_EMIT) acc = block_sum(acc, tmp);
    if (threadIdx.x == 0) {
        if (acc1) atomicAdd(&small->lines[0].first, acc1);
        if (MODE != MODE_EMIT && acc) atomicAdd(&small->lines[0].total, acc);
    }
}

namespace {

// Triples past which the left-deep plan takes over: many times the rows, so
// frequent keys carry them.
uint64_t star_most_triples(uint64_t rows) { return 8 * rows + (1u << 20); }

// Where a result of m triples goes: the caller's buffer, or a new one (*dev).
// A host buffer is filled from *dev = scratch by a copy (*copy_back).
jn_status star_output(jn_ctx* c, Scratch& s, uint64_t m, jn_triple* user, uint64_t capacity, uint64_t* n_out,
                      jn_triple** dev, bool* copy_back) {
    *copy_back = false;
    *dev = nullptr;
    if (user && m > capacity) {
        *n_out = m;
        return fail(c, JN_ERR_CAPACITY, "output buffer holds fewer triples than the result");
    }
    if (!user) {
        if (m) JN_TRY(dalloc(c, reinterpret_cast<void**>(dev), m * sizeof(jn_triple)));
    } else if (m == 0 || is_device_pointer(user)) {
        *dev = user;
    } else {
        JN_TRY(s.get(dev, m));
        *copy_back = true;
    }
    return JN_OK;
}

jn_status too_many_first(jn_ctx* c) {
    return fail(c, JN_ERR_UNSUPPORTED, "star join: the first join has more than 2^31 - 1 pairs");
}

bool device_table(const jn_table* t) {
    return is_device_pointer(t->key) && (!t->payload || is_device_pointer(t->payload));
}

// The one-pass star join; *taken false = nothing was done.
template <typename K, int MODE>
jn_status star_direct(jn_ctx* c, const jn_table* R, const jn_table* S1, const jn_table* S2, jn_triple** out,
                      uint64_t capacity, uint64_t* n_out, uint64_t* count, bool* taken) {
    *taken = false;
    const int64_t big = std::max(S1->n, S2->n);
    // R small against a dimension is joined with it the other way round; a run
    // admitted by its bytes keeps the two joins, which ask for each of theirs
    if (R->n < 1 || S1->n < 1 || S2->n < 1 || big > (int64_t)DJ_MAX || R->n < big / 2 || S1->reserved ||
        S2->reserved || c->mem_limit || c->admit || !direct_allowed(c) || !is_device_pointer(R->key) ||
        !device_table(S1) || !device_table(S2))
        return JN_OK;
    const uint64_t n = (uint64_t)R->n;
    const Cols<K> D1{static_cast<const K*>(S1->key), nullptr, S1->payload, S1->n};
    const Cols<K> D2{static_cast<const K*>(S2->key), nullptr, S2->payload, S2->n};
    const DirectLayout<K, MODE> l1((uint64_t)S1->n), l2((uint64_t)S2->n);
    const size_t head = sizeof(DirectSmall);  // each table has its own counters
    const DirectStage sg(n, DJ_ROOM_LEAST);
    const uint32_t segs = MODE == MODE_EMIT ? sg.segs : 1;
    uint64_t cap = MODE == MODE_EMIT ? sg.cap : 0;
    c->info = jn_run_info();
    Scratch s(c), ss(c);
    unsigned char *a = nullptr, *b = nullptr;
    jn_triple* staged = nullptr;
    if (s.get(&a, head + l1.bytes()) != JN_OK || s.get(&b, head + l2.bytes()) != JN_OK) {
        c->err.clear();  // a device too full for the tables takes the two joins
        return JN_OK;
    }
    if (cap && ss.get(&staged, segs * cap) != JN_OK) {
        c->err.clear();
        cap = 0;
    }
    DirectSmall *m1 = reinterpret_cast<DirectSmall*>(a), *m2 = reinterpret_cast<DirectSmall*>(b);
    JN_TRY(zero(c, a, head + l1.zeroed()));
    JN_TRY(zero(c, b, head + l2.zeroed()));
    DirectTab<K, MODE> t1, t2;
    JN_TRY((direct_build<K, MODE>(c, D1, 1, l1, a + head, m1, &t1)));
    JN_TRY((direct_build<K, MODE>(c, D2, 1, l2, b + head, m2, &t2)));
    auto kp = k_star_probe<K, MODE>;
    int per = 0;
    JN_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kp, DJ_T, 0));
    const uint64_t tiles = ceil_div(n, DJ_T * SJ_U);
    const dim3 g((unsigned)std::min<uint64_t>(tiles, (uint64_t)std::max(per, 1) * c->num_sms));
    auto probe = [&](jn_triple* to, uint32_t parts, uint64_t most) {
        return launch(c, K_STAR, kp, g, dim3(DJ_T), 0, static_cast<const K*>(R->key), static_cast<const K*>(R->key2),
                      R->payload, R->n, t1, t2, m1, reinterpret_cast<int32_t*>(to), parts, (unsigned long long)most);
    };
    JN_TRY(probe(staged, segs, cap));
    DirectResult r;
    JN_TRY(direct_result(c, m1, segs, cap, &r));
    const uint64_t m = r.total;
    const bool done = r.fits;
    if (r.first > (uint64_t)INT32_MAX) {
        *taken = true;
        return too_many_first(c);
    }
    if (MODE == MODE_EMIT && !done && m > star_most_triples(n + (uint64_t)S1->n + (uint64_t)S2->n)) return JN_OK;
    *taken = true;
    c->info.result = m;
    c->info.r_survivors = n;
    c->info.s_survivors = (uint64_t)S2->n;
    c->info.partitions = 1;
    c->info.work_items = tiles;
    c->info.hash_path = 3;
    c->info.cartesian_bound = r.first * (uint64_t)S2->n;
    if (MODE != MODE_EMIT) {
        *count = m;
        return JN_OK;
    }
    (done ? s : ss).release();  // the tables, or the scratch the triples did not fit
    jn_triple *user = *out, *dev = nullptr;
    bool copy_back = false;
    const jn_status st = star_output(c, ss, m, user, capacity, n_out, &dev, &copy_back);
    if (st == JN_ERR_OOM) {  // no memory for the output beside the tables or the kept triples: the two joins
        c->err.clear();
        *taken = false;
        ss.release();
        s.release();
        JN_CUDA(c, cudaStreamSynchronize(c->stream));  // the released memory can take another shape
        return JN_OK;
    }
    if (st != JN_OK) return st;
    if (m && done) {
        JN_TRY((direct_gather<int32_t, 3>(c, K_STAR, staged, segs, cap, r, dev)));
    } else if (m) {
        JN_TRY(zero(c, &m1->lines[0].total, 8));
        JN_TRY(probe(dev, 1, m));
    }
    if (copy_back) JN_CUDA(c, cudaMemcpyAsync(user, dev, m * sizeof(jn_triple), cudaMemcpyDefault, c->stream));
    JN_CUDA(c, cudaStreamSynchronize(c->stream));  // as the two joins' way: the triples are complete on return
    if (!user) *out = dev;
    *n_out = m;
    return JN_OK;
}

// Library-allocated pairs of an inner join, freed (stream-ordered) on scope exit.
struct Pairs {
    jn_ctx* c;
    jn_pair* p = nullptr;
    uint64_t n = 0;
    explicit Pairs(jn_ctx* ctx) : c(ctx) {}
    ~Pairs() {
        if (p) jn_free(c, p);
    }
};

// One block per 256 * ST_ILP elements.
unsigned grid_for(uint64_t n) { return (unsigned)((n + 256 * ST_ILP - 1) / (256 * ST_ILP)); }

template <typename K>
jn_status star_typed(jn_ctx* c, const jn_table* R, const jn_table* S1, const jn_table* S2, jn_triple** out,
                     uint64_t capacity, uint64_t* n_out, uint64_t* count) {
    bool taken = false;
    const jn_status direct = count ? star_direct<K, MODE_COUNT>(c, R, S1, S2, out, capacity, n_out, count, &taken)
                                   : star_direct<K, MODE_EMIT>(c, R, S1, S2, out, capacity, n_out, count, &taken);
    if (direct != JN_OK || taken) return direct;
    // 1. R (fk1, row index) joined with S1
    jn_table r1 = *R;
    r1.key2 = nullptr;
    r1.payload = nullptr;
    Pairs j1(c);
    JN_TRY(jn_hash(c, &r1, S1, &j1.p, 0, &j1.n));
    if (j1.n > (uint64_t)INT32_MAX) return too_many_first(c);
    // 2. the fk2 of each pair's R row
    Scratch s(c);
    K* t1key = nullptr;
    if (j1.n) {
        JN_TRY(s.get(&t1key, j1.n));
        JN_TRY(launch(c, K_STAR, k_star_keys<K>, dim3(grid_for(j1.n)), dim3(256), 0, (const jn_pair*)j1.p,
                      j1.n, (const K*)R->key2, t1key));
    }
    jn_table t1;
    memset(&t1, 0, sizeof(t1));
    t1.key = t1key;
    t1.n = (int64_t)j1.n;
    t1.key_type = R->key_type;
    // 3. joined with S2 (count only when that is all that is asked)
    if (count) return jn_count(c, JN_ALGO_HASH, &t1, S2, nullptr, count);
    Pairs j2(c);
    JN_TRY(jn_hash(c, &t1, S2, &j2.p, 0, &j2.n));
    // 4. the triples, at their exact size, in the caller's buffer or a new one
    const uint64_t m = j2.n;
    jn_triple *user = *out, *dev = nullptr;
    bool copy_back = false;
    JN_TRY(star_output(c, s, m, user, capacity, n_out, &dev, &copy_back));
    if (m)
        JN_TRY(launch(c, K_STAR, k_star_emit, dim3(grid_for(m)), dim3(256), 0, (const jn_pair*)j1.p,
                      (const jn_pair*)j2.p, m, (const int32_t*)R->payload, dev));
    if (copy_back) JN_CUDA(c, cudaMemcpyAsync(user, dev, m * sizeof(jn_triple), cudaMemcpyDefault, c->stream));
    JN_CUDA(c, cudaStreamSynchronize(c->stream));
    if (!user) *out = dev;
    *n_out = m;
    return JN_OK;
}

jn_status star_entry(jn_ctx* c, const jn_table* R, const jn_table* S1, const jn_table* S2, jn_triple** out,
                     uint64_t capacity, uint64_t* n_out, uint64_t* count) {
    if (!c) return JN_ERR_INVALID;
    c->err.clear();
    if (!R || !S1 || !S2) return fail(c, JN_ERR_INVALID, "star join: NULL table");
    if (count ? false : (!out || !n_out)) return fail(c, JN_ERR_INVALID, "star join: NULL output pointer");
    if (R->key_type != S1->key_type || R->key_type != S2->key_type)
        return fail(c, JN_ERR_INVALID, "star join: key types differ");
    if (R->key_type != JN_KEY_I32 && R->key_type != JN_KEY_I64)
        return fail(c, JN_ERR_INVALID, "star join: key_type must be JN_KEY_I32 or JN_KEY_I64");
    if (R->n < 0 || R->n > INT32_MAX || R->reserved)
        return fail(c, JN_ERR_INVALID, "star join: R row count out of range or reserved set");
    if (R->n > 0 && (!R->key || !R->key2)) return fail(c, JN_ERR_INVALID, "star join: R needs key and key2");
    JN_CUDA(c, cudaSetDevice(c->device));
    // R's second join column and payloads are read by this file's kernels
    if (R->n > 0 && (!is_device_pointer(R->key2) || (R->payload && !is_device_pointer(R->payload))))
        return fail(c, JN_ERR_INVALID, "star join: R's key2 and payload must be device memory");
    const uint64_t l0 = c->launches_total;
    const jn_status st = R->key_type == JN_KEY_I32 ? star_typed<int32_t>(c, R, S1, S2, out, capacity, n_out, count)
                                                   : star_typed<int64_t>(c, R, S1, S2, out, capacity, n_out, count);
    c->info.kernel_launches = c->launches_total - l0;
    return st;
}

}  // namespace
}  // namespace jnx

using namespace jnx;

extern "C" {

jn_status jn_star(jn_ctx* ctx, const jn_table* R, const jn_table* S1, const jn_table* S2, jn_triple** out,
                  uint64_t capacity, uint64_t* n_out) {
    return star_entry(ctx, R, S1, S2, out, capacity, n_out, nullptr);
}

jn_status jn_star_count(jn_ctx* ctx, const jn_table* R, const jn_table* S1, const jn_table* S2,
                        uint64_t* count) {
    if (!count) return JN_ERR_INVALID;
    return star_entry(ctx, R, S1, S2, nullptr, 0, nullptr, count);
}

void jn_free_triples(jn_ctx* ctx, jn_triple* p) {
    if (p) cudaFreeAsync(p, ctx ? ctx->stream : (cudaStream_t)0);
}

}  // extern "C"
