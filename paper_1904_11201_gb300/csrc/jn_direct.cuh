// Direct equi join: one hash table of the smaller table's keys in global
// memory, probed by the larger table where it lies, with no partitioning.
//
// The partition passes of the other paths exist so that a build table fits
// shared memory.  A build table that stays in the GPU's 129 MB L2 needs none:
// a probe row costs one 32-byte bucket read from L2 (two or four slots) and is
// read from HBM once, in order, where the partitioned join moves it twice and
// reads it four times.  The paper's hash join (Sec. 3.3.2)
// builds on "the smaller table" too (Sec. 2.3); pairs keep the (R, S) order
// whichever side was built.
//
// Table: any number of 32-byte buckets (multiply-shift), the sector one read
// brings, filled front to back and then into the next bucket; one slot per
// distinct key.  Key 0 marks an empty slot and keeps a bucket of its own
// behind the table, so a table starts as zeros.  A lookup step reads a whole
// bucket: with single slots a warp waited for the longest of its 32 chains,
// about six dependent reads at a load of one half.  A slot is as narrow as
// the run allows, because the table's size in L2 is what limits the method:
//   int32 keys, count:      (key, rows)                          8 bytes
//   int32 keys, emit:       (key, value), rows counted aside     8 bytes
//   int32 keys, aggregate:  (key, rows, sum of f)               16 bytes
//   int64 keys:             (key, rows, value)                  16 bytes,
//                           aggregate: sums of f in an array of their own
// where f (g when S is built) is the checksum's mixer of the payload, and an
// emitting run's value is the payload of a key with one row, or where the
// payloads of a key with several rows start in `runs`.  With int32 keys the
// value is a run's start for every key as soon as any key has several rows,
// and the run begins with its length.  Equal keys of a warp insert once, so
// skewed build columns do not queue on one slot.
#pragma once

#include <algorithm>

#include "jn_algos.h"
#include "jn_common.cuh"

namespace jnx {

#ifndef JN_DJ_T
#define JN_DJ_T 256
#endif
#ifndef JN_DJ_MINB
#define JN_DJ_MINB 8
#endif
#ifndef JN_DJ_BUF
#define JN_DJ_BUF 128
#endif
constexpr int DJ_BUF = JN_DJ_BUF;  // results a probing warp collects before it writes them
constexpr int DJ_T = JN_DJ_T;  // threads per block
constexpr int DJ_U = 1;        // probe rows a thread looks up at once (4 and 8 measured slower)

// Counters at the head of a direct join's scratch (zeroed with its table).
// Segment r of the staged results has its cursor in lines[r].total, each in a
// 128-byte line of its own: adds to one address pass at about one in 2 ns, so
// 2^26 pairs through one cursor, 256 at a time, would take 0.5 ms alone.
constexpr int DJ_SEGS = 8;
struct DirectLine {
    unsigned long long total;   // results counted (of the segment when emitting)
    unsigned long long chk;     // [0]: aggregate checksum
    unsigned long long first;   // [0]: star join: pairs of the first join
    unsigned long long cursor;  // [0]: words placed in `runs`
    unsigned int dup;           // [0]: some key has several build rows (emit)
    unsigned int longs;         // [0]: parts of long runs left to k_direct_long
    unsigned int left;          // [0]: nothing was done (dj_left)
    unsigned int pad[21];
};
struct DirectSmall {
    DirectLine lines[DJ_SEGS];
};
static_assert(sizeof(DirectLine) == 128, "one line per cursor");

template <typename K, int MODE>
struct DirectSlot {
    static constexpr bool W8 = sizeof(K) == 4 && MODE != MODE_AGG;  // 8-byte slots
    using T = typename std::conditional<W8, uint2, uint4>::type;
    static constexpr int B = 32 / (int)sizeof(T);  // slots per bucket
    static constexpr bool COUNTS_ASIDE = sizeof(K) == 4 && MODE == MODE_EMIT;
    static constexpr bool SUMS_ASIDE = sizeof(K) == 8 && MODE == MODE_AGG;
};

// A built table, as the kernels see it.
template <typename K, int MODE>
struct DirectTab {
    using Slot = typename DirectSlot<K, MODE>::T;
    static constexpr int B = DirectSlot<K, MODE>::B;
    Slot* slots;               // nb buckets of B slots, and one bucket for key 0
    uint32_t nb;
    uint32_t* counts;          // rows per slot (COUNTS_ASIDE)
    unsigned long long* sums;  // sum of f per slot (SUMS_ASIDE)
    int32_t* runs;             // payloads of keys with several rows (emit)
    const unsigned int* dup;   // emit: set when `runs` is used

    __device__ __forceinline__ static K key(const Slot& s) {
        if constexpr (sizeof(K) == 4)
            return (K)s.x;
        else
            return (K)(((uint64_t)s.y << 32) | s.x);
    }
    // rows of the key in slot i, for the slots that hold the count
    __device__ __forceinline__ static uint32_t rows(const Slot& s) {
        if constexpr (sizeof(K) == 4)
            return s.y;
        else
            return s.z;
    }
    __device__ __forceinline__ uint32_t* rows_at(uint32_t i) const {
        if constexpr (DirectSlot<K, MODE>::COUNTS_ASIDE)
            return counts + i;
        else
            return reinterpret_cast<uint32_t*>(slots + i) + (sizeof(K) == 4 ? 1 : 2);
    }
    __device__ __forceinline__ static uint32_t value(const Slot& s) {
        if constexpr (sizeof(K) == 4)
            return s.y;
        else
            return s.w;
    }
    __device__ __forceinline__ uint32_t* value_at(uint32_t i) const {
        return reinterpret_cast<uint32_t*>(slots + i) + (sizeof(K) == 4 ? 1 : 3);
    }
    __device__ __forceinline__ unsigned long long* sum_at(uint32_t i) const {
        if constexpr (DirectSlot<K, MODE>::SUMS_ASIDE)
            return sums + i;
        else
            return reinterpret_cast<unsigned long long*>(slots + i) + 1;
    }
    // buckets: the first one of a key, the one after a full one
    __device__ __forceinline__ uint32_t home(K k) const { return k == K(0) ? nb : __umulhi(khash(k), nb); }
    __device__ __forceinline__ uint32_t next(uint32_t b) const { return b + 1 == nb ? 0u : b + 1; }
    __device__ __forceinline__ uint32_t zero_slot() const { return nb * (uint32_t)B; }
};

// One bucket in one 32-byte read (the table is complete: the read-only path).
template <typename Slot>
__device__ __forceinline__ void dj_bucket(const Slot* p, Slot* q) {
    static_assert(sizeof(Slot) == 8 || sizeof(Slot) == 16, "two or four slots to a bucket");
    unsigned long long a, b, c, d;
    asm("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(a), "=l"(b), "=l"(c), "=l"(d) : "l"(p));
    if constexpr (sizeof(Slot) == 8) {
        q[0] = make_uint2((uint32_t)a, (uint32_t)(a >> 32));
        q[1] = make_uint2((uint32_t)b, (uint32_t)(b >> 32));
        q[2] = make_uint2((uint32_t)c, (uint32_t)(c >> 32));
        q[3] = make_uint2((uint32_t)d, (uint32_t)(d >> 32));
    } else {
        q[0] = make_uint4((uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32));
        q[1] = make_uint4((uint32_t)c, (uint32_t)(c >> 32), (uint32_t)d, (uint32_t)(d >> 32));
    }
}

// The slot of key k, claimed if it had none.  A slot is only tried after the
// ones before it in its bucket hold other keys, so a bucket has no gaps.
template <typename K, int MODE>
__device__ __forceinline__ uint32_t dj_claim(const DirectTab<K, MODE>& t, K k) {
    constexpr int B = DirectTab<K, MODE>::B;
    uint32_t b = t.home(k);
    if (k == K(0)) return t.zero_slot();
    for (uint32_t probe = 0; probe <= t.nb; probe++) {
#pragma unroll
        for (int j = 0; j < B; j++) {
            const uint32_t s = b * B + j;
            K old;
            if (sizeof(K) == 4)
                old = (K)atomicCAS(reinterpret_cast<unsigned int*>(t.slots + s), 0u, (unsigned int)k);
            else
                old = (K)atomicCAS(reinterpret_cast<unsigned long long*>(t.slots + s), 0ull, (unsigned long long)k);
            if (old == K(0) || old == k) return s;
        }
        b = t.next(b);
    }
    return t.zero_slot();  // not reached: the table has twice the slots of its rows
}

// ------------------------------------------------------- repeated keys --
// Repeated build keys cost the direct join a run per key: counts, starts and
// payloads, each a random access to a table or an array (int32 rows, ms for a
// build of 2^22: 0.11 without repeats, 0.31 with).  Where that decides between
// the direct and the partitioned join, the rows of one hash in 2^shift are
// counted first, 1024 to 2048 of them, and their keys.  The sample's last block
// gives the verdict, which the build's kernels read themselves: no host round
// trip (25 us here) in between.
constexpr int DUP_SLOTS = 4096;   // per table
constexpr int DUP_ROWS = 2048;    // rows per tile
struct DupCount {
    unsigned long long rows, keys;
};
template <typename K>
struct DupTable {
    const K* key;
    int64_t n;
    int shift, pad;
};
// Tables by value, with their tiles' prefix.
constexpr int DUP_MANY = 32;
template <typename K>
struct DupTables {
    DupTable<K> t[DUP_MANY];
    uint32_t tiles[DUP_MANY + 1];
    int n;
    void add(const K* key, int64_t rows) {  // n < DUP_MANY
        int shift = 0;
        while ((rows >> shift) >= 2048) shift++;
        t[n] = DupTable<K>{key, rows, shift, 0};
        tiles[n + 1] = tiles[n] + (uint32_t)ceil_div((uint64_t)rows, DUP_ROWS);
        n++;
    }
};
// When joins are left to the partitioned join, all of them: base and the sum
// over the tables of once[k], or again[k] where keys have more than `ratio`
// rows, pass `most`.
struct DupRule {
    float base = 0, most = 0, ratio = 1;
    float once[DUP_MANY], again[DUP_MANY];
};
// The sample in memory: this, a DupCount per table, slots; starts as zeros.
struct DupHead {
    unsigned int left;  // the verdict
    unsigned int done;  // blocks
    unsigned int pad[2];
};
template <typename K>
inline size_t dup_bytes(int n) {
    return (sizeof(DupHead) + (size_t)n * (sizeof(DupCount) + DUP_SLOTS * sizeof(K)) + 255) & ~(size_t)255;
}

// Not the tables' and partitions' hash: the keys looked at lie all over them.
__device__ __forceinline__ uint32_t dup_hash(int32_t k) {
    uint32_t h = (uint32_t)k * 0x2C1B3C6Du;
    h = (h ^ (h >> 15)) * 0x297A2D39u;
    return h ^ (h >> 16);
}
__device__ __forceinline__ uint32_t dup_hash(int64_t k) {
    return dup_hash((int32_t)((uint32_t)k ^ (uint32_t)((uint64_t)k >> 32) * 0x9E3779B1u));
}

// Key 0 is left out.
template <typename K>
__global__ void __launch_bounds__(256)
k_dup_sample(const __grid_constant__ DupTables<K> tabs, const __grid_constant__ DupRule rule, DupHead* head) {
    DupCount* const counts = reinterpret_cast<DupCount*>(head + 1);
    K* const slots = reinterpret_cast<K*>(counts + tabs.n);
    const uint32_t ntiles = tabs.tiles[tabs.n];
    int j = 0;
    for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        while (tabs.tiles[j + 1] <= t) j++;
        const DupTable<K> d = tabs.t[j];
        const int64_t r0 = (int64_t)(t - tabs.tiles[j]) * DUP_ROWS, end = min(d.n, r0 + DUP_ROWS);
        K* tab = slots + (size_t)j * DUP_SLOTS;
        unsigned int rows = 0, keys = 0;
        constexpr int U = DUP_ROWS / 256;
        K k[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int64_t i = r0 + u * 256 + threadIdx.x;
            k[u] = i < end ? d.key[i] : K(0);
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const uint32_t h = dup_hash(k[u]);
            if (k[u] == K(0) || (d.shift && h >> (32 - d.shift))) continue;
            rows++;
            uint32_t s = h & (DUP_SLOTS - 1);
            bool known = false;
            for (int probe = 0; probe < 64 && !known; probe++) {
                K old = *(volatile K*)(tab + s);
                if (old == K(0)) {
                    if (sizeof(K) == 4)
                        old = (K)atomicCAS(reinterpret_cast<unsigned int*>(tab + s), 0u, (unsigned int)k[u]);
                    else
                        old = (K)atomicCAS(reinterpret_cast<unsigned long long*>(tab + s), 0ull,
                                           (unsigned long long)k[u]);
                    if (old == K(0)) break;  // a new key
                }
                known = old == k[u];
                s = (s + 1) & (DUP_SLOTS - 1);
            }
            keys += !known;
        }
        rows = warp_sum(rows);
        keys = warp_sum(keys);
        if ((threadIdx.x & 31) == 0 && rows) {
            atomicAdd(&counts[j].rows, (unsigned long long)rows);
            atomicAdd(&counts[j].keys, (unsigned long long)keys);
        }
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x >= 32) return;
    unsigned int before = 0;
    if (threadIdx.x == 0) before = atomicAdd(&head->done, 1u);
    if (__shfl_sync(0xffffffffu, before, 0) != gridDim.x - 1) return;
    __threadfence();
    static_assert(DUP_MANY == 32, "a lane per table");
    float cost = 0;
    if (threadIdx.x < tabs.n) {
        volatile DupCount* d = counts + threadIdx.x;
        cost = (float)d->rows > rule.ratio * (float)d->keys ? rule.again[threadIdx.x] : rule.once[threadIdx.x];
    }
    cost = warp_sum(cost);
    if (threadIdx.x == 0) head->left = rule.base + cost > rule.most;
}

template <typename K>
jn_status dup_sample(jn_ctx* c, const DupTables<K>& tabs, const DupRule& rule, DupHead* head) {
    const uint32_t tiles = std::max(tabs.tiles[tabs.n], 1u);
    return launch(c, K_DIRECT_BUILD, k_dup_sample<K>, dim3(std::min<uint32_t>(tiles, 8 * (uint32_t)c->num_sms)),
                  dim3(256), 0, tabs, rule, head);
}

__device__ __forceinline__ bool dj_left(const DupHead* dup) { return dup && dup->left; }

// n 16-byte words set to zero by the block's share of a grid.
__device__ __forceinline__ void dj_zero(uint4* p, uint64_t n) {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
        p[i] = make_uint4(0, 0, 0, 0);
}
static __global__ void __launch_bounds__(256) k_direct_zero(uint4* p, uint64_t n, const DupHead* __restrict__ dup) {
    if (!dj_left(dup)) dj_zero(p, n);
}

// Inserts the build rows.  Emit: where[i] = (slot, rank among the key's
// rows), and the rank-0 row leaves its payload in the slot, which is final
// when no key has several rows.  use_g: the build side is S.
// The block takes rows [b0, b0 + DJ_T), then the next DJ_T `stride` further, of
// [0, n); so do the other loops over rows here.
template <typename K, int MODE>
__device__ __forceinline__ void dj_insert_rows(const K* __restrict__ key, const int32_t* __restrict__ pay, int64_t b0,
                                               int64_t n, int64_t stride, const DirectTab<K, MODE>& t, int use_g,
                                               uint2* __restrict__ where, DirectLine* __restrict__ line) {
    const int lane = threadIdx.x & 31;
    bool dup = false;
    for (int64_t b = b0 + threadIdx.x - lane; b < n; b += stride) {
        const int64_t i = b + lane;
        const bool in = i < n;
        const unsigned act = __ballot_sync(0xffffffffu, in);
        if (!in) continue;  // the column's last rows: the warp has no further round
        const K k = key[i];
        int32_t p = 0;
        if (MODE != MODE_COUNT) p = pay ? pay[i] : (int32_t)i;
        const unsigned peers = __match_any_sync(act, k);
        const int leader = __ffs(peers) - 1;
        unsigned long long f = 0;
        if (MODE == MODE_AGG) {
            const unsigned long long mine = use_g ? chk_g(p) : chk_f(p);
            for (unsigned m = peers; m; m &= m - 1) f += __shfl_sync(peers, mine, __ffs(m) - 1);
        }
        uint32_t s = 0, rank = 0;
        if (lane == leader) {
            s = dj_claim<K, MODE>(t, k);
            rank = atomicAdd(t.rows_at(s), (uint32_t)__popc(peers));
            if (MODE == MODE_AGG) atomicAdd(t.sum_at(s), f);
        }
        if (MODE == MODE_EMIT) {
            s = __shfl_sync(peers, s, leader);
            rank = __shfl_sync(peers, rank, leader) + __popc(peers & ((1u << lane) - 1));
            where[i] = make_uint2(s, rank);
            if (rank == 0)
                *t.value_at(s) = (uint32_t)p;
            else
                dup = true;
        }
    }
    if (MODE == MODE_EMIT && dup) line->dup = 1;
}

template <typename K, int MODE>
__global__ void __launch_bounds__(DJ_T)
k_direct_insert(const K* __restrict__ key, const int32_t* __restrict__ pay, int64_t n, DirectTab<K, MODE> t, int use_g,
                uint2* __restrict__ where, DirectSmall* __restrict__ small, const DupHead* __restrict__ dup) {
    if (dj_left(dup)) return;
    dj_insert_rows<K, MODE>(key, pay, (int64_t)blockIdx.x * DJ_T, n, (int64_t)gridDim.x * DJ_T, t, use_g, where,
                            small->lines);
}

// Some key has several rows (nothing to do otherwise): the rank-0 row of a
// key reserves its run and leaves the start in the slot.
template <typename K>
__device__ __forceinline__ void dj_runs_rows(int64_t b0, int64_t n, int64_t stride, const DirectTab<K, MODE_EMIT>& t,
                                             const uint2* __restrict__ where, DirectLine* __restrict__ line) {
    if (!line->dup) return;
    constexpr bool HEAD = DirectSlot<K, MODE_EMIT>::COUNTS_ASIDE;  // runs begin with their length
    const int lane = threadIdx.x & 31;
    for (int64_t b = b0 + threadIdx.x - lane; b < n; b += stride) {
        const int64_t i = b + lane;
        uint2 w = make_uint2(0, 1);
        if (i < n) w = where[i];
        const uint32_t rows = w.y == 0 ? *t.rows_at(w.x) : 0u;
        const uint32_t c = HEAD ? (rows ? rows + 1 : 0u) : (rows > 1 ? rows : 0u);
        const uint32_t incl = warp_incl_scan(c);
        const uint32_t tot = __shfl_sync(0xffffffffu, incl, 31);
        if (tot == 0) continue;
        uint32_t at = 0;
        if (lane == 0) at = (uint32_t)atomicAdd(&line->cursor, (unsigned long long)tot);
        at = __shfl_sync(0xffffffffu, at, 0) + incl - c;
        if (c) {
            *t.value_at(w.x) = at;
            if (HEAD) t.runs[at] = (int32_t)rows;
        }
    }
}

template <typename K>
__global__ void __launch_bounds__(DJ_T)
k_direct_runs(int64_t n, DirectTab<K, MODE_EMIT> t, const uint2* __restrict__ where, DirectSmall* __restrict__ small) {
    dj_runs_rows<K>((int64_t)blockIdx.x * DJ_T, n, (int64_t)gridDim.x * DJ_T, t, where, small->lines);
}

// ... and every row writes its payload into its key's run.
template <typename K>
__device__ __forceinline__ void dj_place_rows(const int32_t* __restrict__ pay, int64_t b0, int64_t n, int64_t stride,
                                              const DirectTab<K, MODE_EMIT>& t, const uint2* __restrict__ where,
                                              const DirectLine* __restrict__ line) {
    if (!line->dup) return;
    constexpr bool HEAD = DirectSlot<K, MODE_EMIT>::COUNTS_ASIDE;
    for (int64_t i = b0 + threadIdx.x; i < n; i += stride) {
        const uint2 w = where[i];
        if (HEAD || *t.rows_at(w.x) > 1) t.runs[*t.value_at(w.x) + HEAD + w.y] = pay ? pay[i] : (int32_t)i;
    }
}

template <typename K>
__global__ void __launch_bounds__(DJ_T)
k_direct_place(const int32_t* __restrict__ pay, int64_t n, DirectTab<K, MODE_EMIT> t, const uint2* __restrict__ where,
               const DirectSmall* __restrict__ small) {
    dj_place_rows<K>(pay, (int64_t)blockIdx.x * DJ_T, n, (int64_t)gridDim.x * DJ_T, t, where, small->lines);
}

// Looks U keys up, a step of all of them in flight together.  m[u]: rows of
// the key (0 where valid[u] is false).  v[u]: emit: the key's value (past a
// run's length word); fs[u]: aggregate: its sum of f.
template <typename K, int MODE, int U>
__device__ __forceinline__ void dj_lookup(const DirectTab<K, MODE>& t, bool dup, const K* k, const bool* valid,
                                          uint32_t* m, uint32_t* v, unsigned long long* fs) {
    using Tab = DirectTab<K, MODE>;
    using Slot = typename Tab::Slot;
    constexpr int B = Tab::B;
    uint32_t at[U];
    bool open[U], more = false;
#pragma unroll
    for (int u = 0; u < U; u++) {
        at[u] = t.home(k[u]);
        open[u] = valid[u];
        m[u] = 0;
        v[u] = 0;
        fs[u] = 0;
        more |= open[u];
    }
    while (more) {
        Slot q[U][B];
#pragma unroll
        for (int u = 0; u < U; u++)
            if (open[u]) dj_bucket<Slot>(t.slots + (size_t)at[u] * B, q[u]);
        more = false;
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (!open[u]) continue;
#pragma unroll
            for (int j = 0; j < B; j++) {
                const K kk = Tab::key(q[u][j]);
                if (open[u] && kk == k[u]) {
                    open[u] = false;
                    if constexpr (MODE == MODE_EMIT && DirectSlot<K, MODE>::COUNTS_ASIDE) {
                        m[u] = 1;
                        v[u] = Tab::value(q[u][j]);
                    } else {
                        m[u] = Tab::rows(q[u][j]);
                        if constexpr (MODE == MODE_EMIT) v[u] = Tab::value(q[u][j]);
                        if constexpr (DirectSlot<K, MODE>::SUMS_ASIDE) v[u] = at[u] * B + j;
                        if constexpr (MODE == MODE_AGG && !DirectSlot<K, MODE>::SUMS_ASIDE)
                            fs[u] = ((unsigned long long)q[u][j].w << 32) | q[u][j].z;
                    }
                } else if (kk == K(0)) {
                    open[u] = false;
                }
            }
            at[u] = t.next(at[u]);
            more |= open[u];
        }
    }
    if constexpr (DirectSlot<K, MODE>::SUMS_ASIDE) {
#pragma unroll
        for (int u = 0; u < U; u++)
            if (m[u]) fs[u] = __ldg(t.sums + v[u]);
    }
    if constexpr (DirectSlot<K, MODE>::COUNTS_ASIDE) {
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (m[u] && k[u] == K(0)) m[u] = t.counts[t.zero_slot()] != 0;
            if (dup && m[u]) {
                m[u] = (uint32_t)t.runs[v[u]];
                v[u]++;
            }
        }
    }
}

// Whether a value is a payload itself rather than a place in `runs`.
template <typename K>
__device__ __forceinline__ bool dj_single(bool dup, uint32_t m) {
    return DirectSlot<K, MODE_EMIT>::COUNTS_ASIDE ? !dup : m == 1;
}

// A part of a long run: the pairs of one probe row with n payloads at src, to
// dst.  The row's warp reserves their place and k_direct_long writes them, a
// warp to a part, so frequent keys load the whole device wherever their probe
// rows lie.  A warp that wrote such runs itself, those of a sorted column one
// after the other, was all that ran: 2^14 x 2^14 rows, a key 4096 times in one
// and in 256 neighbouring rows of the other, 0.81 ms (int64).
struct LongRun {
    int2* dst;
    const int32_t* src;
    uint32_t n_swap;  // n, and in the top bit whether the payloads at src are S's
    int32_t pay;      // the probe row's
};
constexpr uint32_t DJ_LONG = 128;       // rows of a key past which its run is a long one
constexpr uint32_t DJ_LONG_PART = 1024;
static_assert(DJ_LONG_PART > DJ_LONG, "a run of m > DJ_LONG rows has at most m / DJ_LONG parts");

static __global__ void __launch_bounds__(256)
k_direct_long(const LongRun* __restrict__ longs, const unsigned int* __restrict__ count) {
    const uint32_t n = *count, lane = threadIdx.x & 31;
    for (uint32_t w = (blockIdx.x * 256 + threadIdx.x) >> 5; w < n; w += gridDim.x * 8) {
        const LongRun r = longs[w];
        const uint32_t m = r.n_swap & 0x7fffffffu;
        const bool swap = r.n_swap >> 31;
        for (uint32_t e = lane; e < m; e += 32) r.dst[e] = swap ? make_int2(r.pay, r.src[e]) : make_int2(r.src[e], r.pay);
    }
}

// A warp's results on their way out: they collect in shared memory and leave
// DJ_BUF at a time, as one reservation of the output cursor and coalesced
// stores.  No warp waits for another: with a reservation per block and round
// of 256 rows, two barriers around one atomic's latency bound the probe
// (0.57 ms for 2^26 rows and 2^25 pairs, where the lookups take 0.25 ms).
// W 32-bit words per result.  Results past `cap` are counted, not written.
template <int W>
struct WarpOut {
    static constexpr int ROOM = DJ_BUF + 32;  // a round adds at most 32 before the next check
    using T = typename std::conditional<W == 2, int2, int32_t>::type;
    static constexpr int PER = W == 2 ? 1 : W;  // T words per result
    T* buf;                  // ROOM results of this warp
    unsigned long long* cursor;
    T* out;
    unsigned long long cap;
    uint32_t fill;
    // long runs are listed here (NULL: written by the warp).  Room for one part
    // per DJ_LONG results that can be reserved always suffices.
    LongRun* longs = nullptr;
    unsigned int* nlongs = nullptr;
    // where the warp's next n results start; false: they do not fit
    __device__ __forceinline__ bool reserve(unsigned long long n, unsigned long long* at) const {
        unsigned long long a = 0;
        if ((threadIdx.x & 31) == 0) a = atomicAdd(cursor, n);
        *at = __shfl_sync(0xffffffffu, a, 0);
        return *at + n <= cap;
    }
    __device__ __forceinline__ void flush() {
        if (fill == 0) return;
        __syncwarp();
        unsigned long long at;
        if (reserve(fill, &at)) {
            T* o = out + at * PER;
            for (uint32_t q = threadIdx.x & 31; q < fill * PER; q += 32) o[q] = buf[q];
        }
        fill = 0;
        __syncwarp();
    }
    // the slot of this lane's result in the buffer, for the lanes with `have`
    __device__ __forceinline__ T* slot(bool have, unsigned* any) {
        const unsigned b = __ballot_sync(0xffffffffu, have);
        T* q = buf + (fill + __popc(b & ((1u << (threadIdx.x & 31)) - 1))) * PER;
        fill += __popc(b);
        *any = b;
        return q;
    }
    __device__ __forceinline__ void check() {
        if (fill >= (uint32_t)DJ_BUF) flush();
    }
};

// Probes the table with the block's rows (of DJ_U * DJ_T at a time).  Emit:
// pairs go out through `wo`, which keeps what it has not written yet.
// Count and aggregate add to acc and csum.  swap: the build side is S.
//
// Bound by the latency of the bucket reads, so what matters is how many are
// in flight: small blocks at full occupancy, the next rows' keys and payloads
// loading while these are looked up, payloads read whether or not their row
// matches.
template <typename K, int MODE>
__device__ __forceinline__ void dj_probe_rows(const K* __restrict__ key, const int32_t* __restrict__ pay, int64_t b0,
                                              int64_t n, int64_t stride, const DirectTab<K, MODE>& t, int swap,
                                              WarpOut<2>& wo, unsigned long long& acc, unsigned long long& csum) {
    constexpr int U = DJ_U;
    const int lane = threadIdx.x & 31;
    const bool dup = MODE == MODE_EMIT && *t.dup != 0;
    K kn[U];
    int32_t pn[U];
    auto load = [&](int64_t t0) {
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int64_t i = t0 + u * DJ_T + threadIdx.x;
            kn[u] = i < n ? __ldcs(key + i) : K(0);
            if (MODE != MODE_COUNT) pn[u] = pay && i < n ? __ldcs(pay + i) : (int32_t)i;
        }
    };
    int64_t t0 = b0;
    load(t0);
    for (; t0 < n; t0 += stride) {
        K k[U];
        int32_t pp[U];
        bool valid[U];
        uint32_t m[U], v[U];
        unsigned long long fs[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            k[u] = kn[u];
            pp[u] = pn[u];
            valid[u] = t0 + u * DJ_T + threadIdx.x < n;
        }
        load(t0 + stride);
        dj_lookup<K, MODE, U>(t, dup, k, valid, m, v, fs);
        if (MODE == MODE_EMIT) {
#pragma unroll
            for (int u = 0; u < U; u++) {
                if (!__any_sync(0xffffffffu, m[u] > 1)) {  // at most one pair per row
                    unsigned any;
                    int2* q = wo.slot(m[u] != 0, &any);
                    if (m[u]) {
                        const int32_t bp = dj_single<K>(dup, 1) ? (int32_t)v[u] : t.runs[v[u]];
                        *q = swap ? make_int2(pp[u], bp) : make_int2(bp, pp[u]);
                    }
                    wo.check();
                    continue;
                }
                const unsigned long long incl = warp_incl_scan((unsigned long long)m[u]);
                unsigned long long at;
                if (!wo.reserve(__shfl_sync(0xffffffffu, incl, 31), &at)) continue;
                jn_pair* o = reinterpret_cast<jn_pair*>(wo.out) + at + (incl - m[u]);
                if (m[u] <= 4) {
                    for (uint32_t e = 0; e < m[u]; e++) {
                        const int32_t bp = dj_single<K>(dup, m[u]) ? (int32_t)v[u] : t.runs[v[u] + e];
                        st_pair(o + e, swap ? pp[u] : bp, swap ? bp : pp[u]);
                    }
                }
                // long runs are listed, in parts
                const uint32_t parts =
                    wo.longs && m[u] > DJ_LONG ? (m[u] + DJ_LONG_PART - 1) / DJ_LONG_PART : 0u;
                if (__any_sync(0xffffffffu, parts)) {
                    const uint32_t before = warp_incl_scan(parts) - parts;
                    uint32_t q = 0;
                    if (lane == 31) q = atomicAdd(wo.nlongs, before + parts);
                    q = __shfl_sync(0xffffffffu, q, 31) + before;
                    for (uint32_t e = 0; e < parts; e++) {
                        const uint32_t at0 = e * DJ_LONG_PART;
                        wo.longs[q + e] = LongRun{reinterpret_cast<int2*>(o) + at0, t.runs + v[u] + at0,
                                                  min(DJ_LONG_PART, m[u] - at0) | (uint32_t)swap << 31, pp[u]};
                    }
                }
                // a shorter one is written by the whole warp, 32 pairs at a time
                for (unsigned lanes = __ballot_sync(0xffffffffu, m[u] > 4 && !parts); lanes; lanes &= lanes - 1) {
                    const int src = __ffs(lanes) - 1;
                    const uint32_t lm = __shfl_sync(0xffffffffu, m[u], src);
                    const uint32_t lv = __shfl_sync(0xffffffffu, v[u], src);
                    const int32_t lp = __shfl_sync(0xffffffffu, pp[u], src);
                    jn_pair* lo = reinterpret_cast<jn_pair*>(
                        __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(o), src));
                    for (uint32_t e = lane; e < lm; e += 32) {
                        const int32_t bp = t.runs[lv + e];
                        st_pair(lo + e, swap ? lp : bp, swap ? bp : lp);
                    }
                }
            }
        } else {
#pragma unroll
            for (int u = 0; u < U; u++) {
                acc += m[u];
                if (MODE == MODE_AGG && m[u]) csum += fs[u] * (swap ? chk_f(pp[u]) : chk_g(pp[u]));
            }
        }
    }
}

// The single join's probe.  Emit: `segs` segments of `cap` pairs each at out,
// block b to segment b mod segs (the segments' totals count pairs past `cap`
// too).
template <typename K, int MODE>
__global__ void __launch_bounds__(DJ_T, JN_DJ_MINB)
k_direct_probe(const K* __restrict__ key, const int32_t* __restrict__ pay, int64_t n, DirectTab<K, MODE> t, int swap,
               DirectSmall* __restrict__ small, jn_pair* __restrict__ out, uint32_t segs, unsigned long long cap,
               LongRun* __restrict__ longs, const DupHead* __restrict__ dup) {
    constexpr int TILE = DJ_T * DJ_U;
    using Out = WarpOut<2>;
    __shared__ int2 s_buf[MODE == MODE_EMIT ? DJ_T / 32 : 1][MODE == MODE_EMIT ? Out::ROOM : 1];
    if (MODE == MODE_EMIT && dj_left(dup)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) small->lines[0].left = 1;
        return;
    }
    const uint32_t seg = blockIdx.x % segs;
    out += seg * cap;
    Out wo{MODE == MODE_EMIT ? s_buf[threadIdx.x >> 5] : nullptr, &small->lines[seg].total,
           reinterpret_cast<int2*>(out), cap, 0, longs, &small->lines[0].longs};
    unsigned long long acc = 0, csum = 0;
    dj_probe_rows<K, MODE>(key, pay, (int64_t)blockIdx.x * TILE, n, (int64_t)gridDim.x * TILE, t, swap, wo, acc, csum);
    if (MODE == MODE_EMIT) {
        wo.flush();
    } else {
        __shared__ unsigned long long tmp[33];
        acc = block_sum(acc, tmp);
        if (MODE == MODE_AGG) csum = block_sum(csum, tmp);
        if (threadIdx.x == 0) {
            if (acc) atomicAdd(&small->lines[0].total, acc);
            if (MODE == MODE_AGG && csum) atomicAdd(&small->lines[0].chk, csum);
        }
    }
}

// Results per segment, by value: the counters' scratch may be reused already
// when the gather runs.
struct DirectCounts {
    unsigned long long n[DJ_SEGS];
};

// Where a partition join's pairs go.  Work item i's pairs belong to segment
// i % segs: its own part of scratch in the first pass or, once the segments'
// pairs are counted, of the output.  A launch takes the segments [lo, lo + w);
// its grid is a multiple of w, so a block stays with one segment.
struct PairSegs {
    uint32_t segs, lo, w;
    unsigned long long at[DJ_SEGS], cap[DJ_SEGS];
    __device__ __forceinline__ uint32_t seg() const { return lo + blockIdx.x % w; }
    __device__ __forceinline__ uint64_t first() const { return (uint64_t)(blockIdx.x / w) * segs + seg(); }
    __device__ __forceinline__ uint64_t step() const { return (uint64_t)(gridDim.x / w) * segs; }
};

// The segments of staged results, one after the other, into out.  PER words
// of type T per result.
template <typename T, int PER>
__global__ void __launch_bounds__(256)
k_direct_gather(const T* __restrict__ staged, uint32_t segs, uint64_t cap, DirectCounts counts, T* __restrict__ out) {
    constexpr int V = 4;
    const uint64_t stride = (uint64_t)gridDim.x * 256;
    for (uint32_t r = 0; r < segs; r++) {
        const uint64_t n = counts.n[r] * PER;
        const T* src = staged + r * cap * PER;
        for (uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += V * stride) {
            T v[V];
#pragma unroll
            for (int e = 0; e < V; e++)
                if (i + e * stride < n) v[e] = __ldcs(src + i + e * stride);
#pragma unroll
            for (int e = 0; e < V; e++)
                if (i + e * stride < n) out[i + e * stride] = v[e];
        }
        out += n;
    }
}

// Host side of a build: sizes, layout and launches.
//
// Build rows at most DJ_MAX, where the table reaches L2's size (64 MB of
// 8-byte slots, 128 MB of 16-byte ones).  Measured on GB300 against the
// better of the partition paths, half of the probe rows matching, ms for
// build x probe rows: int32, pairs written: 2^20 x 2^26 0.78 / 1.34, 2^22 x
// 2^22 0.30 / 0.49, 2^22 x 2^26 0.89 / 1.37, but 2^23 x 2^25 1.19 / 1.05 (the
// keys without repeats; with them see DupRule);
// counted: 2^22 x 2^26 0.51 / 1.19; int64, pairs: 2^22 x 2^22 0.34 / 0.66,
// 2^22 x 2^26 1.23 / 2.60; checksum: 2^22 x 2^24 0.71 / 0.98, but 2^23 x
// 2^25 1.71 / 1.64.  2^16 x 2^18: 0.07 / 0.19.
#ifndef JN_DJ_MAX
#define JN_DJ_MAX (1ull << 22)
#endif
constexpr uint64_t DJ_MAX = JN_DJ_MAX;

// Buckets of a table of n rows: twice the rows in slots (load one half at
// most), three times for tables far below L2's size.
template <typename K, int MODE>
inline uint32_t dj_buckets(uint64_t n) {
    constexpr int B = DirectSlot<K, MODE>::B;
    return (uint32_t)(((n < (1u << 19) ? 3 : 2) * n + B - 1) / B + 8);
}

// Bytes of a table's parts, each rounded to 256 bytes.  Slots, counts and
// sums start as zeros; `where` and `runs` (emit) need no value.
template <typename K, int MODE>
struct DirectLayout {
    size_t slots, counts, sums, where, runs;
    explicit DirectLayout(uint64_t n) {
        auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
        using DS = DirectSlot<K, MODE>;
        const size_t ns = ((size_t)dj_buckets<K, MODE>(n) + 1) * DS::B;
        slots = up(ns * sizeof(typename DS::T));
        counts = DS::COUNTS_ASIDE ? up(ns * sizeof(uint32_t)) : 0;
        sums = DS::SUMS_ASIDE ? up(ns * sizeof(unsigned long long)) : 0;
        where = MODE == MODE_EMIT ? up(n * sizeof(uint2)) : 0;
        runs = MODE == MODE_EMIT ? up((DS::COUNTS_ASIDE ? 2 : 1) * n * sizeof(int32_t)) : 0;  // and the lengths
    }
    size_t zeroed() const { return slots + counts + sums; }
    size_t bytes() const { return zeroed() + where + runs; }
};

// Launches of one table's build in `mem` (already zeroed up to lay.zeroed()).
template <typename K, int MODE>
jn_status direct_build(jn_ctx* c, const Cols<K>& B, int use_g, const DirectLayout<K, MODE>& lay, unsigned char* mem,
                       DirectSmall* small, DirectTab<K, MODE>* t, const DupHead* dup = nullptr) {
    t->slots = reinterpret_cast<typename DirectTab<K, MODE>::Slot*>(mem);
    t->nb = dj_buckets<K, MODE>((uint64_t)B.n);
    t->counts = reinterpret_cast<uint32_t*>(mem + lay.slots);
    t->sums = reinterpret_cast<unsigned long long*>(mem + lay.slots + lay.counts);
    uint2* where = reinterpret_cast<uint2*>(mem + lay.zeroed());
    t->runs = reinterpret_cast<int32_t*>(mem + lay.zeroed() + lay.where);
    t->dup = &small->lines[0].dup;
    const dim3 g((unsigned)std::min<uint64_t>(ceil_div((uint64_t)B.n, DJ_T), (uint64_t)c->num_sms * 8));
    JN_TRY(launch(c, K_DIRECT_BUILD, k_direct_insert<K, MODE>, g, dim3(DJ_T), 0, B.key, B.pay, B.n, *t, use_g, where,
                  small, dup));
    if constexpr (MODE == MODE_EMIT) {
        JN_TRY(launch(c, K_DIRECT_BUILD, k_direct_runs<K>, g, dim3(DJ_T), 0, B.n, *t, (const uint2*)where, small));
        JN_TRY(launch(c, K_DIRECT_BUILD, k_direct_place<K>, g, dim3(DJ_T), 0, B.pay, B.n, *t, (const uint2*)where,
                      (const DirectSmall*)small));
    }
    return JN_OK;
}

// Staged results of a probe of np rows: segments and results per segment, with
// room for `quarters` quarters of a result a row.  Blocks take rows in turn, so
// segments fill evenly.  Pairs past their room are found a second time, so the
// room is for two rows a key and a little more, as random keys have it (int32,
// 2^20 x 2^24, two a key: 0.63 ms, 1.02 with five quarters; 0.77 partitioned).
constexpr uint32_t DJ_ROOM = 9, DJ_ROOM_LEAST = 5;  // quarters
struct DirectStage {
    uint32_t segs;
    uint64_t cap;
    DirectStage(uint64_t np, uint32_t quarters) {
        segs = np >= (1u << 23) ? DJ_SEGS : 1;
        cap = np * quarters / 4 / segs + 1024;
    }
    uint64_t room() const { return segs * cap; }
};

// What a probe left in the counters.
struct DirectResult {
    DirectCounts counts;
    uint64_t total = 0, chk = 0, first = 0;
    bool fits = true;  // every segment's results fit its room
    bool dup = false;  // some build key has several rows
    bool left = false;
    uint32_t longs = 0;
};
// Queues the counters' copy to the host; after the stream is synchronised,
// direct_parse reads them.
constexpr int DJ_HWORD = 8;   // where they land in the context's pinned words
constexpr int DJ_LINE_WORDS = 6;  // words of a line that matter here
inline jn_status direct_fetch(jn_ctx* c, const DirectSmall* small, uint32_t segs) {
    constexpr int W = DJ_LINE_WORDS;
    static_assert(DJ_HWORD + W * DJ_SEGS < 63, "the last pinned word is read_back's error word");
    JN_CUDA(c, cudaMemcpy2DAsync(c->h_small + DJ_HWORD, W * 8, small, sizeof(DirectLine), W * 8, segs,
                                 cudaMemcpyDeviceToHost, c->stream));
    return JN_OK;
}
inline void direct_parse(const jn_ctx* c, uint32_t segs, uint64_t cap, DirectResult* r) {
    const uint64_t* h = c->h_small + DJ_HWORD;
    for (uint32_t i = 0; i < segs; i++) {
        r->counts.n[i] = h[DJ_LINE_WORDS * i];
        r->total += r->counts.n[i];
        r->fits &= r->counts.n[i] <= cap;
    }
    r->chk = h[1];
    r->first = h[2];
    r->dup = (h[4] & 0xffffffffu) != 0;
    r->longs = (uint32_t)(h[4] >> 32);
    r->left = (h[5] & 0xffffffffu) != 0;
}
inline jn_status direct_result(jn_ctx* c, const DirectSmall* small, uint32_t segs, uint64_t cap, DirectResult* r) {
    JN_TRY(direct_fetch(c, small, segs));
    JN_CUDA(c, cudaStreamSynchronize(c->stream));
    direct_parse(c, segs, cap, r);
    return JN_OK;
}

// Writes the long runs that a probe listed.
inline jn_status direct_long(jn_ctx* c, const LongRun* longs, const unsigned int* count) {
    return launch(c, K_DIRECT_PROBE, k_direct_long, dim3(8 * (unsigned)c->num_sms), dim3(256), 0, longs, count);
}

template <typename T, int PER>
jn_status direct_gather(jn_ctx* c, int kid, const void* staged, uint32_t segs, uint64_t cap, const DirectResult& r,
                        void* out) {
    const dim3 g((unsigned)std::min<uint64_t>(ceil_div(r.total * PER, 1024), 8 * (uint64_t)c->num_sms));
    return launch(c, kid, k_direct_gather<T, PER>, g, dim3(256), 0, static_cast<const T*>(staged), segs, cap, r.counts,
                  static_cast<T*>(out));
}

// Whether the context's tuning leaves the choice of path to the library.
inline bool direct_allowed(const jn_ctx* c) {
    const jn_tuning& t = c->tune;
    return t.hash_path == 0 && t.radix_bits == 0 && t.radix_bits1 == 0 && t.filter_bits == 0 && t.prefilter == -1 &&
           t.heavy == -1 && t.table_rows == 0;
}

}  // namespace jnx
