// Sort-merge equi join of one hash partition pair: the third category of
// join algorithms in Sec. 2.3 (sort both tables, then walk them in order),
// beside the nested-loop and hash joins the paper builds.
//
// It takes the same work items as the hash join kernel: a chunk of at most
// cap R rows of one partition against every S row of that partition.
// k_sort_chunks sorts every R chunk once (bitonic network in registers and
// shared memory) into a copy of the partitioned rows; k_sort_join then stages
// the sorted chunk and each S row finds its run of equal R keys by binary
// search, which is the merge step done per probe row instead of by a second
// sorted stream.
//   count: the sum over S rows of the run lengths;
//   agg:   as count, and the sum over matches of f(r) * g(s), from a prefix
//          sum of f over the sorted run order;
//   emit:  a warp finds the runs of 256 S rows, reserves room for all their
//          pairs in a segment of scratch with one addition and writes them:
//          no counting pass goes before it.
//
// Order.  Inside a partition any order will do that R and S agree on.  An
// int32 key is ordered by the bits of its hash below the partition's (the
// hash is a product with an odd number, so equal bits inside a partition mean
// equal keys).  From 2^12 partitions on, that leaves 20 bits and the row's
// number in the chunk fits beneath them: the network then moves one 32-bit
// word per row, and 64-bit words only for tables of few partitions.
//
// The sort is held by shuffles and shared memory, the join by shared memory
// (dependent lookups: eleven to find a run among 2000 rows), so a thread
// searches for four S rows at a time and three blocks share an SM.  Measured
// on GB300, 1.6e7 x 4e7 int32 rows, 2.8e7 of S left by the filter, 2.4e7
// pairs: sort 0.21 ms (0.66 with 64-bit words and a trip through shared
// memory per step), pairs 0.45 with their copy (a counting pass of 0.26 and a
// writing pass of 0.33, searching twice, without sj_swz); eight S rows at a
// time in two blocks: 0.48.
#pragma once

#include "jn_common.cuh"
#include "jn_direct.cuh"
#include "jn_partition.cuh"

namespace jnx {

#ifndef JN_SC_MINB
#define JN_SC_MINB 3
#endif
#ifndef JN_SJ_PER
#define JN_SJ_PER 4
#endif
#ifndef JN_SJ_MINB
#define JN_SJ_MINB 3
#endif
constexpr int SJ_T = 512;      // threads per sort-merge block
constexpr int SJ_IDX = 12;     // bits of a row's number in its chunk
constexpr int SJ_CHUNK = 1 << SJ_IDX;  // rows of the largest chunk
static_assert(8 * SJ_T == SJ_CHUNK, "eight rows per thread");

// What a partition is sorted by: the low bits of an int32 key's hash, the
// order-preserving unsigned image of an int64 key.
__device__ __forceinline__ uint32_t sj_ord(int32_t k, int bits) { return khash(k) << bits; }
__device__ __forceinline__ uint64_t sj_ord(int64_t k, int) { return (uint64_t)k ^ 0x8000000000000000ull; }

// Where word i of a sorted chunk lies: the binary search visits positions a
// power of two apart, which without this share a bank (20 to 28 lanes of a
// warp on one bank at the five middle steps of a 4096-row chunk).
__device__ __forceinline__ uint32_t sj_swz(uint32_t i) { return i ^ (((i >> 5) ^ (i >> 7)) & 31u); }

template <typename K>
struct SortJoinSmem {
    using U = typename std::conditional<sizeof(K) == 4, uint32_t, uint64_t>::type;
    // sort pass, int32 keys: words of W bytes and payloads; int64 keys: keys,
    // row numbers and payloads
    static size_t sort_bytes(int cap, bool narrow) {
        return sizeof(K) == 4 ? (size_t)cap * ((narrow ? 4 : 8) + sizeof(int32_t)) + 16
                              : (size_t)cap * (sizeof(U) + sizeof(uint16_t) + sizeof(int32_t)) + 16;
    }
    // join passes: the sorted chunk's keys (whole groups of 32) and payloads,
    // and (aggregate mode) the prefix sum of f over it
    __host__ __device__ static constexpr int keys(int cap) { return (cap + 31) & ~31; }
    static size_t bytes(int cap, int mode) {
        return (size_t)keys(cap) * sizeof(U) + (size_t)cap * sizeof(int32_t) +
               (mode == MODE_AGG ? (size_t)(cap + 1) * sizeof(unsigned long long) : 0) + 16;
    }
};

// Sorts R rows [rbeg, rbeg + rn) of every item by sj_ord(key) into `sorted`
// (same positions; the key is replaced by sj_ord(key)).  int64 keys.  Shared
// memory: SortJoinSmem<K>::sort_bytes(cap).
template <typename K>
__global__ void __launch_bounds__(SJ_T)
k_sort_chunks(const Row<K, false>* __restrict__ rrows, Row<K, false>* __restrict__ sorted,
              const Item* __restrict__ items, const uint64_t* __restrict__ nitems_p, int cap, int bits) {
    using U = typename SortJoinSmem<K>::U;
    extern __shared__ __align__(128) unsigned char smem[];
    U* s_k = reinterpret_cast<U*>(smem);
    int32_t* s_pay = reinterpret_cast<int32_t*>(s_k + cap);
    uint16_t* s_i = reinterpret_cast<uint16_t*>(s_pay + cap);
    constexpr uint16_t PAD = 0x8000u;
    const uint64_t nitems = *nitems_p;
    for (uint64_t it = blockIdx.x; it < nitems; it += gridDim.x) {
        const Item d = items[it];  // every item owns one R chunk
        const int rn = d.rn;
        int n2 = 1;
        while (n2 < rn) n2 <<= 1;
        for (int i = threadIdx.x; i < n2; i += SJ_T) {
            if (i < rn) {
                const Row<K, false> x = rrows[d.rbeg + i];
                s_k[i] = sj_ord(x.key, bits);
                s_pay[i] = x.pay;
                s_i[i] = (uint16_t)i;
            } else {
                s_k[i] = ~(U)0;
                s_i[i] = (uint16_t)(PAD | i);
            }
        }
        __syncthreads();
        for (int k = 2; k <= n2; k <<= 1) {
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int t = threadIdx.x; t < (n2 >> 1); t += SJ_T) {
                    const int a = 2 * j * (t / j) + (t % j), b = a + j;
                    const U ka = s_k[a], kb = s_k[b];
                    const uint16_t ia = s_i[a], ib = s_i[b];
                    const bool gt = ka > kb || (ka == kb && (ia & PAD) > (ib & PAD));
                    if (gt == ((a & k) == 0)) {
                        s_k[a] = kb;
                        s_k[b] = ka;
                        s_i[a] = ib;
                        s_i[b] = ia;
                    }
                }
                __syncthreads();
            }
        }
        for (int i = threadIdx.x; i < rn; i += SJ_T) {
            Row<K, false> x{};
            x.key = (K)s_k[i];
            x.pay = s_pay[s_i[i] & (PAD - 1)];
            sorted[d.rbeg + i] = x;
        }
        __syncthreads();
    }
}

// One merge step of the network on the 8 consecutive words a thread holds
// (word i = 8 * thread + e), partners j < 256 apart: 8 or more apart they sit
// in another lane of the warp, closer ones in the same thread.  Ascending: a
// descending block holds its words inverted.
template <typename W, int J>
__device__ __forceinline__ void sj_step(W (&v)[8]) {
    const bool lower = ((threadIdx.x << 3) & J) == 0;
#pragma unroll
    for (int e = 0; e < 8; e++) {
        if (J >= 8) {
            const W o = __shfl_xor_sync(0xffffffffu, v[e], J >> 3);
            v[e] = lower ? min(v[e], o) : max(v[e], o);
        } else if (!(e & J)) {
            const W x = v[e], y = v[e | (J & 7)];
            v[e] = min(x, y);
            v[e | (J & 7)] = max(x, y);
        }
    }
}

// The steps j = J, J / 2, .. 1.
template <typename W, int J>
__device__ __forceinline__ void sj_steps(W (&v)[8]) {
    sj_step<W, J>(v);
    if constexpr (J > 1) sj_steps<W, J / 2>(v);
}

// Blocks of up to 256 words, K2 of them at a time, from blocks half as long.
template <typename W, int K2>
__device__ __forceinline__ void sj_warp_sort(W (&v)[8]) {
    if constexpr (K2 > 2) sj_warp_sort<W, K2 / 2>(v);
#pragma unroll
    for (int e = 0; e < 8; e++)
        if ((8 * threadIdx.x + e) & K2) v[e] = ~v[e];
    sj_steps<W, K2 / 2>(v);
#pragma unroll
    for (int e = 0; e < 8; e++)
        if ((8 * threadIdx.x + e) & K2) v[e] = ~v[e];
}

// int32 keys.  A word is the key's order, above a padding flag (64-bit words)
// and the row's number.  Blocks of 256 words are sorted inside a warp; steps
// with j >= 256 go through shared memory, where a thread takes the words 256
// apart and does up to three of them at a time: five trips for a chunk of
// 4096 rows.  Padding words are all ones (a row with an all-ones word is the
// last of a chunk without padding).
template <typename W>
__global__ void __launch_bounds__(SJ_T, sizeof(W) == 4 ? JN_SC_MINB : 2)
k_sort_chunks32(const Row<int32_t, false>* __restrict__ rrows, Row<int32_t, false>* __restrict__ sorted,
                const Item* __restrict__ items, const uint64_t* __restrict__ nitems_p, int cap, int bits) {
    extern __shared__ __align__(128) unsigned char smem[];
    W* s_v = reinterpret_cast<W*>(smem);  // cap words
    int32_t* s_pay = reinterpret_cast<int32_t*>(s_v + cap);
    constexpr bool NARROW = sizeof(W) == 4;
    constexpr W IDX = (W)(SJ_CHUNK - 1);
    const int t = threadIdx.x;
    const uint64_t nitems = *nitems_p;
    // a warp reads or writes its 8 x 32 words without bank conflicts
    auto at = [](int i) { return i ^ ((i >> 5) & 7); };
    for (uint64_t it = blockIdx.x; it < nitems; it += gridDim.x) {
        const Item d = items[it];  // every item owns one R chunk
        const int rn = d.rn;
        int n2 = 256;  // one warp's 8 x 32 words at least
        while (n2 < rn) n2 <<= 1;
        const int nt = n2 >> 3;
        const bool act = t < nt;  // whole warps: n2 is a multiple of 256
        W v[8];
        if (act) {
#pragma unroll
            for (int e = 0; e < 8; e++) {
                const int i = e * nt + t;  // which word a row starts in does not matter
                v[e] = ~(W)0;
                if (i < rn) {
                    const Row<int32_t, false> x = rrows[d.rbeg + i];
                    s_pay[i] = x.pay;
                    const uint32_t o = sj_ord(x.key, bits);
                    v[e] = NARROW ? (W)(o | (uint32_t)i) : ((W)o << (NARROW ? 0 : 16)) | (W)i;
                }
            }
            sj_warp_sort<W, 256>(v);
        }
        for (int k = 512; k <= n2; k <<= 1) {
            if (act) {
                const bool inv = ((8 * t) & k) != 0;
#pragma unroll
                for (int e = 0; e < 8; e++) s_v[at(8 * t + e)] = inv ? ~v[e] : v[e];
            }
            __syncthreads();
            if (k == SJ_CHUNK) {
                for (int a = t; a < SJ_CHUNK / 2; a += SJ_T) {
                    const W x = s_v[at(a)], y = s_v[at(a + SJ_CHUNK / 2)];
                    s_v[at(a)] = min(x, y);
                    s_v[at(a + SJ_CHUNK / 2)] = max(x, y);
                }
                __syncthreads();
            }
            const int base = (t & 255) + 2048 * (t >> 8);
            if (base < n2) {
                W w[8];
#pragma unroll
                for (int e = 0; e < 8; e++) w[e] = base + 256 * e < n2 ? s_v[at(base + 256 * e)] : ~(W)0;
#pragma unroll
                for (int J = 4; J > 0; J >>= 1) {
                    if (256 * J > (k >> 1)) continue;
#pragma unroll
                    for (int e = 0; e < 8; e++) {
                        if (e & J) continue;
                        const W x = w[e], y = w[e | J];
                        w[e] = min(x, y);
                        w[e | J] = max(x, y);
                    }
                }
#pragma unroll
                for (int e = 0; e < 8; e++)
                    if (base + 256 * e < n2) s_v[at(base + 256 * e)] = w[e];
            }
            __syncthreads();
            if (act) {
                const bool inv = ((8 * t) & k) != 0;
#pragma unroll
                for (int e = 0; e < 8; e++) v[e] = s_v[at(8 * t + e)];
                sj_steps<W, 128>(v);
                if (inv) {
#pragma unroll
                    for (int e = 0; e < 8; e++) v[e] = ~v[e];
                }
            }
            // the next trip's writes go where this thread just read
        }
        if (act) {
#pragma unroll
            for (int e = 0; e < 8; e++) s_v[at(8 * t + e)] = v[e];
        }
        __syncthreads();
        for (int i = t; i < rn; i += SJ_T) {
            const W w = s_v[at(i)];
            Row<int32_t, false> x;
            x.key = (int32_t)(NARROW ? (uint32_t)(w & ~IDX) : (uint32_t)(w >> (NARROW ? 0 : 16)));
            x.pay = s_pay[(int)(w & IDX)];
            sorted[d.rbeg + i] = x;
        }
        __syncthreads();  // shared arrays are rewritten by the next chunk
    }
}

template <typename K, int MODE>
__global__ void __launch_bounds__(SJ_T, JN_SJ_MINB)
k_sort_join(const Row<K, false>* __restrict__ rrows, const Row<K, false>* __restrict__ srows,
            const Item* __restrict__ items, const uint64_t* __restrict__ nitems_p, int cap_rows, int bits,
            DirectSmall* __restrict__ small, jn_pair* __restrict__ out, const __grid_constant__ PairSegs ps) {
    using U = typename SortJoinSmem<K>::U;
    extern __shared__ __align__(128) unsigned char smem[];
    U* s_k = reinterpret_cast<U*>(smem);
    const int nk = SortJoinSmem<K>::keys(cap_rows);
    unsigned long long* s_f = reinterpret_cast<unsigned long long*>(s_k + nk);  // agg only
    int32_t* s_pay = reinterpret_cast<int32_t*>(MODE == MODE_AGG ? reinterpret_cast<unsigned char*>(s_f + cap_rows + 1)
                                                                 : reinterpret_cast<unsigned char*>(s_k + nk));
    __shared__ unsigned long long tmp64[33];
    constexpr int PER = JN_SJ_PER;  // S rows a thread searches for at once
    const int tid = threadIdx.x, lane = tid & 31;
    const uint64_t nitems = *nitems_p;
    const uint32_t seg = ps.seg();
    const unsigned long long cap = ps.cap[seg];
    jn_pair* const gout = out + ps.at[seg];
    unsigned long long acc = 0, csum = 0;
    const uint64_t next = ps.step();
    for (uint64_t it = ps.first(); it < nitems; it += next) {
        const Item d = items[it];
        const uint32_t rn = (uint32_t)d.rn;
        const uint32_t sn = (uint32_t)d.sn;  // below 2^31: a row number and a round past it fit 32 bits
        for (uint32_t i = tid; i < rn; i += SJ_T) {  // the chunk, sorted by key
            const Row<K, false> x = rrows[d.rbeg + i];
            s_k[sj_swz(i)] = (U)x.key;
            s_pay[i] = x.pay;
        }
        __syncthreads();
        if (MODE == MODE_AGG) {
            // s_f[e] = sum of f(payload) over sorted positions < e, e <= rn
            const uint32_t base = tid * 8;
            unsigned long long v[8], sum = 0;
#pragma unroll
            for (int q = 0; q < 8; q++) {
                v[q] = base + q < rn ? chk_f(s_pay[base + q]) : 0ull;
                sum += v[q];
            }
            unsigned long long tot;
            unsigned long long pre = block_excl_scan(sum, tmp64, &tot);
            if (tid == 0) s_f[0] = 0;
#pragma unroll
            for (int q = 0; q < 8; q++) {
                pre += v[q];
                if (base + q < rn) s_f[base + q + 1] = pre;
            }
            __syncthreads();
        }
        uint32_t top = 1;  // the largest power of two in rn
        while (2 * top <= rn) top <<= 1;
        // a warp takes groups of 256 consecutive S rows
        const Row<K, false>* sp = srows + d.sbeg;
        for (uint32_t g = (tid >> 5) * 32 * PER; g < sn; g += SJ_T * PER) {
            U q[PER];
            int32_t spay[PER];
            uint32_t lo[PER], m[PER];
#pragma unroll
            for (int e = 0; e < PER; e++) {
                const uint32_t j = g + e * 32 + lane;
                lo[e] = 0;
                m[e] = 0;
                q[e] = 0;
                spay[e] = 0;
                if (j < sn) {
                    const Row<K, false> x = sp[j];
                    q[e] = sj_ord(x.key, bits);
                    spay[e] = x.pay;
                }
            }
            // rows before the first that is not below q: PER searches in step
            for (uint32_t step = top; step; step >>= 1) {
#pragma unroll
                for (int e = 0; e < PER; e++) {
                    const uint32_t p = lo[e] + step;
                    if (p <= rn && s_k[sj_swz(p - 1)] < q[e]) lo[e] = p;
                }
            }
            uint32_t sum = 0;
#pragma unroll
            for (int e = 0; e < PER; e++) {
                if (g + e * 32 + lane < sn && lo[e] < rn && s_k[sj_swz(lo[e])] == q[e]) {
                    // the run's length: by doubling, then by halving
                    uint32_t a = 1, step = 1;
                    while (lo[e] + a < rn && s_k[sj_swz(lo[e] + a)] == q[e]) {
                        step = a;
                        a = min(2 * a, rn - lo[e]);
                    }
                    // rows [lo, lo + b) are known equal; the run ends in (b, a]
                    uint32_t b = step, c = a;
                    while (b < c) {
                        const uint32_t mid = (b + c) >> 1;
                        if (s_k[sj_swz(lo[e] + mid)] == q[e]) b = mid + 1; else c = mid;
                    }
                    m[e] = b;
                    if (MODE == MODE_AGG) csum += (s_f[lo[e] + b] - s_f[lo[e]]) * chk_g(spay[e]);
                }
                sum += m[e];
            }
            if (MODE != MODE_EMIT) {
                acc += sum;
                continue;
            }
            sum = __reduce_add_sync(0xffffffffu, sum);
            if (sum == 0) continue;
            unsigned long long o = 0;
            if (lane == 0) o = atomicAdd(&small->lines[seg].total, (unsigned long long)sum);
            o = __shfl_sync(0xffffffffu, o, 0);
            if (o + sum > cap) continue;  // counted; the caller makes room and asks again
#pragma unroll
            for (int e = 0; e < PER; e++) {
                const uint32_t incl = warp_incl_scan(m[e]);
                const uint32_t wt = __shfl_sync(0xffffffffu, incl, 31);
                const unsigned long long oe = o + (incl - m[e]);
                o += wt;
                // short runs by their lane, long runs by the whole warp
                const bool longr = m[e] > 4;
                if (!longr)
                    for (uint32_t r = 0; r < m[e]; r++) st_pair(gout + oe + r, s_pay[lo[e] + r], spay[e]);
                for (unsigned lanes = __ballot_sync(0xffffffffu, longr); lanes; lanes &= lanes - 1) {
                    const int src = __ffs(lanes) - 1;
                    const uint32_t bm = __shfl_sync(0xffffffffu, m[e], src);
                    const uint32_t bl = __shfl_sync(0xffffffffu, lo[e], src);
                    const int32_t bp = __shfl_sync(0xffffffffu, spay[e], src);
                    const unsigned long long bo = __shfl_sync(0xffffffffu, oe, src);
                    for (uint32_t r = lane; r < bm; r += 32) st_pair(gout + bo + r, s_pay[bl + r], bp);
                }
            }
        }
        __syncthreads();  // the chunk's shared arrays are rewritten by the next item
    }
    if (MODE == MODE_EMIT) return;
    acc = block_sum(acc, tmp64);
    if (MODE == MODE_AGG) csum = block_sum(csum, tmp64);
    if (tid == 0) {
        if (acc) atomicAdd(&small->lines[seg].total, acc);
        if (MODE == MODE_AGG && csum) atomicAdd(&small->lines[0].chk, csum);
    }
}

}  // namespace jnx
