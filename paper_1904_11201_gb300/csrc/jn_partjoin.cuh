// Join of one hash partition pair in shared memory (the join kernel of the
// partitioned hash join).
//
// A work item is a chunk of R rows of one partition against every S row of
// that partition.  The R rows are staged in shared memory (one TMA bulk copy)
// and stay there; the hash table over them is an array of 4-byte entries
// (16 bits of the key's hash, row number), so inserting a row whose key is new
// costs one compare-and-swap and nothing else.  Rows that meet their key
// again count at the key's first row.  S rows are read by the threads that
// probe with them, the first of them before the table is built, so no barrier
// stands between the probing warps.
//   count:     rows of a key = 1 + the count at its first row;
//   aggregate: and f of the first row's payload + the sum of f of the others;
//   emit:      a key with several rows gets its payloads as one run, placed by
//              the ranks that the counting returned.  Pairs leave in WarpOut's
//              manner (jn_direct.cuh) to segments of scratch, once: there is
//              no second pass over the rows to write what a first one counted.
//
// The pass is held by shared-memory latency (dependent compare-and-swaps and
// lookups), so a block is kept small enough, in shared memory and registers,
// for three (emit) or four (count, aggregate) on an SM where its table is
// fitted to the partitions (run_hash); they cover each other's staging and
// barriers.  A full table of 4096 int32 rows leaves two blocks (107 KB; checksum
// one, 123 KB), one of 2048 int64 rows two: with the full table asked for, int32
// pairs go to k_hash_join.  One S row at a time per thread beats two to
// four with fewer blocks.  Measured on GB300, 2^28 x 2^28 uniform int32 rows:
// count 1.42 ms (1.65 with the kernel it replaced), checksum 2.49 (4.22), pairs
// 4.82 with the copy (1.65 + 3.24); 2^26 x 2^26, unique R keys, half matching:
// count 0.29 (0.44), checksum 0.42 (1.08), pairs 0.52 (0.44 + 0.77); int64:
// 0.74 (0.95), 0.90 (2.07), 1.19 (0.95 + 2.86).
#pragma once

#include "jn_async.cuh"
#include "jn_direct.cuh"
#include "jn_partition.cuh"

namespace jnx {

#ifndef JN_PJ_MINB
#define JN_PJ_MINB 4
#endif
#ifndef JN_PJ_ENT
#define JN_PJ_ENT 5  // entries per two rows of a full table
#endif
#ifndef JN_PJ_MINBE
#define JN_PJ_MINBE 3
#endif
constexpr int PJ_T = 512;          // threads per block
constexpr int PJ_BUF = 64;         // pairs a warp collects before it writes them
constexpr uint32_t PJ_EMPTY = 0xFFFFFFFFu;  // no entry: a row number is below 2^15

// First entry of a key hash: the bits below the partition's.  The hash is a
// multiple of the golden ratio (modulo 2^32), so the keys of a dense integer
// range that fall into a partition lie evenly spaced over those bits (the
// three-distance theorem) and rarely meet; mixing the bits again made the
// pass 1.5 times as long, and a second product 1.2 times.
__device__ __forceinline__ uint32_t pj_slot(uint32_t h, int bits, int ts) { return __umulhi(h << bits, (uint32_t)ts); }

template <typename K, int MODE>
struct PartJoinSmem {
    using R = Row<K, false>;
    // staged rows (16-byte widened), entries, counts, then the warps' output
    // buffers (emit) or sums of f, low and high words (aggregate)
    __host__ __device__ static constexpr int entries(int cap) { return JN_PJ_ENT * cap / 2; }
    __host__ __device__ static constexpr size_t rows(int cap) { return (size_t)(cap + 2) * sizeof(R) + 32; }
    static constexpr size_t bytes(int cap) {
        return rows(cap) + (size_t)entries(cap) * 4 + (size_t)cap * 4 +
               (MODE == MODE_EMIT ? (PJ_T / 32) * 2 * PJ_BUF * sizeof(int2)
                : MODE == MODE_AGG ? (size_t)cap * 8
                                   : 0);
    }
};

template <typename K, int MODE>
__global__ void __launch_bounds__(PJ_T, MODE == MODE_EMIT ? JN_PJ_MINBE : JN_PJ_MINB)
k_part_join(const Row<K, false>* __restrict__ rrows, const Row<K, false>* __restrict__ srows,
            const Item* __restrict__ items, const uint64_t* __restrict__ nitems_p, int cap_rows, int bits,
            DirectSmall* __restrict__ small, jn_pair* __restrict__ out, const __grid_constant__ PairSegs ps,
            unsigned int* __restrict__ err) {
    using R = Row<K, false>;
    using L = PartJoinSmem<K, MODE>;
    extern __shared__ __align__(128) unsigned char smem[];
    uint32_t* s_ent = reinterpret_cast<uint32_t*>(smem + L::rows(cap_rows));
    uint32_t* s_cnt = s_ent + L::entries(cap_rows);  // per first row: further rows (emit with runs: rows << 16 | start)
    int2* s_out = reinterpret_cast<int2*>(s_cnt + cap_rows);
    uint32_t* s_flo = s_cnt + cap_rows;
    uint32_t* s_fhi = s_flo + cap_rows;
    __shared__ unsigned long long tmp64[33];
    __shared__ uint32_t tmp32[33];
    __shared__ __align__(8) uint64_t bar;
    constexpr int PER = 8;  // R rows per thread: a chunk is at most 8 * PJ_T rows
    constexpr int PU = 1;   // S rows a thread loads at once (two to four measured slower)
    const int tid = threadIdx.x, lane = tid & 31;
    const uint64_t nitems = *nitems_p;
    const uint32_t seg = ps.seg();
    const uint64_t first_item = ps.first(), step = ps.step();
    const unsigned long long cap = ps.cap[seg];
    if (tid == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    // the warp's pairs on their way out
    int2* const buf = MODE == MODE_EMIT ? s_out + (tid >> 5) * 2 * PJ_BUF : nullptr;
    int2* const gout = reinterpret_cast<int2*>(out) + ps.at[seg];
    uint32_t fill = 0;
    auto reserve = [&](unsigned long long n, unsigned long long* at) {
        unsigned long long a = 0;
        if (lane == 0) a = atomicAdd(&small->lines[seg].total, n);
        *at = __shfl_sync(0xffffffffu, a, 0);
        return *at + n <= cap;
    };
    auto flush = [&]() {
        __syncwarp();
        unsigned long long at;
        if (reserve(fill, &at))
            for (uint32_t q = lane; q < fill; q += 32) gout[at + q] = buf[q];
        fill = 0;
        __syncwarp();
    };
    unsigned long long acc = 0, csum = 0;
    uint32_t phase = 0;
    Item d{};
    if (first_item < nitems) d = items[first_item];
    for (uint64_t it = first_item; it < nitems; it += step) {
        const int rn = d.rn;
        const uint32_t sn = (uint32_t)d.sn;  // below 2^31: a row number and a round past it fit 32 bits
        const uint64_t lo = (d.rbeg * sizeof(R)) & ~15ull;
        // bytes of rows [beg, beg + n), widened to 16-byte boundaries
        auto span = [](uint64_t beg, int n) {
            return (uint32_t)((((beg + n) * sizeof(R) + 15) & ~15ull) - ((beg * sizeof(R)) & ~15ull));
        };
        if (tid == 0) {
            fence_proxy_async();
            mbar_arrive_expect_tx(&bar, span(d.rbeg, rn));
            tma_load_1d(smem, reinterpret_cast<const unsigned char*>(rrows) + lo, span(d.rbeg, rn), &bar);
        }
        // the next item's rows start on their way to L2
        Item dn{};
        if (it + step < nitems) {
            dn = items[it + step];
            if (tid == 0)
                l2_prefetch(reinterpret_cast<const unsigned char*>(rrows) + ((dn.rbeg * sizeof(R)) & ~15ull),
                            span(dn.rbeg, dn.rn));
            if (tid == 32 && dn.sn <= cap_rows)
                l2_prefetch(reinterpret_cast<const unsigned char*>(srows) + ((dn.sbeg * sizeof(R)) & ~15ull),
                            span(dn.sbeg, dn.sn));
        }
        // the thread's first S rows come in while the table is built
        const R* sp = srows + d.sbeg;
        R x[PU];
        auto load = [&](uint32_t j0) {
#pragma unroll
            for (int u = 0; u < PU; u++) {
                const uint32_t j = j0 + u * PJ_T + tid;
                if (j < sn) x[u] = sp[j];
            }
        };
        load(0);
        R* row = reinterpret_cast<R*>(smem + (d.rbeg * sizeof(R) - lo));
        // four entries to a row (load a quarter), as far as the table goes
        const int ts = min(L::entries(cap_rows), max(64, 4 * rn));
        auto fill4 = [&](uint32_t* p, int n, uint32_t v) {
            for (int i = tid; i < (n + 3) / 4; i += PJ_T) reinterpret_cast<uint4*>(p)[i] = make_uint4(v, v, v, v);
        };
        fill4(s_ent, ts, PJ_EMPTY);
        fill4(s_cnt, rn, 0);
        if (MODE == MODE_AGG) {
            fill4(s_flo, rn, 0);
            fill4(s_fhi, rn, 0);
        }
        if (__syncthreads_or(!mbar_wait(&bar, phase, err))) {
            if (tid == 0) mbar_wait(&bar, phase, nullptr);  // let the copy in flight land before leaving
            break;
        }
        phase ^= 1u;
        // ---- build ----
        uint32_t place[PER];  // emit: first row of the row's key << 16 | rank among its rows
        bool dup = false;
#pragma unroll
        for (int k = 0; k < PER; k++) {
            const int i = k * PJ_T + tid;
            place[k] = 0;
            if (i >= rn) continue;
            const K key = row[i].key;
            const uint32_t h = khash(key), mine = (h << 16) | (uint32_t)i;
            uint32_t s = pj_slot(h, bits, ts);
            for (int probe = 0; probe < ts; probe++) {
                const uint32_t old = atomicCAS(s_ent + s, PJ_EMPTY, mine);
                if (old == PJ_EMPTY) {
                    place[k] = (uint32_t)i << 16;
                    break;
                }
                if ((old ^ mine) < 0x10000u && row[old & 0xffffu].key == key) {
                    const uint32_t first = old & 0xffffu;
                    dup = true;
                    place[k] = first << 16 | (atomicAdd(s_cnt + first, 1u) + 1);
                    if (MODE == MODE_AGG) {
                        // a 64-bit sum in two native adds: the low word tells its carry
                        const unsigned long long f = chk_f(row[i].pay);
                        const uint32_t w = (uint32_t)f, o = atomicAdd(s_flo + first, w);
                        atomicAdd(s_fhi + first, (uint32_t)(f >> 32) + (o + w < o ? 1u : 0u));
                    }
                    break;
                }
                s = s + 1 == (uint32_t)ts ? 0u : s + 1;
            }
        }
        const bool runs = __syncthreads_or(dup);
        if (MODE == MODE_EMIT && runs) {
            // run starts: a scan over the counts at the first rows (which count
            // themselves; the others hold 0), PER rows per thread
            const int i0 = tid * PER;
            uint32_t c[PER], sum = 0, tot;
            int32_t pay[PER];
#pragma unroll
            for (int k = 0; k < PER; k++) {
                const int i = k * PJ_T + tid;
                if (i >= rn) continue;
                pay[k] = row[i].pay;
                if ((place[k] & 0xffffu) == 0) s_cnt[i] += 1;
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < PER; k++) {
                c[k] = i0 + k < rn ? s_cnt[i0 + k] : 0u;
                sum += c[k];
            }
            uint32_t pre = block_excl_scan(sum, tmp32, &tot);
#pragma unroll
            for (int k = 0; k < PER; k++) {
                if (c[k]) s_cnt[i0 + k] = c[k] << 16 | pre;
                pre += c[k];
            }
            __syncthreads();
            // the runs take the place of the payloads in the staged rows
#pragma unroll
            for (int k = 0; k < PER; k++) {
                const int i = k * PJ_T + tid;
                if (i < rn) row[(s_cnt[place[k] >> 16] & 0xffffu) + (place[k] & 0xffffu)].pay = pay[k];
            }
            __syncthreads();
        }
        // ---- probe ----
        for (uint32_t j0 = 0; j0 < sn; j0 += PU * PJ_T) {
            R y[PU];
#pragma unroll
            for (int u = 0; u < PU; u++) y[u] = x[u];
            load(j0 + PU * PJ_T);
#pragma unroll
            for (int u = 0; u < PU; u++) {
                if (j0 + u * PJ_T + (tid & ~31) >= sn) break;  // no row of this warp left
                const bool in = j0 + u * PJ_T + tid < sn;
                int first = -1;
                if (in) {
                    const uint32_t h = khash(y[u].key);
                    uint32_t s = pj_slot(h, bits, ts);
                    for (int probe = 0; probe < ts; probe++) {
                        const uint32_t e = s_ent[s];
                        if (e == PJ_EMPTY) break;
                        if ((e >> 16) == (h & 0xffffu) && row[e & 0xffffu].key == y[u].key) {
                            first = (int)(e & 0xffffu);
                            break;
                        }
                        s = s + 1 == (uint32_t)ts ? 0u : s + 1;
                    }
                }
                if (MODE != MODE_EMIT) {
                    if (first < 0) continue;
                    const uint32_t c = runs ? s_cnt[first] : 0u;
                    acc += 1 + c;
                    if (MODE == MODE_AGG) {
                        unsigned long long f = chk_f(row[first].pay);
                        if (c) f += (unsigned long long)s_fhi[first] << 32 | s_flo[first];
                        csum += f * chk_g(y[u].pay);
                    }
                    continue;
                }
                if (!runs) {
                    const unsigned b = __ballot_sync(0xffffffffu, first >= 0);
                    if (first >= 0)
                        buf[fill + __popc(b & ((1u << lane) - 1))] = make_int2(row[first].pay, y[u].pay);
                    fill += __popc(b);
                } else {
                    const uint32_t c = first >= 0 ? s_cnt[first] : 0u;
                    const uint32_t m = c >> 16, at0 = c & 0xffffu;
                    const uint32_t incl = warp_incl_scan(m);
                    const uint32_t tot = __shfl_sync(0xffffffffu, incl, 31);
                    if (tot == 0) continue;
                    // into the buffer when they fit it, else straight out
                    if (fill + tot > 2 * PJ_BUF && fill) flush();
                    int2* o = buf + fill;
                    if (tot > 2 * (uint32_t)PJ_BUF) {
                        unsigned long long at;
                        if (!reserve(tot, &at)) continue;
                        o = gout + at;
                    } else {
                        fill += tot;
                    }
                    o += incl - m;
                    const bool longr = m > 4;
                    if (!longr)
                        for (uint32_t e = 0; e < m; e++) o[e] = make_int2(row[at0 + e].pay, y[u].pay);
                    // a long run is written by the whole warp, 32 pairs at a time
                    for (unsigned lanes = __ballot_sync(0xffffffffu, longr); lanes; lanes &= lanes - 1) {
                        const int src = __ffs(lanes) - 1;
                        const uint32_t bm = __shfl_sync(0xffffffffu, m, src);
                        const uint32_t bb = __shfl_sync(0xffffffffu, at0, src);
                        const int32_t bp = __shfl_sync(0xffffffffu, y[u].pay, src);
                        int2* bo = reinterpret_cast<int2*>(
                            __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(o), src));
                        for (uint32_t e = lane; e < bm; e += 32) bo[e] = make_int2(row[bb + e].pay, bp);
                    }
                }
                if (fill >= (uint32_t)PJ_BUF) flush();
            }
        }
        __syncthreads();  // the staged rows and the table are free
        d = dn;
    }
    if (MODE == MODE_EMIT) {
        if (fill) flush();
        return;
    }
    __syncthreads();
    acc = block_sum(acc, tmp64);
    if (MODE == MODE_AGG) csum = block_sum(csum, tmp64);
    if (tid == 0) {
        if (acc) atomicAdd(&small->lines[seg].total, acc);
        if (MODE == MODE_AGG && csum) atomicAdd(&small->lines[0].chk, csum);
    }
}

}  // namespace jnx
