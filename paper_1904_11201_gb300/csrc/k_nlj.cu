// Nested-loop join (Sec. 3.3.1): every (R, S) pair is tested.
//
// The paper's grid gives each thread NB_S = |S|/(m x) + 1 rows of S and
// NB_T = |T|/(n y) + 1 rows of T (Eqs. NBS, NBT, IDS, IDT) and a private
// result buffer of NB_S * NB_T pairs.  Here a block holds a tile of R rows in
// shared memory and a tile of S rows in registers (NLJ_SPT per thread), so
// every R value read from shared memory is compared against NLJ_SPT S rows.
// The predicate of each S row is turned, once, into an interval test on the
// R value ("R.x op s" <=> R.x in [lo, hi], possibly negated), which makes the
// inner loop a subtract and an unsigned compare per column.  The exact count
// replaces the NB_S * NB_T per-thread buffers: jn_nested_loop compares once
// and keeps the pairs it finds in scratch (k_nlj_once) where that pays; the
// allocation-free entry point counts per tile, scans, and compares again to
// write (k_nlj).
#include <limits.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "jn_algos.h"

namespace jnx {

constexpr int NLJ_T = 256;
#ifndef JN_NLJ_SPT
#define JN_NLJ_SPT 4
#endif
constexpr int NLJ_SPT = JN_NLJ_SPT;  // S rows per thread
constexpr int NLJ_STILE = NLJ_T * NLJ_SPT;

// An R row's two predicate columns, adjacent in shared memory so that one
// load fetches both.
template <typename K>
struct __align__(2 * sizeof(K)) KPair {
    K a, b;
};

// The tile kernel of the allocation-free call and of runs with few pairs a tile
// (nlj_thin).  MODE_COUNT: tile_val[tile] = its pairs; MODE_EMIT: writes them at
// out[tile_off[tile] ..].
template <typename K, bool HAS2, int MODE>
__global__ void __launch_bounds__(NLJ_T)
k_nlj(const K* __restrict__ rk, const K* __restrict__ rk2, const int32_t* __restrict__ rp, int64_t nr,
      const K* __restrict__ sk, const K* __restrict__ sk2, const int32_t* __restrict__ sp, int64_t ns,
      int op_a, int op_k, long long band, int tr, unsigned long long* __restrict__ tile_val,
      const uint64_t* __restrict__ tile_off, jn_pair* __restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem[];
    // R tile: (a, b) pairs with a second column, else the a column alone
    K* s_a = reinterpret_cast<K*>(smem);
    KPair<K>* s_ab = reinterpret_cast<KPair<K>*>(smem);
    int32_t* s_p = reinterpret_cast<int32_t*>(s_a + (HAS2 ? 2 : 1) * tr);
    __shared__ unsigned long long tmp64[33];
    __shared__ uint32_t s_cur;

    const uint64_t tile = (uint64_t)blockIdx.y * gridDim.x + blockIdx.x;
    if (MODE == MODE_EMIT) {
        // tiles without results have nothing to write
        if (tile_off[tile + 1] == tile_off[tile]) return;
    }
    const int64_t r0 = (int64_t)blockIdx.y * tr;
    const int rn = (int)min((int64_t)tr, nr - r0);
    for (int i = threadIdx.x; i < rn; i += NLJ_T) {
        if (HAS2)
            s_ab[i] = KPair<K>{rk[r0 + i], rk2[r0 + i]};
        else
            s_a[i] = rk[r0 + i];
        s_p[i] = rp ? rp[r0 + i] : (int32_t)(r0 + i);
    }
    if (threadIdx.x == 0) s_cur = 0;

    Interval<K> ia[NLJ_SPT], ib[NLJ_SPT];
    int32_t spay[NLJ_SPT];
    bool valid[NLJ_SPT];
    const int64_t s0 = (int64_t)blockIdx.x * NLJ_STILE;
#pragma unroll
    for (int j = 0; j < NLJ_SPT; j++) {
        const int64_t s = s0 + j * NLJ_T + threadIdx.x;
        valid[j] = s < ns;
        K a = valid[j] ? sk[s] : (K)0;
        ia[j] = op_interval<K>(valid[j] ? op_a : JN_ANY, a);
        if (!valid[j]) {  // an empty set: never matches
            ia[j].inv = true;
            ia[j].lo = sizeof(K) == 4 ? (K)INT32_MIN : (K)INT64_MIN;
            ia[j].span = ~(decltype(ia[j].span))0;
        }
        if (HAS2) {
            K b = valid[j] ? sk2[s] : (K)0;
            ib[j] = band >= 0 ? band_interval<K>(b, band) : op_interval<K>(op_k, b);
        }
        spay[j] = valid[j] ? (sp ? sp[s] : (int32_t)s) : 0;
    }
    // Inverted intervals (!=, and the empty sets of invalid rows and of
    // "< min" / "> max") take the general test; a warp whose rows have none
    // runs the plain interval test, which needs no inversion step per pair.
    bool inv = false;
#pragma unroll
    for (int j = 0; j < NLJ_SPT; j++) inv |= ia[j].inv || (HAS2 && ib[j].inv);
    const bool plain = !__any_sync(0xffffffffu, inv);
    __syncthreads();

    unsigned long long acc = 0;
    auto visit = [&](auto test) {
        for (int i = 0; i < rn; i++) {
            K a, b = 0;
            if (HAS2) {
                const KPair<K> ab = s_ab[i];
                a = ab.a;
                b = ab.b;
            } else {
                a = s_a[i];
            }
            if (MODE == MODE_EMIT) {
                // one branch per R row: matches are rare, the tests are not
                uint32_t mask = 0;
#pragma unroll
                for (int j = 0; j < NLJ_SPT; j++) mask |= (uint32_t)test(j, a, b) << j;
                if (mask) {
#pragma unroll
                    for (int j = 0; j < NLJ_SPT; j++) {
                        if ((mask >> j) & 1u) {
                            const uint32_t slot = atomicAdd(&s_cur, 1u);
                            st_pair(out + tile_off[tile] + slot, s_p[i], spay[j]);
                        }
                    }
                }
            } else {
#pragma unroll
                for (int j = 0; j < NLJ_SPT; j++) acc += test(j, a, b);
            }
        }
    };
    if (plain)
        visit([&](int j, K a, K b) {
            bool m = in_range(a, ia[j].lo, ia[j].span);
            if (HAS2) m &= in_range(b, ib[j].lo, ib[j].span);
            return m;
        });
    else
        visit([&](int j, K a, K b) {
            bool m = iv_test(ia[j], a);
            if (HAS2) m &= iv_test(ib[j], b);
            return m;
        });
    if (MODE != MODE_EMIT) {
        const unsigned long long t = block_sum(acc, tmp64);
        if (threadIdx.x == 0) tile_val[tile] = t;
    }
}

// ------------------------------------------------------------- one pass --
// The nested loop of jn_nested_loop, jn_count and jn_aggregate: every pair is
// compared once, and pairs go to scratch as they are found (the copy into the
// exact allocation costs 16 bytes a pair, a second round of comparisons costs
// the whole join again).
//
// Bound by the instructions issued per pair.  A predicate with one selective
// conjunct -- equality on either column, or a narrow band -- is screened
// first, on 16-bit codes, two S rows to an instruction: a code is the band
// column's offset inside the R tile's range (its top 16 bits) or a 16-bit
// hash for equality, and `R code - S code <= limit` (modulo 2^16) holds for
// every pair that the conjunct accepts.  A thread holds NL_SPT S codes and
// takes the minimum of the differences over them, NL_R R rows at a time, so 64
// pairs cost 32 add-min instructions, one shared load and one test; only what
// passes is compared exactly, on the rows themselves.  A warp that finds
// nearly every round passing (a wide band, few distinct keys) finishes the
// tile with the exact comparisons, in groups of four S rows held as intervals.
//
// Measured on GB300, 64K x 1M rows, R.a < S.a and |R.k - S.k| <= 127 of 2^24:
// 2.95 ms, the integer pipe 92 % busy, 1.0 instructions a pair; the count and
// emit passes it replaces took 14.5 + 10.9 ms at 6.5 and 6.3.  With a band of
// 24414 (too wide to screen) 15.4 ms against 27.8.
constexpr int NL_SPT = 16;   // S rows per thread
constexpr int NL_STILE = NLJ_T * NL_SPT;
constexpr int NL_R = 4;      // R rows screened together
constexpr int NL_BUF = 256;  // pairs a warp collects in shared memory
constexpr uint32_t NL_NEVER = 0xFFFFu;  // S code where there is nothing to find (what passes is compared all the same)

enum NlScreen { NL_NONE = 0, NL_BAND = 1, NL_EQ_A = 2, NL_EQ_B = 3 };

struct NlCounters {
    unsigned long long total, chk;
    unsigned long long hits;  // of the sample
};

// A first pass whose sample's hits lie in [lo, hi] does nothing: the predicate
// accepts more than it looks like, or less, and another way is faster.
struct NlSkip {
    unsigned long long lo = 1, hi = 0;
};

__device__ __forceinline__ uint32_t nl_hash(int32_t k) { return khash(k) >> 16; }
__device__ __forceinline__ uint32_t nl_hash(int64_t k) { return khash(k) >> 16; }

template <typename K, bool HAS2, int MODE>
__global__ void __launch_bounds__(NLJ_T, 4)
k_nlj_once(const K* __restrict__ rk, const K* __restrict__ rk2, const int32_t* __restrict__ rp, int64_t nr,
           const K* __restrict__ sk, const K* __restrict__ sk2, const int32_t* __restrict__ sp, int64_t ns, int op_a,
           int op_k, long long band, int tr, int screen, NlCounters* __restrict__ cnt,
           unsigned long long* __restrict__ tile_val, const uint64_t* __restrict__ tile_off, jn_pair* __restrict__ out,
           unsigned long long cap, NlSkip skip) {
    if (cnt->hits >= skip.lo && cnt->hits <= skip.hi) return;
    // emit: to out[0 .. cap) through cnt->total, or, with tile_off, every tile
    // to its own place; tile_val (if given) gets the tile's pairs
    const uint64_t tile = (uint64_t)blockIdx.y * gridDim.x + blockIdx.x;
    if (MODE == MODE_EMIT && tile_off && tile_off[tile + 1] == tile_off[tile]) return;
    if (MODE == MODE_EMIT && tile_off) out += tile_off[tile];
    const bool direct = MODE == MODE_EMIT && tile_off != nullptr;
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t* s_c = reinterpret_cast<uint32_t*>(smem);  // the tile's codes, each in both halves of a word
    KPair<K>* s_ab = reinterpret_cast<KPair<K>*>(s_c + tr + NL_R);
    int32_t* s_p = reinterpret_cast<int32_t*>(s_ab + tr);
    __shared__ int2 s_buf[MODE == MODE_EMIT ? NLJ_T / 32 : 1][MODE == MODE_EMIT ? NL_BUF : 1];
    __shared__ unsigned int s_fill[NLJ_T / 32], s_cur;
    __shared__ long long s_lo[NLJ_T / 32], s_hi[NLJ_T / 32];
    __shared__ unsigned long long tmp64[33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t r0 = (int64_t)blockIdx.y * tr, s0 = (int64_t)blockIdx.x * NL_STILE;
    const int rn = (int)min((int64_t)tr, nr - r0);

    // ---- the R tile, and (band screen) the range of its band column ----
    long long lo = LLONG_MAX, hi = LLONG_MIN;
    for (int i = threadIdx.x; i < rn; i += NLJ_T) {
        const K a = rk[r0 + i], b = HAS2 ? rk2[r0 + i] : K(0);
        s_ab[i] = KPair<K>{a, b};
        s_p[i] = rp ? rp[r0 + i] : (int32_t)(r0 + i);
        lo = min(lo, (long long)b);
        hi = max(hi, (long long)b);
    }
    if (lane == 0) s_fill[w] = 0;
    if (threadIdx.x == 0) s_cur = 0;
    uint64_t limit = 0;
    int q = 0;
    if (HAS2 && screen == NL_BAND) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        if (lane == 0) {
            s_lo[w] = lo;
            s_hi[w] = hi;
        }
        __syncthreads();
        lo = s_lo[0];
        hi = s_hi[0];
        for (int k = 1; k < NLJ_T / 32; k++) {
            lo = min(lo, s_lo[k]);
            hi = max(hi, s_hi[k]);
        }
        while ((((uint64_t)hi - (uint64_t)lo) >> q) > 0xffffu) q++;
        // a window of 2 band + 1 values covers at most this many codes past its first
        limit = band < (1ll << 62) ? ((2 * (uint64_t)band) >> q) + 1 : ~0ull;
        if (limit > 64) screen = NL_NONE;  // one pair in 512 or more would pass
    }
    __syncthreads();
    if (screen != NL_NONE) {
        for (int i = threadIdx.x; i < ((rn + NL_R - 1) & ~(NL_R - 1)); i += NLJ_T) {
            uint32_t c = 0;  // rows behind the last are left out where they pass
            if (i < rn)
                c = screen == NL_BAND ? (uint32_t)(((uint64_t)(long long)s_ab[i].b - (uint64_t)lo) >> q)
                                      : nl_hash(screen == NL_EQ_A ? s_ab[i].a : s_ab[i].b);
            s_c[i] = c | (c << 16);
        }
    }
    __syncthreads();

    unsigned long long acc = 0, csum = 0;
    // writes a pair: to its tile's place, or through the warp's buffer
    auto put = [&](int32_t r, int32_t p) {
        if (direct) {
            st_pair(out + atomicAdd(&s_cur, 1u), r, p);
            return;
        }
        const unsigned int at = atomicAdd(&s_fill[w], 1u);
        if (at < NL_BUF) {
            s_buf[w][at] = make_int2(r, p);
        } else {  // more than a buffer at once
            const unsigned long long g = atomicAdd(&cnt->total, 1ull);
            if (g < cap) st_pair(out + g, r, p);
        }
    };
    // the warp writes what it has collected, once that is `from` pairs (all lanes)
    auto flush = [&](unsigned int from) {
        if (MODE != MODE_EMIT || direct) return;
        __syncwarp();
        // one lane reads the count, so that every lane decides alike
        const unsigned int n = min(__shfl_sync(0xffffffffu, lane == 0 ? s_fill[w] : 0u, 0), (unsigned int)NL_BUF);
        if (n < from) return;
        unsigned long long g = 0;
        if (lane == 0) g = atomicAdd(&cnt->total, (unsigned long long)n);
        g = __shfl_sync(0xffffffffu, g, 0);
        if (g + n <= cap)
            for (unsigned int e = lane; e < n; e += 32) st_pair(out + g + e, s_buf[w][e].x, s_buf[w][e].y);
        __syncwarp();
        if (lane == 0) s_fill[w] = 0;
        __syncwarp();
    };
    int i0 = 0;  // tile rows below it are done

    // ---- screened rounds ----
    if (screen != NL_NONE) {
        uint32_t nc[NL_SPT / 2];  // two S rows' codes, negated
        auto code = [&](int j) -> uint32_t {
            const int64_t s = s0 + (int64_t)j * NLJ_T + threadIdx.x;
            if (s >= ns) return NL_NEVER;
            if (screen == NL_EQ_A) return nl_hash(sk[s]);
            if (!HAS2) return NL_NEVER;
            if (screen == NL_EQ_B) return nl_hash(sk2[s]);
            const Interval<K> iv = band_interval<K>(sk2[s], band);
            const long long first = (long long)iv.lo;
            const long long last = (long long)(K)((decltype(iv.span))iv.lo + iv.span);
            if (last < lo || first > hi) return NL_NEVER;
            return (uint32_t)(((uint64_t)max(first, lo) - (uint64_t)lo) >> q);
        };
#pragma unroll
        for (int e = 0; e < NL_SPT / 2; e++)
            nc[e] = ((0u - code(2 * e)) & 0xffffu) | ((0u - code(2 * e + 1)) << 16);
        const uint32_t lim = (uint32_t)limit;
        int rounds = 0, passed = 0;
        for (; i0 < rn; i0 += NL_R) {
            const uint4 c4 = *reinterpret_cast<const uint4*>(s_c + i0);
            const uint32_t c[NL_R] = {c4.x, c4.y, c4.z, c4.w};
            uint32_t m[NL_R], all = 0xffffffffu;
#pragma unroll
            for (int r = 0; r < NL_R; r++) {
                m[r] = 0xffffffffu;
#pragma unroll
                for (int e = 0; e < NL_SPT / 2; e++) m[r] = __viaddmin_u16x2(c[r], nc[e], m[r]);
                all = __vminu2(all, m[r]);
            }
            const bool pass = min(all & 0xffffu, all >> 16) <= lim;
            rounds++;
            if (!__any_sync(0xffffffffu, pass)) continue;
            passed++;
            if (pass) {
#pragma unroll
                for (int r = 0; r < NL_R; r++) {
                    if (min(m[r] & 0xffffu, m[r] >> 16) > lim) continue;
                    const uint32_t cr = c[r];
                    uint32_t hits = 0;
#pragma unroll
                    for (int e = 0; e < NL_SPT / 2; e++) {
                        const uint32_t d = __viaddmin_u16x2(cr, nc[e], 0xffffffffu);
                        hits |= (uint32_t)((d & 0xffffu) <= lim) << (2 * e) | (uint32_t)((d >> 16) <= lim) << (2 * e + 1);
                    }
                    if (i0 + r >= rn) hits = 0;
                    for (; hits; hits &= hits - 1) {
                        const int64_t s = s0 + (int64_t)(__ffs(hits) - 1) * NLJ_T + threadIdx.x;
                        if (s >= ns) continue;
                        const KPair<K> ab = s_ab[i0 + r];
                        bool ok = iv_test(op_interval<K>(op_a, sk[s]), ab.a);
                        if (HAS2 && ok)
                            ok = iv_test(band >= 0 ? band_interval<K>(sk2[s], band) : op_interval<K>(op_k, sk2[s]), ab.b);
                        if (!ok) continue;
                        acc++;
                        if (MODE == MODE_COUNT) continue;
                        const int32_t p = sp ? sp[s] : (int32_t)s;
                        if (MODE == MODE_AGG)
                            csum += chk_f(s_p[i0 + r]) * chk_g(p);
                        else
                            put(s_p[i0 + r], p);
                    }
                }
            }
            flush(NL_BUF / 2);
            if (passed >= 6 && 16 * passed > 15 * rounds) {
                i0 += NL_R;
                break;
            }
        }
    }

    // ---- exact rounds: four S rows as intervals, the rest of the tile ----
    if (i0 < rn) {
#pragma unroll 1
        for (int g = 0; g < NL_SPT; g += 4) {
            Interval<K> ia[4], ib[4];
            bool inv = false;
            int32_t p[4];
            unsigned long long gs[4];
            const int64_t sg = s0 + (int64_t)g * NLJ_T;
            if (sg >= ns) break;  // no S row left in this tile
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int64_t s = sg + j * NLJ_T + threadIdx.x;
                const bool valid = s < ns;
                ia[j] = op_interval<K>(valid ? op_a : JN_ANY, valid ? sk[s] : K(0));
                if (!valid) {  // an empty set: never matches
                    ia[j].inv = true;
                    ia[j].lo = sizeof(K) == 4 ? (K)INT32_MIN : (K)INT64_MIN;
                    ia[j].span = ~(decltype(ia[j].span))0;
                }
                inv |= ia[j].inv;
                if (HAS2) {
                    const K b = valid ? sk2[s] : K(0);
                    ib[j] = band >= 0 ? band_interval<K>(b, band) : op_interval<K>(op_k, b);
                    inv |= ib[j].inv;
                }
                if (MODE != MODE_COUNT) p[j] = valid ? (sp ? sp[s] : (int32_t)s) : 0;
                if (MODE == MODE_AGG) gs[j] = chk_g(p[j]);
            }
            // `first` (a band alone) rules most rounds out where there is one.  A
            // warp that it ruled out four in 64 for, or fewer, stops asking where
            // that gains: counts (2^15 x 2^18 rows, a band of 2^19 in 2^24: 1.9 ms,
            // 2.5 asked throughout; int64 3.0 and 4.5) and int32 checksums (4.7 and
            // 5.5).  The int64 checksum's loop is the slower one without the
            // question (10.8 and 9.1), and most pairs to write come from narrower
            // bands.  Each kind has a loop of its own: one that carried the numbers
            // of rounds asked and ruled out took 18.1 ms for 2^16 x 2^20 rows, a
            // band of 24414 in 2^24, pairs kept, where 15.4 are enough, and 12.0 to
            // count, where 9.5 are.
            constexpr bool STOPS = MODE == MODE_COUNT || (MODE == MODE_AGG && sizeof(K) == 4);
            auto visit = [&](auto has_first, auto first, auto test) {
                uint32_t count = 0;  // at most four a round
                auto round = [&](auto ask, int i) {  // whether it was ruled out
                    const KPair<K> ab = s_ab[i];
                    if (decltype(ask)::value) {
                        bool any = false;
#pragma unroll
                        for (int j = 0; j < 4; j++) any |= first(j, ab);
                        if (!__any_sync(0xffffffffu, any)) return true;
                    }
                    if (MODE == MODE_COUNT) {
#pragma unroll
                        for (int j = 0; j < 4; j++) count += test(j, ab);
                        return false;
                    }
                    uint32_t mask = 0;
#pragma unroll
                    for (int j = 0; j < 4; j++) mask |= (uint32_t)test(j, ab) << j;
                    if (MODE == MODE_AGG) {
                        if (mask) {
                            acc += __popc(mask);
                            unsigned long long g4 = 0;
#pragma unroll
                            for (int j = 0; j < 4; j++) g4 += (mask >> j) & 1u ? gs[j] : 0ull;
                            csum += chk_f(s_p[i]) * g4;
                        }
                    } else if (direct) {
                        // half of the pairs or fewer: every lane reserves its
                        // own; more: one reservation per warp and the lanes'
                        // pairs side by side, at the price of four ballots
                        const int32_t r = s_p[i];
                        if (__popc(__ballot_sync(0xffffffffu, __popc(mask) > 2)) <= 16) {
                            if (!mask) return false;
                            jn_pair* o = out + atomicAdd(&s_cur, (unsigned int)__popc(mask));
#pragma unroll
                            for (int j = 0; j < 4; j++)
                                if ((mask >> j) & 1u) st_pair(o++, r, p[j]);
                            return false;
                        }
                        unsigned b[4], sum = 0;
#pragma unroll
                        for (int j = 0; j < 4; j++) {
                            b[j] = __ballot_sync(0xffffffffu, (mask >> j) & 1u);
                            sum += __popc(b[j]);
                        }
                        unsigned at = 0;
                        if (lane == 0) at = atomicAdd(&s_cur, sum);
                        at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
                        for (int j = 0; j < 4; j++) {
                            if ((mask >> j) & 1u) st_pair(out + at + __popc(b[j] & ((1u << lane) - 1)), r, p[j]);
                            at += __popc(b[j]);
                        }
                    } else {
                        if (!__any_sync(0xffffffffu, mask)) return false;
                        acc += __popc(mask);
#pragma unroll
                        for (int j = 0; j < 4; j++)
                            if ((mask >> j) & 1u) put(s_p[i], p[j]);
                        flush(NL_BUF / 2);
                    }
                    return false;
                };
                int i = i0;
                if (decltype(has_first)::value && !STOPS) {
                    for (; i < rn; i++) round(has_first, i);
                } else if (decltype(has_first)::value) {
                    int ruled = 0;
#pragma unroll 1
                    for (int end = min(rn, i0 + 64);; end = rn) {
                        for (; i < end; i++) ruled += round(has_first, i);
                        if (end == rn || ruled <= 4) break;
                    }
                }
                for (; i < rn; i++) round(std::false_type(), i);
                acc += count;
            };
            constexpr std::false_type all{};
            constexpr std::true_type band_first{};
            // warps without inverted intervals (!=, empty sets) take the bare
            // range tests
            if (!__any_sync(0xffffffffu, inv)) {
                auto both = [&](int j, const KPair<K>& x) {
                    bool m = in_range(x.a, ia[j].lo, ia[j].span);
                    if (HAS2) m &= in_range(x.b, ib[j].lo, ib[j].span);
                    return m;
                };
                if (HAS2 && band >= 0)
                    visit(band_first, [&](int j, const KPair<K>& x) { return in_range(x.b, ib[j].lo, ib[j].span); },
                          both);
                else
                    visit(all, both, both);
            } else {
                auto both = [&](int j, const KPair<K>& x) {
                    bool m = iv_test(ia[j], x.a);
                    if (HAS2) m &= iv_test(ib[j], x.b);
                    return m;
                };
                visit(all, both, both);
            }
        }
    }
    if (direct) return;
    flush(1);
    acc = block_sum(acc, tmp64);
    if (MODE == MODE_AGG) csum = block_sum(csum, tmp64);
    if (threadIdx.x == 0) {
        if (tile_val) tile_val[tile] = acc;
        if (MODE != MODE_EMIT && acc) atomicAdd(&cnt->total, acc);
        if (MODE == MODE_AGG && csum) atomicAdd(&cnt->chk, csum);
    }
}

// cnt->hits += pairs that the predicate accepts among sampled rows: block x
// compares part x of R's sample with all of S's.
constexpr int NL_SAMPLE_R = 4096, NL_SAMPLE_S = 512, NL_SPARTS = 128;
template <typename K, bool HAS2>
__global__ void __launch_bounds__(NL_SAMPLE_S)
k_nlj_sample(const K* __restrict__ rk, const K* __restrict__ rk2, int64_t nr, const K* __restrict__ sk,
             const K* __restrict__ sk2, int64_t ns, int op_a, int op_k, long long band, NlCounters* __restrict__ cnt) {
    constexpr int PART = NL_SAMPLE_R / NL_SPARTS;
    __shared__ KPair<K> s_r[PART];
    const int mr = (int)min(nr, (int64_t)NL_SAMPLE_R), ms = (int)min(ns, (int64_t)NL_SAMPLE_S);
    const int r0 = blockIdx.x * PART, n = min(PART, mr - r0), q = threadIdx.x;
    if (n <= 0) return;  // the whole block
    if (q < n) {
        const int64_t at = (int64_t)(r0 + q) * nr / mr;
        s_r[q] = KPair<K>{rk[at], HAS2 ? rk2[at] : K(0)};
    }
    __syncthreads();
    unsigned int m = 0;
    if (q < ms) {
        const int64_t at = (int64_t)q * ns / ms;
        const Interval<K> ia = op_interval<K>(op_a, sk[at]);
        Interval<K> ib{};
        if (HAS2) ib = band >= 0 ? band_interval<K>(sk2[at], band) : op_interval<K>(op_k, sk2[at]);
        for (int i = 0; i < n; i++) m += iv_test(ia, s_r[i].a) && (!HAS2 || iv_test(ib, s_r[i].b));
    }
    m = warp_sum(m);
    if ((q & 31) == 0 && m) atomicAdd(&cnt->hits, (unsigned long long)m);
}

// An emitting run counted and then written by k_nlj, every tile to its place.
template <typename K>
static jn_status nlj_thin(jn_ctx* c, const Cols<K>& R, const Cols<K>& S, const jn_pred& pr, bool has2, int tr,
                          OutPlan* plan, RunResult* res) {
    const dim3 grid((unsigned)ceil_div(S.n, NLJ_STILE), (unsigned)ceil_div(R.n, tr));
    const uint64_t tiles = (uint64_t)grid.x * grid.y;
    const size_t smem = (size_t)tr * (sizeof(K) * (has2 ? 2 : 1) + 4);
    Scratch s(c);
    unsigned long long* val;
    uint64_t* off;
    JN_TRY(s.get(&val, tiles));
    JN_TRY(s.get(&off, tiles + 1));
    auto pass = [&](int kid, auto kn, jn_pair* out) {
        return launch(c, kid, kn, grid, dim3(NLJ_T), smem, R.key, R.key2, R.pay, R.n, S.key, S.key2, S.pay, S.n,
                      pr.op_a, pr.op_k, (long long)pr.band, tr, val, (const uint64_t*)off, out);
    };
    JN_TRY(has2 ? pass(K_NLJ_COUNT, k_nlj<K, true, MODE_COUNT>, (jn_pair*)nullptr)
                : pass(K_NLJ_COUNT, k_nlj<K, false, MODE_COUNT>, (jn_pair*)nullptr));
    JN_TRY(scan_u64(c, reinterpret_cast<const uint64_t*>(val), off, (int64_t)tiles));
    uint64_t total;
    JN_TRY(read_back(c, off + tiles, &total, 1));
    jn_run_info& info = c->info;
    res->count = info.result = total;
    info.partitions = info.work_items = tiles;
    info.r_survivors = (uint64_t)R.n;
    info.s_survivors = (uint64_t)S.n;
    info.prefilter = 0;
    info.cartesian_bound = (uint64_t)R.n * (uint64_t)S.n;
    JN_TRY(out_prepare(c, s, total, *plan));
    if (total) {
        JN_TRY(has2 ? pass(K_NLJ_EMIT, k_nlj<K, true, MODE_EMIT>, plan->dev)
                    : pass(K_NLJ_EMIT, k_nlj<K, false, MODE_EMIT>, plan->dev));
        JN_CUDA(c, cudaStreamSynchronize(c->stream));  // this pass reads the caller's columns
    }
    return out_finish(c, total, *plan);
}

static int nlj_screen(const jn_pred& pr, bool has2) {
    return pr.op_a == JN_EQ             ? NL_EQ_A
           : has2 && pr.band >= 0       ? NL_BAND
           : has2 && pr.op_k == JN_EQ   ? NL_EQ_B
                                        : NL_NONE;
}

template <typename K, bool HAS2>
static jn_status nlj_once(jn_ctx* c, int mode, dim3 grid, const Cols<K>& R, const Cols<K>& S, const jn_pred& pr,
                          int tr, NlCounters* cnt, uint64_t* val, const uint64_t* off, jn_pair* out, uint64_t cap,
                          NlSkip skip) {
    const size_t smem = (size_t)(tr + NL_R) * 4 + (size_t)tr * (2 * sizeof(K) + 4);
    auto kn = mode == MODE_EMIT  ? k_nlj_once<K, HAS2, MODE_EMIT>
              : mode == MODE_AGG ? k_nlj_once<K, HAS2, MODE_AGG>
                                 : k_nlj_once<K, HAS2, MODE_COUNT>;
    return launch(c, mode == MODE_EMIT ? K_NLJ_EMIT : K_NLJ_COUNT, kn, grid, dim3(NLJ_T), smem, R.key, R.key2, R.pay,
                  R.n, S.key, S.key2, S.pay, S.n, pr.op_a, pr.op_k, (long long)pr.band, tr, nlj_screen(pr, HAS2), cnt,
                  reinterpret_cast<unsigned long long*>(val), off, out, (unsigned long long)cap, skip);
}

template <typename K>
jn_status run_nlj(jn_ctx* c, const Cols<K>& R, const Cols<K>& S, const jn_pred& pred, int mode,
                  OutPlan* plan, RunResult* res) {
    jn_run_info& info = c->info;
    if (R.n == 0 || S.n == 0) {
        res->count = res->checksum = 0;
        if (mode == MODE_EMIT) {
            Scratch s0(c);
            JN_TRY(out_prepare(c, s0, 0, *plan));
            JN_TRY(out_finish(c, 0, *plan));
        }
        return JN_OK;
    }
    const bool has2 = R.key2 != nullptr && S.key2 != nullptr;
    int tr = c->tune.nlj_tile_r ? c->tune.nlj_tile_r : 1024;
    if (ceil_div(R.n, tr) > 65535)
        return fail(c, JN_ERR_UNSUPPORTED, "nested loop: R has more than 65535 tiles; use a larger nlj_tile_r");
    // small joins: smaller R tiles, until every SM has several
    const uint64_t gx = ceil_div(S.n, NL_STILE);
    while (!c->tune.nlj_tile_r && tr > 64 && gx * ceil_div(R.n, tr) < 8 * (uint64_t)c->num_sms) tr /= 2;
    const dim3 grid((unsigned)gx, (unsigned)ceil_div(R.n, tr));
    const uint64_t tiles = gx * grid.y, pairs = (uint64_t)R.n * (uint64_t)S.n;
    // scratch for the pairs of a selective predicate (one that is screened):
    // a few per row, or one comparison in 128 of a large join; not under a
    // limit that counts scratch
    uint64_t cap = 0;
    if (mode == MODE_EMIT && nlj_screen(pred, has2) != NL_NONE && !c->mem_limit && !c->admit)
        cap = std::min(pairs, std::max<uint64_t>(4 * (uint64_t)(R.n + S.n) + 65536, std::min<uint64_t>(pairs / 128, 1u << 27)));
    Scratch s(c), ss(c);
    NlCounters* cnt;
    jn_pair* staged = nullptr;
    uint64_t *val = nullptr, *off = nullptr;
    JN_TRY(s.get(&cnt, 1));
    JN_TRY(zero(c, cnt, sizeof(NlCounters)));
    if (mode == MODE_EMIT) JN_TRY(s.get(&val, tiles));
    if (cap && ss.get(&staged, cap) != JN_OK) {
        c->err.clear();
        cap = 0;
    }
    auto pass = [&](int m, jn_pair* to, uint64_t room, NlSkip skip) {
        return has2 ? nlj_once<K, true>(c, m, grid, R, S, pred, tr, cnt, val, off, to, room, skip)
                    : nlj_once<K, false>(c, m, grid, R, S, pred, tr, cnt, val, off, to, room, skip);
    };
    // Large joins are sampled (9 us), and the first pass looks at the hits: a
    // predicate that looks selective and accepts more than the scratch holds (a
    // wide band, few distinct keys) would be compared twice with the first
    // time's stores on top (2^15 x 2^18 int32 rows, 3 % accepted: 12.1 ms).
    // Counted and then written to the tiles' places, k_nlj is the faster one
    // below one pair in eight (6.8 ms there, 8.1 here; int64 10.3 and 11.1) and
    // k_nlj_once above (2^13 x 2^15, half accepted: 0.39 ms here, 0.57 there).
    const double looked = (double)std::min(R.n, (int64_t)NL_SAMPLE_R) * (double)std::min(S.n, (int64_t)NL_SAMPLE_S);
    const unsigned long long eighth = (unsigned long long)(looked / 8);
    NlSkip skip;
    const bool screened = nlj_screen(pred, has2) != NL_NONE;
    if (mode == MODE_EMIT && (cap ? pairs >= (1ull << 26) : !screened && pairs >= (1ull << 30))) {
        if (cap)
            skip = NlSkip{(unsigned long long)((double)cap / (double)pairs * looked) + 1, ~0ull};
        else
            skip = NlSkip{0, eighth};
        auto ks = has2 ? k_nlj_sample<K, true> : k_nlj_sample<K, false>;
        JN_TRY(launch(c, K_NLJ_COUNT, ks, dim3(NL_SPARTS), dim3(NL_SAMPLE_S), 0, R.key, R.key2, R.n, S.key, S.key2, S.n,
                      pred.op_a, pred.op_k, (long long)pred.band, cnt));
    }
    // without scratch the first pass only counts
    JN_TRY(pass(mode == MODE_EMIT && !cap ? (int)MODE_COUNT : mode, staged, cap, skip));
    uint64_t h[3];
    JN_TRY(read_back(c, reinterpret_cast<const uint64_t*>(cnt), h, 3));
    if (h[2] >= skip.lo && h[2] <= skip.hi) {
        ss.release();
        cap = 0;
        if (h[2] <= eighth)
            return nlj_thin<K>(c, R, S, pred, has2, c->tune.nlj_tile_r ? c->tune.nlj_tile_r : 1024, plan, res);
        JN_TRY(pass(MODE_COUNT, nullptr, 0, NlSkip()));
        JN_TRY(read_back(c, reinterpret_cast<const uint64_t*>(cnt), h, 2));
    }
    res->count = h[0];
    res->checksum = h[1];
    info.result = h[0];
    info.partitions = tiles;
    info.work_items = tiles;
    info.r_survivors = (uint64_t)R.n;
    info.s_survivors = (uint64_t)S.n;
    info.prefilter = 0;
    info.cartesian_bound = pairs;  // every pair is compared
    if (mode != MODE_EMIT) return JN_OK;
    bool done = h[0] <= cap;
    if (!done) ss.release();
    JN_TRY(out_prepare_or(c, s, h[0], *plan, [&] {
        const bool kept = done && cap;
        ss.release();
        done = done && !cap;
        return kept;
    }));
    if (h[0] && done) {
        // straight to the caller's buffer, host memory included
        JN_CUDA(c, cudaMemcpyAsync(plan->host_copy ? *plan->user_out : plan->dev, staged, h[0] * sizeof(jn_pair),
                                   cudaMemcpyDefault, c->stream));
        plan->copied = plan->host_copy;
    } else if (h[0]) {
        // compared again, every tile's pairs to their place
        JN_TRY(s.get(&off, tiles + 1));
        JN_TRY(scan_u64(c, val, off, (int64_t)tiles));
        JN_TRY(pass(MODE_EMIT, plan->dev, h[0], NlSkip()));
        JN_CUDA(c, cudaStreamSynchronize(c->stream));  // this pass reads the caller's columns
    }
    return out_finish(c, h[0], *plan);
}

// ------------------------------------------------------ allocation-free --
// A nested-loop join for callers that may not allocate device memory at all:
// code running inside a region where the application owns every byte of the
// device (a fixed memory plan, a real-time or serving loop that forbids
// cudaMalloc / cudaFree and the synchronisation they bring), or code that
// must not touch any allocator, the library's pool included.  Its scratch
// (per-tile counts, their scan and the checksum word) lives in the fixed
// device array below, so a call allocates nothing; the caller supplies the
// output buffer.
constexpr int NA_MAX_TILES = 65536;  // R tiles x S tiles per call
static __device__ __align__(256) unsigned long long g_na_scratch[2 * NA_MAX_TILES + 8];

// Device address of g_na_scratch, looked up once per device (host code
// cannot use the symbol itself as an address).
static std::mutex g_na_mu;
static void* g_na_addr[64];

static jn_status na_scratch(void** p) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return JN_ERR_CUDA;
    }
    std::lock_guard<std::mutex> g(g_na_mu);
    if (!g_na_addr[dev]) {
        void* a = nullptr;
        if (cudaGetSymbolAddress(&a, g_na_scratch) != cudaSuccess || !a) {
            cudaGetLastError();
            return JN_ERR_CUDA;
        }
        g_na_addr[dev] = a;
    }
    *p = g_na_addr[dev];
    return JN_OK;
}

// Single-block exclusive scan of n <= NA_MAX_TILES counts; out[n] = total.
static __global__ void k_na_scan(const unsigned long long* __restrict__ in, int n, unsigned long long* __restrict__ out) {
    __shared__ unsigned long long tmp[33];
    unsigned long long carry = 0;
    for (int base = 0; base < n; base += blockDim.x) {
        const int i = base + threadIdx.x;
        const unsigned long long v = i < n ? in[i] : 0ull;
        unsigned long long tot;
        const unsigned long long pre = block_excl_scan(v, tmp, &tot);
        if (i < n) out[i] = carry + pre;
        carry += tot;
    }
    if (threadIdx.x == 0) out[n] = carry;
}

template <typename K, bool HAS2>
static jn_status na_run(const jn_table* R, const jn_table* S, const jn_pred& pr, jn_pair* out, uint64_t capacity,
                        uint64_t* n_out, cudaStream_t st) {
    const int tr = 1024;
    const uint64_t gx = ceil_div((uint64_t)S->n, NLJ_STILE), gy = ceil_div((uint64_t)R->n, tr);
    const uint64_t tiles = gx * gy;
    if (tiles > NA_MAX_TILES || gy > 65535) return JN_ERR_INVALID;  // beyond the fixed scratch
    void* base = nullptr;
    JN_TRY(na_scratch(&base));
    unsigned long long* val = static_cast<unsigned long long*>(base);
    unsigned long long* off = val + NA_MAX_TILES;
    const dim3 grid((unsigned)gx, (unsigned)gy);
    const size_t smem = (size_t)tr * (sizeof(K) * (HAS2 ? 2 : 1) + 4);
    const K* rk = static_cast<const K*>(R->key);
    const K* rk2 = static_cast<const K*>(R->key2);
    const K* sk = static_cast<const K*>(S->key);
    const K* sk2 = static_cast<const K*>(S->key2);
    // the array keeps the previous call's contents: counts are rewritten for
    // every tile of this call
    k_nlj<K, HAS2, MODE_COUNT><<<grid, NLJ_T, smem, st>>>(rk, rk2, R->payload, R->n, sk, sk2, S->payload, S->n,
                                                          pr.op_a, pr.op_k, (long long)pr.band, tr, val,
                                                          nullptr, nullptr);
    k_na_scan<<<1, 1024, 0, st>>>(val, (int)tiles, off);
    if (cudaGetLastError() != cudaSuccess) return JN_ERR_CUDA;
    uint64_t total = 0;
    if (cudaMemcpyAsync(&total, off + tiles, sizeof(uint64_t), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
        cudaGetLastError();
        return JN_ERR_CUDA;
    }
    *n_out = total;
    if (total > capacity) return JN_ERR_CAPACITY;
    if (total > 0) {
        k_nlj<K, HAS2, MODE_EMIT><<<grid, NLJ_T, smem, st>>>(rk, rk2, R->payload, R->n, sk, sk2, S->payload, S->n,
                                                             pr.op_a, pr.op_k, (long long)pr.band, tr, nullptr,
                                                             reinterpret_cast<const uint64_t*>(off), out);
        if (cudaGetLastError() != cudaSuccess) return JN_ERR_CUDA;
    }
    return JN_OK;
}

template jn_status run_nlj<int32_t>(jn_ctx*, const Cols<int32_t>&, const Cols<int32_t>&,
                                    const jn_pred&, int, OutPlan*, RunResult*);
template jn_status run_nlj<int64_t>(jn_ctx*, const Cols<int64_t>&, const Cols<int64_t>&,
                                    const jn_pred&, int, OutPlan*, RunResult*);

}  // namespace jnx

using namespace jnx;

extern "C" jn_status jn_nested_loop_noalloc(const jn_table* R, const jn_table* S, const jn_pred* pred,
                                            jn_pair* out, uint64_t capacity, uint64_t* n_out, void* stream) {
    if (!R || !S || !n_out || (capacity > 0 && !out)) return JN_ERR_INVALID;
    if (R->key_type != S->key_type || (R->key_type != JN_KEY_I32 && R->key_type != JN_KEY_I64)) return JN_ERR_INVALID;
    if (R->n < 0 || S->n < 0 || R->n > INT32_MAX || S->n > INT32_MAX || R->reserved || S->reserved)
        return JN_ERR_INVALID;
    jn_pred pr;
    pr.op_a = JN_EQ;
    pr.op_k = JN_ANY;
    pr.band = -1;
    if (pred) pr = *pred;
    if (pr.op_a < JN_EQ || pr.op_a > JN_ANY || pr.op_k < JN_EQ || pr.op_k > JN_ANY) return JN_ERR_INVALID;
    // columns, output and stream on the current device (whose scratch address
    // the call looks up): nothing may be staged, no other device's array used
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return JN_ERR_CUDA;
    }
    const void* cols[6] = {R->key, R->key2, R->payload, S->key, S->key2, S->payload};
    for (const void* c : cols)
        if (c && pointer_device(c) != dev) return JN_ERR_INVALID;
    if (capacity > 0 && pointer_device(out) != dev) return JN_ERR_INVALID;
    if (((uintptr_t)out & 7) != 0) return JN_ERR_INVALID;  // pairs are stored as 8-byte words
    if (stream) {
        int sdev = -1;
        if (cudaStreamGetDevice((cudaStream_t)stream, &sdev) != cudaSuccess) {
            cudaGetLastError();
            return JN_ERR_INVALID;
        }
        if (sdev != dev) return JN_ERR_INVALID;
    }
    if (R->n == 0 || S->n == 0) {
        *n_out = 0;
        return JN_OK;
    }
    if ((R->n > 0 && !R->key) || (S->n > 0 && !S->key)) return JN_ERR_INVALID;
    const bool has2 = R->key2 && S->key2;
    cudaStream_t st = (cudaStream_t)stream;
    if (R->key_type == JN_KEY_I32)
        return has2 ? na_run<int32_t, true>(R, S, pr, out, capacity, n_out, st)
                    : na_run<int32_t, false>(R, S, pr, out, capacity, n_out, st);
    return has2 ? na_run<int64_t, true>(R, S, pr, out, capacity, n_out, st)
                : na_run<int64_t, false>(R, S, pr, out, capacity, n_out, st);
}
