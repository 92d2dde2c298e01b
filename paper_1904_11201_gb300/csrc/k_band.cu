// Direct band join: (R.a op S.a) AND |R.k - S.k| <= band with one sorted
// index of the smaller table in global memory, probed by the larger table
// where it lies (the band form of jn_direct.cuh; Algorithm 3's regions,
// Sec. 4.2, become the index's buckets).
//
// The smaller table's rows are put in the order of buckets of k, about one
// row to a bucket, by a counting sort (count, scan, place).  A row of the
// other table finds its candidates as one contiguous range, from the offset
// of the first bucket its window [k - band, k + band] touches to the offset
// behind the last, and tests both conjuncts on each.  While index and rows
// stay in L2 (2^22 rows: 80 MB at most with int32 keys), this reads the larger
// table once where the partitioned join (k_theta.cu) moves it once and reads
// it four times.
//
// Every candidate is a read from L2, against one from shared memory there, so
// windows with many candidates belong to the partitioned join.  A sample of
// both tables estimates the candidates of a row first; past the line (below)
// nothing is built.  Where the buckets bring far more rows than the band, the
// check beside the buckets' bounds leaves the join to the partitioned one; should
// both samples be wrong by far, the probe, which counts its candidates, stops.
//
// Measured on GB300, 2^20 x 2^24 int32 rows, ms with (without) the index, at
// 1, 6, 12, 24 candidates a row: count 0.38 (0.61), 0.53 (0.65), 0.70 (0.71),
// 1.07 (0.83); checksum 0.46 (0.74), 0.73 (0.88), 1.04 (1.05), 1.67 (1.34);
// int64 checksum 0.54 (0.97), 0.85 (1.17), 1.20 (1.39), 1.92 (1.81).
//
// One or many joins run in the same launches: blocks take tiles of BD_ROWS
// rows, join by join.  Pairs go to rooms of scratch (several per large join,
// for their cursors' sake) through per-warp buffers, and one copy puts them in
// the exact allocation.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "jn_direct.cuh"
#include "jn_partition.cuh"

namespace jnx {

// Candidates a row up to which a join is taken, by what is asked of it (pairs
// written: 1 candidate 0.53 ms against 0.78, 6 candidates 0.98 against 0.90).
constexpr double BD_LINE_COUNT = 10, BD_LINE_AGG = 8, BD_LINE_EMIT = 4;
constexpr int BD_T = 256;
constexpr int BD_ROWS = 4096;      // rows per tile
constexpr int BD_BUF = 128;        // pairs a warp's buffer holds
constexpr uint64_t BD_MOST = 48;   // candidates a row past which a probe stops
constexpr int BD_SAMPLE_P = 512;   // rows sampled for the estimate: of the probing table,
constexpr int BD_SAMPLE_B = 4096;  // and of the built one, in BD_SPARTS parts
constexpr int BD_SPARTS = 64;      // (the estimate takes 9 us; 13 in 16 parts)
constexpr int BD_CHECK_B = 1024, BD_CPARTS = 16;  // and, of the built one, by k_band_ranges
// Rows of the index a row meets past which nothing is built.  What puts that
// many into a few buckets fills few of the partitioned join's groups too:
// counts with far values, 28 and 128 rows met, take 1.0 and 1.15 times its time.
constexpr double BD_MEET = 128;
constexpr uint64_t BD_ROOM = 1ull << 30;  // pairs of room at most (8 GB)
constexpr int BD_ROOMS = DJ_SEGS;  // rooms of a large join

template <typename K>
struct BandJoin {
    const K *bk, *ba;  // build side: the smaller table's k and a
    const int32_t* bpay;
    const K *pk, *pa;
    const int32_t* ppay;
    int64_t bn, pn;
    uint64_t row0;      // build rows of the joins before this one
    uint64_t off0;      // first of its offsets: `buckets` and one behind
    uint64_t most;      // candidates past which its probe stops
    uint64_t most_hits; // hits past which nothing is built
    long long band;
    uint32_t buckets;   // a power of two
    int32_t op;         // built row's a `op` probing row's a
    int32_t swap;       // the build side is S
    uint32_t room0, rooms;
};

struct BandRange {
    long long lo, hi;  // of the built k
    int shift;         // bucket of k: (k - lo) >> shift
    int pad;
};

// Per join, zeroed: bounds of k as maxima of their unsigned images, and work.
struct BandMark {
    unsigned long long hi, nlo;  // max of ord(k), max of ~ord(k)
    unsigned long long work;     // candidates met
    unsigned long long stop;     // too many, or too many to come
    unsigned long long hits;     // sampled pairs whose rows meet in the index
    unsigned long long pad;
};

struct BandRoom {
    uint64_t at, cap;  // pairs
};

__device__ __forceinline__ unsigned long long bd_ord(long long k) { return (unsigned long long)k ^ (1ull << 63); }

// A built row's two columns side by side.
template <typename K>
struct alignas(2 * sizeof(K)) BandKA {
    K k, a;
};

template <typename K>
struct BandBatch {
    const BandJoin<K>* joins;
    const uint64_t* btiles;  // n + 1 tile offsets of the build tables, and of the probe tables
    const uint64_t* ptiles;
    int n;
    BandMark* mark;
    BandRange* range;
    uint32_t* count;   // rows per bucket, then
    uint32_t* off;     // where they start (of all joins' rows)
    uint32_t* rank;    // a build row's number in its bucket
    BandKA<K>* ka;     // rows in bucket order, and their payloads
    int32_t* pay;
    const BandRoom* rooms;
    DirectLine* lines;  // one per room
};

// hits[j] += pairs within the band among the samples of join j (block
// BD_SPARTS j + x: part x of the built sample against the whole probing one).
// A single join comes by value (joins == NULL).
template <typename K>
__global__ void __launch_bounds__(BD_T)
k_band_sample(const BandJoin<K>* __restrict__ joins, BandJoin<K> only, unsigned int* __restrict__ hits) {
    __shared__ K s_k[BD_SAMPLE_B / BD_SPARTS];
    const int j = blockIdx.x / BD_SPARTS;
    const BandJoin<K> d = joins ? joins[j] : only;
    const int nb = (int)min(d.bn, (int64_t)BD_SAMPLE_B), np = (int)min(d.pn, (int64_t)BD_SAMPLE_P);
    const int b0 = (blockIdx.x % BD_SPARTS) * (BD_SAMPLE_B / BD_SPARTS), cnt = min(BD_SAMPLE_B / BD_SPARTS, nb - b0);
    if (cnt <= 0) return;  // the whole block
    for (int i = threadIdx.x; i < cnt; i += BD_T) s_k[i] = d.bk[(int64_t)(b0 + i) * d.bn / nb];
    __syncthreads();
    unsigned int m = 0;
    for (int p = threadIdx.x; p < np; p += BD_T) {
        const Interval<K> iv = band_interval<K>(d.pk[(int64_t)p * d.pn / np], d.band);
        for (int i = 0; i < cnt; i++) m += in_range(s_k[i], iv.lo, iv.span);
    }
    m = warp_sum(m);
    if ((threadIdx.x & 31) == 0 && m) atomicAdd(hits + j, m);
}

template <typename K>
__global__ void __launch_bounds__(BD_T)
k_band_bounds(BandBatch<K> b) {
    __shared__ unsigned long long s_hi[BD_T / 32], s_nlo[BD_T / 32];
    const uint64_t tiles = b.btiles[b.n];
    for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int j = find_segment(b.btiles, b.n, t);
        const int64_t r0 = (int64_t)(t - b.btiles[j]) * BD_ROWS, end = min(b.joins[j].bn, r0 + BD_ROWS);
        const K* k = b.joins[j].bk;
        unsigned long long hi = 0, nlo = 0;
        for (int64_t i = r0 + threadIdx.x; i < end; i += BD_T) {
            const unsigned long long o = bd_ord((long long)k[i]);
            hi = max(hi, o);
            nlo = max(nlo, ~o);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
            nlo = max(nlo, __shfl_xor_sync(0xffffffffu, nlo, o));
        }
        __syncthreads();
        if ((threadIdx.x & 31) == 0) {
            s_hi[threadIdx.x >> 5] = hi;
            s_nlo[threadIdx.x >> 5] = nlo;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < BD_T / 32; w++) {
                hi = max(hi, s_hi[w]);
                nlo = max(nlo, s_nlo[w]);
            }
            atomicMax(&b.mark[j].hi, hi);
            atomicMax(&b.mark[j].nlo, nlo);
        }
    }
}

__device__ __forceinline__ uint64_t bd_bucket(const BandRange& r, long long k) {
    return ((uint64_t)k - (uint64_t)r.lo) >> r.shift;
}

// The joins' ranges (the first of a join's BD_CPARTS blocks), and mark[j].hits +=
// pairs of sampled rows that meet in the index: the built row lies in a bucket
// that the other's window touches (a block takes a part of the built sample).  The index pays
// for these and not for the rows inside the band alone: one value far from the
// others puts all of them into a few buckets.  A join with more than most_hits
// is left to the partitioned join before it is built; its rows are what every
// window's warp scanned before the probe's own limit was seen (2^16 x 2^16 int32
// rows, one key 300 times further out than the others' range: 0.88 ms, 0.27 now,
// 0.20 partitioned at once).
template <typename K>
__global__ void __launch_bounds__(BD_T)
k_band_ranges(BandBatch<K> b) {
    __shared__ uint64_t s_b[BD_CHECK_B / BD_CPARTS];
    const int j = blockIdx.x / BD_CPARTS, part = blockIdx.x % BD_CPARTS;
    const uint64_t most_hits = b.joins[j].most_hits;
    if (part && most_hits == ~0ull) return;
    BandRange g;
    g.hi = (long long)(b.mark[j].hi ^ (1ull << 63));
    g.lo = (long long)(~b.mark[j].nlo ^ (1ull << 63));
    const uint64_t width = (uint64_t)g.hi - (uint64_t)g.lo;
    const uint32_t buckets = b.joins[j].buckets;
    // the smallest shift with width >> shift < buckets, a power of two
    g.shift = width >= buckets ? (64 - __clzll((long long)width)) - (31 - __clz((int)buckets)) : 0;
    g.pad = 0;
    if (part == 0 && threadIdx.x == 0) b.range[j] = g;
    if (most_hits == ~0ull) return;
    const BandJoin<K> d = b.joins[j];
    const int nb = (int)min(d.bn, (int64_t)BD_CHECK_B), np = (int)min(d.pn, (int64_t)BD_SAMPLE_P);
    const int b0 = part * (BD_CHECK_B / BD_CPARTS), cnt = min(BD_CHECK_B / BD_CPARTS, nb - b0);
    if (cnt <= 0) return;  // the whole block
    for (int i = threadIdx.x; i < cnt; i += BD_T) s_b[i] = bd_bucket(g, (long long)d.bk[(int64_t)(b0 + i) * d.bn / nb]);
    __syncthreads();
    unsigned int m = 0;
    for (int p = threadIdx.x; p < np; p += BD_T) {
        const Interval<K> iv = band_interval<K>(d.pk[(int64_t)p * d.pn / np], d.band);
        const long long first = (long long)iv.lo, last = (long long)(K)((decltype(iv.span))iv.lo + iv.span);
        if (last < g.lo || first > g.hi) continue;
        const uint64_t lo = bd_bucket(g, max(first, g.lo)), span = bd_bucket(g, min(last, g.hi)) - lo;
        for (int i = 0; i < cnt; i++) m += s_b[i] - lo <= span;
    }
    m = warp_sum(m);
    if ((threadIdx.x & 31) == 0 && m) atomicAdd(&b.mark[j].hits, (unsigned long long)m);
}

template <typename K>
__global__ void __launch_bounds__(BD_T)
k_band_count(BandBatch<K> b) {
    const uint64_t tiles = b.btiles[b.n];
    for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int j = find_segment(b.btiles, b.n, t);
        if (b.mark[j].hits > b.joins[j].most_hits) {
            if (threadIdx.x == 0) b.mark[j].stop = 1;
            continue;
        }
        const BandJoin<K> d = b.joins[j];
        const BandRange r = b.range[j];
        const int64_t r0 = (int64_t)(t - b.btiles[j]) * BD_ROWS, end = min(d.bn, r0 + BD_ROWS);
        for (int64_t i = r0 + threadIdx.x; i < end; i += BD_T)
            b.rank[d.row0 + i] = atomicAdd(b.count + d.off0 + bd_bucket(r, (long long)d.bk[i]), 1u);
    }
}

template <typename K>
__global__ void __launch_bounds__(BD_T)
k_band_place(BandBatch<K> b) {
    const uint64_t tiles = b.btiles[b.n];
    for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int j = find_segment(b.btiles, b.n, t);
        if (b.mark[j].stop) continue;
        const BandJoin<K> d = b.joins[j];
        const BandRange r = b.range[j];
        const int64_t r0 = (int64_t)(t - b.btiles[j]) * BD_ROWS, end = min(d.bn, r0 + BD_ROWS);
        for (int64_t i = r0 + threadIdx.x; i < end; i += BD_T) {
            const K k = d.bk[i];
            const uint32_t at = b.off[d.off0 + bd_bucket(r, (long long)k)] + b.rank[d.row0 + i];
            b.ka[at] = BandKA<K>{k, d.ba[i]};
            b.pay[at] = d.bpay ? d.bpay[i] : (int32_t)i;
        }
    }
}

// Emit: pairs to their join's rooms in `out` (off == NULL), or, for the joins
// one of whose rooms was too small, to out + off[j] in a second pass.
template <typename K, int MODE>
__global__ void __launch_bounds__(BD_T, 4)
k_band_probe(BandBatch<K> b, jn_pair* __restrict__ out, const uint64_t* __restrict__ off,
             const uint8_t* __restrict__ redo) {
    __shared__ int2 s_buf[MODE == MODE_EMIT ? BD_T / 32 : 1][MODE == MODE_EMIT ? BD_BUF : 1];
    const int lane = threadIdx.x & 31;
    int2* const buf = s_buf[MODE == MODE_EMIT ? threadIdx.x >> 5 : 0];
    const uint64_t tiles = b.ptiles[b.n];
    for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int j = find_segment(b.ptiles, b.n, t);
        if (MODE == MODE_EMIT && off && !redo[j]) continue;
        const BandJoin<K> d = b.joins[j];
        const BandRange g = b.range[j];
        const int64_t r0 = (int64_t)(t - b.ptiles[j]) * BD_ROWS, end = min(d.pn, r0 + BD_ROWS);
        const uint32_t room = d.room0 + (uint32_t)((t - b.ptiles[j]) % d.rooms);
        DirectLine* line = b.lines + room;
        uint64_t cap = 0;
        int2* to = reinterpret_cast<int2*>(out);
        unsigned long long* cursor = &line->total;
        if (MODE == MODE_EMIT) {
            if (off) {
                to += off[j];
                cap = off[j + 1] - off[j];
                cursor = &b.lines[d.room0].cursor;
            } else {
                to += b.rooms[room].at;
                cap = b.rooms[room].cap;
            }
        }
        uint32_t fill = 0;
        auto reserve = [&](unsigned long long n, unsigned long long* at) {
            unsigned long long a = 0;
            if (lane == 0) a = atomicAdd(cursor, n);
            *at = __shfl_sync(0xffffffffu, a, 0);
            return *at + n <= cap;
        };
        auto flush = [&]() {
            __syncwarp();
            unsigned long long at;
            if (reserve(fill, &at))
                for (uint32_t q = lane; q < fill; q += 32) to[at + q] = buf[q];
            fill = 0;
            __syncwarp();
        };
        unsigned long long acc = 0, csum = 0, work = 0;
        const bool first_pass = MODE != MODE_EMIT || !off;  // the second pass writes what the first counted
        if (first_pass && __shfl_sync(0xffffffffu, *(volatile unsigned long long*)&b.mark[j].stop, 0)) continue;
        K kn{}, an{};
        int32_t pn = 0;
        auto load = [&](int64_t i) {
            if (i >= end) return;
            kn = d.pk[i];
            an = d.pa[i];
            if (MODE != MODE_COUNT) pn = d.ppay ? d.ppay[i] : (int32_t)i;
        };
        load(r0 + threadIdx.x);
        for (int64_t w0 = r0 + (threadIdx.x & ~31); w0 < end; w0 += BD_T) {
            const int64_t i = w0 + lane;
            const K k = kn, a = an;
            const int32_t pay = pn;
            load(i + BD_T);
            uint32_t c0 = 0, c1 = 0;
            Interval<K> ia{}, ib{};
            if (i < end) {
                ia = op_interval<K>(d.op, a);
                ib = band_interval<K>(k, d.band);
                const long long first = (long long)ib.lo;
                const long long last = (long long)(K)((decltype(ib.span))ib.lo + ib.span);
                if (last >= g.lo && first <= g.hi) {
                    c0 = __ldg(b.off + d.off0 + bd_bucket(g, max(first, g.lo)));
                    c1 = __ldg(b.off + d.off0 + bd_bucket(g, min(last, g.hi)) + 1);
                }
            }
            work += c1 - c0;
            // 32 candidates of every row at a time
            while (__any_sync(0xffffffffu, c0 < c1)) {
                uint32_t mask = 0;
                const uint32_t n = min(32u, c1 - c0);
                for (uint32_t e = 0; e < n; e += 4) {
                    BandKA<K> x[4];
#pragma unroll
                    for (int u = 0; u < 4; u++)  // up to three rows past the range are read and left out
                        x[u] = b.ka[c0 + e + u];
#pragma unroll
                    for (int u = 0; u < 4; u++)
                        if (in_range(x[u].k, ib.lo, ib.span) && iv_test(ia, x[u].a) && e + u < n) mask |= 1u << (e + u);
                }
                const uint32_t m = __popc(mask);
                if (MODE == MODE_COUNT) {
                    acc += m;
                } else if (MODE == MODE_AGG) {
                    acc += m;
                    if (mask) {
                        unsigned long long f = 0;
                        for (uint32_t q = mask; q; q &= q - 1) {
                            const int32_t bp = b.pay[c0 + __ffs(q) - 1];
                            f += d.swap ? chk_g(bp) : chk_f(bp);
                        }
                        csum += f * (d.swap ? chk_f(pay) : chk_g(pay));
                    }
                } else {
                    const uint32_t incl = warp_incl_scan(m);
                    const uint32_t tot = __shfl_sync(0xffffffffu, incl, 31);
                    if (tot) {
                        if (fill + tot > (uint32_t)BD_BUF && fill) flush();
                        int2* o = buf + fill;
                        bool room_left = true;
                        if (tot > (uint32_t)BD_BUF) {
                            unsigned long long at;
                            room_left = reserve(tot, &at);
                            o = to + at;
                        } else {
                            fill += tot;
                        }
                        o += incl - m;
                        if (room_left)
                            for (uint32_t q = mask; q; q &= q - 1) {
                                const int32_t bp = b.pay[c0 + __ffs(q) - 1];
                                *o++ = d.swap ? make_int2(pay, bp) : make_int2(bp, pay);
                            }
                    }
                }
                c0 += n;
            }
            // the join's candidates so far; too many: left to the partitioned join
            if (first_pass && __any_sync(0xffffffffu, work >= 4096)) {
                const unsigned long long sum = warp_sum(work);
                unsigned long long before = 0;
                if (lane == 0) before = atomicAdd(&b.mark[j].work, sum);
                before = __shfl_sync(0xffffffffu, before, 0);
                work = 0;
                if (before + sum > d.most) {
                    if (lane == 0) b.mark[j].stop = 1;
                    break;
                }
            }
        }
        if (MODE == MODE_EMIT) {
            if (fill) flush();
        } else {
            warp_add_to(cursor, acc);
            if (MODE == MODE_AGG) warp_add_to(&b.lines[d.room0].chk, csum);
        }
        if (first_pass) warp_add_to(&b.mark[j].work, work);
    }
}

// The rooms' pairs to their places: BD_ROWS pairs of one room per block and round.
__global__ void __launch_bounds__(256)
k_band_gather(const uint64_t* __restrict__ staged, const BandRoom* __restrict__ rooms,
              const uint64_t* __restrict__ place, const uint64_t* __restrict__ chunks, int n, uint64_t* __restrict__ out) {
    const uint64_t total = chunks[n];
    for (uint64_t c = blockIdx.x; c < total; c += gridDim.x) {
        const int j = find_segment(chunks, n, c);
        const uint64_t q0 = (c - chunks[j]) * BD_ROWS;
        const uint64_t m = min((uint64_t)BD_ROWS, place[j + 1] - place[j] - q0);
        const uint64_t* src = staged + rooms[j].at + q0;
        uint64_t* dst = out + place[j] + q0;
        for (uint64_t e = threadIdx.x; e < m; e += 256) dst[e] = __ldcs(src + e);
    }
}

template <typename K, int MODE>
struct BandDirectRun : BandDirect {
    Scratch s, ss;
    jn_ctx* c;
    int n;
    BandBatch<K> b{};
    std::vector<BandJoin<K>> joins;
    std::vector<BandRoom> rooms;
    std::vector<uint64_t> found;  // pairs per room
    std::vector<unsigned char> host;  // what the copies to the device read
    std::vector<uint64_t> words;
    jn_pair* staged = nullptr;
    uint64_t btiles = 0, ptiles = 0;

    BandDirectRun(jn_ctx* ctx, int count) : s(ctx), ss(ctx), c(ctx), n(count) {}

    dim3 grid(const void* fn, uint64_t tiles) const {
        int per = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, BD_T, 0) != cudaSuccess) {
            cudaGetLastError();
            per = 1;
        }
        return dim3((unsigned)std::min<uint64_t>(std::max<uint64_t>(tiles, 1), (uint64_t)std::max(per, 1) * c->num_sms));
    }

    jn_status prepare(const Cols<K>* Rs, const Cols<K>* Ss, const int* ops, const int64_t* bands) {
        joins.resize(n);
        stopped.assign(n, 0);
        for (int i = 0; i < n; i++) {
            const bool swap = Ss[i].n < Rs[i].n;
            const Cols<K>&B = swap ? Ss[i] : Rs[i], &P = swap ? Rs[i] : Ss[i];
            BandJoin<K>& d = joins[i];
            d = BandJoin<K>{};
            d.bk = B.key2, d.ba = B.key, d.bpay = B.pay, d.bn = B.n;
            d.pk = P.key2, d.pa = P.key, d.ppay = P.pay, d.pn = B.n ? P.n : 0;
            d.band = bands[i];
            d.swap = swap;
            // the test is made on the built row: mirrored when that is S's
            static const int mirror[7] = {JN_EQ, JN_NE, JN_GT, JN_GE, JN_LT, JN_LE, JN_ANY};
            d.op = swap ? mirror[ops[i]] : ops[i];
        }
        // candidates a row, estimated; joins past the line are left out
        std::vector<double> est(n);
        JN_TRY(estimate(est.data()));
        const double line = MODE == MODE_EMIT ? BD_LINE_EMIT : MODE == MODE_AGG ? BD_LINE_AGG : BD_LINE_COUNT;
        std::vector<uint64_t> bt(n + 1, 0), pt(n + 1, 0);
        uint64_t rows = 0, offs = 0, stage = 0;
        for (int i = 0; i < n; i++) {
            BandJoin<K>& d = joins[i];
            if (est[i] > line) {
                stopped[i] = 1;
                d.bn = d.pn = 0;
            }
            d.row0 = rows, d.off0 = offs;
            d.buckets = 64;
            while (d.buckets < (uint64_t)d.bn) d.buckets <<= 1;
            d.most = BD_MOST * (uint64_t)d.pn + 65536;
            // sampled pairs that meet where a row meets BD_MEET, with room for
            // chance; small joins meet few rows at worst
            const double meet = d.bn ? BD_MEET * (double)std::min(d.pn, (int64_t)BD_SAMPLE_P) *
                                           (double)std::min(d.bn, (int64_t)BD_CHECK_B) / (double)d.bn
                                     : 0;
            const bool small = (double)d.bn * (double)d.pn < (double)(1u << 28);
            d.most_hits = small ? ~0ull : (uint64_t)(meet + 3 * sqrt(meet) + 4);
            d.room0 = (uint32_t)rooms.size();
            d.rooms = d.pn >= (1 << 21) ? BD_ROOMS : 1;
            const uint64_t cap =
                MODE == MODE_EMIT && d.pn ? (uint64_t)((1.25 + est[i]) * (double)d.pn) / d.rooms + 4096 : 0;
            for (uint32_t r = 0; r < d.rooms; r++) {
                rooms.push_back(BandRoom{stage, cap});
                stage += cap;
            }
            rows += (uint64_t)d.bn;
            offs += (uint64_t)d.buckets + 1;
            bt[i + 1] = bt[i] + ceil_div((uint64_t)d.bn, BD_ROWS);
            pt[i + 1] = pt[i] + ceil_div((uint64_t)d.pn, BD_ROWS);
        }
        offsets.assign((size_t)n + 1, 0);
        redo.assign(n, 0);
        if (rows == 0) return JN_OK;
        if (rows + 4 > UINT32_MAX) return JN_ERR_OOM;  // beyond 32-bit offsets: the partitioned join
        if (stage > BD_ROOM) {  // no room kept: the first pass counts, the second writes
            for (BandRoom& r : rooms) r = BandRoom{0, 0};
            stage = 0;
        }
        btiles = bt[n];
        ptiles = pt[n];
        // one array of words for what the host sends, one of what starts as zeros
        const size_t jb = sizeof(BandJoin<K>) * n, tb = 8 * (size_t)(n + 1), rb = sizeof(BandRoom) * rooms.size();
        host.resize(jb + 2 * tb + rb);
        memcpy(host.data(), joins.data(), jb);
        memcpy(host.data() + jb, bt.data(), tb);
        memcpy(host.data() + jb + tb, pt.data(), tb);
        memcpy(host.data() + jb + 2 * tb, rooms.data(), rb);
        static_assert(sizeof(BandJoin<K>) % 8 == 0, "the tile offsets follow, 8-byte aligned");
        const size_t lines = sizeof(DirectLine) * rooms.size(), marks = sizeof(BandMark) * n, counts = 4 * offs;
        unsigned char *dev, *zeroed;
        JN_TRY(s.get(&dev, host.size()));
        JN_TRY(s.get(&zeroed, lines + marks + counts));
        JN_TRY(s.get(&b.range, (size_t)n));
        JN_TRY(s.get(&b.off, offs + 1));
        JN_TRY(s.get(&b.rank, rows));
        JN_TRY(s.get(&b.ka, rows + 4));  // the last candidates are read four at a time
        JN_TRY(s.get(&b.pay, rows));
        if (stage) JN_TRY(ss.get(&staged, stage));
        b.joins = reinterpret_cast<BandJoin<K>*>(dev);
        b.btiles = reinterpret_cast<uint64_t*>(dev + jb);
        b.ptiles = reinterpret_cast<uint64_t*>(dev + jb + tb);
        b.rooms = reinterpret_cast<BandRoom*>(dev + jb + 2 * tb);
        b.n = n;
        b.lines = reinterpret_cast<DirectLine*>(zeroed);
        b.mark = reinterpret_cast<BandMark*>(zeroed + lines);
        b.count = reinterpret_cast<uint32_t*>(zeroed + lines + marks);
        JN_CUDA(c, cudaMemcpyAsync(dev, host.data(), host.size(), cudaMemcpyHostToDevice, c->stream));
        GraphPhase gp(c, c->tune.graphs != 0 && !c->profiling);
        JN_TRY(gp.begin());
        const jn_status st = queue(zeroed, lines + marks + counts, (int64_t)offs);
        if (st != JN_OK) {
            gp.abort();
            return st;
        }
        JN_TRY(gp.end_and_run());
        // pairs (and checksums) per room, candidates and stops per join; a single
        // join's fit the context's page-locked words
        found.resize(rooms.size());
        std::vector<uint64_t> chks(rooms.size(), 0), line2;
        std::vector<BandMark> m(n);
        if (n > 1) line2.resize(2 * rooms.size());
        uint64_t* lw = n > 1 ? line2.data() : c->h_small;
        void* mw = n > 1 ? (void*)m.data() : (void*)(c->h_small + 2 * BD_ROOMS);
        static_assert(2 * BD_ROOMS + sizeof(BandMark) / 8 < 63, "a single join's results fit the page-locked words");
        JN_CUDA(c, cudaMemcpy2DAsync(lw, 16, b.lines, sizeof(DirectLine), 16, rooms.size(), cudaMemcpyDeviceToHost,
                                     c->stream));
        JN_CUDA(c, cudaMemcpyAsync(mw, b.mark, marks, cudaMemcpyDeviceToHost, c->stream));
        JN_CUDA(c, cudaStreamSynchronize(c->stream));
        if (n == 1) memcpy(&m[0], mw, sizeof(BandMark));
        for (size_t r = 0; r < rooms.size(); r++) {
            found[r] = lw[2 * r];
            chks[r] = lw[2 * r + 1];
        }
        for (int i = 0; i < n; i++) {
            uint64_t pairs = 0;
            stopped[i] |= m[i].stop != 0;
            for (uint32_t r = joins[i].room0; r < joins[i].room0 + joins[i].rooms; r++) {
                if (stopped[i]) found[r] = 0;
                pairs += found[r];
                if (MODE == MODE_EMIT && found[r] > rooms[r].cap) redo[i] = 1;
                checksum += stopped[i] ? 0 : chks[r];
            }
            candidates += stopped[i] ? 0 : m[i].work;
            buckets += joins[i].buckets;
            offsets[i + 1] = offsets[i] + pairs;
        }
        tiles = ptiles;
        total = offsets[n];
        return JN_OK;
    }

    // candidates of a probing row of each join, from the samples
    jn_status estimate(double* est) {
        Scratch t(c);
        BandJoin<K>* dj = nullptr;
        unsigned int* hits;
        JN_TRY(t.get(&hits, (size_t)n));
        if (n > 1) {
            JN_TRY(t.get(&dj, (size_t)n));
            JN_CUDA(c, cudaMemcpyAsync(dj, joins.data(), sizeof(BandJoin<K>) * n, cudaMemcpyHostToDevice, c->stream));
        }
        JN_TRY(zero(c, hits, sizeof(unsigned int) * n));
        JN_TRY(launch(c, K_BAND_BUILD, k_band_sample<K>, dim3(BD_SPARTS * (unsigned)n), dim3(BD_T), 0,
                      (const BandJoin<K>*)dj, joins[0], hits));
        std::vector<unsigned int> many(n > 1 ? n : 0);
        unsigned int* h = n > 1 ? many.data() : reinterpret_cast<unsigned int*>(c->h_small);  // page-locked
        JN_CUDA(c, cudaMemcpyAsync(h, hits, sizeof(unsigned int) * n, cudaMemcpyDeviceToHost, c->stream));
        JN_CUDA(c, cudaStreamSynchronize(c->stream));
        for (int i = 0; i < n; i++) {
            const double nb = (double)std::min(joins[i].bn, (int64_t)BD_SAMPLE_B);
            const double np = (double)std::min(joins[i].pn, (int64_t)BD_SAMPLE_P);
            est[i] = np > 0 ? (double)h[i] / np * ((double)joins[i].bn / nb) : 0;
        }
        return JN_OK;
    }

    jn_status queue(void* zeroed, size_t bytes, int64_t offs) {
        JN_TRY(zero(c, zeroed, bytes));
        auto kb = k_band_bounds<K>;
        auto kc = k_band_count<K>;
        auto kl = k_band_place<K>;
        auto kp = k_band_probe<K, MODE>;
        JN_TRY(launch(c, K_MINMAX, kb, grid((const void*)kb, btiles), dim3(BD_T), 0, b));
        JN_TRY(launch(c, K_MINMAX, k_band_ranges<K>, dim3(BD_CPARTS * (unsigned)n), dim3(BD_T), 0, b));
        JN_TRY(launch(c, K_BAND_BUILD, kc, grid((const void*)kc, btiles), dim3(BD_T), 0, b));
        JN_TRY(scan_u32_u32(c, b.count, b.off, offs));
        JN_TRY(launch(c, K_BAND_BUILD, kl, grid((const void*)kl, btiles), dim3(BD_T), 0, b));
        return launch(c, K_BAND_PROBE, kp, grid((const void*)kp, ptiles), dim3(BD_T), 0, b, staged,
                      (const uint64_t*)nullptr, (const uint8_t*)nullptr);
    }

    std::vector<uint8_t> redo;  // joins one of whose rooms was too small

    jn_status emit(jn_ctx*, jn_pair* out) override {
        if (total == 0) return JN_OK;
        const int nr = (int)rooms.size();
        if (n == 1 && !redo[0]) {  // one join: its rooms follow one another, all of a size
            DirectResult r{};
            for (int i = 0; i < nr; i++) r.counts.n[i] = found[i];
            r.total = total;
            return direct_gather<uint64_t, 1>(c, K_BAND_PROBE, staged, (uint32_t)nr, rooms[0].cap, r, out);
        }
        // places of the rooms' pairs, chunks of those to copy, join offsets, redo flags
        words.assign((size_t)2 * (nr + 1) + n + 1 + (n + 7) / 8, 0);
        uint64_t *place = words.data(), *chunks = place + nr + 1, *offw = chunks + nr + 1;
        bool again = false;
        for (int i = 0; i < n; i++)
            for (uint32_t r = joins[i].room0; r < joins[i].room0 + joins[i].rooms; r++) {
                place[r + 1] = place[r] + found[r];
                chunks[r + 1] = chunks[r] + (redo[i] ? 0 : ceil_div(found[r], BD_ROWS));
            }
        for (int i = 0; i <= n; i++) offw[i] = offsets[i];
        for (int i = 0; i < n; i++) {
            reinterpret_cast<uint8_t*>(offw + n + 1)[i] = redo[i];
            again |= redo[i] != 0;
        }
        uint64_t* d;
        JN_TRY(s.get(&d, words.size()));
        JN_CUDA(c, cudaMemcpyAsync(d, words.data(), 8 * words.size(), cudaMemcpyHostToDevice, c->stream));
        JN_TRY(launch(c, K_BAND_PROBE, k_band_gather,
                      dim3((unsigned)std::min<uint64_t>(std::max<uint64_t>(chunks[nr], 1), 8 * (uint64_t)c->num_sms)),
                      dim3(256), 0, reinterpret_cast<const uint64_t*>(staged), b.rooms, (const uint64_t*)d,
                      (const uint64_t*)(d + nr + 1), nr, reinterpret_cast<uint64_t*>(out)));
        if (again) {
            auto kp = k_band_probe<K, MODE_EMIT>;
            const uint64_t* d_off = d + 2 * (nr + 1);
            JN_TRY(launch(c, K_BAND_PROBE, kp, grid((const void*)kp, ptiles), dim3(BD_T), 0, b, out, d_off,
                          reinterpret_cast<const uint8_t*>(d_off + n + 1)));
            JN_CUDA(c, cudaStreamSynchronize(c->stream));  // this pass reads the caller's columns
        }
        return JN_OK;
    }
};

bool band_direct_takes(const jn_ctx* c, int64_t nr, int64_t ns) {
    return c->tune.theta_groups == 0 && !c->mem_limit && !c->admit && (uint64_t)std::min(nr, ns) <= DJ_MAX;
}

template <typename K>
jn_status band_direct_prepare(jn_ctx* c, int n, const Cols<K>* Rs, const Cols<K>* Ss, const int* ops,
                              const int64_t* bands, int mode, std::unique_ptr<BandDirect>* run) {
    auto go = [&](auto* r) -> jn_status {
        std::unique_ptr<BandDirect> own(r);
        JN_TRY(r->prepare(Rs, Ss, ops, bands));
        *run = std::move(own);
        return JN_OK;
    };
    if (mode == MODE_EMIT) return go(new BandDirectRun<K, MODE_EMIT>(c, n));
    if (mode == MODE_AGG) return go(new BandDirectRun<K, MODE_AGG>(c, n));
    return go(new BandDirectRun<K, MODE_COUNT>(c, n));
}

template jn_status band_direct_prepare<int32_t>(jn_ctx*, int, const Cols<int32_t>*, const Cols<int32_t>*, const int*,
                                                const int64_t*, int, std::unique_ptr<BandDirect>*);
template jn_status band_direct_prepare<int64_t>(jn_ctx*, int, const Cols<int64_t>*, const Cols<int64_t>*, const int*,
                                                const int64_t*, int, std::unique_ptr<BandDirect>*);

}  // namespace jnx
