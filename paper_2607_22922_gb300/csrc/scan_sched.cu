// The work lists of a batch's scans.
//
// What a query has to scan is known on the device only (k_prepare's position
// ranges, the filter's pass counts), so the split into CTAs is made there:
// k_schedule turns the batch into work items, and the scan kernels take items
// from the lists until they are empty.  A grid cut by row chunks of the whole
// index instead left most CTAs without work for a few selective queries (one
// query for 10 % of 10^6 rows: 6 of 58 CTAs busy, 64 us; 16 for 1 % of 10^7
// rows: 225 us) and let one long query end a mixed batch alone.
//
// Units of work: 256-position rounds (sorted copies), 1024-row blocks (pairs),
// and for the bitmap path blocks / 8 + passing rows / 1024 (reading a block's
// bits costs about an eighth of looking its rows up).  With w units in all,
// `slots` CTAs resident and n queries:
//   n <= slots / 2   one wave: items of ceil(w / (slots - n)) units, so that
//                    at most `slots` items arise;
//   otherwise        three to six items per slot (per_slot), a query's count
//                    rounded to nearest (every item pays its table, lists and
//                    merge);
//   pairs of about equal ranges: the count c per pair of the least
//                    ceil(n c / slots) (length / c + start), waves times an
//                    item's time.  Measured, c = 1 / 2: 512 pairs of 5 x 10^6
//                    rows at k = 100 7410 / 7010 us, of 10^6 rows 1869 / 2064;
//                    c = 5 / 7 / 14: 128 bitmap pairs of 4 x 10^6 rows at k =
//                    10 1242 / 1123 / 1178 us.  start = 128 blocks for k <= 32 and
//                    400 above fit these.
// A query's items are equal parts of its range.  Where the bitmap scan's are more
// than one wave, the first parts of all queries come first, then the second ones
// (up to the fourth): CTAs that work at the same time read the same part of the
// codes and share it in the L2, which 8 x 10^6 rows fill (512 queries of M = 16
// that 21 and 32 % of them pass, k = 200: 8946 and 12344 us query by query, 8602 and
// 11866 so; k = 10 8647 and 8470 us at 32 %; 2 x 10^6 rows the same either way).  The
// other groups gained nothing from it.  Each item writes one list of
// k keys (two for a pair), numbered so that a query's lists are contiguous;
// k_merge reads (first list, count) per query.
//
// The pairing of overlapping ranges (M = 12 and 16) comes first in the same
// kernel: see scan_pair.cu for what a pair is worth.  Its sort covers the next
// power of two of the queries (2048 keys for any batch took 14 us).  Bitmap
// queries that many rows pass are paired in their order: any two share every
// block.
#include "scan_common.cuh"

namespace ifvs {

namespace {

constexpr int kSeg = 2048;              // queries sorted and numbered together
constexpr int kSchedThreads = 1024;
// items per slot aimed at in large batches: one-query lists 4 -> 3: 1024 mixed
// ranges of 10^6 rows 700 -> 686 us, 512 of 40,000 157 -> 150; pairs 4 -> 6:
// nothing but where the waves below decide
constexpr int kListPerSlot = 3, kPairPerSlot = 6, kBitmapPerSlot = 4;
static_assert(kSeg == 2 * kSchedThreads, "one neighbour pair per thread");
static_assert(kSortedCopies <= 8, "the pairing key keeps 3 bits of the sorted copy");

// exclusive prefix of v over the block's threads (in thread order) and the
// total; wsum holds one value per warp, which every warp adds up by itself, a
// lane per warp (a loop over 32 warps' values in every thread took half a
// microsecond of shared-memory reads)
template <class T>
__device__ __forceinline__ T warp_prefix(T v, int lane) {   // inclusive
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T t = __shfl_up_sync(0xFFFFFFFFu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

template <class T>
__device__ __forceinline__ T block_prefix(T v, T* wsum, T& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const T incl = warp_prefix(v, lane);
    __syncthreads();
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    const T w = warp_prefix(lane < (int)(blockDim.x >> 5) ? wsum[lane] : T(0), lane);
    total = __shfl_sync(0xFFFFFFFFu, w, 31);
    const T before = __shfl_sync(0xFFFFFFFFu, w, (warp + 31) & 31);
    return (warp > 0 ? before : T(0)) + incl - v;
}

// v[i] <- its sum over the block's threads; wsum holds N values per warp
template <int N>
__device__ __forceinline__ void block_sums(int64_t (&v)[N], int64_t (*wsum)[32]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto warp_sum = [](int64_t x) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
        return x;
    };
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = warp_sum(v[i]);
    __syncthreads();
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < N; ++i) wsum[i][warp] = v[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = warp_sum(lane < (int)(blockDim.x >> 5) ? wsum[i][lane] : 0);
}

__device__ __forceinline__ bool pairable(const ScanPlan& x, const ScanPlan& y, int64_t min_rows) {
    if (!x.list || !y.list || x.col != y.col) return false;
    const int64_t lx = x.b - x.a, ly = y.b - y.a;
    if (lx <= 0 || ly <= 0) return false;
    const int64_t common = min(x.b, y.b) - max(x.a, y.a);
    const int64_t span = max(x.b, y.b) - min(x.a, y.a);
    return 4 * common >= 3 * max(lx, ly) && span >= min_rows;
}

// How a group of ranges is cut (see the file comment).
struct Cut {
    int64_t L;
    bool up;        // count rounded up (one wave) or to nearest
    __device__ __forceinline__ int count(int64_t len) const {
        if (len <= 0) return 0;
        const int64_t c = up ? (len + L - 1) / L : (len + L / 2) / L;
        return c < 1 ? 1 : (int)c;
    }
};

__device__ __forceinline__ Cut cut_of(int64_t work, int64_t n, const SchedGroup& g, bool equal) {
    Cut c;
    c.up = false;
    if (n <= 0) {
        c.L = 1;
        return c;
    }
    if (g.fixed > 0) {
        c.L = g.fixed;
        c.up = true;
    } else if (2 * n <= g.slots) {
        c.L = max((work + g.slots - n - 1) / (g.slots - n), g.least);
        c.up = true;
    } else if (equal) {
        // a count per lane (64-bit divisions: one lane for all took 10 us)
        const int64_t len = work / n;
        const int i = (int)(threadIdx.x & 15) + 1;
        int64_t t = i == 1 || len / i >= g.least ? (n * i + g.slots - 1) / g.slots * (len / i + g.start) : INT64_MAX;
        t = (t < INT64_MAX >> 4 ? t : INT64_MAX >> 4) << 4 | (i - 1);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) t = min(t, __shfl_xor_sync(0xFFFFFFFFu, t, o));
        c.L = max(len / ((t & 15) + 1), (int64_t)1);
    } else {
        c.L = max(work / (g.per_slot * g.slots), 8 * g.least);
    }
    // at most `cap` items in all: each query has at most len / L + 1
    if (g.cap <= n)
        c.L = (int64_t)1 << 62, c.up = false;
    else
        c.L = max(c.L, (work + g.cap - n - 1) / (g.cap - n));
    return c;
}

}  // namespace

// PARTS: the bitmap group's items part by part (a kernel of its own: the ranks'
// code cost a batch without them 3 us).
template <bool PARTS>
__global__ void __launch_bounds__(kSchedThreads) k_schedule(const ScanPlan* __restrict__ plan,
                                                            const unsigned long long* __restrict__ npass, int64_t nq,
                                                            int64_t n_blocks, PairRule rule, ScanSched s) {
    __shared__ uint64_t key[kSeg];          // pairing; then the items' prefix counts
    __shared__ uint64_t rank[PARTS ? kSeg : 1];   // of an element among those with more than c parts, c = 0..3
    __shared__ int wsum[32];
    __shared__ uint64_t wsum_rank[32];
    __shared__ int64_t wsum64[2 * kGroups][32];
    int* pre = reinterpret_cast<int*>(key);
    const int tid = threadIdx.x, nt = blockDim.x;
    int n_pairs = 0, n_bm_pairs = 0;
    int64_t pair_min_rows = plan != nullptr ? rule.span : -1;
    wait_before();
    start_dependents();   // prepare and filter are complete: the tables can start

    // no sort for a batch that cannot pair: 3/4 in common, a pair spans at most
    // 5/4 of its longer range
    if (pair_min_rows >= 0) {
        int64_t t[2] = {0, 0};   // rows, ranges wide enough
        for (int64_t q = tid; q < nq; q += nt)
            if (plan[q].list) {
                const int64_t len = plan[q].b - plan[q].a;
                t[0] += len;
                t[1] += 5 * len >= 4 * pair_min_rows;
            }
        block_sums(t, wsum64);
        if (t[0] < rule.total || t[1] == 0) pair_min_rows = -1;
    }

    // ---- pairs: sorted by (copy, range start, query), neighbours (2j, 2j + 1)
    if (pair_min_rows >= 0) {
        for (int64_t q0 = 0; q0 < nq; q0 += kSeg) {
            const int n = (int)min((int64_t)kSeg, nq - q0);
            int P = 2;
            while (P < n) P <<= 1;
            __syncthreads();
            // key = copy (3 bits) | range start (32 bits) | index in the segment
            // (11 bits); queries of the bitmap path sort last as all ones
            for (int i = tid; i < P; i += nt) {
                uint64_t kk = ~0ull;
                if (i < n) {
                    const ScanPlan p = plan[q0 + i];
                    if (p.list) kk = ((uint64_t)(p.col & 7) << 43) | ((uint64_t)(uint32_t)p.a << 11) | (uint64_t)i;
                    s.paired[q0 + i] = 0;
                }
                key[i] = kk;
            }
            for (int size = 2; size <= P; size <<= 1)
                for (int stride = size >> 1; stride > 0; stride >>= 1) {
                    __syncthreads();
                    for (int t = tid; t < P / 2; t += nt) {
                        const int i = 2 * t - (t & (stride - 1));
                        const int j = i + stride;
                        const bool up = (i & size) == 0;
                        const uint64_t x = key[i], y = key[j];
                        if ((x > y) == up) {
                            key[i] = y;
                            key[j] = x;
                        }
                    }
                }
            __syncthreads();
            for (int j0 = 0; j0 < P / 2; j0 += nt) {
                const int j = j0 + tid;
                int qa = -1, qb = -1, cnt = 0;
                if (j < P / 2) {
                    const uint64_t ka = key[2 * j], kb = key[2 * j + 1];
                    if (ka != ~0ull && kb != ~0ull) {
                        qa = (int)(q0 + (int64_t)(ka & 2047u));
                        qb = (int)(q0 + (int64_t)(kb & 2047u));
                        cnt = pairable(plan[qa], plan[qb], pair_min_rows) ? 1 : 0;
                    }
                }
                int total = 0;
                const int at = n_pairs + block_prefix(cnt, wsum, total);
                if (cnt) {
                    s.pairs[at] = make_int2(qa, qb);
                    s.paired[qa] = s.paired[qb] = 1;
                }
                n_pairs += total;
            }
        }
        __syncthreads();
    }

    // ---- bitmap queries with enough passing rows, two by two
    bool bm_pairs = rule.bm_pass >= 0 && npass != nullptr;
    if (bm_pairs) {
        int* of = reinterpret_cast<int*>(s.pairs + n_pairs);
        auto dense = [&](int64_t q) {
            return (plan == nullptr || !plan[q].list) && npass[q] > 0 && (int64_t)npass[q] >= rule.bm_pass;
        };
        int64_t n[1] = {0};
        for (int64_t q = tid; q < nq; q += nt) n[0] += dense(q);
        block_sums(n, wsum64);
        bm_pairs = n[0] > 1 && n[0] * n_blocks * kBlockRows >= rule.bm_total;
        if (bm_pairs) {
            n_bm_pairs = (int)(n[0] / 2);
            int done = 0;
            for (int64_t q0 = 0; q0 < nq; q0 += nt) {
                const int64_t q = q0 + tid;
                const bool d = q < nq && dense(q);
                int total = 0;
                const int at = done + block_prefix((int)d, wsum, total);
                const bool in = d && at < 2 * n_bm_pairs;   // an odd one stays alone
                if (in) of[at] = (int)q;
                if (q < nq && (plan == nullptr || !plan[q].list)) s.paired[q] = in;
                done += total;
            }
            __syncthreads();
        }
    }

    // lengths in units of work
    auto list_len = [&](int64_t q) -> int64_t {
        if (plan == nullptr) return 0;
        const ScanPlan p = plan[q];
        if (!p.list || p.a >= p.b || (pair_min_rows >= 0 && s.paired[q])) return 0;
        return (p.b + kRoundRows - 1) / kRoundRows - p.a / kRoundRows;
    };
    auto bm_len = [&](int64_t q) -> int64_t {
        if ((plan != nullptr && plan[q].list) || (bm_pairs && s.paired[q])) return 0;
        if (s.group[1].fixed > 0) return n_blocks;
        if (npass == nullptr) return n_blocks;
        const int64_t np = (int64_t)npass[q];
        return np == 0 ? 0 : (n_blocks + 7) / 8 + np / kBlockRows;
    };
    auto pair_span = [&](int64_t j, int64_t& lo, int64_t& hi) {
        const int2 p = s.pairs[j];
        const ScanPlan x = plan[p.x], y = plan[p.y];
        lo = min(x.a, y.a) / kBlockRows;
        hi = (max(x.b, y.b) + kBlockRows - 1) / kBlockRows;
    };
    int64_t sums[2 * kGroups] = {};
    int64_t *work = sums, *cnt = sums + kGroups;
    for (int64_t q = tid; q < nq; q += nt) {
        const int64_t l = list_len(q), b = bm_len(q);
        work[0] += l;
        cnt[0] += l > 0;
        work[1] += b;
        cnt[1] += b > 0;
    }
    for (int64_t j = tid; j < n_pairs; j += nt) {
        int64_t lo, hi;
        pair_span(j, lo, hi);
        work[2] += hi - lo;
        cnt[2] += 1;
    }
    if (tid == 0) {
        work[3] = n_bm_pairs * n_blocks;
        cnt[3] = n_bm_pairs;
    }
    block_sums(sums, wsum64);
    bool longer = false;   // a pair's span is more than 5/4 of the mean
    for (int64_t j = tid; j < n_pairs; j += nt) {
        int64_t lo, hi;
        pair_span(j, lo, hi);
        longer |= 4 * (hi - lo) * cnt[2] > 5 * work[2];
    }
    const bool equal = n_pairs > 0 && __syncthreads_or(longer ? 1 : 0) == 0;   // n_pairs: the same in every thread
    Cut cut[kGroups];
#pragma unroll
    for (int g = 0; g < kGroups; ++g) {
        cut[g] = {1, false};
        if (cnt[g] > 0) cut[g] = cut_of(work[g], cnt[g], s.group[g], g == 3 || (g == 2 && equal));
    }

    // no lists for queries that nothing passes
    for (int64_t q = tid; q < nq; q += nt) s.qlist[q] = make_int2(0, 0);
    __syncthreads();

    // items, numbered segment by segment
    int lists = 0;
#pragma unroll
    for (int g = 0; g < kGroups; ++g) {
        int items = 0;
        const int64_t n_el = g == 2 ? n_pairs : (g == 3 ? n_bm_pairs : nq);
        const int2* pairs = s.pairs + (g == 3 ? n_pairs : 0);
        if (cnt[g] == 0) {   // the same in every thread
            if (tid == 0) s.ctl[g] = s.ctl[kGroups + g] = 0;
            continue;
        }
        const bool by_part = PARTS && g == 1 && (s.group[g].fixed > 0 || 2 * cnt[g] > s.group[g].slots);
        for (int64_t e0 = 0; e0 < n_el; e0 += kSeg) {
            const int n = (int)min((int64_t)kSeg, n_el - e0);
            int total = 0, done = 0;
            uint64_t ranks = 0ull;   // 16 bits per part
            for (int i0 = 0; i0 < n; i0 += nt) {
                const int i = i0 + tid;
                int64_t len = 0;
                if (i < n) {
                    if (g == 0) {
                        len = list_len(e0 + i);
                    } else if (g == 1) {
                        len = bm_len(e0 + i);
                    } else if (g == 3) {
                        len = n_blocks;
                    } else {
                        int64_t lo, hi;
                        pair_span(e0 + i, lo, hi);
                        len = hi - lo;
                    }
                }
                const int c = i < n ? cut[g].count(len) : 0;
                const int at = done + block_prefix(c, wsum, total);
                done += total;
                if (by_part) {
                    const uint64_t has = (uint64_t)(c > 0) | (uint64_t)(c > 1) << 16 | (uint64_t)(c > 2) << 32 |
                                         (uint64_t)(c > 3) << 48;
                    uint64_t all = 0ull;
                    const uint64_t r = ranks + block_prefix(has, wsum_rank, all);
                    ranks += all;
                    if (i < n) rank[i] = r;
                }
                if (i >= n) continue;
                pre[i] = at;
                if (pair_group(g)) {
                    const int2 p = pairs[e0 + i];
                    s.qlist[p.x] = make_int2(lists + 2 * at, c);
                    s.qlist[p.y] = make_int2(lists + 2 * at + c, c);
                } else if (c > 0) {
                    s.qlist[e0 + i] = make_int2(lists + at, c);
                }
            }
            __syncthreads();
            auto field = [](uint64_t v, int c) { return (int)(v >> (16 * c) & 0xFFFFu); };
            const int f1 = field(ranks, 0), f2 = f1 + field(ranks, 1), f3 = f2 + field(ranks, 2), f4 = f3 + field(ranks, 3);
            for (int it = tid; it < done; it += nt) {
                int lo = 0, hi = n;              // the last element whose prefix is <= it
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (pre[mid] <= it)
                        lo = mid;
                    else
                        hi = mid;
                }
                const int c = it - pre[lo];
                const int nc = (lo + 1 < n ? pre[lo + 1] : done) - pre[lo];
                ScanItem w;
                int64_t a, b;
                if (pair_group(g)) {
                    const int2 p = pairs[e0 + lo];
                    a = 0;
                    b = n_blocks;
                    if (g == 2) pair_span(e0 + lo, a, b);
                    w.qa = p.x;
                    w.qb = p.y;
                    w.la = lists + 2 * pre[lo] + c;
                    w.lb = w.la + nc;
                } else {
                    w.qa = (int)(e0 + lo);
                    w.qb = -1;
                    w.la = lists + it;
                    w.lb = -1;
                    if (g == 0) {
                        const ScanPlan p = plan[e0 + lo];
                        a = p.a / kRoundRows;
                        b = (p.b + kRoundRows - 1) / kRoundRows;
                    } else {
                        a = 0;
                        b = n_blocks;
                    }
                }
                w.a = (uint32_t)(a + (b - a) * c / nc);
                w.b = (uint32_t)(a + (b - a) * (c + 1) / nc);
                int to = it;
                if (by_part) {
                    const uint64_t r = rank[lo];
                    to = c == 0   ? field(r, 0)
                         : c == 1 ? f1 + field(r, 1)
                         : c == 2 ? f2 + field(r, 2)
                         : c == 3 ? f3 + field(r, 3)
                                  : f4 + it - 4 - field(r, 0) - field(r, 1) - field(r, 2) - field(r, 3);
                }
                s.items[g][items + to] = w;
            }
            __syncthreads();   // pre is rewritten
            items += done;
            lists += (pair_group(g) ? 2 : 1) * done;
        }
        if (tid == 0) {
            s.ctl[g] = items;        // items of the list
            s.ctl[kGroups + g] = 0;  // work counter
        }
    }
}

// Bounds of the lists and the workspace's layout (offsets from `base`).
size_t scan_sched_layout(int64_t nq, int k, int64_t n_blocks, int row_bytes, const int (&slots)[kGroups],
                         int64_t chunk_blocks, const int64_t (&most)[kGroups], uint8_t* base, ScanSched* s) {
    s->by_part = n_blocks * kBlockRows * row_bytes > (int64_t)1 << 26;   // half of the L2
    size_t at = 0;
    auto take = [&](size_t bytes) {
        uint8_t* p = base + at;
        at = (at + bytes + 255) / 256 * 256;
        return p;
    };
    int64_t lists = 0;
    for (int g = 0; g < kGroups; ++g) {
        SchedGroup& G = s->group[g];
        const int64_t el = pair_group(g) ? nq / 2 : nq;
        G.slots = slots[g];
        G.least = g == 0 ? kScanWarps : (g == 1 ? 2 : 64);
        G.fixed = chunk_blocks > 0 ? chunk_blocks * (g == 0 ? kBlockRows / kRoundRows : 1) : 0;
        G.per_slot = g == 0 ? kListPerSlot : (pair_group(g) ? kPairPerSlot : kBitmapPerSlot);
        G.start = k <= 32 ? 128 : 400;
        int64_t cap = G.per_slot * (int64_t)slots[g] + el;
        if (chunk_blocks > 0) {
            int64_t per = (n_blocks + chunk_blocks - 1) / chunk_blocks + 1;
            if (per > 1024) per = 1024;
            cap = el * (per + 1);
        }
        if (cap > most[g]) cap = most[g];
        G.cap = cap;
        s->items[g] = reinterpret_cast<ScanItem*>(take(sizeof(ScanItem) * (size_t)cap));
        lists += (pair_group(g) ? 2 : 1) * cap;
    }
    s->ctl = reinterpret_cast<int*>(take(2 * kGroups * sizeof(int)));
    s->qlist = reinterpret_cast<int2*>(take(sizeof(int2) * (size_t)nq));
    s->pairs = reinterpret_cast<int2*>(take(sizeof(int2) * (size_t)(nq / 2 + 1)));
    s->paired = take((size_t)nq);
    s->partials = reinterpret_cast<uint64_t*>(take(sizeof(uint64_t) * (size_t)(lists * k)));
    return at;
}

cudaError_t launch_schedule(const ScanPlan* plan, const unsigned long long* npass, int64_t nq, int64_t n_blocks,
                            PairRule rule, const ScanSched& s, bool chain, cudaStream_t st) {
    if (nq <= 0) return cudaSuccess;
    int threads = 128;
    while (threads < kSchedThreads && threads < nq) threads <<= 1;
    return launch_kernel(s.by_part ? k_schedule<true> : k_schedule<false>, dim3(1), dim3((unsigned)threads), 0, chain,
                         st, plan, npass, nq, n_blocks, rule, s);
}

}  // namespace ifvs
