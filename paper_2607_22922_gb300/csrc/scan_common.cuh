// Stage 2 of §2 (Rank) with the per-CTA part of stage 3 (Select): every
// passing row v gets dist(v) = sum_m LUT[m][code_v[m]] (the weighted ADC
// form of the printed score), and each CTA keeps the k smallest
// (dist, row id) of its chunk exactly.
//
// Work split.  A CTA of 8 warps takes items, parts of a query's rows, from a
// list made on the device (scan_sched.cu).  Warp w of the bitmap path owns
// the item's bitmap blocks b0 + w, b0 + w + 8, ...; lane l owns, in each of
// them, the 32 rows b*1024 + 32*j + l, whose pass bits form its lane-major
// bitmap word.
//
// LUT placement.  The scan issues one shared-memory load per code byte, so
// bank conflicts set its speed.  The table of query q is stored as 256 rows
// (one per codeword) of S words, S a multiple of 32, word w of row c holding
// LUT[w mod M][c] for w < M + 31.  Row i's codes are stored rotated by
// (i mod 32) mod M, so the lane that owns row i (lane i mod 32) reads at
// step s the code of subspace (l + s) mod M and finds its entry at word
// l + s of that codeword's row: bank (l + s) mod 32, distinct across the
// warp whatever the codes.  For M = 16 the row stride is 256 bytes and the
// address is one byte permute, code * 256 + 4l, with the table base and the
// step 4s in the load's immediate offset (the table starts the CTA's dynamic
// shared memory, whose address the kernel checks).
//
// Compaction.  Each lane visits only its own passing rows, so it keeps its
// residue class and the conflict-free banks at any selectivity.  The warp's
// bitmap words sit in a ring of 16 blocks in shared memory (lane l's word in
// bank l); lanes advance through the ring at their own pace, eight rows per
// round, and the ring is refilled by halves, from words prefetched into
// registers, once every lane has left the older half.  Lanes at different
// blocks read rows that lie far apart, one cache line per lane; a block
// with at least kDenseRows passing rows (of 1024) is therefore taken in
// lockstep instead: each lane stops at it until the whole warp has arrived,
// then the warp walks its 32 columns, 32 neighbouring rows per load, with
// the lanes whose row fails masked.
//
// Top-k.  Each warp keeps a sorted list of its KP best keys (in registers for
// k <= 64, a key or two per lane) and a candidate area; a key (dist bits << 32 |
// row) enters the area when it is below the bound of its CTA (the smallest of
// the warps' k-th keys and the largest of their ceil(k / warps)-th ones), and a
// full area is sorted and merged.  Keys are unique (row ids are), so the result
// is exact and independent of scheduling.  At the end the warps' lists are
// merged pairwise and warp 0 writes the CTA's k keys.
//
// The tile constants (warps per CTA, ring depth, rows per round) were chosen
// by measurement on the 10^8-row workload; the macros below only exist to
// rebuild variants for such sweeps.
#pragma once
#include <climits>

#include "internal.cuh"

namespace ifvs {

#ifndef IFVS_SCAN_WARPS
#define IFVS_SCAN_WARPS 8
#endif
#ifndef IFVS_SCAN_RING
#define IFVS_SCAN_RING 16
#endif
#ifndef IFVS_SCAN_ROWS
#define IFVS_SCAN_ROWS 8
#endif
#ifndef IFVS_SCAN_DENSE
#define IFVS_SCAN_DENSE 448
#endif
constexpr int kScanWarps = IFVS_SCAN_WARPS;
constexpr int kScanThreads = kScanWarps * 32;
constexpr int kRing = IFVS_SCAN_RING;    // bitmap words per lane in the ring
constexpr int kHalf = kRing / 2;
constexpr int kU = IFVS_SCAN_ROWS;       // rows per lane per round (even)
constexpr int kDenseRows = IFVS_SCAN_DENSE;   // passing rows from which a block goes in lockstep
static_assert(kRing <= 32 && 32 % kU == 0, "one mask bit per ring slot; whole column groups");

__device__ __forceinline__ void warp_sort(uint64_t* a, int n, int lane) {
    for (int size = 2; size <= n; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            __syncwarp();
            for (int t = lane; t < (n >> 1); t += 32) {
                const int i = 2 * t - (t & (stride - 1));
                const int j = i + stride;
                const bool up = (i & size) == 0;
                const uint64_t x = a[i], y = a[j];
                if ((x > y) == up) {
                    a[i] = y;
                    a[j] = x;
                }
            }
        }
    __syncwarp();
}

// a[0, n) and a[n, 2n) ascending (n a power of two) -> a[0, n) holds the n
// smallest keys of both, ascending; a[n, 2n) is left unspecified.  The first
// step pairs a[i] with a[2n-1-i] (the second run read backwards, which makes
// the 2n keys one bitonic sequence) and keeps the smaller key: the n smallest
// of the union, as a bitonic sequence; the half-cleaners of a bitonic merge
// then sort it.
__device__ __forceinline__ void warp_merge_low(uint64_t* a, int n, int lane) {
    __syncwarp();
    for (int i = lane; i < n; i += 32) {
        const uint64_t x = a[i], y = a[2 * n - 1 - i];
        if (y < x) a[i] = y;
    }
    for (int stride = n >> 1; stride > 0; stride >>= 1) {
        __syncwarp();
        for (int t = lane; t < (n >> 1); t += 32) {
            const int i = 2 * t - (t & (stride - 1));
            const int j = i + stride;
            const uint64_t x = a[i], y = a[j];
            if (x > y) {
                a[i] = y;
                a[j] = x;
            }
        }
    }
    __syncwarp();
}

__device__ __forceinline__ uint64_t min_max_step(uint64_t x, int j, bool low) {
    const uint64_t y = __shfl_xor_sync(0xFFFFFFFFu, x, j);
    return (x < y) == low ? x : y;
}

// 32 keys, one per lane, descending
__device__ __forceinline__ uint64_t sort32_down(uint64_t c, int lane) {
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
        for (int j = size >> 1; j > 0; j >>= 1) c = min_max_step(c, j, ((lane & j) == 0) != ((lane & size) == 0));
    return c;
}

// ---- the bound shared by a CTA's warps ----------------------------------------
//
// NW warps of a CTA serve one query.  share[0] is the bound, share[1 + w] the
// smallest (kw + 1)-th key that warp w has published, kw + 1 = ceil(k / NW).
// Two kinds of key bound the CTA's k-th from above: any warp's own k-th key
// (it holds k distinct rows), and, once every warp has published, the largest
// of the published keys (NW ceil(k / NW) >= k distinct rows are at or below
// it).  The second is close to the CTA's true k-th key, as a warp's own k-th
// over an NW-th of the rows is not: a warp then offers about ceil(k / NW)
// rows per e-fold of rows instead of k.  A row above the bound cannot be in the
// CTA's top-k, so the lists still hold every row of it; the rows at the bound
// are in a list already.
template <int NW>
__device__ __forceinline__ void share_publish(uint64_t* share, uint64_t own_kth, uint64_t own_kw, int lane) {
    const int warp = (int)(threadIdx.x >> 5);
    if (lane == 0) {
        volatile uint64_t* mine = reinterpret_cast<volatile uint64_t*>(share + 1 + warp);
        if (own_kw < *mine) *mine = own_kw;
    }
    __syncwarp();
    uint64_t b = lane < NW ? *reinterpret_cast<volatile uint64_t*>(share + 1 + lane) : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const uint64_t y = __shfl_xor_sync(0xFFFFFFFFu, b, o);
        b = y > b ? y : b;
    }
    b = own_kth < b ? own_kth : b;
    if (lane == 0 && b != ~0ull) atomicMin(reinterpret_cast<unsigned long long*>(share), b);
}

// The bound before anything is offered.  Each lane brings the smallest distance
// (as bits) of its rows of the warp's first round; the lanes' minima are 32
// distinct rows, so the sorted minima bound the warp's k-th (k <= 32) and
// (kw + 1)-th key.  All warps of the CTA call it, or prime_none, once per item;
// after the barrier in it the CTA's bound holds over all their first rounds.
// Without it every row of a warp's first rounds went through its list: eight
// sorts of 32 keys per warp and item (with each candidate's row id loaded by
// itself; 512 queries of 40,000 rows, M = 12: 113 us, 90 now; 16 of 100,000
// at k = 100: 46, 35; 1024 of 100,000 at k = 42: 374, 332).  k_scan_list_gen, with 24 warps
// of 64 rows, gained nothing (484 us with and without).  The two-query kernel:
// 512 pairs of 10^6 rows at k = 100 2109 -> 1869 us per batch.
__device__ __forceinline__ void prime_none() { __syncthreads(); }

// the lanes' minima sorted and published; the warp's own k-th key (k <= 32)
template <int NW>
__device__ __forceinline__ uint64_t prime_publish(uint32_t c, int k, int kw, uint64_t* share, int lane) {
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
        for (int j = size >> 1; j > 0; j >>= 1) {
            const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, c, j);
            c = ((lane & j) == 0) == ((lane & size) == 0) ? min(c, y) : max(c, y);
        }
    // the last key of a distance: rows at it are offered
    auto key = [&](int i) { return (uint64_t)__shfl_sync(0xFFFFFFFFu, c, i) << 32 | 0xFFFFFFFFull; };
    const uint64_t own = k <= 32 ? key(k - 1) : ~0ull;
    share_publish<NW>(share, own, key(kw), lane);
    __syncthreads();
    return own;
}

// The same out of line, for the scan by per-lane loads: inlined in its loop it
// left the loads of a round waiting for one another at M = 12 (512 queries of
// 8 x 10^6 rows: k = 50 10333 us, 8923 so; k = 100 13017, 9093).  The other kernels
// measured the same or 1 % slower with it.
template <int NW>
__device__ __noinline__ uint64_t prime_publish_out(uint32_t c, int k, int kw, uint64_t* share, int lane) {
    return prime_publish<NW>(c, k, kw, share, lane);
}

template <int NW, bool OUT = false, class TK>
__device__ __forceinline__ void prime_bound(TK& tk, uint32_t smallest, int lane) {
    if constexpr (OUT)
        tk.primed(prime_publish_out<NW>(smallest, tk.k, tk.kw, tk.share, lane));
    else
        tk.primed(prime_publish<NW>(smallest, tk.k, tk.kw, tk.share, lane));
    tk.refresh(lane);
}

constexpr size_t share_bytes(int warps) { return (size_t)(1 + warps) * 8; }

// before a barrier, by the CTA's first threads
template <int NW>
__device__ __forceinline__ void share_init(uint64_t* share) {
    if (threadIdx.x <= NW) share[threadIdx.x] = ~0ull;
}

// A candidate whose low word is a position of a sorted copy -> its key.  The row
// ids of a scan's candidates are loaded when their list takes them, 32 at a
// time: loaded round by round, half of a warp's rounds waited for one (512 queries of 40,000 rows 157 ->
// 150 us per batch).
__device__ __forceinline__ uint64_t row_key(const uint32_t* rows, uint64_t c) {
    return c == ~0ull ? c : ((c & 0xFFFFFFFF00000000ull) | __ldg(rows + (uint32_t)c));
}

// Merges a warp's candidates [KP, 2KP) of buf into its sorted list [0, KP),
// clears the candidates, publishes (NW > 0) and returns the new k-th key.  The
// candidates are sorted and the KP smallest of both runs kept by one bitonic
// merge (half the compare-exchanges of one sort of 2 KP; 10^8 rows at KP = 128:
// 0.1 % and 1 % bins 1.51 -> 1.41 and 4.33 -> 4.04 ms).  Out of line: the scan
// loops offer keys at many sites and flush rarely, and one copy of the sort
// keeps their code small (instruction-fetch stalls led the two-query kernel's
// profile).
template <int KP, int NW>
__device__ __noinline__ uint64_t flush_list(uint64_t* buf, int k, int kw, uint64_t* share, const uint32_t* rows,
                                            int lane) {
    if (rows != nullptr) {
        __syncwarp();
#pragma unroll
        for (int i = KP + lane; i < 2 * KP; i += 32) buf[i] = row_key(rows, buf[i]);
    }
    warp_sort(buf + KP, KP, lane);
    warp_merge_low(buf, KP, lane);
    const uint64_t thr = buf[k - 1];
    for (int i = KP + lane; i < 2 * KP; i += 32) buf[i] = ~0ull;
    if constexpr (NW > 0) share_publish<NW>(share, thr, buf[kw], lane);
    __syncwarp();
    return thr;
}

// A warp's first 32 candidates: enough for a first published key.
template <int NW>
__device__ __noinline__ void publish_first(const uint64_t* cand, int kw, uint64_t* share, int lane) {
    const uint64_t c = sort32_down(cand[lane], lane);
    share_publish<NW>(share, ~0ull, __shfl_sync(0xFFFFFFFFu, c, 31 - kw), lane);
}

template <int KP, int NW = 0>
struct WarpTopK {
    uint64_t* buf;   // [0, KP): sorted best keys; [KP, 2KP): candidates
    uint64_t* share; // the CTA's shared bound for this query (NW > 0)
    const uint32_t* rows;   // null: candidates are keys; else (distance, position)
    int cnt;
    int k, kw;
    bool first;      // nothing published yet
    uint64_t thr;    // keys below thr are offered: min(own k-th key, shared bound)

    __device__ __forceinline__ void init(uint64_t* b, int k_, int lane, uint64_t* share_ = nullptr,
                                         const uint32_t* rows_ = nullptr) {
        buf = b;
        share = share_;
        rows = rows_;
        k = k_;
        kw = NW > 0 ? (k_ + NW - 1) / (NW > 0 ? NW : 1) - 1 : 0;
        cnt = 0;
        first = NW > 0;
        thr = ~0ull;
        for (int i = lane; i < 2 * KP; i += 32) buf[i] = ~0ull;
        __syncwarp();
    }
    // lower thr to the shared bound: every lane loads the same word in one
    // broadcast (measured faster than a lane-0 load and a shuffle); any value
    // a lane sees is a valid bound, so thr stays correct in every lane
    __device__ __forceinline__ void refresh(int) {
        if (NW == 0) return;
        const uint64_t t = *reinterpret_cast<volatile uint64_t*>(share);
        if (t < thr) thr = t;
    }
    __device__ __forceinline__ void primed(uint64_t own) {
        if (own < thr) thr = own;
        first = false;
    }
    __device__ __forceinline__ void flush(int lane) {
        const uint64_t t = flush_list<KP, NW>(buf, k, kw, share, rows, lane);
        if (t < thr) thr = t;
        cnt = 0;
        first = false;
        refresh(lane);
    }
    __device__ __forceinline__ void offer(uint64_t key, bool want, int lane) {
        const unsigned ball = __ballot_sync(0xFFFFFFFFu, want);
        if (ball == 0) return;
        if (want) buf[KP + cnt + __popc(ball & ((1u << lane) - 1u))] = key;
        cnt += __popc(ball);
        if (NW > 0 && first && cnt >= 32) {
            __syncwarp();
            publish_first<NW>(buf + KP, kw, share, lane);
            first = false;
            refresh(lane);
        }
        if (cnt > KP - 32) {
            __syncwarp();
            flush(lane);
        }
    }
};

// k <= 32: the sorted list is one key per lane, in registers, and up to 63
// candidates wait in shared memory; every 32 of them are sorted and merged
// across the lanes by shuffles (15 + 6 steps of about 25 cycles; the sort of 64
// keys in shared memory took three times as long and ran for every offer).
// Out of line, as flush_list.
// `mine` ascending over the lanes, `c` any: the 32 smallest keys of both, ascending
static __device__ __noinline__ uint64_t absorb32(uint64_t mine, uint64_t c, int lane) {
    c = sort32_down(c, lane);
    mine = c < mine ? c : mine;
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) mine = min_max_step(mine, j, (lane & j) == 0);
    return mine;
}

// k <= 64: the same with two rows of 32 keys, every key of `lo` below those of
// `hi`: the candidates meet `lo` first, what falls out of it meets `hi`.
static __device__ __noinline__ ulonglong2 absorb64(uint64_t lo, uint64_t hi, uint64_t c, int lane) {
    c = sort32_down(c, lane);
    uint64_t out = c < lo ? lo : c;      // the 32 larger keys, bitonic
    lo = c < lo ? c : lo;
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
        lo = min_max_step(lo, j, (lane & j) == 0);
        out = min_max_step(out, j, (lane & j) != 0);   // descending
    }
    hi = out < hi ? out : hi;
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) hi = min_max_step(hi, j, (lane & j) == 0);
    return make_ulonglong2(lo, hi);
}

template <int NW>
struct WarpTopK<64, NW> {
    uint64_t* buf;   // candidates, 64 slots (of 128)
    uint64_t* share;
    const uint32_t* rows;
    int cnt;
    int k, kw;
    uint64_t thr;
    uint64_t lo, hi;   // the lane's keys of the sorted list

    __device__ __forceinline__ void init(uint64_t* b, int k_, int, uint64_t* share_ = nullptr,
                                         const uint32_t* rows_ = nullptr) {
        buf = b;
        share = share_;
        rows = rows_;
        k = k_;
        kw = NW > 0 ? (k_ + NW - 1) / (NW > 0 ? NW : 1) - 1 : 0;
        cnt = 0;
        thr = ~0ull;
        lo = hi = ~0ull;
    }
    __device__ __forceinline__ void refresh(int) {
        if (NW == 0) return;
        const uint64_t t = *reinterpret_cast<volatile uint64_t*>(share);
        if (t < thr) thr = t;
    }
    __device__ __forceinline__ void primed(uint64_t own) {
        if (own < thr) thr = own;
    }
    __device__ __forceinline__ void drain(int n, int lane) {
        cnt -= n;
        __syncwarp();
        uint64_t c = lane < n ? buf[cnt + lane] : ~0ull;
        if (rows != nullptr) c = row_key(rows, c);
        __syncwarp();   // the drained slots take the next candidates
        const ulonglong2 r = absorb64(lo, hi, c, lane);
        lo = r.x;
        hi = r.y;
        const uint64_t t = __shfl_sync(0xFFFFFFFFu, k > 32 ? hi : lo, (k - 1) & 31);
        if (t < thr) thr = t;
        if (NW > 0) share_publish<(NW > 0 ? NW : 1)>(share, thr, __shfl_sync(0xFFFFFFFFu, lo, kw), lane);
        refresh(lane);
    }
    __device__ __forceinline__ void flush(int lane) {
        if (cnt > 0) drain(cnt, lane);
    }
    __device__ __forceinline__ void offer(uint64_t key, bool want, int lane) {
        const unsigned ball = __ballot_sync(0xFFFFFFFFu, want);
        if (ball == 0) return;
        if (want) buf[cnt + __popc(ball & ((1u << lane) - 1u))] = key;
        cnt += __popc(ball);
        if (cnt >= 32) drain(32, lane);
    }
};

template <int NW>
struct WarpTopK<32, NW> {
    uint64_t* buf;   // candidates, 64 slots
    uint64_t* share;
    const uint32_t* rows;
    int cnt;
    int k, kw;
    uint64_t thr;
    uint64_t mine;   // the lane's key of the sorted list

    __device__ __forceinline__ void init(uint64_t* b, int k_, int, uint64_t* share_ = nullptr,
                                         const uint32_t* rows_ = nullptr) {
        buf = b;
        share = share_;
        rows = rows_;
        k = k_;
        kw = NW > 0 ? (k_ + NW - 1) / (NW > 0 ? NW : 1) - 1 : 0;
        cnt = 0;
        thr = ~0ull;
        mine = ~0ull;
    }
    __device__ __forceinline__ void refresh(int) {
        if (NW == 0) return;
        const uint64_t t = *reinterpret_cast<volatile uint64_t*>(share);
        if (t < thr) thr = t;
    }
    __device__ __forceinline__ void primed(uint64_t own) {
        if (own < thr) thr = own;
    }
    __device__ __forceinline__ void drain(int n, int lane) {
        cnt -= n;
        __syncwarp();
        uint64_t c = lane < n ? buf[cnt + lane] : ~0ull;
        if (rows != nullptr) c = row_key(rows, c);
        __syncwarp();   // the drained slots take the next candidates
        mine = absorb32(mine, c, lane);
        const uint64_t t = __shfl_sync(0xFFFFFFFFu, mine, k - 1);
        if (t < thr) thr = t;
        if (NW > 0) share_publish<(NW > 0 ? NW : 1)>(share, thr, __shfl_sync(0xFFFFFFFFu, mine, kw), lane);
        refresh(lane);
    }
    __device__ __forceinline__ void flush(int lane) {
        if (cnt > 0) drain(cnt, lane);
    }
    __device__ __forceinline__ void offer(uint64_t key, bool want, int lane) {
        const unsigned ball = __ballot_sync(0xFFFFFFFFu, want);
        if (ball == 0) return;
        if (want) buf[cnt + __popc(ball & ((1u << lane) - 1u))] = key;
        cnt += __popc(ball);
        if (cnt >= 32) drain(32, lane);
    }
};

// L2 policies: code rows are read by every query of a batch (keep them, so
// the CTAs that walk the same chunk share them); bitmap words are read once.
__device__ __forceinline__ uint64_t policy_evict_last() {
    uint64_t pol;
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

__device__ __forceinline__ uint4 ldg_nc_v4(const uint8_t* p, uint64_t pol) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p), "l"(pol));
    return v;
}

__device__ __forceinline__ uint32_t ldg_nc_u32(const uint32_t* p, uint64_t pol) {
    uint32_t v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.u32 %0, [%1], %2;"
                 : "=r"(v) : "l"(p), "l"(pol));
    return v;
}

template <int IMM>
__device__ __forceinline__ float lds_imm(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(v) : "r"(addr), "n"(IMM));
    return v;
}

// Two packed fp32 additions at once (Blackwell f32x2 pipe).
__device__ __forceinline__ uint64_t add_f32x2(uint64_t acc, float a, float b) {
    uint64_t r;
    asm("{\n\t.reg .b64 t;\n\tmov.b64 t, {%1, %2};\n\tadd.rn.f32x2 %0, %3, t;\n\t}"
        : "=l"(r) : "f"(a), "f"(b), "l"(acc));
    return r;
}

__device__ __forceinline__ void unpack_f32x2(uint64_t v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}

// Shared address at which the dynamic shared memory of a CTA begins on this
// architecture (after the 1 KB the hardware reserves); the kernel checks it.
constexpr uint32_t kDynSmemBase = 0x400u;

// Distances of two rows of MM <= 16 subspaces (codes ca, cb: 16-byte rows,
// table rows of 64 words).  One byte permute forms code * 256 + 4 * w0, w0 =
// the row's index mod 32 (the lane that owns it in the bitmap path); FAST
// (table at kDynSmemBase): the table base and the step go into the load's
// immediate offset; otherwise the base is added.
template <int MM, bool FAST>
__device__ __forceinline__ void lookup2(const uint4 ca, const uint4 cb, uint32_t tba, uint32_t tbb,
                                        uint32_t base, float& da, float& db) {
    static_assert(MM >= 1 && MM <= 16, "16-byte rows");
    const uint32_t wa[4] = {ca.x, ca.y, ca.z, ca.w};
    const uint32_t wb[4] = {cb.x, cb.y, cb.z, cb.w};
    uint64_t acc = 0ull;
#pragma unroll
    for (int s = 0; s < MM; ++s) {
        const uint32_t sel = 0x5504u | ((uint32_t)(s & 3) << 4);
        uint32_t oa = __byte_perm(wa[s >> 2], tba, sel);
        uint32_t ob = __byte_perm(wb[s >> 2], tbb, sel);
        if (!FAST) {
            oa += base;
            ob += base;
        }
        constexpr uint32_t B0 = FAST ? kDynSmemBase : 0u;
        float va, vb;
        switch (s) {
#define IFVS_LDS_CASE(S)                  \
    case S:                               \
        va = lds_imm<B0 + 4 * S>(oa);     \
        vb = lds_imm<B0 + 4 * S>(ob);     \
        break;
            IFVS_LDS_CASE(0) IFVS_LDS_CASE(1) IFVS_LDS_CASE(2) IFVS_LDS_CASE(3)
            IFVS_LDS_CASE(4) IFVS_LDS_CASE(5) IFVS_LDS_CASE(6) IFVS_LDS_CASE(7)
            IFVS_LDS_CASE(8) IFVS_LDS_CASE(9) IFVS_LDS_CASE(10) IFVS_LDS_CASE(11)
            IFVS_LDS_CASE(12) IFVS_LDS_CASE(13) IFVS_LDS_CASE(14) IFVS_LDS_CASE(15)
#undef IFVS_LDS_CASE
            default: va = 0.f; vb = 0.f; break;
        }
        acc = add_f32x2(acc, va, vb);
    }
    unpack_f32x2(acc, da, db);
}

// Distances of NU rows for any M, all owned by one lane (so they share the
// table word offset w0 = the lane): the rows' code words are read together
// and their look-ups go into NU/2 packed f32x2 chains, independent of each
// other; each row's entries are still added one by one for s ascending, from
// subspace w0 mod M on.  Rows whose bit in `valid` is clear read no codes.
template <int NU>
__device__ __forceinline__ void lookup_rows(const uint8_t* __restrict__ codes, const uint32_t (&idx)[NU],
                                            unsigned valid, int row_bytes, int M, int S, const float* tab,
                                            int w0, float (&d)[NU]) {
    static_assert(NU % 2 == 0, "rows in pairs");
    uint64_t acc[NU / 2];
#pragma unroll
    for (int u = 0; u < NU / 2; ++u) acc[u] = 0ull;
    const float* tw = tab + w0;
    for (int w = 0; w * 4 < M; ++w) {
        uint32_t wd[NU];
#pragma unroll
        for (int u = 0; u < NU; ++u)
            wd[u] = (valid >> u & 1u)
                        ? __ldg(reinterpret_cast<const uint32_t*>(codes + (size_t)idx[u] * row_bytes) + w)
                        : 0u;
#pragma unroll
        for (int bb = 0; bb < 4; ++bb) {
            const int s = 4 * w + bb;
            if (s < M) {
#pragma unroll
                for (int u = 0; u < NU; u += 2) {
                    const float va = tw[(int)((wd[u] >> (8 * bb)) & 0xFFu) * S + s];
                    const float vb = tw[(int)((wd[u + 1] >> (8 * bb)) & 0xFFu) * S + s];
                    acc[u / 2] = add_f32x2(acc[u / 2], va, vb);
                }
            }
        }
    }
#pragma unroll
    for (int u = 0; u < NU; u += 2) unpack_f32x2(acc[u / 2], d[u], d[u + 1]);
}

// merge the warps' lists of one query pairwise (both sorted: one bitonic merge
// per level); warp 0 writes k keys
template <int KP, int WARPS, class TK>
__device__ __forceinline__ void merge_warps(TK& tk, uint64_t* tkbuf, int k, int lane, int warp, uint64_t* out) {
    tk.flush(lane);
    if constexpr (KP == 32) {
        __syncwarp();
        tk.buf[lane] = tk.mine;
    } else if constexpr (KP == 64) {
        __syncwarp();
        tk.buf[lane] = tk.lo;
        tk.buf[32 + lane] = tk.hi;
    }
#pragma unroll 1
    for (int step = 1; step < WARPS; step <<= 1) {
        __syncthreads();
        if ((warp & (2 * step - 1)) == 0 && warp + step < WARPS) {
            const uint64_t* other = tkbuf + (warp + step) * 2 * KP;
            if constexpr (KP == 32) {
                const uint64_t o = other[31 - lane];
                uint64_t m = o < tk.mine ? o : tk.mine;
#pragma unroll
                for (int j = 16; j > 0; j >>= 1) m = min_max_step(m, j, (lane & j) == 0);
                tk.mine = m;
                tk.buf[lane] = m;
            } else {
                for (int i = lane; i < KP; i += 32) tk.buf[KP + i] = other[i];
                warp_merge_low(tk.buf, KP, lane);
            }
        }
    }
    if (warp == 0 && out != nullptr) {
        if constexpr (KP == 32) {
            if (lane < k) out[lane] = tk.mine;
        } else {
            for (int i = lane; i < k; i += 32) out[i] = tk.buf[i];
        }
    }
}

// ---- bulk copies into shared memory (cp.async.bulk) and their mbarriers ----
//
// The untiled form of TMA: one instruction copies a contiguous, 16-byte
// aligned run of global memory into shared memory and reports its bytes to
// an mbarrier (complete_tx); threads wait on the barrier's phase parity.
// Every wait is bounded (kWaitCycles SM cycles, about half a second at
// 2 GHz): a wait that runs out returns false and the kernel reports it.

constexpr long long kWaitCycles = 1ll << 30;

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

// makes barrier initialisations visible to the bulk-copy (async) proxy
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// orders this thread's earlier shared-memory accesses before later
// bulk-copy writes to the same bytes
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// one arrival that also announces `bytes` of bulk-copy traffic
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// global -> shared copy of `bytes` (a multiple of 16, both addresses 16-byte
// aligned), completion counted on `bar`, with an L2 cache policy
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar,
                                         uint64_t pol) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], "
        "%4;" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar), "l"(pol)
        : "memory");
}

// a thread whose phase has not completed may sleep in the instruction for
// up to kSuspendNs (it wakes when the phase completes) instead of spinning;
// 0: no hint (the hardware's own time limit)
#ifndef IFVS_SUSPEND_NS
#define IFVS_SUSPEND_NS 20000
#endif
constexpr uint32_t kSuspendNs = IFVS_SUSPEND_NS;

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    if constexpr (kSuspendNs > 0) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, "
            "p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity), "n"(kSuspendNs)
            : "memory");
    } else {
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
    }
    return ok != 0u;
}

// Waits, with every lane of the warp, until the barrier's phase of parity
// `parity` has completed; false (for the whole warp) when kWaitCycles pass
// first.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity) {
    const long long t0 = clock64();
    for (;;) {
        const bool ok = mbar_try_wait(bar, parity);
        if (__all_sync(0xFFFFFFFFu, ok)) return true;
        if (__any_sync(0xFFFFFFFFu, clock64() - t0 > kWaitCycles)) return false;
    }
}

// largest dynamic shared memory per CTA the current device allows (opt-in)
inline int max_smem_optin() {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return 0;
    return v;
}

// Subspace count the fixed-M scan loops are compiled for when the index
// stores 16-byte rows with 64-word tables (M = 12 rows padded to 16 bytes,
// or M = 16); 0: the generic-M loop.
inline int fixed_m(const ScanShape& sh) {
    if (sh.row_bytes != 16 || sh.tab_words != 64) return 0;
    return (sh.M == 16 || sh.M == 12) ? sh.M : 0;
}

// A scan kernel's CTA takes items from its group's list until it is empty: the
// first by its block index, the others from the work counter (after another
// group's items, the first one too).  `slot`: a word
// of the CTA's dynamic shared memory (static shared memory would move the
// dynamic window off the base that the look-ups' immediate offsets assume).
struct ItemLoop {
    const ScanItem* items;
    int n;
    int* counter;
    volatile int* slot;
    int own;   // items given out by block index
    int at;
    __device__ __forceinline__ ItemLoop(const ScanSched& s, int group, void* slot_, bool later = false)
        : items(s.items[group]), n(s.ctl[group]), counter(s.ctl + kGroups + group),
          slot(reinterpret_cast<volatile int*>(slot_)), own(later ? 0 : (int)gridDim.x), at((int)blockIdx.x) {
        if (later && n > 0) next();
    }
    __device__ __forceinline__ bool more() const { return at < n; }
    // all threads; a barrier on both sides: shared memory may be reused after it
    __device__ __forceinline__ void next() {
        if (threadIdx.x == 0) *slot = own + atomicAdd(counter, 1);
        __syncthreads();
        at = *slot;
        __syncthreads();
    }
};

// A batch's scans share no data and overlap: the first waits for the tables and
// lets the next start, which fills the SMs that the first leaves at its end;
// the others wait for the one before them at their end.
//
// The others read the work lists, the plan and the tables without a wait of their
// own, which PTX does not promise to be enough: it speaks of what a grid sees
// after its own griddepcontrol.wait.  They rely on the grids that wrote these
// having completed, and their writes being in memory, before the first scan's
// wait returned, and on the first scan letting them start only after that; no
// CTA of theirs has read those addresses earlier.  A wait of their own would hold
// them until the first scan has ended, which is what the overlap avoids.
__device__ __forceinline__ void scan_begin(bool first) {
    if (first) wait_before();
    start_dependents();
}
__device__ __forceinline__ void scan_end(bool first) {
    if (!first) wait_before();
}

// CTAs to launch for a group: all that fit the device, or the items there can be
inline unsigned item_grid(const SchedGroup& g) { return (unsigned)(g.cap < g.slots ? (g.cap < 1 ? 1 : g.cap) : g.slots); }

}  // namespace ifvs
