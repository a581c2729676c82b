// Rank (§2 stage 2) over a one-column predicate's pool read as a position
// range of that column's sorted copy of the codes: the one-query kernel
// k_scan_list and its forms on bulk-copied tiles.  Design notes in
// scan_common.cuh.
#include "scan_common.cuh"

namespace ifvs {

// ---- sorted-copy scan ---------------------------------------------------
//
// For a query of the list path (ScanPlan) the pool is the position range
// [a, b) of one column's sorted copy of the codes, whose position p holds
// row rows[p]'s codes rotated by (p mod 32) mod M.  An item is a run of
// 256-position rounds of that range, walked exactly as the bitmap path walks
// dense blocks: lane l takes the positions = l (mod 32), so its look-ups hit
// banks (l + s) mod 32 and the code loads are coalesced; rounds cut by a or b
// mask their positions.  No bitmap, no per-row bit handling.  The row id, needed for
// the key, is loaded only for positions whose distance can enter the top-k.
// The sum order (the subspaces from (p mod 32) mod M on) differs from the
// bitmap path's, so the two agree to float32 rounding.

size_t scan_list_smem_bytes(int tab_words, int kp) {
    return (size_t)256 * tab_words * 4 + (size_t)kScanWarps * 2 * kp * 8 + share_bytes(kScanWarps) + 24;
}

// the smallest distance (as bits) of the rows with a bit in `valid`
template <int NU>
__device__ __forceinline__ uint32_t smallest(const float (&d)[NU], unsigned valid) {
    uint32_t m = 0xFFFFFFFFu;
#pragma unroll
    for (int u = 0; u < NU; ++u) m = (valid >> u & 1u) ? min(m, __float_as_uint(d[u])) : m;
    return m;
}

// The candidates of a round (bits of `cand`: distance at most the bound's).  Their
// row ids are looked up when the list takes them (row_key), except where the
// distance equals the bound's: there the id decides now, so that rows of equal
// distance do not all go through the list.
template <class TK>
__device__ __forceinline__ void offer_round(TK& tk, const float (&d)[kU], const uint32_t (&pos)[kU], unsigned cand,
                                            uint32_t thr_hi, const uint32_t* __restrict__ rows, int lane) {
    unsigned tie = 0u;
#pragma unroll
    for (int u = 0; u < kU; ++u) tie |= (unsigned)(__float_as_uint(d[u]) == thr_hi) << u;
    tie &= cand;
    if (__any_sync(0xFFFFFFFFu, tie != 0u)) {
        const uint32_t thr_lo = (uint32_t)tk.thr;
#pragma unroll
        for (int u = 0; u < kU; ++u)
            if ((tie >> u & 1u) && __ldg(rows + pos[u]) >= thr_lo) cand &= ~(1u << u);
    }
#pragma unroll
    for (int u = 0; u < kU; ++u)
        tk.offer(((uint64_t)__float_as_uint(d[u]) << 32) | pos[u],
                 (cand >> u & 1u) && __float_as_uint(d[u]) <= (uint32_t)(tk.thr >> 32), lane);
}

template <int KP, int MM, bool FAST, class TK>
__device__ __forceinline__ void scan_positions(const uint8_t* __restrict__ codes, const uint32_t* __restrict__ rows,
                                               int64_t a, int64_t b, uint32_t r0, uint32_t r1, uint32_t base,
                                               TK& tk, int lane, int warp) {
    const uint32_t tb = 4u * (uint32_t)lane;
    const uint64_t keep = policy_evict_last();
    // positions fit in 32 bits: N < 2^32 - 2048
    const uint32_t a32 = (uint32_t)a, b32 = (uint32_t)b;
    const uint32_t first = r0 + (uint32_t)warp;
    if (first >= r1) prime_none();
#pragma unroll 1
    for (uint32_t r = first; r < r1; r += kScanWarps) {
        const uint32_t P = r * kRoundRows;
        const bool full = P >= a32 && P + kRoundRows <= b32;
        tk.refresh(lane);
        uint32_t pos[kU];
        unsigned valid = 0u;
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            pos[u] = P + 32u * (uint32_t)u + (uint32_t)lane;
            valid |= (unsigned)(full || (pos[u] >= a32 && pos[u] < b32)) << u;
        }
        float d[kU];
        uint4 c[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u)
            c[u] = (valid >> u & 1u) ? ldg_nc_v4(codes + (size_t)pos[u] * 16, keep) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < kU; u += 2) lookup2<MM, FAST>(c[u], c[u + 1], tb, tb, base, d[u], d[u + 1]);
        if (r == first) prime_bound<kScanWarps, true>(tk, smallest(d, valid), lane);
        // a position can enter the top-k only if its distance is at most the
        // current k-th one; only those load their row id
        const uint32_t thr_hi = (uint32_t)(tk.thr >> 32);
        unsigned cand = 0u;
#pragma unroll
        for (int u = 0; u < kU; ++u) cand |= (unsigned)(__float_as_uint(d[u]) <= thr_hi) << u;
        cand &= valid;
        if (!__any_sync(0xFFFFFFFFu, cand != 0u)) continue;
        offer_round(tk, d, pos, cand, thr_hi, rows, lane);
    }
}

template <int KP, int MM, int MINB>
__global__ void __launch_bounds__(kScanThreads, MINB)
k_scan_list(const float* __restrict__ tables, SortedCols sc, const ScanPlan* __restrict__ plan, int k,
            ScanSched sched, bool first) {
    extern __shared__ __align__(256) uint8_t smem[];
    constexpr int S = 64;
    float* tab = reinterpret_cast<float*>(smem);
    uint64_t* tkbuf = reinterpret_cast<uint64_t*>(smem + (size_t)256 * S * 4);
    uint64_t* share = tkbuf + kScanWarps * 2 * KP;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(tab);
    scan_begin(first);
    for (ItemLoop loop(sched, 0, share + 1 + kScanWarps); loop.more(); loop.next()) {
        const ScanItem item = loop.items[loop.at];
        const ScanPlan p = plan[item.qa];
        {
            const float4* src = reinterpret_cast<const float4*>(tables + item.qa * (int64_t)256 * S);
            float4* dst = reinterpret_cast<float4*>(tab);
            for (int i = threadIdx.x; i < 64 * S; i += kScanThreads) dst[i] = __ldg(src + i);
        }
        share_init<kScanWarps>(share);
        WarpTopK<KP, kScanWarps> tk;
        tk.init(tkbuf + warp * 2 * KP, k, lane, share, sc.rows_of(p.col));
        __syncthreads();
        const uint8_t* codes = sc.codes_of(p.col);
        const uint32_t* rows = sc.rows_of(p.col);
        if (base == kDynSmemBase)
            scan_positions<KP, MM, true>(codes, rows, p.a, p.b, item.a, item.b, base, tk, lane, warp);
        else
            scan_positions<KP, MM, false>(codes, rows, p.a, p.b, item.a, item.b, base, tk, lane, warp);
        merge_warps<KP, kScanWarps>(tk, tkbuf, k, lane, warp, sched.partials + (int64_t)item.la * k);
    }
    scan_end(first);
}

// ---- sorted-copy scan with bulk-copied code tiles (M = 12, 16) --------------
//
// The walk of k_scan_list with the code rows of every round brought into
// shared memory by the bulk-copy engine (cp.async.bulk, the untiled form of
// TMA) instead of per-lane vector loads.  A warp's round is 256 consecutive
// positions (lane l takes positions 32u + l, u < kU = 8): 4 KB of codes, one
// copy.  Each warp owns one such tile with an mbarrier; lane 0 issues the copy
// of its next round as soon as this round's rows sit in registers, so a warp
// keeps a round of codes in flight while it computes, in shared memory rather
// than in registers.  A warp whose tile
// has not arrived within the bounded wait sets bit 4 of *err (the search
// returns IFVS_ERR_TIMEOUT), waits (bounded again) for its copies still in
// flight, and stops scanning; its CTA still merges and writes its lists.
// tx_extra (0 in normal use) is added to the bytes each barrier expects; a
// positive value makes every wait run out, which exercises that path.
// One tile per warp keeps two 8-warp CTAs per SM; measured on the
// 10^8-row workload it beat vector loads by 3 % (0.1 % pools) and 7 % (1 %),
// while two or four tiles per warp (one CTA per SM) lost 38 % and 36 %.

constexpr uint32_t kTileBytes = 32u * kU * 16u;    // one warp round: 256 positions x 16 bytes
static_assert(32 % kU == 0, "whole rounds per block");
static_assert(32 * kU == kRoundRows, "a warp's round is the unit of the work lists");

__host__ __device__ constexpr size_t bulk_ring_offset(int kp) {
    return ((size_t)256 * 64 * 4 + (size_t)kScanWarps * 2 * kp * 8 + (1 + kScanWarps) * 8 + 127) / 128 * 128;
}

// tiles, one barrier per tile, and the barrier of the table copy
size_t scan_bulk_smem_bytes(int kp) {
    return bulk_ring_offset(kp) + (size_t)kScanWarps * (kTileBytes + 8) + 32;
}

// `phase`: the tile barrier's parity before this item, updated; false when a
// wait ran out (the barrier must not be used again)
template <int KP, int MM, bool FAST, class TK>
__device__ __forceinline__ bool scan_positions_bulk(const uint8_t* __restrict__ codes,
                                                    const uint32_t* __restrict__ rows, int64_t a, int64_t b,
                                                    uint32_t r0, uint32_t r1, const float* tab, uint8_t* tile_mem,
                                                    uint32_t bar_s, uint32_t& phase, uint32_t tx_extra, int* err,
                                                    TK& tk, int lane, int warp) {
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(tab);
    const uint32_t tb = 4u * (uint32_t)lane;
    const uint64_t keep = policy_evict_last();
    const uint32_t a32 = (uint32_t)a, b32 = (uint32_t)b;   // positions fit in 32 bits
    const uint32_t tile_s = (uint32_t)__cvta_generic_to_shared(tile_mem);
    auto issue = [&](uint32_t r) {
        mbar_arrive_expect_tx(bar_s, kTileBytes + tx_extra);
        bulk_g2s(tile_s, codes + (size_t)r * kTileBytes, kTileBytes, bar_s, keep);
    };
    const uint32_t first = r0 + (uint32_t)warp;
    if (lane == 0 && first < r1) {
        fence_proxy_async_smem();   // the tile's readers of the previous item are past a barrier
        issue(first);
    }
    if (first >= r1) prime_none();
#pragma unroll 1
    for (uint32_t r = first; r < r1; r += kScanWarps) {
        if (!mbar_wait_warp(bar_s, phase)) {
            if (lane == 0) atomicOr(err, 4);
            mbar_wait_warp(bar_s, phase);   // this round's copy may still be in flight
            if (r == first) prime_none();
            return false;
        }
        phase ^= 1u;
        tk.refresh(lane);
        const uint32_t P = r * kRoundRows;
        const uint4* tile = reinterpret_cast<const uint4*>(tile_mem);
        uint4 c[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) c[u] = tile[32 * u + lane];
        __syncwarp();
        if (lane == 0 && r + kScanWarps < r1) {
            fence_proxy_async_smem();
            issue(r + kScanWarps);
        }
        const bool full = P >= a32 && P + 32u * kU <= b32;
        uint32_t pos[kU];
        unsigned valid = 0u;
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            pos[u] = P + 32u * (uint32_t)u + (uint32_t)lane;
            valid |= (unsigned)(full || (pos[u] >= a32 && pos[u] < b32)) << u;
        }
        float d[kU];
#pragma unroll
        for (int u = 0; u < kU; u += 2) lookup2<MM, FAST>(c[u], c[u + 1], tb, tb, base, d[u], d[u + 1]);
        if (r == first) prime_bound<kScanWarps>(tk, smallest(d, valid), lane);
        // as in scan_positions: only candidates load their row id
        const uint32_t thr_hi = (uint32_t)(tk.thr >> 32);
        unsigned cand = 0u;
#pragma unroll
        for (int u = 0; u < kU; ++u) cand |= (unsigned)(__float_as_uint(d[u]) <= thr_hi) << u;
        cand &= valid;
        if (!__any_sync(0xFFFFFFFFu, cand != 0u)) continue;
        offer_round(tk, d, pos, cand, thr_hi, rows, lane);
    }
    return true;
}

template <int KP, int MM, int MINB>
__global__ void __launch_bounds__(kScanThreads, MINB)
k_scan_list_bulk(const float* __restrict__ tables, SortedCols sc, const ScanPlan* __restrict__ plan, int k,
                 ScanSched sched, uint32_t tx_extra, int* __restrict__ err, bool first) {
    extern __shared__ __align__(256) uint8_t smem[];
    float* tab = reinterpret_cast<float*>(smem);
    uint64_t* tkbuf = reinterpret_cast<uint64_t*>(smem + (size_t)256 * 64 * 4);
    uint8_t* ring_all = smem + bulk_ring_offset(KP);
    uint64_t* bars_all = reinterpret_cast<uint64_t*>(ring_all + (size_t)kScanWarps * kTileBytes);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint8_t* tile = ring_all + (size_t)warp * kTileBytes;
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(bars_all + warp);
    const uint32_t tbar = (uint32_t)__cvta_generic_to_shared(bars_all + kScanWarps);
    if (lane == 0) {
        mbar_init(bar, 1u);
        if (threadIdx.x == 0) mbar_init(tbar, 1u);
        fence_mbar_init();
    }
    uint64_t* share = tkbuf + kScanWarps * 2 * KP;
    uint32_t phase = 0u, tphase = 0u;
    scan_begin(first);
    for (ItemLoop loop(sched, 0, bars_all + kScanWarps + 1); loop.more(); loop.next()) {
        const ScanItem item = loop.items[loop.at];
        // the query's 64 KB table (rows replicated and rotated, as k_tables
        // describes) in one bulk copy, while the lists are set up
        if (threadIdx.x == 0) {
            fence_proxy_async_smem();   // the last item's readers are past a barrier
            mbar_arrive_expect_tx(tbar, 256u * 64u * 4u);
            bulk_g2s((uint32_t)__cvta_generic_to_shared(tab), tables + item.qa * (int64_t)256 * 64, 256u * 64u * 4u,
                     tbar, policy_evict_first());
        }
        share_init<kScanWarps>(share);
        const ScanPlan p = plan[item.qa];
        WarpTopK<KP, kScanWarps> tk;
        tk.init(tkbuf + warp * 2 * KP, k, lane, share, sc.rows_of(p.col));
        __syncthreads();
        bool ok = mbar_wait_warp(tbar, tphase);
        if (!ok) {
            if (lane == 0) atomicOr(err, 4);
            mbar_wait_warp(tbar, tphase);   // the copy may still be in flight
        }
        tphase ^= 1u;
        if (ok) {
            const uint8_t* codes = sc.codes_of(p.col);
            const uint32_t* rows = sc.rows_of(p.col);
            if ((uint32_t)__cvta_generic_to_shared(tab) == kDynSmemBase)
                ok = scan_positions_bulk<KP, MM, true>(codes, rows, p.a, p.b, item.a, item.b, tab, tile, bar, phase,
                                                       tx_extra, err, tk, lane, warp);
            else
                ok = scan_positions_bulk<KP, MM, false>(codes, rows, p.a, p.b, item.a, item.b, tab, tile, bar, phase,
                                                        tx_extra, err, tk, lane, warp);
        } else {
            prime_none();
        }
        merge_warps<KP, kScanWarps>(tk, tkbuf, k, lane, warp, sched.partials + (int64_t)item.la * k);
        if (__syncthreads_or(ok ? 0 : 1)) break;   // the search reports a timeout; its lists are incomplete
    }
    scan_end(first);
}

// ---- generic M ----------------------------------------------------------------
//
// For M other than 12 and 16 a sorted copy is stored by groups of 32 positions,
// word by word ([group][word][lane], k_relayout_sorted): a warp reads word
// w of its 32 rows as one 128-byte line, with no shared-memory tile between
// (rows of 120 bytes one after the other cost an L1 wavefront per row and word,
// or a bulk-copied tile per warp whose row reads met two-way bank conflicts and
// whose space left eight warps per SM).  Without tiles the table (160 KB at
// M = 120) leaves room for 24 warps; lane l owns two positions, 32 apart, whose
// entries are added as packed pairs for s ascending, as in lookup_rows.  The
// next four words of both are loaded while the 32 entries of these are looked
// up.  Bound: the shared-memory look-ups, one wavefront per 32.
// 256 queries on 5 x 10^5 rows at M = 120, pools of 10 %: 866 us with tiles, 370 us
// here.
size_t scan_gen_smem_bytes(int tab_words, int kp, int warps) {
    return (size_t)256 * tab_words * 4 + (size_t)warps * 2 * kp * 8 + share_bytes(warps) + 24;
}

constexpr int kGenWords = 4;   // words per block: 16 codes of each row

// entry at byte `addr` + 4 s of the shared table, s in the load's immediate
__device__ __forceinline__ float lds_step(uint32_t addr, int s) {
    switch (s) {
#define IFVS_LDS_CASE(S) \
    case S: return lds_imm<4 * S>(addr);
        IFVS_LDS_CASE(0) IFVS_LDS_CASE(1) IFVS_LDS_CASE(2) IFVS_LDS_CASE(3)
        IFVS_LDS_CASE(4) IFVS_LDS_CASE(5) IFVS_LDS_CASE(6) IFVS_LDS_CASE(7)
        IFVS_LDS_CASE(8) IFVS_LDS_CASE(9) IFVS_LDS_CASE(10) IFVS_LDS_CASE(11)
        IFVS_LDS_CASE(12) IFVS_LDS_CASE(13) IFVS_LDS_CASE(14) IFVS_LDS_CASE(15)
#undef IFVS_LDS_CASE
        default: return 0.f;
    }
}

// The look-ups of a block's codes of two rows.  `at`: shared address of word
// (lane + the block's first code index) of codeword 0's row; codeword rows S4
// bytes apart: one byte extraction and one multiply-add per address.  Codes
// from `left` on are the row's padding.
template <bool CHECK>
__device__ __forceinline__ uint64_t gen_block(const uint32_t (&wa)[kGenWords], const uint32_t (&wb)[kGenWords],
                                              uint32_t at, uint32_t S4, int left, uint64_t acc) {
#pragma unroll
    for (int s = 0; s < 4 * kGenWords; ++s) {
        if (CHECK && s >= left) break;
        const uint32_t sel = 0x4440u | (uint32_t)(s & 3);
        const float va = lds_step(__byte_perm(wa[s >> 2], 0u, sel) * S4 + at, s);
        const float vb = lds_step(__byte_perm(wb[s >> 2], 0u, sel) * S4 + at, s);
        acc = add_f32x2(acc, va, vb);
    }
    return acc;
}

template <int KP, int WARPS, class TK>
__device__ __forceinline__ void scan_positions_gen(const uint32_t* __restrict__ codes,
                                                   const uint32_t* __restrict__ rows, int64_t a, int64_t b,
                                                   uint32_t r0, uint32_t r1, const ScanShape& sh, uint32_t base,
                                                   TK& tk, int lane, int warp) {
    const int M = sh.M, nw = sh.row_bytes / 4, nblk = (nw + kGenWords - 1) / kGenWords;
    const uint32_t S4 = 4u * (uint32_t)sh.tab_words, a32 = (uint32_t)a, b32 = (uint32_t)b;
    const uint64_t keep = policy_evict_last();
    constexpr uint32_t kPer = kRoundRows / 64;  // pairs of groups per round
    const uint32_t last = r1 * kPer;
    // words [first, first + kGenWords) of the two rows, `row` words apart
    auto load = [&](const uint32_t* p, int left, uint32_t (&wa)[kGenWords], uint32_t (&wb)[kGenWords]) {
#pragma unroll
        for (int i = 0; i < kGenWords; ++i) {
            wa[i] = i < left ? ldg_nc_u32(p + 32 * i, keep) : 0u;
            wb[i] = i < left ? ldg_nc_u32(p + 32 * (nw + i), keep) : 0u;
        }
    };
    uint32_t g = r0 * kPer + (uint32_t)warp;
    const uint32_t* p = codes + (size_t)g * 2 * nw * 32 + lane;    // the block to load next
    const size_t step = (size_t)(WARPS * 2 * nw) * 32 - (size_t)(nblk - 1) * kGenWords * 32;
    uint32_t wa[kGenWords], wb[kGenWords];
    const uint32_t first = g;
    if (g < last)
        load(p, nw, wa, wb);
#pragma unroll 1
    for (; g < last; g += WARPS) {
        tk.refresh(lane);
        uint64_t acc = 0ull;
        uint32_t at = base + 4u * (uint32_t)lane;
#pragma unroll 1
        for (int blk = 0; blk < nblk; ++blk, at += 16u * kGenWords) {
            uint32_t na[kGenWords], nb[kGenWords];
            const bool end = blk + 1 == nblk;
            p += end ? step : kGenWords * 32;
            if (!end || g + WARPS < last) load(p, end ? nw : nw - (blk + 1) * kGenWords, na, nb);
            const int left = M - blk * 4 * kGenWords;
            if (left >= 4 * kGenWords)
                acc = gen_block<false>(wa, wb, at, S4, left, acc);
            else
                acc = gen_block<true>(wa, wb, at, S4, left, acc);
#pragma unroll
            for (int i = 0; i < kGenWords; ++i) {
                wa[i] = na[i];
                wb[i] = nb[i];
            }
        }
        float d[2];
        unpack_f32x2(acc, d[0], d[1]);
        const uint32_t pos = 64u * g + (uint32_t)lane;
        unsigned valid = 0u;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const uint32_t p = pos + 32u * (uint32_t)u;
            valid |= (unsigned)(p >= a32 && p < b32) << u;
        }
        const uint32_t thr_hi = (uint32_t)(tk.thr >> 32);
        bool cand[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) cand[u] = (valid >> u & 1u) && __float_as_uint(d[u]) <= thr_hi;
        if (!__any_sync(0xFFFFFFFFu, cand[0] || cand[1])) continue;
        uint32_t id[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) id[u] = cand[u] ? __ldg(rows + pos + 32u * (uint32_t)u) : 0u;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const uint64_t key = ((uint64_t)__float_as_uint(d[u]) << 32) | id[u];
            tk.offer(key, cand[u] && key < tk.thr, lane);
        }
    }
}

template <int KP, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, WARPS > 12 ? 1 : 2)
k_scan_list_gen(const float* __restrict__ tables, SortedCols sc, const ScanPlan* __restrict__ plan, int k,
                ScanShape sh, ScanSched sched, bool first) {
    extern __shared__ __align__(256) uint8_t smem[];
    const int S = sh.tab_words;
    float* tab = reinterpret_cast<float*>(smem);
    uint64_t* tkbuf = reinterpret_cast<uint64_t*>(smem + (size_t)256 * S * 4);
    uint64_t* share = tkbuf + WARPS * 2 * KP;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(tab);
    scan_begin(first);
    for (ItemLoop loop(sched, 0, share + 1 + WARPS); loop.more(); loop.next()) {
        const ScanItem item = loop.items[loop.at];
        const ScanPlan p = plan[item.qa];
        {
            const float4* src = reinterpret_cast<const float4*>(tables + item.qa * (int64_t)256 * S);
            float4* dst = reinterpret_cast<float4*>(tab);
#pragma unroll 4
            for (int i = threadIdx.x; i < 64 * S; i += WARPS * 32) dst[i] = __ldg(src + i);
        }
        share_init<WARPS>(share);
        WarpTopK<KP, WARPS> tk;
        tk.init(tkbuf + warp * 2 * KP, k, lane, share);
        __syncthreads();
        scan_positions_gen<KP, WARPS>(reinterpret_cast<const uint32_t*>(sc.codes_of(p.col)), sc.rows_of(p.col), p.a,
                                      p.b, item.a, item.b, sh, base, tk, lane, warp);
        merge_warps<KP, WARPS>(tk, tkbuf, k, lane, warp, sched.partials + (int64_t)item.la * k);
    }
    scan_end(first);
}

template <class Kernel, class... Args>
static cudaError_t launch_items(Kernel kern, const ScanSched& sched, int threads, size_t smem, ScanOrder o,
                                cudaStream_t s, Args... args) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_kernel(kern, dim3(item_grid(sched.group[0])), dim3((unsigned)threads), smem, o.chain, s, args...,
                         o.first);
}

// The kernel for a shape.  M = 12 and 16: bulk copies where asked for, else
// per-lane loads, 8 warps and one or two CTAs per SM.  Other M: 24 warps per SM
// at 80 registers, in one CTA where the SM holds one table and in two of 12
// where it holds two; fewer where the lists do not fit.
struct ListKernel {
    enum { kBulk, kPlain, kGen } kind;
    int warps;
    size_t smem;
    int ctas;      // per SM
};
static ListKernel list_kernel(const ScanShape& sh, int kp, bool bulk) {
    const int mm = fixed_m(sh);
    const size_t most = (size_t)max_smem_optin(), sm = 233472;
    ListKernel lk;
    lk.warps = kScanWarps;
    if (mm > 0) {
        lk.kind = bulk && scan_bulk_smem_bytes(kp) <= most ? ListKernel::kBulk : ListKernel::kPlain;
        lk.smem = lk.kind == ListKernel::kBulk ? scan_bulk_smem_bytes(kp) : scan_list_smem_bytes(sh.tab_words, kp);
    } else {
        lk.kind = ListKernel::kGen;
        const bool two = sm / (scan_gen_smem_bytes(sh.tab_words, kp, 8) + 1024) >= 2;
        lk.warps = 24;
        if (two || scan_gen_smem_bytes(sh.tab_words, kp, 24) > most) {
            const size_t need = scan_gen_smem_bytes(sh.tab_words, kp, 12);
            lk.warps = (two ? sm / (need + 1024) >= 2 : need <= most) ? 12 : 8;
        }
        lk.smem = scan_gen_smem_bytes(sh.tab_words, kp, lk.warps);
    }
    const int by_smem = (int)(sm / (lk.smem + 1024));
    lk.ctas = by_smem >= 2 && lk.warps <= 12 ? 2 : 1;
    return lk;
}

int scan_list_ctas_per_sm(const ScanShape& sh, int k, bool bulk) { return list_kernel(sh, scan_kp(k), bulk).ctas; }

template <int KP>
static cudaError_t launch_list_kp(const float* tab, SortedCols sc, const ScanPlan* plan, int k, const ScanShape& sh,
                                  const ScanSched& sched, const ListOpts& lo, ScanOrder o,
                                  cudaStream_t s) {
    const int mm = fixed_m(sh);
    const ListKernel lk = list_kernel(sh, KP, lo.bulk);
    const bool two = lk.ctas == 2;
    const int threads = lk.warps * 32;
    if (lk.kind == ListKernel::kBulk) {
        auto kern = mm == 16 ? (two ? k_scan_list_bulk<KP, 16, 2> : k_scan_list_bulk<KP, 16, 1>)
                             : (two ? k_scan_list_bulk<KP, 12, 2> : k_scan_list_bulk<KP, 12, 1>);
        return launch_items(kern, sched, threads, lk.smem, o, s, tab, sc, plan, k, sched, lo.tx_extra, lo.err);
    }
    if (lk.kind == ListKernel::kPlain) {
        auto kern = mm == 16 ? (two ? k_scan_list<KP, 16, 2> : k_scan_list<KP, 16, 1>)
                             : (two ? k_scan_list<KP, 12, 2> : k_scan_list<KP, 12, 1>);
        return launch_items(kern, sched, threads, lk.smem, o, s, tab, sc, plan, k, sched);
    }
    auto kern = lk.warps == 24   ? k_scan_list_gen<KP, 24>
                : lk.warps == 12 ? k_scan_list_gen<KP, 12>
                                 : k_scan_list_gen<KP, 8>;
    return launch_items(kern, sched, threads, lk.smem, o, s, tab, sc, plan, k, sh, sched);
}

cudaError_t launch_scan_list(const float* tab, SortedCols sc, const ScanPlan* plan, int64_t nq, int k,
                             const ScanShape& sh, const ScanSched& sched, const ListOpts& lo, ScanOrder o,
                                  cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    switch (scan_kp(k)) {
        case 32: return launch_list_kp<32>(tab, sc, plan, k, sh, sched, lo, o, s);
        case 64: return launch_list_kp<64>(tab, sc, plan, k, sh, sched, lo, o, s);
        case 128: return launch_list_kp<128>(tab, sc, plan, k, sh, sched, lo, o, s);
        default: return launch_list_kp<256>(tab, sc, plan, k, sh, sched, lo, o, s);
    }
}
}  // namespace ifvs
