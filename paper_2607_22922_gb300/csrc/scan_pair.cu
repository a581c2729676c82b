// Rank (§2 stage 2) for two queries per CTA (M = 12 and 16), on the sorted copy
// of the codes or, for bitmap queries, on the index layout: the two-query
// kernel k_scan_list_pair.  Design notes in scan_common.cuh.
#include <algorithm>

#include "scan_common.cuh"

namespace ifvs {

// When k_schedule pairs two queries on the sorted copy of the same
// column, one CTA serves both, and one shared-memory load serves
// both queries' look-ups.  A 64 KB table with the rows, replication and rotation
// of the float32 one holds, in word w of codeword row c, the pair
// qA[w mod M][c] | qB[w mod M][c] << 16 of quantised entries,
// q[m][c] = floor((LUT[m][c] - lo_m) * inv), lo_m the smallest entry of
// subspace m, inv = Q / (the widest subspace's range), Q = floor(32767 / M).
// M entries sum to less than 2^15, so one integer add accumulates both queries with no
// carry between the halves (and bit 15 of each half stays free for the
// candidate test, pack_bounds), and a row's sum S bounds its float32 distance
// from below (quant_bound).  A row whose S exceeds the bound of its query's
// current k-th key cannot enter that top-k and is dropped; every other row
// gets its exact float32 distance from the query's unreplicated table,
// added in the order of the one-query loop (subspace (p mod 32) mod 16
// first), so the top-k receives the keys the one-query loop would give it.
// Since the dropped rows are decided by integers, the shared-memory traffic
// of the dense loop is half that of two float32 tables.  Blocks that meet
// one query's range only run the same loop with the other query masked.
// 16 warps, one CTA per SM.
//
// Two bitmap queries run the same rounds over all rows of the index, with
// their pass bits as masks: neighbouring rows are read together and every
// look-up serves both, where one query's loop (k_scan) visits its own passing
// rows only, each lane a row in a line of its own (256 queries that 40 % of
// 4 x 10^6 rows of 12 codes pass: 2270 us single, 1090 us paired; the look-ups
// alone take 0.61 ms at one per bank and clock).
constexpr int kPairWarps = 16;
constexpr int kPairThreads = kPairWarps * 32;
constexpr uint32_t kTabBytes16 = 256u * 64u * 4u;    // one replicated M = 16 table
constexpr uint32_t kExactBytes16 = 256u * 16u * 4u;  // one unreplicated table, [c][m]
constexpr size_t kPairShare = 2 * share_bytes(kPairWarps);   // both queries' shared bounds
template <int MM>
constexpr int kQMax = 32767 / MM;                     // MM entries sum to less than 2^15

// Deferred rescoring.  The rows of a round that pass a query's quantised
// test (about 0.5 % of the rows on the dense bins, but in a third of the
// warps' rounds) are not rescored where they are found, which ran the exact
// sum for one or two lanes of the warp at a time; each warp appends them
// (codes, position, query flags) to a buffer of kCandCap entries in shared
// memory, and every 32 entries the warp rescores them with one entry per
// lane.  The exact sums, the keys and the offers are the same as in place
// (the offers only in another order, which the exact top-k does not see).
// Lists of KP = 256 leave no room for the buffer: they rescore in place.
#ifndef IFVS_PAIR_DEFER
#define IFVS_PAIR_DEFER 1
#endif
constexpr int kCandCap = 64;   // a warp drains at 32: at most 31 + 32 entries are held
constexpr size_t kCandWarpBytes = (size_t)kCandCap * (16 + 4 + 4);

__host__ __device__ constexpr bool pair_defers(int kp) { return IFVS_PAIR_DEFER != 0 && kp <= 128; }

template <int KP>
using PairTopK = WarpTopK<KP, kPairWarps>;

// packed table, two exact tables, extremes + the two shared bounds, lists,
// the candidate buffers, the current work item (no static shared memory:
// it would move the dynamic window off the base the look-ups' immediate
// offsets assume)
size_t scan_pair_smem_bytes(int kp) {
    return (size_t)kTabBytes16 + 2 * (size_t)kExactBytes16 + 64 * 4 + kPairShare + (size_t)kPairWarps * 2 * 2 * kp * 8 +
           (pair_defers(kp) ? (size_t)kPairWarps * kCandWarpBytes : 0) + 16;
}

template <int IMM>
__device__ __forceinline__ uint32_t lds_u32_imm(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(addr), "n"(IMM));
    return v;
}

template <int MM>
__device__ __forceinline__ uint32_t quantised(float L, float lo, float inv) {
    const float y = __fmul_rn(__fsub_rn(L, lo), inv);
    return (uint32_t)fminf((float)kQMax<MM>, fmaxf(0.f, y));   // truncation: floor of y >= 0
}

// The largest quantised sum S a row can have and still reach a top-k whose
// k-th key is thr (INT_MAX: every row; -1: none).  With u = 2^-24 and
// entries L >= 0 (so lo_m >= 0): the float32 distance d, at most sixteen rounded
// additions from 0, is at least (sum_m L_m)(1 - 15u); each q_m is at most
// (L_m - lo_m)(1 + u)^2 inv (two roundings, then floor); so
// S <= (1 + u)^2 inv (d / (1 - 15u) - sum_m lo_m).  At d = dist(thr) the
// bound below is at least that: each of its float32 steps carries a factor
// 1 +- 2^-12 beyond its rounding, and sl, the float32 sum of the lo_m, is at
// most (1 + 15u) sum_m lo_m.  A row with S above it has d > dist(thr).
__device__ __forceinline__ int quant_bound(uint64_t thr, float sl, float inv) {
    const uint32_t hi = (uint32_t)(thr >> 32);
    if (inv == 0.f || hi >= 0x7F800000u) return INT_MAX;   // list not full, inf, NaN or -0
    const float a = __fmul_rn(__uint_as_float(hi), 1.f + 0x1p-12f);
    const float b = __fmul_rn(sl, 1.f - 0x1p-12f);
    const float t = __fmul_rn(__fsub_rn(a, b), __fmul_rn(inv, 1.f + 0x1p-12f));
    if (!(t < 1.0e9f)) return INT_MAX;
    return t < 0.f ? -1 : (int)t;
}

// Quantised sums of two rows (codes ca, cb), both queries at once:
// the addresses of lookup2, integer loads and adds.
template <int MM, bool FAST>
__device__ __forceinline__ void lookup2_q(const uint4 ca, const uint4 cb, uint32_t tb, uint32_t base,
                                             uint32_t& sa, uint32_t& sb) {
    const uint32_t wa[4] = {ca.x, ca.y, ca.z, ca.w};
    const uint32_t wb[4] = {cb.x, cb.y, cb.z, cb.w};
    uint32_t va[MM], vb[MM];
#pragma unroll
    for (int s = 0; s < MM; ++s) {
        const uint32_t sel = 0x5504u | ((uint32_t)(s & 3) << 4);
        uint32_t oa = __byte_perm(wa[s >> 2], tb, sel);
        uint32_t ob = __byte_perm(wb[s >> 2], tb, sel);
        if (!FAST) {
            oa += base;
            ob += base;
        }
        constexpr uint32_t B0 = FAST ? kDynSmemBase : 0u;
        switch (s) {
#define IFVS_LDQ_CASE(S)                         \
    case S:                                      \
        va[s] = lds_u32_imm<B0 + 4 * S>(oa);     \
        vb[s] = lds_u32_imm<B0 + 4 * S>(ob);     \
        break;
            IFVS_LDQ_CASE(0) IFVS_LDQ_CASE(1) IFVS_LDQ_CASE(2) IFVS_LDQ_CASE(3)
            IFVS_LDQ_CASE(4) IFVS_LDQ_CASE(5) IFVS_LDQ_CASE(6) IFVS_LDQ_CASE(7)
            IFVS_LDQ_CASE(8) IFVS_LDQ_CASE(9) IFVS_LDQ_CASE(10) IFVS_LDQ_CASE(11)
            IFVS_LDQ_CASE(12) IFVS_LDQ_CASE(13) IFVS_LDQ_CASE(14) IFVS_LDQ_CASE(15)
#undef IFVS_LDQ_CASE
            default: break;
        }
    }
    uint32_t xa = 0u, xb = 0u;
#pragma unroll
    for (int s = 0; s < MM; ++s) {
        xa += va[s];
        xb += vb[s];
    }
    sa = xa;
    sb = xb;
}

// Exact float32 distance of one row from an unreplicated table ex[c * 16 + m]:
// byte s holds subspace (s + rot) mod MM, rot = (its index mod 32) mod MM,
// added for s ascending from 0, as lookup2 does.
// Called for the rare candidate rows only: kept out of line, the round's
// code is smaller (measured 1-2 % faster than inlining its eight copies).
template <int MM>
__device__ __noinline__ float exact_row(const uint4 c, const float* ex, int rot) {
    const uint32_t w[4] = {c.x, c.y, c.z, c.w};
    float d = 0.f;
#pragma unroll
    for (int s = 0; s < MM; ++s) {
        const uint32_t code = (w[s >> 2] >> (8 * (s & 3))) & 0xFFu;
        const int m = MM == 16 ? (s + rot) & 15 : (s + rot >= MM ? s + rot - MM : s + rot);
        d = __fadd_rn(d, ex[code * 16u + (uint32_t)m]);
    }
    return d;
}

// Both queries' bounds in one word: half h holds bound_h + 0x8000, bound_h
// clamped to [-1, 0x7FFF].  A row's packed sums (each half < 0x8000) are candidates where (packed bounds - sums) keeps bit 15 (query A)
// or bit 31 (query B): no borrow crosses the halves.
__device__ __forceinline__ uint32_t pack_bounds(int ta, int tb) {
    ta = ta > 0x7FFF ? 0x7FFF : ta;
    tb = tb > 0x7FFF ? 0x7FFF : tb;
    return (uint32_t)(ta + 0x8000) | (uint32_t)(tb + 0x8000) << 16;
}

constexpr uint32_t kCandA = 0x00008000u, kCandB = 0x80000000u;

// kU2 rows per lane per round in the paired loop.  Measured on the 10^8-row
// dense bin with candidates rescored in batches: 8 rows 137.4 ms, 4 rows
// 142.1 ms, 2 rows 200.1 ms per batch; 16 rows spill at the 128-register cap
// of a 16-warp CTA.  (With in-place rescoring 4 rows had been the fastest.)
#ifndef IFVS_PAIR_ROWS
#define IFVS_PAIR_ROWS 8
#endif
constexpr int kU2 = IFVS_PAIR_ROWS;
static_assert(kU2 % 2 == 0 && 32 % kU2 == 0, "rows in pairs, whole rounds per block");

// A warp's candidate buffer (shared memory): entry i = codes[i], pos[i],
// flags[i] (kCandA | kCandB for the queries whose test it passed).
struct CandBuf {
    uint4* codes;
    uint32_t* pos;
    uint32_t* flags;
    int cnt;
};

// Rescoring of entries [first, first + n) (n <= 32), entry first + l by lane
// l: the exact float32 distance of each flagged query in the one-query
// kernel's order, the row id for those within the query's k-th key, the
// offers (warp-collective).  Here and below, BM: positions are row ids.
template <int KP, int MM, bool BM>
__device__ __forceinline__ void rescore_entries(const CandBuf& cbuf, int first, int n,
                                                const uint32_t* __restrict__ rows, PairTopK<KP>& tkA,
                                                PairTopK<KP>& tkB, const float* exA, const float* exB, int lane) {
    uint4 c = make_uint4(0, 0, 0, 0);
    uint32_t pos = 0u, f = 0u;
    if (lane < n) {
        c = cbuf.codes[first + lane];
        pos = cbuf.pos[first + lane];
        f = cbuf.flags[first + lane];
    }
    const int rot = (int)((pos & 31u) % MM);
    bool cA = (f & kCandA) != 0u;
    bool cB = (f & kCandB) != 0u;
    float dA = 0.f, dB = 0.f;
    if (cA) dA = exact_row<MM>(c, exA, rot);
    if (cB) dB = exact_row<MM>(c, exB, rot);
    cA = cA && __float_as_uint(dA) <= (uint32_t)(tkA.thr >> 32);
    cB = cB && __float_as_uint(dB) <= (uint32_t)(tkB.thr >> 32);
    const uint32_t row = BM ? pos : ((cA || cB) ? __ldg(rows + pos) : 0u);
    const uint64_t kA = ((uint64_t)__float_as_uint(dA) << 32) | row;
    const uint64_t kB = ((uint64_t)__float_as_uint(dB) << 32) | row;
    tkA.offer(kA, cA && kA < tkA.thr, lane);
    tkB.offer(kB, cB && kB < tkB.thr, lane);
}

// One round of kU2 positions of a block: the shared bounds refreshed,
// quantised sums of both queries, candidates by the packed bounds, exact
// distances and top-k offers for the candidates.  mask(u) holds kCandA / kCandB
// where the position counts for each query.
template <int KP, int MM, bool FAST, bool BM, typename Mask>
__device__ __forceinline__ void pair_round(const uint4 (&c)[kU2], const uint32_t* __restrict__ rows,
                                           uint32_t pos0, Mask mask, PairTopK<KP>& tkA,
                                           PairTopK<KP>& tkB, const float* exA, const float* exB, float slA,
                                           float invA, float slB, float invB, uint32_t tb, uint32_t base,
                                           int rot, int lane, uint32_t& Tpk, CandBuf& cbuf) {
    {
        const uint64_t oa = tkA.thr, ob = tkB.thr;
        tkA.refresh(lane);
        tkB.refresh(lane);
        if (tkA.thr != oa || tkB.thr != ob)
            Tpk = pack_bounds(quant_bound(tkA.thr, slA, invA), quant_bound(tkB.thr, slB, invB));
    }
    uint32_t sq[kU2];
#pragma unroll
    for (int u = 0; u < kU2; u += 2) lookup2_q<MM, FAST>(c[u], c[u + 1], tb, base, sq[u], sq[u + 1]);
    uint32_t cb[kU2], any = 0u;
#pragma unroll
    for (int u = 0; u < kU2; ++u) {
        cb[u] = Tpk - sq[u];
        if (!BM) cb[u] &= mask(u);
        any |= cb[u];
    }
    if (BM) {   // the bits of the bitmap words only where a row is within a bound
        if (!__any_sync(0xFFFFFFFFu, (any & (kCandA | kCandB)) != 0u)) return;
        any = 0u;
#pragma unroll
        for (int u = 0; u < kU2; ++u) {
            cb[u] &= mask(u);
            any |= cb[u];
        }
    }
    if (!__any_sync(0xFFFFFFFFu, any != 0u)) return;
    if constexpr (pair_defers(KP)) {
        const unsigned lt = (1u << lane) - 1u;
#pragma unroll
        for (int u = 0; u < kU2; ++u) {
            const unsigned ball = __ballot_sync(0xFFFFFFFFu, cb[u] != 0u);
            if (ball == 0u) continue;
            if (cb[u] != 0u) {
                const int at = cbuf.cnt + __popc(ball & lt);
                cbuf.codes[at] = c[u];
                cbuf.pos[at] = pos0 + 32u * (uint32_t)u;
                cbuf.flags[at] = cb[u];
            }
            cbuf.cnt += __popc(ball);
            if (cbuf.cnt >= 32) {
                __syncwarp();
                cbuf.cnt -= 32;
                rescore_entries<KP, MM, BM>(cbuf, cbuf.cnt, 32, rows, tkA, tkB, exA, exB, lane);
                __syncwarp();   // the drained slots take the next entries
                Tpk = pack_bounds(quant_bound(tkA.thr, slA, invA), quant_bound(tkB.thr, slB, invB));
            }
        }
        return;
    }
#pragma unroll
    for (int u = 0; u < kU2; ++u) {
        const uint32_t pos = pos0 + 32u * (uint32_t)u;
        bool cA = (cb[u] & kCandA) != 0u;
        bool cB = (cb[u] & kCandB) != 0u;
        float dA = 0.f, dB = 0.f;
        if (cA) dA = exact_row<MM>(c[u], exA, rot);
        if (cB) dB = exact_row<MM>(c[u], exB, rot);
        cA = cA && __float_as_uint(dA) <= (uint32_t)(tkA.thr >> 32);
        cB = cB && __float_as_uint(dB) <= (uint32_t)(tkB.thr >> 32);
        const uint32_t row = BM ? pos : ((cA || cB) ? __ldg(rows + pos) : 0u);
        const uint64_t kA = ((uint64_t)__float_as_uint(dA) << 32) | row;
        const uint64_t kB = ((uint64_t)__float_as_uint(dB) << 32) | row;
        tkA.offer(kA, cA && kA < tkA.thr, lane);
        tkB.offer(kB, cB && kB < tkB.thr, lane);
    }
    Tpk = pack_bounds(quant_bound(tkA.thr, slA, invA), quant_bound(tkB.thr, slB, invB));
}

// Where a pair's rows lie: positions [a, b) of each query on a sorted copy
// (rows: their ids), or the two queries' bitmap words.
struct PairRange {
    const uint8_t* codes;
    const uint32_t* rows;
    uint32_t a1, b1, a2, b2;
    const uint32_t *bmA, *bmB;
};

template <int KP, int MM, bool FAST, bool BM>
__device__ __forceinline__ void scan_positions_pair(const PairRange& r, int64_t blk0, int64_t blk1, PairTopK<KP>& tkA,
                                                    PairTopK<KP>& tkB, const float* exA, const float* exB, float slA,
                                                    float invA, float slB, float invB, uint32_t base, int lane,
                                                    int warp, CandBuf& cbuf) {
    const uint8_t* codes = r.codes;
    const uint32_t* rows = r.rows;
    const uint32_t tb = 4u * (uint32_t)lane;
    const int rot = lane % MM;
    const uint64_t keep = policy_evict_last();
    // the bounds before the first offer (prime_bound): of each lane's rows of the
    // warp's first round the one with the smallest quantised sum, exactly
    {
        uint32_t mA = 0xFFFFFFFFu, mB = 0xFFFFFFFFu;
        const int64_t blk = blk0 + warp;
        if (blk < blk1) {
            const uint32_t pos0 = (uint32_t)(blk * kBlockRows) + (uint32_t)lane;
            uint4 c[kU2];
#pragma unroll
            for (int u = 0; u < kU2; ++u) c[u] = ldg_nc_v4(codes + (size_t)(pos0 + 32u * (uint32_t)u) * 16, keep);
            uint32_t inA = 0u, inB = 0u;   // bit u: row u counts for the query
            if constexpr (BM) {
                inA = ldg_nc_u32(r.bmA + blk * 32 + lane, keep);
                inB = ldg_nc_u32(r.bmB + blk * 32 + lane, keep);
            } else {
#pragma unroll
                for (int u = 0; u < kU2; ++u) {
                    const uint32_t p = pos0 + 32u * (uint32_t)u;
                    inA |= (uint32_t)(p >= r.a1 && p < r.b1) << u;
                    inB |= (uint32_t)(p >= r.a2 && p < r.b2) << u;
                }
            }
            uint32_t sq[kU2], bA = 0xFFFFFFFFu, bB = 0xFFFFFFFFu;   // sum << 8 | row
#pragma unroll
            for (int u = 0; u < kU2; u += 2) lookup2_q<MM, FAST>(c[u], c[u + 1], tb, base, sq[u], sq[u + 1]);
#pragma unroll
            for (int u = 0; u < kU2; ++u) {
                if (inA >> u & 1u) bA = min(bA, (sq[u] & 0xFFFFu) << 8 | (uint32_t)u);
                if (inB >> u & 1u) bB = min(bB, (sq[u] >> 16) << 8 | (uint32_t)u);
            }
            uint4 cA = c[0], cB = c[0];
#pragma unroll
            for (int u = 1; u < kU2; ++u) {
                if ((bA & 0xFFu) == (uint32_t)u) cA = c[u];
                if ((bB & 0xFFu) == (uint32_t)u) cB = c[u];
            }
            const float dA = exact_row<MM>(cA, exA, rot), dB = exact_row<MM>(cB, exB, rot);
            if (bA != 0xFFFFFFFFu) mA = __float_as_uint(dA);
            if (bB != 0xFFFFFFFFu) mB = __float_as_uint(dB);
        }
        prime_bound<kPairWarps>(tkA, mA, lane);
        prime_bound<kPairWarps>(tkB, mB, lane);
    }
    uint32_t Tpk = pack_bounds(quant_bound(tkA.thr, slA, invA), quant_bound(tkB.thr, slB, invB));
    if constexpr (BM) {
        const uint64_t once = policy_evict_first();
        uint32_t nA = 0u, nB = 0u;   // the next block's words
        if (blk0 + warp < blk1) {
            nA = ldg_nc_u32(r.bmA + (blk0 + warp) * 32 + lane, once);
            nB = ldg_nc_u32(r.bmB + (blk0 + warp) * 32 + lane, once);
        }
        for (int64_t blk = blk0 + warp; blk < blk1; blk += kPairWarps) {
            uint32_t wA = nA, wB = nB;
            if (blk + kPairWarps < blk1) {
                nA = ldg_nc_u32(r.bmA + (blk + kPairWarps) * 32 + lane, once);
                nB = ldg_nc_u32(r.bmB + (blk + kPairWarps) * 32 + lane, once);
            }
            if (!__any_sync(0xFFFFFFFFu, (wA | wB) != 0u)) continue;
            const uint32_t pb = (uint32_t)(blk * kBlockRows) + (uint32_t)lane;
#pragma unroll 1
            for (int j0 = 0; j0 < 32; j0 += kU2) {
                uint4 c[kU2];
#pragma unroll
                for (int u = 0; u < kU2; ++u)
                    c[u] = ldg_nc_v4(codes + (size_t)(pb + 32u * (uint32_t)(j0 + u)) * 16, keep);
                auto mask = [&](int u) { return (wA << (15 - u) & kCandA) | (wB << (31 - u) & kCandB); };
                pair_round<KP, MM, FAST, BM>(c, rows, pb + 32u * (uint32_t)j0, mask, tkA, tkB, exA, exB, slA, invA,
                                             slB, invB, tb, base, rot, lane, Tpk, cbuf);
                wA >>= kU2;
                wB >>= kU2;
            }
        }
    } else {
        const uint32_t a1 = r.a1, b1 = r.b1, a2 = r.a2, b2 = r.b2;
        for (int64_t blk = blk0 + warp; blk < blk1; blk += kPairWarps) {
            const uint32_t p0 = (uint32_t)(blk * kBlockRows);
            const uint32_t pe = p0 + kBlockRows;
            const bool inA = p0 < b1 && pe > a1, inB = p0 < b2 && pe > a2;
            if (!(inA || inB)) continue;
            const bool fullA = inA && p0 >= a1 && pe <= b1, fullB = inB && p0 >= a2 && pe <= b2;
            if ((fullA || !inA) && (fullB || !inB)) {
                // each query takes all or none of the block: one mask for all rows
                const uint32_t mc = (fullA ? kCandA : 0u) | (fullB ? kCandB : 0u);
                const uint32_t pb = p0 + (uint32_t)lane;
#pragma unroll 1
                for (int j0 = 0; j0 < 32; j0 += kU2) {
                    uint4 c[kU2];
#pragma unroll
                    for (int u = 0; u < kU2; ++u)
                        c[u] = ldg_nc_v4(codes + (size_t)(pb + 32u * (uint32_t)(j0 + u)) * 16, keep);
                    pair_round<KP, MM, FAST, BM>(c, rows, pb + 32u * (uint32_t)j0, [&](int) { return mc; }, tkA, tkB,
                                                 exA, exB, slA, invA, slB, invB, tb, base, rot, lane, Tpk, cbuf);
                }
                continue;
            }
#pragma unroll 1
            for (int j0 = 0; j0 < 32; j0 += kU2) {
                const uint32_t pos0 = p0 + 32u * (uint32_t)j0 + (uint32_t)lane;
                uint32_t mask[kU2];
#pragma unroll
                for (int u = 0; u < kU2; ++u) {
                    const uint32_t pos = pos0 + 32u * (uint32_t)u;
                    mask[u] = ((fullA || (inA && pos >= a1 && pos < b1)) ? kCandA : 0u) |
                              ((fullB || (inB && pos >= a2 && pos < b2)) ? kCandB : 0u);
                }
                uint4 c[kU2];
#pragma unroll
                for (int u = 0; u < kU2; ++u)
                    c[u] = mask[u] != 0u ? ldg_nc_v4(codes + (size_t)(pos0 + 32u * (uint32_t)u) * 16, keep)
                                         : make_uint4(0, 0, 0, 0);
                pair_round<KP, MM, FAST, BM>(c, rows, pos0, [&](int u) { return mask[u]; }, tkA, tkB, exA, exB, slA,
                                             invA, slB, invB, tb, base, rot, lane, Tpk, cbuf);
            }
        }
    }
    if constexpr (pair_defers(KP)) {
        if (cbuf.cnt > 0) {   // warp-uniform
            __syncwarp();
            rescore_entries<KP, MM, BM>(cbuf, 0, cbuf.cnt, rows, tkA, tkB, exA, exB, lane);
            cbuf.cnt = 0;
        }
    }
}

// Quantisation parameters of one query from the per-subspace extremes
// lo[16], hi[16]: inv (0 turns the test off: every row is rescored) and sl.
template <int MM>
__device__ __forceinline__ void quant_params(const float* lo, const float* hi, float& inv, float& sl) {
    float r = 0.f, s = 0.f;
    bool ok = true;
#pragma unroll
    for (int m = 0; m < MM; ++m) {
        r = fmaxf(r, __fsub_rn(hi[m], lo[m]));
        s = __fadd_rn(s, lo[m]);
        ok = ok && lo[m] >= 0.f;
    }
    inv = __fdiv_rn((float)kQMax<MM>, r);
    if (!(ok && r > 0.f && isfinite(inv) && isfinite(s))) inv = 0.f;
    sl = s;
}

// Two queries are worth one CTA when they read the same column's copy, their
// ranges mostly coincide (at least 3/4 of the longer range is common to both;
// the rows of only one range then run with the other query masked) and the
// two ranges together span at least min_rows positions (pair_rule, api.cu).
// k_schedule makes the pairs (scan_sched.cu).

// Offset of the current work item in the two-query kernel's shared memory.
__host__ __device__ constexpr size_t scan_pair_item_offset(int kp) {
    return (size_t)kTabBytes16 + 2 * (size_t)kExactBytes16 + 64 * 4 + kPairShare + (size_t)kPairWarps * 2 * 2 * kp * 8 +
           (pair_defers(kp) ? (size_t)kPairWarps * kCandWarpBytes : 0);
}

// One work item of the two-query kernel.
template <int KP, int MM, bool BM>
__device__ __forceinline__ void pair_item(uint8_t* smem, const float* __restrict__ tables, const PairRange& range,
                                          const ScanItem& it, int k, uint64_t* __restrict__ partials) {
    uint32_t* ptab = reinterpret_cast<uint32_t*>(smem);
    float* exA = reinterpret_cast<float*>(smem + kTabBytes16);
    float* exB = reinterpret_cast<float*>(smem + kTabBytes16 + kExactBytes16);
    float* prm = reinterpret_cast<float*>(smem + kTabBytes16 + 2 * kExactBytes16);   // lo/hi of A, lo/hi of B
    uint64_t* shareA = reinterpret_cast<uint64_t*>(smem + kTabBytes16 + 2 * kExactBytes16 + 64 * 4);
    uint64_t* shareB = shareA + 1 + kPairWarps;
    uint64_t* tkbufA = reinterpret_cast<uint64_t*>(smem + kTabBytes16 + 2 * kExactBytes16 + 64 * 4 + kPairShare);
    uint64_t* tkbufB = tkbufA + kPairWarps * 2 * KP;
    float* red = reinterpret_cast<float*>(tkbufA);   // [warp][4][16], before the lists are set up
    uint8_t* cand_base = reinterpret_cast<uint8_t*>(tkbufB + kPairWarps * 2 * KP);   // 16-byte aligned
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t qA = it.qa, qB = it.qb;
    uint64_t* outA = partials + (int64_t)it.la * k;
    uint64_t* outB = partials + (int64_t)it.lb * k;
    // 1) unreplicated float32 tables ex[c * 16 + m] (from the replicated
    //    tables of k_tables: word m < 16 of row c is LUT[m][c]) and the
    //    extremes of each subspace; a thread keeps one subspace m
    {
        const float* srcA = tables + qA * (int64_t)256 * 64;
        const float* srcB = tables + qB * (int64_t)256 * 64;
        const int m = threadIdx.x & 15;
        float loA = INFINITY, hiA = -INFINITY, loB = INFINITY, hiB = -INFINITY;
        for (int i = threadIdx.x; i < 4096; i += kPairThreads) {
            const int c = i >> 4;
            const float x = __ldg(srcA + c * 64 + m), y = __ldg(srcB + c * 64 + m);
            exA[i] = x;
            exB[i] = y;
            loA = fminf(loA, x);
            hiA = fmaxf(hiA, x);
            loB = fminf(loB, y);
            hiB = fmaxf(hiB, y);
        }
        loA = fminf(loA, __shfl_xor_sync(0xFFFFFFFFu, loA, 16));
        hiA = fmaxf(hiA, __shfl_xor_sync(0xFFFFFFFFu, hiA, 16));
        loB = fminf(loB, __shfl_xor_sync(0xFFFFFFFFu, loB, 16));
        hiB = fmaxf(hiB, __shfl_xor_sync(0xFFFFFFFFu, hiB, 16));
        if (lane < 16) {
            red[warp * 64 + m] = loA;
            red[warp * 64 + 16 + m] = hiA;
            red[warp * 64 + 32 + m] = loB;
            red[warp * 64 + 48 + m] = hiB;
        }
    }
    __syncthreads();
    if (threadIdx.x < 64) {
        const int j = threadIdx.x;   // 0-15 lo A, 16-31 hi A, 32-47 lo B, 48-63 hi B
        const bool is_lo = (j & 16) == 0;
        float v = red[j];
        for (int w = 1; w < kPairWarps; ++w) v = is_lo ? fminf(v, red[w * 64 + j]) : fmaxf(v, red[w * 64 + j]);
        prm[j] = v;
    }
    __syncthreads();
    float invA, slA, invB, slB;
    quant_params<MM>(prm, prm + 16, invA, slA);
    quant_params<MM>(prm + 32, prm + 48, invB, slB);
    // 2) the packed table: word w of row c = qA[w mod MM][c] | qB[..] << 16
    for (int i = threadIdx.x; i < 256 * 64; i += kPairThreads) {
        const int c = i >> 6, m = (i & 63) % MM;
        ptab[i] = quantised<MM>(exA[c * 16 + m], prm[m], invA) | quantised<MM>(exB[c * 16 + m], prm[32 + m], invB) << 16;
    }
    __syncthreads();   // the reduction scratch becomes the lists
    share_init<kPairWarps>(shareA);
    share_init<kPairWarps>(shareB);
    PairTopK<KP> tkA, tkB;
    tkA.init(tkbufA + warp * 2 * KP, k, lane, shareA);
    tkB.init(tkbufB + warp * 2 * KP, k, lane, shareB);
    __syncthreads();
    const int64_t lo = it.a, hi = it.b;
    CandBuf cbuf;
    {
        uint8_t* wb = cand_base + (size_t)warp * kCandWarpBytes;
        cbuf.codes = reinterpret_cast<uint4*>(wb);
        cbuf.pos = reinterpret_cast<uint32_t*>(wb + kCandCap * 16);
        cbuf.flags = reinterpret_cast<uint32_t*>(wb + kCandCap * 20);
        cbuf.cnt = 0;
    }
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(ptab);
    if (base == kDynSmemBase)
        scan_positions_pair<KP, MM, true, BM>(range, lo, hi, tkA, tkB, exA, exB, slA, invA, slB, invB, base, lane,
                                              warp, cbuf);
    else
        scan_positions_pair<KP, MM, false, BM>(range, lo, hi, tkA, tkB, exA, exB, slA, invA, slB, invB, base, lane,
                                               warp, cbuf);
    merge_warps<KP, kPairWarps>(tkA, tkbufA, k, lane, warp, outA);
    merge_warps<KP, kPairWarps>(tkB, tkbufB, k, lane, warp, outB);
}

// Persistent: one CTA per SM takes work items, so no SM idles through a ragged
// last wave of long ones (512 pairs as one item each over 152 SMs left the last
// of 3.4 waves 0.6 empty).
template <int KP, int MM>
__global__ void __launch_bounds__(kPairThreads, 1)
k_scan_list_pair(const float* __restrict__ tables, SortedCols sc, const ScanPlan* __restrict__ plan,
                 const uint8_t* __restrict__ codes, const uint32_t* __restrict__ bm, int64_t bm_words, int k,
                 ScanSched sched, bool first) {
    extern __shared__ __align__(256) uint8_t smem[];
    scan_begin(first);
    for (ItemLoop loop(sched, 2, smem + scan_pair_item_offset(KP)); loop.more(); loop.next()) {
        const ScanItem it = loop.items[loop.at];
        const ScanPlan pA = plan[it.qa], pB = plan[it.qb];
        const PairRange r{sc.codes_of(pA.col), sc.rows_of(pA.col), (uint32_t)pA.a, (uint32_t)pA.b,
                          (uint32_t)pB.a,      (uint32_t)pB.b,     nullptr,        nullptr};
        pair_item<KP, MM, false>(smem, tables, r, it, k, sched.partials);
    }
    for (ItemLoop loop(sched, 3, smem + scan_pair_item_offset(KP), true); loop.more(); loop.next()) {
        const ScanItem it = loop.items[loop.at];
        const PairRange r{codes, nullptr, 0u, 0u, 0u, 0u, bm + it.qa * bm_words, bm + it.qb * bm_words};
        pair_item<KP, MM, true>(smem, tables, r, it, k, sched.partials);
    }
    scan_end(first);
}

bool scan_pairs_fit(const ScanShape& sh, int k) {
    return fixed_m(sh) != 0 && scan_pair_smem_bytes(scan_kp(k)) <= (size_t)max_smem_optin();
}

cudaError_t launch_scan_pairs(const float* tab, SortedCols sc, const ScanPlan* plan, const uint8_t* codes,
                              const uint32_t* bm, int64_t nq, int k, const ScanShape& sh, const ScanSched& sched,
                              ScanOrder o, cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    const int kp = scan_kp(k);
    const bool m16 = fixed_m(sh) == 16;
    auto kern = kp == 32    ? (m16 ? k_scan_list_pair<32, 16> : k_scan_list_pair<32, 12>)
                : kp == 64  ? (m16 ? k_scan_list_pair<64, 16> : k_scan_list_pair<64, 12>)
                : kp == 128 ? (m16 ? k_scan_list_pair<128, 16> : k_scan_list_pair<128, 12>)
                            : (m16 ? k_scan_list_pair<256, 16> : k_scan_list_pair<256, 12>);
    const size_t ps = scan_pair_smem_bytes(kp);
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ps);
    if (e != cudaSuccess) return e;
    const unsigned grid = std::max(item_grid(sched.group[2]), item_grid(sched.group[3]));
    return launch_kernel(kern, dim3(grid), dim3(kPairThreads), ps, o.chain, s, tab, sc, plan, codes, bm,
                         sh.n_blocks * 32, k, sched, o.first);
}

}  // namespace ifvs
