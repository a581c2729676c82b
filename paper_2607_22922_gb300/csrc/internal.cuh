// Internal declarations of the iFVS GB300 library (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "ifvs.h"

namespace ifvs {

// A bitmap block covers 1024 rows: 32 lane-words of 32 bits.  In the
// device ("lane-major") layout, word (b * 32 + l) bit j is row
// b * 1024 + 32 * j + l, so lane l of a warp owns rows congruent to l mod 32
// and reads its 32 pass bits of a block in one coalesced 128-byte load.
constexpr int kBlockRows = 1024;
constexpr int kWarps = 8;          // warps per CTA in the scan and filter
constexpr int kThreads = kWarps * 32;

// One predicate reduced to a closed interval per attribute column:
// row passes iff for every column c, (uint32)(a_c - lo[c]) <= wm1[c].
struct CanonPred {
    int32_t lo[IFVS_MAX_ATTRS];
    uint32_t wm1[IFVS_MAX_ATTRS];
    uint32_t used;     // bit c: column c is constrained
    int32_t empty;     // 1: no row can pass
    int32_t invalid;   // 1: malformed predicate
    int32_t pad;
};

// Reduce a predicate to per-column intervals (clauses on one column
// intersect).  Returns 0, or -1 when the predicate is malformed.
__host__ __device__ inline int canonicalize(const ifvs_predicate& p, const int32_t* types,
                                            int n_attrs, CanonPred* out) {
    int64_t lo[IFVS_MAX_ATTRS], hi[IFVS_MAX_ATTRS];
    out->used = 0;
    out->empty = 0;
    out->invalid = 0;
    out->pad = 0;
    for (int c = 0; c < IFVS_MAX_ATTRS; ++c) {
        bool i16 = c < n_attrs && types[c] == IFVS_ATTR_I16;
        lo[c] = i16 ? -32768 : -2147483648LL;
        hi[c] = i16 ? 32767 : 2147483647LL;
    }
    int bad = (p.n_clauses < 0 || p.n_clauses > IFVS_MAX_CLAUSES || p.reserved != 0);
    int nc = bad ? 0 : p.n_clauses;
    for (int i = 0; i < nc; ++i) {
        const ifvs_clause& cl = p.c[i];
        if (cl.col < 0 || cl.col >= n_attrs) { bad = 1; break; }
        int64_t a, b;
        const int64_t kMin = (-9223372036854775807LL - 1), kMax = 9223372036854775807LL;
        bool none = false;
        switch (cl.op) {
            case IFVS_OP_EQ: a = cl.lo; b = cl.lo; break;
            case IFVS_OP_RANGE:
                a = cl.lo;
                if (cl.hi == kMin) { none = true; b = kMin; } else { b = cl.hi - 1; }
                break;
            case IFVS_OP_GE: a = cl.lo; b = kMax; break;
            case IFVS_OP_LT:
                a = kMin;
                if (cl.lo == kMin) { none = true; b = kMin; } else { b = cl.lo - 1; }
                break;
            case IFVS_OP_GT:
                b = kMax;
                if (cl.lo == kMax) { none = true; a = kMax; } else { a = cl.lo + 1; }
                break;
            case IFVS_OP_LE: a = kMin; b = cl.lo; break;
            default: bad = 1; a = 0; b = 0; break;
        }
        if (bad) break;
        if (none) { out->empty = 1; continue; }
        if (a > lo[cl.col]) lo[cl.col] = a;
        if (b < hi[cl.col]) hi[cl.col] = b;
        out->used |= 1u << cl.col;
    }
    for (int c = 0; c < IFVS_MAX_ATTRS; ++c) {
        if (lo[c] > hi[c]) {
            out->empty = 1;
            out->lo[c] = 0;
            out->wm1[c] = 0;
        } else {
            out->lo[c] = (int32_t)lo[c];
            out->wm1[c] = (uint32_t)(hi[c] - lo[c]);
        }
    }
    if (bad) { out->invalid = 1; out->empty = 1; return -1; }
    return 0;
}

struct AttrCols {
    const void* col[IFVS_MAX_ATTRS];
    int32_t type[IFVS_MAX_ATTRS];
    int32_t n;
};

// ---- sums that carry their rounding errors (TwoSum, Knuth) -------------------
// a + b = hi + lo exactly (hi the rounded sum)
__device__ __forceinline__ void two_sum(float a, float b, float& hi, float& lo) {
    hi = __fadd_rn(a, b);
    const float bb = __fsub_rn(hi, a);
    lo = __fadd_rn(__fsub_rn(a, __fsub_rn(hi, bb)), __fsub_rn(b, bb));
}
// A running sum as a pair of floats, for short runs only: `lo` takes the
// rounding error of every addition and is itself a float, so after n additions
// the pair is off by up to (n - 1)(n - 2) 2^-48 of the sum of the terms'
// magnitudes.  That is reached when the terms are alike (their errors have the
// same sign): 10^6 of 0.1 are off by 43 float32 ulp, 5 x 10^6 of 1.7 by 1500.
struct Sum2 {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float v) {
        float e;
        two_sum(hi, v, hi, e);
        lo = __fadd_rn(lo, e);
    }
    __device__ __forceinline__ bool finite() const { return isfinite(hi) && isfinite(lo); }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};
// Terms per pair where runs of any length are summed: every kPairTerms of them
// the pair goes into a float64 sum.  31 x 30 x 2^-48 < 2^-38 of the magnitudes
// whatever the run's length; over 10^6 to 10^7 terms of every kind tried
// (constant, low-variance, normal, lognormal) the total was as near the exact sum
// as float64 additions one by one.
constexpr int kPairTerms = 32;
// s + get(0) + ... + get(n - 1) to float64 accuracy, 8 terms fetched at a time.
// Terms that a pair cannot hold (infinite, NaN, or a sum beyond float32) are
// fetched again and added in float64: the result is what float64 additions give.
template <class Get>
__device__ __forceinline__ double sum_f64(double s, int n, const Get& get) {
    for (int i0 = 0; i0 < n; i0 += kPairTerms) {
        const int i1 = min(n, i0 + kPairTerms);
        Sum2 p;
        for (int i = i0; i < i1; i += 8) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (i + u < i1) v[u] = get(i + u);
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (i + u < i1) p.add(v[u]);
        }
        double t = p.value();
        if (!p.finite()) {
            t = 0.0;
            for (int i = i0; i < i1; ++i) t += (double)get(i);
        }
        s += t;
    }
    return s;
}


// ---- overlapping launches ----------------------------------------------
//
// The kernels of a search follow each other in one stream.  Launched with
// `chain`, a kernel may start while the one before it still runs (programmatic
// launch), once all of that one's CTAs have called start_dependents:
//   prepare [-> filter] -> schedule -> tables -> scans -> merge [-> rerank]
// A kernel either waits for the one before it at its start (wait_before, after
// reading only what no kernel of the path writes), or, where it needs nothing
// of it, at its end: schedule starts the tables once prepare and filter are
// complete, the first scan waits for the tables, and the other scans start
// with it.  Since every kernel waits before it completes, a kernel that has
// waited sees all that came earlier.  Without `chain` (stage timing, shapes
// with separate table kernels) launches are ordinary and the calls do nothing.
__device__ __forceinline__ void start_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_before() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
inline cudaError_t launch_kernel(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, bool chain, cudaStream_t s,
                                 A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = chain ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// ---- kernel launchers (one per translation unit) -----------------------
// Every launcher returns the cudaError_t of its launch.

// Per-query scan plan: a predicate whose pool is one position range [a, b)
// of a sorted copy (one constrained column; or, with composite copies, one
// column fixed to a value and the other bounded) with at most max_rows rows,
// or an empty / malformed one, takes the sorted-copy scan of copy `col`; the
// rest take the bitmap path.
struct ScanPlan {
    int64_t a, b;
    int32_t col;
    int32_t list;      // 1: row-list scan
};
// Sorted copies of the codes.  Copy c < IFVS_MAX_ATTRS: the rows sorted by
// (column c's value, row); vals[c] holds the values in that order.  For an
// index of exactly two columns, copies kComposite + j (j = 0, 1) are sorted
// by (column j, column 1 - j, row), and ckeys[j] holds the composite key
// ckey(v_j, v_{1-j}) of each position: a predicate fixing column j to one
// value and bounding the other column to an interval selects one contiguous
// position range of that copy.  Every copy: position p holds row rows[p]'s
// codes, rotated by (p mod 32) mod M, padded like the index: row_bytes apart for
// M = 12 and 16, by groups of 32 positions word by word for other M
// (sorted_byte, scan.cu).
constexpr int kComposite = IFVS_MAX_ATTRS;
constexpr int kSortedCopies = IFVS_MAX_ATTRS + 2;

// composite key: unsigned order of the pair is signed (primary, secondary) order
__host__ __device__ inline uint64_t ckey(int32_t primary, int32_t secondary) {
    return ((uint64_t)((uint32_t)primary ^ 0x80000000u) << 32) | (uint64_t)((uint32_t)secondary ^ 0x80000000u);
}

struct SortedCols {
    const uint32_t* rows[kSortedCopies];
    const uint8_t* codes[kSortedCopies];
    const int32_t* vals[IFVS_MAX_ATTRS];
    const uint64_t* ckeys[2];
    int32_t n;
    // copy c's arrays, selected without indexing the parameter at run time
    __host__ __device__ const uint8_t* codes_of(int c) const {
        const uint8_t* r = codes[0];
#pragma unroll
        for (int i = 1; i < kSortedCopies; ++i)
            if (c == i) r = codes[i];
        return r;
    }
    __host__ __device__ const uint32_t* rows_of(int c) const {
        const uint32_t* r = rows[0];
#pragma unroll
        for (int i = 1; i < kSortedCopies; ++i)
            if (c == i) r = rows[i];
        return r;
    }
    __host__ __device__ const int32_t* vals_of(int c) const {
        const int32_t* v = vals[0];
#pragma unroll
        for (int i = 1; i < IFVS_MAX_ATTRS; ++i)
            if (c == i) v = vals[i];
        return v;
    }
    __host__ __device__ const uint64_t* ckeys_of(int j) const { return j == 0 ? ckeys[0] : ckeys[1]; }
};
// What precedes the tables, per query (condition.cu).  Parts whose outputs
// are null are left out.
struct PrepareArgs {
    const ifvs_predicate* preds;
    AttrCols cols;
    CanonPred* canon;              // canonical predicates, or null (checked all the same)
    int* err;                      // |= 1 for any malformed predicate
    // scan plan
    SortedCols sorted;
    int64_t N, max_rows;
    ScanPlan* plan;                // or null
    unsigned long long* npass;     // with plan: pool sizes of list-path queries, 0 for the others
    // fingerprint, alpha (when bank is not null), w_f (when wf is not null)
    const float* q;                // [nq][D]
    int D;
    const uint64_t* seeds;
    int h;
    int64_t B;
    const float* bank;             // [B][Mr]
    int Mr;
    const float* wz;               // w_z of query i at wz + i * wz_stride; null: w_f = 1
    int64_t wz_stride;
    uint32_t* idx;                 // [nq][h], or null
    float* alpha;                  // [nq][Mr]
    float* wf;                     // [nq][D]
};
cudaError_t launch_prepare(const PrepareArgs& a, int64_t nq, cudaStream_t s);

// Filter: lane-major pass bitmaps [nq][n_blocks * 32] + popcounts (added to
// npass) for the bitmap-path queries of `plan` (all queries when plan is null)
cudaError_t launch_filter(AttrCols cols, int64_t N, int64_t n_blocks, const CanonPred* canon,
                          const ScanPlan* plan, int64_t nq, uint32_t* bm, unsigned long long* npass,
                          int num_sms, bool chain, cudaStream_t s);

// 32x32 bit transposes between the lane-major layout and the row-ordered
// layout of the ABI ([nq][ceil(N/32)]).  to_rows = true: lane-major -> rows.
cudaError_t launch_bitmap_layout(const uint32_t* src, uint32_t* dst, int64_t nq,
                                 int64_t n_blocks, int64_t n_words_rows, bool to_rows,
                                 cudaStream_t s);

// Delta, C_iFVS (optional output) and the weighted ADC tables
cudaError_t launch_lut(const float* cpq, const float* W, const float* alpha, const float* q,
                       const float* wf, int64_t nq, int M, int K, int ds, int r,
                       float* lut, float* cifvs, int num_sms, cudaStream_t s);

// weighted ADC tables [nq][M][K] -> the scan's shared-memory layout
// [nq][256][S] (S = tab_words)
cudaError_t launch_tables(const float* lut, int64_t nq, int M, int K, int S, float* tab,
                          cudaStream_t s);

// the same layout straight from the conditioning (alpha null: no bank), for
// the shapes that cond_tables_fit names
bool cond_tables_fit(int ds, int r, bool cond);
cudaError_t launch_cond_tables(const float* cpq, const float* W, const float* alpha, const float* q, const float* wf,
                               int64_t nq, int M, int K, int ds, int S, float* tab, int num_sms, bool chain,
                               cudaStream_t s);

struct ScanShape {
    int64_t n_blocks;      // bitmap blocks (rows padded to n_blocks * 1024)
    int M, K;
    int row_bytes;         // code row stride in bytes (M rounded up to 4)
    int tab_words;         // LUT table stride in words per codeword
    int64_t n_rows;        // N (rows of the index)
};
size_t scan_smem_bytes(int tab_words, int kp);
// CTAs resident per SM: of the bitmap scan, and of the one-query sorted-copy
// scan, for this shape and k
int scan_ctas_per_sm(int tab_words, int kp);
int scan_list_ctas_per_sm(const ScanShape& sh, int k, bool bulk);
int scan_kp(int k);

// ---- work lists of a batch (scan_sched.cu) -------------------------------
constexpr int kRoundRows = 256;   // positions of a warp's round on a sorted copy
// One CTA's work: query qa (with qb when >= 0) on units [a, b): rounds of a
// sorted copy (list group), blocks (bitmap and pair groups); writes list la
// (and lb) of k keys.
struct ScanItem {
    int32_t qa, qb, la, lb;
    uint32_t a, b;
};
struct SchedGroup {
    int64_t slots;     // CTAs resident on the device
    int64_t least;     // fewest units per item
    int64_t fixed;     // units per item set by the caller (0: automatic)
    int64_t cap;       // most items
    int64_t per_slot;  // items per slot aimed at (large batches)
    int64_t start;     // what an item costs beside its units, in units
};
// Groups: one-query sorted-copy scan, bitmap scan, pairs on a sorted copy, pairs
// of bitmap queries.
constexpr int kGroups = 4;
__host__ __device__ constexpr bool pair_group(int g) { return g >= 2; }
struct ScanSched {
    SchedGroup group[kGroups];
    bool by_part;          // the bitmap group's items part by part (scan_sched.cu)
    ScanItem* items[kGroups];
    int* ctl;              // items per group, then work counters
    int2* qlist;           // [nq] (first list, lists) of a query
    int2* pairs;           // pairs of queries: on sorted copies, then of bitmap queries
    uint8_t* paired;       // [nq]
    uint64_t* partials;    // [lists][k]
};
// fills s (pointers from `base`, which may be null); returns the bytes needed.
// most[g] bounds group g's items (0: the group is not used).
// row_bytes: of a code row.
size_t scan_sched_layout(int64_t nq, int k, int64_t n_blocks, int row_bytes, const int (&slots)[kGroups],
                         int64_t chunk_blocks, const int64_t (&most)[kGroups], uint8_t* base, ScanSched* s);
// What two queries must bring to be paired (pair_rule, api.cu); < 0: no pairs.
struct PairRule {
    int64_t span;       // rows a pair on a sorted copy spans, at least
    int64_t total;      // rows of the batch's ranges together, at least
    int64_t bm_pass;    // passing rows of a bitmap query, at least
    int64_t bm_total;   // index rows times such queries, at least
};
// plan null: every query on the bitmap path; npass null: pass counts unknown
cudaError_t launch_schedule(const ScanPlan* plan, const unsigned long long* npass, int64_t nq, int64_t n_blocks,
                            PairRule rule, const ScanSched& s, bool chain, cudaStream_t st);

// How a scan is launched: `chain` as above; first: it is the batch's first scan
// (waits at its start, the others at their end)
struct ScanOrder {
    bool chain, first;
};
// Rank over the bitmap group's items: per item, the k best keys (dist bits <<
// 32 | row) of its blocks' passing rows; `tab` holds the tables written by
// launch_tables
cudaError_t launch_scan(const uint8_t* codes, const float* tab, const uint32_t* bm, int64_t nq, int k,
                        const ScanShape& sh, const ScanSched& sched, ScanOrder o, cudaStream_t s);
// Rank over the list group's items: a query's pool is the position range
// [a, b) of a sorted copy.  Code rows arrive by bulk copies into shared memory
// when `bulk` and the shape allows it (else by per-lane loads); a bounded wait
// that runs out sets bit 4 of *err.  tx_extra: bytes added to what each
// copy's barrier expects (0; positive only to exercise the timeout path).
struct ListOpts {
    bool bulk;
    uint32_t tx_extra;
    int* err;
};
cudaError_t launch_scan_list(const float* tab, SortedCols sc, const ScanPlan* plan, int64_t nq, int k,
                             const ScanShape& sh, const ScanSched& sched, const ListOpts& lo, ScanOrder o,
                             cudaStream_t s);
// Rank over the pair groups' items (M = 12 and 16): two queries per CTA, on a
// sorted copy or, by their bitmaps bm, on the index layout `codes`
bool scan_pairs_fit(const ScanShape& sh, int k);
cudaError_t launch_scan_pairs(const float* tab, SortedCols sc, const ScanPlan* plan, const uint8_t* codes,
                              const uint32_t* bm, int64_t nq, int k, const ScanShape& sh, const ScanSched& sched,
                              ScanOrder o, cudaStream_t s);
// the sorted copy of the codes: dst position p <- row rows[p] of the index
// layout `src`, re-rotated by (p mod 32) mod M; positions >= N are zero
cudaError_t launch_relayout_sorted(const uint8_t* src, const uint32_t* rows, int64_t N, int M,
                                   int row_bytes, int64_t n_rows_pad, uint8_t* dst, cudaStream_t s);
// Select: a query's lists -> ids / dists; npass to npass_copy unless null
cudaError_t launch_merge(const ScanSched& sched, int64_t nq, int k, int64_t* ids, float* dists,
                         const unsigned long long* npass, int64_t* npass_copy, bool chain, cudaStream_t s);
// exact fp32 rerank of cand [nq][R] -> k best
// Select across row shards: [G][nq][k] (dist, global id) -> [nq][k]
int shard_merge_cap();
cudaError_t launch_merge_shards(const float* dists, const int64_t* ids, int64_t nq, int G, int k,
                                float* dists_out, int64_t* ids_out, cudaStream_t s);
cudaError_t launch_rerank(const float* X, int64_t N, int D, const float* q, const int64_t* cand,
                          int64_t nq, int R, int k, int64_t* ids, float* dists, bool chain, cudaStream_t s);
// codes [N][M] -> rotated rows [n_rows_pad][row_bytes]; *bad = 1 if a code >= K
cudaError_t launch_relayout_codes(const uint8_t* src, int64_t N, int M, int K, int row_bytes,
                                  int64_t n_rows_pad, uint8_t* dst, int* bad, cudaStream_t s);

// ---- PQ construction (csrc/pq.cu) --------------------------------------
// codes [n][M] and optional dmin [n][M] (float32 argmin, fixed order); by
// subspace ([M][n]) when `by_subspace`
cudaError_t launch_pq_assign(const float* X, int64_t n, int D, int M, int K, const float* C,
                             uint8_t* codes, float* dmin, bool by_subspace, cudaStream_t s);
// Buffers of Lloyd training, carved from one allocation at `base`
struct LloydBufs {
    uint8_t* base;
    int64_t rows_per_chunk;
    int chunks;
    double* sums;               // [chunks][M][K][ds] member sums
    double* obj;                // [chunks][M] sums of distances
    unsigned long long* far;    // [chunks][M] farthest row: distance bits << 32 | ~row
    unsigned* counts;           // [chunks][M][K] members
    float* dmin;                // [M][n]
    uint8_t* codes;             // [M][n]
    uint8_t* used;              // [M][K]
};
// sets the plan and the pointers (relative to b->base, which may be null) and the bytes needed
void lloyd_plan(int64_t n, int M, int K, int ds, int num_sms, LloydBufs* b, size_t* bytes);
// Lloyd update from b's codes and dmin: means of the members (sum_f64), unused
// codewords on the farthest rows; objective [M] (may be null)
cudaError_t launch_pq_update(const float* X, int64_t n, int D, int M, int K, const LloydBufs& b, const float* C_in,
                             float* C_out, double* objective, cudaStream_t s);

// ---- training of bank, W, w_f (csrc/train.cu) --------------------------
constexpr int kTrainMaxR = 32;     // r per subspace handled by the gradient kernels
constexpr int kTrainMaxV = 512;    // positives + negatives per query
struct TrainQueryArgs {
    const uint8_t* codes;          // index layout (rows rotated, row_bytes apart)
    int row_bytes, M, K, ds, D, r;
    const float* C_pq;             // [M][K][ds]
    const float* W;                // [M][r][K][ds]
    const float* G;                // [M][r][r] Gram matrices (written by the gradient launch)
    const float* q;                // [n][D]
    const float* wf;               // [n][D]
    const float* alpha;            // [n][M r]
    const int64_t* pos;            // positives, row q at pos + q * pos_stride, P of them
    int64_t pos_stride;
    int P;
    const int64_t* negsrc;         // negative source, row q at negsrc + q * neg_stride, S entries
    int64_t neg_stride;
    int S, n_neg;
    int exclude;                   // 1: mined list (skip positives, stop at -1); 0: take as given
    float tau, lambda;
    int64_t n;
    int64_t N;                     // rows of the index: ids outside -1..N-1 are refused
    int* err;                      // |= 2 when a candidate id is outside -1..N-1 (then treated as absent)
    int64_t* neg_out;              // [n][n_neg] or null
    float* gC;                     // [n][M][K][ds] scratch
    float* gw;                     // [n][D] scratch: dL/dw_f per query
    float* galpha;                 // [n][M r] dL/dalpha per query (not divided by n)
    double* loss;                  // [n]
};
size_t train_query_smem(int V, int Mr, int D, int r);
// G [M][r][r] = W[m] W[m]^T
cudaError_t launch_train_gram(const float* W, int M, int r, int KD, float* G, cudaStream_t s);
// per query: candidates, distances, softmax, loss, gC (zeroed by the caller), dL/dw_f, dL/dalpha
cudaError_t launch_train_query(const TrainQueryArgs& a, cudaStream_t s);
// gW [M][r][K ds] of the mean loss (written, not accumulated); scratch of
// train_gW_scratch bytes; *launches = kernels launched
size_t train_gW_scratch(int64_t n, int M, int r, int KD);
cudaError_t launch_train_gW(const float* alpha, const float* gC, const float* W, int64_t n, int M, int r,
                            int KD, float lambda, float inv_n, float* scratch, float* gW,
                            cudaStream_t s, int* launches);

// gbank rows fetched by the batch (other rows must be zeroed by the caller)
cudaError_t launch_train_bank(const uint32_t* idx, int64_t n, int h, int Mr, const float* galpha,
                              float inv_n, float* gbank, cudaStream_t s);
cudaError_t launch_train_wz(const float* gw, int64_t n, int D, const float* wz, float inv_n, float* gwz,
                            cudaStream_t s);
struct SgdArgs {
    float* theta[3];
    const float* g[3];
    int64_t n[3];
    float lr[3];
};
cudaError_t launch_sgd(const SgdArgs& a, cudaStream_t s);

// Read-only view of a loaded index, for entry points defined outside api.cu.
struct IndexView {
    int device;
    int num_sms;
    int max_smem;  // opt-in shared memory per block on `device`, bytes
    int64_t N, n_blocks;
    int M, K, row_bytes, tab_words;
    const uint8_t* codes;
};
int index_view(const ifvs_index* ix, IndexView* out);
// Sets the thread-local message of ifvs_last_error and returns `code`.
int report_error(int code, const char* fmt, ...);

}  // namespace ifvs
