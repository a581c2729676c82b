// Conditioning and table build of §2.
//
// k_prepare (one CTA per query): the predicate's canonical form and scan plan;
// the pair <q, f> is fingerprinted by h hash functions into the memory bank
// (FNV-1a-64 of the key bytes, then the SplitMix64 finalizer of base XOR
// seed_i, mod B — the paper names no hash function), alpha = sum of the h
// fetched bank rows, and the filter weights w_f = softplus(w_z) (w_f = 1 when
// no w_z is given: the paper's initial state).
//
// k_lut (grid: subspace m x query group; thread = codeword k): the
// adjustment Delta[m][k][:] = sum_j alpha[m][j] W[m][j][k][:] is formed with
// the thread's slice of W held in registers across the whole query group,
// C_iFVS = C_PQ + Delta, and the weighted ADC table
// LUT[m][k] = sum_t w_f[m ds + t] (q[m ds + t] - C_iFVS[m][k][t])^2, which
// turns the Rank score of §2 into an additive distance (score = sum w q^2 -
// dist).  C_iFVS is only written out on request.
#include "internal.cuh"

namespace ifvs {

// ---- fingerprint ----------------------------------------------------------
//
// FNV-1a-64 (h <- (h xor byte) P for every byte) by one warp instead of one
// thread, whose chain of 64-bit multiplications took 11 us for a 532-byte key
// and 86 us for a 3868-byte one.  Three facts make it parallel:
//  * The low byte evolves by itself: l <- ((l xor b) 0xb3) mod 256, and bit j
//    of the product is bit j of x = l xor b (0xb3 is odd) xor a carry c_j of
//    the lower bits of x.  So bit j of every l in a run of bytes is a prefix
//    xor of (b_j xor c_j), once the bits below j are known: eight rounds of
//    bitwise work on 32 bytes per lane, a ballot each.
//  * 0xb3 x = s + 16 s + 128 x with s = 3 x: two ripple carries.
//  * From a start value whose low byte is known the run is affine in the rest:
//    F(h) = F(l) + (h - l) P^len; every lane hashes its 32 bytes from its l and
//    five combinations join the lanes.

constexpr uint64_t kFnvPrime = 1099511628211ull;
constexpr uint64_t kFnvBasis = 14695981039346656037ull;

__device__ __forceinline__ uint64_t splitmix64_finalizer(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

// bit 8 i + j <-> bit 8 j + i: the 8 x 8 bit matrix of 8 bytes, transposed
__device__ __forceinline__ uint64_t transpose8(uint64_t x) {
    uint64_t t = (x ^ (x >> 7)) & 0x00AA00AA00AA00AAull;
    x ^= t ^ (t << 7);
    t = (x ^ (x >> 14)) & 0x0000CCCC0000CCCCull;
    x ^= t ^ (t << 14);
    t = (x ^ (x >> 28)) & 0x00000000F0F0F0F0ull;
    return x ^ t ^ (t << 28);
}

__device__ __forceinline__ uint32_t majority(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (c & (a | b)); }

// h after the key's words [first, first + 256), word(i) giving word i (words
// before 0 are absent: the run is right-aligned); every lane takes 8 words
template <class Word>
__device__ __forceinline__ uint64_t fnv_run(uint64_t h, int first, const Word& word, int lane) {
    uint32_t w[8];
    uint32_t mask = 0u;    // bytes present
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int at = first + lane * 8 + i;
        w[i] = at >= 0 ? word(at) : 0u;
        mask |= at >= 0 ? 0xFu << (4 * i) : 0u;
    }
    uint32_t b[8];         // bit i of b[j]: bit j of byte i
    {
        uint32_t lo[4], hi[4];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const uint64_t t = transpose8((uint64_t)w[2 * g + 1] << 32 | w[2 * g]);
            lo[g] = (uint32_t)t;
            hi[g] = (uint32_t)(t >> 32);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t sel = (uint32_t)(j | (j + 4) << 4);
            b[j] = __byte_perm(__byte_perm(lo[0], lo[1], sel), __byte_perm(lo[2], lo[3], sel), 0x5410);
            b[j + 4] = __byte_perm(__byte_perm(hi[0], hi[1], sel), __byte_perm(hi[2], hi[3], sel), 0x5410);
        }
    }
    uint32_t x[8], s[8], k1 = 0u, k2 = 0u, start = 0u;
    const uint32_t before = (1u << lane) - 1u;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const uint32_t below = j > 0 ? x[j - 1] : 0u;
        uint32_t c = below ^ k1 ^ k2;
        if (j >= 4) c ^= s[j - 4];
        if (j == 7) c ^= x[0];
        uint32_t t = (b[j] ^ c) & mask;
        t ^= t << 1;
        t ^= t << 2;
        t ^= t << 4;
        t ^= t << 8;
        t ^= t << 16;
        const unsigned odd = __ballot_sync(0xFFFFFFFFu, (t >> 31) != 0u);
        const uint32_t flip = (uint32_t)(__popc(odd & before) & 1) ^ (uint32_t)(h >> j & 1u);
        const uint32_t l = (t << 1) ^ (0u - flip);
        start |= (l & 1u) << j;
        x[j] = l ^ b[j];
        s[j] = x[j] ^ below ^ k1;
        k1 = majority(x[j], below, k1);
        if (j >= 4) k2 = majority(s[j], s[j - 4], k2);
    }
    uint64_t r = start, A = 1ull;
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (first + lane * 8 + i >= 0) {
#pragma unroll
            for (int e = 0; e < 4; ++e) r = (r ^ (uint64_t)(w[i] >> (8 * e) & 0xFFu)) * kFnvPrime;
            A *= kFnvPrime * kFnvPrime * kFnvPrime * kFnvPrime;
        }
    uint64_t C = r - start * A;     // h -> A h + C
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t A2 = __shfl_down_sync(0xFFFFFFFFu, A, o), C2 = __shfl_down_sync(0xFFFFFFFFu, C, o);
        C = A2 * C + C2;            // lanes that are multiples of 2 o hold their group's map
        A *= A2;
    }
    return __shfl_sync(0xFFFFFFFFu, A * h + C, 0);
}

__device__ __forceinline__ float softplus_f32(float x) {
    // log(1 + e^x) without overflow on either side
    return x > 0.f ? x + log1pf(expf(-x)) : log1pf(expf(x));
}

// ---- scan plan --------------------------------------------------------------
//
// A predicate that constrains one column selects, for that column's canonical
// interval [lo, lo + wm1], a contiguous segment of the rows sorted by (value,
// row): two searches give it, and its length is the exact pool size.  On an
// index with composite copies a predicate that fixes one of the two columns
// and bounds the other does the same.  Pools up to max_rows take the
// row-list scan (no filter pass, no bitmap); empty and malformed predicates
// take it with an empty segment, and a predicate that constrains no column
// (every row passes) takes it with all N positions of column 0's copy; every
// other query takes the bitmap path.

// first index in [0, n] whose value is not below x; the warp probes 32 places
// a round (5 rounds at 10^7 values, against 24 dependent loads of a thread)
template <class T>
__device__ __forceinline__ int64_t first_not_below(const T* __restrict__ v, int64_t n, T x, int lane) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t step = (hi - lo) <= 32 ? 1 : (hi - lo) / 33 + 1;
        const int64_t at = lo + (lane + 1) * step - 1;
        const bool below = at < hi && __ldg(v + at) < x;
        const int64_t cnt = __popc(__ballot_sync(0xFFFFFFFFu, below));
        const int64_t top = lo + (cnt + 1) * step - 1;   // probe cnt, if there is one, is not below
        lo += cnt * step;
        if (step == 1) break;
        hi = top < hi ? top : hi;
    }
    return lo;
}

// Where a predicate's segment starts (end = 0) or ends (end = 1): the copy and
// the value (or composite key) to search for; false: no search is needed
// (*edge is the answer) or there is no segment (*copy < 0).
__device__ __forceinline__ bool segment_bound(const CanonPred& cp, const SortedCols& sc, int64_t N, int end, int* copy,
                                              int64_t* value, uint64_t* key, int64_t* edge) {
    *copy = -1;
    *edge = 0;
    if (cp.empty) {
        *copy = 0;
        return false;
    }
    if (cp.used == 0u) {
        if (sc.n > 0 && sc.vals_of(0) != nullptr) *copy = 0;
        *edge = end ? N : 0;
        return false;
    }
    if (__popc(cp.used) == 1) {
        const int c = __ffs(cp.used) - 1;
        if (c >= sc.n || sc.vals_of(c) == nullptr) return false;
        int64_t lo = 0, wm1 = 0;
#pragma unroll
        for (int i = 0; i < IFVS_MAX_ATTRS; ++i)
            if (c == i) {
                lo = cp.lo[i];
                wm1 = cp.wm1[i];
            }
        *copy = c;
        *value = end ? lo + wm1 + 1 : lo;
        *edge = N;
        return *value <= 2147483647ll;     // above every value: N
    }
    if (cp.used == 3u && sc.ckeys[0] != nullptr && (cp.wm1[0] == 0u || cp.wm1[1] == 0u)) {
        // columns 0 and 1, one of them fixed to a value: a position range of
        // the composite copy keyed by that column first
        const int j = cp.wm1[0] == 0u ? 0 : 1;
        const int32_t v = cp.lo[j], lo2 = cp.lo[1 - j];
        *copy = kComposite + j;
        // one past (v, lo2 + w2) is the next composite key (it carries into
        // the primary half when the secondary value is the largest int32)
        const uint64_t k = ckey(v, (int32_t)((uint32_t)lo2 + (end ? cp.wm1[1 - j] : 0u)));
        *key = k + (end ? 1ull : 0ull);
        *edge = N;
        return !(end && k == ~0ull);
    }
    return false;
}

// Everything about a query that comes before its tables, one CTA each: the
// predicate's canonical form, its scan plan (warps 0 and 1 search the two ends
// of the segment), the fingerprint of <q, f> (warp 2) and from it alpha, and
// the filter weights.  One launch for what took three and a memset, 28 us for
// one query on 10^6 rows and 40 us on 10^7.
constexpr int kPrepThreads = 128;

__global__ void __launch_bounds__(kPrepThreads) k_prepare(PrepareArgs a) {
    const int64_t qi = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ uint32_t s_idx[64];
    __shared__ int64_t s_end[2];
    __shared__ CanonPred s_cp;
    start_dependents();
    if (tid == 0) {
        const ifvs_predicate p = a.preds[qi];
        CanonPred cp;
        if (canonicalize(p, a.cols.type, a.cols.n, &cp) != 0) atomicOr(a.err, 1);
        if (a.canon != nullptr) a.canon[qi] = cp;
        s_cp = cp;
    }
    if (a.plan != nullptr) __syncthreads();
    if (a.plan != nullptr && warp < 2) {
        int copy = -1;
        int64_t value = 0, at = 0;
        uint64_t key = 0ull;
        if (segment_bound(s_cp, a.sorted, a.N, warp, &copy, &value, &key, &at))
            at = copy >= kComposite ? first_not_below<uint64_t>(a.sorted.ckeys_of(copy - kComposite), a.N, key, lane)
                                    : first_not_below<int32_t>(a.sorted.vals_of(copy), a.N, (int32_t)value, lane);
        if (lane == 0) s_end[warp] = at;
    }
    if (a.bank != nullptr && warp == 2) {
        const uint32_t* qw = reinterpret_cast<const uint32_t*>(a.q + qi * a.D);
        const uint32_t* pw = reinterpret_cast<const uint32_t*>(a.preds + qi);
        int nc = (int)pw[0];
        nc = nc < 0 ? 0 : (nc > IFVS_MAX_CLAUSES ? IFVS_MAX_CLAUSES : nc);
        // the key: q, n_clauses, then each clause's col, op, lo, hi (24 bytes)
        const int D = a.D, nw = D + 1 + 6 * nc;
        auto word = [&](int i) { return __ldg(i < D ? qw + i : (i == D ? pw : pw + (i - D + 1))); };
        uint64_t h = kFnvBasis;
        for (int first = nw - (nw + 255) / 256 * 256; first < nw; first += 256) h = fnv_run(h, first, word, lane);
        for (int i = lane; i < a.h; i += 32)
            s_idx[i] = (uint32_t)(splitmix64_finalizer(h ^ a.seeds[i]) % (uint64_t)a.B);
    }
    if (a.wf != nullptr)
        for (int d = tid; d < a.D; d += kPrepThreads)
            a.wf[qi * a.D + d] = a.wz != nullptr ? softplus_f32(a.wz[qi * a.wz_stride + d]) : 1.0f;
    __syncthreads();
    if (a.plan != nullptr && tid == 0) {
        ScanPlan p;
        p.a = p.b = 0;
        p.col = p.list = 0;
        int copy;
        int64_t value, at;
        uint64_t key;
        segment_bound(s_cp, a.sorted, a.N, 0, &copy, &value, &key, &at);
        const int64_t len = s_end[1] - s_end[0];
        if (copy >= 0 && len <= a.max_rows) {
            p.a = s_end[0];
            p.b = s_end[1];
            p.col = copy;
            p.list = 1;
        }
        a.plan[qi] = p;
        a.npass[qi] = p.list ? (unsigned long long)len : 0ull;   // the filter adds to the others
    }
    if (a.bank != nullptr) {
        if (a.idx != nullptr)
            for (int i = tid; i < a.h; i += kPrepThreads) a.idx[qi * a.h + i] = s_idx[i];
        for (int t = tid; t < a.Mr; t += kPrepThreads) {
            float s = 0.f;
            for (int i = 0; i < a.h; ++i) s += a.bank[(int64_t)s_idx[i] * a.Mr + t];
            a.alpha[qi * a.Mr + t] = s;
        }
    }
}

cudaError_t launch_prepare(const PrepareArgs& a, int64_t nq, cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    k_prepare<<<(unsigned)nq, kPrepThreads, 0, s>>>(a);
    return cudaGetLastError();
}

// Fixed (ds, r): the thread keeps W[m][:][k][:] and C_PQ[m][k][:] in registers.
template <int DS, int R>
__global__ void __launch_bounds__(256) k_lut_fixed(const float* __restrict__ cpq,
                                                   const float* __restrict__ W,
                                                   const float* __restrict__ alpha,
                                                   const float* __restrict__ q,
                                                   const float* __restrict__ wf, int64_t nq,
                                                   int M, int K, int q_per_cta,
                                                   float* __restrict__ lut,
                                                   float* __restrict__ cifvs) {
    const int m = blockIdx.x;
    const int k = threadIdx.x;
    if (k >= K) return;
    const int D = M * DS;
    float c0[DS];
    float w[R][DS];
#pragma unroll
    for (int t = 0; t < DS; ++t) c0[t] = cpq[((int64_t)m * K + k) * DS + t];
    if (alpha != nullptr) {
#pragma unroll
        for (int j = 0; j < R; ++j)
#pragma unroll
            for (int t = 0; t < DS; ++t) w[j][t] = W[(((int64_t)m * R + j) * K + k) * DS + t];
    }
    const int64_t q0 = (int64_t)blockIdx.y * q_per_cta;
    const int64_t q1 = min(nq, q0 + (int64_t)q_per_cta);
    for (int64_t qi = q0; qi < q1; ++qi) {
        float c[DS];
        if (alpha != nullptr) {
            float a[R];
#pragma unroll
            for (int j = 0; j < R; ++j) a[j] = alpha[(qi * M + m) * R + j];
#pragma unroll
            for (int t = 0; t < DS; ++t) {
                float delta = 0.f;
#pragma unroll
                for (int j = 0; j < R; ++j) delta = fmaf(a[j], w[j][t], delta);
                c[t] = c0[t] + delta;
            }
        } else {
#pragma unroll
            for (int t = 0; t < DS; ++t) c[t] = c0[t];
        }
        float s = 0.f;
#pragma unroll
        for (int t = 0; t < DS; ++t) {
            const float diff = q[qi * D + m * DS + t] - c[t];
            s = fmaf(wf[qi * D + m * DS + t] * diff, diff, s);
        }
        lut[(qi * M + m) * K + k] = s;
        if (cifvs != nullptr) {
#pragma unroll
            for (int t = 0; t < DS; ++t) cifvs[((qi * M + m) * K + k) * DS + t] = c[t];
        }
    }
}

// Any (ds, r): W and C_PQ are read through the cache inside the query loop.
__global__ void __launch_bounds__(256) k_lut_any(const float* __restrict__ cpq,
                                                 const float* __restrict__ W,
                                                 const float* __restrict__ alpha,
                                                 const float* __restrict__ q,
                                                 const float* __restrict__ wf, int64_t nq, int M,
                                                 int K, int ds, int r, int q_per_cta,
                                                 float* __restrict__ lut,
                                                 float* __restrict__ cifvs) {
    const int m = blockIdx.x;
    const int k = threadIdx.x;
    if (k >= K) return;
    const int D = M * ds;
    const int64_t q0 = (int64_t)blockIdx.y * q_per_cta;
    const int64_t q1 = min(nq, q0 + (int64_t)q_per_cta);
    for (int64_t qi = q0; qi < q1; ++qi) {
        float s = 0.f;
        for (int t = 0; t < ds; ++t) {
            float delta = 0.f;
            if (alpha != nullptr)
                for (int j = 0; j < r; ++j)
                    delta = fmaf(alpha[(qi * M + m) * r + j],
                                 __ldg(W + (((int64_t)m * r + j) * K + k) * ds + t), delta);
            const float c = __ldg(cpq + ((int64_t)m * K + k) * ds + t) + delta;
            const float diff = q[qi * D + m * ds + t] - c;
            s = fmaf(wf[qi * D + m * ds + t] * diff, diff, s);
            if (cifvs != nullptr) cifvs[((qi * M + m) * K + k) * ds + t] = c;
        }
        lut[(qi * M + m) * K + k] = s;
    }
}

cudaError_t launch_lut(const float* cpq, const float* W, const float* alpha, const float* q,
                       const float* wf, int64_t nq, int M, int K, int ds, int r, float* lut,
                       float* cifvs, int num_sms, cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    // query groups: enough CTAs to cover the GPU, while each CTA reuses its
    // registers' W slice across as many queries as possible
    int64_t groups = ((int64_t)num_sms * 4 + M - 1) / M;
    if (groups > nq) groups = nq;
    if (groups < 1) groups = 1;
    if (groups > 65535) groups = 65535;
    const int64_t qpc = (nq + groups - 1) / groups;
    groups = (nq + qpc - 1) / qpc;
    dim3 grid((unsigned)M, (unsigned)groups);
    const int threads = K <= 32 ? 32 : (K <= 64 ? 64 : (K <= 128 ? 128 : 256));
    if (ds == 8 && (r == 8 || alpha == nullptr))
        k_lut_fixed<8, 8><<<grid, threads, 0, s>>>(cpq, W, alpha, q, wf, nq, M, K, (int)qpc,
                                                   lut, cifvs);
    else
        k_lut_any<<<grid, threads, 0, s>>>(cpq, W, alpha, q, wf, nq, M, K, ds, r, (int)qpc, lut,
                                           cifvs);
    return cudaGetLastError();
}

// ---- tables in the scan's layout, straight from the conditioning ---------------
//
// For ds = 4, 8, 16 and r = 8 (or no bank) a query's weighted tables are
// formed and written in the scan's layout (below) by one kernel, without the
// [M][K] table in between.  CTA (8 subspaces x 32 codewords, query group):
// warp m, lane c keeps W[m][:][c][:] and C_PQ[m][c] in registers across the
// group.  alpha, q and w_f of 8 queries at a time arrive in shared memory by
// asynchronous copies, one stage ahead, and are read as broadcasts: fetched by
// every lane for itself they filled the L1 data pipe (78 % busy).  The entries
// pass through shared memory so that 8 lanes write a codeword's 8 words as one
// sector, to each of their places in row c.  The arithmetic is k_lut_fixed's.
// Words from M + 31 on are never read and stay unwritten.  1024 queries at
// M = 16 took 95 us as two kernels, 28 us here; 256 queries at M = 120 145 us,
// 59 us here.
constexpr int kTabM = 8, kTabC = 32, kTabQ = 8;
constexpr int kTabThreads = kTabM * kTabC;

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

template <int DS, bool COND>
__global__ void __launch_bounds__(kTabThreads, DS > 8 ? 1 : 2)
k_cond_tables(const float* __restrict__ cpq, const float* __restrict__ W, const float* __restrict__ alpha,
              const float* __restrict__ q, const float* __restrict__ wf, int64_t nq, int M, int K, int S,
              int q_per_cta, int vec, float* __restrict__ tab) {
    constexpr int R = 8, NX = kTabM * DS, NA = kTabM * R, NP = NA + 2 * NX;   // floats per query of a stage
    __shared__ __align__(16) float par[2][kTabQ][NP];                         // alpha, q, w_f
    __shared__ float st[kTabQ][kTabC * (kTabM + 1)];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = (int)(blockIdx.x / (256 / kTabC)) * kTabM, c0 = (int)(blockIdx.x % (256 / kTabC)) * kTabC;
    const int D = M * DS, mg = min(kTabM, M - m0);
    const int64_t q0 = (int64_t)blockIdx.y * q_per_cta;
    const int64_t q1 = min(nq, q0 + (int64_t)q_per_cta);
    start_dependents();
    auto stage = [&](int64_t s0, int b) {   // queries [s0, s0 + kTabQ)
        const int ns = (int)min((int64_t)kTabQ, q1 - s0);
        if (COND)
            for (int e = tid; e < ns * (NA / 4); e += kTabThreads) {
                const int i = e / (NA / 4), o = (e - i * (NA / 4)) * 4;
                if (o < mg * R) cp_async16(&par[b][i][o], alpha + ((s0 + i) * M + m0) * R + o);
            }
        for (int e = tid; e < ns * (NX / 4); e += kTabThreads) {
            const int i = e / (NX / 4), o = (e - i * (NX / 4)) * 4;
            if (o >= mg * DS) continue;
            const int64_t at = (s0 + i) * D + m0 * DS + o;
            cp_async16(&par[b][i][NA + NX + o], wf + at);
            if (vec)
                cp_async16(&par[b][i][NA + o], q + at);
            else
#pragma unroll
                for (int u = 0; u < 4; ++u) cp_async4(&par[b][i][NA + o + u], q + at + u);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    stage(q0, 0);
    const int m = m0 + warp, c = c0 + lane;
    const bool real = m < M && c < K;
    float base[DS], w[R][DS];
#pragma unroll
    for (int t = 0; t < DS; ++t) base[t] = real ? __ldg(cpq + ((int64_t)m * K + c) * DS + t) : 0.f;
    if (COND) {
#pragma unroll
        for (int j = 0; j < R; ++j)
#pragma unroll
            for (int t = 0; t < DS; t += 4) {
                const float4 v =
                    real ? __ldg(reinterpret_cast<const float4*>(W + (((int64_t)m * R + j) * K + c) * DS + t))
                         : make_float4(0.f, 0.f, 0.f, 0.f);
                w[j][t] = v.x, w[j][t + 1] = v.y, w[j][t + 2] = v.z, w[j][t + 3] = v.w;
            }
    }
    // where this thread writes: codeword wc, subspace wm
    const int wc = tid / kTabM, wm = tid % kTabM;
    float* out = tab + (q0 * 256 + c0 + wc) * (int64_t)S;
    int b = 0;
#pragma unroll 1
    for (int64_t s0 = q0; s0 < q1; s0 += kTabQ, b ^= 1) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();   // the stage is here, the other buffer and the entries are read
        if (s0 + kTabQ < q1) stage(s0 + kTabQ, b ^ 1);
        const int ns = (int)min((int64_t)kTabQ, q1 - s0);
#pragma unroll 1
        for (int i = 0; i < ns; ++i) {
            const float4* pa = reinterpret_cast<const float4*>(&par[b][i][warp * R]);
            const float4* px = reinterpret_cast<const float4*>(&par[b][i][NA + warp * DS]);
            const float4* pf = reinterpret_cast<const float4*>(&par[b][i][NA + NX + warp * DS]);
            float a[R];
            if (COND) {
                const float4 v0 = pa[0], v1 = pa[1];
                a[0] = v0.x, a[1] = v0.y, a[2] = v0.z, a[3] = v0.w;
                a[4] = v1.x, a[5] = v1.y, a[6] = v1.z, a[7] = v1.w;
            }
            float s = 0.f;
#pragma unroll
            for (int t = 0; t < DS; t += 4) {
                const float4 x4 = px[t / 4], f4 = pf[t / 4];
                const float x[4] = {x4.x, x4.y, x4.z, x4.w}, f[4] = {f4.x, f4.y, f4.z, f4.w};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    float cv = base[t + u];
                    if (COND) {
                        float delta = 0.f;
#pragma unroll
                        for (int j = 0; j < R; ++j) delta = fmaf(a[j], w[j][t + u], delta);
                        cv += delta;
                    }
                    const float diff = x[u] - cv;
                    s = fmaf(f[u] * diff, diff, s);
                }
            }
            st[i][lane * (kTabM + 1) + warp] = real ? s : 0.f;
        }
        __syncthreads();
        for (int i = 0; i < ns; ++i, out += (int64_t)256 * S)
            if (wm < mg) {
                const float s = st[i][wc * (kTabM + 1) + wm];
                for (int o = m0 + wm; o < M + 31; o += M) out[o] = s;
            }
    }
    wait_before();
}

template <int DS>
static cudaError_t start_cond_tables(dim3 grid, bool chain, cudaStream_t s, const float* cpq, const float* W,
                                     const float* alpha, const float* q, const float* wf, int64_t nq, int M, int K,
                                     int S, int qpc, int vec, float* tab) {
    auto kern = alpha != nullptr ? k_cond_tables<DS, true> : k_cond_tables<DS, false>;
    return launch_kernel(kern, grid, dim3(kTabThreads), 0, chain, s, cpq, W, alpha, q, wf, nq, M, K, S, qpc, vec, tab);
}

bool cond_tables_fit(int ds, int r, bool cond) { return (ds == 4 || ds == 8 || ds == 16) && (!cond || r == 8); }

cudaError_t launch_cond_tables(const float* cpq, const float* W, const float* alpha, const float* q, const float* wf,
                               int64_t nq, int M, int K, int ds, int S, float* tab, int num_sms, bool chain,
                               cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    const int tiles = (M + kTabM - 1) / kTabM * (256 / kTabC);
    // two CTAs per SM; a group of queries shares a CTA's registers
    int64_t groups = ((int64_t)num_sms * 2 + tiles - 1) / tiles;
    if (groups > nq) groups = nq;
    const int64_t qpc = (nq + groups - 1) / groups;
    groups = (nq + qpc - 1) / qpc;
    const dim3 grid((unsigned)tiles, (unsigned)groups);
    const int vec = (uintptr_t)q % 16 == 0;
    auto start = ds == 4 ? start_cond_tables<4> : (ds == 8 ? start_cond_tables<8> : start_cond_tables<16>);
    return start(grid, chain, s, cpq, W, alpha, q, wf, nq, M, K, S, (int)qpc, vec, tab);
}

// ---- scan tables -------------------------------------------------------------
//
// The scan keeps each query's table in shared memory as 256 rows (one per
// codeword) of S words, word w of row c = LUT[w mod M][c] for w < M + 31
// (zero above).  This kernel writes that layout once per query so that every
// scan CTA fetches it with coalesced 16-byte loads.  Grid: query x 32-codeword
// tile; the tile passes through shared memory padded to 33 words per row so
// that both the coalesced reads and the rotated writes are conflict-free.
__global__ void __launch_bounds__(256) k_tables(const float* __restrict__ lut, int M, int K, int S,
                                                float* __restrict__ tab) {
    __shared__ float st[IFVS_MAX_M * 33];
    const int64_t q = blockIdx.x;
    const int c0 = blockIdx.y * 32;
    const float* src = lut + q * (int64_t)M * K;
    for (int i = threadIdx.x; i < M * 32; i += blockDim.x) {
        const int m = i >> 5, cc = i & 31, c = c0 + cc;
        st[m * 33 + cc] = c < K ? src[(int64_t)m * K + c] : 0.f;
    }
    __syncthreads();
    float* dst = tab + q * (int64_t)256 * S + (int64_t)c0 * S;
    const int wu = M + 31;
    for (int i = threadIdx.x; i < 32 * S; i += blockDim.x) {
        const int cc = i / S, w = i - cc * S;
        dst[i] = w < wu ? st[(w % M) * 33 + cc] : 0.f;
    }
}

cudaError_t launch_tables(const float* lut, int64_t nq, int M, int K, int S, float* tab,
                          cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    dim3 grid((unsigned)nq, 8);
    k_tables<<<grid, 256, 0, s>>>(lut, M, K, S, tab);
    return cudaGetLastError();
}

}  // namespace ifvs
