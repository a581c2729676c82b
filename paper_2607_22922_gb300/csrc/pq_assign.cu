// PQ assignment: the codeword of every subspace that is nearest to a row's
// sub-vector, decided in float32 in a fixed order — s = s + (x_t - c_t)^2 for
// t ascending, every operation rounded on its own (no fused multiply-add) —
// with ties to the smallest codeword, so that the codes are bit-exact with
// the same decision made in float32 on the CPU.
//
// k_pq_assign_mma (sub-vectors of 4, 8 and 16 dimensions).  Evaluating all K
// codewords in that order costs 3 ds rounded operations each, 24 at ds = 8:
// the FP32 pipe was the bound (3.5 ms for 2^20 rows x 16 subspaces, 0.76 of
// its peak).  Here the tensor cores rank the codewords and the float32
// decision is made only between those that the ranking cannot separate:
//   score_k = |c_k|^2 - 2 x.c_k        (= distance - |x|^2)
// as one tcgen05.mma chain per 128 rows and subspace on bf16 operands split
// in two, x = xh + xl and -2c = ch + cl (|c|^2 in three parts against a
// column of ones), accumulated in float32 in TMEM: 128 lanes (rows) x 256
// columns (codewords).  Error of a score: the products dropped or rounded
// away are at most 3 x 2^-18 of 2 sum |x_t c_t| <= |x|^2 + |c|^2, and the
// float32 accumulation of up to 64 products at most 64 x 2^-24 x 3 of it; the
// float32 distance it stands for is within 20 x 2^-24 x 2 (|x|^2 + |c|^2) of
// the true one.  So the float32 argmin's score is within
// 2 (1.2e-5 + 1.2e-5 + 2.4e-6) (|x|^2 + max|c|^2) = 5.3e-5 of the smallest
// score, and every codeword within kMargin = 2^-14 (6.1e-5) of it is a
// candidate; kFloor covers what underflow takes (64 products and three parts of
// |c|^2 on either side, 2^-126 each).  The
// unit is a group of 4 codewords: the groups whose smallest score is a
// candidate (one for almost every row) are compared exactly, codewords
// ascending.
//
// Data that would have many candidates, or none that the bound vouches for
// (2^19 rows x 16 subspaces of 8: ordinary data 0.42 ms; every codeword evaluated
// for every row 1.84 ms; each of these up to 2.73 ms before it had its rule):
//  * A codebook far from the origin (is_far) is ranked relative to its mean mu,
//    whose rounding adds 4 x 2^-24 (|x - mu|^2 + |c - mu|^2) to a score's error:
//    0.58 ms (offset 30 times the spread or more).
//  * A codeword that is not finite is at an infinite or NaN distance, never
//    smaller than another, unless it is the first, whose distance stands until
//    a smaller one is found: it gets the score of the columns beyond K.  A row
//    that is not finite takes codeword 0 for the same reason: 0.38 ms.
//  * Rows with more than kMaxCand candidate groups (equal codewords: padding,
//    codebooks trained on few distinct values) and rows for which the bound does
//    not hold (huge values) take scan_all, which measures one codeword of each
//    class of equal ones: 0.50 ms for zeros against zeros, 1.56 ms with 16
//    distinct codewords.  Codebooks of nearly equal codewords and values below
//    1e-18 are left: 2.7 ms.
//
// A thread owns a row.  It reads its scores from TMEM once, keeps the minimum
// of every four (half an ALU operation per score with the three-input min),
// then finds the groups within the margin (one packed subtraction per two
// groups and one funnel shift each that collects the sign).  A CTA of 128
// threads works on half a codebook (128 TMEM columns) at a time, so that four
// CTAs share an SM's 512 columns: their decisions cover each other's MMAs.
// The rows being decided wait in shared memory: in registers they made the
// main loop spill (0.75 ms).  The issue slots are the bound (63 % used; tensor pipe 18 %).  Measured,
// 2^20 rows x 16 subspaces: 3.49 ms with every codeword evaluated in float32,
// 0.68 ms now; with whole codebooks (256 columns, two CTAs per SM) 0.80 ms;
// with two passes over the scores and a bit per codeword 1.22 ms.
#include "scan_common.cuh"

namespace ifvs {

namespace {

constexpr int kTile = 128;              // rows per MMA (TMEM lanes), threads per CTA
constexpr int kMaxTiles = 4;            // tiles per CTA: one codebook image serves them
constexpr float kMargin = 0x1p-14f;
constexpr float kFloor = 0x1p-116f;
constexpr float kHuge = 1e28f;          // |x|^2 + max|c|^2 from which the bound does not hold
constexpr float kAbsent = 0x1p100f;     // |c|^2 of a column that can never be a candidate
constexpr int kHalf2 = 128;             // codewords (TMEM columns) per MMA: half a codebook
constexpr int kMaxCand = 8;             // candidate groups per row; more: all codewords

template <int DS>
struct AssignShape {
    static constexpr int NB = (DS + 7) / 8;          // 16-byte chunks (8 bf16) per operand part
    static constexpr int A_CHUNKS = 2 * NB + 1 + (NB & 1 ? 0 : 1);   // xh, xl, ones (, zeros)
    static constexpr int B_CHUNKS = 3 * NB + 1 + (NB & 1 ? 0 : 1);   // ch, ch, cl, |c|^2 (+ a zero chunk: whole K = 16 steps)
    static constexpr int STEPS = B_CHUNKS / 2;
    static constexpr uint32_t A_BYTES = A_CHUNKS * kTile * 16;
    static constexpr uint32_t B_BYTES = B_CHUNKS * 256 * 16;
};

// floats of one float32 codebook slot (halves of 128 codewords): 4 codewords
// and 16 bytes of padding per group, so that the lanes' groups spread over
// the banks
__host__ __device__ constexpr int code_floats(int ds, int K) { return (K > kHalf2 ? 2 : 1) * (kHalf2 * ds + kHalf2); }

// Slots of the float32 codebook: a warp may still compare with subspace
// m - 1 while another stores m + 1, unless a barrier lies between (two halves).
__host__ __device__ constexpr int code_slots(int K) { return K > kHalf2 ? 2 : 3; }

// dynamic shared memory: A, B, the codebook slots, the codes of the CTA's rows and subspaces
template <int DS>
size_t assign_smem_bytes(int K, int tiles, int group) {
    using S = AssignShape<DS>;
    return S::A_BYTES + S::B_BYTES + (size_t)code_slots(K) * code_floats(DS, K) * 4 + (size_t)tiles * kTile * group;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// K-major operand without swizzle: core matrices of 8 rows x 16 bytes, rows
// 16 bytes apart, 8-row groups 128 bytes apart, K chunks `lbo` bytes apart
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t lbo) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(128u >> 4) << 32) |
           (1ull << 46);
}

__device__ __forceinline__ void umma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t addr, float (&v)[16]) {
    uint32_t* r = reinterpret_cast<uint32_t*>(v);
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(addr));
}

// the loaded registers pass through the wait, so that no use of them can be
// moved above it
__device__ __forceinline__ void tmem_wait_ld(float (&v)[16]) {
    uint32_t* r = reinterpret_cast<uint32_t*>(v);
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
                   "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]),
                   "+r"(r[14]), "+r"(r[15])::"memory");
}

__device__ __forceinline__ float min3(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// two floats -> packed bf16 (lo half = a), round to nearest
__device__ __forceinline__ uint32_t bf16x2(float a, float b) {
    uint32_t d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
    return d;
}
__device__ __forceinline__ float bf16_lo(uint32_t p) { return __uint_as_float(p << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t p) { return __uint_as_float(p & 0xFFFF0000u); }

// the two bf16 parts of v[0..7] (zero beyond n)
template <int N>
__device__ __forceinline__ void split8(const float* v, uint4& h, uint4& l) {
    float x[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) x[t] = t < N ? v[t] : 0.f;
    uint32_t hh[4], ll[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        hh[t] = bf16x2(x[2 * t], x[2 * t + 1]);
        ll[t] = bf16x2(x[2 * t] - bf16_lo(hh[t]), x[2 * t + 1] - bf16_hi(hh[t]));
    }
    h = make_uint4(hh[0], hh[1], hh[2], hh[3]);
    l = make_uint4(ll[0], ll[1], ll[2], ll[3]);
}

template <int DS>
__device__ __forceinline__ void load_vec(const float* __restrict__ p, bool vec, float (&x)[DS]) {
    if (vec) {
#pragma unroll
        for (int t = 0; t < DS; t += 4) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(p + t));
            x[t] = v.x;
            x[t + 1] = v.y;
            x[t + 2] = v.z;
            x[t + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int t = 0; t < DS; ++t) x[t] = __ldg(p + t);
    }
}

template <int DS>
__device__ __forceinline__ bool finite_vec(const float (&x)[DS]) {
    bool ok = true;
#pragma unroll
    for (int t = 0; t < DS; ++t) ok &= fabsf(x[t]) < INFINITY;   // false for NaN
    return ok;
}

// the float32 distance, in its defined order
template <int DS>
__device__ __forceinline__ float exact_dist(const float (&x)[DS], const float* c) {
    float s = 0.f;
#pragma unroll
    for (int t = 0; t < DS; t += 4) {
        const float4 v = *reinterpret_cast<const float4*>(c + t);
        const float d0 = __fsub_rn(x[t], v.x), d1 = __fsub_rn(x[t + 1], v.y);
        const float d2 = __fsub_rn(x[t + 2], v.z), d3 = __fsub_rn(x[t + 3], v.w);
        s = __fadd_rn(s, __fmul_rn(d0, d0));
        s = __fadd_rn(s, __fmul_rn(d1, d1));
        s = __fadd_rn(s, __fmul_rn(d2, d2));
        s = __fadd_rn(s, __fmul_rn(d3, d3));
    }
    return s;
}

// Codeword k's column of the operand image, from g = -2 c and n = |c|^2.
template <int DS>
__device__ __forceinline__ void store_column(uint8_t* B, int k, const float (&g)[DS], float n) {
    using S = AssignShape<DS>;
#pragma unroll
    for (int b = 0; b < S::NB; ++b) {
        uint4 h, l;
        split8<(DS < 8 ? DS : 8)>(g + 8 * b, h, l);
        *reinterpret_cast<uint4*>(B + (size_t)(b * 256 + k) * 16) = h;
        *reinterpret_cast<uint4*>(B + (size_t)((S::NB + b) * 256 + k) * 16) = h;
        *reinterpret_cast<uint4*>(B + (size_t)((2 * S::NB + b) * 256 + k) * 16) = l;
    }
    const uint32_t p1 = bf16x2(n, 0.f);   // |c|^2 in three parts
    const float r1 = n - bf16_lo(p1);
    const uint32_t p2 = bf16x2(r1, 0.f);
    const uint32_t p3 = bf16x2(r1 - bf16_lo(p2), 0.f);
    *reinterpret_cast<uint4*>(B + (size_t)(3 * S::NB * 256 + k) * 16) =
        make_uint4((p1 & 0xFFFFu) | (p2 << 16), p3 & 0xFFFFu, 0u, 0u);
    if (S::B_CHUNKS > 3 * S::NB + 1)
        *reinterpret_cast<uint4*>(B + (size_t)((3 * S::NB + 1) * 256 + k) * 16) = make_uint4(0u, 0u, 0u, 0u);
}

// Codewords `tid` and `tid + 128` of one subspace, in registers.
template <int DS>
struct CodeRegs {
    float c[2][DS];
    __device__ __forceinline__ void load(const float* __restrict__ C, int m, int K, int tid, bool vec) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int k = tid + i * kTile;
            if (k < K)
                load_vec<DS>(C + ((int64_t)m * K + k) * DS, vec, c[i]);
            else
#pragma unroll
                for (int t = 0; t < DS; ++t) c[i][t] = 0.f;
        }
    }
    // the float32 codebook, the operand image, and the largest and the smallest
    // |c|^2 (as float bits: order-preserving for values >= 0; the largest +inf
    // when the error bound does not hold for a codeword)
    __device__ __forceinline__ void store(int K, int tid, float* cbf, uint8_t* B, unsigned* cmax,
                                          unsigned* cmin) const {
        unsigned mx = 0u, mn = 0x7F800000u;
        const float nan = __uint_as_float(0x7FC00000u);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int k = tid + i * kTile;
            if (i == 1 && K <= kHalf2) break;   // one half
            float n = 0.f;
            float4* f = reinterpret_cast<float4*>(cbf + k * DS + (k >> 2) * 4);
#pragma unroll
            for (int t = 0; t < DS; t += 4) {
                f[t / 4] = k < K ? make_float4(c[i][t], c[i][t + 1], c[i][t + 2], c[i][t + 3])
                                 : make_float4(nan, nan, nan, nan);   // never nearest
                n += c[i][t] * c[i][t] + c[i][t + 1] * c[i][t + 1];
                n += c[i][t + 2] * c[i][t + 2] + c[i][t + 3] * c[i][t + 3];
            }
            float g[DS];
#pragma unroll
            for (int t = 0; t < DS; ++t) g[t] = -2.f * c[i][t];
            if (k >= K || !(n < kHuge)) {
                // not finite: only the first can be the answer
                const bool absent = k >= K || (k > 0 && !finite_vec<DS>(c[i]));
                if (!absent) mx = 0x7F800000u;
                n = kAbsent;
#pragma unroll
                for (int t = 0; t < DS; ++t) g[t] = 0.f;
            } else {
                mx = max(mx, __float_as_uint(n));
                mn = min(mn, __float_as_uint(n));
            }
            store_column<DS>(B, k, g, n);
        }
        mx = __reduce_max_sync(0xFFFFFFFFu, mx);
        mn = __reduce_min_sync(0xFFFFFFFFu, mn);
        if ((tid & 31) == 0) {
            atomicMax(cmax, mx);
            atomicMin(cmin, mn);
        }
    }
};

// A codebook far from the origin: every score carries the offset, and the margin
// that follows it takes in more groups than kMaxCand in some row of every warp
// from about 20 times the spread.  The smallest |c|^2 is above 3/4 of the largest from 12
// to 15 times (normal data, ds = 8), where a second image costs 0.07 ms of 0.50.
__device__ __forceinline__ bool is_far(unsigned cmax, unsigned cmin, int K) {
    return K > 4 * kMaxCand && cmax < 0x7F800000u && __uint_as_float(cmin) > 0.75f * __uint_as_float(cmax);
}
// The whole CTA calls this: the operand image again, relative to mu, the mean of
// 32 of the codewords, and the largest |c - mu|^2.
template <int DS>
__device__ __noinline__ void recentre(int K, const float* cbf, uint8_t* B, float* mu, unsigned* far_max) {
    const int tid = threadIdx.x;
    if (tid < DS) {
        float s = 0.f;
        for (int i = 0; i < 32; ++i) {
            const int k = i * K / 32;
            const float v = cbf[k * DS + (k >> 2) * 4 + tid];
            s += fabsf(v) < 1e14f ? v : 0.f;
        }
        mu[tid] = s * (1.f / 32.f);
    }
    if (tid == 0) *far_max = 0u;
    __syncthreads();
    unsigned mx = 0u;
#pragma unroll 1
    for (int k = tid; k < K; k += kTile) {
        const float* c = cbf + k * DS + (k >> 2) * 4;
        float g[DS], n = 0.f;
        bool finite = true;
#pragma unroll
        for (int t = 0; t < DS; ++t) {
            const float d = c[t] - mu[t];
            finite &= fabsf(c[t]) < INFINITY;
            n = fmaf(d, d, n);
            g[t] = -2.f * d;
        }
        if (!(n < kHuge)) {
            if (k == 0 || finite) mx = 0x7F800000u;
            n = kAbsent;
#pragma unroll
            for (int t = 0; t < DS; ++t) g[t] = 0.f;
        } else {
            mx = max(mx, __float_as_uint(n));
        }
        store_column<DS>(B, k, g, n);
    }
    mx = __reduce_max_sync(0xFFFFFFFFu, mx);
    if ((tid & 31) == 0) atomicMax(far_max, mx);
}

// The float32 decision over all codewords, for the lanes that ask; the whole
// warp calls it.  While whole classes of equal codewords are met (padding, a
// codebook trained on few distinct values) only the first of each is measured:
// the others lose the tie.  NaN distances as in the definition: the first
// codeword stands until a smaller distance is found, so that a row that is not
// finite (every distance infinite or NaN) needs no other.
template <int DS>
struct Vec {
    float v[DS];
};
// (distance, codeword)
template <int DS>
__device__ __noinline__ float2 scan_all(const Vec<DS> row, const float* cb, int K, bool ask) {
    const int lane = threadIdx.x & 31;
    float x[DS];
#pragma unroll
    for (int t = 0; t < DS; ++t) x[t] = row.v[t];
    float best = exact_dist<DS>(x, cb);
    int bk = 0;
    if (!__any_sync(0xFFFFFFFFu, ask && finite_vec<DS>(x))) return make_float2(best, __int_as_float(0));
    uint32_t left[8];    // bit l of left[j]: codeword 32 j + l
#pragma unroll
    for (int j = 0; j < 8; ++j) left[j] = K >= 32 * j + 32 ? 0xFFFFFFFFu : (K > 32 * j ? (1u << (K - 32 * j)) - 1u : 0u);
    auto measure = [&](int k) {
        const float s = exact_dist<DS>(x, cb + k * DS + (k >> 2) * 4);
        if (s < best) {
            best = s;
            bk = k;
        }
    };
    // a class at a time, while that is cheaper than measuring its members (a
    // round costs about four distances)
    for (int k = 0, gone = 4; gone >= 4;) {
        const float* e = cb + k * DS + (k >> 2) * 4;
        if (k > 0) measure(k);
        gone = 0;
        int next = -1;
#pragma unroll
        for (int j = 7; j >= 0; --j) {
            const int o = 32 * j + lane;
            const float* c = cb + (left[j] >> lane & 1u ? o * DS + (o >> 2) * 4 : 0);
            bool same = true;
#pragma unroll
            for (int t = 0; t < DS; ++t) same &= c[t] == e[t];
            const uint32_t drop = __ballot_sync(0xFFFFFFFFu, same || o == k) & left[j];
            gone += __popc(drop);
            left[j] &= ~drop;
            if (left[j] != 0u) next = 32 * j + __ffs(left[j]) - 1;
        }
        if (next < 0) break;
        k = next;
    }
#pragma unroll 1
    for (int j = 0; j < 8; ++j) {
        uint32_t w = left[0];
#pragma unroll
        for (int i = 1; i < 8; ++i) w = j == i ? left[i] : w;
        for (; w != 0u; w &= w - 1u) measure(32 * j + __ffs(w) - 1);
    }
    return make_float2(best, __int_as_float(bk));
}

}  // namespace

// CTA (row chunk of `tiles` x 128 rows, group of `group` subspaces).  Codes
// and distances [n][M], or [M][n] (BY_SUBSPACE).
template <int DS, bool BY_SUBSPACE>
__global__ void __launch_bounds__(kTile, DS > 8 ? 2 : 4)
k_pq_assign_mma(const float* __restrict__ X, int64_t n, int D, int M, int K, const float* __restrict__ C, int tiles,
                int group, int vec, uint8_t* __restrict__ codes, float* __restrict__ dmin) {
    using S = AssignShape<DS>;
    extern __shared__ __align__(1024) uint8_t sm[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tmem_base;
    __shared__ unsigned cmax[3], cmin[3];   // slots as the float32 codebooks
    __shared__ float mu[DS];                // of a subspace far from the origin
    __shared__ unsigned far_max;
    __shared__ float4 xs[DS / 4][kTile];    // the rows being decided
    const int nslots = code_slots(K);
    uint8_t* A = sm;
    uint8_t* B = sm + S::A_BYTES;
    float* cbf = reinterpret_cast<float*>(B + S::B_BYTES);
    uint8_t* out = B + S::B_BYTES + nslots * code_floats(DS, K) * 4;   // [tiles * 128][group]
    const int tid = threadIdx.x, warp = tid >> 5;
    const int64_t row0 = (int64_t)blockIdx.x * tiles * kTile;
    const int m0 = blockIdx.y * group;
    const int g = min(group, M - m0);
    const int nt = (int)min((int64_t)tiles, (n - row0 + kTile - 1) / kTile);
    const int halves = K > kHalf2 ? 2 : 1;
    // instruction: D float32, A and B bf16, both K-major, N = 128, M = 128
    constexpr uint32_t idesc =
        (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kHalf2 >> 3) << 17) | ((128u >> 4) << 24);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 128;" ::"r"(smem_u32(&tmem_base))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        mbar_init(smem_u32(&bar), 1u);
        fence_mbar_init();
        cmax[0] = cmax[1] = cmax[2] = 0u;
        cmin[0] = cmin[1] = cmin[2] = 0x7F800000u;
    }
    // the constant chunks of A: ones against the parts of |c|^2, zeros
    *reinterpret_cast<uint4*>(A + (size_t)(2 * S::NB * kTile + tid) * 16) =
        make_uint4(0x3F803F80u, 0x00003F80u, 0u, 0u);
    if (S::A_CHUNKS > 2 * S::NB + 1)
        *reinterpret_cast<uint4*>(A + (size_t)((2 * S::NB + 1) * kTile + tid) * 16) = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();

    CodeRegs<DS> cr;
    float x1[DS];   // the next tile's row (loading)
    // the rows run ahead of the tile being decided: tile xt of subspace xm is next
    const int rows = (int)min((int64_t)tiles * kTile, n - row0);
    int xm = 0, xt = 0;
    auto load_x = [&](float (&v)[DS]) {
        const int r = xt * kTile + tid;
        if (r < rows)
            load_vec<DS>(X + (row0 + r) * D + (m0 + xm) * DS, vec != 0, v);
        else
#pragma unroll
            for (int t = 0; t < DS; ++t) v[t] = 0.f;
        if (++xt == nt) {
            xt = 0;
            ++xm;
        }
    };
    auto store_a = [&](const float (&u)[DS], bool centred) {
        float v[DS];
#pragma unroll
        for (int t = 0; t < DS; ++t) v[t] = u[t];
        if (centred)
#pragma unroll
            for (int t = 0; t < DS; ++t) v[t] -= mu[t];
#pragma unroll
        for (int b = 0; b < S::NB; ++b) {
            uint4 h, l;
            split8<(DS < 8 ? DS : 8)>(v + 8 * b, h, l);
            *reinterpret_cast<uint4*>(A + (size_t)(b * kTile + tid) * 16) = h;
            *reinterpret_cast<uint4*>(A + (size_t)((S::NB + b) * kTile + tid) * 16) = l;
        }
    };
    // the row becomes this tile's; its squared norm (relative to the centre)
    auto keep = [&](const float (&v)[DS], bool centred) -> float {
        float s = 0.f;
#pragma unroll
        for (int t = 0; t < DS; t += 4) xs[t / 4][tid] = make_float4(v[t], v[t + 1], v[t + 2], v[t + 3]);
        if (centred) {
#pragma unroll
            for (int t = 0; t < DS; ++t) s = fmaf(v[t] - mu[t], v[t] - mu[t], s);
        } else {
#pragma unroll
            for (int t = 0; t < DS; ++t) s = fmaf(v[t], v[t], s);
        }
        return s;
    };
    // A's chunk of K chunk j of B: (ch, xh), (ch, xl), (cl, xh), (|c|^2, ones), (0, zeros)
    auto a_chunk = [](int j) { return j < 2 * S::NB ? j : (j < 3 * S::NB ? j - 2 * S::NB : j - S::NB); };
    auto issue = [&](int half) {   // one thread
        const uint32_t a = smem_u32(A), b = smem_u32(B) + (uint32_t)half * kHalf2 * 16;
#pragma unroll
        for (int st = 0; st < S::STEPS; ++st) {
            const int c0 = a_chunk(2 * st), c1 = a_chunk(2 * st + 1);
            umma_bf16(tmem_base, umma_desc(a + (uint32_t)c0 * kTile * 16, (uint32_t)(c1 - c0) * kTile * 16),
                      umma_desc(b + (uint32_t)(2 * st) * 256 * 16, 256 * 16), idesc, st > 0 ? 1u : 0u);
        }
        umma_commit(smem_u32(&bar));
    };

    const int iters = g * nt;
    cr.load(C, m0, K, tid, vec != 0);
    load_x(x1);
    cr.store(K, tid, cbf, B, &cmax[0], &cmin[0]);
    store_a(x1, false);
    fence_proxy_async_smem();
    __syncthreads();
    bool far = is_far(cmax[0], cmin[0], K);
    if (far) {   // the same in every thread
        recentre<DS>(K, cbf, B, mu, &far_max);
        store_a(x1, true);
        fence_proxy_async_smem();
        __syncthreads();
    }
    float nx = keep(x1, far);
    if (iters > 1) load_x(x1);
    const uint32_t tm = tmem_base + ((uint32_t)(warp * 32) << 16);
    if (tid == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        issue(0);
    }
    // mma_ok false, late = 0 or 1: the bounded wait for an MMA (of that
    // barrier parity) ran out; its rows and all later ones are scanned exactly
    bool mma_ok = true;
    int late = -1;
    uint32_t phase = 0u;
    int mi = 0, ti = 0, slot = 0;   // subspace and tile of iteration it; the subspace's codebook slot
#pragma unroll 1
    for (int it = 0; it < iters; ++it) {
        const bool more = it + 1 < iters;
        const bool new_m = more && ti + 1 == nt;
        const float span = nx + __uint_as_float(far ? far_max : cmax[slot]);
        const float margin = kMargin * span + kFloor;
        bool all = !(span < kHuge);
        const int next = new_m ? (slot + 1 == nslots ? 0 : slot + 1) : slot;
        bool next_far = far;
        // per half: the smallest score and the groups within the margin of
        // it (bit j: group j of the half)
        uint32_t mask[2] = {0u, 0u};
        float low[2] = {0x1p120f, 0x1p120f};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (h >= halves) break;
            float gm[32];
            if (mma_ok) mma_ok = mbar_wait_warp(smem_u32(&bar), phase);
            if (mma_ok) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // the smallest score of every 4 codewords
                float vv[2][16];
                tmem_ld16(tm, vv[0]);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    float(&v)[16] = vv[i & 1];
                    tmem_wait_ld(v);
                    if (i < 7) tmem_ld16(tm + 16 * (i + 1), vv[(i + 1) & 1]);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        gm[4 * i + j] = fminf(min3(v[4 * j], v[4 * j + 1], v[4 * j + 2]), v[4 * j + 3]);
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            }
            const bool read = mma_ok;
            // the next MMA: the other half, or the next tile, whose operands
            // replace this one's now that its MMAs are done
            const bool last = h + 1 == halves;
            if (last && more) {
                store_a(x1, far && !new_m);
                if (new_m) {
                    cr.load(C, m0 + mi + 1, K, tid, vec != 0);
                    cr.store(K, tid, cbf + next * code_floats(DS, K), B, &cmax[next], &cmin[next]);
                }
                fence_proxy_async_smem();
            }
            if (__syncthreads_or(mma_ok ? 0 : 1) != 0 && late < 0) late = (int)phase;
            mma_ok = late < 0;
            phase ^= 1u;
            // a subspace far from the origin starts when this tile is decided
            if (last && new_m) next_far = is_far(cmax[next], cmin[next], K);
            if (mma_ok && (!last || (more && !(new_m && next_far))) && tid == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                issue(last ? 0 : 1);
            }
            if (read) {
                float lo[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) lo[i] = fminf(gm[i], gm[i + 4]);
#pragma unroll
                for (int j = 8; j < 32; j += 8)
#pragma unroll
                    for (int i = 0; i < 4; ++i) lo[i] = min3(lo[i], gm[j + i], gm[j + i + 4]);
                low[h] = fminf(fminf(lo[0], lo[1]), fminf(lo[2], lo[3]));
                const float thr = low[h] + margin;
                const uint64_t nthr = add_f32x2(0ull, -thr, -thr);
                // the signs of (score - thr), eight per chain of funnel shifts
                uint32_t w[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) w[i] = 0u;
#pragma unroll
                for (int j = 6; j >= 0; j -= 2)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float a, b;
                        unpack_f32x2(add_f32x2(nthr, gm[8 * i + j], gm[8 * i + j + 1]), a, b);
                        w[i] = __funnelshift_l(__float_as_uint(b), w[i], 1);
                        w[i] = __funnelshift_l(__float_as_uint(a), w[i], 1);
                    }
                mask[h] = w[0] | w[1] << 8 | w[2] << 16 | w[3] << 24;
            }
        }
        // a half whose smallest score is beyond the other's margin has no candidate
        if (low[1] > low[0] + margin) mask[1] = 0u;
        if (low[0] > low[1] + margin) mask[0] = 0u;
        const int cnt = __popc(mask[0]) + __popc(mask[1]);
        all = all || cnt == 0 || cnt > kMaxCand || (late >= 0);
        const float* cb = cbf + slot * code_floats(DS, K);
        float best = INFINITY;
        int bk = 0;
        float x[DS];
#pragma unroll
        for (int t = 0; t < DS; t += 4) {
            const float4 v = xs[t / 4][tid];
            x[t] = v.x;
            x[t + 1] = v.y;
            x[t + 2] = v.z;
            x[t + 3] = v.w;
        }
        if (__any_sync(0xFFFFFFFFu, all)) {
            Vec<DS> row;
#pragma unroll
            for (int t = 0; t < DS; ++t) row.v[t] = x[t];
            const float2 r = scan_all<DS>(row, cb, K, all);
            if (all) {
                mask[0] = mask[1] = 0u;
                best = r.x;
                bk = __float_as_int(r.y);
            }
        }
        // the float32 decision over the candidate groups, codewords
        // ascending; their distances are finite, those of columns beyond K NaN
#pragma unroll 1
        while ((mask[0] | mask[1]) != 0u) {
            int g4;
            if (mask[0] != 0u) {
                g4 = __ffs(mask[0]) - 1;
                mask[0] &= mask[0] - 1u;
            } else {
                g4 = 31 + __ffs(mask[1]);
                mask[1] &= mask[1] - 1u;
            }
            const float* c = cb + g4 * (4 * DS + 4);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float s = exact_dist<DS>(x, c + j * DS);
                if (s < best) {
                    best = s;
                    bk = 4 * g4 + j;
                }
            }
        }
        const int lr = ti * kTile + tid;
        out[BY_SUBSPACE ? mi * (nt * kTile) + lr : lr * g + mi] = (uint8_t)bk;
        if (dmin != nullptr && lr < rows)
            dmin[BY_SUBSPACE ? (m0 + mi) * n + row0 + lr : (row0 + lr) * M + m0 + mi] = best;
        if (new_m && tid == 0) {   // its last readers passed the barrier above
            cmax[slot] = 0u;
            cmin[slot] = 0x7F800000u;
        }
        far = next_far;
        if (new_m && far) {   // mu and far_max: their last readers are past the barrier above
            recentre<DS>(K, cbf + next * code_floats(DS, K), B, mu, &far_max);
            store_a(x1, true);
            fence_proxy_async_smem();
            __syncthreads();
            if (mma_ok && tid == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                issue(0);
            }
        }
        if (more) nx = keep(x1, far);
        if (it + 2 < iters) load_x(x1);
        if (++ti == nt) {
            ti = 0;
            ++mi;
            slot = slot + 1 == nslots ? 0 : slot + 1;
        }
    }
    __syncthreads();
    if (late >= 0) {   // that MMA may still be in flight: wait again (bounded) before TMEM is freed
        mbar_wait_warp(smem_u32(&bar), (uint32_t)late);
        __syncthreads();
    }
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 128;" ::"r"(tmem_base));
    if (BY_SUBSPACE) {
        for (int j = 0; j < g; ++j)
            for (int r = tid; r < rows; r += kTile)
                codes[(m0 + j) * n + row0 + r] = out[j * nt * kTile + r];
    } else {
        for (int e = tid; e < rows * g; e += kTile) {
            const int r = e / g;
            codes[(row0 + r) * M + m0 + (e - r * g)] = out[e];
        }
    }
}

// any ds: one thread per row, the codebook of one subspace in shared memory
constexpr int kPqThreads = 256;
__global__ void __launch_bounds__(kPqThreads) k_pq_assign_any(const float* __restrict__ X, int64_t n,
                                                              int D, int M, int K, int ds,
                                                              const float* __restrict__ C, int64_t row_stride,
                                                              int64_t sub_stride, uint8_t* __restrict__ codes,
                                                              float* __restrict__ dmin) {
    extern __shared__ __align__(16) float cb[];
    const int64_t i = (int64_t)blockIdx.x * kPqThreads + threadIdx.x;
    for (int m = 0; m < M; ++m) {
        __syncthreads();
        for (int e = threadIdx.x; e < K * ds; e += kPqThreads) cb[e] = C[(int64_t)m * K * ds + e];
        __syncthreads();
        if (i >= n) continue;
        const float* x = X + i * D + m * ds;
        float best = 0.f;
        int bk = 0;
        for (int k = 0; k < K; ++k) {
            float s = 0.f;
            for (int t = 0; t < ds; ++t) {
                const float d = __fsub_rn(__ldg(x + t), cb[k * ds + t]);
                s = __fadd_rn(s, __fmul_rn(d, d));
            }
            if (k == 0 || s < best) {
                best = s;
                bk = k;
            }
        }
        const int64_t at = i * row_stride + m * sub_stride;
        codes[at] = (uint8_t)bk;
        if (dmin != nullptr) dmin[at] = best;
    }
}

template <int DS>
static cudaError_t launch_assign_mma(const float* X, int64_t n, int D, int M, int K, const float* C, uint8_t* codes,
                                     float* dmin, bool by_subspace, cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    // Tiles per CTA share one codebook image (worth about a fourth of a tile);
    // fewer, and the subspaces split over CTAs, where the rows alone would
    // leave the resident CTAs without four waves of work.
    const int64_t want = (int64_t)sms * (DS > 8 ? 2 : 4) * 4;
    const int64_t all = (n + kTile - 1) / kTile;
    int tiles = (int)(all / want);
    tiles = tiles < 1 ? 1 : (tiles > kMaxTiles ? kMaxTiles : tiles);
    const int64_t chunks = (all + tiles - 1) / tiles;
    int64_t groups = (want + chunks - 1) / chunks;
    if (groups > M) groups = M;
    int group = (int)((M + groups - 1) / groups);
    if (group > (DS > 8 ? 8 : 32)) group = DS > 8 ? 8 : 32;   // two CTAs' shared memory per SM
    if ((M + group - 1) / group > 65535) group = (M + 65534) / 65535;   // the grid's second dimension
    groups = (M + group - 1) / group;
    const bool vec = ((uintptr_t)X | (uintptr_t)C) % 16 == 0;   // ds is a multiple of 4: so are D and every offset
    const size_t smem = assign_smem_bytes<DS>(K, tiles, group);
    auto kern = by_subspace ? k_pq_assign_mma<DS, true> : k_pq_assign_mma<DS, false>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3((unsigned)chunks, (unsigned)groups), kTile, smem, s>>>(X, n, D, M, K, C, tiles, group, vec ? 1 : 0,
                                                                       codes, dmin);
    return cudaGetLastError();
}

cudaError_t launch_pq_assign(const float* X, int64_t n, int D, int M, int K, const float* C,
                             uint8_t* codes, float* dmin, bool by_subspace, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int ds = D / M;
    const int64_t rs = by_subspace ? 1 : M, ss = by_subspace ? n : 1;
    if (ds == 4) return launch_assign_mma<4>(X, n, D, M, K, C, codes, dmin, by_subspace, s);
    if (ds == 8) return launch_assign_mma<8>(X, n, D, M, K, C, codes, dmin, by_subspace, s);
    if (ds == 16) return launch_assign_mma<16>(X, n, D, M, K, C, codes, dmin, by_subspace, s);
    const size_t smem = (size_t)K * ds * sizeof(float);
    const int64_t blocks = (n + kPqThreads - 1) / kPqThreads;
    cudaError_t e = cudaFuncSetAttribute(k_pq_assign_any, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_pq_assign_any<<<(unsigned)blocks, kPqThreads, smem, s>>>(X, n, D, M, K, ds, C, rs, ss, codes, dmin);
    return cudaGetLastError();
}

}  // namespace ifvs
