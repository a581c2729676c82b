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
// 2 (1.2e-5 + 1.2e-5 + 2.4e-6) (|x|^2 + max|c|^2) of the smallest score, and
// every codeword within kMargin = 2^-13 (1.2e-4) of it is a candidate: one
// for almost every row (data whose offset from the origin is ~30 times its
// spread would see several), and several are compared exactly, smallest
// first.  Rows for which the bound does not hold (non-finite or huge values,
// all values below 1e-12) and rows with more than kMaxCand candidates scan
// all codewords exactly.
//
// A thread owns a row.  Two passes over its 256 scores in TMEM: the minimum
// (three-input min: half an ALU operation per score), then a bit per score
// within the margin (half a packed subtraction and one funnel shift that
// collects the sign).  The ALU pipe is the bound: 1.5 operations per score at
// 64 lanes per SM and cycle.  A CTA of 128 threads holds 256 TMEM columns,
// two CTAs share an SM: one's epilogue covers the other's MMA, whose operands
// for the next tile are prepared while the current tile's MMA runs.
#include "scan_common.cuh"

namespace ifvs {

namespace {

constexpr int kTile = 128;              // rows per MMA (TMEM lanes), threads per CTA
constexpr int kMaxTiles = 4;            // tiles per CTA: one codebook image serves them
constexpr float kMargin = 0x1p-13f;
constexpr int kMaxCand = 16;

template <int DS>
struct AssignShape {
    static constexpr int NB = (DS + 7) / 8;          // 16-byte chunks (8 bf16) per operand part
    static constexpr int A_CHUNKS = 2 * NB + 2;      // xh, xl, ones, zeros
    static constexpr int B_CHUNKS = 3 * NB + 1 + (NB & 1 ? 0 : 1);   // ch, ch, cl, |c|^2 (+ a zero chunk: whole K = 16 steps)
    static constexpr int STEPS = B_CHUNKS / 2;
    static constexpr uint32_t A_BYTES = A_CHUNKS * kTile * 16;
    static constexpr uint32_t B_BYTES = B_CHUNKS * 256 * 16;
    static constexpr uint32_t C_BYTES = 256 * DS * 4;
};

// dynamic shared memory: A (two buffers), B, codebook in float32 (three
// slots: a warp may still compare with subspace m - 1 while another, one
// barrier ahead, stores m + 1), codes of the CTA's rows and subspaces
template <int DS>
size_t assign_smem_bytes(int tiles, int group) {
    using S = AssignShape<DS>;
    return 2 * S::A_BYTES + S::B_BYTES + 3 * S::C_BYTES + (size_t)tiles * kTile * group;
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

__device__ __forceinline__ void tmem_ld32(uint32_t addr, float (&v)[32]) {
    uint32_t* r = reinterpret_cast<uint32_t*>(v);
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(addr));
}

// the loaded registers pass through the wait, so that no use of them can be
// moved above it
__device__ __forceinline__ void tmem_wait_ld(float (&v)[32]) {
    uint32_t* r = reinterpret_cast<uint32_t*>(v);
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                   "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                   "+r"(r[29]), "+r"(r[30]), "+r"(r[31])::"memory");
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

// the first set bit of mask[0..8) (bit j of word w: codeword 32 w + j), cleared; -1 when none is set
__device__ __forceinline__ int take_first(uint32_t (&mask)[8]) {
    int w = -1;
    uint32_t v = 0u;
#pragma unroll
    for (int i = 7; i >= 0; --i)
        if (mask[i] != 0u) {
            w = i;
            v = mask[i];
        }
    if (w < 0) return -1;
    const int j = __ffs(v) - 1;
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (i == w) mask[i] = v & (v - 1u);
    return 32 * w + j;
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
    // the float32 codebook, the operand image, and the largest |c|^2 (as
    // float bits: order-preserving for values >= 0; +inf when a codeword is
    // not finite or too large for the error bound)
    __device__ __forceinline__ void store(int K, int tid, float* cbf, uint8_t* B, unsigned* cmax) const {
        using S = AssignShape<DS>;
        unsigned mx = 0u;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int k = tid + i * kTile;
            float n = 0.f;
#pragma unroll
            for (int t = 0; t < DS; ++t) {
                cbf[k * DS + t] = c[i][t];
                n += c[i][t] * c[i][t];
            }
            if (k < K) mx = max(mx, n < 1e28f ? __float_as_uint(n) : 0x7F800000u);
            float g[DS];
#pragma unroll
            for (int t = 0; t < DS; ++t) g[t] = -2.f * c[i][t];
#pragma unroll
            for (int b = 0; b < S::NB; ++b) {
                uint4 h, l;
                split8<(DS < 8 ? DS : 8)>(g + 8 * b, h, l);
                *reinterpret_cast<uint4*>(B + (size_t)(b * 256 + k) * 16) = h;
                *reinterpret_cast<uint4*>(B + (size_t)((S::NB + b) * 256 + k) * 16) = h;
                *reinterpret_cast<uint4*>(B + (size_t)((2 * S::NB + b) * 256 + k) * 16) = l;
            }
            // |c|^2 in three parts; columns beyond K can never be candidates
            const float nn = k < K ? n : 0x1p100f;
            const uint32_t p1 = bf16x2(nn, 0.f);
            const float r1 = nn - bf16_lo(p1);
            const uint32_t p2 = bf16x2(r1, 0.f);
            const uint32_t p3 = bf16x2(r1 - bf16_lo(p2), 0.f);
            *reinterpret_cast<uint4*>(B + (size_t)(3 * S::NB * 256 + k) * 16) =
                make_uint4((p1 & 0xFFFFu) | (p2 << 16), p3 & 0xFFFFu, 0u, 0u);
            if (S::B_CHUNKS > 3 * S::NB + 1)
                *reinterpret_cast<uint4*>(B + (size_t)((3 * S::NB + 1) * 256 + k) * 16) = make_uint4(0u, 0u, 0u, 0u);
        }
        mx = __reduce_max_sync(0xFFFFFFFFu, mx);
        if ((tid & 31) == 0) atomicMax(cmax, mx);
    }
};

}  // namespace

// CTA (row chunk of `tiles` x 128 rows, group of `group` subspaces).
template <int DS>
__global__ void __launch_bounds__(kTile, 2) k_pq_assign_mma(const float* __restrict__ X, int64_t n, int D, int M, int K,
                                                         const float* __restrict__ C, int tiles, int group, int vec,
                                                         uint8_t* __restrict__ codes, float* __restrict__ dmin) {
    using S = AssignShape<DS>;
    extern __shared__ __align__(1024) uint8_t sm[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tmem_base;
    __shared__ unsigned cmax[3];   // slots as the float32 codebooks
    uint8_t* A = sm;
    uint8_t* B = sm + 2 * S::A_BYTES;
    float* cbf = reinterpret_cast<float*>(B + S::B_BYTES);
    uint8_t* out = B + S::B_BYTES + 3 * S::C_BYTES;      // [tiles * 128][group]
    const int tid = threadIdx.x, warp = tid >> 5;
    const int64_t row0 = (int64_t)blockIdx.x * tiles * kTile;
    const int m0 = blockIdx.y * group;
    const int g = min(group, M - m0);
    const int nt = (int)min((int64_t)tiles, (n - row0 + kTile - 1) / kTile);
    const int ncol = (K + 31) & ~31;                      // columns read back
    // instruction: D float32, A and B bf16, both K-major, N = 256, M = 128
    constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((256u >> 3) << 17) | ((128u >> 4) << 24);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(smem_u32(&tmem_base))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        mbar_init(smem_u32(&bar), 1u);
        fence_mbar_init();
        cmax[0] = cmax[1] = cmax[2] = 0u;
    }
    // the constant chunks of both A buffers: ones against the parts of |c|^2, zeros
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        uint8_t* a = A + b * S::A_BYTES;
        *reinterpret_cast<uint4*>(a + (size_t)(2 * S::NB * kTile + tid) * 16) =
            make_uint4(0x3F803F80u, 0x00003F80u, 0u, 0u);
        *reinterpret_cast<uint4*>(a + (size_t)((2 * S::NB + 1) * kTile + tid) * 16) = make_uint4(0u, 0u, 0u, 0u);
    }
    __syncthreads();

    CodeRegs<DS> cr;
    float x[DS], x1[DS], x2[DS];   // this tile's row, the next one's, the one after that (loading)
    auto load_x = [&](int it, float (&v)[DS]) {
        const int m = m0 + it / nt;
        const int64_t r = row0 + (int64_t)(it % nt) * kTile + tid;
        if (r < n)
            load_vec<DS>(X + r * D + m * DS, vec != 0, v);
        else
#pragma unroll
            for (int t = 0; t < DS; ++t) v[t] = 0.f;
    };
    auto store_a = [&](int it, const float (&v)[DS]) {
        uint8_t* a = A + (it & 1) * S::A_BYTES;
#pragma unroll
        for (int b = 0; b < S::NB; ++b) {
            uint4 h, l;
            split8<(DS < 8 ? DS : 8)>(v + 8 * b, h, l);
            *reinterpret_cast<uint4*>(a + (size_t)(b * kTile + tid) * 16) = h;
            *reinterpret_cast<uint4*>(a + (size_t)((S::NB + b) * kTile + tid) * 16) = l;
        }
    };
    // A's chunk of K chunk j of B: (ch, xh), (ch, xl), (cl, xh), (|c|^2, ones), (0, zeros)
    auto a_chunk = [](int j) { return j < 2 * S::NB ? j : (j < 3 * S::NB ? j - 2 * S::NB : j - S::NB); };
    auto issue = [&](int it) {   // one thread
        const uint32_t a = smem_u32(A + (it & 1) * S::A_BYTES), b = smem_u32(B);
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
    load_x(0, x);
    if (iters > 1) load_x(1, x1);
    cr.store(K, tid, cbf, B, &cmax[0]);
    store_a(0, x);
    if (g > 1) cr.load(C, m0 + 1, K, tid, vec != 0);
    fence_proxy_async_smem();
    __syncthreads();
    const uint32_t tm = tmem_base + ((uint32_t)(warp * 32) << 16);
    if (tid == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        issue(0);
    }
    // mma_ok false, late >= 0: the bounded wait for tile `late`'s MMA ran out;
    // its rows and all later ones are scanned exactly
    bool mma_ok = true;
    int late = -1;
#pragma unroll 1
    for (int it = 0; it < iters; ++it) {
        const int mi = it / nt;
        const bool more = it + 1 < iters;
        const bool new_m = more && (it + 1) / nt != mi;
        if (it + 2 < iters) load_x(it + 2, x2);
        if (more) store_a(it + 1, x1);
        float nx = 0.f;
#pragma unroll
        for (int t = 0; t < DS; ++t) nx = fmaf(x[t], x[t], nx);
        const float span = nx + __uint_as_float(cmax[mi % 3]);
        bool all = !(span > 1e-24f && span < 1e28f);
        uint32_t mask[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) mask[i] = 0u;
        if (mma_ok) mma_ok = mbar_wait_warp(smem_u32(&bar), (uint32_t)it & 1u);
        if (mma_ok) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // both passes read 32 columns ahead
            float lo = 0x1p120f;
            float vv[2][32];
            tmem_ld32(tm, vv[0]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (32 * i >= ncol) break;
                float(&v)[32] = vv[i & 1];
                tmem_wait_ld(v);
                if (32 * (i + 1) < ncol) tmem_ld32(tm + 32 * (i + 1), vv[(i + 1) & 1]);
                float p = min3(v[0], v[1], v[2]), q = min3(v[3], v[4], v[5]);
#pragma unroll
                for (int j = 6; j < 30; j += 4) {
                    p = min3(p, v[j], v[j + 1]);
                    q = min3(q, v[j + 2], v[j + 3]);
                }
                lo = min3(lo, min3(p, v[30], v[31]), q);
            }
            const float thr = lo + kMargin * span;
            const uint64_t nthr = add_f32x2(0ull, -thr, -thr);
            tmem_ld32(tm, vv[0]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (32 * i >= ncol) break;
                float(&v)[32] = vv[i & 1];
                tmem_wait_ld(v);
                if (32 * (i + 1) < ncol) tmem_ld32(tm + 32 * (i + 1), vv[(i + 1) & 1]);
                uint32_t w = 0u;
#pragma unroll
                for (int j = 30; j >= 0; j -= 2) {
                    float a, b;
                    unpack_f32x2(add_f32x2(nthr, v[j], v[j + 1]), a, b);
                    w = __funnelshift_l(__float_as_uint(b), w, 1);
                    w = __funnelshift_l(__float_as_uint(a), w, 1);
                }
                mask[i] = w;
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        }
        const bool mma_was_ok = mma_ok;
        // the next tile's MMA: its operands are in place, this tile's scores are read
        if (new_m) {
            cr.store(K, tid, cbf + ((mi + 1) % 3) * (256 * DS), B, &cmax[(mi + 1) % 3]);
            if (mi + 2 < g) cr.load(C, m0 + mi + 2, K, tid, vec != 0);
        }
        fence_proxy_async_smem();
        if (__syncthreads_or(mma_ok ? 0 : 1) != 0 && late < 0) late = it;
        mma_ok = late < 0;
        if (mma_ok && more && tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            issue(it + 1);
        }
        // the decision
        int cnt = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) cnt += __popc(mask[i]);
        all = all || !mma_was_ok || cnt == 0 || cnt > kMaxCand;
        const float* cb = cbf + (mi % 3) * (256 * DS);
        float best = 0.f;
        int bk = 0;
        if (!all) {
            bk = take_first(mask);
            if (cnt > 1 || dmin != nullptr) best = exact_dist<DS>(x, cb + bk * DS);
            for (int left = cnt - 1; left > 0; --left) {
                const int k = take_first(mask);
                const float s = exact_dist<DS>(x, cb + k * DS);
                if (s < best) {
                    best = s;
                    bk = k;
                }
            }
        } else {
            best = exact_dist<DS>(x, cb);
#pragma unroll 1
            for (int k = 1; k < K; ++k) {
                const float s = exact_dist<DS>(x, cb + k * DS);
                if (s < best) {
                    best = s;
                    bk = k;
                }
            }
        }
        const int lr = (it % nt) * kTile + tid;
        out[lr * g + mi] = (uint8_t)bk;
        if (dmin != nullptr && row0 + lr < n) dmin[(row0 + lr) * M + m0 + mi] = best;
        if (new_m && tid == 0) cmax[mi % 3] = 0u;   // its last readers passed the barrier above
#pragma unroll
        for (int t = 0; t < DS; ++t) {
            x[t] = x1[t];
            x1[t] = x2[t];
        }
    }
    __syncthreads();
    if (late >= 0) {   // that MMA may still be in flight: wait again (bounded) before TMEM is freed
        mbar_wait_warp(smem_u32(&bar), (uint32_t)late & 1u);
        __syncthreads();
    }
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem_base));
    const int64_t rows = min((int64_t)nt * kTile, n - row0);
    for (int e = tid; e < (int)rows * g; e += kTile) {
        const int r = e / g;
        codes[(row0 + r) * M + m0 + (e - r * g)] = out[e];
    }
}

// any ds: one thread per row, the codebook of one subspace in shared memory
constexpr int kPqThreads = 256;
__global__ void __launch_bounds__(kPqThreads) k_pq_assign_any(const float* __restrict__ X, int64_t n,
                                                              int D, int M, int K, int ds,
                                                              const float* __restrict__ C,
                                                              uint8_t* __restrict__ codes,
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
        codes[i * M + m] = (uint8_t)bk;
        if (dmin != nullptr) dmin[i * M + m] = best;
    }
}

template <int DS>
static cudaError_t launch_assign_mma(const float* X, int64_t n, int D, int M, int K, const float* C, uint8_t* codes,
                                     float* dmin, cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    // Tiles per CTA share one codebook image (worth about a fifth of a tile);
    // fewer, and the subspaces split over CTAs, where the rows alone would
    // leave the two CTAs per SM without four waves of work.
    const int64_t want = (int64_t)sms * 2 * 4;
    const int64_t all = (n + kTile - 1) / kTile;
    int tiles = (int)(all / want);
    tiles = tiles < 1 ? 1 : (tiles > kMaxTiles ? kMaxTiles : tiles);
    const int64_t chunks = (all + tiles - 1) / tiles;
    int64_t groups = (want + chunks - 1) / chunks;
    if (groups > M) groups = M;
    int group = (int)((M + groups - 1) / groups);
    if (group > (DS > 8 ? 16 : 32)) group = DS > 8 ? 16 : 32;   // two CTAs' shared memory per SM
    groups = (M + group - 1) / group;
    const bool vec = ((uintptr_t)X | (uintptr_t)C) % 16 == 0;   // ds is a multiple of 4: so are D and every offset
    const size_t smem = assign_smem_bytes<DS>(tiles, group);
    e = cudaFuncSetAttribute(k_pq_assign_mma<DS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_pq_assign_mma<DS><<<dim3((unsigned)chunks, (unsigned)groups), kTile, smem, s>>>(X, n, D, M, K, C, tiles, group,
                                                                                    vec ? 1 : 0, codes, dmin);
    return cudaGetLastError();
}

cudaError_t launch_pq_assign(const float* X, int64_t n, int D, int M, int K, const float* C,
                             uint8_t* codes, float* dmin, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int ds = D / M;
    if (ds == 4) return launch_assign_mma<4>(X, n, D, M, K, C, codes, dmin, s);
    if (ds == 8) return launch_assign_mma<8>(X, n, D, M, K, C, codes, dmin, s);
    if (ds == 16) return launch_assign_mma<16>(X, n, D, M, K, C, codes, dmin, s);
    const size_t smem = (size_t)K * ds * sizeof(float);
    const int64_t blocks = (n + kPqThreads - 1) / kPqThreads;
    cudaError_t e = cudaFuncSetAttribute(k_pq_assign_any, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_pq_assign_any<<<(unsigned)blocks, kPqThreads, smem, s>>>(X, n, D, M, K, ds, C, codes, dmin);
    return cudaGetLastError();
}

}  // namespace ifvs
