// Stage 1 of §2 (Filter): every row's attribute values are tested against
// the query's predicate (the conjunctive form of Listing 1), giving the
// candidate pool P as a pass bitmap.
//
// One warp owns one 1024-row block: lane l holds the 32 attribute values of
// rows b*1024 + 32*j + l (j = 0..31), loaded with 32 coalesced 128-byte
// column reads, and then evaluates every query of its group against them,
// so the columns are read once per query group.  The lane's 32 pass bits
// form its word of the lane-major bitmap directly (no ballot needed), one
// 128-byte store per warp and query.  Popcounts go through a warp reduction
// into npass.
#include "internal.cuh"

namespace ifvs {

// Fail bits of 8 rows against one interval, shifted into `fail` (row j0 + 7
// first, so that after four calls bit j is row j).  For each row:
// off = v - lo (mod 2^32); the carry out of off + ~wm1 is 1 exactly when
// off > wm1, i.e. when the row fails; addc shifts the carry in.  The carry
// never leaves the asm block.
__device__ __forceinline__ uint32_t fail8(uint32_t fail, const int32_t* v, int32_t lo, uint32_t nwm1) {
    asm("{\n\t.reg .u32 t;\n\t"
        "sub.u32 t, %8, %9;\n\tadd.cc.u32 t, t, %10;\n\taddc.u32 %0, %0, %0;\n\t"
        "sub.u32 t, %7, %9;\n\tadd.cc.u32 t, t, %10;\n\taddc.u32 %0, %0, %0;\n\t"
        "sub.u32 t, %6, %9;\n\tadd.cc.u32 t, t, %10;\n\taddc.u32 %0, %0, %0;\n\t"
        "sub.u32 t, %5, %9;\n\tadd.cc.u32 t, t, %10;\n\taddc.u32 %0, %0, %0;\n\t"
        "sub.u32 t, %4, %9;\n\tadd.cc.u32 t, t, %10;\n\taddc.u32 %0, %0, %0;\n\t"
        "sub.u32 t, %3, %9;\n\tadd.cc.u32 t, t, %10;\n\taddc.u32 %0, %0, %0;\n\t"
        "sub.u32 t, %2, %9;\n\tadd.cc.u32 t, t, %10;\n\taddc.u32 %0, %0, %0;\n\t"
        "sub.u32 t, %1, %9;\n\tadd.cc.u32 t, t, %10;\n\taddc.u32 %0, %0, %0;\n\t"
        "}"
        : "+r"(fail)
        : "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(lo), "r"(nwm1));
    return fail;
}

constexpr int kFilterQ = 256;   // queries staged in shared memory at a time

template <int NA>
__global__ void __launch_bounds__(kThreads) k_filter(AttrCols cols, int64_t N, int64_t n_blocks,
                                                     const CanonPred* __restrict__ canon,
                                                     const ScanPlan* __restrict__ plan,
                                                     int64_t nq, int q_per_cta,
                                                     uint32_t* __restrict__ bm,
                                                     unsigned long long* __restrict__ npass) {
    static_assert(kThreads >= kFilterQ, "one staging pass per query group");
    __shared__ int2 s_iv[kFilterQ][NA];      // (lo, ~wm1) per query and column
    __shared__ uint32_t s_keep[kFilterQ];    // 0 for a predicate no row can pass
    __shared__ uint32_t s_used[kFilterQ];
    __shared__ int s_q[kFilterQ];            // query (offset from the group start)
    __shared__ int s_wcnt[kWarps];
    const int lane = threadIdx.x & 31;
    const int64_t b = (int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5);
    const bool live = b < n_blocks;
    const int64_t q0 = (int64_t)blockIdx.y * q_per_cta;
    const int64_t q1 = min(nq, q0 + (int64_t)q_per_cta);
    const int64_t row0 = (live ? b : 0) * kBlockRows + lane;

    // rows beyond N keep their bits at 0 (columns are padded, so the loads
    // themselves stay inside the allocation)
    uint32_t valid = 0xFFFFFFFFu;
    if (b * kBlockRows + kBlockRows > N) {
        valid = 0;
#pragma unroll
        for (int j = 0; j < 32; ++j) valid |= (uint32_t)(row0 + 32 * j < N) << j;
    }

    int32_t v[NA][32];
#pragma unroll
    for (int c = 0; c < NA; ++c) {
        if (cols.type[c] == IFVS_ATTR_I16) {
            const int16_t* col = (const int16_t*)cols.col[c] + row0;
#pragma unroll
            for (int j = 0; j < 32; ++j) v[c][j] = __ldg(col + 32 * j);
        } else {
            const int32_t* col = (const int32_t*)cols.col[c] + row0;
#pragma unroll
            for (int j = 0; j < 32; ++j) v[c][j] = __ldg(col + 32 * j);
        }
    }

    wait_before();         // the columns are the index's; what follows is prepare's
    start_dependents();
    const int64_t words = n_blocks * 32;
    const int warp = threadIdx.x >> 5;
    for (int64_t g0 = q0; g0 < q1; g0 += kFilterQ) {
        const int ng = (int)min((int64_t)kFilterQ, q1 - g0);
        __syncthreads();
        // stage the group's bitmap-path queries, in order (list-path queries
        // need no bitmap and cost nothing here)
        const int t = threadIdx.x;
        const bool mine = t < ng && (plan == nullptr || !plan[g0 + t].list);
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, mine);
        if (lane == 0) s_wcnt[warp] = __popc(bal);
        __syncthreads();
        int pos = __popc(bal & ((1u << lane) - 1u));
        for (int w = 0; w < warp; ++w) pos += s_wcnt[w];
        int ngd = 0;
        for (int w = 0; w < kWarps; ++w) ngd += s_wcnt[w];
        if (mine) {
            const CanonPred cp = canon[g0 + t];
#pragma unroll
            for (int c = 0; c < NA; ++c) s_iv[pos][c] = make_int2(cp.lo[c], (int32_t)~cp.wm1[c]);
            s_keep[pos] = cp.empty ? 0u : 0xFFFFFFFFu;
            s_used[pos] = cp.used;
            s_q[pos] = t;
        }
        __syncthreads();
        if (!live) continue;
        for (int i = 0; i < ngd; ++i) {
            uint32_t m = valid & s_keep[i];
            const uint32_t used = s_used[i];
#pragma unroll
            for (int c = 0; c < NA; ++c) {
                if (NA == 1 || (used >> c & 1u)) {
                    const int2 iv = s_iv[i][c];
                    uint32_t fail = 0;
#pragma unroll
                    for (int j8 = 24; j8 >= 0; j8 -= 8) fail = fail8(fail, &v[c][j8], iv.x, (uint32_t)iv.y);
                    m &= ~fail;
                }
            }
            const int64_t q = g0 + s_q[i];
            bm[q * words + b * 32 + lane] = m;
            const unsigned cnt = __reduce_add_sync(0xFFFFFFFFu, (unsigned)__popc(m));
            if (lane == 0 && cnt) atomicAdd(npass + q, (unsigned long long)cnt);
        }
    }
}

cudaError_t launch_filter(AttrCols cols, int64_t N, int64_t n_blocks, const CanonPred* canon,
                          const ScanPlan* plan, int64_t nq, uint32_t* bm, unsigned long long* npass,
                          int num_sms, bool chain, cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    const int64_t tiles = (n_blocks + kWarps - 1) / kWarps;
    // enough CTAs to fill the GPU a few times over; each CTA walks a group
    // of queries so that a column tile is read once per group
    const int64_t target = (int64_t)num_sms * 8;
    int64_t groups = (target + tiles - 1) / tiles;
    if (groups < 1) groups = 1;
    if (groups > nq) groups = nq;
    if (groups > 65535) groups = 65535;
    const int64_t qpc = (nq + groups - 1) / groups;
    groups = (nq + qpc - 1) / qpc;
    dim3 grid((unsigned)tiles, (unsigned)groups);
    int na = cols.n < 1 ? 1 : cols.n;
    auto kern = na == 1 ? k_filter<1> : (na == 2 ? k_filter<2> : (na == 3 ? k_filter<3> : k_filter<4>));
    return launch_kernel(kern, grid, dim3(kThreads), 0, chain, s, cols, N, n_blocks, canon, plan, nq, (int)qpc, bm,
                         npass);
}

// ---- layout conversion ---------------------------------------------------

// Transpose the 32x32 bit matrix held one row per lane (lane l, bit j =
// element (l, j)) so that lane l ends up with column l.  Five butterfly
// stages swap the off-diagonal s x s sub-blocks for s = 16, 8, 4, 2, 1.
__device__ __forceinline__ uint32_t transpose32(uint32_t x, int lane) {
    const uint32_t masks[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const int s = 16 >> i;
        const uint32_t mk = masks[i];
        const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x, s);
        x = (lane & s) ? ((x & ~mk) | ((y >> s) & mk)) : ((x & mk) | ((y & mk) << s));
    }
    return x;
}

__global__ void k_bitmap_layout(const uint32_t* __restrict__ src, uint32_t* __restrict__ dst,
                                int64_t nq, int64_t n_blocks, int64_t n_words_rows,
                                bool to_rows) {
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (gw >= nq * n_blocks) return;
    const int64_t q = gw / n_blocks, b = gw - q * n_blocks;
    const int64_t lm = q * n_blocks * 32 + b * 32 + lane;
    const int64_t ri = b * 32 + lane;
    const int64_t rows_off = q * n_words_rows + ri;
    uint32_t x;
    if (to_rows) {
        x = src[lm];
    } else {
        x = ri < n_words_rows ? src[rows_off] : 0u;
    }
    // lane-major word (b, l) bit j == row-ordered word (b*32 + j) bit l
    x = transpose32(x, lane);
    if (to_rows) {
        if (ri < n_words_rows) dst[rows_off] = x;
    } else {
        dst[lm] = x;
    }
}

cudaError_t launch_bitmap_layout(const uint32_t* src, uint32_t* dst, int64_t nq,
                                 int64_t n_blocks, int64_t n_words_rows, bool to_rows,
                                 cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    const int64_t warps = nq * n_blocks;
    const int threads = 256;
    const int64_t blocks = (warps * 32 + threads - 1) / threads;
    k_bitmap_layout<<<(unsigned)blocks, threads, 0, s>>>(src, dst, nq, n_blocks, n_words_rows,
                                                        to_rows);
    return cudaGetLastError();
}

}  // namespace ifvs
