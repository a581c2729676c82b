// Building the PQ index on the GPU (the offline step before the query path
// of §2: the base codebook C_PQ and the uint8 codes stay fixed afterwards).
// The assignment is in pq_assign.cu; here is the Lloyd update.
//
// Training keeps the codes and distances of an iteration by subspace
// ([M][n]), so that every pass over one subspace is coalesced.
//
// k_pq_accumulate: CTA (row chunk, subspace), the subspaces of a chunk in a row.  The chunk's rows are sorted by
// codeword (counting sort in shared memory, 4096 rows at a time), then thread
// (codeword, dimension) adds its members' values, in registers, into its own
// float64 accumulator in shared memory.  Float64 additions bound the same kernel
// with one per member (this part adds some two per SM and cycle: 77 us for
// 65 536 rows x 16 subspaces; 140 us with float64 atomics on shared memory,
// which are compare-and-swap loops), so up to 32 members go into a pair of
// floats with the rounding error of every addition carried along (TwoSum,
// Knuth) before it is added (sum_f64): 39 us, as with one pair per codeword and
// chunk, which was up to 1500 float32 ulp off on long runs of alike values.  The
// latency of the members' loads is what is left (issue slots 32 % used).  Infinite, huge
// and NaN values give what float64 sums give.  The same CTA
// adds up the chunk's distances and finds its farthest row.
//
// k_pq_finalize: the chunks' sums, in order, to float32 means; the objective.
//
// k_pq_reseed: each unused codeword of a subspace, in increasing order, takes
// the row farthest from its codeword (largest float32 distance, ties to the
// smallest row: the maximum of distance bits << 32 | ~row), whose distance
// then counts as 0.  Only the chunk that lost its farthest row is searched
// again, on the device: training needs no host synchronisation between
// iterations.
#include "internal.cuh"

namespace ifvs {

constexpr int kLloydThreads = 256;
constexpr int kSortRows = 4096;
static_assert(kSortRows <= 65536 && kSortRows % kLloydThreads == 0, "16-bit row offsets, whole rounds");

__device__ __forceinline__ unsigned long long far_key(float d, int64_t row) {
    return ((unsigned long long)__float_as_uint(d) << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)row);
}

// the block's maximum, in every thread
__device__ __forceinline__ unsigned long long block_max(unsigned long long v, unsigned long long* scratch) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long other = __shfl_xor_sync(0xFFFFFFFFu, v, o);
        v = other > v ? other : v;
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
    __syncthreads();
    for (int w = 0; w < kLloydThreads / 32; ++w) v = scratch[w] > v ? scratch[w] : v;
    return v;
}

__global__ void __launch_bounds__(kLloydThreads) k_pq_accumulate(const float* __restrict__ X, int64_t n, int D, int M,
                                                                 int K, int ds, LloydBufs b) {
    extern __shared__ __align__(16) double acc[];   // [K * ds]
    __shared__ uint16_t order[kSortRows];
    __shared__ int cnt[256], start[257], wsum[kLloydThreads / 32];
    __shared__ unsigned total[256];
    __shared__ unsigned long long red[kLloydThreads / 32];
    __shared__ double dred[kLloydThreads / 32];
    const int m = (int)(blockIdx.x % (unsigned)M), ch = (int)(blockIdx.x / (unsigned)M), tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    const int64_t r0 = (int64_t)ch * b.rows_per_chunk;
    const int64_t r1 = min(n, r0 + b.rows_per_chunk);
    const int KD = K * ds;
    const uint8_t* codes = b.codes + (int64_t)m * n;
    const float* dmin = b.dmin + (int64_t)m * n;
    for (int e = tid; e < KD; e += kLloydThreads) acc[e] = 0.0;
    total[tid] = 0u;
    constexpr int PER = kSortRows / kLloydThreads;
    for (int64_t s0 = r0; s0 < r1; s0 += kSortRows) {
        const int ns = (int)min((int64_t)kSortRows, r1 - s0);
        cnt[tid] = 0;
        __syncthreads();
        int code[PER], rank[PER];
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int r = i * kLloydThreads + tid;
            code[i] = r < ns ? codes[s0 + r] : -1;
        }
#pragma unroll
        for (int i = 0; i < PER; ++i) rank[i] = code[i] >= 0 ? atomicAdd(&cnt[code[i]], 1) : 0;
        __syncthreads();
        {   // start[c]: exclusive prefix of the counts
            const int v = cnt[tid];
            total[tid] += (unsigned)v;
            int incl = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= o) incl += t;
            }
            if (lane == 31) wsum[warp] = incl;
            __syncthreads();
            int before = 0;
            for (int w = 0; w < warp; ++w) before += wsum[w];
            start[tid] = before + incl - v;
            if (tid == 255) start[256] = before + incl;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (code[i] >= 0) order[start[code[i]] + rank[i]] = (uint16_t)(i * kLloydThreads + tid);
        __syncthreads();
        const float* base = X + s0 * D + m * ds;
        for (int e = tid; e < KD; e += kLloydThreads) {
            const int k = e / ds, t = e - k * ds;
            const int j0 = start[k];
            acc[e] = sum_f64(acc[e], start[k + 1] - j0,
                             [&](int j) { return __ldg(base + (int64_t)order[j0 + j] * D + t); });
        }
        __syncthreads();   // order and the counts are rewritten
    }
    double obj = 0.0;
    unsigned long long far = 0ull;
    for (int64_t r = r0 + tid; r < r1; r += kLloydThreads) {
        const float d = dmin[r];
        const unsigned long long key = far_key(d, r);
        far = key > far ? key : far;
        obj += (double)d;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) obj += __shfl_xor_sync(0xFFFFFFFFu, obj, o);
    if (lane == 0) dred[warp] = obj;
    far = block_max(far, red);   // its barriers publish dred and total too
    const int64_t cm = (int64_t)ch * M + m;
    if (tid == 0) {
        double t = 0.0;
        for (int w = 0; w < kLloydThreads / 32; ++w) t += dred[w];
        b.obj[cm] = t;
        b.far[cm] = far;
    }
    for (int e = tid; e < KD; e += kLloydThreads) b.sums[cm * KD + e] = acc[e];
    if (tid < K) b.counts[cm * K + tid] = total[tid];
}

// thread (m, k, t): float32 mean of the members; thread m of the first CTA:
// the objective of subspace m
__global__ void k_pq_finalize(LloydBufs b, int M, int K, int ds, const float* __restrict__ C_in,
                              float* __restrict__ C_out, double* __restrict__ objective) {
    if (blockIdx.x == 0 && objective != nullptr)
        for (int m = threadIdx.x; m < M; m += blockDim.x) {
            double t = 0.0;
            for (int ch = 0; ch < b.chunks; ++ch) t += b.obj[(int64_t)ch * M + m];
            objective[m] = t;
        }
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t all = (int64_t)M * K * ds;
    if (e >= all) return;
    const int64_t mk = e / ds;
    unsigned long long c = 0ull;
    double v = 0.0;
#pragma unroll 8
    for (int ch = 0; ch < b.chunks; ++ch) {
        v += b.sums[ch * all + e];
        c += b.counts[(int64_t)ch * M * K + mk];
    }
    C_out[e] = c > 0 ? (float)(v / (double)c) : C_in[e];
    if (e - mk * ds == 0) b.used[mk] = c > 0 ? 1 : 0;
}

// CTA m: the unused codewords of subspace m
__global__ void __launch_bounds__(kLloydThreads) k_pq_reseed(const float* __restrict__ X, int64_t n, int D, int M,
                                                             int K, int ds, LloydBufs b, float* __restrict__ C_out) {
    __shared__ unsigned long long red[kLloydThreads / 32];
    const int m = blockIdx.x, tid = threadIdx.x;
    if (!__syncthreads_or(tid < K && b.used[(int64_t)m * K + tid] == 0)) return;
    float* dmin = b.dmin + (int64_t)m * n;
    for (int c = 0; c < K; ++c) {
        if (b.used[(int64_t)m * K + c] != 0) continue;
        unsigned long long best = 0ull;
        for (int ch = tid; ch < b.chunks; ch += kLloydThreads) {
            const unsigned long long k = b.far[(int64_t)ch * M + m];
            best = k > best ? k : best;
        }
        best = block_max(best, red);
        const int64_t row = (int64_t)(0xFFFFFFFFu - (uint32_t)(best & 0xFFFFFFFFull));
        for (int t = tid; t < ds; t += kLloydThreads) C_out[((int64_t)m * K + c) * ds + t] = X[row * D + m * ds + t];
        const int64_t ch = row / b.rows_per_chunk;
        const int64_t r0 = ch * b.rows_per_chunk, r1 = min(n, r0 + b.rows_per_chunk);
        if (tid == 0) dmin[row] = 0.f;
        unsigned long long far = 0ull;
        for (int64_t r = r0 + tid; r < r1; r += kLloydThreads) {
            const unsigned long long k = far_key(r == row ? 0.f : dmin[r], r);
            far = k > far ? k : far;
        }
        far = block_max(far, red);
        if (tid == 0) b.far[ch * M + m] = far;
        __syncthreads();
    }
}

// Chunks: as many as give about two CTAs per SM, of at least 1024 rows.
void lloyd_plan(int64_t n, int M, int K, int ds, int num_sms, LloydBufs* b, size_t* bytes) {
    int64_t chunks = (int64_t)num_sms * 2 / M;
    if (chunks < 1) chunks = 1;
    int64_t rows = (n + chunks - 1) / chunks;
    if (rows < 1024) rows = 1024;
    b->rows_per_chunk = rows;
    b->chunks = (int)((n + rows - 1) / rows);
    const int64_t KD = (int64_t)K * ds, cm = (int64_t)b->chunks * M;
    size_t at = 0;
    auto take = [&](size_t sz) {
        const size_t p = at;
        at = (at + sz + 255) / 256 * 256;
        return p;
    };
    uint8_t* p = b->base;
    b->sums = reinterpret_cast<double*>(p + take(sizeof(double) * (size_t)(cm * KD)));
    b->obj = reinterpret_cast<double*>(p + take(sizeof(double) * (size_t)cm));
    b->far = reinterpret_cast<unsigned long long*>(p + take(sizeof(unsigned long long) * (size_t)cm));
    b->counts = reinterpret_cast<unsigned*>(p + take(sizeof(unsigned) * (size_t)(cm * K)));
    b->dmin = reinterpret_cast<float*>(p + take(sizeof(float) * (size_t)n * M));
    b->codes = p + take((size_t)n * M);
    b->used = p + take((size_t)M * K);
    *bytes = at;
}

cudaError_t launch_pq_update(const float* X, int64_t n, int D, int M, int K, const LloydBufs& b, const float* C_in,
                             float* C_out, double* objective, cudaStream_t s) {
    const int ds = D / M;
    const size_t smem = (size_t)K * ds * sizeof(double);
    cudaError_t e = cudaFuncSetAttribute(k_pq_accumulate, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // one grid dimension: M may be above the 65535 of the second
    k_pq_accumulate<<<(unsigned)((int64_t)b.chunks * M), kLloydThreads, smem, s>>>(X, n, D, M, K, ds, b);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int64_t total = (int64_t)M * K * ds;
    k_pq_finalize<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(b, M, K, ds, C_in, C_out, objective);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_pq_reseed<<<(unsigned)M, kLloydThreads, 0, s>>>(X, n, D, M, K, ds, b, C_out);
    return cudaGetLastError();
}

}  // namespace ifvs
