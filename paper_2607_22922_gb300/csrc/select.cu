// Stage 3 of §2 (Select) across CTAs, and the optional exact rerank.
//
// k_merge: one CTA per query folds its items' sorted lists of k keys
// (dist bits << 32 | row) into the query's k smallest; keys are unique, so
// ties in distance fall to the smaller row id exactly as the definition asks.
//
// k_merge_shards: Select across row shards.  Each of G shards returns its
// k best (dist, global row id) per query; one CTA per query sorts the G k
// entries by (dist, id) — a block bitonic sort on an order-preserving
// integer image of the distance and the id (padding, id -1, sorts last) —
// and keeps the k smallest.
//
// k_rerank: one CTA per query computes the exact fp32 squared L2 distance
// (the Pre_IndexFlatL2 distance of §3.2) between the query and each
// candidate's raw vector — one warp per candidate, lanes over dimensions,
// a fixed-order shuffle reduction — and keeps the k best the same way.
#include <math.h>

#include "scan_common.cuh"

namespace ifvs {

__device__ __forceinline__ void block_sort(uint64_t* a, int n) {
    for (int size = 2; size <= n; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            __syncthreads();
            for (int t = threadIdx.x; t < (n >> 1); t += blockDim.x) {
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
    __syncthreads();
}

__device__ __forceinline__ void write_key(uint64_t key, int64_t* id, float* d) {
    if (key == ~0ull) {
        *id = -1;
        *d = INFINITY;
    } else {
        *id = (int64_t)(uint32_t)(key & 0xFFFFFFFFull);
        *d = __uint_as_float((uint32_t)(key >> 32));
    }
}

// One CTA per query; a query with one list only copies it.  The warps split
// the lists: each keeps a sorted list of KP keys and folds the next one in with
// one bitonic merge (both runs are sorted), unless its first key is already
// beyond the k-th; then the warps' lists are merged pairwise.  Sorting all keys
// of all lists again took 45 us for 38 lists of 100 keys, this 12 us.
template <int KP, int WARPS>
__global__ void __launch_bounds__(WARPS * 32) k_merge(const uint64_t* __restrict__ partials,
                                                      const int2* __restrict__ qlist, int k,
                                                      int64_t* __restrict__ ids, float* __restrict__ dists,
                                                      const unsigned long long* __restrict__ npass,
                                                      int64_t* __restrict__ npass_copy) {
    __shared__ uint64_t a[WARPS * 2 * KP];
    const int64_t q = blockIdx.x;
    wait_before();
    start_dependents();
    const int2 ql = qlist[q];
    const uint64_t* src = partials + (int64_t)ql.x * k;
    if (npass_copy != nullptr && threadIdx.x == 0) npass_copy[q] = (int64_t)npass[q];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (ql.y > 1) {
        uint64_t* buf = a + warp * 2 * KP;
        for (int i = lane; i < KP; i += 32) buf[i] = warp < ql.y && i < k ? src[(int64_t)warp * k + i] : ~0ull;
        __syncwarp();
        for (int l = warp + WARPS; l < ql.y; l += WARPS) {
            const uint64_t* list = src + (int64_t)l * k;
            if (__ldg(list) >= buf[k - 1]) continue;
            for (int i = lane; i < KP; i += 32) buf[KP + i] = i < k ? __ldg(list + i) : ~0ull;
            warp_merge_low(buf, KP, lane);
        }
        for (int step = 1; step < WARPS; step <<= 1) {
            __syncthreads();
            if ((warp & (2 * step - 1)) == 0 && warp + step < ql.y) {
                const uint64_t* other = a + (warp + step) * 2 * KP;
                for (int i = lane; i < KP; i += 32) buf[KP + i] = other[i];
                warp_merge_low(buf, KP, lane);
            }
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < k; i += WARPS * 32) {
        const uint64_t key = ql.y > 1 ? a[i] : (ql.y == 1 ? src[i] : ~0ull);
        write_key(key, ids + q * k + i, dists + q * k + i);
    }
}

cudaError_t launch_merge(const ScanSched& sched, int64_t nq, int k, int64_t* ids, float* dists,
                         const unsigned long long* npass, int64_t* npass_copy, bool chain, cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    auto kern = k <= 32 ? k_merge<32, 16> : (k <= 64 ? k_merge<64, 16> : (k <= 128 ? k_merge<128, 16> : k_merge<256, 8>));
    return launch_kernel(kern, dim3((unsigned)nq), dim3(k <= 128 ? 512 : 256), 0, chain, s,
                         (const uint64_t*)sched.partials, (const int2*)sched.qlist, k, ids, dists, npass, npass_copy);
}

constexpr int kShardMergeCap = 4096;   // G * k entries per query, at most

// float -> uint32 whose unsigned order is the float order (NaN aside)
__device__ __forceinline__ uint32_t float_order(float x) {
    const uint32_t b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__global__ void __launch_bounds__(512) k_merge_shards(const float* __restrict__ dists, const int64_t* __restrict__ ids,
                                                      int64_t nq, int G, int k, int n,
                                                      float* __restrict__ dists_out, int64_t* __restrict__ ids_out) {
    __shared__ uint32_t dk[kShardMergeCap];
    __shared__ uint64_t ik[kShardMergeCap];
    const int64_t q = blockIdx.x;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        uint32_t d = 0xFFFFFFFFu;
        uint64_t id = ~0ull;
        if (i < G * k) {
            const int g = i / k, j = i - g * k;
            const int64_t at = ((int64_t)g * nq + q) * k + j;
            const int64_t r = ids[at];
            if (r >= 0) {
                d = float_order(dists[at]);
                id = (uint64_t)r;
            }
        }
        dk[i] = d;
        ik[i] = id;
    }
    for (int size = 2; size <= n; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            __syncthreads();
            for (int t = threadIdx.x; t < (n >> 1); t += blockDim.x) {
                const int i = 2 * t - (t & (stride - 1));
                const int j = i + stride;
                const bool up = (i & size) == 0;
                const uint32_t dx = dk[i], dy = dk[j];
                const uint64_t ix = ik[i], iy = ik[j];
                const bool gt = dx > dy || (dx == dy && ix > iy);
                if (gt == up) {
                    dk[i] = dy;
                    dk[j] = dx;
                    ik[i] = iy;
                    ik[j] = ix;
                }
            }
        }
    __syncthreads();
    for (int i = threadIdx.x; i < k; i += blockDim.x) {
        const bool pad = ik[i] == ~0ull;
        const uint32_t b = dk[i];
        ids_out[q * k + i] = pad ? -1 : (int64_t)ik[i];
        dists_out[q * k + i] = pad ? INFINITY : __uint_as_float((b & 0x80000000u) ? (b & 0x7FFFFFFFu) : ~b);
    }
}

int shard_merge_cap() { return kShardMergeCap; }

cudaError_t launch_merge_shards(const float* dists, const int64_t* ids, int64_t nq, int G, int k,
                                float* dists_out, int64_t* ids_out, cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    int n = 2;
    while (n < G * k) n <<= 1;
    k_merge_shards<<<(unsigned)nq, 512, 0, s>>>(dists, ids, nq, G, k, n, dists_out, ids_out);
    return cudaGetLastError();
}

// WARPS warps, U candidates of a warp in flight: the rows lie anywhere in DRAM.
// While all queries' CTAs are resident at once (four of 16 warps per SM), 16 warps
// with two candidates, from 256 dimensions on one (eight loads of a row are there
// to be in flight); for more queries 8 warps with one.  us per call, 8 warps with
// one / 16 with two / 16 with one:
//   D = 128, 256 candidates: 1 query 32.2 / 25.3 / 24.5, 600 36.4 / 32.5 / 34.5,
//     1024 49.6 / 52.8 / 54.0
//   D = 192, 256 candidates: 600 queries - / 35.9 / 39.2; D = 256: - / 47.1 / 44.1
//   D = 960, 100 candidates: 150 queries 42.5 / 40.5 / 30.8, 1024 82 / 140 / 92,
//     4000 265 / 431 / 280
template <int WARPS, int U>
__global__ void __launch_bounds__(WARPS * 32) k_rerank(const float* __restrict__ X, int64_t N, int D,
                                                       const float* __restrict__ q,
                                                       const int64_t* __restrict__ cand, int R, int k, int rp,
                                                       int64_t* __restrict__ ids, float* __restrict__ dists) {
    __shared__ uint64_t a[IFVS_MAX_K];
    const int64_t qi = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < rp; i += blockDim.x) a[i] = ~0ull;
    wait_before();
    __syncthreads();
    const float* qv = q + qi * D;
    for (int j = warp; j < R; j += U * WARPS) {
        int64_t id[U];
        const float* x[U];
        float s[U] = {};
        bool any = false;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int c = j + u * WARPS;
            id[u] = c < R ? cand[qi * R + c] : -1;
            if (id[u] >= N) id[u] = -1;
            x[u] = X + (id[u] < 0 ? 0 : id[u]) * D;
            any |= id[u] >= 0;
        }
        if (!any) continue;
#pragma unroll 4
        for (int d = lane; d < D; d += 32) {
            const float y = qv[d];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float diff = y - x[u][d];
                s[u] = fmaf(diff, diff, s[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s[u] += __shfl_xor_sync(0xFFFFFFFFu, s[u], o);
            if (lane == 0 && id[u] >= 0)
                a[j + u * WARPS] = ((uint64_t)__float_as_uint(s[u]) << 32) | (uint64_t)(uint32_t)id[u];
        }
    }
    block_sort(a, rp);
    for (int i = threadIdx.x; i < k; i += blockDim.x) write_key(a[i], ids + qi * k + i, dists + qi * k + i);
}

cudaError_t launch_rerank(const float* X, int64_t N, int D, const float* q, const int64_t* cand,
                          int64_t nq, int R, int k, int64_t* ids, float* dists, bool chain, cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    int rp = 32;
    while (rp < R) rp <<= 1;
    int dev = 0, sms = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const bool many = nq > 4 * (int64_t)sms;
    auto kern = many ? k_rerank<8, 1> : (D < 256 ? k_rerank<16, 2> : k_rerank<16, 1>);
    return launch_kernel(kern, dim3((unsigned)nq), dim3(many ? 256 : 512), 0, chain, s, X, N, D, q, cand, R, k, rp,
                         ids, dists);
}

}  // namespace ifvs
