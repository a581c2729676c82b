// Learning the memory bank, W and w_f (§2 "Learning"), one mini-batch of
// queries per step.  The loss (per positive g: softmax cross-entropy of g
// against the mined hard negatives N at temperature tau, averaged over the
// query's positives; plus lambda ||Delta||^2; averaged over the queries) and
// its gradient:
//   dL/ddist_g = (1 - p_g) / tau / |G|,   dL/ddist_n = -sum_g p_n(g) / tau / |G|
//   dL/dC[m][c_v[m]][t] = sum_v gamma_v (-2 w_f (q - C))        (gC, sparse)
//   dL/dw_f[d]          = sum_v gamma_v (q - C)^2
//   dL/dDelta           = gC + 2 lambda Delta,   Delta = alpha . W
//   dL/dW[m][j]         = sum_q alpha_q[m][j] gC_q[m] + 2 lambda sum_j' A_m[j][j'] W[m][j']
//                         with A_m = sum_q alpha_q[m] alpha_q[m]^T
//   dL/dalpha_q[m][j]   = <gC_q[m], W[m][j]> + 2 lambda sum_j' G_m[j][j'] alpha_q[m][j']
//                         with the Gram matrix G_m = W[m] W[m]^T, formed per candidate
//                         while gC is scattered (the W values are already loaded)
//   dL/dbank[b]         = sum over the fetches (q, i) with idx_i(q) = b of dL/dalpha_q
//   dL/dw_z             = dL/dw_f sigmoid(w_z)
// (each divided by the number of queries).  Every sum runs in a fixed order
// (no atomics), so a step is deterministic.
#include "internal.cuh"

namespace ifvs {

namespace {
constexpr int kTrainThreads = 256;
constexpr int kTrainWarps = kTrainThreads / 32;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}
__device__ __forceinline__ double warp_min(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}
}  // namespace

// G[m][j][j'] = sum over (k, t) of W[m][j][k][t] W[m][j'][k][t]; one CTA per entry
__global__ void __launch_bounds__(kTrainThreads) k_train_gram(const float* __restrict__ W, int M,
                                                              int r, int KD, float* __restrict__ G) {
    __shared__ float part[kTrainWarps];
    const int b = blockIdx.x;
    const int m = b / (r * r), j = (b / r) % r, j2 = b % r;
    const float* a = W + ((int64_t)m * r + j) * KD;
    const float* c = W + ((int64_t)m * r + j2) * KD;
    float s = 0.f;
    for (int e = threadIdx.x; e < KD; e += kTrainThreads) s += a[e] * c[e];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < kTrainWarps; ++w) t += part[w];
        G[b] = t;
    }
}

// One CTA per query: candidate list, distances, softmax weights, loss, the
// scatter of dL/dC into the query's dense gC slice and dL/dw_f.  Each thread
// owns the dimensions d = tid + i * blockDim, so every gC address (m, *, t)
// is written by one thread only, in candidate order.
//
// What bounded it was latency and the float64 pipe (about two additions per SM
// and cycle): one thread made the candidate list, every candidate waited for
// the one before it (10 dependent loads each) and was summed over the CTA in
// float64.  Now a warp makes the list by ballots, two candidates' code and W
// values are loaded together, the differences go to shared memory and four
// threads per candidate add its terms (sum_f64).  dL/dw_f, a float32 result, is
// summed over the at most 512 candidates as one float pair (Sum2: within 2^-30 of
// the terms' magnitudes; each term holds a square rounded to float32).  1024 queries with 42 candidates:
// 228 us before.  What is left is the latency of those loads, so CTAs per SM
// count for more than loads per thread: at 128 registers, four candidates in
// flight and 36 KB the grid ran as 1.7 waves of four CTAs per SM (195 us); at 72
// registers, two in flight and 26 KB seven fit (114 us, 40 % of the issue slots, the
// loads' latency still first; the training step 735 -> 673 us; six with two 738, six
// with four, which spill, 764).
//
// Twice the threads per query (three CTAs per SM, two for r > 8) where the
// batch leaves room for them or the shared memory (D r floats) holds fewer than
// seven CTAs anyway; a gradient call in us with 128 / 256 threads, 42 candidates:
//   D = 256, r = 8: 1 query 188 / 151, 400 298 / 254, 1024 421 / 504
//   D = 960, r = 8: 128 queries 820 / 541, 1024 2171 / 1823
//   D = 960, r = 4: 128 queries 819 / 536, 1024 1384 / 1769
//   D = 960, r = 16: 128 queries 1522 / 987, 1024 5081 / 4005
//   D = 2048, r = 8: 1024 queries 4297 / 3118
// At D = 960 the 128 threads alone were slower than the kernel before them, which
// had 256 (r = 4, 128 queries: 641 us).
constexpr int kQueryThreads = 128;
constexpr int kTrainDiffs = 5632;      // floats of the differences held at a time
constexpr int kTrainBatch = 2;         // candidates whose loads are in flight together

// floats shared by the differences (pass 1) and dL/dalpha per dimension (pass
// 2), and the candidates whose differences they hold
__host__ __device__ inline int train_floats(int D, int r) {
    const int need = D * r > D + 1 ? D * r : D + 1;
    return need > kTrainDiffs ? need : kTrainDiffs;
}
__host__ __device__ inline int train_chunk(int V, int D, int r) {
    const int c = train_floats(D, r) / (D + 1);
    return c < V ? c : V;
}

// EXACT: r = RMAX, so no load is behind a test of r and a batch's are all in
// flight at once.
template <int RMAX, bool EXACT, int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS == kQueryThreads ? (RMAX <= 8 ? 7 : 3) : (RMAX <= 8 ? 3 : 2))
k_train_query(TrainQueryArgs a) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int V = a.P + a.n_neg;
    const int Mr = a.M * a.r;
    const int CH = train_chunk(V, a.D, a.r);
    int64_t* cand = reinterpret_cast<int64_t*>(sm);
    double* dist = reinterpret_cast<double*>(cand + V);       // [V]
    double* gam = dist + V;                                   // [V]
    double* red = gam + V;                                    // [warps + 1]
    float* alpha = reinterpret_cast<float*>(red + kTrainWarps + 1);   // [Mr]
    float* dfs = alpha + Mr;                                      // [CH][D + 1] differences
    float* gas = dfs;                                             // [D][r]: dL/dalpha per dimension
    const int64_t q = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nwarps = blockDim.x >> 5;
    const float* qv = a.q + q * a.D;
    const float* wf = a.wf + q * a.D;

    if (warp == 0) {
        const int64_t* pos = a.pos + q * a.pos_stride;
        const int64_t* src = a.negsrc + q * a.neg_stride;
        bool bad = false;
        auto checked = [&](int64_t id) {
            const bool out = id < -1 || id >= a.N;
            bad |= out;
            return out ? (int64_t)-1 : id;
        };
        // positives as given while the mined list is compared with them
        for (int g = lane; g < a.P; g += 32) cand[g] = pos[g];
        __syncwarp();
        int got = 0;
        for (int s0 = 0; s0 < a.S && got < a.n_neg; s0 += 32) {
            const int s = s0 + lane;
            const int64_t id = s < a.S ? src[s] : -1;
            bool keep = s < a.S;
            unsigned end = 0u;
            if (a.exclude) {
                end = __ballot_sync(0xFFFFFFFFu, s < a.S && id < 0);   // a mined list ends at its first -1
                keep = keep && (end == 0u || lane < __ffs(end) - 1);
                for (int g = 0; g < a.P; ++g) keep = keep && cand[g] != id;
            }
            const unsigned ball = __ballot_sync(0xFFFFFFFFu, keep);
            const int at = got + __popc(ball & ((1u << lane) - 1u));
            if (keep && at < a.n_neg) cand[a.P + at] = checked(id);
            got = min(a.n_neg, got + __popc(ball));
            if (end != 0u) break;
        }
        for (int n = got + lane; n < a.n_neg; n += 32) cand[a.P + n] = -1;
        for (int g = lane; g < a.P; g += 32) cand[g] = checked(cand[g]);
        if (bad) atomicOr(a.err, 2);
        __syncwarp();
        if (a.neg_out)
            for (int n = lane; n < a.n_neg; n += 32) a.neg_out[q * a.n_neg + n] = cand[a.P + n];
    }
    for (int e = tid; e < Mr; e += blockDim.x) alpha[e] = a.alpha[q * Mr + e];
    __syncthreads();

    const int64_t KD = (int64_t)a.K * a.ds;
    // code of candidate `id` in subspace m
    auto code_of = [&](int64_t id, int m) -> int {
        int s = m - (int)(id & 31) % a.M;
        if (s < 0) s += a.M;
        return a.codes[id * a.row_bytes + s];
    };

    // pass 1: weighted distances (float32 terms, sum_f64).  The term of
    // dimension d = m ds + t is w_f (q - C)^2 with C_iFVS[m][c][t] = C_PQ +
    // sum_j alpha[m][j] W[m][j][c][t].
    for (int v0 = 0; v0 < V; v0 += CH) {
        const int nv = min(CH, V - v0);
        for (int d = tid; d < a.D; d += blockDim.x) {
            const int m = d / a.ds, t = d - m * a.ds;
            const float* Cm = a.C_pq + (int64_t)m * KD + t;
            const float* Wm = a.W + (int64_t)m * a.r * KD + t;
            for (int i0 = 0; i0 < nv; i0 += kTrainBatch) {
                int c[kTrainBatch];
                float C[kTrainBatch];
#pragma unroll
                for (int u = 0; u < kTrainBatch; ++u) {
                    const int64_t id = i0 + u < nv ? cand[v0 + i0 + u] : -1;
                    c[u] = id >= 0 ? code_of(id, m) * a.ds : 0;
                }
#pragma unroll
                for (int u = 0; u < kTrainBatch; ++u) C[u] = __ldg(Cm + c[u]);
                if constexpr (EXACT && RMAX <= 8) {
                    float w[kTrainBatch][RMAX];
#pragma unroll
                    for (int u = 0; u < kTrainBatch; ++u)
#pragma unroll
                        for (int j = 0; j < RMAX; ++j) w[u][j] = __ldg(Wm + (int64_t)j * KD + c[u]);
#pragma unroll
                    for (int j = 0; j < RMAX; ++j)
#pragma unroll
                        for (int u = 0; u < kTrainBatch; ++u) C[u] += alpha[m * RMAX + j] * w[u][j];
                } else {
#pragma unroll
                    for (int j = 0; j < RMAX; ++j)
                        if (j < a.r) {
                            const float al = alpha[m * a.r + j];
#pragma unroll
                            for (int u = 0; u < kTrainBatch; ++u) C[u] += al * __ldg(Wm + (int64_t)j * KD + c[u]);
                        }
                }
#pragma unroll
                for (int u = 0; u < kTrainBatch; ++u)
                    if (i0 + u < nv) dfs[(i0 + u) * (a.D + 1) + d] = qv[d] - C[u];
            }
        }
        __syncthreads();
        // 4 neighbouring threads per candidate, every fourth dimension each
        for (int x = tid; x < ((4 * nv + 31) & ~31); x += blockDim.x) {
            const int i = x >> 2, p = x & 3;
            auto term = [&](int u) {
                const int d = p + 4 * u;
                const float df = dfs[i * (a.D + 1) + d];
                return __ldg(wf + d) * df * df;
            };
            const int terms = i < nv && p < a.D ? (a.D - p + 3) / 4 : 0;
            double t = sum_f64(0.0, terms, term);
            t += __shfl_xor_sync(0xFFFFFFFFu, t, 1);
            t += __shfl_xor_sync(0xFFFFFFFFu, t, 2);
            if (i < nv && p == 0) dist[v0 + i] = cand[v0 + i] >= 0 ? t : 0.0;
        }
        __syncthreads();
    }

    // Softmax of each positive g against the negatives N, with the shift
    // m_g = min(dist_g, m_N), m_N = min over N:
    //   Z_g = exp(-(d_g - m_g)/tau) + exp(-(m_N - m_g)/tau) S,  S = sum_n u_n,
    //   u_n = exp(-(d_n - m_N)/tau),  p_n(g) = u_n exp(-(m_N - m_g)/tau) / Z_g,
    // so each negative's exponential is shared by all positives (warp 0).
    if (warp == 0) {
        double mN = INFINITY;
        for (int n = a.P + lane; n < V; n += 32)
            if (cand[n] >= 0) mN = fmin(mN, dist[n]);
        mN = warp_min(mN);
        double S = 0.0;
        for (int n = a.P + lane; n < V; n += 32) {
            const double u = cand[n] >= 0 ? exp(-(dist[n] - mN) / a.tau) : 0.0;
            gam[n] = u;
            S += u;
        }
        S = warp_sum(S);
        double lpos = 0.0, csum = 0.0;
        int npos = 0;
        for (int g = lane; g < a.P; g += 32) {
            gam[g] = 0.0;
            if (cand[g] < 0) continue;
            ++npos;
            const double mg = fmin(dist[g], mN);
            const double eg = exp(-(dist[g] - mg) / a.tau);
            const double en = S > 0.0 ? exp(-(mN - mg) / a.tau) : 0.0;
            const double z = eg + en * S;
            lpos += dist[g] / a.tau - mg / a.tau + log(z);
            gam[g] = (1.0 - eg / z) / a.tau;
            csum += en / z;
        }
        lpos = warp_sum(lpos);
        csum = warp_sum(csum);
        npos = __reduce_add_sync(0xFFFFFFFFu, npos);
        __syncwarp();
        const double inv = npos > 0 ? 1.0 / npos : 0.0;
        for (int n = a.P + lane; n < V; n += 32) gam[n] = -gam[n] * csum / a.tau * inv;
        for (int g = lane; g < a.P; g += 32) gam[g] *= inv;
        if (lane == 0) red[kTrainWarps] = npos > 0 ? lpos * inv : 0.0;
    }
    // anchor ||Delta||^2 = sum_m alpha[m]^T G_m alpha[m], a row of G_m per thread
    double an = 0.0;
    for (int x = tid; x < Mr; x += blockDim.x) {
        const int m = x / a.r;
        double row = 0.0;
        for (int j2 = 0; j2 < a.r; ++j2)
            row += (double)a.G[(int64_t)x * a.r + j2] * (double)alpha[m * a.r + j2];
        an += (double)alpha[x] * row;
    }
    an = warp_sum(an);
    if (lane == 0) red[warp] = an;
    __syncthreads();
    if (tid == 0) {
        double s = 0.0;
        for (int w = 0; w < nwarps; ++w) s += red[w];
        a.loss[q] = red[kTrainWarps] + (double)a.lambda * s;
    }

    // pass 2: gC scatter, dL/dw_f, and dL/dalpha through the same W values:
    // dL/dalpha[m][j] = sum over (v, t) of gC contribution x W[m][j][c_v][t]
    float* gC = a.gC + q * (int64_t)a.M * KD;
    for (int d = tid; d < a.D; d += blockDim.x) {
        const int m = d / a.ds, t = d - m * a.ds;
        const float* Cm = a.C_pq + (int64_t)m * KD + t;
        const float* Wm = a.W + (int64_t)m * a.r * KD + t;
        float* gm = gC + (int64_t)m * KD + t;
        Sum2 gw;
        float ga[RMAX];
#pragma unroll
        for (int j = 0; j < RMAX; ++j) ga[j] = 0.f;
        constexpr int B = RMAX <= 8 ? kTrainBatch : 1;
        for (int v0 = 0; v0 < V; v0 += B) {
            int c[B];
            float C[B], w[B][RMAX];
#pragma unroll
            for (int u = 0; u < B; ++u) {
                const int64_t id = v0 + u < V ? cand[v0 + u] : -1;
                c[u] = id >= 0 ? code_of(id, m) * a.ds : -1;
            }
#pragma unroll
            for (int u = 0; u < B; ++u) C[u] = __ldg(Cm + max(c[u], 0));
#pragma unroll
            for (int j = 0; j < RMAX; ++j)
                if (EXACT || j < a.r)
#pragma unroll
                    for (int u = 0; u < B; ++u) w[u][j] = __ldg(Wm + (int64_t)j * KD + max(c[u], 0));
#pragma unroll
            for (int u = 0; u < B; ++u) {
                if (c[u] < 0) continue;
#pragma unroll
                for (int j = 0; j < RMAX; ++j)
                    if (EXACT || j < a.r) C[u] += alpha[m * a.r + j] * w[u][j];
                const float df = qv[d] - C[u];
                const double g = gam[v0 + u];
                const float gf = (float)g;
                const float ge = gf * (-2.f * __ldg(wf + d) * df);
                gm[c[u]] += ge;
                // gam (df df) to 48 bits: gam as two floats, exact products
                const float sq = df * df, p = __fmul_rn(gf, sq);
                gw.add(p);
                gw.lo = __fadd_rn(gw.lo, fmaf((float)(g - (double)gf), sq, fmaf(gf, sq, -p)));
#pragma unroll
                for (int j = 0; j < RMAX; ++j)
                    if (EXACT || j < a.r) ga[j] += ge * w[u][j];
            }
        }
        double gwd = gw.value();
        if (!gw.finite()) {   // beyond float32, infinite or NaN: in float64
            gwd = 0.0;
            for (int v = 0; v < V; ++v) {
                const int64_t id = cand[v];
                if (id < 0) continue;
                const int c = code_of(id, m) * a.ds;
                float C = Cm[c];
                for (int j = 0; j < a.r; ++j) C += alpha[m * a.r + j] * Wm[(int64_t)j * KD + c];
                const float df = qv[d] - C;
                gwd += gam[v] * (double)(df * df);
            }
        }
        a.gw[q * a.D + d] = (float)gwd;
#pragma unroll
        for (int j = 0; j < RMAX; ++j)
            if (EXACT || j < a.r) gas[d * a.r + j] = ga[j];
    }
    __syncthreads();
    // sum over the subspace's dimensions in order, plus the anchor 2 lambda G_m alpha[m]
    for (int x = tid; x < Mr; x += blockDim.x) {
        const int m = x / a.r, j = x - m * a.r;
        float sg = 0.f;
        for (int t = 0; t < a.ds; ++t) sg += gas[(m * a.ds + t) * a.r + j];
        float an = 0.f;
        for (int j2 = 0; j2 < a.r; ++j2) an += a.G[((int64_t)m * a.r + j) * a.r + j2] * alpha[m * a.r + j2];
        a.galpha[q * Mr + x] = sg + 2.f * a.lambda * an;
    }
}

// A[m][j][j'] = sum over the queries of alpha_q[m][j] alpha_q[m][j'] (one CTA per entry)
__global__ void __launch_bounds__(kTrainThreads) k_train_acov(const float* __restrict__ alpha, int64_t n,
                                                              int M, int r, float* __restrict__ A) {
    __shared__ float part[kTrainWarps];
    const int b = blockIdx.x;
    const int m = b / (r * r), j = (b / r) % r, j2 = b % r;
    const int Mr = M * r;
    float s = 0.f;
    for (int64_t q = threadIdx.x; q < n; q += kTrainThreads)
        s += alpha[q * Mr + m * r + j] * alpha[q * Mr + m * r + j2];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < kTrainWarps; ++w) t += part[w];
        A[b] = t;
    }
}

// Partial sums of alpha_q[m][j] gC_q[m][e] over one slice of kGWQueries
// queries: grid (M, ceil(KD / 256), slices); part [slices][M][r][KD]
constexpr int kGWQueries = 64;
template <int RMAX>
__global__ void __launch_bounds__(kTrainThreads) k_train_gW_part(const float* __restrict__ alpha,
                                                                 const float* __restrict__ gC, int64_t n,
                                                                 int M, int r, int KD,
                                                                 float* __restrict__ part) {
    __shared__ float as[kGWQueries * kTrainMaxR];
    const int m = blockIdx.x;
    const int e = blockIdx.y * kTrainThreads + threadIdx.x;
    const int64_t q0 = (int64_t)blockIdx.z * kGWQueries;
    const int nc = (int)min((int64_t)kGWQueries, n - q0);
    const int Mr = M * r;
    for (int t = threadIdx.x; t < nc * r; t += kTrainThreads)
        as[t] = alpha[(q0 + t / r) * Mr + m * r + t % r];
    __syncthreads();
    if (e >= KD) return;
    float acc[RMAX];
#pragma unroll
    for (int j = 0; j < RMAX; ++j) acc[j] = 0.f;
#pragma unroll 8
    for (int i = 0; i < nc; ++i) {
        const float g = gC[((q0 + i) * M + m) * (int64_t)KD + e];
#pragma unroll
        for (int j = 0; j < RMAX; ++j)
            if (j < r) acc[j] += as[i * r + j] * g;
    }
    float* out = part + (((int64_t)blockIdx.z * M + m) * r) * KD + e;
#pragma unroll
    for (int j = 0; j < RMAX; ++j)
        if (j < r) out[(int64_t)j * KD] = acc[j];
}

// dL/dW[m][j][e] = inv_n (sum over slices of part + 2 lambda sum_j' A_m[j][j'] W[m][j'][e]),
// slices summed in order
__global__ void k_train_gW_sum(const float* __restrict__ part, int slices, const float* __restrict__ A,
                               const float* __restrict__ W, int M, int r, int KD, float lambda,
                               float inv_n, float* __restrict__ gW) {
    const int64_t total = (int64_t)M * r * KD;
    const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= total) return;
    const int e = (int)(x % KD);
    const int j = (int)((x / KD) % r);
    const int m = (int)(x / ((int64_t)KD * r));
    float s = 0.f;
    for (int z = 0; z < slices; ++z) s += part[(int64_t)z * total + x];
    float an = 0.f;
    for (int j2 = 0; j2 < r; ++j2)
        an += A[((int64_t)m * r + j) * r + j2] * W[((int64_t)m * r + j2) * KD + e];
    gW[x] = (s + 2.f * lambda * an) * inv_n;
}

// dL/dbank: one CTA per fetch p = (q, i).  The first fetch of each bank row
// gathers, in fetch order, the fetches of that row and sums their dL/dalpha.
constexpr int kBankList = 512;
__global__ void __launch_bounds__(kTrainThreads) k_train_bank(const uint32_t* __restrict__ idx,
                                                              int64_t n_fetch, int h, int Mr,
                                                              const float* __restrict__ galpha,
                                                              float inv_n, float* __restrict__ gbank) {
    __shared__ int64_t list[kBankList];
    __shared__ int wcnt[kTrainWarps];
    __shared__ int total;
    const int64_t p = blockIdx.x;
    const uint32_t b = idx[p];
    int earlier = 0;
    for (int64_t p2 = threadIdx.x; p2 < p; p2 += blockDim.x) earlier |= idx[p2] == b;
    if (__syncthreads_or(earlier)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    for (int64_t c0 = p; c0 < n_fetch; c0 += blockDim.x) {
        const int64_t p2 = c0 + threadIdx.x;
        const bool f = p2 < n_fetch && idx[p2] == b;
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, f);
        if (lane == 0) wcnt[warp] = __popc(bal);
        __syncthreads();
        int off = total;
        for (int w = 0; w < warp; ++w) off += wcnt[w];
        off += __popc(bal & ((1u << lane) - 1u));
        if (f && off < kBankList) list[off] = p2;
        __syncthreads();
        if (threadIdx.x == 0)
            for (int w = 0; w < nw; ++w) total += wcnt[w];
        __syncthreads();
    }
    const int cnt = total;
    for (int e = threadIdx.x; e < Mr; e += blockDim.x) {
        float s = 0.f;
        if (cnt <= kBankList) {
            for (int i = 0; i < cnt; ++i) s += galpha[(list[i] / h) * Mr + e];
        } else {
            for (int64_t p2 = p; p2 < n_fetch; ++p2)
                if (idx[p2] == b) s += galpha[(p2 / h) * Mr + e];
        }
        gbank[(int64_t)b * Mr + e] = s * inv_n;
    }
}

// dL/dw_z[d] = inv_n sum_q dL/dw_f[q][d] sigmoid(w_z[d]); block (32 dims, 32
// query lanes), lane y sums the queries q = y (mod 32) in order, then the 32
// lanes are added in order
__global__ void __launch_bounds__(1024) k_train_wz(const float* __restrict__ gw, int64_t n, int D,
                                                   const float* __restrict__ wz, float inv_n,
                                                   float* __restrict__ gwz) {
    __shared__ double part[32][33];
    const int d = blockIdx.x * 32 + threadIdx.x;
    double s = 0.0;
    if (d < D) {
        // a float pair over at most 32 terms (1024 queries): the float64 adders took 22 us at D = 128
        Sum2 p;
#pragma unroll 8
        for (int64_t q = threadIdx.y; q < n; q += 32) p.add(gw[q * D + d]);
        s = p.value();
        if (!p.finite()) {
            s = 0.0;
            for (int64_t q = threadIdx.y; q < n; q += 32) s += (double)gw[q * D + d];
        }
    }
    part[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y != 0 || d >= D) return;
    double t = 0.0;
    for (int y = 0; y < 32; ++y) t += part[y][threadIdx.x];
    const float x = wz[d];
    const float sg = x >= 0.f ? 1.f / (1.f + expf(-x)) : expf(x) / (1.f + expf(x));
    gwz[d] = (float)t * sg * inv_n;
}

// theta <- theta - lr * g for the bank, W and w_z
__global__ void k_sgd(SgdArgs a) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (e < a.n[i]) a.theta[i][e] = a.theta[i][e] - a.lr[i] * a.g[i][e];
        if (e < a.n[i]) return;
        e -= a.n[i];
    }
}

size_t train_query_smem(int V, int Mr, int D, int r) {
    return sizeof(int64_t) * V + sizeof(double) * ((size_t)2 * V + kTrainWarps + 1) +
           sizeof(float) * (Mr + (size_t)train_floats(D, r));
}

cudaError_t launch_train_gram(const float* W, int M, int r, int KD, float* G, cudaStream_t s) {
    k_train_gram<<<(unsigned)(M * r * r), kTrainThreads, 0, s>>>(W, M, r, KD, G);
    return cudaGetLastError();
}

cudaError_t launch_train_query(const TrainQueryArgs& a, cudaStream_t s) {
    const size_t smem = train_query_smem(a.P + a.n_neg, a.M * a.r, a.D, a.r);
    int dev = 0, sms = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const bool wide = a.D > kQueryThreads && (a.n <= 3 * (int64_t)sms || 7 * (smem + 1024) > 233472);
    // threads own dimensions: no more threads than (32-rounded) dimensions
    const int most = wide ? 2 * kQueryThreads : kQueryThreads;
    const int threads = a.D >= most ? most : ((a.D + 31) / 32) * 32;
    auto kern = wide ? (a.r == 8  ? k_train_query<8, true, 2 * kQueryThreads>
                        : a.r < 8 ? k_train_query<8, false, 2 * kQueryThreads>
                                  : k_train_query<kTrainMaxR, false, 2 * kQueryThreads>)
                     : (a.r == 8  ? k_train_query<8, true, kQueryThreads>
                        : a.r < 8 ? k_train_query<8, false, kQueryThreads>
                                  : k_train_query<kTrainMaxR, false, kQueryThreads>);
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)a.n, threads, smem, s>>>(a);
    return cudaGetLastError();
}

size_t train_gW_scratch(int64_t n, int M, int r, int KD) {
    const int64_t slices = (n + kGWQueries - 1) / kGWQueries;
    return sizeof(float) * (size_t)(slices * M * r * KD + M * r * r);
}

cudaError_t launch_train_gW(const float* alpha, const float* gC, const float* W, int64_t n, int M, int r,
                            int KD, float lambda, float inv_n, float* scratch, float* gW,
                            cudaStream_t s, int* launches) {
    const int slices = (int)((n + kGWQueries - 1) / kGWQueries);
    float* A = scratch;
    float* part = scratch + M * r * r;
    k_train_acov<<<(unsigned)(M * r * r), kTrainThreads, 0, s>>>(alpha, n, M, r, A);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)M, (unsigned)((KD + kTrainThreads - 1) / kTrainThreads), (unsigned)slices);
    if (r <= 8)
        k_train_gW_part<8><<<grid, kTrainThreads, 0, s>>>(alpha, gC, n, M, r, KD, part);
    else
        k_train_gW_part<kTrainMaxR><<<grid, kTrainThreads, 0, s>>>(alpha, gC, n, M, r, KD, part);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int64_t total = (int64_t)M * r * KD;
    k_train_gW_sum<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(part, slices, A, W, M, r, KD, lambda,
                                                                    inv_n, gW);
    if (launches) *launches = 3;
    return cudaGetLastError();
}

cudaError_t launch_train_bank(const uint32_t* idx, int64_t n, int h, int Mr, const float* galpha,
                              float inv_n, float* gbank, cudaStream_t s) {
    const int threads = Mr < kTrainThreads ? ((Mr + 31) / 32) * 32 : kTrainThreads;
    k_train_bank<<<(unsigned)(n * h), threads, 0, s>>>(idx, n * h, h, Mr, galpha, inv_n, gbank);
    return cudaGetLastError();
}

cudaError_t launch_train_wz(const float* gw, int64_t n, int D, const float* wz, float inv_n, float* gwz,
                            cudaStream_t s) {
    k_train_wz<<<(unsigned)((D + 31) / 32), dim3(32, 32), 0, s>>>(gw, n, D, wz, inv_n, gwz);
    return cudaGetLastError();
}

cudaError_t launch_sgd(const SgdArgs& a, cudaStream_t s) {
    const int64_t n = a.n[0] + a.n[1] + a.n[2];
    if (n <= 0) return cudaSuccess;
    k_sgd<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace ifvs
