// Collapsed log marginal likelihood of fixed labels and its gradient with
// respect to log alpha and a gene-wise log beta (theta integrated out of
// eq. 12 against eq. 28 with lambda generalised to beta_u, pi out of eq. 10).
//
//   k_lml_stats     (logml_stats.cuh) n_k, S_ku, T_k of the labelled cells
//                   (integer, exact); for a sampler's chain (dpmm_logml_grad)
//                   k_lml_from_chain sums its sub-cluster statistics
//   k_lml_terms     FP64, blocks of kLmlGenes genes: the gene terms
//                   sum_{u, k: S_ku > 0} [lgamma(beta_u + S_ku) - lgamma(beta_u)]
//                   and B = sum beta_u; the last block adds the cluster terms
//                   lgamma(n_k) + lgamma(B) - lgamma(B + T_k) and the partition
//                   terms (from the host), and for the gradient forms
//                   c = sum_k [psi(B) - psi(B + T_k)] and
//                   d/d log alpha = K + alpha (psi(alpha) - psi(alpha + N))
//   k_lml_backward  beta_u (c + sum_{k: S_ku > 0} [psi(beta_u + S_ku) - psi(beta_u)]),
//                   FP32 digammas summed in FP64
#include <math_constants.h>

#include <cmath>

#include "logml.cuh"
#include "logml_stats.cuh"

namespace dpmm {

constexpr int kLmlGenes = 8;      // genes per block
constexpr int kLmlLanes = 32;     // threads per gene, each every 32nd cluster
constexpr int kLmlThreads = kLmlGenes * kLmlLanes;
constexpr int kLmlChainThreads = 256;

// Block sums of M values at once (every thread gets them); red: 32 M doubles.
template <int M>
__device__ __forceinline__ void block_sums(double (&v)[M], double* red) {
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = (int)(blockDim.x >> 5);
#pragma unroll
    for (int o = 16; o; o >>= 1)
#pragma unroll
        for (int m = 0; m < M; ++m) v[m] += __shfl_xor_sync(0xFFFFFFFFu, v[m], o);
    __syncthreads();
    if (l == 0)
#pragma unroll
        for (int m = 0; m < M; ++m) red[32 * m + w] = v[m];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < M; ++m) v[m] = l < nw ? red[32 * m + l] : 0.0;
#pragma unroll
    for (int o = 16; o; o >>= 1)
        if (o < nw)
#pragma unroll
            for (int m = 0; m < M; ++m) v[m] += __shfl_xor_sync(0xFFFFFFFFu, v[m], o);
#pragma unroll
    for (int m = 0; m < M; ++m) v[m] = __shfl_sync(0xFFFFFFFFu, v[m], 0);
}

// Block g: genes 8 g .. 8 g + 7, 32 threads a gene (every 32nd cluster each).
// GB300 issues 1.7 FP64 operations per SM and cycle, 65 cycles deep (measured;
// a library lgamma takes about 2,400 cycles alone and 20 cycles per thread of
// a full SM), so the cost is the number of FP64 operations, how evenly they
// lie on the SMs and how many follow one another: a term is one lgamma;
// exp(log beta_u) and lgamma(beta_u) are taken once per gene, beside the
// terms, instead of once per term; B is summed by all blocks (the exponentials
// of 2,000 genes on one SM took 23 us); the last block to finish adds the
// cluster terms, one lgamma per thread.  100,000 x 2,000 with K = 25 (ncu,
// cold): value and gradients 93 -> 34 us.  The per-block sums are added in block order,
// so the value is the same in every run.
// value: the log ML itself; grad: c and d/d log alpha.  part_value, part_grad:
// lgamma(alpha) - lgamma(alpha + N), alpha (psi(alpha) - psi(alpha + N)).
__global__ void __launch_bounds__(kLmlThreads)
k_lml_terms(const uint32_t* __restrict__ n, const uint32_t* __restrict__ S,
            const unsigned long long* __restrict__ T, const float* __restrict__ log_beta,
            int32_t D, int32_t K, double log_alpha, double part_value, double part_grad,
            int32_t value, int32_t grad, double* part, int32_t* ticket, double* __restrict__ out,
            double* __restrict__ grad_alpha, double* __restrict__ common, uint32_t* wrap_flag) {
    __shared__ double red[3 * 32];
    __shared__ double sb[kLmlGenes], slg[kLmlGenes], slgB;
    __shared__ int last;
    const int j = threadIdx.x % kLmlGenes, q = threadIdx.x / kLmlGenes;
    const int u = blockIdx.x * kLmlGenes + j;
    if (q == 0) sb[j] = u < D ? exp((double)log_beta[u]) : 0.0;
    __syncthreads();
    double acc[1] = {0.0};
    if (value) {
        const double b = sb[j];
        int terms = 0;
        if (u < D) {
            for (int k = q; k < K; k += kLmlLanes) {
                const uint32_t s = S[(size_t)k * D + u];
                if (s) {
                    acc[0] += lgamma(b + (double)s);
                    ++terms;
                }
            }
            // (the last warp, with the fewest clusters, takes lgamma(beta_u) as well)
            if (q == kLmlLanes - 1) slg[j] = lgamma(b);
        }
        __syncthreads();
        if (terms) acc[0] -= (double)terms * slg[j];
        block_sums(acc, red);
    }
    if (threadIdx.x == 0) {
        double sum = 0.0;
        for (int i = 0; i < kLmlGenes; ++i) sum += sb[i];
        part[2 * (size_t)blockIdx.x] = acc[0];
        part[2 * (size_t)blockIdx.x + 1] = sum;
        __threadfence();
        last = atomicAdd(ticket, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (threadIdx.x == 0) *ticket = 0;
    double ab[2] = {0.0, 0.0};
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) {
        ab[0] += __ldcg(part + 2 * (size_t)i);
        ab[1] += __ldcg(part + 2 * (size_t)i + 1);
    }
    block_sums(ab, red);
    const double B = ab[1];
    // items 0 .. K - 1: lgamma(n_k) and c's term; K .. 2K - 1: lgamma(B + T_k);
    // 2K: lgamma(B), once per cluster
    const float Bf = (float)B;
    const float psiB = grad ? digamma<float>(Bf) : 0.0f;
    double t[3] = {0.0, 0.0, 0.0};   // value, c, clusters
    for (int i = threadIdx.x; i < 2 * K + 1; i += blockDim.x) {
        if (i == 2 * K) {
            slgB = value ? lgamma(B) : 0.0;
        } else if (i >= K) {
            if (value && n[i - K]) t[0] -= lgamma(B + (double)T[i - K]);
        } else if (n[i]) {
            t[2] += 1.0;
            if (wrap_flag && (T[i] >> 32)) atomicOr(wrap_flag, kLmlWrapFlag);
            if (value) t[0] += lgamma((double)n[i]);
            if (grad) t[1] += (double)(psiB - digamma<float>(Bf + (float)T[i]));
        }
    }
    block_sums(t, red);
    if (threadIdx.x == 0) {
        if (value) *out = ab[0] + (t[0] + t[2] * slgB) + (t[2] * log_alpha + part_value);
        if (grad) {
            *common = t[1];
            *grad_alpha = t[2] + part_grad;
        }
    }
}

// Threads as in k_lml_terms.  The digammas are FP32, their sum over the
// clusters FP64 (the terms cancel against c).
__global__ void __launch_bounds__(kLmlThreads)
k_lml_backward(const uint32_t* __restrict__ S, const float* log_beta, int32_t D, int32_t K,
               const double* __restrict__ common, float* grad) {
    __shared__ double sacc[kLmlLanes][kLmlGenes];
    const int j = threadIdx.x % kLmlGenes, q = threadIdx.x / kLmlGenes;
    const int u = blockIdx.x * kLmlGenes + j;
    double acc = 0.0;
    float b = 0.0f;
    if (u < D) {
        b = expf(log_beta[u]);
        const float psib = digamma<float>(b);
        for (int k = q; k < K; k += kLmlLanes) {
            const uint32_t s = S[(size_t)k * D + u];
            if (s) acc += (double)(digamma<float>(b + (float)s) - psib);
        }
    }
    sacc[q][j] = acc;
    __syncthreads();
    if (q == 0 && u < D) {
        acc = *common;
        for (int i = 0; i < kLmlLanes; ++i) acc += sacc[i][j];
        grad[u] = (float)((double)b * acc);
    }
}

// Cluster statistics of a sampler's current state from its sub-cluster
// statistics: n_k = n-bar_k0 + n-bar_k1, S_ku = S-bar_k0u + S-bar_k1u,
// T_k = sum_u S_ku.  One block per cluster.
__global__ void k_lml_from_chain(const uint32_t* __restrict__ nsub,
                                 const uint32_t* __restrict__ Ssub, int32_t D,
                                 uint32_t* __restrict__ n, uint32_t* __restrict__ S,
                                 unsigned long long* __restrict__ T) {
    __shared__ unsigned long long red[32];
    const int k = blockIdx.x;
    const uint32_t* S0 = Ssub + (size_t)(2 * k) * D;
    const uint32_t* S1 = S0 + D;
    unsigned long long t = 0;
    for (int u = threadIdx.x; u < D; u += blockDim.x) {
        const uint32_t v = S0[u] + S1[u];
        S[(size_t)k * D + u] = v;
        t += v;
    }
    t = warp_sum(t);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long s = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
        T[k] = s;
        n[k] = nsub[2 * k] + nsub[2 * k + 1];
    }
}

// n_k, S_ku, T_k with the additions in global memory: for clusters whose counters
// fit no shared memory (see logml_stats.cuh).
template <class Rows>
__global__ void k_lml_stats_global(Rows csr, const int32_t* __restrict__ labels, int64_t N,
                                   int32_t D, int32_t K, uint32_t* __restrict__ n,
                                   uint32_t* __restrict__ S, unsigned long long* __restrict__ T) {
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t cell = w0; cell < N; cell += nw) {
        const int32_t k = labels[cell];
        if (k < 0 || k >= K) continue;
        const int64_t beg = csr.indptr[cell], end = csr.indptr[cell + 1];
        unsigned long long rowsum = 0;
        for (int64_t e = beg + lane; e < end; e += 32) {
            int32_t u, x;
            csr.get(e, u, x);
            if (x) {
                atomicAdd(&S[(size_t)k * D + u], (uint32_t)x);
                rowsum += (unsigned long long)x;
            }
        }
        rowsum = warp_sum(rowsum);
        if (lane == 0) {
            atomicAdd(&n[k], 1u);
            if (rowsum) atomicAdd(&T[k], rowsum);
        }
    }
}

cudaError_t lml_stats_from_chain(LmlPlan& p, const uint32_t* nsub, const uint32_t* Ssub) {
    k_lml_from_chain<<<p.K, kLmlChainThreads, 0, p.stream>>>(nsub, Ssub, p.D, p.n, p.S, p.T);
    return cudaGetLastError();
}

namespace {

template <class Rows>
cudaError_t lml_count(LmlPlan& p, const Rows& rows, const int32_t* labels) {
    cudaError_t e;
    if ((e = cudaMemsetAsync(p.n, 0, sizeof(uint32_t) * p.K, p.stream))) return e;
    if ((e = cudaMemsetAsync(p.S, 0, sizeof(uint32_t) * (size_t)p.K * p.D, p.stream))) return e;
    if ((e = cudaMemsetAsync(p.T, 0, sizeof(unsigned long long) * p.K, p.stream))) return e;
    if ((e = lml_launch_stats<false>(p, rows, labels, nullptr)) != cudaErrorNotSupported) return e;
    k_lml_stats_global<<<p.num_sms * 4, 256, 0, p.stream>>>(rows, labels, p.N, p.D, p.K, p.n, p.S,
                                                            p.T);
    return cudaGetLastError();
}

}  // namespace

cudaError_t lml_stats_from_csr(LmlPlan& p, const Csr& csr, const int32_t* labels) {
    return lml_count(p, csr, labels);
}

cudaError_t lml_compute_stats(LmlPlan& p) {
    return lml_count(p, PlainCsr{p.indptr, p.cols, p.counts}, p.labels);
}

size_t lml_part_count(int32_t D) { return 2 * (size_t)((D + kLmlGenes - 1) / kLmlGenes); }

cudaError_t lml_terms(LmlPlan& p, double log_alpha, const float* log_beta, double* value_dev,
                      double* grad_alpha_dev, uint32_t* wrap_flag) {
    const double alpha = std::exp(log_alpha), an = alpha + (double)p.N;
    k_lml_terms<<<(p.D + kLmlGenes - 1) / kLmlGenes, kLmlThreads, 0, p.stream>>>(
        p.n, p.S, p.T, log_beta, p.D, p.K, log_alpha, std::lgamma(alpha) - std::lgamma(an),
        alpha * (digamma(alpha) - digamma(an)), value_dev != nullptr, grad_alpha_dev != nullptr,
        p.part, p.ticket, value_dev, grad_alpha_dev, p.common, wrap_flag);
    return cudaGetLastError();
}

cudaError_t lml_backward(LmlPlan& p, const float* log_beta, float* grad_dev) {
    k_lml_backward<<<(p.D + kLmlGenes - 1) / kLmlGenes, kLmlThreads, 0, p.stream>>>(
        p.S, log_beta, p.D, p.K, p.common, grad_dev);
    return cudaGetLastError();
}

}  // namespace dpmm
