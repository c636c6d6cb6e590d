// Cluster statistics n_k, S_ku, T_k of labelled cells for the collapsed log
// marginal likelihood, counted in shared memory.
//
// Every count is one addition into S[k][u].  Done in global memory (one L2
// atomic per entry) the 22.6 M entries of 100,000 x 2,000 cells with K = 25
// took 298-323 us, against 27 us to read them (8 bytes each at 6.8 TB/s): the
// atomics on 50,000 hot words were the bound.  Here a block owns a private
// copy of the counters of a range of clusters ([kg][D] words, all K when they
// fit) and adds them into S with bulk reductions (cp.reduce.async.bulk), which
// the L2 performs a sector at a time: 152 blocks x 200 KB; 323 -> 58 us.
//
// Clusters that do not fit together are split into G contiguous groups of kg
// clusters (a multiple of four, so that every group starts on 16 bytes); a
// block belongs to one group and skips the other groups' cells, whose entries
// it never reads.  The blocks are dealt to the groups in proportion to the
// groups' cells among kSampled evenly spaced labels, at least one each; every
// block works out the same split, and the counts are exact integers whatever
// the split is.
#pragma once

#include <algorithm>

#include "logml.cuh"
#include "tc.cuh"

namespace dpmm {

constexpr int kLmlStatsThreads = 1024;
constexpr int kLmlSampled = 4096;        // labels looked at to weigh the groups
constexpr int kLmlMaxGroups = 32;
constexpr int kLmlFlushWords = 4096;     // one bulk reduction: 16 KB
constexpr int kLmlStatsFixed = 2048;     // static shared memory of the kernel, at most

// Shared-memory plan of one launch: kg clusters per group, G groups; kg = 0:
// one cluster's row does not fit, or there would be more groups than
// kLmlMaxGroups (the caller counts in global memory then).
struct LmlStatsPlan {
    int32_t kg, G;
    size_t smem;
};
inline LmlStatsPlan lml_stats_plan(int32_t D, int32_t K, size_t smem_optin, int num_sms) {
    LmlStatsPlan p{0, 0, 0};
    if (smem_optin <= kLmlStatsFixed + 16) return p;
    const size_t per = 4 * (size_t)D + 16;           // counters, n (padded) and T of a cluster
    const size_t fit = (smem_optin - kLmlStatsFixed - 16) / per;
    int64_t kg = (int64_t)fit >= K ? K : (int64_t)fit & ~(int64_t)3;
    if (kg < 1) return p;
    const int64_t G = (K + kg - 1) / kg;
    if (G > kLmlMaxGroups || G > num_sms) return p;
    p.kg = (int32_t)kg;
    p.G = (int32_t)G;
    p.smem = (size_t)kg * per + 16;
    return p;
}

// smem words [0, words) added into global g (both 16-byte aligned); called by
// the whole block after its writes.
__device__ __forceinline__ void bulk_add_u32(uint32_t* g, const uint32_t* s, int64_t words,
                                             int rotate) {
    tc::fence_async_smem();
    __syncthreads();
    const int64_t whole = words & ~(int64_t)3;
    const int64_t pieces = (whole + kLmlFlushWords - 1) / kLmlFlushWords;
    if (threadIdx.x < 32) {
        // each block starts at another piece, so that the blocks' additions
        // do not all meet on the same lines
        for (int64_t i = threadIdx.x; i < pieces; i += 32) {
            int64_t p = i + rotate % pieces;
            if (p >= pieces) p -= pieces;
            const int64_t w0 = p * kLmlFlushWords;
            const uint32_t n = (uint32_t)min((int64_t)kLmlFlushWords, whole - w0);
            tc::bulk_reduce_add_u32(g + w0, s + w0, n * 4u);
        }
        tc::bulk_commit();
        tc::bulk_wait_all();
    }
    if (threadIdx.x < (unsigned)(words - whole)) {
        const uint32_t v = s[whole + threadIdx.x];
        if (v) atomicAdd(g + whole + threadIdx.x, v);
    }
}

// Two int32 arrays as a caller gives them.
struct PlainCsr {
    const int32_t* indptr;
    const int32_t* cols;
    const int32_t* counts;
    __device__ __forceinline__ void get(int64_t e, int32_t& u, int32_t& x) const {
        u = __ldg(cols + e);
        x = __ldg(counts + e);
    }
};

// kChecked: the arrays were not validated; rows with a decreasing indptr or one
// beyond indptr[N], columns outside [0, D), negative counts and labels outside
// [0, K) are skipped and reported in *flag (bit 0: row or label, bit 1: entry).
// A warp takes up to 32 cells at a time (a lane reads one cell's label and
// bounds; fewer when that would leave the block's warps unevenly loaded), then
// the rows of those in the block's group one after the other, eight entries per
// lane in flight.
template <bool kChecked, class Rows>
__global__ void __launch_bounds__(kLmlStatsThreads, 1)
k_lml_stats(Rows csr, const int32_t* __restrict__ labels, int64_t N, int32_t D, int32_t K,
            int32_t kg, int32_t G, uint32_t* __restrict__ n, uint32_t* __restrict__ S,
            unsigned long long* __restrict__ T, uint32_t* flag) {
    extern __shared__ __align__(16) uint32_t sm[];
    __shared__ int32_t weight[kLmlMaxGroups];
    __shared__ int32_t mine[3];              // group, index in the group, blocks of the group
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    constexpr int nw = kLmlStatsThreads / 32;
    const int64_t words = (int64_t)kg * D;
    uint32_t* sS = sm;
    uint32_t* sn = sS + ((words + 3) & ~(int64_t)3);                              // [kg]
    unsigned long long* sT = reinterpret_cast<unsigned long long*>(sn + ((kg + 1) & ~1));   // [kg]
    for (int64_t i = threadIdx.x; i < words; i += blockDim.x) sS[i] = 0u;
    for (int i = threadIdx.x; i < kg; i += blockDim.x) {
        sn[i] = 0u;
        sT[i] = 0ull;
    }
    if (threadIdx.x < kLmlMaxGroups) weight[threadIdx.x] = 1;
    __syncthreads();
    if (G > 1) {
        const int64_t m = min(N, (int64_t)kLmlSampled);
        for (int64_t i = threadIdx.x; i < m; i += blockDim.x) {
            const int32_t k = labels[i * N / m];
            if (k >= 0 && k < K) atomicAdd(&weight[k / kg], 1);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const int64_t B = gridDim.x;
        int64_t W = 0, cum = 0;
        for (int g = 0; g < G; ++g) W += weight[g];
        for (int g = 0; g < G; ++g) {
            const int64_t b0 = g + (B - G) * cum / W;
            cum += weight[g];
            const int64_t b1 = g + 1 + (B - G) * cum / W;
            if ((int64_t)blockIdx.x >= b0 && (int64_t)blockIdx.x < b1) {
                mine[0] = g;
                mine[1] = (int32_t)(blockIdx.x - b0);
                mine[2] = (int32_t)(b1 - b0);
            }
        }
    }
    __syncthreads();
    const int32_t k0 = mine[0] * kg, k1 = min(K, k0 + kg);
    const int64_t c0 = N * mine[1] / mine[2], c1 = N * (mine[1] + 1) / mine[2];
    const int64_t nnz = kChecked ? (int64_t)csr.indptr[N] : 0;
    const int batch = (int)max((int64_t)1, min((int64_t)32, (c1 - c0) / (8 * nw)));
    for (int64_t base = c0 + (int64_t)batch * w; base < c1; base += (int64_t)batch * nw) {
        const int64_t cell = base + lane;
        int32_t k = -1, beg = 0, len = 0;
        if (lane < batch && cell < c1) {
            k = labels[cell];
            beg = csr.indptr[cell];
            const int32_t end = csr.indptr[cell + 1];
            if (kChecked && (k < 0 || k >= K || beg < 0 || end < beg || end > nnz)) {
                if (mine[0] == 0) atomicOr(flag, 1u);
                k = -1;
            } else {
                len = end - beg;
            }
        }
        unsigned todo = __ballot_sync(0xFFFFFFFFu, k >= k0 && k < k1);
        while (todo) {
            const int q = __ffs(todo) - 1;
            todo &= todo - 1;
            const int32_t kr = __shfl_sync(0xFFFFFFFFu, k, q) - k0;
            const int32_t rb = __shfl_sync(0xFFFFFFFFu, beg, q);
            const int32_t rl = __shfl_sync(0xFFFFFFFFu, len, q);
            uint32_t* dst = sS + (size_t)kr * D;
            unsigned long long sum = 0;
            bool bad = false;
            for (int64_t i0 = lane; i0 < rl; i0 += 32 * 8) {
                int32_t u[8], x[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    u[j] = x[j] = 0;
                    if (i0 + 32 * j < rl) csr.get(rb + i0 + 32 * j, u[j], x[j]);
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    if (kChecked && (u[j] < 0 || u[j] >= D || x[j] < 0)) {
                        bad = true;
                    } else if (x[j]) {
                        atomicAdd(dst + u[j], (uint32_t)x[j]);
                        sum += (unsigned long long)x[j];
                    }
                }
            }
            if (kChecked && __any_sync(0xFFFFFFFFu, bad) && lane == 0) atomicOr(flag, 2u);
            // the row's total: one 32-bit reduction unless a lane's share is large
            if (__all_sync(0xFFFFFFFFu, sum < (1ull << 26)))
                sum = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)sum);
            else
                sum = warp_sum(sum);
            if (lane == 0) {
                atomicAdd(sn + kr, 1u);
                if (sum) atomicAdd(sT + kr, sum);
            }
        }
    }
    __syncthreads();
    bulk_add_u32(S + (size_t)k0 * D, sS, (int64_t)(k1 - k0) * D, blockIdx.x);
    for (int i = threadIdx.x; i < k1 - k0; i += blockDim.x) {
        if (sn[i]) atomicAdd(n + k0 + i, sn[i]);
        if (sT[i]) atomicAdd(T + k0 + i, sT[i]);
    }
}

// Launches k_lml_stats for the plan's N, D, K into its (cleared) n, S, T;
// cudaErrorNotSupported if the counters of one cluster do not fit.
template <bool kChecked, class Rows>
cudaError_t lml_launch_stats(const LmlPlan& p, const Rows& rows, const int32_t* labels,
                             uint32_t* flag) {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    const LmlStatsPlan sp = lml_stats_plan(p.D, p.K, (size_t)optin, p.num_sms);
    if (!sp.kg) return cudaErrorNotSupported;
    // (always the largest, so that concurrent calls never shrink one another's)
    if ((e = cudaFuncSetAttribute(k_lml_stats<kChecked, Rows>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  optin - kLmlStatsFixed)))
        return e;
    // a block per SM, fewer where that would leave a block under 128 cells (its
    // counters are cleared and added whatever it counts)
    const int64_t want = (p.N + 127) / 128 * sp.G;
    const int grid = (int)std::max<int64_t>(sp.G, std::min<int64_t>(p.num_sms, want));
    k_lml_stats<kChecked, Rows><<<grid, kLmlStatsThreads, sp.smem, p.stream>>>(
        rows, labels, p.N, p.D, p.K, sp.kg, sp.G, p.n, p.S, p.T, flag);
    return cudaGetLastError();
}

}  // namespace dpmm
