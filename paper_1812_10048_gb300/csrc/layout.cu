// Device-side preparation of a chain's count matrix (dpmm_init): validation
// of the CSR, the packed entry copy and the blocked copy of the dense-tile
// engine, built from one host-to-device copy of the caller's CSR instead of
// host loops over every entry.
//
// The blocked copy groups the entries by segment (128-cell tile, 64-gene
// chunk) and, inside a segment, by quarter (32-cell row block); inside a
// (segment, quarter) bucket the entries keep their CSR order (cell, then
// gene).  It is therefore a stable partition of the CSR by bucket: a block per
// (tile, quarter) counts its 32 rows' chunks, a warp each, a scan over the rows
// gives every (row, chunk) its first place in the bucket, and
// __match_any_sync on the chunk ranks an entry among the warp's entries of the
// same bucket (a running offset per chunk carries it across iterations).  Every
// segment starts on a 16-byte boundary (padding entries have count 0).
#include <algorithm>
#include <climits>

#include "common.cuh"

namespace dpmm {

namespace {

constexpr int kLayoutThreads = 256;

__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// First decreasing row of indptr.
__global__ void k_check_rows(const int32_t* __restrict__ indptr, int64_t N, CsrCheck* chk) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x)
        if (indptr[i + 1] < indptr[i]) atomicMin(&chk->bad_row, (long long)i);
}

// One pass over the caller's entries: the first with a column outside [0, D) or
// a negative count, the largest count, the sum of all counts, and (entries not
// null) the packed copy, padded with zero entries to a multiple of four.  The
// gene sums, one 64-bit atomic an entry, took 350 of the 370 us a check of
// 9.8 M entries lasted; no gene can reach 2^32 while the sum of all counts does
// not, so they are left to k_gene_sums for the matrices where it does.  VEC:
// 16-byte loads (both arrays 16-byte aligned).
template <bool VEC>
__global__ void __launch_bounds__(kLayoutThreads)
k_check_pack(const int32_t* __restrict__ idx, const int32_t* __restrict__ val, int64_t nnz,
             int32_t D, uint32_t* __restrict__ entries, CsrCheck* chk) {
    __shared__ int smax[kLayoutThreads / 32];
    __shared__ unsigned long long ssum[kLayoutThreads / 32];
    int mx = 0;
    unsigned long long sum = 0;
    const int64_t quads = (nnz + 3) >> 2;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < quads;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t u[4], x[4];
        if (VEC && 4 * i + 4 <= nnz) {
            const int4 a = __ldg(reinterpret_cast<const int4*>(idx) + i);
            const int4 b = __ldg(reinterpret_cast<const int4*>(val) + i);
            u[0] = a.x, u[1] = a.y, u[2] = a.z, u[3] = a.w;
            x[0] = b.x, x[1] = b.y, x[2] = b.z, x[3] = b.w;
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                u[q] = x[q] = 0;
                if (4 * i + q < nnz) {
                    u[q] = __ldg(idx + 4 * i + q);
                    x[q] = __ldg(val + 4 * i + q);
                }
            }
        }
        uint32_t e[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (u[q] < 0 || u[q] >= D || x[q] < 0) {
                atomicMin(&chk->bad_entry, (long long)(4 * i + q));
            } else {
                mx = max(mx, x[q]);
                sum += (unsigned long long)x[q];
            }
            e[q] = ((uint32_t)u[q] << 16) | ((uint32_t)x[q] & 0xFFFFu);
        }
        if (entries) reinterpret_cast<uint4*>(entries)[i] = make_uint4(e[0], e[1], e[2], e[3]);
    }
    for (int o = 16; o; o >>= 1) mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
    sum = warp_sum(sum);
    if ((threadIdx.x & 31) == 0) {
        smax[threadIdx.x >> 5] = mx;
        ssum[threadIdx.x >> 5] = sum;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int m = 0;
        unsigned long long t = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            m = max(m, smax[w]);
            t += ssum[w];
        }
        if (m) atomicMax(&chk->max_count, m);
        if (t) atomicAdd(&chk->total, t);
    }
}

// Per-gene sums (64-bit).
__global__ void __launch_bounds__(kLayoutThreads)
k_gene_sums(const int32_t* __restrict__ idx, const int32_t* __restrict__ val, int64_t nnz,
            unsigned long long* __restrict__ colsum) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz;
         e += (int64_t)gridDim.x * blockDim.x)
        if (val[e]) atomicAdd(colsum + idx[e], (unsigned long long)val[e]);
}

// First gene whose counts sum to 2^32 or more (the statistics are 32-bit).
__global__ void k_check_colsum(const unsigned long long* __restrict__ colsum, int32_t D,
                               CsrCheck* chk) {
    for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < D; u += gridDim.x * blockDim.x)
        if (colsum[u] >= (1ull << 32)) atomicMin(&chk->overflow_gene, u);
}

// Block (tile, quarter): its 32 rows, a warp each.  COUNT: bucket sizes into
// qcount[4 (t C + chunk) + q].  Otherwise each entry is written to its
// bucket's start + its stable rank in the bucket, the segment's padding is
// cleared, and a count beyond the label kernel's lo digit sets the segment's
// flag in qptr.  (One warp for all 32 rows left a chain of dependent loads 32
// rows long: 68,000 x 1,000 88 + 101 us, 30 + 51 us with a warp a row.)
constexpr int kBucketThreads = 1024;

template <bool COUNT>
__global__ void __launch_bounds__(kBucketThreads)
k_tile_bucket(const int32_t* __restrict__ indptr, const uint32_t* __restrict__ entries, int64_t N,
              int32_t C, int32_t* __restrict__ qcount, int32_t* qptr, uint32_t* __restrict__ tent) {
    extern __shared__ int32_t cnt_all[];   // [32 rows][C]: counts, then next places
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int32_t* cnt = cnt_all + (size_t)w * C;
    const int64_t t = blockIdx.x >> 2;
    const int q = (int)(blockIdx.x & 3);
    const int64_t cell = t * 128 + 32 * q + w;
    int64_t e0 = 0, e1 = 0;
    if (cell < N) {
        e0 = indptr[cell];
        e1 = indptr[cell + 1];
    }
    for (int j = lane; j < C; j += 32) cnt[j] = 0;
    __syncwarp();
    uint32_t v = e0 + lane < e1 ? __ldg(entries + e0 + lane) : 0u;
    for (int64_t b = e0; b < e1; b += 32) {
        const bool live = b + lane < e1;
        const int chunk = live ? (int)(v >> 22) : -1;
        v = b + 32 + lane < e1 ? __ldg(entries + b + 32 + lane) : 0u;
        const uint32_t peers = __match_any_sync(0xFFFFFFFFu, chunk);
        if (live && !(peers & lanemask_lt())) cnt[chunk] += __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // counts -> places (a thread per chunk over the 32 rows)
    for (int j = threadIdx.x; j < C; j += blockDim.x) {
        const int64_t bucket = 4 * (t * C + j) + q;
        int32_t run = COUNT ? 0 : qptr[bucket] & kTilePtrMask;
#pragma unroll 8
        for (int r = 0; r < 32; ++r) {
            const int32_t n = cnt_all[(size_t)r * C + j];
            cnt_all[(size_t)r * C + j] = run;
            run += n;
        }
        if (COUNT) {
            qcount[bucket] = run;
        } else if (q == 3) {
            for (const int32_t end = qptr[bucket + 1] & kTilePtrMask; run < end; ++run)
                tent[run] = 0u;      // the segment's padding
        }
    }
    if (COUNT) return;
    __syncthreads();
    v = e0 + lane < e1 ? __ldg(entries + e0 + lane) : 0u;
    for (int64_t b = e0; b < e1; b += 32) {
        const bool live = b + lane < e1;
        const uint32_t e = v;
        const int chunk = live ? (int)(e >> 22) : -1;
        v = b + 32 + lane < e1 ? __ldg(entries + b + 32 + lane) : 0u;
        const uint32_t peers = __match_any_sync(0xFFFFFFFFu, chunk);
        const int rank = __popc(peers & lanemask_lt());
        const int at = live ? cnt[chunk] + rank : 0;
        __syncwarp();
        if (live) {
            if (rank == 0) cnt[chunk] = at + __popc(peers);
            tent[at] = ((uint32_t)(32 * q + w) << 22) | (((e >> 16) & 63u) << 16) | (e & 0xFFFFu);
            uint32_t* flags = reinterpret_cast<uint32_t*>(qptr) + 4 * (t * C + chunk);
            if ((e & 0xFFFFu) > (uint32_t)kTileLoMax) atomicOr(flags + 1, kTileFlag);
        }
        __syncwarp();
    }
}

// Segment starts: each segment's four quarter sizes, padded to a multiple of
// four entries, laid end to end, a thread per segment.  k_tile_sums: per-block
// totals and the longest padded segment (out[1]); k_tile_starts: each block adds
// up the totals before it, then scans its own; out[0] = total entries (padding
// included).
constexpr int kScanThreads = 1024;

__device__ __forceinline__ long long padded_size(const int32_t* __restrict__ qcount, int64_t s,
                                                 int64_t TC, int4* q) {
    *q = s < TC ? reinterpret_cast<const int4*>(qcount)[s] : make_int4(0, 0, 0, 0);
    return ((long long)q->x + q->y + q->z + q->w + 3) & ~3ll;
}

__global__ void __launch_bounds__(kScanThreads)
k_tile_sums(const int32_t* __restrict__ qcount, int64_t TC, long long* __restrict__ sums,
            long long* __restrict__ out) {
    __shared__ unsigned long long part[32];
    __shared__ long long lmax;
    if (threadIdx.x == 0) lmax = 0;
    __syncthreads();
    int4 q;
    const long long n = padded_size(qcount, (int64_t)blockIdx.x * kScanThreads + threadIdx.x, TC, &q);
    const unsigned long long s = warp_sum((unsigned long long)n);
    long long m = n;
    for (int o = 16; o; o >>= 1) m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
    if ((threadIdx.x & 31) == 0) {
        part[threadIdx.x >> 5] = s;
        atomicMax(&lmax, m);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t = 0;
        for (int i = 0; i < kScanThreads / 32; ++i) t += part[i];
        sums[blockIdx.x] = (long long)t;
        atomicMax(out + 1, lmax);
    }
}

__global__ void __launch_bounds__(kScanThreads)
k_tile_starts(const int32_t* __restrict__ qcount, int64_t TC, const long long* __restrict__ sums,
              int32_t* __restrict__ qptr, long long* __restrict__ out) {
    __shared__ unsigned long long part[32], wpart[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned long long before = 0;
    for (int64_t b = threadIdx.x; b < (int64_t)blockIdx.x; b += kScanThreads)
        before += (unsigned long long)sums[b];
    before = warp_sum(before);
    int4 q;
    const int64_t s = (int64_t)blockIdx.x * kScanThreads + threadIdx.x;
    const long long n = padded_size(qcount, s, TC, &q);
    long long x = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 0) part[w] = before;
    if (lane == 31) wpart[w] = (unsigned long long)x;
    __syncthreads();
    long long pos = x - n;
    for (int i = 0; i < kScanThreads / 32; ++i) {
        pos += (long long)part[i];
        if (i < w) pos += (long long)wpart[i];
    }
    if (s >= TC) return;
    auto at = [](long long p) { return (int32_t)min(p, (long long)INT_MAX); };
    reinterpret_cast<int4*>(qptr)[s] =
        make_int4(at(pos), at(pos + q.x), at(pos + q.x + q.y), at(pos + q.x + q.y + q.z));
    if (s == TC - 1) {
        out[0] = pos + n;
        qptr[4 * TC] = at(pos + n);
    }
}

int grid_for(int64_t n, int num_sms) {
    const int64_t b = (n + kLayoutThreads - 1) / kLayoutThreads;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, 8 * (int64_t)num_sms));
}

}  // namespace

cudaError_t launch_check_csr(const int32_t* indptr, const int32_t* idx, const int32_t* val,
                             int64_t N, int64_t nnz, int32_t D, uint32_t* entries, CsrCheck* chk,
                             int num_sms, cudaStream_t st) {
    k_check_rows<<<grid_for(N, num_sms), kLayoutThreads, 0, st>>>(indptr, N, chk);
    if (nnz > 0) {
        const int grid = grid_for((nnz + 3) / 4, num_sms);
        if (((reinterpret_cast<uintptr_t>(idx) | reinterpret_cast<uintptr_t>(val)) & 15) == 0)
            k_check_pack<true><<<grid, kLayoutThreads, 0, st>>>(idx, val, nnz, D, entries, chk);
        else
            k_check_pack<false><<<grid, kLayoutThreads, 0, st>>>(idx, val, nnz, D, entries, chk);
    }
    return cudaGetLastError();
}

cudaError_t launch_gene_sums(const int32_t* idx, const int32_t* val, int64_t nnz, int32_t D,
                             unsigned long long* colsum, CsrCheck* chk, int num_sms,
                             cudaStream_t st) {
    k_gene_sums<<<grid_for(nnz, num_sms), kLayoutThreads, 0, st>>>(idx, val, nnz, colsum);
    k_check_colsum<<<grid_for(D, num_sms), kLayoutThreads, 0, st>>>(colsum, D, chk);
    return cudaGetLastError();
}

template <bool COUNT>
static cudaError_t launch_bucket(const int32_t* indptr, const uint32_t* entries, int64_t N,
                                 int32_t T, int32_t C, int32_t* qcount, int32_t* qptr,
                                 uint32_t* tent, cudaStream_t st) {
    // (the attribute is always that of the widest matrix, D = 65,536, so that
    // concurrent calls never shrink one another's)
    const size_t smem = (size_t)32 * C * sizeof(int32_t);
    cudaError_t e = cudaFuncSetAttribute(k_tile_bucket<COUNT>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         32 * 1024 * (int)sizeof(int32_t));
    if (e != cudaSuccess) return e;
    k_tile_bucket<COUNT><<<(unsigned)(4 * T), kBucketThreads, smem, st>>>(indptr, entries, N, C,
                                                                         qcount, qptr, tent);
    return cudaGetLastError();
}

cudaError_t launch_tile_count(const int32_t* indptr, const uint32_t* entries, int64_t N, int32_t T,
                              int32_t C, int32_t* qcount, cudaStream_t st) {
    return launch_bucket<true>(indptr, entries, N, T, C, qcount, nullptr, nullptr, st);
}

int64_t tile_scan_words(int64_t TC) { return 2 + (TC + kScanThreads - 1) / kScanThreads; }

// scan: tile_scan_words(TC) words, the first two zero; scan[0] = total entries,
// scan[1] = the longest padded segment.
cudaError_t launch_tile_scan(const int32_t* qcount, int64_t TC, int32_t* qptr, long long* scan,
                             cudaStream_t st) {
    const unsigned blocks = (unsigned)((TC + kScanThreads - 1) / kScanThreads);
    k_tile_sums<<<blocks, kScanThreads, 0, st>>>(qcount, TC, scan + 2, scan);
    k_tile_starts<<<blocks, kScanThreads, 0, st>>>(qcount, TC, scan + 2, qptr, scan);
    return cudaGetLastError();
}

cudaError_t launch_tile_scatter(const int32_t* indptr, const uint32_t* entries, int64_t N,
                                int32_t T, int32_t C, int32_t* qptr, uint32_t* tent,
                                cudaStream_t st) {
    return launch_bucket<false>(indptr, entries, N, T, C, nullptr, qptr, tent, st);
}

}  // namespace dpmm
