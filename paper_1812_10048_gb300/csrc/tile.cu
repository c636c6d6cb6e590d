// Dense-tile engine on the 5th-generation tensor cores.
//
// This file holds the tensor-core self-test used to validate the operand
// layout, descriptors and tensor-memory path: C[128][N] = A[128][Kd] B[N][Kd]^T
// for BF16 operands with FP32 accumulation, one CTA.
#include <cuda_bf16.h>
#include <math_constants.h>

#include <type_traits>

#include "common.cuh"
#include "tc.cuh"

namespace dpmm {

constexpr uint32_t kWaitLimit = 1u << 24;   // mbarrier polls before giving up

__host__ __device__ __forceinline__ uint32_t tmem_cols_for(uint32_t n) {
    uint32_t c = 32;
    while (c < n) c <<= 1;
    return c;
}

__global__ void __launch_bounds__(128)
k_debug_tc_gemm(const uint16_t* __restrict__ A, const uint16_t* __restrict__ B, int Kd, int N,
                float* __restrict__ C, int* __restrict__ err) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* sA = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int nch = Kd / 64;
    unsigned char* sB = sA + nch * 16384;
    uint64_t* bar = reinterpret_cast<uint64_t*>(sB + (size_t)nch * N * 128);
    uint32_t* taddr_s = reinterpret_cast<uint32_t*>(bar + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < 128 * Kd; i += blockDim.x) {
        const int r = i / Kd, k = i - r * Kd, ch = k >> 6;
        *reinterpret_cast<uint16_t*>(sA + ch * 16384 + tc::swz_offset(r, k & 63)) = A[i];
    }
    for (int i = tid; i < N * Kd; i += blockDim.x) {
        const int r = i / Kd, k = i - r * Kd, ch = k >> 6;
        *reinterpret_cast<uint16_t*>(sB + (size_t)ch * N * 128 + tc::swz_offset(r, k & 63)) = B[i];
    }
    const uint32_t ncols = tmem_cols_for((uint32_t)N);
    if (tid == 0) tc::mbar_init(bar, 1);
    if (warp == 0) {
        tc::tmem_alloc(taddr_s, ncols);
        tc::tmem_relinquish();
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t taddr = *taddr_s;
    if (tid == 0) {
        const uint32_t idesc = tc::idesc_bf16(128, (uint32_t)N);
        for (int ch = 0; ch < nch; ++ch)
            for (int k = 0; k < 4; ++k) {
                const uint64_t ad = tc::desc_sw128(tc::smem_addr(sA + ch * 16384) + 32 * k);
                const uint64_t bd =
                    tc::desc_sw128(tc::smem_addr(sB + (size_t)ch * N * 128) + 32 * k);
                tc::mma_bf16(taddr, ad, bd, idesc, (ch | k) != 0);
            }
        tc::mma_commit(bar);
    }
    bool ok = tc::mbar_wait(bar, 0, kWaitLimit);
    tc::fence_after_sync();
    if (ok) {
        for (int c0 = 0; c0 < N; c0 += 16) {
            float v[16];
            tc::tmem_ld16(taddr + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
            tc::tmem_ld_wait();
            for (int i = 0; i < 16; ++i) C[(size_t)(warp * 32 + lane) * N + c0 + i] = v[i];
        }
    } else {
        if (lane == 0) atomicExch(err, DPMM_ETIMEOUT);
        tc::mbar_wait(bar, 0, kWaitLimit);   // let in-flight MMAs drain (bounded)
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after_sync();
        tc::tmem_dealloc(taddr, ncols);
    }
}

cudaError_t launch_debug_tc_gemm(const uint16_t* A, const uint16_t* B, int Kd, int N, float* C,
                                 int* err) {
    const size_t smem = 1024 + (size_t)(Kd / 64) * (16384 + (size_t)N * 128) + 64;
    cudaError_t e = cudaFuncSetAttribute(k_debug_tc_gemm,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_debug_tc_gemm<<<1, 128, smem>>>(A, B, Kd, N, C, err);
    return cudaGetLastError();
}


// ===========================================================================
// Dense-tile label engine (eq. 4 third line and eq. 8 on the tensor cores).
//
// Tiles of 128 consecutive cells, 64-gene chunks.  Per (tile, chunk) item the
// CTA zeroes a 128 x 64 BF16 operand in shared memory (128-byte swizzled
// K-major layout) and scatters the counts into it; counts above 255 are split
// into two exact digits, the second of which goes through another stage as a
// second plane, only for items that have such counts (flagged when the blocked
// copy is built).  The B operand (bulk-copied per chunk) holds the centred log
// theta table split into BF16 hi + lo parts, so that one M=128 MMA per 16 genes
// accumulates, in FP32 tensor memory, every cluster and sub-cluster score of
// the 128 cells:
//   TMEM / B column 2k, 2k+1            cluster k, hi and lo part
//   column S0 + 4k + 2r, S0 + 4k + 2r + 1  sub-cluster (k, r), hi and lo part
// with S0 = 2K rounded up to 16 and Ntot = (S0 + 4K) rounded up to 16 <= 256
// (K <= 40).  Centring subtracts m_u, the mean of the 3K log theta values of
// gene u, from every row; it shifts all of a cell's scores by the same
// sum_u x_u m_u, which leaves the Gumbel argmax, the eq. 8 draw and log q_i
// unchanged.  The epilogue (two groups of four warps, a thread of each per
// cell) takes the Gumbel-max over the cell's K scores and the eq. 8 sub-label
// from the two sub-cluster scores of the chosen cluster, writes the cell state
// and adds log q_i to its cluster's accumulator; the statistics are counted
// afterwards from the blocked copy (k_stats_tile).
// ===========================================================================

constexpr int kNtotMax = 256;
constexpr uint32_t kBChunkBytes = kNtotMax * 128;   // one chunk of B in global memory

__host__ __device__ __forceinline__ bool tile_usable(int K) {
    return K >= 1 && K <= kTileMaxK;
}
__host__ __device__ __forceinline__ int tile_s0(int K) { return (2 * K + 15) & ~15; }
__host__ __device__ __forceinline__ int tile_ntot(int K) { return (tile_s0(K) + 4 * K + 15) & ~15; }

// BF16 takes every log theta that a draw or a caller can give (FP16 ends at
// 65,504, which drawn values pass from beta = 2.8e-4 down), and its coarse hi
// part leaves the FP32 accumulator's additions nearly exact where few clusters
// meet many counts: own-cluster scores of 4,000 cells x 3,000 genes, K = 3,
// libraries of 3,000, differ from 64 bits by 3.8e-3 rms, with FP16 hi + lo by
// 1.3e-2.
__device__ __forceinline__ uint16_t bf16_bits_rn(float f) {
    const __nv_bfloat16 h = __float2bfloat16_rn(f);
    return *reinterpret_cast<const uint16_t*>(&h);
}
__device__ __forceinline__ float bf16_value(uint16_t b) {
    return __uint_as_float((uint32_t)b << 16);
}

// B operand of one sweep: block (c, q, b) fills rows rb q .. rb q + rb - 1 of
// chunk c (genes 64c .. 64c + 63) of chain b (rb = 16 rows for one chain, 64
// for a batch).  Each block reads the chunk's 3K log theta values per gene
// into shared memory with all of a thread's loads in flight at once, then
// forms m_u and its rows from there.  In a step (force = 0) the blocks of
// chain b first clear its main S-bar rows.
constexpr int kBuildThreads = 256;
constexpr int kBuildStage = 3 * kTileMaxK * 64 / kBuildThreads;   // values per thread

template <class Tab>
__global__ void __launch_bounds__(kBuildThreads)
k_build_b(const __grid_constant__ Tab tab, int32_t force, int32_t rb) {
    __shared__ float sv[3 * kTileMaxK * 64];   // [3K][64]: row j of gene 64c + g
    __shared__ float part[4][64];
    __shared__ float m[64];
    const ChainArgs& ch = tab[blockIdx.z];
    const DevScalars* sc = ch.sc;
    const float* __restrict__ Lc = ch.Lc;
    const float* __restrict__ Ls = ch.Ls;
    unsigned char* __restrict__ B = ch.tile_B;
    uint32_t* __restrict__ Ssub = ch.Ssub;
    const int32_t D = ch.D, kmax = ch.kmax;
    const int K = sc->K;
    if (!force) {
        // the main S-bar rows are dead from here until the statistics kernel
        // adds this sweep's counts into them: clear rows 0 .. 2K-1
        const int64_t words = (int64_t)2 * K * D;
        const int64_t nthr = (int64_t)gridDim.x * gridDim.y * blockDim.x;
        for (int64_t i = ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x;
             i < words; i += nthr)
            Ssub[i] = 0u;
    }
    if (!ch.tile_enabled || !tile_usable(K) || (!force && !sc->tile_used)) return;
    const int c = blockIdx.x;
    if (c >= ch.tile_C) return;
    const int S0 = tile_s0(K), Ntot = tile_ntot(K);
    if ((int)blockIdx.y * rb >= Ntot) return;
    // rows j < K: cluster j (log theta); K <= j < 3K: sub-cluster (j - K) / 2,
    // r = (j - K) % 2 (log theta-bar).  Every load first, then the stores.
    const int n3 = 3 * K * 64;
    float v[kBuildStage];
#pragma unroll
    for (int r = 0; r < kBuildStage; ++r) {
        const int i = threadIdx.x + kBuildThreads * r;
        const int j = i >> 6, u = c * 64 + (i & 63);
        v[r] = 0.0f;
        if (i < n3 && u < D)
            v[r] = j < K ? __ldg(Lc + (size_t)u * kmax + j) : __ldg(Ls + (size_t)u * kmax * 2 + (j - K));
    }
#pragma unroll
    for (int r = 0; r < kBuildStage; ++r) {
        const int i = threadIdx.x + kBuildThreads * r;
        if (i < n3) sv[i] = v[r];
    }
    __syncthreads();
    {
        // m_u: 4 threads per gene, each a quarter of the 3K rows, fixed order
        const int g = threadIdx.x & 63, qq = threadIdx.x >> 6;
        float s = 0.0f;
        if (c * 64 + g < D)
            for (int j = qq; j < 3 * K; j += 4) s += sv[j * 64 + g];
        part[qq][g] = s;
        __syncthreads();
        if (threadIdx.x < 64)
            m[g] = ((part[0][g] + part[1][g]) + (part[2][g] + part[3][g])) / (float)(3 * K);
        __syncthreads();
    }
    unsigned char* dst = B + (size_t)c * kBChunkBytes;
    for (int i = blockIdx.y * rb * 64 + threadIdx.x; i < min(Ntot, (int)(blockIdx.y + 1) * rb) * 64;
         i += blockDim.x) {
        const int row = i >> 6, g = i & 63, u = c * 64 + g;
        float L = 0.0f;
        int part = 0;
        bool live = u < D;
        if (row < 2 * K) {
            part = row & 1;
            L = sv[(row >> 1) * 64 + g];
        } else if (row >= S0 && row < S0 + 4 * K) {
            const int q = row - S0;
            part = q & 1;
            L = sv[(K + (q >> 1)) * 64 + g];
        } else {
            live = false;
        }
        uint16_t v = 0;
        if (live) {
            const float d = L - m[g];
            const uint16_t hi = bf16_bits_rn(d);
            v = part ? bf16_bits_rn(d - bf16_value(hi)) : hi;
        }
        *reinterpret_cast<uint16_t*>(dst + tc::swz_offset((uint32_t)row, (uint32_t)g)) = v;
    }
}


// Chains the dense-tile engine labels in this launch.  Their tiles form one
// list (chain order) dealt round-robin to the CTAs: chain b's tiles handled
// by this CTA are first, first + gridDim.x, ... (cnt of them), where off is
// the number of listed tiles before chain b.
__device__ __forceinline__ void chain_tiles(int64_t off, int T, int& first, int& cnt) {
    const int G = (int)gridDim.x;
    const int skip = off ? (int)((uint64_t)off % (uint32_t)G) : 0;   // CTA of the first tile
    first = (int)blockIdx.x - skip;
    if (first < 0) first += G;
    cnt = first < T ? (T - 1 - first) / G + 1 : 0;
}

// Warp roles of the pipelined engine (32 warp numbers; 20, 24 and 28 idle):
//   warps 0-7   epilogue, two halves of four warps over the same 128 cells
//               (warp w reads TMEM lanes 32 (w % 4) ..): each half takes every
//               other 8-cluster column group of the Gumbel-max, then (the
//               winner exchanged) every other block of sub-cluster columns,
//               and finishes the cells whose sub-cluster columns it met
//   warps from 8 with w % 4 != 0  producers, up to four sets of four warps
//               taking items in turn; warp q of a set densifies rows 32q ..
//               32q + 31 of its item (the entries of one quarter) from the
//               staged segment, so the four warps never wait on one another
//   warp 8      issues the MMAs
//   warp 12     segment loader: bulk-copies each item's entries into a ring,
//               one lane per producer set, reading the segment table a round
//               ahead.  The items lie end to end in the ring: a few deep cells
//               make one segment several times the mean, and slots of that
//               size left room for fewer A stages (1.3 M x 2,000 with 2% deep
//               cells: 1,714 us with slots, 1,611 us)
//   warp 16     lane 0 bulk-copies the B operand of each chunk into its ring
// The roles that feed the tensor core are alone on their scheduler (w % 4 = 0)
// but for two epilogue warps: each item costs them the latency of a chain of
// instructions.
// Every role walks the same sequence of items (tile, chunk): the chains in
// order, this CTA's tiles of each chain in pairs, the chunks, and for each chunk
// the tiles of the pair, so that one copy of a chunk's B operand serves both
// tiles (B, the same for every CTA, is otherwise the largest stream from the
// L2: 32 KB an item at K = 40, against 4 KB of entries).  A tile's chunks are
// accumulated in the same order as without the pairing.  The accumulators are
// nAcc slots of TMEM (512 columns / the score columns, at most four) that the
// tiles take in turn.
// Hand-offs are mbarriers: ent_full / ent_free (segment slots), a_full (the
// four producer warps -> MMA), b_full (B copy -> MMA), stage_free, b_free (MMA
// commit -> producers, B loader), acc_full (MMA -> epilogue) / acc_empty
// (epilogue -> MMA).  The A operand is written by ordinary stores, each
// producer lane's proxy fence before its arrival makes them visible to the MMA.
// Every wait is bounded; a timeout records DPMM_ETIMEOUT, every role leaves
// its loop, and each role that issued asynchronous work waits (bounded) for
// it before the block exits.
constexpr int kMaxStages = 8;        // A stages
constexpr uint32_t kStageBytes = 16384;   // 128 cells x 64 genes x 2 bytes
constexpr int kMaxBStages = 4;
constexpr int kMaxAcc = 4;
constexpr int kPair = 2;             // tiles that share a chunk's B operand
constexpr int kMaxESlots = 16;
constexpr int kEpiWarps = 8;
constexpr int kProdSets = 4;        // producer sets (4 warps each) on alternate items
constexpr int kProdWarp0 = 8;
constexpr int kMmaWarp = 8, kELoadWarp = 12, kBLoadWarp = 16;
constexpr int kTileThreadsP = (kProdWarp0 + (4 * kProdSets + 2) / 3 * 4) * 32;
constexpr int kBarEpi = 1, kBarHalf = 2;   // kBarHalf + h: one half
constexpr int kEpiGroups = (kTileMaxK + 15) / 16;   // 8-cluster groups of a half
constexpr int kSmallBytes = 8192;
constexpr int kScatterDefault = 12;  // entries per producer lane and batch (tunable: 8, 12, 16)

// A digit of a count, x & 255 or x & 0xFF00: at most eight significant bits, so
// that its FP32 pattern truncates exactly to BF16.
__device__ __forceinline__ uint16_t digit_bits(uint32_t v) {
    return (uint16_t)(__float_as_uint((float)v) >> 16);
}

// One producer warp's share of a staged segment into its quarter q of the A stage
// (kPlanes 1: the lo digits into A, 2: the hi ones into H, 3: both): the 16-byte
// groups that hold entries [i0, i1), kScatter entries per lane in flight.  A group at
// either end may hold
// entries of a neighbouring quarter, which their rows tell apart, and the
// segment's padding, whose counts are 0.  An entry row << 22 | gene << 16 | count
// shifted right by 15 has its row and gene at the bytes row * 128 + gene * 2 of
// the stage; the 128-byte swizzle exchanges bits 4-6 with the row's low bits.
template <int kPlanes, int kScatter>
__device__ __forceinline__ void scatter_entries(const uint32_t* ring, int i0, int i1, int q,
                                                int lane, unsigned char* A, unsigned char* H) {
    constexpr uint32_t mask = kPlanes == 1 ? 0xFFu : kPlanes == 2 ? 0xFF00u : 0xFFFFu;
    constexpr int U = kScatter / 4;
    const uint4* ring4 = reinterpret_cast<const uint4*>(ring);
    const int j1 = (i1 + 3) >> 2;
    for (int j = (i0 >> 2) + lane; j < j1; j += 32 * U) {
        uint4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            v[u] = j + 32 * u < j1 ? ring4[j + 32 * u] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t e[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t x = e[k] & mask, t = e[k] >> 15;
                if (x && (e[k] >> 27) == (uint32_t)q) {
                    const uint32_t at = (t & 0x3FFEu) ^ ((t >> 3) & 0x70u);
                    if (kPlanes & 1)
                        *reinterpret_cast<uint16_t*>(A + at) = digit_bits(x & 0xFFu);
                    if (kPlanes == 2 || (kPlanes == 3 && x > 0xFFu))
                        *reinterpret_cast<uint16_t*>(H + at) = digit_bits(x & 0xFF00u);
                }
            }
        }
    }
}

// A producer warp's quarter of an A stage, cleared.
__device__ __forceinline__ void clear_quarter(unsigned char* A, int q, int lane) {
    uint4* zl = reinterpret_cast<uint4*>(A + q * 4096);
#pragma unroll
    for (int i = 0; i < 8; ++i) zl[lane + 32 * i] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
}

// A chain's tiles for one CTA: first, first + gridDim.x, ... (cnt of them).
struct TileJob {
    int32_t b, first, cnt;
    uint32_t k;      // K | second planes << 16
    __device__ __forceinline__ int K() const { return (int)(k & 0xFFFFu); }
    __device__ __forceinline__ bool planes() const { return (k >> 16) & 1u; }
};

// The jobs of this CTA in chain order (called by the whole block; jobs, at most
// kMaxTileJobs by the host's choice of runs, and scratch, 70 words: shared memory).
// A batch's chains are read side by side, one thread each: the roles
// used to walk the table themselves, three dependent loads a chain for each of
// them.
template <class Tab>
__device__ __forceinline__ void list_jobs(const Tab& tab, bool dbg, TileJob* jobs, int& njobs,
                                          uint32_t& total, int& ntot_max, int& lslot_max,
                                          int& lmean_max, bool& planes_any, int& C,
                                          int32_t* scratch) {
    if (tab.n() == 1) {     // one chain: every thread by itself
        const ChainArgs& ch = tab[0];
        const int K = ch.sc->K, used = ch.sc->tile_used;
        if (!ch.tile_enabled || !tile_usable(K) || !(dbg || used)) return;
        TileJob job{0, 0, 0, (uint32_t)K | (ch.max_count > kTileLoMax ? 1u << 16 : 0u)};
        chain_tiles(0, ch.tile_T, job.first, job.cnt);
        if (!job.cnt) return;
        if (threadIdx.x == 0) jobs[0] = job;
        njobs = 1;
        C = ch.tile_C;
        total = (uint32_t)job.cnt * (uint32_t)C;
        ntot_max = tile_ntot(K);
        lslot_max = max(4, ch.tile_Lslot);
        lmean_max = max(4, ch.tile_Lmean);
        planes_any = job.planes();
        return;
    }
    int32_t *wtiles = scratch, *wjobs = wtiles + 32, *smax = wjobs + 32;   // [32], [32], [6]
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = (int)(blockDim.x >> 5);
    if (tid < 6) smax[tid] = 0;      // tiles, ntot, lslot, planes, lmean, C
    int64_t tiles_before = 0;
    for (int b0 = 0; b0 < tab.n(); b0 += blockDim.x) {
        const int b = b0 + tid;
        int T = 0, lslot = 0, lmean = 0;
        uint32_t k = 0;
        if (b < tab.n()) {
            const ChainArgs& ch = tab[b];
            const bool enabled = ch.tile_enabled;
            const int K = ch.sc->K, used = ch.sc->tile_used;
            if (enabled && tile_usable(K) && (dbg || used)) {
                T = ch.tile_T;
                lslot = ch.tile_Lslot;
                lmean = ch.tile_Lmean;
                k = (uint32_t)K | (ch.max_count > kTileLoMax ? 1u << 16 : 0u);
            }
        }
        int x = T;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wtiles[w] = x;
        __syncthreads();
        int64_t off = tiles_before + x - T;
        for (int i = 0; i < nw; ++i) {
            if (i < w) off += wtiles[i];
            tiles_before += wtiles[i];
        }
        int first = 0, cnt = 0;
        if (T) chain_tiles(off, T, first, cnt);
        const unsigned own = __ballot_sync(0xFFFFFFFFu, cnt > 0);
        if (lane == 0) wjobs[w] = __popc(own);
        __syncthreads();
        int pos = njobs + __popc(own & ((1u << lane) - 1u));
        for (int i = 0; i < nw; ++i) {
            if (i < w) pos += wjobs[i];
            njobs += wjobs[i];
        }
        if (cnt > 0) {
            jobs[pos] = TileJob{b, first, cnt, k};
            atomicAdd(&smax[0], cnt);
            atomicMax(&smax[1], tile_ntot((int)(k & 0xFFFFu)));
            atomicMax(&smax[2], lslot);
            atomicMax(&smax[4], lmean);
            if (k >> 16) smax[3] = 1;
            smax[5] = tab[b].tile_C;     // (the chains share D)
        }
        __syncthreads();
    }
    C = smax[5];
    total = (uint32_t)smax[0] * (uint32_t)C;
    ntot_max = smax[1];
    lslot_max = max(4, smax[2]);
    lmean_max = max(4, smax[4]);
    planes_any = smax[3] != 0;
}

// A 64-bit sum kept as two 32-bit words in shared memory (the 32-bit shared
// atomics are single instructions, the 64-bit one is a loop).
__device__ __forceinline__ void add_words64(uint32_t* w, unsigned long long v) {
    const uint32_t lo = (uint32_t)v;
    const uint32_t old = atomicAdd(w, lo);
    const uint32_t hi = (uint32_t)(v >> 32) + (old + lo < old ? 1u : 0u);
    if (hi) atomicAdd(w + 1, hi);
}

// dbg: optional [N][3K] centred scores of a single chain (no state or
// statistics writes).
// kScatter: row entries a producer lane loads per batch; stages_pref: 2 to
// keep two A stages to every producer set rather than four sets of one.
template <class Tab, int kScatter>
__global__ void __launch_bounds__(kTileThreadsP, 1)
k_assign_tc(const __grid_constant__ Tab tab, float* dbg_out, int64_t smem_bytes,
            int32_t stages_pref) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool dbg = dbg_out != nullptr;
    // this CTA's chains with their tiles, and the largest operand / segment
    TileJob* jobs = reinterpret_cast<TileJob*>(base);
    uint32_t total = 0;   // items of this block
    int njobs = 0, ntot_max = 0, lslot_max = 4, lmean_max = 4, C = 0;
    bool planes_any = false;
    list_jobs(tab, dbg, jobs, njobs, total, ntot_max, lslot_max, lmean_max, planes_any, C,
              reinterpret_cast<int32_t*>(smem_raw + smem_bytes - 512));
    if (total == 0) return;
    base += (njobs * (int)sizeof(TileJob) + 1023) & ~1023;
    // shared-memory plan (identical in every thread): A stages, B stages,
    // segments, then the small area.  (In 32-bit integers: 64-bit divisions here
    // and in the roles' starts cost a block 1 us.)
    const int b_slot = (ntot_max * 128 + 1023) & ~1023;
    const int e_max = min(lslot_max, 1 << 20) * 4, e_mean = min(lmean_max, 1 << 20) * 4;
    const int avail = (int)(smem_bytes - (base - smem_raw)) - kSmallBytes;
    // Producer sets and A stages, the most that fit beside a segment ring for two
    // items of a set and the longest segment.  A set takes every nsets-th item
    // and always meets the same stages and slots, so nsets divides nS and nE:
    // slot g % nE is then refilled for item g only after the same set consumed
    // item g - nE, and a set's parity wait can never be two phases ahead.  Two
    // stages a set let it fill one while the MMAs read the other.
    auto ring_left = [&](int stages, int b_stages) {
        return avail - stages * (int)kStageBytes - b_stages * b_slot;
    };
    auto fit = [&](int sets, int stages) {
        return ring_left(stages, 2) >= max(e_max, 2 * sets * e_mean);
    };
    // Four sets of two stages against three: 68,000 x 1,000, K = 10 44 and 48 us,
    // 1.3 M x 2,000, K = 40 1,611 and 1,711; three of two against four of one:
    // 24 datasets 81 and 95.
    int nsets = 2, nS = 2;
    if (fit(4, 8)) nsets = 4, nS = 8;
    else if (fit(3, 6)) nsets = 3, nS = 6;
    else if (stages_pref != 2 && fit(4, 4)) nsets = 4, nS = 4;
    else if (fit(2, 4)) nsets = 2, nS = 4;
    // more than two B stages only where they leave room for twelve segments
    int nB = 2;
    while (nB < kMaxBStages && ring_left(nS, nB + 1) >= max(e_max, 12 * e_mean)) ++nB;
    const int e_ring = ring_left(nS, nB) & ~15;
    // An item's two planes filled and multiplied together, where every set of four has
    // two stages and an item's MMAs are short (N <= 128 columns: the MMA warp's waits
    // are what an item costs); else the second plane follows the first.  68,000 x 1,000,
    // libraries of 8,000: K = 5 67 -> 55 us, K = 20 (N = 128) 70 -> 60; K = 40 (N = 240)
    // 87 us one after the other, 90 together, 1.3 M x 2,000 1,611 and 1,743.  For a
    // batch one after the other: 24 datasets 80 us, 85 together.
    const bool both = std::is_same<Tab, TabV>::value && nsets == 4 && nS == 8 && ntot_max <= 128;
    // items in the ring at most: as many as it nearly always has room for, so
    // that a round seldom waits for more than its own slots
    // (fixed slots for the longest segment where two a set fit: a round of the
    // loader is shorter then; 68,000 x 1,000 44.3 us, 45.7 in the ring)
    const bool fixed = e_ring >= 2 * nsets * e_max;
    const int e_item = fixed ? e_max : e_mean + e_mean / 4;
    const int nE = min(kMaxESlots / nsets, max(2, e_ring / (e_item * nsets))) * nsets;
    if (e_ring < e_max) {
        if (tid == 0) atomicExch(&tab[0].sc->error, DPMM_ECAPACITY);
        return;
    }
    const uint32_t ldN = ((uint32_t)ntot_max + 31u) & ~31u;        // TMEM columns of a slot
    const uint32_t nAcc = min((uint32_t)kMaxAcc, 512u / ldN);      // >= 2
    unsigned char* A_base = base;
    unsigned char* B_base = A_base + nS * kStageBytes;
    unsigned char* E_base = B_base + nB * b_slot;
    unsigned char* small = E_base + e_ring;
    small = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(small) + 15) & ~(uintptr_t)15);
    int4* meta = reinterpret_cast<int4*>(small);                   // [kMaxESlots] quarter ends
    uint64_t* a_full = reinterpret_cast<uint64_t*>(meta + kMaxESlots);   // [kMaxStages]
    uint64_t* stage_free = a_full + kMaxStages;                     // [kMaxStages]
    uint64_t* b_full = stage_free + kMaxStages;                     // [kMaxBStages]
    uint64_t* b_free = b_full + kMaxBStages;                        // [kMaxBStages]
    uint64_t* ent_full = b_free + kMaxBStages;                      // [kMaxESlots]
    uint64_t* ent_free = ent_full + kMaxESlots;                     // [kMaxESlots]
    uint64_t* acc_full = ent_free + kMaxESlots;                     // [kMaxAcc]
    uint64_t* acc_empty = acc_full + kMaxAcc;                       // [kMaxAcc]
    uint64_t* drain = acc_empty + kMaxAcc;                          // [1]
    uint32_t* taddr_s = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* err = reinterpret_cast<volatile int*>(taddr_s + 1);
    int* stop = const_cast<int*>(err) + 1;                          // [2]
    int32_t* stage_hi = stop + 2;                                   // [kMaxStages]
    int32_t* slot_off = stage_hi + kMaxStages;                      // [kMaxESlots] ring offsets
    int32_t* meta_hi = slot_off + kMaxESlots;                       // [kMaxESlots]
    float* spi = reinterpret_cast<float*>(meta_hi + kMaxESlots);    // [K]
    float* slw = spi + kTileMaxK;                                   // [4K]
    float* xbest = slw + 4 * kTileMaxK;                             // [2][half][128]
    int* xc = reinterpret_cast<int*>(xbest + 512);                  // [2][half][128]
    uint32_t* wsq = reinterpret_cast<uint32_t*>(xc + 512);          // [4][K][2] sum log q

    if (tid == 0) {
        *err = 0;
        stop[0] = stop[1] = 0;
        for (int i = 0; i < kMaxStages; ++i) {
            tc::mbar_init(&a_full[i], 4);   // four producer warps
            tc::mbar_init(&stage_free[i], 1);
        }
        for (int i = 0; i < kMaxBStages; ++i) {
            tc::mbar_init(&b_full[i], 1);
            tc::mbar_init(&b_free[i], 1);
        }
        tc::mbar_init(drain, 1);
        for (int i = 0; i < kMaxESlots; ++i) {
            tc::mbar_init(&ent_full[i], 1);
            tc::mbar_init(&ent_free[i], 4);
        }
        for (int i = 0; i < kMaxAcc; ++i) {
            tc::mbar_init(&acc_full[i], 1);
            tc::mbar_init(&acc_empty[i], 2);   // the epilogue's halves
        }
        tc::fence_mbar_init();
    }
    if (warp == 0) {
        tc::tmem_alloc(taddr_s, 512);
        tc::tmem_relinquish();
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *taddr_s;

    if (warp >= kProdWarp0 && (warp & 3)) {
        // ---------------- producers ----------------
        const int pi = (warp - kProdWarp0) / 4 * 3 + (warp & 3) - 1, set = pi >> 2, q = pi & 3;
        // this set's stages and slots, one after the other
        uint32_t st = (uint32_t)set % (uint32_t)nS, sph = 1u;   // parity of the stage's last use
        uint32_t es = (uint32_t)set % (uint32_t)nE, eph = 0u;
        uint32_t g = set < nsets ? (uint32_t)set : total;
        auto next_stage = [&]() {
            if ((st += (uint32_t)nsets) >= (uint32_t)nS) {
                st -= (uint32_t)nS;
                sph ^= 1u;
            }
        };
        bool ok = true;
        for (; g < total && ok; g += (uint32_t)nsets) {
            int i0 = 0, i1 = 0, hi = 0;
            const uint32_t* ring = nullptr;
            // the item's plane of lo digits, then, if it has counts above 255, that of
            // its hi digits in the set's next stage, a stage like any other: the MMA
            // warp goes on to other items while it fills.  (Stages of its own that the
            // MMA warp had to drain before they were used again: 68,000 x 1,000 step
            // 96 -> 89 us, 1.3 M x 2,000 2,430 -> 2,260 us.)
            for (int pl = 0; pl <= hi; ++pl) {
                unsigned char* A = A_base + st * kStageBytes;
                // (at a stage's first use the parity of the phase before the first)
                ok = tc::mbar_wait(&stage_free[st], sph, kWaitLimit);
                if (__all_sync(0xFFFFFFFFu, ok)) {
                    clear_quarter(A, q, lane);      // while the segment is still on its way
                    if (!pl) ok = tc::mbar_wait(&ent_full[es], eph, kWaitLimit);
                }
                const bool mine = ok;
                ok = __all_sync(0xFFFFFFFFu, ok && *err == 0);
                if (!ok) {
                    if (lane == 0 && !mine) *err = DPMM_ETIMEOUT;
                    break;
                }
                if (!pl) {
                    const int4 mt = meta[es];
                    i0 = q == 0 ? 0 : q == 1 ? mt.x : q == 2 ? mt.y : mt.z;
                    i1 = q == 0 ? mt.x : q == 1 ? mt.y : q == 2 ? mt.z : mt.w;
                    if (planes_any) hi = meta_hi[es];
                    ring = reinterpret_cast<const uint32_t*>(E_base + slot_off[es]);
                    if (both && hi) {
                        // both planes at once; the second stage is full when the first is
                        const uint32_t st1 = st;
                        next_stage();
                        ok = tc::mbar_wait(&stage_free[st], sph, kWaitLimit);
                        const bool mine2 = ok;
                        ok = __all_sync(0xFFFFFFFFu, ok && *err == 0);
                        if (!ok) {
                            if (lane == 0 && !mine2) *err = DPMM_ETIMEOUT;
                            break;
                        }
                        unsigned char* H = A_base + st * kStageBytes;
                        clear_quarter(H, q, lane);
                        scatter_entries<3, kScatter>(ring, i0, i1, q, lane, A, H);
                        tc::fence_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            if (q == 0) stage_hi[st1] = hi;
                            tc::mbar_arrive(&a_full[st]);
                            tc::mbar_arrive(&a_full[st1]);
                            tc::mbar_arrive(&ent_free[es]);
                        }
                        next_stage();
                        break;
                    }
                    scatter_entries<1, kScatter>(ring, i0, i1, q, lane, A, nullptr);
                } else {
                    scatter_entries<2, kScatter>(ring, i0, i1, q, lane, nullptr, A);
                }
                tc::fence_async_smem();
                __syncwarp();
                if (lane == 0) {
                    if (planes_any && q == 0 && !pl) stage_hi[st] = hi;
                    tc::mbar_arrive(&a_full[st]);
                    if (pl == hi) tc::mbar_arrive(&ent_free[es]);
                }
                next_stage();
            }
            if ((es += (uint32_t)nsets) >= (uint32_t)nE) {
                es -= (uint32_t)nE;
                eph ^= 1u;
            }
        }
    } else if (warp == kELoadWarp) {
        // ---------------- segment loader ----------------
        // the five quarter pointers of a job's item j and (last) its second-plane flag
        auto seg_ptrs = [&](const TileJob& job, uint32_t j, int32_t (&p)[6]) {
            const uint32_t Cu = (uint32_t)C;
            const uint32_t pr = j / (kPair * Cu);          // pair, then chunk, then tile
            const uint32_t m = min((uint32_t)kPair, (uint32_t)job.cnt - kPair * pr);
            const uint32_t r = j - pr * kPair * Cu, ci = r / m;
            const int64_t sgm =
                ((int64_t)job.first + (int64_t)(kPair * pr + (r - ci * m)) * gridDim.x) *
                    (int64_t)Cu + ci;
            const int32_t* ptr = tab[job.b].tile_ptr + 4 * sgm;
#pragma unroll
            for (int k = 0; k < 5; ++k) p[k] = __ldg(ptr + k);
            p[5] = p[1] < 0;
            p[1] &= kTilePtrMask;
        };
        // an item's segment into slot es, at byte `at` of the ring
        auto issue = [&](const uint32_t* ent, const int32_t (&p)[6], uint32_t es, int32_t at) {
            const int32_t len = p[4] - p[0];
            slot_off[es] = at;
            meta[es] = make_int4(p[1] - p[0], p[2] - p[0], p[3] - p[0], len);
            if (planes_any) meta_hi[es] = p[5];
            if (len) {
                tc::mbar_arrive_expect_tx(&ent_full[es], (uint32_t)len * 4u);
                tc::bulk_g2s(E_base + at, ent + p[0], (uint32_t)len * 4u, &ent_full[es]);
            } else {
                tc::mbar_arrive(&ent_full[es]);
            }
        };
        if (fixed) {
            // Lane l < nsets loads for set l by itself, so that a set that is late
            // (second planes) keeps no other's entries back: the next item's pointers
            // are read one item ahead, its slot is polled.  (In rounds of all sets
            // 68,000 x 1,000, K = 10 44.1 us, 42.7 so; libraries of 1,500, K = 16, a
            // step 111 and 109.)
            uint32_t g = lane < nsets ? (uint32_t)lane : total;     // next item
            uint32_t es = (uint32_t)lane, eph = 0, n = 0;           // its slot; items started
            int jn = -1;                                            // its job, whose items are
            uint32_t j0 = 0, jend = 0;                              // j0 .. jend - 1
            int32_t cur[6], nxt[6];
            auto fetch = [&](uint32_t item, int32_t (&p)[6]) {
                while (item >= jend && jn + 1 < njobs) {
                    j0 = jend;
                    jend += (uint32_t)jobs[++jn].cnt * (uint32_t)C;
                }
                if (item < total) seg_ptrs(jobs[jn], item - j0, p);
            };
            int jcur = 0;
            if (g < total) {
                fetch(g, cur);
                jcur = jn;
                fetch(g + (uint32_t)nsets, nxt);
            }
            const uint32_t* ent = tab[jobs[jcur].b].tile_ent;
            uint32_t polls = 0;
            while (__any_sync(0xFFFFFFFFu, g < total)) {
                const bool ready = g < total && tc::mbar_test(&ent_free[es], eph ^ 1u);
                if (ready) {
                    issue(ent, cur, es, (int32_t)(es * (uint32_t)e_max));
                    ++n;
                    g += (uint32_t)nsets;
                    if ((es += (uint32_t)nsets) >= (uint32_t)nE) {
                        es -= (uint32_t)nE;
                        eph ^= 1u;
                    }
#pragma unroll
                    for (int k = 0; k < 6; ++k) cur[k] = nxt[k];
                    if (jn != jcur) {
                        jcur = jn;
                        ent = tab[jobs[jn].b].tile_ent;
                    }
                    fetch(g + (uint32_t)nsets, nxt);
                }
                polls = __any_sync(0xFFFFFFFFu, ready) ? 0u : polls + 1u;
                if (polls >= kWaitLimit || __any_sync(0xFFFFFFFFu, *err != 0)) {
                    if (lane == 0 && *err == 0) *err = DPMM_ETIMEOUT;
                    break;
                }
            }
            // every started copy has landed before the block can exit
            const uint32_t per = (uint32_t)(nE / nsets);
            for (uint32_t q = n > per ? n - per : 0u; q < n; ++q)
                tc::mbar_wait(&ent_full[(uint32_t)lane + (uint32_t)nsets * (q % per)],
                              (q / per) & 1u, kWaitLimit);
            __syncwarp();
        } else {
            uint32_t g = 0;        // items started (slot sequence)
            uint32_t es = (uint32_t)lane % (uint32_t)nE, eph = 0;   // this lane's slot, its use's parity
            uint32_t tail = 0;     // oldest item that may still be in the ring
            int32_t head = 0;      // the ring's next free byte (the items lie between)
            bool stop_l = false;
            for (int jn = 0; jn < njobs && !stop_l; ++jn) {
                const TileJob job = jobs[jn];
                const uint32_t* ent = tab[job.b].tile_ent;
                const uint32_t nitem = (uint32_t)job.cnt * (uint32_t)C;
                // lane l < nsets takes the items l, l + nsets, ...: their pointers, read
                // one round ahead
                auto ptrs = [&](uint32_t j, int32_t (&p)[6]) {
#pragma unroll
                    for (int k = 0; k < 6; ++k) p[k] = 0;
                    if (lane < nsets && j < nitem) seg_ptrs(job, j, p);
                };
                int32_t cur[6], nxt[6];
                ptrs((uint32_t)lane, cur);
                for (uint32_t jb = 0; jb < nitem; jb += (uint32_t)nsets) {
                    ptrs(jb + (uint32_t)nsets + (uint32_t)lane, nxt);
                    const uint32_t n = min((uint32_t)nsets, nitem - jb);
                    const int32_t len = cur[4] - cur[0];
                    const int32_t room = (uint32_t)lane < n ? max(len, 4) * 4 : 0;   // ring bytes
                    // the slots' previous items have been consumed (a lane each; at a
                    // slot's first use the parity of the phase before the first)
                    bool ok = (uint32_t)lane >= n || tc::mbar_wait(&ent_free[es], eph ^ 1u, kWaitLimit);
                    ok = __all_sync(0xFFFFFFFFu, ok && *err == 0);
                    // a lane's copy may land where the item of another lane's slot lay: each
                    // lane takes over what the others have seen consumed
                    __syncwarp();
                    if (g + n > tail + (uint32_t)nE) tail = g + n - (uint32_t)nE;
                    // the round's items side by side when the ring has room for all
                    int32_t off = room;
#pragma unroll
                    for (int o = 1; o < kProdSets; o <<= 1) {
                        const int32_t y = __shfl_up_sync(0xFFFFFFFFu, off, o);
                        if (lane >= o) off += y;
                    }
                    const int32_t all = __shfl_sync(0xFFFFFFFFu, off, kProdSets - 1);
                    off -= room;
                    if (tail == g) head = 0;
                    int32_t toff = tail == g ? -1 : slot_off[tail % (uint32_t)nE];
                    if (ok && (head > toff ? (int32_t)e_ring - head : toff - head) >= all) {
                        if ((uint32_t)lane < n) issue(ent, cur, es, head + off);
                        head += all;
                    } else {
                        // one after the other, wrapping, and waiting for the oldest
                        // items in the ring as needed
                        for (uint32_t j = 0; j < n && ok; ++j) {
                            const int32_t need = __shfl_sync(0xFFFFFFFFu, room, (int)j);
                            int32_t at = -1;
                            while (ok && at < 0) {
                                if (tail == g + j) {
                                    at = 0;
                                } else {
                                    const uint32_t ts = tail % (uint32_t)nE;
                                    toff = slot_off[ts];
                                    if (head > toff) {
                                        if ((int32_t)e_ring - head >= need) at = head;
                                        else if (toff >= need) at = 0;
                                    } else if (toff - head >= need) {
                                        at = head;
                                    }
                                    if (at < 0) {
                                        ok = tc::mbar_wait_warp(&ent_free[ts],
                                                                (tail / (uint32_t)nE) & 1u,
                                                                kWaitLimit) &&
                                             __all_sync(0xFFFFFFFFu, *err == 0);
                                        ++tail;
                                    }
                                }
                            }
                            if (ok && (uint32_t)lane == j) issue(ent, cur, es, at);
                            head = at + need;
                            __syncwarp();
                        }
                    }
                    if (!ok) {
                        if (lane == 0) *err = DPMM_ETIMEOUT;
                        stop_l = true;
                        break;
                    }
                    __syncwarp();
                    if ((es += n) >= (uint32_t)nE) {
                        es -= (uint32_t)nE;
                        eph ^= 1u;
                    }
                    g += n;
#pragma unroll
                    for (int k = 0; k < 6; ++k) cur[k] = nxt[k];
                }
            }
            // every started copy has landed before the block can exit (after a
            // timeout perhaps some of the round that was cut short)
            const uint32_t issued = g + (stop_l ? (uint32_t)nsets : 0u);
            if (lane == 0)
                for (uint32_t q = issued > (uint32_t)nE ? issued - (uint32_t)nE : 0u; q < issued; ++q)
                    tc::mbar_wait(&ent_full[q % (uint32_t)nE], (q / (uint32_t)nE) & 1u,
                                  stop_l ? kWaitLimit >> 8 : kWaitLimit);
        }
    } else if (warp == kBLoadWarp) {
        // ---------------- B loader ----------------
        if (lane == 0) {
            uint32_t g = 0, bs = 0, bph = 0;    // chunks started
            bool stop_b = false;
            for (int jn = 0; jn < njobs && !stop_b; ++jn) {
                const TileJob job = jobs[jn];
                const unsigned char* B = tab[job.b].tile_B;
                const uint32_t bytes = (uint32_t)tile_ntot(job.K()) * 128u;
                for (int i = 0; i < job.cnt && !stop_b; i += kPair) {
                    for (int c = 0; c < C; ++c, ++g) {
                        if (g >= (uint32_t)nB &&
                            !tc::mbar_wait(&b_free[bs], bph ^ 1u, kWaitLimit)) {
                            *err = DPMM_ETIMEOUT;
                            stop_b = true;
                            break;
                        }
                        if (*err) {
                            stop_b = true;
                            break;
                        }
                        tc::mbar_arrive_expect_tx(&b_full[bs], bytes);
                        tc::bulk_g2s(B_base + bs * b_slot, B + (size_t)c * kBChunkBytes,
                                     bytes, &b_full[bs]);
                        if (++bs == (uint32_t)nB) {
                            bs = 0;
                            bph ^= 1u;
                        }
                    }
                }
            }
            const uint32_t issued = g;
            for (uint32_t q = issued > (uint32_t)nB ? issued - (uint32_t)nB : 0u; q < issued; ++q)
                tc::mbar_wait(&b_full[q % (uint32_t)nB], (q / (uint32_t)nB) & 1u, kWaitLimit);
        }
    } else if (warp == kMmaWarp) {
        // ---------------- MMA issue ----------------
        // An item costs this warp the latency of its instructions, not the tensor
        // core's time, while N <= 128 (alone: four MMAs and a commit 200-260
        // cycles, a wait for a barrier that is already complete another 200, 340
        // beside busy producers; the tensor core needs 257 at N = 128, 480 at
        // N = 240).  So the whole warp walks the items converged and an elected
        // lane issues (from a branch of one lane the same sequence took 282, its
        // waits 270 - 500), and one wait serves two items: lanes poll the barriers of
        // two A stages and their B stages side by side.
        // Lane l < nsets follows the stages of producer set l (index and parity of
        // the next one); lane 5 polls a round's second B stage.
        uint32_t s0 = 0, bs = 0, bph = 0;       // next item's set; next B stage, its parity
        uint32_t idx = (uint32_t)lane % (uint32_t)nsets, ph = 0;
        auto advance = [&]() {                  // a set's lane: one stage on
            if ((idx += (uint32_t)nsets) >= (uint32_t)nS) {
                idx -= (uint32_t)nS;
                ph ^= 1u;
            }
        };
        uint32_t slot = 0, aph = 1;             // accumulator slot, its reads' parity
        const uint64_t desc = tc::desc_sw128(0);
        const uint32_t alo = tc::smem_addr(A_base) >> 4, blo = tc::smem_addr(B_base) >> 4;
        const uint32_t bstep = (uint32_t)(b_slot >> 4);
        auto four = [&](uint32_t acc, uint32_t a, uint32_t bb, uint32_t idesc, uint32_t accum) {
            const uint64_t ad = desc | a, bd = desc | bb;
            tc::mma_bf16(acc, ad, bd, idesc, accum);
#pragma unroll
            for (int k = 1; k < 4; ++k) tc::mma_bf16(acc, ad + 2 * k, bd + 2 * k, idesc, 1u);
        };
        bool go = true;
        for (int jn = 0; jn < njobs && go; ++jn) {
            const TileJob job = jobs[jn];
            const int cnt = job.cnt;
            const uint32_t ntot = (uint32_t)tile_ntot(job.K());
            const uint32_t idesc = tc::idesc_bf16(128, ntot);
            const bool planes = job.planes();
            for (int i = 0; i < cnt && go; i += kPair) {
                const int m = min(kPair, cnt - i);
                uint32_t acc[kPair] = {0u, 0u};
                uint64_t* full[kPair] = {nullptr, nullptr};
#pragma unroll
                for (int p = 0; p < kPair; ++p) {
                    if (p < m) {
                        // the slot's previous tile has been read (at the slot's
                        // first use the parity of the phase before the first)
                        go = go && tc::mbar_wait_warp(&acc_empty[slot], aph, kWaitLimit);
                        acc[p] = tmem + slot * ldN;
                        full[p] = &acc_full[slot];
                        if (++slot == nAcc) {
                            slot = 0;
                            aph ^= 1u;
                        }
                    }
                }
                if (m == 1) acc[1] = acc[0];
                tc::fence_after_sync();
                go = go && __all_sync(0xFFFFFFFFu, *err == 0);
                // Rounds of two items: a chunk of both tiles, or two chunks of one
                // (the last may be one chunk alone).
                const uint32_t nb = (uint32_t)(kPair / m);      // B stages of a round
                const int rounds = (C + (int)nb - 1) / (int)nb;
                for (int rd = 0; rd < rounds && go; ++rd) {
                    const bool two = m == kPair || 2 * rd + 1 < C;
                    const uint32_t s1 = s0 + 1 == (uint32_t)nsets ? 0 : s0 + 1;
                    const uint32_t bs1 = nb == 1 ? bs : bs + 1 == (uint32_t)nB ? 0 : bs + 1;
                    const bool item = (uint32_t)lane == s0 || (two && (uint32_t)lane == s1);
                    uint32_t a0 = __shfl_sync(0xFFFFFFFFu, idx, (int)s0);
                    uint32_t a1 = __shfl_sync(0xFFFFFFFFu, idx, (int)s1);
                    // (lanes without a barrier of their own poll the first B stage's)
                    uint64_t* bar = item ? a_full + idx : b_full + bs;
                    uint32_t par = item ? ph : bph;
                    if (lane == 5 && two && nb == 2) {
                        bar = b_full + bs1;
                        par = bs1 ? bph : bph ^ 1u;
                    }
                    go = tc::mbar_wait_warp(bar, par, kWaitLimit);
                    // each of the lanes has seen one of the round's barriers complete:
                    // the lane that issues takes over what all of them have seen
                    __syncwarp();
                    tc::fence_after_sync();
                    if (!go) break;
                    const unsigned hq =
                        planes ? __ballot_sync(0xFFFFFFFFu,
                                               item && reinterpret_cast<volatile int32_t*>(
                                                           stage_hi)[idx])
                               : 0u;
                    if (item) advance();
                    if (two && !hq) {
                        if (tc::elect_one()) {
                            four(acc[0], alo + a0 * (kStageBytes >> 4), blo + bs * bstep, idesc,
                                 rd != 0);
                            tc::mma_commit(&stage_free[a0]);
                            if (nb == 2) tc::mma_commit(&b_free[bs]);
                            four(acc[1], alo + a1 * (kStageBytes >> 4), blo + bs1 * bstep, idesc,
                                 (rd != 0) | (nb - 1u));
                            tc::mma_commit(&stage_free[a1]);
                            tc::mma_commit(&b_free[bs1]);
                        }
                        __syncwarp();
                    } else {
                        // one item, or some with a second plane: its set's next stage (both:
                        // full when the first is)
#pragma unroll 1
                        for (uint32_t x = 0; x < (two ? 2u : 1u) && go; ++x) {
                            const uint32_t sx = x ? s1 : s0, bx = x ? bs1 : bs;
                            const uint32_t ax = x ? acc[1] : acc[0];
                            const uint32_t a = x ? a1 : a0;
                            const bool h = (hq >> sx) & 1u;
                            const uint32_t e = __shfl_sync(0xFFFFFFFFu, idx, (int)sx);
                            if (tc::elect_one()) {
                                four(ax, alo + a * (kStageBytes >> 4), blo + bx * bstep, idesc,
                                     (rd != 0) | (x & (nb - 1u)));
                                tc::mma_commit(&stage_free[a]);
                                if (h && both) {
                                    four(ax, alo + e * (kStageBytes >> 4), blo + bx * bstep,
                                         idesc, 1u);
                                    tc::mma_commit(&stage_free[e]);
                                }
                            }
                            __syncwarp();
                            if (h && !both) {
                                go = tc::mbar_wait_warp(a_full + e,
                                                        __shfl_sync(0xFFFFFFFFu, ph, (int)sx),
                                                        kWaitLimit);
                                tc::fence_after_sync();
                                if (go && tc::elect_one()) {
                                    four(ax, alo + e * (kStageBytes >> 4), blo + bx * bstep,
                                         idesc, 1u);
                                    tc::mma_commit(&stage_free[e]);
                                }
                                __syncwarp();
                            }
                            if (h && (uint32_t)lane == sx) advance();
                            if ((nb == 2 || x == 1) && tc::elect_one()) tc::mma_commit(&b_free[bx]);
                            __syncwarp();
                        }
                    }
                    if ((s0 += two ? 2u : 1u) >= (uint32_t)nsets) s0 -= (uint32_t)nsets;
                    if ((bs += two ? nb : 1u) >= (uint32_t)nB) {
                        bs -= (uint32_t)nB;
                        bph ^= 1u;
                    }
                }
                if (go && tc::elect_one()) {
                    tc::mma_commit(full[0]);
                    if (m == kPair) tc::mma_commit(full[1]);
                }
                __syncwarp();
            }
        }
        if (!go && lane == 0) *err = DPMM_ETIMEOUT;
        // every MMA issued has completed (and signalled) before exit
        if (tc::elect_one()) tc::mma_commit(drain);
        __syncwarp();
        tc::mbar_wait_warp(drain, 0u, kWaitLimit);
    } else if (warp < kEpiWarps) {
        // ---------------- epilogue (warps 0-7) ----------------
        const int h = warp >> 2, qw = warp & 3;
        const int r = 32 * qw + lane;
        uint32_t it = 0;
        bool halt = false;
        for (int jn = 0; jn < njobs && !halt; ++jn) {
            const TileJob job = jobs[jn];
            const ChainArgs& ch = tab[job.b];
            const int first = job.first, cnt = job.cnt, K = job.K();
            const int S0 = tile_s0(K), Ntot = tile_ntot(K);
            // this chain's log pi, eq. 8 weights and log q sums in shared memory
            tc::named_bar(kBarEpi, 32 * kEpiWarps);
            for (int k = tid; k < K; k += 32 * kEpiWarps) spi[k] = ch.logpi[k];
            for (int i = tid; i < 2 * K; i += 32 * kEpiWarps) {
                const float n = (float)ch.nsub[i];
                slw[2 * i] = n > 0.0f ? logf(n) : -CUDART_INF_F;
                slw[2 * i + 1] = n > 1.0f ? logf(n - 1.0f) : -CUDART_INF_F;
            }
            for (int i = tid; i < 8 * K; i += 32 * kEpiWarps) wsq[i] = 0u;
            tc::named_bar(kBarEpi, 32 * kEpiWarps);
            for (int ti = 0; ti < cnt; ++ti, ++it) {
                const int tile = first + ti * (int)gridDim.x;
                const uint32_t slot = it % nAcc, xb = it & 1;
                const int64_t cell = (int64_t)tile * 128 + r;
                const bool live = cell < ch.N;
                // this cell's noise and old state, loaded before the accumulator is
                // ready (clusters 16 j + 8 h .. + 7 for this half)
                float gq[kEpiGroups][8], gs0 = 0.0f, gs1 = 0.0f;
                uint32_t old = 0u;
#pragma unroll
                for (int j = 0; j < kEpiGroups; ++j)
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int k = 16 * j + 8 * h + i;
                        gq[j][i] = live && k < K ? __ldg(ch.noise + (size_t)k * ch.N + cell) : 0.0f;
                    }
                if (live) {
                    gs0 = __ldg(ch.noise + (size_t)K * ch.N + cell);
                    gs1 = __ldg(ch.noise + (size_t)(K + 1) * ch.N + cell);
                    old = ch.state[cell];
                }
                const bool ok = tc::mbar_wait(&acc_full[slot], (it / nAcc) & 1u, kWaitLimit);
                if (!ok) *err = DPMM_ETIMEOUT;
                tc::fence_after_sync();
                const bool okw = __all_sync(0xFFFFFFFFu, ok);
                const uint32_t trow = tmem + slot * ldN + ((uint32_t)(32 * qw) << 16);
                float best = -CUDART_INF_F;
                int c = h ? K : 0;   // half 1's "none" loses every tie
                if (okw) {
#pragma unroll
                    for (int j = 0; j < kEpiGroups; ++j) {
                        const int q = 2 * j + h;
                        if (q >= S0 / 16) continue;
                        float v[16];
                        tc::tmem_ld16(trow + (uint32_t)(16 * q), v);
                        tc::tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const int k = 8 * q + i;
                            if (k < K) {
                                const float sc = v[2 * i] + v[2 * i + 1];
                                if (dbg && live) dbg_out[(size_t)cell * 3 * K + k] = sc;
                                const float val = (spi[k] + sc) + gq[j][i];
                                if (val > best) {
                                    best = val;
                                    c = k;
                                }
                            }
                        }
                    }
                }
                // both halves learn the winner: half 0's unless half 1's is larger
                // (half 0's wins a tie with a lower index, half 1's otherwise)
                xbest[128 * (2 * xb + h) + r] = best;
                xc[128 * (2 * xb + h) + r] = c;
                if (tid == 0) stop[xb] = *err;
                tc::named_bar(kBarEpi, 32 * kEpiWarps);
                if (stop[xb]) {
                    halt = true;
                    break;
                }
                {
                    const float bo = xbest[128 * (2 * xb + (h ^ 1)) + r];
                    const int co = xc[128 * (2 * xb + (h ^ 1)) + r];
                    if (bo > best || (bo == best && co < c)) c = co;
                }
                // its sub-cluster scores: each half reads every other block of 16
                // columns, the half that meets the cell's columns finishes it
                float t0 = 0.0f, t1 = 0.0f;
                const int s0 = S0 + 4 * c;
                for (int q = S0 / 16 + h; q < Ntot / 16; q += 2) {
                    float v[16];
                    tc::tmem_ld16(trow + (uint32_t)(16 * q), v);
                    tc::tmem_ld_wait();
                    if (dbg && live) {
#pragma unroll
                        for (int i = 0; i < 16; i += 2) {
                            const int col = 16 * q + i - S0;
                            if (col < 4 * K)
                                dbg_out[(size_t)cell * 3 * K + K + (col >> 1)] = v[i] + v[i + 1];
                        }
                    }
                    if ((s0 >> 4) == q) {
                        const int o = s0 & 15;
                        if (o == 0) { t0 = v[0] + v[1]; t1 = v[2] + v[3]; }
                        else if (o == 4) { t0 = v[4] + v[5]; t1 = v[6] + v[7]; }
                        else if (o == 8) { t0 = v[8] + v[9]; t1 = v[10] + v[11]; }
                        else { t0 = v[12] + v[13]; t1 = v[14] + v[15]; }
                    }
                }
                // this half has read the accumulator (both: the slot's next tile may
                // start)
                tc::fence_before_sync();
                tc::named_bar(kBarHalf + h, 128);
                if (qw == 0 && lane == 0) tc::mbar_arrive(&acc_empty[slot]);
                if (live && !dbg && (((s0 >> 4) - S0 / 16) & 1) == h) {
                    const bool stays = state_label(old) == (uint32_t)c;
                    const uint32_t so = state_sub(old);
                    const float lw0 = slw[4 * c + (stays && so == 0 ? 1 : 0)];
                    const float lw1 = slw[4 * c + 2 + (stays && so == 1 ? 1 : 0)];
                    const bool both_empty = lw0 == -CUDART_INF_F && lw1 == -CUDART_INF_F;
                    const float l0 = (both_empty ? 0.0f : lw0) + t0;
                    const float l1 = (both_empty ? 0.0f : lw1) + t1;
                    const uint32_t s = (l1 + gs1 > l0 + gs0) ? 1u : 0u;
                    const float mx = fmaxf(l0, l1), mn = fminf(l0, l1);
                    const float logq = (s ? l1 : l0) - (mx + log1pf(expf(mn - mx)));
                    ch.state[cell] = pack_state((uint32_t)c, s);
                    add_words64(wsq + 2 * (qw * K + c), logq_fixed(logq));
                }
            }
            if (halt) break;
            // this chain's sum log q (per cluster, over its tiles of this block)
            tc::named_bar(kBarEpi, 32 * kEpiWarps);
            if (!dbg)
                for (int k = tid; k < K; k += 32 * kEpiWarps) {
                    unsigned long long v = 0ull;
                    for (int w = 0; w < 4; ++w)
                        v += (unsigned long long)wsq[2 * (w * K + k)] +
                             ((unsigned long long)wsq[2 * (w * K + k) + 1] << 32);
                    if (v) atomicAdd(&ch.acc_logq[k], v);
                }
        }
    }
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(tmem, 512);
    if (*err && tid == 0)
        for (int jn = 0; jn < njobs; ++jn) atomicExch(&tab[jobs[jn].b].sc->error, *err);
}

// Statistics n-bar[k][r], S-bar[k][r][u] of the sweep's labels (from either
// engine), read from the blocked entries: S-bar added into the main rows
// (cleared by k_build_b), n-bar into the accumulator nsub (the compaction
// moves it into the main one).  Blocks are partitioned by gene chunk: block b
// takes chunk c = b % C of the tiles t = b / C, b / C + nt, ... (nt tile
// groups), so its private counters cover only 64 genes ([2K][64] words in
// shared memory; K > kTileMaxK counts straight into global memory) and its
// flush adds at most 2K x 64 words.  A warp takes one (tile, chunk) segment at a
// time, with the counter row (2 k + r) ld of each of the tile's 128 cells cached
// (0xFFFFFFFF past the last cell), or (kQuarter) one quarter of a segment.  An
// item of fewer tiles than half the warps is taken by quarters: a segment alone
// is several dependent batches of loads long (2,000 x 500: 12.4 -> 6.9 us), but
// its quarters fill those batches less well (68,000 x 1,000, 14 tiles an item:
// 16.0 us by segments, 20.7 by quarters).  Integer sums, exact.
constexpr int kStatsTileThreads = 512;

template <bool kQuarter, typename T_>
__device__ __forceinline__ void count_segments(T_* priv, int ld, uint32_t* pn, uint32_t* my,
                                               const uint32_t* __restrict__ state,
                                               const uint32_t* __restrict__ ent,
                                               const int32_t* __restrict__ ptr, int32_t T,
                                               int32_t C, int64_t N, int c, int tg, int nt,
                                               int lane, int w, int nw) {
    constexpr int parts = kQuarter ? 4 : 1, rows = 4 / parts;   // 32-cell row blocks of a unit
    const int units = parts * ((T - tg + nt - 1) / nt);
    for (int un = w; un < units; un += nw) {
        const int tile = tg + nt * (un / parts), q0 = un % parts;
        const int64_t seg = (int64_t)tile * C + c;
        const int p0 = ptr[4 * seg + q0] & kTilePtrMask;
        const int p1 = ptr[4 * seg + (kQuarter ? q0 + 1 : 4)] & kTilePtrMask;
#pragma unroll
        for (int j = 0; j < rows; ++j) {
            const int64_t cell = (int64_t)tile * 128 + 32 * (q0 + j) + lane;
            uint32_t row = 0xFFFFFFFFu;
            if (cell < N) {
                const uint32_t st = state[cell];
                const uint32_t kr = 2 * state_label(st) + state_sub(st);
                row = kr * (uint32_t)ld;
                if (c == 0) atomicAdd(&pn[kr], 1u);
            }
            my[32 * (q0 + j) + lane] = row;
        }
        __syncwarp();
        // an entry of count 0 (segment padding) adds nothing; its cell may lie
        // past the last one, so it is skipped before its row is read
        auto add = [&](uint32_t v) {
            const uint32_t x = v & 0xFFFFu;
            if (x) atomicAdd(&priv[my[v >> 22] + ((v >> 16) & 63u)], x);
        };
        int e = p0 + lane;
        for (; e + 32 * 15 < p1; e += 32 * 16) {      // whole batches: 16 loads in flight
            const uint32_t* pe = ent + e;
            uint32_t v[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = __ldg(pe + 32 * j);
#pragma unroll
            for (int j = 0; j < 16; ++j) add(v[j]);
        }
        if (e < p1) {                                  // the rest, bounds-checked
            uint32_t v[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = e + 32 * j < p1 ? __ldg(ent + e + 32 * j) : 0u;
#pragma unroll
            for (int j = 0; j < 16; ++j) add(v[j]);
        }
        __syncwarp();
    }
}

// Item (chunk c, tile group tg of nt) of a chain: tiles tg, tg + nt, ... of
// gene chunk c, counted into the block's private counters and flushed.
__device__ __forceinline__ void
stats_tile_item(const ChainArgs& ch, int c, int tg, int nt, uint32_t (*cache)[128],
                uint32_t* priv, uint32_t* pn) {
    const DevScalars* sc = ch.sc;
    const uint32_t* __restrict__ state = ch.state;
    const uint32_t* __restrict__ ent = ch.tile_ent;
    const int32_t* __restrict__ ptr = ch.tile_ptr;
    const int32_t T = ch.tile_T, C = ch.tile_C, D = ch.D;
    const int64_t N = ch.N;
    uint32_t* __restrict__ acc_nsub = ch.acc_nsub;
    uint32_t* __restrict__ Ssub = ch.Ssub;
    const int K = sc->K;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int gene0 = c * 64;
    if (K > kTileMaxK) {
        // counts straight into the main rows (global atomics)
        count_segments<false>(Ssub + gene0, D, acc_nsub, cache[w], state, ent, ptr, T, C, N, c, tg, nt,
                       lane, w, nw);
        return;
    }
    for (int i = threadIdx.x; i < 2 * K * 64; i += blockDim.x) priv[i] = 0u;
    for (int i = threadIdx.x; i < 2 * K; i += blockDim.x) pn[i] = 0u;
    __syncthreads();
    if ((T - tg + nt - 1) / nt < nw / 2)
        count_segments<true>(priv, 64, pn, cache[w], state, ent, ptr, T, C, N, c, tg, nt, lane, w,
                             nw);
    else
        count_segments<false>(priv, 64, pn, cache[w], state, ent, ptr, T, C, N, c, tg, nt, lane,
                              w, nw);
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * K * 64; i += blockDim.x) {
        const int u = gene0 + (i & 63);
        if (priv[i] && u < D) atomicAdd(&Ssub[(size_t)(i >> 6) * D + u], priv[i]);
    }
    if (c == 0)
        for (int i = threadIdx.x; i < 2 * K; i += blockDim.x)
            if (pn[i]) atomicAdd(&acc_nsub[i], pn[i]);
}

// The items of every chain with the blocked copy (chain b: tile_C chunks x g_b
// tile groups) form one list dealt round-robin to the blocks, so the chains of
// a batch are counted side by side, each with as many items as its size
// warrants: g_b = ceil(T_b / S) clamped to [1, min(T_b, nt)], with nt the tile
// groups per chunk of the launch and S the tiles per item that give the whole
// table about two items per block (one item per block for a single chain).
// The counts are integer sums, so the split into items changes nothing.  With
// several chains (at most kStatsTable) the threads read the table side by side
// first, so that a block finds its items without a round trip per chain.
constexpr int kStatsTable = kStatsTileThreads;

__device__ __forceinline__ int stats_groups(const ChainArgs& ch, int32_t nt, int64_t S) {
    return (int)max((int64_t)1,
                    min(((int64_t)ch.tile_T + S - 1) / S, (int64_t)min(ch.tile_T, nt)));
}

template <class Tab>
__global__ void __launch_bounds__(kStatsTileThreads)
k_stats_tile(const __grid_constant__ Tab tab, int32_t nt, int64_t S) {
    __shared__ uint32_t cache[kStatsTileThreads / 32][128];
    __shared__ uint32_t priv[2 * kTileMaxK * 64];
    __shared__ uint32_t pn[2 * kTileMaxK];
    __shared__ int32_t before[kStatsTable + 1], groups[kStatsTable];   // items, tile groups
    const int64_t G = gridDim.x;
    const int n = tab.n();
    if (n > 1 && n <= kStatsTable) {
        const int b = threadIdx.x, lane = b & 31, w = b >> 5;
        int g = 0, items = 0;
        if (b < n && tab[b].tile_enabled) {
            g = stats_groups(tab[b], nt, S);
            items = tab[b].tile_C * g;
        }
        int x = items;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) pn[w] = (uint32_t)x;
        __syncthreads();
        int off = x - items;
        for (int i = 0; i < w; ++i) off += (int)pn[i];
        if (b < n) {
            before[b] = off;
            groups[b] = g;
            if (b == n - 1) before[n] = off + items;
        }
        __syncthreads();
        int c = 0;
        for (int id = blockIdx.x; id < before[n]; id += (int)G) {
            while (before[c + 1] <= id) ++c;
            const ChainArgs& ch = tab[c];
            const int i = id - before[c], C = ch.tile_C;
            stats_tile_item(ch, i % C, i / C, groups[c], cache, priv, pn);
            __syncthreads();
        }
        return;
    }
    int64_t base = 0;
    for (int b = 0; b < n; ++b) {
        const ChainArgs& ch = tab[b];
        if (!ch.tile_enabled) continue;
        const int C = ch.tile_C;
        const int g = stats_groups(ch, nt, S);
        const int64_t items = (int64_t)C * g;
        const int64_t first = base + (((int64_t)blockIdx.x - base) % G + G) % G;
        for (int64_t id = first; id < base + items; id += G) {
            const int64_t i = id - base;
            stats_tile_item(ch, (int)(i % C), (int)(i / C), g, cache, priv, pn);
            __syncthreads();
        }
        base += items;
    }
}

// Tile groups per gene chunk of the statistics launch: four blocks per SM
// for one chain, two for a batch, unless tuned (dpmm_set_tuning).
int32_t tile_stat_groups(const Ctx& c) {
    const int per_sm = c.tune_stats_per_sm ? c.tune_stats_per_sm : (c.nchains > 1 ? 2 : 4);
    return max(1, (per_sm * c.num_sms) / max(1, c.tile_C));
}

size_t tile_b_bytes(int32_t C) { return (size_t)C * kBChunkBytes; }

cudaError_t configure_tile(Ctx& c) {
    const void* fns[6] = {(const void*)k_assign_tc<TabV, 8>, (const void*)k_assign_tc<TabV, 12>,
                          (const void*)k_assign_tc<TabV, 16>, (const void*)k_assign_tc<TabP, 8>,
                          (const void*)k_assign_tc<TabP, 12>, (const void*)k_assign_tc<TabP, 16>};
    for (const void* f : fns) {
        cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)c.smem_optin);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_build_b(Ctx& c, bool force) {
    return with_table(c, [&](auto tab) {
        const int rb = c.nchains > 1 ? 64 : 16;
        k_build_b<<<dim3(c.tile_C, kNtotMax / rb, c.nchains), kBuildThreads, 0, c.stream>>>(
            tab, force ? 1 : 0, rb);
        return cudaGetLastError();
    });
}

// A stages of the label kernel (see k_assign_tc): 4 for one chain, 2 for a
// batch, unless tuned; they differ only where neither eight nor six stages fit.
int32_t tile_label_stages(const Ctx& c) {
    return c.tune_tile_stages ? c.tune_tile_stages : (c.nchains > 1 ? 2 : 4);
}

cudaError_t launch_tile_label(Ctx& c, float* dbg) {
    const int scatter = c.tune_tile_scatter ? c.tune_tile_scatter : kScatterDefault;
    const int32_t stages = tile_label_stages(c);
    auto launch = [&](auto tab) {
        using T = decltype(tab);
        const int64_t sm = (int64_t)c.smem_optin;
        if (scatter == 8)
            k_assign_tc<T, 8><<<c.num_sms, kTileThreadsP, c.smem_optin, c.stream>>>(
                tab, dbg, sm, stages);
        else if (scatter == 16)
            k_assign_tc<T, 16><<<c.num_sms, kTileThreadsP, c.smem_optin, c.stream>>>(
                tab, dbg, sm, stages);
        else
            k_assign_tc<T, 12><<<c.num_sms, kTileThreadsP, c.smem_optin, c.stream>>>(
                tab, dbg, sm, stages);
        return cudaGetLastError();
    };
    if (c.label_runs.size() <= 2) return with_table(c, launch);
    cudaError_t e = cudaSuccess;
    for (size_t i = 0; i + 1 < c.label_runs.size() && e == cudaSuccess; ++i)
        e = launch(TabP{c.d_chains + c.label_runs[i], c.label_runs[i + 1] - c.label_runs[i]});
    return e;
}

cudaError_t launch_tile_stats(Ctx& c) {
    const int nt = tile_stat_groups(c);   // tile groups per gene chunk
    const int64_t C = std::max(1, c.tile_C);
    const int64_t S = std::max<int64_t>(1, (c.tile_sumT * C + 2 * (int64_t)nt * C - 1) /
                                               (2 * (int64_t)nt * C));
    return with_table(c, [&](auto tab) {
        k_stats_tile<<<nt * c.tile_C, kStatsTileThreads, 0, c.stream>>>(tab, nt, S);
        return cudaGetLastError();
    });
}

// The whole dense-tile labelling: B operand, labels, statistics (dbg: scores
// only, no state or statistics writes).
cudaError_t launch_tile_assign(Ctx& c, float* dbg) {
    cudaError_t e = launch_build_b(c, dbg != nullptr);
    if (e == cudaSuccess) e = launch_tile_label(c, dbg);
    if (e == cudaSuccess && !dbg) e = launch_tile_stats(c);
    return e;
}

}  // namespace dpmm
