// Grouped (MoE) block-scaled FP4 GEMM on CTA pairs, for experts with many tokens each (grouped_pairs_pay in prq_api.cu draws the line): per expert the product of Eq. (3) as
// in prq_gemm.cu, with the prefill kernel's tile -- 256 tokens of one expert x 240 output features, computed by two
// CTAs of a cluster as one tcgen05 cta_group::2 unit (prq_pair.cuh).
//
// Why.  The tile-per-CTA kernel (128 features x 128 tokens) spends 110 KB of operands per 32 KB of output; at the
// 64 - 70 bytes per cycle that an SM takes in from L2 its main loop alone is 72 us of the 116 us at 8192 tokens x 8
// experts of 2048 x 768 (k = 64).  The pair's tile needs 113 KB per CTA for 61 KB of output: 104 us, against 63 us of HBM
// traffic.  Without its stores it takes 70 us, without the loads of its steady state 70 us too: operand reads and 268 MB of y
// add up on the way through L2, and neither instructions nor the tensor pipe are what it waits for.  With K + k = 832 a tile is only 3.25 stages, so the epilogue must be short: eight warps
// per CTA, 32 rows x 128 columns each, write rows of 128 contiguous bytes through a swizzled staging tile of their own.
// Plain 16-byte stores, not tiled ones: the last rows of an expert are followed by the next expert's, which no tensor map
// clips.
//
// Tiles are counted over all experts (256-token tiles; an expert's last one may be short), feature tiles innermost, so
// that the rows of y are completed while their lines are still in L2 (a tile's 480 bytes per row end inside a line; with
// feature tiles outermost 111 us).  A pair takes a contiguous range of them: stepping to the next is a few shared-memory
// reads, and neighbouring pairs share an expert's weights in L2.  Codes of the next expert's rows that a short tile loads
// are computed and dropped.
//
// Roles per CTA: warp 0 TMA producer, warp 1 tcgen05 issuer (leader CTA only), warps 2 - 9 epilogue.  Every wait is
// bounded; on expiry the roles of both CTAs unwind, tensor memory is freed and PRQ_ERR_TIMEOUT is recorded.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "prq_kernels.h"
#include "prq_pair.cuh"
#include "prq_ptx.cuh"

namespace prq {
namespace {

constexpr int kGpThreads = 320;
constexpr int kGpEpiWarps = 8;
constexpr int kGpStaging = 4096;                  // per epilogue warp: 32 rows x 128 bytes
constexpr int kGpTokens = 256;                    // tokens per tile
constexpr int kGpRowCache = 256;                  // experts whose row ranges are kept in shared memory

template <int BN>
constexpr int gp_smem() { return kStages * PCfg<BN>::kStageBytes + kGpEpiWarps * kGpStaging + 1024; }

// The tiles of one pair, in order.
struct GpTiles {
    const int* tile_start;
    int n_tiles, left;
    int e, mt, ni;
    __device__ __forceinline__ GpTiles(const int* ts, int E, int n_tiles_, int pair, int pairs) : tile_start(ts), n_tiles(n_tiles_) {
        const int T = ts[E] * n_tiles, base = T / pairs, extra = T - base * pairs;
        const int begin = pair * base + min(pair, extra);
        left = base + (pair < extra ? 1 : 0);
        e = mt = ni = 0;
        if (left > 0) {
            mt = begin / n_tiles;
            ni = begin - mt * n_tiles;
            int lo = 0, hi = E - 1;
            while (lo < hi) {   // last expert whose first tile is <= mt
                const int mid = (lo + hi + 1) >> 1;
                if (ts[mid] <= mt) lo = mid; else hi = mid - 1;
            }
            e = lo;
        }
    }
    __device__ __forceinline__ bool valid() const { return left > 0; }
    __device__ __forceinline__ void next() {
        if (--left > 0) {
            if (++ni == n_tiles) {
                ni = 0;
                ++mt;
                while (tile_start[e + 1] <= mt) ++e;   // experts without rows have no tile
            }
        }
    }
};

template <int BN>
__global__ void __launch_bounds__(kGpThreads, 1)
gemm_grouped_pair_kernel(const __grid_constant__ CUtensorMap tm_act, const __grid_constant__ CUtensorMap tm_w,
                         const __grid_constant__ CUtensorMap tm_sfa, const __grid_constant__ CUtensorMap tm_sfw,
                         const GemmParams p) {
    using C = PCfg<BN>;
    static_assert(BN > 128 && BN <= 240, "two accumulators, two scale groups, 128 columns per epilogue warp");
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[kStages], bar_empty[kStages], bar_acc_full[2], bar_acc_empty[2];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag_s;
    __shared__ int tile_start[kMaxExperts + 1], group_start[kMaxExperts + 1];
    __shared__ int row_cache[kGpRowCache + 1];
    volatile int* abort_flag = &abort_flag_s;
    const int* row_start = p.n_experts <= kGpRowCache ? row_cache : p.expert_offsets;

    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t smem_base = smem_u32(smem);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();          // 0 = leader of the pair
    const StagePlan plan(p.K, p.k_tail);
    const int S = plan.S, S1 = plan.S1;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) { mbar_init(smem_u32(&bar_full[i]), 1); mbar_init(smem_u32(&bar_empty[i]), 1); }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&bar_acc_full[i]), 1);
            mbar_init(smem_u32(&bar_acc_empty[i]), 2 * kGpEpiWarps);   // the epilogue warps of both CTAs
        }
        abort_flag_s = 0;
        fence_mbar_init();
        tma_prefetch_desc(&tm_act);
        tma_prefetch_desc(&tm_w);
        tma_prefetch_desc(&tm_sfa);
        tma_prefetch_desc(&tm_sfw);
    }
    if (warp == 1) {
        tmem_alloc_pair(smem_u32(&tmem_slot), kTmemCols);
        tmem_relinquish_pair();
    }
    // everything above overlaps the kernel before this one; from here on its results are read
    grid_dependency_wait();
    if (p.n_experts <= kGpRowCache)
        for (int e = threadIdx.x; e <= p.n_experts; e += kGpThreads) row_cache[e] = p.expert_offsets[e];
    __syncthreads();
    if (warp == 2) warp_expert_starts(row_start, p.n_experts, kGpTokens, tile_start, group_start);
    // both CTAs' barriers and tensor memory must exist before either CTA signals the other
    tc_fence_before_sync();
    __syncthreads();
    cluster_arrive();
    cluster_wait();
    tc_fence_after_sync();
    const uint32_t tmem_base = tmem_slot;
    const uint32_t lo_base = ((smem_base & 0x3FFFF) >> 4) | (1u << 16);
    const int n_tiles = (p.N + BN - 1) / BN;
    GpTiles t(tile_start, p.n_experts, n_tiles, static_cast<int>(blockIdx.x >> 1), static_cast<int>(gridDim.x >> 1));

    if (warp == 0) {
        // ------------------------------------------------------------ producer (both CTAs)
        int st = 0;
        uint32_t ph = 0;
        bool ok = true;
        const uint32_t leader_full0 = cluster_map(smem_u32(&bar_full[0]), 0);
        for (; t.valid() && ok; t.next()) {
            const int lt = t.mt - tile_start[t.e];
            const int row = row_start[t.e] + lt * kGpTokens + static_cast<int>(rank) * 128;
            const int wrow = t.e * p.N + t.ni * BN + static_cast<int>(rank) * C::kHalfN;
            // scale bytes: rows of 256 bytes, 4 per 128-row group
            const int sfa0 = (group_start[t.e] + lt * 2 + static_cast<int>(rank)) * 4, sfa_stride = p.act_groups * 4;
            const int sfw0 = (t.e * S * p.w_groups + t.ni * C::kSfqGroups) * 4, sfw_stride = p.w_groups * 4;
            for (int s = 0; s < S; ++s) {
                if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_empty[st]), ph ^ 1, abort_flag))) { ok = false; break; }
                if (elect_one()) {
                    if (rank == 0) mbar_arrive_expect_tx(smem_u32(&bar_full[st]), 2 * C::kTxBytes);
                    const uint32_t full = leader_full0 + st * 8, sb = smem_base + st * C::kStageBytes;
                    const int xw = s < S1 ? s * 128 : p.K / 2 + (s - S1) * 128;
                    const int xa = s < S1 ? s * 128 : (p.K - p.k_tail) / 2 + (s - S1) * 128;
                    tma_load_2d_pair(sb + kPTile, &tm_w, xw, wrow, full);
                    tma_load_2d_pair(sb, &tm_act, xa, row, full);
                    tma_load_2d_pair(sb + kPTile + C::kQTile, &tm_sfa, 0, sfa0 + s * sfa_stride, full);
                    tma_load_2d_pair(sb + kPTile + C::kQTile + C::kSfp, &tm_sfw, 0, sfw0 + s * sfw_stride, full);
                }
                if (++st == kStages) { st = 0; ph ^= 1; }
            }
        }
        // gave up: copies in flight still target this CTA's shared memory and are counted on the leader's barrier, which
        // this CTA cannot poll: give them time to land (microseconds) before the CTA moves on to the teardown
        if (!ok) __nanosleep(50000);
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer (leader CTA only)
        if (rank == 0) {
            const bool leader = elect_one();
            int st = 0, tile_it = 0;
            uint32_t ph = 0;
            bool ok = true, ready = false;   // ready: the next slot was already seen full by the probe one stage earlier
            const uint32_t sf_t = tmem_base + C::kSfCol;
            for (int left = t.left; left > 0 && ok; --left, ++tile_it) {
                const int buf = tile_it & 1;
                if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_acc_empty[buf]), ((tile_it >> 1) & 1) ^ 1, abort_flag))) break;
                tc_fence_after_sync();
                const uint32_t d_tmem = tmem_base + buf * BN;
                uint32_t accumulate = 0;
                for (int s = 0; s < S; ++s) {
                    if (!ready && !__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_full[st]), ph, abort_flag))) { ok = false; break; }
                    const int rem = s < S1 ? p.K - s * kStageK : p.k_tail - (s - S1) * kStageK;
                    const int nst = st + 1 == kStages ? 0 : st + 1;
                    const uint32_t nph = nst == 0 ? ph ^ 1 : ph;
                    ready = __all_sync(0xffffffffu, mbar_test_wait(smem_u32(&bar_full[nst]), nph));
                    if (leader) {
                        const uint32_t eb = smem_u32(&bar_empty[0]);
                        switch (st) {
                            case 0: issue_stage<BN, false, 0>(lo_base, d_tmem, sf_t, rem, accumulate, eb); break;
                            case 1: issue_stage<BN, false, 1>(lo_base, d_tmem, sf_t, rem, accumulate, eb); break;
                            case 2: issue_stage<BN, false, 2>(lo_base, d_tmem, sf_t, rem, accumulate, eb); break;
                            case 3: issue_stage<BN, false, 3>(lo_base, d_tmem, sf_t, rem, accumulate, eb); break;
                            default: issue_stage<BN, false, 4>(lo_base, d_tmem, sf_t, rem, accumulate, eb); break;
                        }
                    }
                    accumulate = 1;
                    st = nst; ph = nph;
                }
                if (!ok) break;
                if (leader) tc_commit_pair(smem_u32(&bar_acc_full[buf]), 3);
                __syncwarp();
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue (warps 2..9, both CTAs)
        const int q4 = warp & 3;                        // tensor-memory lane quarter of this warp
        const int half = (warp - 2) >> 2;               // which 128 columns of the tile
        const uint32_t stg = smem_base + kStages * C::kStageBytes + (warp - 2) * kGpStaging;
        const uint32_t leader_acc_empty0 = cluster_map(smem_u32(&bar_acc_empty[0]), 0);
        int tile_it = 0;
        for (; t.valid(); t.next(), ++tile_it) {
            const int buf = tile_it & 1;
            const int lt = t.mt - tile_start[t.e];
            const int row0 = row_start[t.e] + lt * kGpTokens + static_cast<int>(rank) * 128 + q4 * 32;   // this warp's first row
            const int n_rows = min(32, row_start[t.e + 1] - row0);
            const int n0 = t.ni * BN, col0 = n0 + half * 128, col_end = min(p.N, n0 + BN);
            if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_acc_full[buf]), (tile_it >> 1) & 1, abort_flag))) break;
            tc_fence_after_sync();
            const int cols = n_rows > 0 ? max(0, min(128, col_end - col0)) : 0;   // columns of this warp to store
            const uint32_t acc_t = tmem_base + buf * BN + half * 128 + (static_cast<uint32_t>(q4 * 32) << 16);
            if (cols == 0) {
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(leader_acc_empty0 + buf * 8);
                continue;
            }
            // 128 bytes of every row at a time (64 bf16 or 32 fp32 columns): registers, a swizzled staging tile (16-byte unit
            // index ^= row % 8), whole rows out.  One compact loop: unrolled over the chunks and both types the code
            // outgrew the instruction cache and took 6 us per tile.
            const int rsub = lane >> 3, u = lane & 7;
            const int chunk = p.y_bf16 ? 64 : 32, es = p.y_bf16 ? 2 : 4, per16 = 16 / es;
            uint8_t* yp0 = static_cast<uint8_t*>(p.y) + (static_cast<size_t>(row0 + rsub) * p.ldy + col0 + u * per16) * es;
            const size_t step4 = static_cast<size_t>(4) * p.ldy * es;
#pragma unroll 1
            for (int c0 = 0; c0 < cols; c0 += chunk, yp0 += 128) {
                uint32_t h[32];
                if (p.y_bf16) {
                    // (the second half of a 240-column tile reads 16 columns past it: the other accumulator's or scales, dropped)
                    uint32_t r[64];
                    tmem_ld_32x32(acc_t + c0, *reinterpret_cast<uint32_t (*)[32]>(&r[0]));
                    tmem_ld_32x32(acc_t + c0 + 32, *reinterpret_cast<uint32_t (*)[32]>(&r[32]));
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        const __nv_bfloat162 t2 = __floats2bfloat162_rn(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
                        h[i] = *reinterpret_cast<const uint32_t*>(&t2);
                    }
                } else {
                    tmem_ld_32x32(acc_t + c0, h);
                    tmem_ld_wait();
                }
                if (c0 + chunk >= cols) {
                    // the warp's share has been read: hand the accumulator back before the stores
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(leader_acc_empty0 + buf * 8);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    st_shared_v4(stg + lane * 128 + ((i ^ (lane & 7)) << 4), h[4 * i], h[4 * i + 1], h[4 * i + 2], h[4 * i + 3]);
                __syncwarp();
                const int left = cols - c0 - u * per16;   // columns from this lane's first one on
                uint8_t* yp = yp0;
                uint4 v[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int row = j * 4 + rsub;
                    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v[j].x), "=r"(v[j].y), "=r"(v[j].z), "=r"(v[j].w) : "r"(stg + row * 128 + ((u ^ (row & 7)) << 4)));
                }
#pragma unroll
                for (int j = 0; j < 8; ++j, yp += step4)
                    if (j * 4 + rsub < n_rows && left >= per16) *reinterpret_cast<uint4*>(yp) = v[j];
                if (__any_sync(0xffffffffu, left > 0 && left < per16)) {
                    // a right edge narrower than 16 bytes, element by element
#pragma unroll 1
                    for (int j = 0; j < 8; ++j) {
                        const int row = j * 4 + rsub;
                        if (row < n_rows && left > 0 && left < per16)
                            for (int i = 0; i < left * es; i += 2) {
                                uint16_t x;
                                asm volatile("ld.shared.u16 %0, [%1];" : "=h"(x) : "r"(stg + row * 128 + ((u ^ (row & 7)) << 4) + i));
                                *reinterpret_cast<uint16_t*>(yp0 + j * step4 + i) = x;
                            }
                    }
                }
                __syncwarp();   // the staging tile is read before the next chunk overwrites it
            }
        }
    }

    // ------------------------------------------------------------ teardown (normal and aborted)
    // a CTA that gave up tells its peer, whose waits would otherwise run to their own limit
    __syncwarp();
    if (abort_flag_s && lane == 0) st_cluster_u32(cluster_map(smem_u32(&abort_flag_s), rank ^ 1), 1);
    tc_fence_before_sync();
    __syncwarp();
    cluster_arrive();
    cluster_wait();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after_sync();
        tmem_dealloc_pair(tmem_base, kTmemCols);
    }
    if (threadIdx.x == 0 && abort_flag_s) atomicExch(p.status, static_cast<int>(PRQ_ERR_TIMEOUT));
}

}  // namespace

cudaError_t launch_gemm_grouped_pair(const CUtensorMap& tm_act, const CUtensorMap& tm_w, const CUtensorMap& tm_sfa,
                                     const CUtensorMap& tm_sfw, const GemmParams& p, int pairs, cudaStream_t stream) {
    constexpr int BN = kPrefillTileWide;
    static OncePerDevice opt_in;
    const cudaError_t e = opt_in([] { return cudaFuncSetAttribute(gemm_grouped_pair_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, gp_smem<BN>()); });
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * pairs);
    cfg.blockDim = dim3(kGpThreads);
    cfg.dynamicSmemBytes = gp_smem<BN>();
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, gemm_grouped_pair_kernel<BN>, tm_act, tm_w, tm_sfa, tm_sfw, p);
}

}  // namespace prq
