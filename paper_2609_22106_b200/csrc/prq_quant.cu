// Activation quantisation kernel: the one MXFP4 quantisation of the reordered activation per layer call
// (Kernel design paragraph; Eq. (1) activation side when the scale and permutation are applied online).
//
// One CTA owns 128 rows x 128 columns: exactly one 512-byte scale atom of the GEMM's layout.  In
// identity mode a lane takes one whole 32-element block (a row of the tile is 4 lanes, a warp covers
// eight rows per step, two steps), with all eight 16-byte loads of a lane issued first, so that about
// 100 KB per SM are in flight -- the kernel is HBM-bound (2 bytes read + 0.5 + 1/32 written per element),
// latency is hidden by loads in flight rather than by occupancy, and the instruction count per element
// is what decides how close it gets (8 elements per lane: 11.3 us, 16: 10.3 us, 32: 9.8 us at 2048 x
// 9728).  Block amax by packed 16-bit maxima without any shuffle, E8M0 byte from the exponent field, 32
// round-to-nearest-even E2M1 conversions per lane, one 16-byte packed store per lane.  (Scale +
// permute mode keeps 8 elements per lane and 4 lanes per block.)  The atom's scale bytes are collected in shared memory and
// written out as one coalesced 512-byte piece; the bytes of tail blocks are also duplicated into the
// residual stages, which is all the "tail copy" this design needs (the GEMM re-reads the tail codes).
//
// The scale + permute mode has two structures.  quant_act_cols_kernel (see there) brings whole rows into shared memory
// by bulk copies and keeps the columns with the lanes.  The column-atom CTAs of quant_act_kernel serve what it does not serve
// better: very wide rows, and some calls on few rows (the launcher has the lines and what both measured there).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdlib>
#include <type_traits>

#include "prq_internal.h"
#include "prq_kernels.h"
#include "prq_ptx.cuh"
#include "prq_quant_block.cuh"

namespace prq {
namespace {

constexpr int kQuantThreads = 256;
constexpr int kAtomK = 128;    // columns per CTA (4 blocks = one scale atom)
constexpr int kSteps = kGroupRows / (2 * (kQuantThreads / 32));  // 8 steps of 16 rows
constexpr int kPermBatch = 4;   // scale + permute mode: steps whose loads are in flight together

// Scale byte from the block's largest magnitude given as fp32 bits: biased exponent - 2, floored at 0.
__device__ __forceinline__ uint32_t scale_byte(uint32_t amax_f32_bits) {
    const int eb = static_cast<int>(amax_f32_bits >> 23) - 2;
    return eb < 0 ? 0u : static_cast<uint32_t>(eb);
}

// Eight values (as fp32) -> 4 bytes of codes under the block scale 2^(byte - 127).
__device__ __forceinline__ uint32_t encode8(const float (&v)[8], uint32_t byte) {
    const float inv = __uint_as_float((254u - byte) << 23);  // 2^(127 - byte), exact multiply
    return cvt_e2m1x8(v[0] * inv, v[1] * inv, v[2] * inv, v[3] * inv, v[4] * inv, v[5] * inv, v[6] * inv, v[7] * inv);
}

// A launch on few rows leaves the memory idle, and the product behind it then waits for its weights: every CTA asks for its
// share of them (`part` of `parts`) in L2.  Weights depend on no kernel, so this needs no wait.  Quantise + multiply, us:
// 2560 x 9728, k = 256, at 16 / 64 / 128 tokens 7.13 / 9.21 / 11.33 -> 6.39 / 8.51 / 10.72, 4096 x 2560, k = 128, 5.26 / 7.01 / 8.86 -> 5.12 /
// 6.78 / 7.99, 9728 x 2560, k = 256, 6.57 / 7.75 / 9.81 -> 6.42 / 7.01 / 9.04.  (Not for stacked experts: 89 MB keep the memory busy longer than the
// quantiser runs, and its rows wait behind them; 64 tokens over 128 experts 27.5 -> 29.9.)
__device__ __forceinline__ void ask_for(const uint8_t* base, uint32_t bytes, int part, int parts) {
    const uint32_t share = ((bytes + parts - 1) / parts + 127) & ~127u, at = share * part;
    if (at < bytes) prefetch_l2(base + at, min(share, (bytes - at)) & ~15u);
}

// The hints are parameters of instances of their own: 100 bytes more in the parameters of every launch made the quantiser
// 0.06 - 0.1 us slower alone and up to 4 % at 2048 rows (2560 x 9728 10.7 -> 11.1 us, 256 x 256 at 16 tokens 1.54 -> 1.63).
constexpr int kAskNothing = 0, kAskRows = 1, kAskWeights = 2;   // (the last one: both)
template <int kAsk>
struct AskParam {};
template <>
struct AskParam<kAskWeights> : WeightHints {};

template <bool kScalePerm, bool kBatch, int kAsk>
__global__ void __launch_bounds__(kQuantThreads, kScalePerm ? 3 : 4)
quant_act_kernel(const QuantBatch b, const __grid_constant__ AskParam<kAsk> ask) {
    __shared__ __align__(16) uint8_t sf_atom[512];
    __shared__ int s_tile_start[kMaxExperts + 1];

    // Launched with programmatic stream serialisation: this CTA may be running while the previous kernel
    // of the stream still is.  Nothing that an earlier kernel may write or still read is touched before the
    // wait (x may be that kernel's output, and it may still be reading the buffers written here); the
    // layer's own permutation and reciprocal scales are constants of the prepared weights, and a dense
    // launch requests them first so that their latency overlaps the wait.
    grid_launch_dependents();

    // which of the batched layers this CTA works for (one launch may quantise the same activation for
    // several layers, each with its own scale, permutation and outputs)
    // (kBatch = false: a single layer, nothing to look up -- the division alone costs the small-batch
    // launches 0.2 us)
    const int lin = kBatch ? static_cast<int>(blockIdx.y) / b.groups_per_lin : 0;
    QuantParams p;
    p.x = b.x; p.M = b.M; p.ldx = b.ldx; p.K = b.K; p.n_experts = b.n_experts; p.act_groups = b.act_groups;
    p.expert_offsets = b.expert_offsets;
    {
        const QuantLayer& l = b.lay[lin];
        p.k_tail = l.k_tail; p.perm = l.perm; p.inv_s_perm = l.inv_s_perm;
        p.codes = l.codes; p.scales_row = l.scales_row; p.scales_sf = l.scales_sf;
    }
    // Which (128-column atom, 128-row group, share of the group's rows) this CTA takes.  In scale + permute mode the
    // atoms of the tail are some twenty times slower than the others: their source columns are scattered over the
    // whole row, every 2-byte read is a 32-byte sector of its own, and the CTA runs at the rate at which its SM's L1
    // takes sectors (about 20 us for 128 rows against 1 us for a head atom, whose window is nearly contiguous).  A
    // launch could not end before its slowest CTA, which the next kernel of the stream then waited for.  So the tail
    // atoms are cut into `tail_split` shares of the rows each and come first in the grid, the head atoms after them
    // (quantise + multiply, K = 28672, k = 256, without / with: 300 rows 43.5 / 30.2 us, 1024: 88 / 60, 4096: 198 / 183).
    // (counted over the whole layer: the tail units of ALL row groups precede every head atom.)
    int group = static_cast<int>(blockIdx.y) - lin * b.groups_per_lin;
    int atom = blockIdx.x, tail_share = 0, tail_split = 1;
    if (kScalePerm && b.n_tail > 0) {
        const int units = b.n_tail * b.tail_split, n_head = b.n_atoms - b.n_tail;
        const int id = group * static_cast<int>(gridDim.x) + atom, first = units * b.groups_per_lin;
        if (id < first) {
            group = id / units;
            const int u = id - group * units;
            tail_split = b.tail_split; tail_share = u % tail_split; atom = n_head + u / tail_split;
        } else {
            const int r = id - first;
            group = r / n_head; atom = r - group * n_head;
        }
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int half = lane >> 4, hl = lane & 15;   // which of the warp's two rows, lane inside the row
    float inv_s[8];
    int src[8];
    auto load_layer_constants = [&](int expert_) {
        const int c0 = atom * kAtomK + hl * 8;
        if (c0 < p.K) {
            const int32_t* perm = p.perm + static_cast<size_t>(expert_) * p.K + c0;
            const float* isp = p.inv_s_perm + static_cast<size_t>(expert_) * p.K + c0;
            const int4 p0 = *reinterpret_cast<const int4*>(perm), p1 = *reinterpret_cast<const int4*>(perm + 4);
            const float4 s0 = *reinterpret_cast<const float4*>(isp), s1 = *reinterpret_cast<const float4*>(isp + 4);
            src[0] = p0.x; src[1] = p0.y; src[2] = p0.z; src[3] = p0.w;
            src[4] = p1.x; src[5] = p1.y; src[6] = p1.z; src[7] = p1.w;
            inv_s[0] = s0.x; inv_s[1] = s0.y; inv_s[2] = s0.z; inv_s[3] = s0.w;
            inv_s[4] = s1.x; inv_s[5] = s1.y; inv_s[6] = s1.z; inv_s[7] = s1.w;
        }
    };
    const bool dense = p.expert_offsets == nullptr;
    if constexpr (kAsk == kAskWeights) {
        if (threadIdx.x == 0) {
            const int parts = static_cast<int>(gridDim.x * gridDim.z) * b.groups_per_lin;
            const int part = static_cast<int>(blockIdx.x + gridDim.x * (blockIdx.z + gridDim.z * (blockIdx.y - lin * b.groups_per_lin)));
            ask_for(ask.lay[lin].codes, ask.lay[lin].code_bytes, part, parts);
            ask_for(ask.lay[lin].sf, ask.lay[lin].sf_bytes, part, parts);
        }
    }
    if (kScalePerm && dense) load_layer_constants(0);
    // Identity mode: this CTA's rows in L2 before the wait, one 128-byte line per thread.  The CTAs that come up beside the GEMM
    // before this launch (four per SM) thereby read memory while that computes.  A hint only: what an earlier kernel still writes
    // is read behind the wait.  Quantise + multiply, 2560 x 9728, 512 / 2048 (fp32 y) / 2048 / 4096 tokens: 23.4 / 33.2 / 32.3 / 65.5 ->
    // 22.2 / 32.0 / 31.2 / 62.0 us, 9728 x 2560 at 3000: 41.7 -> 41.0.  (Asking for the rows of the CTAs behind them too disturbs the
    // one-wave GEMM: 33.6 with fp32 y.)  Alone the quantiser only pays for it, 2 to 7 % (2560 x 9728 at 2048 tokens 7.41 -> 7.70).
    if (!kScalePerm && kAsk) {
        const int row = group * kGroupRows + (threadIdx.x >> 1), col = atom * kAtomK + (threadIdx.x & 1) * 64;
        if (row < p.M && col < p.K) asm volatile("prefetch.global.L2 [%0];" ::"l"(p.x + static_cast<size_t>(row) * p.ldx + col));
    }
    grid_dependency_wait();

    // Which rows does this CTA own?  Dense: group g covers rows [128 g, 128 g + 128).  Grouped: the
    // scale groups are padded per expert, so walk the expert offsets to find ours.
    int row0, row_end, expert = 0;
    if (p.expert_offsets == nullptr) {
        row0 = group * kGroupRows;
        row_end = min(p.M, row0 + kGroupRows);
    } else {
        if (threadIdx.x < 32) warp_expert_starts(p.expert_offsets, p.n_experts, kGroupRows, s_tile_start, nullptr);
        __syncthreads();
        if (group >= s_tile_start[p.n_experts]) return;  // padding CTA of the launch grid
        int lo = 0, hi = p.n_experts - 1;
        while (lo < hi) {  // last expert whose first tile is <= group
            int mid = (lo + hi + 1) >> 1;
            if (s_tile_start[mid] <= group) lo = mid; else hi = mid - 1;
        }
        expert = lo;
        row0 = p.expert_offsets[expert] + (group - s_tile_start[expert]) * kGroupRows;
        row_end = min(p.expert_offsets[expert + 1], row0 + kGroupRows);
    }

    if (threadIdx.x < 128) reinterpret_cast<uint32_t*>(sf_atom)[threadIdx.x] = 0;
    __syncthreads();

    const int K = p.K, k_tail = p.k_tail;
    const int col0 = atom * kAtomK + hl * 8;      // first of this lane's 8 columns
    const bool col_ok = col0 < K;                 // K % 32 == 0, so a lane is all in or all out
    const int blk_in_atom = hl >> 2;
    const int gblk = atom * (kAtomK / kBlock) + blk_in_atom;
    const int tail_blk0 = (K - k_tail) / kBlock;  // first tail block (global block index)
    const StagePlan plan(K, k_tail);
    const int stage = atom >> 1;
    uint8_t* sf_base = p.scales_sf;
    const size_t sf_stage_stride = static_cast<size_t>(p.act_groups) * kSfGroupBytes;
    uint8_t* sf_group = sf_base + static_cast<size_t>(group) * kSfGroupBytes;
    const int n_rows = row_end - row0;            // 1..128
    // With few groups the rows of a group are split over gridDim.z CTAs (1, 2, 4 or 8 parts of whole
    // 16-row steps) so that a small batch still fills the GPU; only the scale + permute mode is split.
    const int n_parts = kScalePerm ? static_cast<int>(gridDim.z) * tail_split : 1;
    const int part = kScalePerm ? static_cast<int>(blockIdx.z) * tail_split + tail_share : 0;
    const int part_steps = kSteps / n_parts;

    if (kScalePerm && !dense) load_layer_constants(expert);   // grouped: the expert is known only now

    // row of step i: 16 rows per step, 2 per warp
    auto row_of = [&](int i) { return i * 16 + warp * 2 + half; };

    if (!kScalePerm) {
        // ---- identity.  Here a lane takes one whole 32-element block (64 contiguous bytes, four 16-byte
        // loads): no shuffle at all, a row of the tile is 4 lanes, a warp covers 8 rows and the tile is
        // done in 2 steps of 64 rows.  All eight loads are issued first, then the arithmetic runs on
        // packed bf16 pairs. ----
        const int l4 = lane & 3, rw = lane >> 2;
        const int c8 = warp * 8 + rw;                        // row inside a 64-row step
        const int colb = atom * kAtomK + l4 * 32;            // first of this lane's 32 columns
        const bool okb = colb < K;                           // K % 32 == 0: a lane is all in or all out
        const int gb = atom * (kAtomK / kBlock) + l4;        // this lane's block
        const uint16_t* xp = p.x + static_cast<size_t>(row0 + c8) * p.ldx + colb;
        const size_t x_step = static_cast<size_t>(64) * p.ldx;
        uint4 q[2][4];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                q[i][h] = make_uint4(0, 0, 0, 0);
                if (okb && i * 64 + c8 < n_rows) q[i][h] = __ldg(reinterpret_cast<const uint4*>(xp + i * x_step + 8 * h));
            }
        }
        uint8_t* cp = p.codes + static_cast<size_t>(row0 + c8) * (K / 2) + colb / 2;
        const size_t c_step = static_cast<size_t>(64) * (K / 2);
        uint8_t* rp = p.scales_row ? p.scales_row + static_cast<size_t>(row0 + c8) * (K / kBlock) + gb : nullptr;
        const size_t r_step = static_cast<size_t>(64) * (K / kBlock);
        const bool tail_lane = okb && gb >= tail_blk0;
        uint8_t* tp = nullptr;                                // this lane's duplicate slot in the residual stages
        if (tail_lane) {
            const int t = gb - tail_blk0;
            tp = sf_group + (plan.S1 + t / 8) * sf_stage_stride + ((t % 8) >> 2) * 512 + ((t % 8) & 3);
        }
        // row r = 64 i + c8 of the group: atom offset (r % 32) * 16 + (r / 32) * 4 + block
        const int in_atom0 = (c8 & 31) * 16 + (c8 >> 5) * 4;
        uint8_t* ap = sf_atom + in_atom0 + l4;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            uint4 packed;
            const uint32_t byte = quant_block32(q[i], packed);
            const bool row_ok = i * 64 + c8 < n_rows;
            if (okb && row_ok) {
                *reinterpret_cast<uint4*>(cp + i * c_step) = packed;
                ap[i * 8] = static_cast<uint8_t>(byte);
                if (rp) rp[i * r_step] = static_cast<uint8_t>(byte);
                if (tail_lane) tp[in_atom0 + i * 8] = static_cast<uint8_t>(byte);
            }
        }
    } else {
        // ---- scale + permute: gathered 2-byte loads (the head of the permutation is nearly the identity,
        // so they coalesce), multiply by the stored reciprocal scale in fp32.  The loads of four steps
        // (32 per lane) are issued before any arithmetic. ----
        // Everything that does not depend on the row is computed once: per-lane pointers that advance by
        // a fixed stride per 16-row step, the lane's slot in the residual stages, and -- for lanes past K --
        // zero sources and factors so that the arithmetic below needs no per-element select.
        const int w2h = warp * 2 + half;                       // row inside a 16-row step
        const size_t x_step = static_cast<size_t>(16) * p.ldx;
        const size_t c_step = static_cast<size_t>(16) * (K / 2);
        const size_t r_step = static_cast<size_t>(16) * (K / kBlock);
        const bool sf_lane = col_ok && (hl & 3) == 0;          // the lane that writes the block's scale byte
        const bool tail_lane = sf_lane && gblk >= tail_blk0;
        uint8_t* tp = nullptr;
        if (tail_lane) {
            const int t = gblk - tail_blk0;
            tp = sf_group + (plan.S1 + t / 8) * sf_stage_stride + ((t % 8) >> 2) * 512 + ((t % 8) & 3);
        }
        if (!col_ok) {
#pragma unroll
            for (int e = 0; e < 8; ++e) { src[e] = 0; inv_s[e] = 0.f; }
        }
#pragma unroll 1
        for (int i0 = part * part_steps; i0 < (part + 1) * part_steps; i0 += kPermBatch) {
            if (i0 * 16 >= n_rows) break;   // nothing but padding rows from here on (their scale bytes are zero already)
            const int rb = i0 * 16 + w2h;   // this lane's row in the batch's first step
            const uint16_t* xb = p.x + static_cast<size_t>(row0 + rb) * p.ldx;
            uint8_t* cp = p.codes + static_cast<size_t>(row0 + rb) * (K / 2) + col0 / 2;
            uint8_t* rp = p.scales_row ? p.scales_row + static_cast<size_t>(row0 + rb) * (K / kBlock) + gblk : nullptr;
            uint32_t raw[kPermBatch][8];
#pragma unroll
            for (int ii = 0; ii < kPermBatch; ++ii) {
                if (ii >= part_steps) break;
                const bool ld_ok = col_ok && rb + 16 * ii < n_rows;
                const uint16_t* xrow = xb + ii * x_step;
#pragma unroll
                for (int e = 0; e < 8; ++e) raw[ii][e] = ld_ok ? static_cast<uint32_t>(__ldg(xrow + src[e])) : 0u;
            }
#pragma unroll
            for (int ii = 0; ii < kPermBatch; ++ii) {
                if (ii >= part_steps) break;
                const int r = rb + 16 * ii;
                float v[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = __uint_as_float(raw[ii][e] << 16) * inv_s[e];
                const float a01 = fmaxf(fabsf(v[0]), fabsf(v[1])), a23 = fmaxf(fabsf(v[2]), fabsf(v[3]));
                const float a45 = fmaxf(fabsf(v[4]), fabsf(v[5])), a67 = fmaxf(fabsf(v[6]), fabsf(v[7]));
                uint32_t am = __float_as_uint(fmaxf(fmaxf(a01, a23), fmaxf(a45, a67)));
                am = max(am, __shfl_xor_sync(0xffffffffu, am, 1));
                am = max(am, __shfl_xor_sync(0xffffffffu, am, 2));
                const uint32_t byte = scale_byte(am);
                const uint32_t packed = encode8(v, byte);
                if (col_ok && r < n_rows) {
                    *reinterpret_cast<uint32_t*>(cp + ii * c_step) = packed;
                    if (sf_lane) {
                        const int in_atom = (r & 31) * 16 + (r >> 5) * 4;
                        sf_atom[in_atom + blk_in_atom] = static_cast<uint8_t>(byte);
                        if (rp) rp[ii * r_step] = static_cast<uint8_t>(byte);
                        if (tail_lane) tp[in_atom] = static_cast<uint8_t>(byte);
                    }
                }
            }
        }
    }
    __syncthreads();
    // the atom's scale bytes, coalesced (rows past the end and blocks past K stay zero = 2^-127)
    if (n_parts == 1) {
        if (threadIdx.x < 32) {
            reinterpret_cast<uint4*>(sf_group + stage * sf_stage_stride + (atom & 1) * 512)[threadIdx.x] =
                reinterpret_cast<const uint4*>(sf_atom)[threadIdx.x];
        }
    } else if (threadIdx.x < kGroupRows / n_parts) {
        // this part's rows only: the four scale bytes of row r sit at (r % 32) * 16 + (r / 32) * 4
        const int r = part * (kGroupRows / n_parts) + threadIdx.x;
        const int off = (r & 31) * 16 + (r >> 5) * 4;
        *reinterpret_cast<uint32_t*>(sf_group + stage * sf_stage_stride + (atom & 1) * 512 + off) =
            *reinterpret_cast<const uint32_t*>(sf_atom + off);
    }
    if (part != 0) return;
    const int n_atoms = b.n_atoms;
    // An odd atom count leaves the second half of the last main stage without an owner: zero it.
    if (atom == n_atoms - 1 && (n_atoms & 1) && threadIdx.x >= 32 && threadIdx.x < 64)
        reinterpret_cast<uint4*>(sf_group + stage * sf_stage_stride + 512)[threadIdx.x - 32] = make_uint4(0, 0, 0, 0);
    // The CTA of the last atom also zero-fills what nobody else writes in the residual stages:
    // blocks past k_tail, and every byte of rows past the end of the group.
    if (atom == n_atoms - 1 && plan.S > plan.S1) {
        const int nb = kStageK / kBlock;
        for (int idx = threadIdx.x; idx < (plan.S - plan.S1) * kGroupRows * nb; idx += kQuantThreads) {
            const int ts = idx / (kGroupRows * nb);
            const int r = (idx / nb) % kGroupRows;
            const int b = idx % nb;
            const bool live = (r < n_rows) && (ts * nb + b) < k_tail / kBlock;
            if (!live) sf_group[(plan.S1 + ts) * sf_stage_stride + sf_offset_in_group(r, b)] = 0;
        }
    }
}


// ---------------------------------------------------------------------------------------------------------
// Scale + permute mode, second structure: columns stay with their lanes.  A lane owns kCols consecutive destination
// columns of one layer and keeps their source offsets and reciprocal scales in registers while rows stream past it:
// whole rows arrive in shared memory by bulk copies (one warp does nothing else), and every gather of the permutation
// is a 2-byte shared-memory read.
//
// Why.  The mode is bound by instruction issue and by a launch's fixed latencies, not by memory (2.53 bytes per element).
// Gathering from global memory costs about 20 instructions per element (64-bit addresses, one 32-byte sector per
// scattered 2-byte read).  Rows that stay with their lanes need a 16-byte record per column pair fetched from shared
// memory for every row (12.7 per element), and the records of a wide layer (K = 9728) do not fit beside its rows.  Here
// the core is 5 per element -- gather, its address, widening, two packed fp32 products and a conversion per pair, half
// a three-input maximum -- and 10.5 - 10.7 in all at 4096 x 2560 (ncu), where a CTA sees only three or four slices; a row is
// all that shared memory holds.  Measured figures stand at the launcher.  Of the 8.9 us at 4096 x 2560 (2.53 B per
// element: 4.1 us of memory time) about 3 are set-up, the first rows' latency and the last stores.
//
// The lanes of a warp read the same row, kCols columns apart: where the permutation is locally the identity, four
// (eight) lanes would meet in a bank.  A lane therefore walks its columns from another start (`rot`, chosen from its
// first source column so that the lanes of a bank group read different words), which one rotation of the packed
// codes undoes.
//
// A slice is kRowsC rows of one 128-row group.  The block maxima of two rows travel in one register (only exponents
// are needed), the four scale bytes of (row, atom) meet by shuffles and leave as the one word the GEMM's layout has
// for them; tail bytes are stored once more where the residual stages read them.  Rows and blocks that do not exist
// get zero bytes.  gridDim.y cuts the columns where the warps of one CTA do not cover them, gridDim.z runs over
// batched layers.
struct ColsPlan {
    int n_slices;        // slices of all 128-row groups (grouped: of all groups the launch could need)
    int n_stages;        // slices of rows in flight per CTA
    int warps;           // computing warps per CTA (one more loads the rows)
    int strided;         // a CTA takes slices g, g + G, ... instead of consecutive ones (one 128-row group only)
};
constexpr int kColsMaxStages = 8;
constexpr size_t kColsSmem = 220 * 1024;   // shared memory of an SM that the rows in flight may take

__device__ __forceinline__ const QuantBatch& batch_of(const QuantBatch& b, const ColsPlan&) { return b; }
__device__ __forceinline__ const QuantBatch& batch_of(const ColsPlan&, const QuantBatch& b) { return b; }
__device__ __forceinline__ const ColsPlan& plan_of(const QuantBatch&, const ColsPlan& c) { return c; }
__device__ __forceinline__ const ColsPlan& plan_of(const ColsPlan& c, const QuantBatch&) { return c; }

// kCols: columns per lane, 8 or 16.  kRowsC: rows per slice, 1, 2 or 4.
// With hints the plan stands in front of the batch, so that what every CTA reads first shares two 64-byte lines of parameters (2560 x
// 9728 at 64 tokens 9.23 -> 8.49 us with the product behind it, 4096 x 2560 7.13 -> 6.78).
template <int kCols, int kRowsC, bool kGrouped, int kMaxT, bool kAsk>
__global__ void __launch_bounds__(kMaxT, 1)
quant_act_cols_kernel(const std::conditional_t<kAsk, ColsPlan, QuantBatch> first, const std::conditional_t<kAsk, QuantBatch, ColsPlan> second,
                      const __grid_constant__ AskParam<kAsk ? kAskWeights : kAskNothing> ask) {
    const QuantBatch& b = batch_of(first, second);
    const ColsPlan& plan_c = plan_of(first, second);
    constexpr int kPairs = kCols / 2;
    constexpr int kBlkLanes = kBlock / kCols;            // lanes per 32-element block: 4 or 2
    constexpr int kAtomLanes = kAtomK / kCols;           // lanes per scale atom: 16 or 8
    constexpr int kBankLanes = 64 / kCols;               // lanes whose columns take the 32 banks once: 8 or 4
    constexpr int kSlicesC = kGroupRows / kRowsC;        // slices per group
    extern __shared__ __align__(128) uint8_t cols_smem[];
    __shared__ __align__(8) uint64_t bar_full[kColsMaxStages], bar_empty[kColsMaxStages];
    __shared__ int s_tile_start[kGrouped ? kMaxExperts + 1 : 1];
    __shared__ int s_row_start[kGrouped ? kMaxExperts + 1 : 1];
    __shared__ int abort_flag_s;
    volatile int* abort_flag = &abort_flag_s;
    grid_launch_dependents();
    const int K = b.K, nblk = K / kBlock;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_stages = plan_c.n_stages, n_warps = plan_c.warps;
    const bool loader = warp == n_warps;
    const uint32_t row_bytes = static_cast<uint32_t>(K) * 2, stage_bytes = kRowsC * row_bytes;
    const QuantLayer& l = b.lay[blockIdx.z];
    if (threadIdx.x == 0) {
        for (int i = 0; i < kColsMaxStages; ++i) { mbar_init(smem_u32(&bar_full[i]), 1); mbar_init(smem_u32(&bar_empty[i]), n_warps); }
        abort_flag_s = 0;
        fence_mbar_init();
    }

    // this lane's columns, block and place in the block
    const int my = (static_cast<int>(blockIdx.y) * n_warps + warp) * 32 + lane;   // lane index over the whole row
    const int col0 = my * kCols;
    const bool col_ok = !loader && col0 < K;             // K % 32 == 0: a lane is all in or all out
    uint32_t src[kCols];                                 // byte offsets in a row; slot u = column (u + rot) % kCols
    uint64_t inv2[kPairs];
    uint32_t rot = 0;
    auto load_constants = [&](int expert) {
        const int4* pp = reinterpret_cast<const int4*>(l.perm + static_cast<size_t>(expert) * K + col0);
        const uint4* ip = reinterpret_cast<const uint4*>(l.inv_s_perm + static_cast<size_t>(expert) * K + col0);
        uint32_t inv[kCols];
#pragma unroll
        for (int i = 0; i < kCols / 4; ++i) {
            int4 p4 = make_int4(0, 0, 0, 0);
            uint4 s4 = make_uint4(0, 0, 0, 0);
            if (col_ok) { p4 = __ldg(pp + i); s4 = __ldg(ip + i); }
            src[4 * i] = p4.x; src[4 * i + 1] = p4.y; src[4 * i + 2] = p4.z; src[4 * i + 3] = p4.w;
            inv[4 * i] = s4.x; inv[4 * i + 1] = s4.y; inv[4 * i + 2] = s4.z; inv[4 * i + 3] = s4.w;
        }
        rot = (2u * (lane / kBankLanes) - src[0]) % kCols;
#pragma unroll
        for (int d = 1; d < kCols; d <<= 1) {
            uint32_t a[kCols], c[kCols];
#pragma unroll
            for (int u = 0; u < kCols; ++u) { a[u] = (rot & d) ? src[(u + d) % kCols] : src[u]; c[u] = (rot & d) ? inv[(u + d) % kCols] : inv[u]; }
#pragma unroll
            for (int u = 0; u < kCols; ++u) { src[u] = a[u]; inv[u] = c[u]; }
        }
#pragma unroll
        for (int u = 0; u < kCols; ++u) src[u] *= 2;
#pragma unroll
        for (int t = 0; t < kPairs; ++t) inv2[t] = pack_f32x2(inv[2 * t], inv[2 * t + 1]);
    };
    __syncthreads();
    if (!kGrouped) {
        // a dense layer's constants belong to the prepared weights, not to an earlier kernel of the stream
        if (!loader) load_constants(0);
        if constexpr (kAsk) {
            if (loader && lane == 0) {
                const int part = blockIdx.x + gridDim.x * blockIdx.y, parts = gridDim.x * gridDim.y;
                ask_for(ask.lay[blockIdx.z].codes, ask.lay[blockIdx.z].code_bytes, part, parts);
                ask_for(ask.lay[blockIdx.z].sf, ask.lay[blockIdx.z].sf_bytes, part, parts);
            }
        }
        grid_dependency_wait();
    } else {
        grid_dependency_wait();
        // the experts' row ranges, once per CTA
        for (int e = threadIdx.x; e <= b.n_experts; e += blockDim.x) s_row_start[e] = b.expert_offsets[e];
        __syncthreads();
        if (threadIdx.x < 32) warp_expert_starts(s_row_start, b.n_experts, kGroupRows, s_tile_start, nullptr);
        __syncthreads();
    }
    const int n_slices = kGrouped ? min(plan_c.n_slices, s_tile_start[b.n_experts] * kSlicesC) : plan_c.n_slices;

    // A CTA's slices are consecutive (with stacked experts the constants then change a few times, not per slice), and
    // the CTAs' shares differ by one slice at most.  A few rows of one dense group are dealt out in turn instead: the
    // group's padding follows its rows, and nobody then has two slices of rows beside others that have none.
    const int G = static_cast<int>(gridDim.x), g = static_cast<int>(blockIdx.x);
    const int base = n_slices / G, extra = n_slices - base * G;
    const bool strided = !kGrouped && plan_c.strided;
    const int sl_begin = strided ? g : g * base + min(g, extra), n_mine = base + (g < extra ? 1 : 0);
    const int step_rows = strided ? G * kRowsC : kRowsC;
    // where a slice sits: its group, its first row inside the group, the expert and the rows (in x) of the group
    int group = sl_begin / kSlicesC, r_first = (sl_begin % kSlicesC) * kRowsC, expert = 0, g_row0 = 0, g_end = 0;
    auto enter_group = [&]() {
        if (!kGrouped) {
            g_row0 = group * kGroupRows; g_end = min(b.M, g_row0 + kGroupRows);
        } else {
            while (s_tile_start[expert + 1] <= group) ++expert;   // last expert whose first group is <= group
            g_row0 = s_row_start[expert] + (group - s_tile_start[expert]) * kGroupRows;
            g_end = min(s_row_start[expert + 1], g_row0 + kGroupRows);
        }
    };
    auto next_slice = [&]() {
        r_first += step_rows;
        if (r_first >= kGroupRows) { r_first -= kGroupRows; ++group; return true; }
        return false;
    };
    if (n_mine > 0) {
        if (kGrouped) {
            int lo = 0, hi = b.n_experts - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (s_tile_start[mid] <= group) lo = mid; else hi = mid - 1;
            }
            expert = lo;
        }
        enter_group();
    }

    int it = 0;   // slices whose rows were asked for (the loading warp)
    if (loader) {
        int st = 0;
        uint32_t ph = 0;
        for (int i = 0; i < n_mine; ++i) {
            const int row0 = g_row0 + r_first, n_rows = min(kRowsC, g_end - row0);
            if (n_rows > 0) {
                if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_empty[st]), ph ^ 1, abort_flag))) break;
                const uint32_t full = smem_u32(&bar_full[st]);
                if (lane == 0) mbar_arrive_expect_tx(full, n_rows * row_bytes);
                __syncwarp();
                if (lane < n_rows)
                    bulk_load(smem_u32(cols_smem) + st * stage_bytes + lane * row_bytes, b.x + static_cast<size_t>(row0 + lane) * b.ldx, row_bytes, full);
                ++it;
                if (++st == n_stages) { st = 0; ph ^= 1; }
            }
            if (next_slice() && i + 1 < n_mine) enter_group();
        }
    } else {
        const StagePlan plan(K, l.k_tail);
        const int blk = my / kBlkLanes, sub = my % kBlkLanes, ba = blk & 3;   // block of the row, lane in it, block of its atom
        const int atom = blk >> 2;
        const int n_tail_blk = l.k_tail / kBlock, tail_t = blk - (nblk - n_tail_blk);   // >= 0: a tail block
        const int n_res = (plan.S - plan.S1) * (kStageK / kBlock);                      // block positions of the residual stages
        const size_t sf_stage_stride = static_cast<size_t>(b.act_groups) * kSfGroupBytes;
        // the pointers that every slice needs, held in registers (the layer is looked up with an index)
        uint8_t* codes = l.codes + col0 / 2;
        uint8_t* sf_atom = l.scales_sf + (atom >> 1) * sf_stage_stride + (atom & 1) * 512;
        uint8_t* sf_tail = l.scales_sf + (plan.S1 + (max(tail_t, 0) >> 3)) * sf_stage_stride + ((tail_t >> 2) & 1) * 512 + (tail_t & 3);
        asm volatile("" : "+l"(codes), "+l"(sf_atom), "+l"(sf_tail));
        const bool has_row_scales = l.scales_row != nullptr;
        const bool word_lane = ba == 0 && atom < 2 * plan.S1;   // an odd atom count leaves half a stage that must read as zeros
        const bool tail_lane = col_ok && tail_t >= 0;
        const bool fill = n_res > n_tail_blk && blockIdx.y == 0;
        const uint32_t smem0 = smem_u32(cols_smem), code_row = K / 2;
        int st = 0, expert_now = kGrouped ? -1 : 0;
        uint32_t ph = 0;
        for (int i_sl = 0; i_sl < n_mine; ++i_sl) {
            const int row0 = g_row0 + r_first, n_rows = min(kRowsC, g_end - row0);   // n_rows <= 0: padding of the group
            uint32_t bytes[kRowsC];
#pragma unroll
            for (int r = 0; r < kRowsC; ++r) bytes[r] = 0;
            if (n_rows > 0) {
                if (kGrouped && expert != expert_now) { load_constants(expert); expert_now = expert; }
                if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_full[st]), ph, abort_flag))) break;
                const uint32_t sbase = smem0 + st * stage_bytes;
                uint64_t v[kRowsC][kPairs];
                float am[kRowsC];
#pragma unroll
                for (int r = 0; r < kRowsC; ++r) {
                    // rows that do not exist read the last one that does; their results are dropped below
                    const uint32_t rb = sbase + min(r, n_rows - 1) * row_bytes;
#pragma unroll
                    for (int p = 0; p < kPairs; ++p) {
                        uint32_t x0, x1;
                        asm volatile("{\n\t.reg .b16 h;\n\tld.shared.b16 h, [%1];\n\tmov.b32 %0, {0, h};\n\t}" : "=r"(x0) : "r"(rb + src[2 * p]));
                        asm volatile("{\n\t.reg .b16 h;\n\tld.shared.b16 h, [%1];\n\tmov.b32 %0, {0, h};\n\t}" : "=r"(x1) : "r"(rb + src[2 * p + 1]));
                        v[r][p] = mul_f32x2(pack_f32x2(x0, x1), inv2[p]);
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bar_empty[st]));   // every value of the slice is in registers
                if (++st == n_stages) { st = 0; ph ^= 1; }
#pragma unroll
                for (int r = 0; r < kRowsC; ++r) {
                    am[r] = 0.f;
#pragma unroll
                    for (int p = 0; p < kPairs; ++p) {
                        float lo, hi;
                        unpack_f32x2(v[r][p], lo, hi);
                        am[r] = max3_abs(am[r], lo, hi);
                    }
                }
                // largest exponent over the block's lanes, two rows per register
#pragma unroll
                for (int r = 0; r < kRowsC; r += 2) {
                    uint32_t e = __float_as_uint(am[r]) >> 23;
                    if (r + 1 < kRowsC) e |= (__float_as_uint(am[r + 1]) >> 23) << 16;
#pragma unroll
                    for (int d = 1; d < kBlkLanes; d <<= 1) e = __vmaxu2(e, __shfl_xor_sync(0xffffffffu, e, d));
                    bytes[r] = max(static_cast<int>(e & 0xffffu) - 2, 0);
                    if (r + 1 < kRowsC) bytes[r + 1] = max(static_cast<int>(e >> 16) - 2, 0);
                }
                uint8_t* cp = codes + static_cast<size_t>(row0) * code_row;
#pragma unroll
                for (int r = 0; r < kRowsC; ++r) {
                    const uint32_t up = (254u - bytes[r]) << 23;   // 2^(127 - byte), exact multiply
                    const uint64_t up2 = pack_f32x2(up, up);
                    uint32_t pk[kCols / 8];
#pragma unroll
                    for (int h = 0; h < kCols / 8; ++h) {
                        float f[8];
#pragma unroll
                        for (int i = 0; i < 4; ++i) unpack_f32x2(mul_f32x2(v[r][4 * h + i], up2), f[2 * i], f[2 * i + 1]);
                        pk[h] = cvt_e2m1x8(f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7]);
                    }
                    // nibble u holds column (u + rot) % kCols: put them in order by a rotation of the packed word(s)
                    const bool live = col_ok && r < n_rows;
                    if (kCols == 8) {
                        pk[0] = __funnelshift_l(pk[0], pk[0], 4 * rot);
                        if (live) *reinterpret_cast<uint32_t*>(cp) = pk[0];
                    } else {
                        const uint32_t lo = (rot & 8) ? pk[kCols / 8 - 1] : pk[0], hi = (rot & 8) ? pk[0] : pk[kCols / 8 - 1];
                        const uint2 w = make_uint2(__funnelshift_l(hi, lo, 4 * (rot & 7)), __funnelshift_l(lo, hi, 4 * (rot & 7)));
                        if (live) *reinterpret_cast<uint2*>(cp) = w;
                    }
                    cp += code_row;
                    bytes[r] = live ? bytes[r] : 0u;
                }
                if (has_row_scales && sub == 0 && col_ok) {
#pragma unroll
                    for (int r = 0; r < kRowsC; ++r)
                        if (r < n_rows) l.scales_row[static_cast<size_t>(row0 + r) * nblk + blk] = static_cast<uint8_t>(bytes[r]);
                }
            }
            const size_t group_off = static_cast<size_t>(group) * kSfGroupBytes;
            // the lanes of a block share out the slice's rows: lane `sub` brings the words of rows sub, sub + lanes, ...
#pragma unroll
            for (int r0 = 0; r0 < kRowsC; r0 += kBlkLanes) {
                uint32_t mine = bytes[r0];
#pragma unroll
                for (int i = 1; i < kBlkLanes; ++i)
                    if (r0 + i < kRowsC) mine = sub == i ? bytes[r0 + i] : mine;
                const int r = r0 + sub;
                const int gr = r_first + r, off = (gr & 31) * 16 + (gr >> 5) * 4;   // row inside its group
                uint32_t w = mine << (8 * ba);
#pragma unroll
                for (int d = kBlkLanes; d < kAtomLanes; d <<= 1) w |= __shfl_xor_sync(0xffffffffu, w, d);
                if (r < kRowsC && word_lane) *reinterpret_cast<uint32_t*>(sf_atom + group_off + off) = w;
                if (r < kRowsC && tail_lane) sf_tail[group_off + off] = static_cast<uint8_t>(mine);
            }
            // residual block positions past the tail
            if (fill) {
                uint8_t* const sf_res = l.scales_sf + group_off + plan.S1 * sf_stage_stride;
                for (int i = static_cast<int>(threadIdx.x); i < (n_res - n_tail_blk) * kRowsC; i += n_warps * 32) {
                    const int p = n_tail_blk + i / kRowsC, gr = r_first + i % kRowsC;
                    sf_res[(p >> 3) * sf_stage_stride + sf_offset_in_group(gr, p & 7)] = 0;
                }
            }
            if (next_slice() && i_sl + 1 < n_mine) enter_group();
        }
    }
    __syncthreads();
    // gave up: let the copies in flight land before the CTA's shared memory is given up (bounded)
    if (loader && lane == 0 && abort_flag_s)
        for (int j = max(0, it - n_stages); j < it; ++j)
            mbar_wait_after_abort(smem_u32(&bar_full[j % n_stages]), (j / n_stages) & 1);
    if (threadIdx.x == 0 && abort_flag_s && b.status) atomicExch(b.status, static_cast<int>(PRQ_ERR_TIMEOUT));
}

// Registers of one instance as built (they decide how many of its CTAs an SM holds).
template <int kCols, int kRowsC, bool kGrouped, int kMaxT, bool kAsk = false>
cudaError_t launch_cols_impl(const QuantBatch& b, int sm_count, cudaStream_t stream, const WeightHints* ask = nullptr) {
    auto kernel = quant_act_cols_kernel<kCols, kRowsC, kGrouped, kMaxT, kAsk>;
    const int lanes = (b.K + kStageK - 1) / kStageK * (kStageK / kCols);
    const int all_warps = (lanes + 31) / 32, max_warps = kMaxT / 32 - 1;
    const int chunks = (all_warps + max_warps - 1) / max_warps, warps = (all_warps + chunks - 1) / chunks;
    static std::atomic<int> regs{0};   // the same on every device
    static OncePerDevice opt_in;
    const cudaError_t e = opt_in([&] {
        cudaError_t r = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kColsSmem - (kGrouped ? 9216 : 0));
        cudaFuncAttributes fa;
        if (r == cudaSuccess) r = cudaFuncGetAttributes(&fa, kernel);
        if (r == cudaSuccess) regs.store(fa.numRegs);
        return r;
    });
    if (e != cudaSuccess) return e;
    const int threads = 32 * (warps + 1);
    const size_t stage = static_cast<size_t>(kRowsC) * b.K * 2;
    // CTAs per SM: as many as the registers hold, while each still has room for three slices of rows
    int per_sm = 65536 / (((regs.load() + 7) / 8 * 8) * threads);
    per_sm = per_sm < 1 ? 1 : per_sm > 16 ? 16 : per_sm;
    const size_t fixed = 1024 + (kGrouped ? 8 * (kMaxExperts + 1) : 0) + 256;
    while (per_sm > 1 && kColsSmem / per_sm < 3 * stage + fixed) --per_sm;
    // slices in flight: about 100 KB per SM hide the memory latency
    size_t n_stages = (kColsSmem / per_sm - fixed) / stage;
    const size_t in_flight = (98304 / per_sm + stage - 1) / stage;
    n_stages = n_stages > in_flight ? in_flight : n_stages;
    n_stages = n_stages > kColsMaxStages ? kColsMaxStages : n_stages < 2 ? 2 : n_stages;
    ColsPlan cp;
    cp.n_slices = b.groups_per_lin * (kGroupRows / kRowsC);
    cp.n_stages = static_cast<int>(n_stages);
    cp.warps = warps;
    cp.strided = 0;
    int want = per_sm * sm_count / (chunks * b.n_lin);
    // a CTA of a grouped launch first looks the experts up: two slices at least, or that is all it does
    if (kGrouped && want > cp.n_slices / 2) want = cp.n_slices / 2;
    // A launch on a few rows must leave room for the CTAs of the next one, which set themselves up beside it.  Where it would
    // take more than two thirds of the CTAs the GPU holds, half as many take two slices each (rows first, padding last).
    // Quantise + multiply, three layers of K = 2560 (q / k / v, 384 of 444 places), 1 / 16 / 64 tokens: 8.5 / 9.1 / 9.9 ->
    // 6.5 / 7.0 / 9.0 us; four layers 9.6 / 9.9 / 11.0 -> 7.2 / 7.9 / 10.0; two of K = 8192 6.8 / 7.4 / 9.7 -> 6.4 / 7.0 / 9.5.
    // (Two layers of K = 2560, 256 places, lose by it at 32 tokens: 10.1 -> 10.5.)
    if (!kGrouped && b.M <= kGroupRows) {
        const int grid = want < cp.n_slices ? want : cp.n_slices;
        const int live = (b.M + kRowsC - 1) / kRowsC, half = cp.n_slices / 2, fewer = live > half ? live : half;
        if (3LL * grid * chunks * b.n_lin > 2LL * per_sm * sm_count && fewer < grid) { cp.strided = 1; want = fewer; }
        // Where the CTAs ask for weights, no more stages of rows than a CTA has slices: they then come up beside a GEMM that
        // fills its SMs and ask while it ends.  (Without weights to ask for that only disturbs it: 1024 x 2560 at 16 tokens 4.43 / 4.70.)
        const int g2 = want < 1 ? 1 : want < cp.n_slices ? want : cp.n_slices, mine = ((cp.strided ? live : cp.n_slices) + g2 - 1) / g2;
        if (kAsk && cp.n_stages > mine) cp.n_stages = mine;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(want < 1 ? 1 : want < cp.n_slices ? want : cp.n_slices, chunks, b.n_lin);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = cp.n_stages * stage;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    AskParam<kAsk ? kAskWeights : kAskNothing> asked;
    if constexpr (kAsk) {
        static_cast<WeightHints&>(asked) = *ask;
        return cudaLaunchKernelEx(&cfg, kernel, cp, b, asked);
    } else {
        return cudaLaunchKernelEx(&cfg, kernel, b, cp, asked);
    }
}

}  // namespace

cudaError_t launch_quant_act_batch(const QuantBatch& b, bool scale_perm, bool rows, const WeightHints* weights, cudaStream_t stream) {
    const QuantBatch& p = b;
    const int grid_groups = b.groups_per_lin * b.n_lin;
    cudaLaunchConfig_t cfg = {};
    const int n_atoms = (p.K + kAtomK - 1) / kAtomK;
    int parts = 1, k_max = 0;
    for (int i = 0; i < b.n_lin; ++i) k_max = b.lay[i].k_tail > k_max ? b.lay[i].k_tail : k_max;
    if (scale_perm) {
        // split the rows of a group (a CTA has a fixed cost of about a microsecond, so no further than needed)
        int sms = 0;
        const cudaError_t e = current_sm_count(&sms);
        if (e != cudaSuccess) return e;
        const long long tiles = static_cast<long long>(n_atoms) * grid_groups;
        while (parts < 4 && tiles * parts < 8LL * sms) parts *= 2;   // 3 CTAs per SM: keep the last wave short
        if (parts == 4 && tiles * parts < 4LL * sms) parts = 8;
        if (const char* ev = dev_knobs_enabled() ? getenv("PRQ_QUANT_PARTS") : nullptr) { const int v = atoi(ev); if (v == 1 || v == 2 || v == 4 || v == 8) parts = v; }
        // The column-stationary structure, in the instance that measured best (microseconds in a chain of launches, K and
        // k as given; column atoms -> this structure):
        //   up to 128 rows of K <= 4096: one row per slice, CTAs of at most five computing warps (64 x 2560: 2.7 -> 2.0);
        //   large batches: four rows per slice amortise a slice's bookkeeping (4096 x 2560: 15.3 -> 8.9, four rows against
        //   two: 8.9 / 9.8; 4096 x 4096: 22.6 -> 11.0); beyond 8192 columns two rows, so that one CTA's registers hold the
        //   whole width (4096 x 9728: 46.7 -> 20.9, against 22.0 with the columns cut in two);
        //   in between two rows per slice (600 x 2560: 5.5 -> 3.6, 1000 x 6144: 11.5 -> 6.7, 16 x 9728: 2.9 -> 2.8);
        //   stacked experts: eight columns per lane, more warps for narrow rows (K = 768, 128 experts: 1024 tokens 19.5 -> 11.5,
        //   8192 tokens 62 -> 34).
        // ... and the column atoms where they are the better ones, judged with the product behind them (quantise + multiply,
        // column atoms / this structure):
        //   rows of which two do not fit twice (K > 25728; stacked experts, four rows, 12864).  With one row per slice a CTA has
        //   five warps for a whole row in shared memory, and every one of the 12 - 21 cuts of the columns brings all of it:
        //   K = 28672, 16 / 300 / 4096 rows 10.6 / 27 / 149 against 13.9 / 37 / 271; K = 51456 16 / 36 / 263 against 22 / 58 / 464;
        //   2 to 32 rows where the atoms alone have a CTA per SM (K = 22016, 8 / 32 rows: 8.6 / 9.5 against 9.4 / 10.7;
        //   K = 18432, below that line: 8.9 / 9.8 against 8.8 / 9.7);
        //   no tail, or one block of it, and 41 (65) to 128 rows of a narrow layer: there are no scattered reads to save (k = 0,
        //   64 / 128 rows: K = 2560 7.5 / 8.5 against 7.7 / 9.2, K = 6144 8.2 / 9.8 against 8.7 / 10.4; K = 8192 8.0 / 10.2 against 7.7 /
        //   9.8; k = 128, K = 2560: 9.2 / 10.0 against 7.7 / 9.2);
        //   stacked experts of one atom (128 experts of K = 128, 4096 / 65536 rows: 14.4 / 45 against 16.0 / 50); up to 64 atoms, where
        //   looking the experts up is all there is to it; up to 128 rows while the atoms' launch is small (2 experts of K = 3072,
        //   8 / 128 rows: 10.2 / 11.0 against 10.7 / 12.1, 32 of K = 256, 64 rows: 8.0 against 8.7; beyond those lines 8 of K = 2048:
        //   11.3 / 12.2 against 9.7 / 10.8, 16 of K = 640, 64 rows: 9.2 against 9.0); three atoms, which leave every second warp half
        //   idle, while the atoms' CTAs fit the GPU at once (64 experts of K = 384, 64 / 512 rows: 10.0 / 12.3 against 11.0 / 13.1).
        const bool grouped = b.expert_offsets != nullptr;
        auto fits = [&](int rows) { return 4 * static_cast<size_t>(rows) * p.K + 10240 <= kColsSmem - 9216; };
        bool cols;
        if (grouped) {
            const bool few = b.M <= 128 && tiles * parts <= (b.n_experts <= 4 ? 768 : 576);
            const bool three = n_atoms == 3 && b.M <= 1024 && parts == 4 && tiles <= 216;
            cols = n_atoms > 1 && tiles > 64 && !few && !three;
        } else {
            const bool wide_few = b.M > 1 && b.M <= 32 && tiles >= sms;
            const bool narrow_flat = b.M <= 128 && p.K <= 6144 && tiles >= 16 && tiles <= 80 &&
                                     ((k_max == 0 && b.M > 40) || (k_max <= kBlock && b.M > 64));
            cols = !wide_few && !narrow_flat;
        }
        if (const char* ev = dev_knobs_enabled() ? getenv("PRQ_QUANT_ROWS") : nullptr) cols = atoi(ev) != 0;
        if (cols && grouped && fits(4)) return launch_cols_impl<8, 4, true, 544>(b, sms, stream);
        if (cols && !grouped) {
            const bool large = b.M >= 1500 && p.K >= 2048;
            if (b.M <= 128 && p.K <= 4096)
                return weights ? launch_cols_impl<16, 1, false, 192, true>(b, sms, stream, weights) : launch_cols_impl<16, 1, false, 192>(b, sms, stream);
            if (large && p.K <= 8192) return launch_cols_impl<16, 4, false, 384>(b, sms, stream);
            if (large && fits(2)) return launch_cols_impl<16, 2, false, 640>(b, sms, stream);
            if (fits(2)) return weights ? launch_cols_impl<16, 2, false, 320, true>(b, sms, stream, weights) : launch_cols_impl<16, 2, false, 320>(b, sms, stream);
        }
    }
    // the tail atoms of the scale + permute mode in shares of 16 rows (128 / 8), see the kernel
    QuantBatch bb = b;
    bb.n_atoms = n_atoms;
    bb.n_tail = 0; bb.tail_split = 1;
    // (dense launches only: a grouped launch has a CTA per expert group and column atom already, each with the fixed
    // cost of finding its expert -- eight times as many tail CTAs made the 128-expert quantiser 35-50 % slower, and its
    // launches are long enough for a 20 us CTA not to be their end)
    if (scale_perm && b.expert_offsets == nullptr) {
        bb.n_tail = (k_max + kAtomK - 1) / kAtomK < n_atoms ? (k_max + kAtomK - 1) / kAtomK : n_atoms;
        bb.tail_split = 8 / parts;
    }
    cfg.gridDim = dim3(n_atoms - bb.n_tail + bb.n_tail * bb.tail_split, grid_groups, parts);
    cfg.blockDim = dim3(kQuantThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    auto launch = [&](auto batch) {
        constexpr bool kBatch = decltype(batch)::value;
        if (weights) {
            AskParam<kAskWeights> asked;
            static_cast<WeightHints&>(asked) = *weights;
            return scale_perm ? cudaLaunchKernelEx(&cfg, quant_act_kernel<true, kBatch, kAskWeights>, bb, asked)
                              : cudaLaunchKernelEx(&cfg, quant_act_kernel<false, kBatch, kAskWeights>, bb, asked);
        }
        if (scale_perm) return cudaLaunchKernelEx(&cfg, quant_act_kernel<true, kBatch, kAskNothing>, bb, AskParam<kAskNothing>{});
        return rows ? cudaLaunchKernelEx(&cfg, quant_act_kernel<false, kBatch, kAskRows>, bb, AskParam<kAskRows>{})
                    : cudaLaunchKernelEx(&cfg, quant_act_kernel<false, kBatch, kAskNothing>, bb, AskParam<kAskNothing>{});
    };
    return b.n_lin > 1 ? launch(std::true_type{}) : launch(std::false_type{});
}

cudaError_t launch_quant_act(const QuantParams& p, bool scale_perm, int grid_groups, bool rows, const WeightHints* weights, cudaStream_t stream) {
    QuantBatch b = {};
    b.x = p.x; b.expert_offsets = p.expert_offsets; b.M = p.M; b.ldx = p.ldx; b.K = p.K;
    b.n_experts = p.n_experts; b.act_groups = p.act_groups;
    b.n_lin = 1;
    b.groups_per_lin = grid_groups;
    b.lay[0] = QuantLayer{p.perm, p.inv_s_perm, p.codes, p.scales_row, p.scales_sf, p.k_tail};
    b.status = p.status;
    return launch_quant_act_batch(b, scale_perm, rows, weights, stream);
}

}  // namespace prq
