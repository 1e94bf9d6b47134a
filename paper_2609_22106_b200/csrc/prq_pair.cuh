// What the two CTA-pair kernels share (prefill of a dense layer, prq_gemm_prefill_pair.cu; stacked experts,
// prq_gemm_grouped_pair.cu): tile geometry, shared- and tensor-memory budgets, and the issue of one reduction stage.
#pragma once
#include <cstdint>

#include "prq_kernels.h"
#include "prq_ptx.cuh"

namespace prq {
namespace {

constexpr int kPTile = 128 * 128;                 // activation tile bytes (128 rows x 256 codes)
constexpr int kStages = 5;
constexpr int kStagingPerWarp = 2 * 4096;         // two 32-row x 128-byte chunks per epilogue warp
constexpr int kTmemCols = 512;
constexpr int kChunkCols = 32;                    // accumulator columns per epilogue chunk

// Everything that depends on the tile width BN (weight rows per tile): 224, 240 or 288.
//   224 / 240: two accumulators of BN columns and the scale columns must fit the 512 columns of tensor memory,
//   which 240 still does; the wider tile needs fewer operand bytes per multiply-add, its main loop runs within a
//   few percent of the tensor time, and it pads N = 2560 less (11 x 240 against 12 x 224).
//   288: ONE accumulator, for calls whose tiles all fit one wave of pairs at this width (the host decides): no
//   pair takes a second tile, so nothing needs a second accumulator, and no tile is split along K.  An MMA takes at
//   most 256 columns, so a reduction step is two instructions of 144 columns each (an MMA of 32 columns costs about as
//   much as one of 64: 256 + 32 measured 9 % slower than 144 + 144 predicts); each CTA loads 72 + 72 weight rows -- rows
//   [72 r, +72) and [144 + 72 r, +72) of the tile -- so that the accumulator's columns are the tile's weight rows in
//   order, and the scale bytes are tiled per 144-row half (two groups each).
// kFp8: the second format (MXFP8, one byte per element).  A stage is still one 128-byte swizzled row per operand row,
// which then holds 128 elements = four blocks = ONE 512-byte scale atom per 128-row group, and an MMA takes 32 of them.
template <int BN, bool kFp8 = false>
struct PCfg {
    static constexpr int kStageElems = kFp8 ? 128 : kStageK;
    static constexpr int kSfGroup = kFp8 ? 512 : kSfGroupBytes;   // scale bytes per (stage, 128-row group)
    static constexpr int kSfRows = kSfGroup / 256;                // rows of the scale tensor maps per group
    static constexpr int kSfp = kSfGroup;                         // one group of 128 activation rows
    static constexpr bool kWide = BN > 256;
    static constexpr int kHalfN = BN / 2;                    // weight rows each CTA of the pair loads
    static constexpr int kQTile = kHalfN * 128;              // half weight tile bytes
    static constexpr int kHalfGroups = kWide ? (BN / 2 + 127) / 128 : 0;                    // scale groups per 144-row half
    static constexpr int kSfqGroups = kWide ? 2 * kHalfGroups : (BN + 127) / 128;           // 128-row scale groups of a weight tile
    static constexpr int kSfq = kSfqGroups * kSfGroup;
    static constexpr int kTxBytes = kPTile + kQTile + kSfp + kSfq;     // 33792 / 34816 / 39936; MXFP8 32256 / 33280 / 37376
    static constexpr int kStageBytes = (kTxBytes + 1023) / 1024 * 1024;
    // the alternating staging buffers serve epilogues that run under a main loop; the one-wave tile has only a last
    // epilogue, which stages in the idle ring
    static constexpr int kStagingBytes = kWide ? 0 : 4 * kStagingPerWarp;
    static constexpr int kSmemBytes = kStages * kStageBytes + kStagingBytes + 1024;
    static constexpr int kAccBufs = kWide ? 1 : 2;
    static constexpr int kSfCol = kAccBufs * BN;             // scale columns start behind the accumulator(s)
    static constexpr int kSfCols = kFp8 ? 4 : 8;             // scale columns per group: 4 per atom
    static constexpr int kSfSetCols = kSfCols * (1 + kSfqGroups);
    static constexpr int kChunks = (BN + kChunkCols - 1) / kChunkCols;   // 7, 7 and a 16-column one, or 9
    static constexpr int kLastCols = BN - (kChunks - 1) * kChunkCols;    // 32 or 16
    static constexpr int kSlotUnits = kChunks * 8 * 128;     // float4 per workspace slot (128 rows)
    static_assert(kQTile % 1024 == 0 && kStageBytes % 1024 == 0, "operand tiles must keep 1024-byte alignment");
    static_assert(kSmemBytes <= 232448 - 256, "shared memory budget");
    static_assert(kSfCol + kSfSetCols <= kTmemCols, "tensor memory budget");
    static_assert(kLastCols == 32 || kLastCols == 16, "epilogue chunks are 32 columns, the last one 32 or 16");
    static_assert(kWide || static_cast<size_t>(kSlotUnits) * 16 <= kPrefillSlotBytes, "workspace slot");
};

__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void st_cluster_u32(uint32_t cluster_addr, uint32_t v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}

constexpr uint32_t kHiSw128 = (1024u >> 4) | (1u << 14) | (2u << 29);  // SBO 1024, version 1, 128B swizzle
constexpr uint32_t kHiPlain = (128u >> 4) | (1u << 14);                // SBO 128, version 1, no swizzle
__device__ __forceinline__ uint64_t desc64(uint32_t hi, uint32_t lo) { return (static_cast<uint64_t>(hi) << 32) | lo; }

// One reduction stage of the issue loop with the ring slot Q known at compile time: every
// shared-memory descriptor is `lo_base` plus a constant.  Scale atoms first, then up to four steps, then the commit that
// frees the slot in both CTAs.  A step is one MMA over all BN columns, or for the 288-column tile two of 144 columns (the
// second reads the second half of the CTA's weight rows and the scale columns of the second half's groups).  The copies and
// the MMAs are issued by one thread, so tensor memory sees them in order and one set of scale columns is enough.
// MXFP4: K = 64 steps, two atoms per 128-row group and stage: the activation's in scale columns +0 / +4 (first / second half of
// the stage), the weight groups' (G = 2 of them, 288 columns: 4) in +8 + 4 g / +8 + 4 G + 4 g; a step's scale id picks the byte
// pair.  MXFP8: K = 32 steps, one atom per group: activation +0, weights +4 + 4 g; step j takes byte j.  `rem` = reduction
// elements this stage still covers.
template <int BN, bool kFp8, int Q>
__device__ __forceinline__ void issue_stage(uint32_t lo_base, uint32_t d_tmem, uint32_t sf_t, int rem,
                                            uint32_t accumulate, uint32_t empty_bar0) {
    using C = PCfg<BN, kFp8>;
    constexpr int kStageBytes = C::kStageBytes, kQTile = C::kQTile, G = C::kSfqGroups;
    constexpr uint32_t so = (Q * kStageBytes) >> 4;  // stage offset in 16-byte units
    constexpr uint32_t sfo = so + ((kPTile + kQTile) >> 4);
    // E2M1 x E2M1, E8M0 scales, both operands K-major, N = N1 (and N2), M = 256 (two CTAs)
    constexpr int N1 = C::kWide ? BN / 2 : BN, N2 = BN - N1;
    constexpr uint32_t idesc0 = (1u << 7) | (1u << 10) | ((N1 >> 3) << 17) | (1u << 23) | ((256u >> 4) << 24);
    constexpr uint32_t idesc2 = idesc0 | (2u << 4) | (2u << 29);
    constexpr uint32_t jdesc0 = (1u << 7) | (1u << 10) | (((N2 > 0 ? N2 : 16) >> 3) << 17) | (1u << 23) | ((256u >> 4) << 24);
    constexpr uint32_t jdesc2 = jdesc0 | (2u << 4) | (2u << 29);
    const uint32_t plo = lo_base + so, qlo = lo_base + so + (kPTile >> 4), slo = lo_base + sfo;
    constexpr int kSfp = C::kSfp;
    const uint32_t sfp_t = sf_t, sfq_t = sf_t + C::kSfCols;
    // the second instruction of a step reads the CTA's weight rows from row N1 / 2 on and the scale columns of
    // the second half's groups
    constexpr uint32_t q2 = ((N1 / 2) * 128) >> 4, s2 = 4 * C::kHalfGroups;
    if constexpr (kFp8) {
        // E4M3 x E4M3 (format 0); step j takes byte j of the scale words
        constexpr uint32_t id = ((N1 >> 3) << 17) | (1u << 23) | ((256u >> 4) << 24);
        constexpr uint32_t jd = (((N2 > 0 ? N2 : 16) >> 3) << 17) | (1u << 23) | ((256u >> 4) << 24);
        tc_copy_sf_atom_pair(sfp_t, desc64(kHiPlain, slo));
#pragma unroll
        for (int g = 0; g < G; ++g) tc_copy_sf_atom_pair(sfq_t + 4 * g, desc64(kHiPlain, slo + ((kSfp + g * C::kSfGroup) >> 4)));
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (rem > 32 * j) {
                const uint32_t sid = (static_cast<uint32_t>(j) << 4) | (static_cast<uint32_t>(j) << 29), acc = j ? 1u : accumulate;
                tc_mma_mxf8_pair(d_tmem, desc64(kHiSw128, plo + 2 * j), desc64(kHiSw128, qlo + 2 * j), id | sid, sfp_t, sfq_t, acc);
                if (N2 > 0) tc_mma_mxf8_pair(d_tmem + N1, desc64(kHiSw128, plo + 2 * j), desc64(kHiSw128, qlo + q2 + 2 * j), jd | sid, sfp_t, sfq_t + s2, acc);
            }
        }
        tc_commit_pair(empty_bar0 + Q * 8, 3);
        return;
    }
    tc_copy_sf_atom_pair(sf_t, desc64(kHiPlain, slo));
#pragma unroll
    for (int g = 0; g < G; ++g)
        tc_copy_sf_atom_pair(sfq_t + 4 * g, desc64(kHiPlain, slo + ((kSfp + g * kSfGroupBytes) >> 4)));
    if (rem > 128) {
        tc_copy_sf_atom_pair(sf_t + 4, desc64(kHiPlain, slo + (512 >> 4)));
#pragma unroll
        for (int g = 0; g < G; ++g)
            tc_copy_sf_atom_pair(sfq_t + 4 * G + 4 * g, desc64(kHiPlain, slo + ((kSfp + g * kSfGroupBytes + 512) >> 4)));
    }
    tc_mma_mxf4_pair(d_tmem, desc64(kHiSw128, plo), desc64(kHiSw128, qlo), idesc0, sfp_t, sfq_t, accumulate);
    if (N2 > 0) tc_mma_mxf4_pair(d_tmem + N1, desc64(kHiSw128, plo), desc64(kHiSw128, qlo + q2), jdesc0, sfp_t, sfq_t + s2, accumulate);
    if (rem > 64) {
        tc_mma_mxf4_pair(d_tmem, desc64(kHiSw128, plo + 2), desc64(kHiSw128, qlo + 2), idesc2, sfp_t, sfq_t, 1);
        if (N2 > 0) tc_mma_mxf4_pair(d_tmem + N1, desc64(kHiSw128, plo + 2), desc64(kHiSw128, qlo + q2 + 2), jdesc2, sfp_t, sfq_t + s2, 1);
    }
    if (rem > 128) {
        tc_mma_mxf4_pair(d_tmem, desc64(kHiSw128, plo + 4), desc64(kHiSw128, qlo + 4), idesc0, sfp_t + 4, sfq_t + 4 * G, 1);
        if (N2 > 0) tc_mma_mxf4_pair(d_tmem + N1, desc64(kHiSw128, plo + 4), desc64(kHiSw128, qlo + q2 + 4), jdesc0, sfp_t + 4, sfq_t + 4 * G + s2, 1);
    }
    if (rem > 192) {
        tc_mma_mxf4_pair(d_tmem, desc64(kHiSw128, plo + 6), desc64(kHiSw128, qlo + 6), idesc2, sfp_t + 4, sfq_t + 4 * G, 1);
        if (N2 > 0) tc_mma_mxf4_pair(d_tmem + N1, desc64(kHiSw128, plo + 6), desc64(kHiSw128, qlo + q2 + 6), jdesc2, sfp_t + 4, sfq_t + 4 * G + s2, 1);
    }
    tc_commit_pair(empty_bar0 + Q * 8, 3);
}

}  // namespace
}  // namespace prq
