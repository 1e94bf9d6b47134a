// Offline weight preparation (Algorithm 1 steps 3-7 and 11) with the heavy steps on the GPU.
//
// The result is bit-for-bit the one of the host path (prq_prep.cu): same scale rule, same rounding, same
// FP64 summation order.  What runs where:
//   host    s_j = max(amax_j, 1e-5)^alpha and 1 / s_j                        (K values, FP64)
//   kernel  err_j = sum_n (W0[n,j] - deq(Q(W0))[n,j])^2, W0 = fl32(W * s)    col_err_kernel
//   host    error-ranked top-k, permutation                                  (a selection among K numbers)
//   kernel  Wt = W0[:, perm], Q(Wt), R = Wt_tail - deq(Q(Wt))_tail, Q(R), packing, optionally with the block-scale
//           search (floor-rule exponent and its two neighbours, FP64 squared error in element order)   quant_perm_kernel
//   kernel  the row-major scale bytes in every layout the GEMMs read         sf_layout_kernel
// W is read from device memory twice (50 MB at the paper's down-projection shape, 15 us at the measured copy rate);
// codes and scale bytes are produced where the GEMMs read them and never visit the host.
#include <cuda_runtime.h>

#include <cstdint>

#include "prq_internal.h"
#include "prq_quant_block.cuh"

namespace prq {
namespace {

__device__ __forceinline__ float bf16_to_float(uint32_t h) { return __uint_as_float(h << 16); }

// E8M0 byte from the bit pattern of the block's largest magnitude: biased exponent - 2, floored at 0
__device__ __forceinline__ uint32_t scale_byte(uint32_t amax_bits) {
    const int e = static_cast<int>((amax_bits >> 23) & 0xff) - 2;
    return e < 0 ? 0u : static_cast<uint32_t>(e);
}
__device__ __forceinline__ float code_scale(uint32_t byte) { return __uint_as_float((254u - byte) << 23); }                    // 2^(127 - byte)
__device__ __forceinline__ float value_scale(uint32_t byte) { return __uint_as_float(byte == 0 ? 0x00400000u : byte << 23); }  // 2^(byte - 127)

// Two values already multiplied by 2^(127 - byte), rounded to the nearest E2M1 (ties to the even code, saturating).
// The conversions are exact both ways, so times 2^(byte - 127) this is the dequantised value (at most two significant
// bits times a power of two: exact in fp32, subnormal results included).
__device__ __forceinline__ void round_e2m1x2(float a0, float a1, float& q0, float& q1) {
    uint32_t h;
    asm("{\n\t.reg .b8 t;\n\tcvt.rn.satfinite.e2m1x2.f32 t, %2, %1;\n\tcvt.rn.f16x2.e2m1x2 %0, t;\n\t}" : "=r"(h) : "f"(a0), "f"(a1));
    asm("{\n\t.reg .b16 l, u;\n\tmov.b32 {l, u}, %2;\n\tcvt.f32.f16 %0, l;\n\tcvt.f32.f16 %1, u;\n\t}" : "=f"(q0), "=f"(q1) : "r"(h));
}

// ---------------------------------------------------------------------------------------------- column errors
// The FP64 sum of a column runs over the rows in ascending order (its bits depend on that), so a column's sum is a
// serial chain of N additions: 2560 rows cannot take less than 2560 FP64 latencies, whatever the rest does.  A CTA takes
// one 32-channel block of the original order: eight warps quantise 128 rows at a time and leave the differences in
// shared memory (exact in fp32: a value and its own rounding lie within a factor of two, or the rounding is zero or
// saturates), a ninth warp -- lane = channel -- squares and adds the 128 rows before.  One warp that did everything itself
// paid the whole quantisation on that chain: 580 us at 2560 x 9728 against 38 now, 2180 against 93 at 9728 x 2560.
constexpr int kErrWarps = 8, kErrChunk = 128;

template <bool kAligned>   // kAligned: W on 8 bytes
__global__ void __launch_bounds__(32 * (kErrWarps + 1)) col_err_kernel(const uint16_t* __restrict__ W, const float* __restrict__ s, int N, int K,
                                                                      double* __restrict__ err, int* __restrict__ nonfinite) {
    __shared__ __align__(16) float diff[2][kErrChunk][kBlock];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int expert = blockIdx.y, j0 = static_cast<int>(blockIdx.x) * kBlock;
    W += static_cast<size_t>(expert) * N * K + j0;
    s += static_cast<size_t>(expert) * K + j0;
    const int n_chunks = (N + kErrChunk - 1) / kErrChunk;
    if (warp < kErrWarps) {
        // a lane holds four channels of one row, a warp four rows per step, four steps per chunk; the next chunk's
        // loads are issued before this chunk is worked on
        constexpr int kSteps = kErrChunk / (4 * kErrWarps);
        const int c4 = (lane & 7) * 4, r4 = warp * 4 + (lane >> 3);
        const float4 sj = *reinterpret_cast<const float4*>(s + c4);
        bool ok = true;
        uint2 h[kSteps];
        auto load = [&](int chunk) {
#pragma unroll
            for (int i = 0; i < kSteps; ++i) {
                const int n = chunk * kErrChunk + i * 4 * kErrWarps + r4;
                h[i] = make_uint2(0, 0);
                if (n < N) {
                    const uint16_t* p = W + static_cast<size_t>(n) * K + c4;
                    if (kAligned) h[i] = __ldg(reinterpret_cast<const uint2*>(p));
                    else h[i] = make_uint2(__ldg(p) | static_cast<uint32_t>(__ldg(p + 1)) << 16, __ldg(p + 2) | static_cast<uint32_t>(__ldg(p + 3)) << 16);
                }
            }
        };
        load(0);
        for (int c = 0; c < n_chunks; ++c) {
            uint2 w[kSteps];
#pragma unroll
            for (int i = 0; i < kSteps; ++i) w[i] = h[i];
            if (c + 1 < n_chunks) load(c + 1);
#pragma unroll
            for (int i = 0; i < kSteps; ++i) {
                const float v0 = __fmul_rn(__uint_as_float(w[i].x << 16), sj.x), v1 = __fmul_rn(__uint_as_float(w[i].x & 0xffff0000u), sj.y);
                const float v2 = __fmul_rn(__uint_as_float(w[i].y << 16), sj.z), v3 = __fmul_rn(__uint_as_float(w[i].y & 0xffff0000u), sj.w);
                const uint32_t m0 = __float_as_uint(v0) & 0x7fffffffu, m1 = __float_as_uint(v1) & 0x7fffffffu;
                const uint32_t m2 = __float_as_uint(v2) & 0x7fffffffu, m3 = __float_as_uint(v3) & 0x7fffffffu;
                uint32_t m = max(max(m0, m1), max(m2, m3));
                ok = ok && m < 0x7f800000u;
#pragma unroll
                for (int d = 1; d < 8; d <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, d));
                const uint32_t byte = scale_byte(m);
                const float up = code_scale(byte), down = value_scale(byte);
                float q0, q1, q2, q3;
                round_e2m1x2(__fmul_rn(v0, up), __fmul_rn(v1, up), q0, q1);
                round_e2m1x2(__fmul_rn(v2, up), __fmul_rn(v3, up), q2, q3);
                *reinterpret_cast<float4*>(&diff[c & 1][i * 4 * kErrWarps + r4][c4]) =
                    make_float4(__fsub_rn(v0, __fmul_rn(q0, down)), __fsub_rn(v1, __fmul_rn(q1, down)),
                                __fsub_rn(v2, __fmul_rn(q2, down)), __fsub_rn(v3, __fmul_rn(q3, down)));
            }
            __syncthreads();   // this chunk is there; the ninth warp is through with the buffer that comes next
        }
        if (!ok) atomicExch(nonfinite, 1);
    } else {
        double acc = 0.0;
        for (int c = 0; c < n_chunks; ++c) {
            __syncthreads();
            const int rows = min(kErrChunk, N - c * kErrChunk);
            const float(*d)[kBlock] = diff[c & 1];
            int r = 0;
            for (; r + 16 <= rows; r += 16) {
                double dd[16];
#pragma unroll
                for (int u = 0; u < 16; ++u) { const double x = static_cast<double>(d[r + u][lane]); dd[u] = __dmul_rn(x, x); }
#pragma unroll
                for (int u = 0; u < 16; ++u) acc = __dadd_rn(acc, dd[u]);
            }
            for (; r < rows; ++r) { const double x = static_cast<double>(d[r][lane]); acc = __dadd_rn(acc, __dmul_rn(x, x)); }
        }
        err[static_cast<size_t>(expert) * K + j0 + lane] = acc;
    }
}

// ---------------------------------------------------------------------------------------------- quantise + pack
// codes of a block under `byte`, packed with element i in nibble i % 8 of word i / 8
__device__ __forceinline__ uint4 block_codes(const float (&v)[kBlock], uint32_t byte) {
    const float up = code_scale(byte);
    uint32_t c[4];
#pragma unroll
    for (int w = 0; w < 4; ++w)
        c[w] = cvt_e2m1x8(__fmul_rn(v[8 * w], up), __fmul_rn(v[8 * w + 1], up), __fmul_rn(v[8 * w + 2], up), __fmul_rn(v[8 * w + 3], up),
                          __fmul_rn(v[8 * w + 4], up), __fmul_rn(v[8 * w + 5], up), __fmul_rn(v[8 * w + 6], up), __fmul_rn(v[8 * w + 7], up));
    return make_uint4(c[0], c[1], c[2], c[3]);
}
// squared error of the block under `byte`, FP64, element order (the differences are exact in fp32 under the floor-rule
// exponent and its neighbours: at most 24 bits between the value's last place and three binades above the scale)
__device__ __forceinline__ double block_error(const float (&v)[kBlock], uint32_t byte) {
    const float up = code_scale(byte), down = value_scale(byte);
    double err = 0.0;
#pragma unroll
    for (int i = 0; i < kBlock; i += 2) {
        float q0, q1;
        round_e2m1x2(__fmul_rn(v[i], up), __fmul_rn(v[i + 1], up), q0, q1);
        const double d0 = static_cast<double>(v[i]) - static_cast<double>(__fmul_rn(q0, down));
        const double d1 = static_cast<double>(v[i + 1]) - static_cast<double>(__fmul_rn(q1, down));
        err = __dadd_rn(err, __dmul_rn(d0, d0));
        err = __dadd_rn(err, __dmul_rn(d1, d1));
    }
    return err;
}
// Floor-rule byte, or with `search` the best of it and its two neighbours: a neighbour wins only if strictly better,
// byte - 1 is looked at before byte + 1, and an all-zero block keeps the floor rule.
template <bool kSearch>
__device__ __forceinline__ uint32_t choose_byte(const float (&v)[kBlock]) {
    uint32_t amax = 0;
#pragma unroll
    for (int i = 0; i < kBlock; ++i) amax = max(amax, __float_as_uint(v[i]) & 0x7fffffffu);
    const uint32_t byte0 = scale_byte(amax);
    if (!kSearch || amax == 0) return byte0;
    double best_err = block_error(v, byte0);
    uint32_t best = byte0;
#pragma unroll 1
    for (int c = -1; c <= 1; c += 2) {
        const int cand = static_cast<int>(byte0) + c;
        if (cand < 0 || cand > 254) continue;
        const double e = block_error(v, static_cast<uint32_t>(cand));
        if (e < best_err) { best_err = e; best = static_cast<uint32_t>(cand); }
    }
    return best;
}

// One thread per 32-channel block of the permuted order; it keeps its block's source positions and scales in registers
// while rows pass by in shared memory (two buffers, the next row on its way).  The lanes of a warp read 16 words apart,
// so a row is stored with word w at w ^ ((w >> 4) & 15): two lanes share a bank instead of sixteen.  Gathering the 2-byte
// weights from global memory instead took 205 us at 2560 x 9728; this takes 38 (119 with the search).
// kStage: 2 = rows copied asynchronously in 4-byte words (W on 4 bytes), 1 = copied by 2-byte loads, 0 = rows too wide
// for shared memory, gathered from global memory.
constexpr int kPermThreads = 320;
__device__ __forceinline__ uint32_t swizzled(uint32_t word) { return word ^ ((word >> 4) & 15u); }

template <bool kSearch, int kStage>
__global__ void __launch_bounds__(kPermThreads) quant_perm_kernel(const uint16_t* __restrict__ W, const float* __restrict__ s,
                                                                  const int32_t* __restrict__ perm, int N, int K, int k_tail,
                                                                  uint8_t* __restrict__ codes, uint8_t* __restrict__ scales) {
    extern __shared__ __align__(16) uint8_t perm_smem[];
    const int nblk = K / kBlock, expert = blockIdx.z;
    const int b = static_cast<int>(blockIdx.y) * blockDim.x + threadIdx.x;
    const bool live = b < nblk;
    const size_t Ka = static_cast<size_t>(K) + k_tail;
    W += static_cast<size_t>(expert) * N * K;
    s += static_cast<size_t>(expert) * K;
    perm += static_cast<size_t>(expert) * K;
    codes += static_cast<size_t>(expert) * N * (Ka / 2);
    scales += static_cast<size_t>(expert) * N * (Ka / kBlock);
    uint32_t src[kBlock];   // byte position of element i in a (staged) row
    float sc[kBlock];
#pragma unroll
    for (int i = 0; i < kBlock; ++i) {
        const uint32_t j = live ? static_cast<uint32_t>(__ldg(perm + b * kBlock + i)) : 0u;
        sc[i] = live ? __ldg(s + j) : 0.f;
        src[i] = kStage ? swizzled(j >> 1) * 4 + (j & 1) * 2 : j * 2;
    }
    const uint32_t row_bytes = static_cast<uint32_t>(K) * 2;
    auto stage = [&](int n, int buf) {
        if (kStage == 2) {
            const uint32_t* p = reinterpret_cast<const uint32_t*>(W + static_cast<size_t>(n) * K);
            const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(perm_smem)) + buf * row_bytes;
            for (int w = threadIdx.x; w < K / 2; w += blockDim.x)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(base + swizzled(w) * 4), "l"(p + w) : "memory");
            asm volatile("cp.async.commit_group;" ::: "memory");
        } else if (kStage == 1) {
            const uint16_t* p = W + static_cast<size_t>(n) * K;
            for (int j = threadIdx.x; j < K; j += blockDim.x)
                *reinterpret_cast<uint16_t*>(perm_smem + buf * row_bytes + swizzled(j >> 1) * 4 + (j & 1) * 2) = __ldg(p + j);
        }
    };
    const int tail_blk0 = (K - k_tail) / kBlock;
    int n = blockIdx.x;
    if (n < N) stage(n, 0);
    for (int it = 0; n < N; ++it, n += gridDim.x) {
        if (kStage == 2) asm volatile("cp.async.wait_all;" ::: "memory");
        if (kStage) __syncthreads();   // this row is there; everybody is through with the other buffer
        if (n + static_cast<int>(gridDim.x) < N) stage(n + gridDim.x, (it + 1) & 1);
        if (!live) continue;
        const uint8_t* row = kStage ? perm_smem + (it & 1) * row_bytes : reinterpret_cast<const uint8_t*>(W + static_cast<size_t>(n) * K);
        float v[kBlock];
#pragma unroll
        for (int i = 0; i < kBlock; ++i) v[i] = __fmul_rn(bf16_to_float(*reinterpret_cast<const uint16_t*>(row + src[i])), sc[i]);
        const uint32_t byte = choose_byte<kSearch>(v);
        uint8_t* crow = codes + static_cast<size_t>(n) * (Ka / 2);
        uint8_t* srow = scales + static_cast<size_t>(n) * (Ka / kBlock);
        *reinterpret_cast<uint4*>(crow + static_cast<size_t>(b) * 16) = block_codes(v, byte);
        srow[b] = static_cast<uint8_t>(byte);
        if (b >= tail_blk0) {
            // Eq. (2): residual of the tail block against its own quantisation (exact in fp32), quantised again
            const float up = code_scale(byte), down = value_scale(byte);
#pragma unroll
            for (int i = 0; i < kBlock; i += 2) {
                float q0, q1;
                round_e2m1x2(__fmul_rn(v[i], up), __fmul_rn(v[i + 1], up), q0, q1);
                v[i] = __fsub_rn(v[i], __fmul_rn(q0, down));
                v[i + 1] = __fsub_rn(v[i + 1], __fmul_rn(q1, down));
            }
            const uint32_t rbyte = choose_byte<kSearch>(v);
            const int rb = nblk + (b - tail_blk0);
            *reinterpret_cast<uint4*>(crow + static_cast<size_t>(rb) * 16) = block_codes(v, rbyte);
            srow[rb] = static_cast<uint8_t>(rbyte);
        }
    }
}

// ---------------------------------------------------------------------------------------------- scale-byte layouts
// Every layout is [expert][stage][128-row group][1024 bytes] (second format: 512, four blocks per stage); a weight tile of
// `tile_rows` rows has `groups_per_tile` groups of its own, the last one partly empty.  One thread per word: the four blocks of one (row, atom).  Words that
// hold no row or block are zero bytes (2^-127, finite).
__global__ void __launch_bounds__(256) sf_layout_kernel(const uint8_t* __restrict__ scales, int N, int K, int k_tail, SfLayouts t) {
    const SfLayout l = t.l[blockIdx.y];
    const int nb = t.group_bytes / 128;   // blocks per stage: 8 or 4
    const int nblk = K / kBlock, n_all = nblk + k_tail / kBlock;
    const int S1 = (nblk + nb - 1) / nb, S = S1 + (k_tail / kBlock + nb - 1) / nb;
    for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < l.bytes / 4; i += static_cast<size_t>(gridDim.x) * blockDim.x) {
        const int off = static_cast<int>(i % (t.group_bytes / 4)) * 4;
        size_t g = i / (t.group_bytes / 4);
        uint32_t w = 0;
        const int group = static_cast<int>(g % l.groups);
        g /= l.groups;
        const int stage = static_cast<int>(g % S);
        const size_t expert = g / S;
        const int in_tile = (group % l.groups_per_tile) * kGroupRows + (off & 12) * 8 + ((off & 511) >> 4);
        const int n = group / l.groups_per_tile * l.tile_rows + in_tile;
        if (expert < static_cast<size_t>(t.n_experts) && in_tile < l.tile_rows && n < N) {
            const int bis = (off >> 9) * 4;
            const int b = stage < S1 ? stage * nb + bis : nblk + (stage - S1) * nb + bis;
            const int end = stage < S1 ? nblk : n_all;
            const uint8_t* p = scales + (expert * N + n) * n_all + b;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (b + j < end) w |= static_cast<uint32_t>(__ldg(p + j)) << (8 * j);
        }
        reinterpret_cast<uint32_t*>(l.dst)[i] = w;
    }
}

template <bool kSearch, int kStage>
cudaError_t launch_quant_perm_impl(const uint16_t* W, const float* s, const int32_t* perm, int E, int N, int K, int k_tail,
                                   uint8_t* codes, uint8_t* scales, int sm_count, cudaStream_t stream) {
    const size_t smem = kStage ? 4 * static_cast<size_t>(K) : 0;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(quant_perm_kernel<kSearch, kStage>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (e != cudaSuccess) return e;
    }
    const int nblk = K / kBlock, chunks = (nblk + kPermThreads - 1) / kPermThreads;
    const int threads = ((nblk + chunks - 1) / chunks + 31) / 32 * 32;
    // as many CTAs as stay resident with at most 168 registers a thread; a CTA's constants are worth a few rows
    int per_sm = 65536 / (168 * threads);
    if (smem) per_sm = per_sm < static_cast<int>(200 * 1024 / (smem + 1024)) ? per_sm : static_cast<int>(200 * 1024 / (smem + 1024));
    per_sm = per_sm < 1 ? 1 : per_sm > 16 ? 16 : per_sm;
    long long gx = static_cast<long long>(per_sm) * sm_count / (static_cast<long long>(chunks) * E);
    gx = gx < 1 ? 1 : gx > N ? N : gx;
    quant_perm_kernel<kSearch, kStage><<<dim3(static_cast<unsigned>(gx), chunks, E), threads, smem, stream>>>(W, s, perm, N, K, k_tail, codes, scales);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_col_err(const uint16_t* W, const float* s, int E, int N, int K, double* err, int* nonfinite, cudaStream_t stream) {
    const dim3 grid(K / kBlock, E);
    if (reinterpret_cast<uintptr_t>(W) % 8 == 0) col_err_kernel<true><<<grid, 32 * (kErrWarps + 1), 0, stream>>>(W, s, N, K, err, nonfinite);
    else col_err_kernel<false><<<grid, 32 * (kErrWarps + 1), 0, stream>>>(W, s, N, K, err, nonfinite);
    return cudaGetLastError();
}

cudaError_t launch_quant_perm(const uint16_t* W, const float* s, const int32_t* perm, int E, int N, int K, int k_tail, bool search,
                              uint8_t* codes, uint8_t* scales, int sm_count, cudaStream_t stream) {
    const int stage = K > 49152 ? 0 : reinterpret_cast<uintptr_t>(W) % 4 ? 1 : 2;
    if (search)
        return stage == 2 ? launch_quant_perm_impl<true, 2>(W, s, perm, E, N, K, k_tail, codes, scales, sm_count, stream)
               : stage == 1 ? launch_quant_perm_impl<true, 1>(W, s, perm, E, N, K, k_tail, codes, scales, sm_count, stream)
                            : launch_quant_perm_impl<true, 0>(W, s, perm, E, N, K, k_tail, codes, scales, sm_count, stream);
    return stage == 2 ? launch_quant_perm_impl<false, 2>(W, s, perm, E, N, K, k_tail, codes, scales, sm_count, stream)
           : stage == 1 ? launch_quant_perm_impl<false, 1>(W, s, perm, E, N, K, k_tail, codes, scales, sm_count, stream)
                        : launch_quant_perm_impl<false, 0>(W, s, perm, E, N, K, k_tail, codes, scales, sm_count, stream);
}

cudaError_t launch_sf_layout(const uint8_t* scales, int N, int K, int k_tail, const SfLayouts& t, int sm_count, cudaStream_t stream) {
    size_t most = 0;
    for (int i = 0; i < t.n; ++i) most = t.l[i].bytes > most ? t.l[i].bytes : most;
    const size_t blocks = (most / 4 + 255) / 256, cap = static_cast<size_t>(sm_count) * 8;
    sf_layout_kernel<<<dim3(static_cast<unsigned>(blocks < cap ? blocks : cap), t.n), 256, 0, stream>>>(scales, N, K, k_tail, t);
    return cudaGetLastError();
}

}  // namespace prq
