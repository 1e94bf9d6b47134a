// Decode GEMM (M <= 128 tokens): the block-scaled FP4 product of Eq. (3) as a weight-streaming kernel.
//
// With few tokens the layer is bound by reading its 4-bit weights once.  The weight rows sit on the MMA
// M axis (128-row tiles), the tokens on the N axis (16, 32, 64 or 128 columns), and the reduction axis
// K + k is split over the CTAs of a thread-block cluster so that every SM streams a share of the
// weights.  Each CTA of a cluster accumulates its K-range in tensor memory and then pushes, through
// distributed shared memory, the partial sums of token t into a receive buffer of the CTA that owns
// token t (t mod cluster size); the owner adds up what it received and writes its tokens to y.  The pushes are asynchronous
// stores whose bytes are counted on an mbarrier of the owner, which therefore waits for exactly its own tokens (the 32 KB
// of a 64-token tile among seven CTAs: 1500 cycles, with plain stores and a cluster barrier 2800; one bulk copy per
// owner 2170).  Two CTAs with more than 64 tokens park their sums instead and copy the other one's half with plain stores, whole
// rows at a time, and a cluster barrier (256 x 256 at 80 / 128 tokens: asynchronous 4.14 / 5.36 us, parked 3.90 / 4.94, 6144 x 2560
// 7.01 / 8.06 and 6.76 / 7.59; with three CTAs the asynchronous stores are ahead, 2304 x 2304 at 128 tokens 6.04 against 6.30).
// No global scratch, no atomics, and the summation order is fixed (peer 0, 1, ...), so
// the result is reproducible.  For up to 32 tokens two CTAs fit on an SM, so that the
// CTAs of the next kernel of the stream (the next layer's GEMM) are resident and streaming their weights
// while this one finishes.
//
// Roles per CTA (6 warps, 10 from 64 tokens on): warp 0 TMA producer, warp 1 tcgen05 issuer (scale copies + MMAs), warps 2-5 (2-9)
// epilogue and reduction.  The activation tail is re-read: stages past the K main columns load the
// token tile from column K - k and the weight tile from column K onwards (Kernel design paragraph).
// Every wait is bounded; the cluster barriers sit on the common path so that a CTA that gave up still
// arrives and its peers are released, and a CTA that gave up under the asynchronous exchange stays until its
// peers' deliveries into its receive buffer have landed.
// The kernel is latency-bound, not bandwidth-bound (with the weights resident in L2 it is only 0.5-1 us faster): what a
// launch costs is the chain token copies -> five stages of tcgen05 issue -> accumulator read -> exchange -> store behind
// its dependency, plus the hand-over to the next kernel.  Everything in it runs once per launch, so what counts is the
// number of instructions and waits between the dependency and the last store.  What that gave (N = 2560, K = 9728, k = 256,
// us a launch in a chain, before -> now): one token in one launch 4.53 -> 3.88 (N = 1024, K = 2560: 2.84 -> 2.40), quantise +
// multiply 16 / 64 / 128 tokens 7.73 / 9.45 / 11.70 -> 7.13 / 9.21 / 11.33 (6.4 / 8.5 / 10.7 where the quantiser asks for the weights):
//   * weight scales copied to tensor memory before the tokens are there; no wait, branch or commit between the stages of
//     the first ring pass (393 -> 190 cycles per stage);
//   * a few tokens' stages quantised side by side;
//   * partial sums sent from registers (a 4 x 4 transpose by shuffles) instead of through a parked tile, no divisions.
// Rehearsing the code on no data while the CTA waits for its dependency (to have the instructions at hand) made every launch
// slower (4.55 -> 5.25 with the code of the time): it runs beside the launch before.
//
// Fused variant (up to 16 tokens, activation already scaled and reordered by its producer): the kernel
// takes the bf16 activation itself.  The four epilogue warps first act as the activation quantiser of
// their CTA -- one 32-element block per thread and stage, codes written straight into the 128-byte-
// swizzled token tile of the pipeline slot, scale bytes into the slot's scale atom -- so that the
// separate quantiser launch, its round trip through global memory and one kernel-to-kernel hand-over
// leave the decode step (the Kernel design paragraph asks for one quantisation of the reordered activation
// per layer call; here it happens inside the product kernel).
// Every cluster quantises the K-range it reduces over, i.e. the bf16 activation is read once per 128-row
// weight tile; that extra L2 traffic grows with the token count and is why the variant stops at 16 tokens.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstring>

#include "prq_kernels.h"
#include "prq_ptx.cuh"
#include "prq_quant_block.cuh"

namespace prq {
namespace {

constexpr int kPTile = 128 * 128;   // weight tile bytes: 128 rows x 256 codes
constexpr int kSf = kSfGroupBytes;  // one 128-row scale group per operand and stage

constexpr uint32_t kHiSw128 = (1024u >> 4) | (1u << 14) | (2u << 29);
constexpr uint32_t kHiPlain = (128u >> 4) | (1u << 14);
__device__ __forceinline__ uint64_t desc64(uint32_t hi, uint32_t lo) { return (static_cast<uint64_t>(hi) << 32) | lo; }
constexpr int pow2_cols(int x) { int p = 32; while (p < x) p *= 2; return p; }

// kDense: the variant for layers with more 128-row weight tiles than the GPU has SMs (from 64 tokens on one
// CTA fills an SM, so tile 149 would wait for a second wave that leaves most SMs idle).  Such a layer is not
// K-split, so its CTAs need no receive buffer; with a 3-slot ring two of them share an SM and all tiles are
// resident at once (stacked gate / up projection, 152 tiles: 16.2 -> 12.1 us at 64 tokens, 20.0 -> 14.1 at 128).
template <int BN, bool kDense = false>
struct DCfg {
    static_assert(!kDense || BN >= 64, "up to 32 tokens two CTAs share an SM anyway");
    static constexpr int kQTile = BN * 128;
    // a ring slot: weight tile, token tile, weight scales; the token scales of all slots lie behind the ring, in stage order
    // (as in global memory, so that one copy brings those of a whole ring pass)
    static constexpr int kStageBytes = kPTile + kQTile + kSf;
    // ring depth: 5 / 4 stages leave room for two CTAs per SM at 16 / 32 tokens
    static constexpr int kStages = kDense ? 3 : BN == 16 ? 5 : BN == 32 ? 4 : BN == 64 ? 6 : 4;
    static constexpr int kCtasPerSm = (kDense || BN <= 32) ? 2 : 1;
    // epilogue warps: four (one per tensor-memory lane quarter); eight from 64 tokens on, where moving the
    // partial sums is most of the kernel -- two warps per quarter then take alternate 16-token chunks
    static constexpr int kEpiWarps = BN >= 64 ? 8 : 4;
    static constexpr int kThreads = 64 + 32 * kEpiWarps;
    // receive buffer of the split-K exchange: [peer][token slot][128 rows] fp32, ceil(BN / splits) token
    // slots per peer, i.e. at most BN + 7 token rows of 512 bytes
    static constexpr int kRecvBytes = kDense ? 0 : (BN + 7) * 512;
    static constexpr int kRingBytes = kStages * (kStageBytes + kSf);
    static constexpr int kSmemBytes = kRingBytes + kRecvBytes + 1024;
    static constexpr int kAccCols = BN < 32 ? 32 : BN;
    // behind the accumulator every ring slot has 8 weight-scale and 8 token-scale columns of its own, so that the weights'
    // scales can be in tensor memory before the tokens are there
    static constexpr int kSfCol = kAccCols, kSfSlotCols = 16;
    static constexpr int kTmemCols = pow2_cols(kAccCols + kSfSlotCols * kStages);
    static_assert(kStageBytes % 1024 == 0, "stage slots must keep 1024-byte alignment");
    static_assert(kCtasPerSm * kTmemCols <= 512, "tensor memory budget");
    static_assert(kCtasPerSm * (kSmemBytes + 256) <= 232448, "shared memory budget");
};

// Address of `local_addr` in the shared memory of CTA `peer` of this cluster.
__device__ __forceinline__ uint32_t peer_addr(uint32_t local_addr, uint32_t peer) {
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(local_addr), "r"(peer));
    return ra;
}
// The tensor-core instructions of a stage.  The whole warp comes here and `on` holds for its elected thread alone: predicated
// instructions in code that the warp runs together, because behind a branch that one thread takes alone every wait costs
// 200 cycles instead of 95.  The ring slot is a run-time value on purpose: a CTA runs only a handful of stages, so one
// compact code path beats a specialised copy per slot, each of which would be fetched cold.
// Scale atoms of one operand's stage: shared -> tensor memory, two atoms of four columns (the second one only if the stage
// covers more than 128 reduction elements).
__device__ __forceinline__ void copy_stage_scales(bool on, uint32_t sf_t, uint32_t slo, int rem) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %0, 0;\n\t@q tcgen05.cp.cta_group::1.32x128b.warpx4 [%1], %2;\n\t}"
                 ::"r"(static_cast<uint32_t>(on)), "r"(sf_t), "l"(desc64(kHiPlain, slo)));
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %0, 0;\n\t@q tcgen05.cp.cta_group::1.32x128b.warpx4 [%1], %2;\n\t}"
                 ::"r"(static_cast<uint32_t>(on && rem > 128)), "r"(sf_t + 4), "l"(desc64(kHiPlain, slo + (512 >> 4))));
}
__device__ __forceinline__ void mma_if(bool on, uint32_t d_tmem, uint32_t plo, uint32_t qlo, uint32_t idesc, uint32_t sfp_t, uint32_t sfq_t,
                                       uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 q, %7, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::mxf4.block_scale.block32 [%0], %1, %2, %3, [%5], [%6], p;\n\t}"
        ::"r"(d_tmem), "l"(desc64(kHiSw128, plo)), "l"(desc64(kHiSw128, qlo)), "r"(idesc), "r"(accumulate), "r"(sfp_t), "r"(sfq_t),
        "r"(static_cast<uint32_t>(on)));
}
__device__ __forceinline__ void commit_if(bool on, uint32_t bar) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
                 ::"r"(bar), "r"(static_cast<uint32_t>(on)) : "memory");
}
template <int BN>
__device__ __forceinline__ void issue_stage(bool on, uint32_t plo, uint32_t d_tmem, uint32_t sfp_t, int rem, uint32_t accumulate) {
    constexpr uint32_t idesc0 = (1u << 7) | (1u << 10) | ((BN >> 3) << 17) | (1u << 23) | ((128u >> 4) << 24);
    constexpr uint32_t idesc2 = idesc0 | (2u << 4) | (2u << 29);
    const uint32_t qlo = plo + (kPTile >> 4), sfq_t = sfp_t + 8;
    mma_if(on, d_tmem, plo, qlo, idesc0, sfp_t, sfq_t, accumulate);
    mma_if(on && rem > 64, d_tmem, plo + 2, qlo + 2, idesc2, sfp_t, sfq_t, 1);
    mma_if(on && rem > 128, d_tmem, plo + 4, qlo + 4, idesc0, sfp_t + 4, sfq_t + 4, 1);
    mma_if(on && rem > 192, d_tmem, plo + 6, qlo + 6, idesc2, sfp_t + 4, sfq_t + 4, 1);
}

template <int BN, bool kFused, bool kBatch, bool kDense = false>
__global__ void __launch_bounds__(DCfg<BN, kDense>::kThreads, DCfg<BN, kDense>::kCtasPerSm)
decode_kernel(const __grid_constant__ DecodeMaps maps, const DecodeBatch b) {
    using C = DCfg<BN, kDense>;
    // which of the batched layers this cluster works for (one launch may run several layers over the same
    // tokens, each with its own weights, activation codes and output)
    const int tile_all = static_cast<int>(blockIdx.x) / b.splits;
    int lin = 0;   // (kBatch = false: a single layer, nothing to look up)
    if (kBatch)
        while (lin + 1 < b.n_lin && tile_all >= b.lay[lin].tile_end) ++lin;
    DecodeParams p;
    p.M = b.M; p.K = b.K; p.k_tail = b.k_tail; p.x = b.x; p.ldx = b.ldx; p.y_bf16 = b.y_bf16; p.splits = b.splits;
    p.status = b.status; p.trace = b.trace; p.dbg = b.dbg;
    {
        const DecodeLayer& l = b.lay[lin];
        p.N = l.N; p.w_groups = l.w_groups; p.act_sf = l.act_sf; p.w_sf = l.w_sf; p.y = l.y; p.ldy = l.ldy;
    }
    const CUtensorMap* const tm_act = &maps.act[lin];
    const CUtensorMap* const tm_w = &maps.w[lin];
    extern __shared__ uint8_t smem_raw[];
    constexpr int kStages = C::kStages;
    // per ring slot: the weight side has landed (later ring passes: both sides); the tensor cores are done with both.
    // bar_t: the token side of the first ring pass (one barrier), or fused the quantiser's groups of items
    __shared__ __align__(8) uint64_t bar_w[kStages], bar_t[kStages], bar_empty[kStages], bar_acc_full;
    __shared__ __align__(8) uint64_t bar_recv;   // counts the bytes of partial sums that the peers deliver to this CTA
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag_s;
    volatile int* abort_flag = &abort_flag_s;

    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t smem_base = smem_u32(smem);
    constexpr int kTokSf = kStages * C::kStageBytes;   // token scales of slot i at kTokSf + i * kSf
    // (the warp and the tensor-memory address by way of a shuffle: uniform over the warp, as far as the compiler can see)
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const StagePlan plan(p.K, p.k_tail);
    const int S = plan.S, S1 = plan.S1;
    const int splits = p.splits;
    const int tile = tile_all - (lin ? b.lay[lin - 1].tile_end : 0);   // 128-row weight tile of this layer
    const int split = static_cast<int>(blockIdx.x) - tile_all * splits;   // = rank in the cluster
    const int s_begin = static_cast<int>(static_cast<uint32_t>(S) * split / splits);   // (S <= 2^24 stages, splits <= 8)
    const int s_end = static_cast<int>(static_cast<uint32_t>(S) * (split + 1) / splits);
    const int n_st = s_end - s_begin;
    const int n0 = tile * 128;
    // t / splits without a division: exact for t <= 135 and splits <= 8.  Token t belongs to CTA t mod splits of the cluster.
    const uint32_t rcp = 65536u / splits + 1;
    auto slot_of = [&](int tok) { return static_cast<int>((tok * rcp) >> 16); };

    long long* const ptrace = kTraceBuild ? p.trace : nullptr;
    const long long t_entry = kTraceBuild ? clock64() : 0;
    __shared__ int trace_slot_s;
    if (ptrace && blockIdx.x == 0 && threadIdx.x == 0) {
        unsigned long long g; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(g));
        const int sl = static_cast<int>(atomicAdd(reinterpret_cast<unsigned long long*>(ptrace + 2040), 1ull)) & 63;
        trace_slot_s = sl;
        ptrace[2048 + sl * 4] = static_cast<long long>(g);
    }
    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(smem_u32(&bar_w[i]), 1);
            mbar_init(smem_u32(&bar_t[i]), kFused ? C::kEpiWarps : 1);
            mbar_init(smem_u32(&bar_empty[i]), 1);
        }
        mbar_init(smem_u32(&bar_acc_full), 1);
        mbar_init(smem_u32(&bar_recv), 1);
        abort_flag_s = 0;
        fence_mbar_init();
        if (!kFused) tma_prefetch_desc(tm_act);
        tma_prefetch_desc(tm_w);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&tmem_slot), C::kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    // Split-K exchange, receiving side: this CTA owns tokens split, split + splits, ...; every CTA of the
    // cluster (itself included) delivers 512 bytes per owned token, counted on bar_recv.  The cluster
    // barrier only tells the peers that this CTA (and its bar_recv) is there before they push: arrive here, wait just
    // before the pushes, so that it costs nothing.
    const int n_own = split < p.M ? slot_of(p.M - split + splits - 1) : 0;
    const bool parked = BN == 128 && splits == 2;   // two CTAs, more than 64 tokens: see the exchange
    if (splits > 1) {
        if (!parked && threadIdx.x == 0) mbar_arrive_expect_tx(smem_u32(&bar_recv), static_cast<uint32_t>(n_own) * splits * 512u);
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    }
    // set-up done: let the next kernel of the stream be scheduled (its launch latency then overlaps this
    // kernel).  The roles that touch what earlier kernels wrote (activation codes and scales) or may
    // still read (y) pass grid_dependency_wait() first; the weights depend on no kernel, so the producer
    // requests them before it waits and they stream in while the previous kernel (normally the
    // activation quantiser) is still running.
    const long long t_setup = kTraceBuild ? clock64() : 0;
    // Up to 32 tokens the next kernel may be scheduled from here on: two CTAs share an SM, and the next GEMM's set-up and
    // weight stream overlap this one.  From 64 tokens on a CTA fills its SM and what comes next in a decode step is the
    // small-CTA activation quantiser, whose blocks would squeeze in beside this kernel's CTAs and slow their chain for
    // nothing (they wait for this kernel's result anyway): there the trigger comes once the reduction has been issued
    // (quantise + GEMM step 9.1 -> 8.5 us at 64 tokens, 11.75 -> 11.67 at 128; GEMM-only loops unchanged).
    // So does a launch of whole reductions that fill the ring more than once (more tiles than clusters of two would find room for):
    // the loads of the launch after next, which come up with the quantiser, only delay its own; there the trigger comes with the
    // tokens (two of 9728 x 2560, quantise + multiply, 16 / 32 tokens: 9.12 / 10.23 -> 8.84 / 9.78 us, 19456 x 2560 alone 7.28 / 8.27 ->
    // 6.17 / 7.37; 19456 x 1024, one ring pass, would lose: 3.62 -> 4.49).
    const bool late_trigger = BN >= 64 || (!kFused && splits == 1 && n_st > kStages);
    if (!late_trigger) grid_launch_dependents();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, tmem_slot, 0);
    long long* trace = (ptrace && blockIdx.x < 4) ? ptrace + blockIdx.x * 512 : nullptr;
    if (trace && threadIdx.x == 0) { trace[500] = clock64(); trace[502] = t_entry; trace[503] = t_setup; }
    const uint32_t lo_base = ((smem_base & 0x3FFFF) >> 4) | (1u << 16);

    if (warp == 0) {
        // ------------------------------------------------------------ producer
        const uint8_t* sfp = p.w_sf + (static_cast<size_t>(s_begin) * p.w_groups + tile) * kSfGroupBytes;
        const size_t sfp_stride = static_cast<size_t>(p.w_groups) * kSfGroupBytes;
        const uint8_t* sfq = p.act_sf + static_cast<size_t>(s_begin) * kSfGroupBytes;   // one token group per stage
        auto load_weights = [&](int it, int st, uint32_t more) {
            const int s = s_begin + it;
            const uint32_t sb = smem_base + st * C::kStageBytes, bar = smem_u32(&bar_w[st]);
            mbar_arrive_expect_tx(bar, kPTile + kSf + more);
            tma_load_2d(sb, tm_w, s < S1 ? s * 128 : p.K / 2 + (s - S1) * 128, n0, bar);
            bulk_load(sb + kPTile + C::kQTile, sfp + it * sfp_stride, kSf, bar);
        };
        // `sf_stages`: stages whose scale bytes come with this one (contiguous in both memories)
        auto load_tokens = [&](int it, int st, int sf_stages, uint32_t bar) {
            const int s = s_begin + it;
            if (sf_stages) bulk_load(smem_base + kTokSf + st * kSf, sfq + static_cast<size_t>(it) * kSfGroupBytes, sf_stages * kSf, bar);
            tma_load_2d(smem_base + st * C::kStageBytes + kPTile, tm_act, s < S1 ? s * 128 : (p.K - p.k_tail) / 2 + (s - S1) * 128, 0, bar);
        };
        // first ring pass: the weight side now, the token side after the dependency wait on a barrier of its own
        const int pre = min(kStages, n_st);
        if (elect_one())
            for (int i = 0; i < pre; ++i) load_weights(i, i, 0);
        __syncwarp();
        if (!kFused) {
            grid_dependency_wait();
            if (elect_one()) {
                mbar_arrive_expect_tx(smem_u32(&bar_t[0]), pre * (C::kQTile + kSf));
                for (int i = 0; i < pre; ++i) load_tokens(i, i, i == 0 ? pre : 0, smem_u32(&bar_t[0]));
            }
            __syncwarp();
        }
        // later passes: both sides together
        int st = 0, it = pre;
        uint32_t ph = 0;
        bool ok = true;
        for (; it < n_st; ++it) {
            if (!mbar_wait(smem_u32(&bar_empty[st]), ph, abort_flag)) { ok = false; break; }
            if (elect_one()) {
                load_weights(it, st, kFused ? 0 : C::kQTile + kSf);
                if (!kFused) load_tokens(it, st, 1, smem_u32(&bar_w[st]));
            }
            __syncwarp();
            if (++st == kStages) { st = 0; ph ^= 1; }
        }
        // gave up: the copies in flight land before the CTA leaves (bounded)
        if (!ok && lane == 0) {
            for (int j = max(0, it - kStages); j < it; ++j) {
                const uint32_t php = (j / kStages) & 1;
                for (int tries = 0; tries < (1 << 16) && !mbar_try_wait(smem_u32(&bar_w[j % kStages]), php); ++tries) {}
            }
            for (int tries = 0; !kFused && tries < (1 << 16) && !mbar_try_wait(smem_u32(&bar_t[0]), 0); ++tries) {}
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ tcgen05 issuer
        const bool leader = elect_one();
        const uint32_t d_tmem = tmem_base, sf_base = tmem_base + C::kSfCol;
        // the weights' scales of the first ring pass go to tensor memory as they land, normally long before the tokens
        const int pre = min(kStages, n_st);
        int s = s_begin, rem = s < S1 ? p.K - s * kStageK : p.k_tail - (s - S1) * kStageK;   // what stage s still covers
        auto next_stage = [&]() { rem = ++s == S1 ? p.k_tail : rem - kStageK; };
        uint32_t plo = lo_base, sfp_t = sf_base, tlo = lo_base + (kTokSf >> 4);
        bool ok = true;
        for (int it = 0; it < pre && ok; ++it) {
            ok = mbar_wait(smem_u32(&bar_w[it]), 0, abort_flag);
            copy_stage_scales(leader && ok, sfp_t, plo + ((kPTile + C::kQTile) >> 4), rem);
            plo += C::kStageBytes >> 4; sfp_t += C::kSfSlotCols;
            next_stage();
        }
        s = s_begin; rem = s < S1 ? p.K - s * kStageK : p.k_tail - (s - S1) * kStageK;
        plo = lo_base; sfp_t = sf_base;
        // Fused: the quantiser's items come in groups of 128, stage by stage; stage `it` of a pass needs the first
        // ceil((it + 1) M / 16) groups.  Otherwise the token side of the first ring pass is waited for as a whole: a wait
        // between two stages' instructions costs half a stage (issued back to back, two scale copies and four MMAs of 16
        // columns take 173 cycles, with one barrier probe per stage 260 - 320).
        int groups = 0, need = p.M + 15;
        if (!kFused) ok = ok && mbar_wait(smem_u32(&bar_t[0]), 0, abort_flag);
        if (BN < 64 && late_trigger) grid_launch_dependents();
        if (trace && lane == 0) trace[64] = clock64();
#pragma unroll 1
        for (int it = 0; it < pre && ok; ++it) {
            if (kFused) {
                while (ok && groups < (need >> 4)) { ok = mbar_wait(smem_u32(&bar_t[groups]), 0, abort_flag); ++groups; }
                need += p.M;
            }
            copy_stage_scales(leader && ok, sfp_t + 8, tlo, rem);
            issue_stage<BN>(leader && ok, plo, d_tmem, sfp_t, rem, it > 0);
            if (it + kStages < n_st) commit_if(leader && ok, smem_u32(&bar_empty[it]));
            plo += C::kStageBytes >> 4; sfp_t += C::kSfSlotCols; tlo += kSf >> 4;
            next_stage();
        }
        // later ring passes
        int st = 0;
        uint32_t ph = 1;
#pragma unroll 1
        for (int it = kStages; it < n_st && ok; ++it) {
            if (st == 0) { plo = lo_base; sfp_t = sf_base; tlo = lo_base + (kTokSf >> 4); groups = 0; need = p.M + 15; }
            ok = mbar_wait(smem_u32(&bar_w[st]), ph, abort_flag);
            copy_stage_scales(leader && ok, sfp_t, plo + ((kPTile + C::kQTile) >> 4), rem);
            if (kFused) {
                while (ok && groups < (need >> 4)) { ok = mbar_wait(smem_u32(&bar_t[groups]), ph, abort_flag); ++groups; }
                need += p.M;
            }
            copy_stage_scales(leader && ok, sfp_t + 8, tlo, rem);
            issue_stage<BN>(leader && ok, plo, d_tmem, sfp_t, rem, 1);
            if (it + kStages < n_st) commit_if(leader && ok, smem_u32(&bar_empty[st]));
            plo += C::kStageBytes >> 4; sfp_t += C::kSfSlotCols; tlo += kSf >> 4;
            next_stage();
            if (++st == kStages) { st = 0; ph ^= 1; }
        }
        commit_if(leader && ok, smem_u32(&bar_acc_full));
        if (trace && lane == 0) trace[128] = clock64();
        if (BN >= 64) grid_launch_dependents();
    } else {
        // ------------------------------------------------------------ epilogue warps: activation quantiser of this CTA
        // (fused), accumulator -> y or the owners' receive buffers, sums of this CTA's tokens
        const int q4 = warp & 3, ew = warp - 2;
        const int chunk0 = ew >> 2;                  // which of the quarter's warps this is
        const uint32_t acc_t = tmem_base + (static_cast<uint32_t>(q4 * 32) << 16);
        const uint32_t recv_base = smem_base + C::kRingBytes;
        const int slots = slot_of(p.M + splits - 1);                // token slots per peer in a receive buffer
        if constexpr (kFused) {
            // ---- An item is one token's 32-column block of a stage, and a thread takes item 128 j + its number of every group
            // of 128; items run block, token, stage, so that a few tokens' stages are quantised side by side (one token: all
            // five stages at once instead of one after the other, 2400 -> 1000 cycles).  Where a thread's items sit is
            // worked out before the wait. ----
            static_assert(BN == 16 && C::kEpiWarps == 4, "five groups of 128 items cover a ring pass of sixteen tokens");
            const int et = threadIdx.x - 64;
            // token-scale atoms of all slots start as zeros (rows past M and the unused atom rows stay so)
            for (int i = et; i < kStages * kSf / 16; i += 128) *reinterpret_cast<uint4*>(smem + kTokSf + i * 16) = make_uint4(0, 0, 0, 0);
            const int blk = et & 7;
            const uint32_t rcp_m = 65536u / p.M + 1;                          // row / M, exact for the 80 rows of a pass
            int stage_of[kStages], tok_of[kStages];
#pragma unroll
            for (int j = 0; j < kStages; ++j) {
                const int row = (et >> 3) + 16 * j;                           // (stage, token) of the pass
                stage_of[j] = static_cast<int>((row * rcp_m) >> 16);
                tok_of[j] = row - stage_of[j] * p.M;
            }
            asm volatile("bar.sync 1, 128;" ::: "memory");
            bool first = true;
#pragma unroll 1
            for (int base = 0; base < n_st; base += kStages) {
                const int n = min(kStages, n_st - base), n_groups = (n * p.M + 15) >> 4;
                const uint16_t* xp[kStages];
#pragma unroll
                for (int j = 0; j < kStages; ++j) {
                    const int s = s_begin + base + stage_of[j];
                    const int col = (s < S1 ? s * kStageK : p.K - p.k_tail + (s - S1) * kStageK) + blk * kBlock;
                    xp[j] = stage_of[j] < n && col < p.K ? p.x + static_cast<size_t>(tok_of[j]) * p.ldx + col : nullptr;
                }
                if (first) {
                    grid_dependency_wait();   // x is the previous kernel's output
                    if (ptrace && blockIdx.x == 0 && threadIdx.x == 64) { unsigned long long g; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(g)); ptrace[2048 + trace_slot_s * 4 + 1] = static_cast<long long>(g); }
                    if (trace && et == 0) trace[200] = clock64();
                }
                // the loads of all groups of a ring pass are in flight together
                uint4 q[kStages][4];
#pragma unroll
                for (int j = 0; j < kStages; ++j) {
                    if (j >= n_groups) break;
#pragma unroll
                    for (int w4 = 0; w4 < 4; ++w4)
                        q[j][w4] = xp[j] ? __ldg(reinterpret_cast<const uint4*>(xp[j] + 8 * w4)) : make_uint4(0, 0, 0, 0);
                }
                bool qok = true;
#pragma unroll
                for (int j = 0; j < kStages; ++j) {
                    if (j >= n_groups || !qok) break;
                    // a reused slot must have been drained by the tensor core (threads without an item wait too: their warp's
                    // arrival below must not run a pass ahead)
                    if (!first) qok = mbar_wait(smem_u32(&bar_empty[min(stage_of[j], n - 1)]), (base / kStages - 1) & 1, abort_flag);
                    if (stage_of[j] < n) {
                        uint8_t* slot = smem + stage_of[j] * C::kStageBytes;
                        uint4 codes;
                        const uint32_t byte = quant_block32(q[j], codes);
                        const int tok = tok_of[j];
                        // token tile: rows of 128 bytes, 16-byte piece c of row r at piece c ^ (r % 8)
                        *reinterpret_cast<uint4*>(slot + kPTile + tok * 128 + ((blk ^ (tok & 7)) << 4)) = codes;
                        smem[kTokSf + stage_of[j] * kSf + (blk >> 2) * 512 + tok * 16 + (blk & 3)] = static_cast<uint8_t>(byte);
                    }
                    qok = __all_sync(0xffffffffu, qok);
                    fence_proxy_async_smem();   // the tensor core reads the slot through the async proxy
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&bar_t[j]));
                    if (trace && lane == 0 && first && ew == 0) trace[201 + j] = clock64();
                }
                if (!qok) break;
                first = false;
            }
        } else {
            grid_dependency_wait();   // y may still be read by an earlier kernel
            if (ptrace && blockIdx.x == 0 && threadIdx.x == 64) { unsigned long long g; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(g)); ptrace[2048 + trace_slot_s * 4 + 1] = static_cast<long long>(g); }
            if (trace && threadIdx.x == 64) trace[200] = clock64();
        }
        // Accumulator -> registers -> y (splits == 1), or straight into the receive buffers of the tokens' owners: token
        // t belongs to CTA t mod splits, its slot there is t / splits, a receive buffer is [peer][slot][row].  (Or, of two CTAs,
        // -> the pipeline's buffers, which nothing reads any more, token by token: the other one's tokens go from there to its
        // receive buffer, this one's own are added from there.)
        if (splits > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // every peer is there
        if (mbar_wait(smem_u32(&bar_acc_full), 0, abort_flag)) {
            if (trace && threadIdx.x == 64) trace[192] = clock64();
            tc_fence_after_sync();
#pragma unroll 1
            for (int c = chunk0; c < (BN + 15) / 16; c += C::kEpiWarps / 4) {
                if (c * 16 >= p.M) break;
                uint32_t v[16];
                tmem_ld_32x16(acc_t + c * 16, v);
                tmem_ld_wait();
                if (splits == 1) {
                    const int n = n0 + q4 * 32 + lane;   // this lane's weight row
                    if (n < p.N) {
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const int tok = c * 16 + i;
                            if (tok < p.M) {
                                if (p.y_bf16)
                                    reinterpret_cast<__nv_bfloat16*>(p.y)[static_cast<size_t>(tok) * p.ldy + n] =
                                        __float2bfloat16_rn(__uint_as_float(v[i]));
                                else
                                    reinterpret_cast<float*>(p.y)[static_cast<size_t>(tok) * p.ldy + n] = __uint_as_float(v[i]);
                            }
                        }
                    }
                } else if (parked) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) reinterpret_cast<float*>(smem)[(c * 16 + i) * 128 + q4 * 32 + lane] = __uint_as_float(v[i]);
                } else {
                    // 4 x 4 transposes among the lanes of four weight rows: lane `sub` gets token 4 g + sub of those rows and
                    // sends them with one 16-byte asynchronous store, whose bytes are counted on the owner's barrier
                    const int sub = lane & 3;
                    const uint32_t recv_mine = recv_base + (split * slots * 128 + q4 * 32 + lane - sub) * 4;
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        if (c * 16 + 4 * g >= p.M) break;
                        uint32_t a0 = v[4 * g], a1 = v[4 * g + 1], a2 = v[4 * g + 2], a3 = v[4 * g + 3];
                        const uint32_t x0 = __shfl_xor_sync(0xffffffffu, (sub & 1) ? a0 : a1, 1);
                        const uint32_t x1 = __shfl_xor_sync(0xffffffffu, (sub & 1) ? a2 : a3, 1);
                        if (sub & 1) { a0 = x0; a2 = x1; } else { a1 = x0; a3 = x1; }
                        const uint32_t y0 = __shfl_xor_sync(0xffffffffu, (sub & 2) ? a0 : a2, 2);
                        const uint32_t y1 = __shfl_xor_sync(0xffffffffu, (sub & 2) ? a1 : a3, 2);
                        if (sub & 2) { a0 = y0; a1 = y1; } else { a2 = y0; a3 = y1; }
                        const int tok = c * 16 + 4 * g + sub;
                        const int slot = slot_of(tok), owner = tok - slot * splits;
                        if (tok < p.M) {
                            const uint32_t dst = peer_addr(recv_mine + slot * 512, owner);
                            const uint32_t rbar = peer_addr(smem_u32(&bar_recv), owner);
                            asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                                         ::"r"(dst), "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(rbar) : "memory");
                        }
                    }
                }
            }
            if (trace && threadIdx.x == 64) trace[195] = clock64();
        }
        tc_fence_before_sync();
        if (splits > 1) {
            if (parked) {
                asm volatile("bar.sync 1, %0;" ::"n"(32 * C::kEpiWarps) : "memory");   // the parked tile is complete
                for (int tok = abort_flag_s ? p.M : (split ^ 1) + 2 * ew; tok < p.M; tok += 2 * C::kEpiWarps) {
                    uint4 v;
                    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(smem_base + tok * 512 + lane * 16));
                    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};"
                                 ::"r"(peer_addr(recv_base + ((split * slots + (tok >> 1)) * 128 + 4 * lane) * 4, split ^ 1)), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
                }
                __syncwarp();
                asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
            } else if (n_own > 0) {
                // all partial sums of this CTA's tokens have arrived (nobody writes to this CTA after that)
                mbar_wait(smem_u32(&bar_recv), 0, abort_flag);
            }
            // this CTA's tokens: split, split + splits, ...; a thread owns 4 consecutive weight rows and
            // every kEpiWarps-th slot; the sum runs in peer order
            const int n = n0 + 4 * lane;
            const int n_sum = abort_flag_s ? 0 : n_own;
#pragma unroll 1
            for (int slot = ew; slot < n_sum; slot += C::kEpiWarps) {
                const int tok = split + slot * splits;
                float4 v[8];
#pragma unroll
                for (int peer = 0; peer < 8; ++peer)
                    if (peer < splits)
                        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                                     : "=f"(v[peer].x), "=f"(v[peer].y), "=f"(v[peer].z), "=f"(v[peer].w)
                                     : "r"(parked && peer == split ? smem_base + tok * 512 + lane * 16
                                                                   : recv_base + ((peer * slots + slot) * 128 + 4 * lane) * 4));
                float4 sum = v[0];
#pragma unroll
                for (int peer = 1; peer < 8; ++peer)
                    if (peer < splits) { sum.x += v[peer].x; sum.y += v[peer].y; sum.z += v[peer].z; sum.w += v[peer].w; }
                if (n + 3 < p.N) {
                    if (p.y_bf16) {
                        __nv_bfloat162 lo = __floats2bfloat162_rn(sum.x, sum.y), hi = __floats2bfloat162_rn(sum.z, sum.w);
                        uint2 pk = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
                        *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.y) + static_cast<size_t>(tok) * p.ldy + n) = pk;
                    } else {
                        *reinterpret_cast<float4*>(reinterpret_cast<float*>(p.y) + static_cast<size_t>(tok) * p.ldy + n) = sum;
                    }
                } else {
                    const float e[4] = {sum.x, sum.y, sum.z, sum.w};
                    for (int i = 0; i < 4 && n + i < p.N; ++i) {
                        if (p.y_bf16)
                            reinterpret_cast<__nv_bfloat16*>(p.y)[static_cast<size_t>(tok) * p.ldy + n + i] = __float2bfloat16_rn(e[i]);
                        else
                            reinterpret_cast<float*>(p.y)[static_cast<size_t>(tok) * p.ldy + n + i] = e[i];
                    }
                }
            }
            if (trace && threadIdx.x == 64) trace[194] = clock64();
        }
        // A CTA that gave up pushes nothing and sums nothing, but healthy peers still deliver their partial
        // sums into its receive buffer and count them on its barrier: it stays until they have (bounded), so
        // that no store of a peer reaches the shared memory of a CTA that has left.
        if (splits > 1 && !parked && abort_flag_s && n_own > 0 && threadIdx.x == 64)
            mbar_wait_after_abort(smem_u32(&bar_recv), 0);
    }
    // the cluster barrier that the epilogue warps have passed
    if (splits > 1 && warp < 2) {
        __syncwarp();
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (parked) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }

    // ------------------------------------------------------------ teardown (normal and aborted)
    tc_fence_before_sync();
    __syncthreads();
    if (trace && threadIdx.x == 0) trace[501] = clock64();
    if (ptrace && blockIdx.x == 0 && threadIdx.x == 64) { unsigned long long g; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(g)); ptrace[2048 + trace_slot_s * 4 + 2] = static_cast<long long>(g); }
    if (warp == 1) {
        __syncwarp();
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, C::kTmemCols);
    }
    if (threadIdx.x == 0 && abort_flag_s) atomicExch(p.status, static_cast<int>(PRQ_ERR_TIMEOUT));
}

template <int BN, bool kFused, bool kBatch, bool kDense = false>
cudaError_t launch_one(const DecodeMaps& maps, const DecodeBatch& b, cudaStream_t stream) {
    const DecodeBatch& p = b;
    const int n_tiles = b.lay[b.n_lin - 1].tile_end;
    using C = DCfg<BN, kDense>;
    if (kDense && p.splits != 1) return cudaErrorInvalidValue;   // the dense variant has no receive buffer
    static OncePerDevice opt_in;
    const cudaError_t e = opt_in([] { return cudaFuncSetAttribute(decode_kernel<BN, kFused, kBatch, kDense>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes); });
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_tiles * p.splits);
    cfg.blockDim = dim3(C::kThreads);
    cfg.dynamicSmemBytes = C::kSmemBytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = p.splits;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, decode_kernel<BN, kFused, kBatch, kDense>, maps, b);
}

// more weight tiles than SMs, no K split, 64 tokens or more: the two-CTAs-per-SM variant
bool wants_dense(int bn, const DecodeBatch& b) {
    if (bn < 64 || b.splits != 1) return false;
    int sms = 0;
    if (current_sm_count(&sms) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return b.lay[b.n_lin - 1].tile_end > sms;
}

// The occupancy query counts one CTA per SM for every kernel that allocates tensor memory, however little; two do run beside
// each other up to 32 tokens (a launch's CTAs enter while the one before it computes).  A kernel without it, of the same
// threads and shared memory, gives the number that is wanted there.
template <int kThreads>
__global__ void __launch_bounds__(kThreads) occupancy_stand_in(int* p) {
    extern __shared__ int stand_in_smem[];
    if (p) *p = stand_in_smem[threadIdx.x];
}

template <int BN>
int max_clusters(int splits) {
    using C = DCfg<BN>;
    const void* kernel = C::kCtasPerSm > 1 ? reinterpret_cast<const void*>(occupancy_stand_in<C::kThreads>) : reinterpret_cast<const void*>(decode_kernel<BN, false, false>);
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes + 256) != cudaSuccess) { cudaGetLastError(); return 0; }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(splits);
    cfg.blockDim = dim3(C::kThreads);
    cfg.dynamicSmemBytes = C::kSmemBytes + (C::kCtasPerSm > 1 ? 256 : 0);   // (the stand-in has no static shared memory)
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = splits;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
    return n;
}

}  // namespace

cudaError_t launch_decode_batch(int bn, const DecodeMaps& maps, const DecodeBatch& b, cudaStream_t stream) {
    if (b.n_lin < 1 || b.n_lin > kMaxBatch) return cudaErrorInvalidValue;
    if (b.x != nullptr)   // fused activation quantiser: one layer, the 16-token tile only
        return (bn == 16 && b.n_lin == 1) ? launch_one<16, true, false>(maps, b, stream) : cudaErrorInvalidValue;
    const bool dense = wants_dense(bn, b);
    if (b.n_lin > 1) {
        switch (bn) {
            case 16: return launch_one<16, false, true>(maps, b, stream);
            case 32: return launch_one<32, false, true>(maps, b, stream);
            case 64: return dense ? launch_one<64, false, true, true>(maps, b, stream) : launch_one<64, false, true>(maps, b, stream);
            default: return dense ? launch_one<128, false, true, true>(maps, b, stream) : launch_one<128, false, true>(maps, b, stream);
        }
    }
    if (dense)
        return bn == 64 ? launch_one<64, false, false, true>(maps, b, stream) : launch_one<128, false, false, true>(maps, b, stream);
    switch (bn) {
        case 16: return launch_one<16, false, false>(maps, b, stream);
        case 32: return launch_one<32, false, false>(maps, b, stream);
        case 64: return launch_one<64, false, false>(maps, b, stream);
        default: return launch_one<128, false, false>(maps, b, stream);
    }
}

cudaError_t launch_decode(int bn, const CUtensorMap& tm_act, const CUtensorMap& tm_w, const DecodeParams& p,
                          int n_tiles, cudaStream_t stream) {
    DecodeMaps maps;
    std::memset(&maps, 0, sizeof(maps));
    maps.act[0] = tm_act; maps.w[0] = tm_w;
    DecodeBatch b = {};
    b.x = p.x; b.status = p.status; b.trace = p.trace;
    b.M = p.M; b.K = p.K; b.k_tail = p.k_tail; b.ldx = p.ldx;
    b.y_bf16 = p.y_bf16; b.splits = p.splits; b.dbg = p.dbg;
    b.n_lin = 1;
    b.lay[0] = DecodeLayer{p.act_sf, p.w_sf, p.y, p.N, p.w_groups, p.ldy, n_tiles};
    return launch_decode_batch(bn, maps, b, stream);
}

int decode_max_active_clusters(int bn, int splits) {
    switch (bn) {
        case 16: return max_clusters<16>(splits);
        case 32: return max_clusters<32>(splits);
        case 64: return max_clusters<64>(splits);
        default: return max_clusters<128>(splits);
    }
}

}  // namespace prq
