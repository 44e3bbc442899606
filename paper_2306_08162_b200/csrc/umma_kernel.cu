// Tensor-core kernel of the quantized-linear + LoRA layer for sm_100a: TMA-staged packed codes and group parameters,
// register-level unpack + dequantisation to bf16 in shared memory, tcgen05 MMA with fp32 accumulators in tensor
// memory, LoRA update fused as one extra MMA per tile, bf16 epilogue.
//
// One kernel template serves both directions (Figure 1 of the paper):
//   forward        Out[m, n] = sum_k X[m, k]  W[n, k] + s sum_j H[m, j] B[n, j]      contraction over k
//   backward-input Out[m, k] = sum_n dY[m, n] W[n, k] + s sum_j G[m, j] A[j, k]      contraction over n
// The backward direction is the paper's fused "transpose + unpack + matmul" (Section 3.1): nothing is transposed in
// memory.  The packed word still yields consecutive-k codes; they are written as one 16-byte chunk of a shared-memory
// operand whose *non-contraction* dimension is contiguous, and the MMA descriptor's major-ness bit does the rest.
//
// Orientation: the dequantised weight tile is the MMA's A operand (128 rows), the activation tile is the B operand
// (up to 256 token rows), so every dequantised weight is reused by up to 256 tokens inside one CTA.  The accumulator
// D[weight row, token] lives in tensor memory (two buffers of 256 columns, so the epilogue of one tile overlaps the
// main loop of the next).
//
// Warp roles (480 threads): warp 0 = TMA producer of activation tiles, warp 1 = MMA issuer (+ tensor-memory
// allocation), warp 2 = TMA producer of packed codes + group parameters (its ring runs ahead of the activation ring),
// warps 3-6 = epilogue (+ LoRA operand staging), warps 7-14 = unpack/dequant (two groups taking alternate stages).  In the DOWN
// build warps 3-14 are three dequant groups, and all warps finish the tile.
// Every mbarrier wait is bounded; on a timeout the kernel records a status word, drains and returns.
#include <cuda.h>

#include <mutex>

#include "common.cuh"
#include "device_state.h"
#include "launch.h"
#include "lora_down.cuh"
#include "umma_plan.h"

namespace qlora {

__device__ unsigned int g_device_status = 0;   // sticky; bit 0: an mbarrier wait timed out

// The producer clusters of a launch signal its tile CTAs through a pair of counters in the CALLER's workspace (the layer
// calls carve two words out of it): [0] producer CTAs that have published their rows, [1] tile CTAs that have seen the
// full count.  A one-warp kernel ahead of the launch sets the pair to zero (in stream order, with programmatic dependent
// launch, so the main kernel's set-up still overlaps its predecessor); the last tile CTA zeroes it again.

namespace {

constexpr int kThreads = 480;
constexpr int kDequantWarp0 = 7, kGroupWarps = 4;   // two dequant groups of four warps (DOWN: a third in the epilogue's place)
constexpr int kEpiWarp0 = 3, kEpiWarps = 4;
constexpr int kSyncWords = 64;                       // counters in the workspace: [0], [1] producer clusters, [2 ..] one per split tile
constexpr size_t kSplitTileBytes = 2 * 2 * 8 * 8 * 128 * 16;   // exchange area of one split tile: 2 halves x 2 CTAs x 8 chunks x 4 KiB
constexpr int kAccStride = 256;      // tensor-memory columns per accumulator buffer
constexpr uint32_t kSpinLimit = 1u << 26;
constexpr int kWaitLimitUs = 250000;   // default limit of a wait, a launch parameter: far beyond any healthy wait (microseconds), short for a hang

struct Params : TilePlan {
    float s;
    const float* Pmat;               // H (forward) or G (backward), fp32 [M, r]
    const __nv_bfloat16* L;          // B [N, r] (forward) or A [r, K] (backward)
    __nv_bfloat16* Out;
    // producer clusters (n_prod > 0, as in the CTA-pair kernel): the first n_prod clusters of the grid compute
    // P = In * Ldown into Pout (== Pmat) beside the tiles and publish it through the counter pair `sync`
    int n_prod, T, lds_stages;
    unsigned int* sync;   // the counter pair (n_prod > 0)
    int wait_limit_us;    // every wait inside the kernel gives up after this long
    const __nv_bfloat16* In;         // [M, T]
    const __nv_bfloat16* Ldown;      // A [r, K] (forward) or B [N, r] (backward)
    float* Pout;
};

// ---------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok;
}
__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait: gives up after abort_flag[1] microseconds of wall time (the launch's limit, set beside the flag when the
// kernel starts) or kSpinLimit polls.  Returns false when the kernel is
// aborting (this wait or another one ran out).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    uint64_t t0 = 0;
    for (uint32_t i = 0; i < kSpinLimit; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 63u) == 63u) {
            if (*abort_flag) return false;
            const uint64_t now = global_ns();
            if (t0 == 0) t0 = now;
            else if (now - t0 > (uint64_t)abort_flag[1] * 1000ull) break;
        }
    }
    *abort_flag = 1;
    atomicOr(&g_device_status, 1u);
    return false;
}
// Whole-warp wait: lane 0 polls (so a waiting warp costs one lane's issue slots), the outcome is broadcast, and every
// lane then observes the completed phase itself before touching the data the barrier guards.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int lane) {
    if (__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, parity) != 0u)) return true;   // already complete: one instruction per lane
    uint32_t ok = 1;
    if (lane == 0) ok = mbar_wait(bar, parity, abort_flag) ? 1u : 0u;
    ok = __shfl_sync(0xFFFFFFFFu, ok, 0);
    if (ok) (void)mbar_try_wait(bar, parity);
    return ok != 0;
}
// The same for the MMA issuer, whose wait ends a stage's chain: every lane polls, so no lane hands the outcome on and the phase is not read again.
// INT4, rank 8, from warp_wait to this: 512 x 512, 64 tokens 6.0 -> 5.65 us; 11008 -> 4096, 256 tokens 33.8 -> 33.3, 200 tokens 31.2 -> 30.7; 4096 x 4096,
// 700 tokens 33.2 -> 32.6; four ranks on 32 tiles up to 1 % slower.  (In the roles that issue copies it gives nothing: 2048 x 2048, 300 tokens 13.85 -> 14.0.)
__device__ __forceinline__ bool warp_poll(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    uint64_t t0 = 0;
    for (uint32_t i = 0; i < kSpinLimit; ++i) {
        if (__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, parity) != 0u)) return true;
        if ((i & 63u) == 63u) {
            if (__any_sync(0xFFFFFFFFu, *abort_flag != 0)) return false;
            const uint64_t now = __shfl_sync(0xFFFFFFFFu, global_ns(), 0);
            if (t0 == 0) t0 = now;
            else if (now - t0 > (uint64_t)abort_flag[1] * 1000ull) break;
        }
    }
    *abort_flag = 1;
    atomicOr(&g_device_status, 1u);
    return false;
}
// One lane of a converged warp, the same one every time.  The roles that issue TMA copies and MMAs run as whole warps and elect a lane for
// the instructions alone, so that ring positions, addresses and descriptors are warp-uniform values, which these instructions want: run by
// lane 0 of a diverged warp they cost 75 to 150 cycles each (a trace of one CTA had the dequant warps 3000 cycles ahead of the MMAs).
// INT4, rank 0, 64 tokens: 4096 -> 11008 29.3 -> 25.9, 4096 x 4096 13.3 -> 12.2 us; rank 8, 300 tokens, 11008 -> 4096 44.6 -> 41.3.  Tiles of
// 200 to 256 tokens, which wait for their products, gain nothing (4096 -> 11008, 256 tokens 33.0 -> 32.9; 11008 -> 4096 33.1 -> 33.3).
__device__ __forceinline__ bool elect_one() {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) ::"memory");
    return ok != 0;
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                 ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, {%5, %5, %5, %5}, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(0u) : "memory");
}
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ---------------------------------------------------------------- thread-block cluster helpers
__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// shared::cluster address of the same shared-memory offset in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_cta(uint32_t local_addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local_addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void st_cluster_16(uint32_t cluster_addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(cluster_addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ float4 ld_cluster_f32x4(uint32_t cluster_addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(cluster_addr) : "memory");
    return v;
}


// Bounded wait until a counter in global memory reaches `target` (written by other CTAs of the same launch).
__device__ __forceinline__ bool wait_counter(const unsigned* ctr, unsigned target, volatile int* abort_flag) {
    uint64_t t0 = 0;
    for (uint32_t i = 0; i < kSpinLimit; ++i) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
        if (v >= target) return true;
        __nanosleep(256);
        if ((i & 63u) == 63u) {
            if (*abort_flag) return false;
            const uint64_t now = global_ns();
            if (t0 == 0) t0 = now;
            else if (now - t0 > (uint64_t)abort_flag[1] * 1000ull) break;
        }
    }
    *abort_flag = 1;
    atomicOr(&g_device_status, 1u);
    return false;
}

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

#include "lora_down_stream.cuh"

// Eight of s * P as bf16 (the LoRA operand), and -- where it is wanted -- in `low` what that rounding left over, again as bf16.
__device__ __forceinline__ uint4 lora_p_chunk(const float4& a, const float4& b, float s, bool want_low, uint4& low) {
    const float f[8] = {s * a.x, s * a.y, s * a.z, s * a.w, s * b.x, s * b.y, s * b.z, s * b.w};
    uint32_t o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
        o[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
    if (want_low) {
        uint32_t l[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {    // (nothing is left of a value that became infinite or was no number)
            const float l0 = f[2 * i] - bf16_lo(o[i]), l1 = f[2 * i + 1] - bf16_hi(o[i]);
            const __nv_bfloat162 r = __floats2bfloat162_rn(fabsf(l0) < INFINITY ? l0 : 0.f, fabsf(l1) < INFINITY ? l1 : 0.f);
            l[i] = *reinterpret_cast<const uint32_t*>(&r);
        }
        low = make_uint4(l[0], l[1], l[2], l[3]);
    }
    return make_uint4(o[0], o[1], o[2], o[3]);
}

// Eight bf16 with 0 in the place of infinities and NaN: the adapter rows that meet the low pieces.  (An infinite element has had its say
// in the product with the high piece; times a low piece that is zero, or of the other sign, it would make the sum a NaN.)
__device__ __forceinline__ uint4 finite_only(uint4 v) {
    uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if ((w[i] & 0x7F80u) == 0x7F80u) w[i] &= 0xFFFF0000u;
        if ((w[i] & 0x7F800000u) == 0x7F800000u) w[i] &= 0xFFFFu;
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// Shared-memory matrix descriptor (version 1).  Offsets in bytes; layout 0 = no swizzle, 2 = 128-byte swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo, uint32_t layout) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46) | ((uint64_t)layout << 61);
}
// Instruction descriptor: bf16 x bf16 -> fp32, M = m_mma, N = n_mma; majors: 0 = contraction-contiguous, 1 = other.
__device__ __forceinline__ uint32_t instr_desc(uint32_t n_mma, uint32_t a_mn_major, uint32_t b_mn_major, uint32_t m_mma = 128) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (a_mn_major << 15) | (b_mn_major << 16) | ((n_mma >> 3) << 17) |
           ((m_mma >> 4) << 24);
}

// Ring position: slot index plus the phase bit of the current lap (no division in the hot loops).
struct Ring {
    uint32_t slot = 0, phase = 0;
    __device__ __forceinline__ void advance(uint32_t n) { if (++slot == n) { slot = 0; phase ^= 1u; } }
};

// Eight ranks of the adapter applied second, for one weight row (zero beyond the last).
template <bool TRANSPOSED>
__device__ __forceinline__ uint4 lora_up_chunk(const Params& p, int wrow, int jc) {
    if (wrow >= p.C) return make_uint4(0, 0, 0, 0);
    if constexpr (!TRANSPOSED) {
        return __ldg(reinterpret_cast<const uint4*>(p.L + (size_t)wrow * p.r + jc * 8));      // B[n, j..j+7]
    } else {
        uint32_t e[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) e[j] = __bfloat16_as_ushort(__ldg(p.L + (size_t)(jc * 8 + j) * p.K + wrow));     // A[j, k]
        return make_uint4(e[0] | (e[1] << 16), e[2] | (e[3] << 16), e[4] | (e[5] << 16), e[6] | (e[7] << 16));
    }
}

// DOWN (split tiles of ranks 8 and 16 up to 128 tokens, where down_pays says so): no producer clusters.  Every rank forms its part of P = In * Ldown beside its
// part of the tile, from the activation stages it has anyway -- four more MMAs per stage, the adapter as their 64-row operand -- and the
// parts of P meet where the tile's parts do; s P L is added in fp32 there.  So nothing has to be counted in device memory, nor the counters
// set to zero by a launch ahead, and a tile waits for no other.
template <int BITS, bool TRANSPOSED, bool DOWN>
__global__ void __launch_bounds__(kThreads, 1)
umma_gemm_kernel(const __grid_constant__ CUtensorMap tm_act, const __grid_constant__ CUtensorMap tm_q,
                 const __grid_constant__ CUtensorMap tm_scales, const __grid_constant__ CUtensorMap tm_zeros,
                 const __grid_constant__ CUtensorMap tm_down, const Params p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag_s[2];   // [0] set when a wait gave up, [1] the launch's wait limit in microseconds
    volatile int* abort_flag = abort_flag_s;
    pdl_launch_dependents();

    const uint32_t smem0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem0 - smem_u32(smem_raw));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t S = (uint32_t)p.S, P = (uint32_t)p.P;

    // barrier addresses
    const uint32_t bar_full_x = smem0 + p.off_bar;          // [S]  stage full: activation tile landed (TMA) and weight tile
    const uint32_t bar_full_w = bar_full_x;                 //      written by one dequant group (one wait for the MMA issuer)
    const uint32_t bar_empty = bar_full_x + 8 * S;          // [S]  MMAs reading the stage have completed
    const uint32_t bar_full_p = bar_empty + 8 * S;          // [P]  packed words + group parameters landed (TMA)
    const uint32_t bar_empty_p = bar_full_p + 8 * P;        // [P]  the dequant group has read them into registers
    const uint32_t bar_acc_full = bar_empty_p + 8 * P;      // [2]  accumulator buffer complete
    const uint32_t bar_acc_empty = bar_acc_full + 16;       // [2]  accumulator buffer drained by the epilogue
    const uint32_t bar_lora_full = bar_acc_empty + 16;      // [1]  LoRA operand tiles staged

    if (threadIdx.x == 0) {
        abort_flag_s[0] = 0; abort_flag_s[1] = p.wait_limit_us;
        for (uint32_t i = 0; i < S; ++i) {
            mbar_init(bar_full_x + 8 * i, 1 + kGroupWarps);
            mbar_init(bar_empty + 8 * i, 1);
        }
        for (uint32_t i = 0; i < P; ++i) {
            mbar_init(bar_full_p + 8 * i, 1);
            mbar_init(bar_empty_p + 8 * i, kGroupWarps);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar_acc_full + 8 * i, 1);
            mbar_init(bar_acc_empty + 8 * i, kEpiWarps);
        }
        mbar_init(bar_lora_full, kEpiWarps);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {   // whole warp: allocate all 512 tensor-memory columns (one CTA per SM owns them)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    // Set-up done.  The frozen weights are read-only for every call of the library, so their producer starts at once; the
    // roles that touch what the preceding work in the stream may have produced (activations, P) or may still be reading
    // (the output) call pdl_wait() first.

    // Few tokens give few tiles: the contraction of a tile is then split over a cluster of p.split CTAs (rank i takes steps
    // i * p.steps ...), each accumulates its part in tensor memory, and the parts are added through distributed shared
    // memory at the end.  One tile per cluster in that mode.
    const int rank = p.split > 1 ? (int)cluster_ctarank() : 0;
    const int first_tile = (int)blockIdx.x / p.split - p.n_prod, tile_stride = (int)gridDim.x / p.split - p.n_prod;
    const int step0 = rank * p.steps;

    if (!DOWN && first_tile < 0) {
        // ------------------------------------------------------------------ producer cluster: LoRA down-projection on SMs
        // the tiles leave idle (one CTA per row block or more; lowest block indices, so they wait for nobody)
        const int n_ctas = p.n_prod * p.split;
        if (p.M <= 256) {   // ask all lines this CTA will read (its share of the adapter) into L2 at once; nothing is read into the SM
            const size_t row = (size_t)p.T * 2, share = (size_t)p.r * row / (size_t)n_ctas;
            const char* l = reinterpret_cast<const char*>(p.Ldown) + (size_t)blockIdx.x * share;
            for (size_t o = (size_t)threadIdx.x * 128; o < share; o += kThreads * 128) prefetch_l2(l + o);
            for (int m = (int)blockIdx.x * 16; m < p.M; m += n_ctas * 16) {
                const char* x = reinterpret_cast<const char*>(p.In) + (size_t)m * row;
                const size_t n = (size_t)min(16, p.M - m) * row;
                for (size_t o = (size_t)threadIdx.x * 128; o < n; o += kThreads * 128) prefetch_l2(x + o);
            }
        }
        pdl_wait();
        if (p.M <= 256) {
            // few row blocks (two per CTA at most) and a short main loop: 16-byte row loads (the bulk copies of the streaming form bring
            // 10 - 30 GB/s per SM: P came 5000 cycles after the main loops at 128 tokens, 4096 x 4096).  INT8, 128 tokens, forward:
            // activations in L2 18.0 -> 15.6 us, from DRAM 18.2 -> 16.4 (without the request ahead 19.0: a round of loads is in flight at a time).
            float* red = reinterpret_cast<float*>(smem_gen);
            const bool one = (p.M + 15) / 16 <= n_ctas;           // one row block per CTA
            if (p.r <= 8) {
                if (one) lora_down_rows<!TRANSPOSED, 1, 1, 6>(p.M, p.T, p.r, p.In, p.Ldown, p.Pout, (int)blockIdx.x * 16, n_ctas * 16, kThreads / 32, red);
                else     lora_down_rows<!TRANSPOSED, 1, 2, 4>(p.M, p.T, p.r, p.In, p.Ldown, p.Pout, (int)blockIdx.x * 16, n_ctas * 16, kThreads / 32, red);
            } else {
                if (one) lora_down_rows<!TRANSPOSED, 2, 1, 5>(p.M, p.T, p.r, p.In, p.Ldown, p.Pout, (int)blockIdx.x * 16, n_ctas * 16, kThreads / 32, red);
                else     lora_down_rows<!TRANSPOSED, 2, 2, 2>(p.M, p.T, p.r, p.In, p.Ldown, p.Pout, (int)blockIdx.x * 16, n_ctas * 16, kThreads / 32, red);
            }
        } else {
            if (p.r <= 8) lora_down_stream<!TRANSPOSED, 1>(p.M, p.T, p.r, p.In, p.Ldown, p.Pout, (int)blockIdx.x, n_ctas, smem_gen, p.lds_stages, abort_flag);
            else          lora_down_stream<!TRANSPOSED, 2>(p.M, p.T, p.r, p.In, p.Ldown, p.Pout, (int)blockIdx.x, n_ctas, smem_gen, p.lds_stages, abort_flag);
        }
        __threadfence();       // every thread's rows of P are visible device-wide before the CTA is counted
        __syncthreads();
        if (threadIdx.x == 0) atomicAdd(&p.sync[0], 1u);
    } else if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer: activation tiles
        pdl_wait();
        Ring ring;
        for (int tile = first_tile; tile < p.n_tiles; tile += tile_stride) {
            const int m0 = (tile % p.n_tok_tiles) * p.BT;
            for (int step = 0; step < p.steps; ++step) {
                if (!warp_wait(bar_empty + 8 * ring.slot, ring.phase ^ 1u, abort_flag, lane)) goto done;
                const uint32_t bar = bar_full_x + 8 * ring.slot, dst = smem0 + p.off_x + ring.slot * p.x_stage_bytes;
                const int c0 = (step0 + step) * kStepC;
                const uint32_t dst_l = smem0 + p.off_l + ring.slot * p.down_bytes;
                if (elect_one()) {
                    mbar_expect_tx(bar, p.x_stage_bytes + (DOWN ? p.down_bytes : 0u));
                    tma_load_2d(dst, &tm_act, bar, c0, m0);
                    if constexpr (DOWN) {                    // the stage's part of the adapter: eight ranks in 1 KiB
                        tma_load_2d(dst_l, &tm_down, bar, TRANSPOSED ? 0 : c0, TRANSPOSED ? c0 : 0);
                        if (TRANSPOSED && p.r > 8) tma_load_2d(dst_l + 1024, &tm_down, bar, 8, c0);
                    }
                }
                ring.advance(S);
            }
        }
    } else if (warp == 2) {
        // ------------------------------------------------------------------ TMA producer: packed codes, scales, zeros
        Ring ring;
        const uint32_t tx_bytes = p.words_bytes + 2 * p.scale_bytes;
        for (int tile = first_tile; tile < p.n_tiles; tile += tile_stride) {
            // forward: weight rows n = w0.., contraction k = c0..;  backward: weight rows k = w0.., contraction n = c0..
            const int w0 = (tile / p.n_tok_tiles) * kWRows;
            for (int step = 0; step < p.steps; ++step) {
                if (!warp_wait(bar_empty_p + 8 * ring.slot, ring.phase ^ 1u, abort_flag, lane)) goto done;
                const uint32_t dst = smem0 + p.off_p + ring.slot * p.packed_slot_bytes, bar = bar_full_p + 8 * ring.slot;
                const int c0 = (step0 + step) * kStepC, x = TRANSPOSED ? c0 : w0, k = TRANSPOSED ? w0 : c0, gr = k / p.g;
                if (elect_one()) {
                    mbar_expect_tx(bar, tx_bytes);
                    tma_load_2d(dst, &tm_q, bar, x, k * BITS / 32);
                    tma_load_2d(dst + p.words_bytes, &tm_scales, bar, x, gr);
                    tma_load_2d(dst + p.words_bytes + p.scale_bytes, &tm_zeros, bar, x, gr);
                }
                ring.advance(P);
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (one elected thread)
        const uint32_t idesc = instr_desc((uint32_t)p.BT, TRANSPOSED ? 1u : 0u, 0u);
        const uint32_t idesc_lora = instr_desc((uint32_t)p.BT, 0u, 0u);
        // Descriptors of slot 0; the start-address field (16-byte units) is advanced per slot and per 16-wide MMA step.
        // activation tile: contraction-contiguous rows of 128 B, 128-byte swizzle, 8-row groups 1024 B apart.
        // weight tile: forward = the same layout (rows n); backward = rows are the contraction (n) with 64 k contiguous:
        //   MN-major, 64-element atoms 8192 B apart (LBO), 8-row contraction groups 1024 B apart (SBO).
        const uint64_t b_desc0 = smem_desc(smem0 + p.off_x, 16, 1024, 2);
        const uint64_t a_desc0 = TRANSPOSED ? smem_desc(smem0 + p.off_w, 8192, 1024, 2) : smem_desc(smem0 + p.off_w, 16, 1024, 2);
        constexpr uint32_t a_k16 = TRANSPOSED ? (2048u >> 4) : (32u >> 4);
        const uint32_t x_step = p.x_stage_bytes >> 4;
        // DOWN: the adapter as the 64-row operand (rows beyond r are whatever lies there; their sums are not looked at); the sums go to the
        // second accumulator, which a split tile does not use.
        //   forward A [r, k]: rows of 128 B, 128-byte swizzle;  backward B [n, r]: 16-byte rows of eight ranks, so 8 x 8 core matrices
        //   of 128 B, consecutive along the contraction, 1 KiB from one eight ranks to the next
        const uint32_t idesc_down = instr_desc((uint32_t)p.BT, TRANSPOSED ? 1u : 0u, 0u, 64u);
        const uint64_t l_desc0 = TRANSPOSED ? smem_desc(smem0 + p.off_l, 128, 1024, 0) : smem_desc(smem0 + p.off_l, 16, 1024, 2);
        constexpr uint32_t l_k16 = TRANSPOSED ? (256u >> 4) : (32u >> 4);
        Ring ring;
        uint32_t tile_it = 0;
        for (int tile = first_tile; tile < p.n_tiles; tile += tile_stride, ++tile_it) {
            const uint32_t buf = tile_it & 1u;
            const uint32_t d_tmem = tmem_base + buf * kAccStride;
            if (!warp_poll(bar_acc_empty + 8 * buf, ((tile_it >> 1) & 1u) ^ 1u, abort_flag)) goto done;
            tc_fence_after();
            uint32_t acc = 0;
            for (int step = 0; step < p.steps; ++step) {
                if (!warp_poll(bar_full_x + 8 * ring.slot, ring.phase, abort_flag)) goto done;
                tc_fence_after();
                const uint64_t b_desc = b_desc0 + ring.slot * x_step;
                const uint64_t a_desc = a_desc0 + ring.slot * (uint32_t)(kWStageBytes >> 4);
                const uint64_t l_desc = l_desc0 + ring.slot * (p.down_bytes >> 4);
                const uint32_t bar = bar_empty + 8 * ring.slot;
                if (elect_one()) {
#pragma unroll
                    for (int k16 = 0; k16 < kStepC / 16; ++k16)
                        tc_mma(d_tmem, a_desc + k16 * a_k16, b_desc + k16 * 2, idesc, acc | (uint32_t)(k16 > 0));
                    if constexpr (DOWN)
#pragma unroll
                        for (int k16 = 0; k16 < kStepC / 16; ++k16)
                            tc_mma(tmem_base + kAccStride, l_desc + k16 * l_k16, b_desc + k16 * 2, idesc_down, acc | (uint32_t)(k16 > 0));
                    tc_commit(bar);
                }
                acc = 1;
                ring.advance(S);
            }
            if (!DOWN && p.r > 0 && rank == 0) {   // the LoRA update goes into one rank's part only
                if (!warp_poll(bar_lora_full, tile_it & 1u, abort_flag)) goto done;
                tc_fence_after();
                if (elect_one())
                    for (int jb = 0; jb < p.r_pad / 16; ++jb) {
                        // un-swizzled operands: 8-row x 16-byte core matrices 128 B apart (SBO), contraction halves LBO apart
                        const uint64_t a_desc = smem_desc(smem0 + p.off_lora_a + jb * 2 * (kWRows * 16), kWRows * 16, 128, 0);
                        const uint64_t b_desc = smem_desc(smem0 + p.off_lora_p + jb * 2 * (p.BT * 16), p.BT * 16, 128, 0);
                        tc_mma(d_tmem, a_desc, b_desc, idesc_lora, 1u);
                    }
                __syncwarp();
            }
            if (elect_one()) tc_commit(bar_acc_full + 8 * buf);
        }
    } else if (!DOWN && warp >= kEpiWarp0 && warp < kDequantWarp0) {
        // ------------------------------------------------------------------ epilogue (+ LoRA operand staging)
        const int q = warp & 3;                      // tensor-memory lane quarter this warp may read
        const int et = threadIdx.x - kEpiWarp0 * 32; // 0..127
        pdl_wait();
        uint32_t tile_it = 0;
        for (int tile = first_tile; tile < p.n_tiles; tile += tile_stride, ++tile_it) {
            const int wt = tile / p.n_tok_tiles, tt = tile % p.n_tok_tiles;
            const int w0 = wt * kWRows, m0 = tt * p.BT;
            const uint32_t buf = tile_it & 1u;
            if (p.n_prod > 0 && tile_it == 0 && rank == 0) {
                // P is being computed by this launch's producer clusters: one thread waits for all of their CTAs, is counted
                // as done with the counter, and the last such CTA of the launch zeroes the pair for the next one.
                if (et == 0 && wait_counter(&p.sync[0], (unsigned)(p.n_prod * p.split), abort_flag)) {
                    const unsigned n_cons = gridDim.x / (unsigned)p.split - (unsigned)p.n_prod;   // one waiting CTA per tile cluster
                    if (atomicAdd(&p.sync[1], 1u) == n_cons - 1u) {
                        atomicExch(&p.sync[0], 0u);
                        atomicExch(&p.sync[1], 0u);
                    }
                }
                asm volatile("bar.sync 2, %0;" ::"r"(kEpiWarps * 32) : "memory");
                if (*abort_flag) break;
            }
            if (p.r > 0 && rank == 0) {   // (the LoRA update goes into rank 0's part only)
                // (the previous tile's LoRA MMA has completed: its accumulator-full barrier was observed below)
                uint8_t* la = smem_gen + p.off_lora_a;
                uint8_t* lp = smem_gen + p.off_lora_p;
                const int row = et, wrow = w0 + row;
                const int n8 = p.r >> 3;                      // chunks of eight ranks; the low pieces' chunks follow, then padding
                for (int jc = 0; jc < p.r_pad / 8; ++jc) {
                    if (p.lora_lo && jc >= n8) break;         // (no padding then: r_pad == 2 r)
                    const uint4 v = jc < n8 ? lora_up_chunk<TRANSPOSED>(p, wrow, jc) : make_uint4(0, 0, 0, 0);
                    uint8_t* dst = la + jc * (kWRows * 16) + (row >> 3) * 128 + (row & 7) * 16;
                    *reinterpret_cast<uint4*>(dst) = v;
                    if (p.lora_lo) *reinterpret_cast<uint4*>(dst + n8 * (kWRows * 16)) = finite_only(v);
                }
                for (int row_t = et; row_t < p.BT; row_t += 128) {
                    const int m = m0 + row_t;
                    for (int jc = 0; jc < p.r_pad / 8; ++jc) {
                        if (p.lora_lo && jc >= n8) break;
                        uint4 v = make_uint4(0, 0, 0, 0), low = v;
                        if (jc < n8 && m < p.M) {
                            // (not the read-only path: P may have been written by this launch's producer clusters)
                            const float4* src = reinterpret_cast<const float4*>(p.Pmat + (size_t)m * p.r + jc * 8);
                            v = lora_p_chunk(__ldcg(src), __ldcg(src + 1), p.s, p.lora_lo != 0, low);
                        }
                        uint8_t* dst = lp + jc * (p.BT * 16) + (row_t >> 3) * 128 + (row_t & 7) * 16;
                        *reinterpret_cast<uint4*>(dst) = v;
                        if (p.lora_lo) *reinterpret_cast<uint4*>(dst + n8 * (p.BT * 16)) = low;
                    }
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_lora_full);
            }
            if (!warp_wait(bar_acc_full + 8 * buf, (tile_it >> 1) & 1u, abort_flag, lane)) break;
            tc_fence_after();
            const int c = w0 + q * 32 + lane;                 // output column owned by this thread
            const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + buf * kAccStride;
            if (p.split > 1) break;                           // (the parts of a split tile: below, with the dequant warps' help)
#pragma unroll 1
            for (int cb = 0; cb < p.BT; cb += 16) {
                uint32_t v[16];
                tc_ld16(taddr + cb, v);
                tc_wait_ld();
                if (c < p.C) {
                    __nv_bfloat16* optr = p.Out + (size_t)(m0 + cb) * p.C + c;
                    const int rows_left = p.M - (m0 + cb);
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        if (j < rows_left) *optr = __float2bfloat16_rn(__uint_as_float(v[j]));
                        optr += p.C;
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_acc_empty + 8 * buf);
        }
    } else if (warp >= (DOWN ? kEpiWarp0 : kDequantWarp0)) {
        // ------------------------------------------------------------------ unpack + dequant
        // (DOWN: one tile per CTA, so the epilogue's warps would be idle until the end; they are a third group.)
        constexpr int kGroups = DOWN ? kDownGroups : kDequantGroups, kWarp0 = DOWN ? kEpiWarp0 : kDequantWarp0;
        // The groups of four warps take the pipeline stages in turn, so each has as many stage times as there are groups for its serial chain
        // (wait, shared-memory loads, arithmetic, wait, stores, fence, arrive); rings_sound says which ring lengths that allows.  Inside a group a thread owns one column of
        // the packed tile and two blocks of 32 consecutive-k codes.
        const int group = (warp - kWarp0) / kGroupWarps;
        const int gt = threadIdx.x - (kWarp0 + group * kGroupWarps) * 32;   // 0..127 inside the group
        const int col = gt % p.packed_cols;                       // column of the packed tile (n in both directions)
        const int kb0 = gt / p.packed_cols;                       // forward: 0; backward: 0..1
        const int kb_stride = TRANSPOSED ? 2 : 1;                 // the thread's two code blocks are kb0 and kb0 + kb_stride
        const uint32_t row_base = (uint32_t)(col >> 3) * 1024u + (uint32_t)(col & 7) * 128u;   // row `col` of a swizzled tile
        const uint32_t sw = (uint32_t)(col & 7);
        uint32_t w_off[2], chunk0[2], soff[2];
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int kb = kb0 + b * kb_stride;                   // 32-code block along k: 0..1 forward, 0..3 backward
            w_off[b] = row_base + (TRANSPOSED ? (uint32_t)(kb >> 1) * 8192u : 0u);
            chunk0[b] = (uint32_t)((TRANSPOSED ? (kb & 1) : kb) * 4);
            soff[b] = (uint32_t)((((kb * 32) / p.g) % p.scale_rows) * p.packed_cols + col);   // (a stage holds several group rows when groups are short)
        }
        const uint32_t pcols = (uint32_t)p.packed_cols;
        const int my_tiles = first_tile < p.n_tiles ? (p.n_tiles - first_tile + tile_stride - 1) / tile_stride : 0;
        const int total = my_tiles * p.steps;
        Ring ring_w, ring_p;
        for (int i = 0; i < group; ++i) { ring_w.advance(S); ring_p.advance(P); }
        for (int it = group; it < total; it += kGroups) {
            if (!warp_wait(bar_full_p + 8 * ring_p.slot, ring_p.phase, abort_flag, lane)) break;
            const uint8_t* pk = smem_gen + p.off_p + ring_p.slot * p.packed_slot_bytes;
            const uint32_t* pw = reinterpret_cast<const uint32_t*>(pk);
            const __half* ps = reinterpret_cast<const __half*>(pk + p.words_bytes);
            const __half* pz = reinterpret_cast<const __half*>(pk + p.words_bytes + p.scale_bytes);
            uint32_t w[2][BITS];
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const uint32_t kb = (uint32_t)(kb0 + b * kb_stride);
#pragma unroll
                for (int i = 0; i < BITS; ++i) w[b][i] = pw[(kb * BITS + i) * pcols + col];
            }
            GroupParams gp[2];
            gp[0] = gp[1] = group_params(ps[soff[0]], pz[soff[0]]);
            if (p.scale_rows > 1) gp[1] = group_params(ps[soff[1]], pz[soff[1]]);   // (else the stage lies inside one group: 11008 -> 4096, 700 tokens 81.0 -> 79.3 us)
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_empty_p + 8 * ring_p.slot);

            uint32_t out[2][16];
#pragma unroll
            for (int b = 0; b < 2; ++b) dequant32<BITS>(w[b], gp[b], out[b]);

            if (!warp_wait(bar_empty + 8 * ring_w.slot, ring_w.phase ^ 1u, abort_flag, lane)) break;
            uint8_t* ws = smem_gen + p.off_w + ring_w.slot * kWStageBytes;
#pragma unroll
            for (int b = 0; b < 2; ++b)
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    *reinterpret_cast<uint4*>(ws + w_off[b] + (((chunk0[b] + c) ^ sw) << 4)) =
                        make_uint4(out[b][4 * c], out[b][4 * c + 1], out[b][4 * c + 2], out[b][4 * c + 3]);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_full_w + 8 * ring_w.slot);
#pragma unroll
            for (int i = 0; i < kGroups; ++i) { ring_w.advance(S); ring_p.advance(P); }
        }
        if (DOWN && group == 0) {         // the adapter applied second, [8 ranks][weight row]: every rank adds the update to its tokens below
            pdl_wait();
            uint8_t* la = smem_gen + p.off_lora_a;
            for (int jc = 0; jc < p.r / 8; ++jc) *reinterpret_cast<uint4*>(la + (jc * kWRows + gt) * 16) = lora_up_chunk<TRANSPOSED>(p, first_tile / p.n_tok_tiles * kWRows + gt, jc);
        }
    }

done:
    if constexpr (DOWN) {
        // The parts meet at the ranks that finish them: rank i takes tokens i * BT / split ...  Every rank stores its fp32 sums from tensor
        // memory straight into the owners' shared memory, over the operand ring, which is idle once every rank's products are
        // through: that is what the first cluster barrier says; the second says that the parts have arrived, and after it nobody touches a
        // peer's memory again.  Bound by what comes into an SM from its neighbours, about 13 bytes a cycle whichever way it is moved: the other
        // form below (parts put down, read by their owners) is 0.2 - 0.3 us slower up to 64 tokens and 10 % faster at 256; st.async on the
        // owners' mbarriers and bulk copies were 0.4 - 1.2 us slower.
        // Layout: [rank][token / 4][128 weight rows][4 tokens], a warp's store is 512 contiguous bytes; behind it P's, [rank][token / 4][r][4 tokens].
        __syncwarp();
        bool mine = warp >= kEpiWarp0;                         // the epilogue and the dequant warps, three per lane quarter, 16 tokens in turn
        if (mine) mine = warp_wait(bar_acc_full, 0u, abort_flag, lane);
        tc_fence_after();
        cluster_arrive();
        const uint32_t quarter = (uint32_t)warp & 3u, tpr4 = (uint32_t)(p.BT / p.split) >> 2, r = (uint32_t)p.r;
        const uint32_t taddr = tmem_base + ((quarter * 32u) << 16);
        int cb = 16 * ((warp - kEpiWarp0) >> 2);
        uint32_t v[16];
        if (mine && cb < p.BT) { tc_ld16(taddr + cb, v); tc_wait_ld(); }
        cluster_wait();
        if (mine) {
            const uint32_t row = quarter * 32u + (uint32_t)lane;
            // (lane: the first lanes of P's accumulator are its ranks)
            auto send = [&](uint32_t base, uint32_t width, uint32_t col) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t t4 = (uint32_t)(cb >> 2) + j, owner = t4 / tpr4;
                    const uint32_t off = base + (((uint32_t)rank * tpr4 + (t4 - owner * tpr4)) * width + col) * 16u;
                    st_cluster_16(map_to_cta(smem0 + off, owner), v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                }
            };
#pragma unroll 1
            while (cb < p.BT) {
                send(0u, kWRows, row);
                if (quarter == 0) {
                    tc_ld16(taddr + kAccStride + cb, v);
                    tc_wait_ld();
                    if (lane < p.r) send((uint32_t)p.BT * (kWRows * 4u), r, (uint32_t)lane);
                    __syncwarp();
                }
                cb += 48;
                if (cb < p.BT) { tc_ld16(taddr + cb, v); tc_wait_ld(); }
            }
        }
        __syncwarp();
        cluster_arrive();
        cluster_wait();
        pdl_wait();             // every thread stores part of the output
        const bool go = __all_sync(0xFFFFFFFFu, !*abort_flag) != 0;
        const int wt = first_tile / p.n_tok_tiles, tt = first_tile % p.n_tok_tiles;
        const int m_own = tt * p.BT + rank * (p.BT / p.split), c = wt * kWRows;
        const float4* parts = reinterpret_cast<const float4*>(smem_gen);
        float4* sp = reinterpret_cast<float4*>(smem_gen + p.off_lora_p);     // s * P of this rank's tokens, [token / 4][r][4 tokens]
        if (go)
            for (uint32_t i = threadIdx.x; i < tpr4 * r; i += kThreads) {
                const float4* part = parts + (uint32_t)p.BT * (kWRows / 4) + i;
                float4 y = part[0];
                for (uint32_t rk = 1; rk < (uint32_t)p.split; ++rk) {
                    const float4 x = part[rk * tpr4 * r];
                    y.x += x.x; y.y += x.y; y.z += x.z; y.w += x.w;
                }
                if (wt == 0) {                                 // one tile of a token's many writes P out
                    const uint32_t t4 = i / r, j = i - t4 * r;
                    const int m = m_own + 4 * (int)t4;
                    float* out = p.Pout + (size_t)m * p.r + j;
                    if (m < p.M) out[0] = y.x;
                    if (m + 1 < p.M) out[p.r] = y.y;
                    if (m + 2 < p.M) out[2 * p.r] = y.z;
                    if (m + 3 < p.M) out[3 * p.r] = y.w;
                }
                sp[i] = make_float4(p.s * y.x, p.s * y.y, p.s * y.z, p.s * y.w);
            }
        __syncthreads();
        if (go) {
            const bool odd = (lane & 1) != 0;
            // four tokens of one weight row (output column) at a time; the ranks' parts are added in rank order (the same bits on every run)
#pragma unroll 1
            for (uint32_t e = threadIdx.x; e < tpr4 * kWRows; e += kThreads) {
                float4 x[4];
#pragma unroll
                for (int rk = 0; rk < 4; ++rk)
                    if (rk < p.split) x[rk] = parts[(uint32_t)rk * tpr4 * kWRows + e];
                float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int rk = 0; rk < 4; ++rk)
                    if (rk < p.split) { y.x += x[rk].x; y.y += x[rk].y; y.z += x[rk].z; y.w += x[rk].w; }
                const uint32_t t4 = e / kWRows, n = e % kWRows;
                const uint4* up = reinterpret_cast<const uint4*>(smem_gen + p.off_lora_a) + n;
#pragma unroll 1
                for (uint32_t jc = 0; jc < r / 8; ++jc) {      // + s P L, in fp32
                    const uint4 l = up[jc * kWRows];
                    const float lf[8] = {bf16_lo(l.x), bf16_hi(l.x), bf16_lo(l.y), bf16_hi(l.y), bf16_lo(l.z), bf16_hi(l.z), bf16_lo(l.w), bf16_hi(l.w)};
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float4 q4 = sp[t4 * r + jc * 8 + j];
                        y.x = fmaf(q4.x, lf[j], y.x); y.y = fmaf(q4.y, lf[j], y.y); y.z = fmaf(q4.z, lf[j], y.z); y.w = fmaf(q4.w, lf[j], y.w);
                    }
                }
                // neighbouring lanes trade two tokens each, so that a lane stores two columns of two tokens
                const float r0 = __shfl_xor_sync(0xFFFFFFFFu, odd ? y.x : y.z, 1), r1 = __shfl_xor_sync(0xFFFFFFFFu, odd ? y.y : y.w, 1);
                const __nv_bfloat162 o0 = odd ? __floats2bfloat162_rn(r0, y.z) : __floats2bfloat162_rn(y.x, r0);
                const __nv_bfloat162 o1 = odd ? __floats2bfloat162_rn(r1, y.w) : __floats2bfloat162_rn(y.y, r1);
                const int m = m_own + (int)t4 * 4 + (odd ? 2 : 0), col = c + (int)(n & ~1u);
                if (col < p.C) {                                  // C is a multiple of 64: both columns or none
                    __nv_bfloat16* out = p.Out + (size_t)m * p.C + col;
                    if (m < p.M) *reinterpret_cast<__nv_bfloat162*>(out) = o0;
                    if (m + 1 < p.M) *reinterpret_cast<__nv_bfloat162*>(out + p.C) = o1;
                }
            }
        }
    }
    if (!DOWN && p.split > 1 && warp >= kEpiWarp0 && first_tile >= 0 && first_tile < p.n_tiles) {
        // This rank's part of the tile, fp32 [token][128 weight rows], over the (now idle) operand ring: the epilogue and the dequant
        // warps, three per lane quarter, take 16 tokens at a time in turn.
        __syncwarp();
        if (warp_wait(bar_acc_full, 0u, abort_flag, lane)) {
            tc_fence_after();
            const int quarter = warp & 3;
            float* part = reinterpret_cast<float*>(smem_gen) + quarter * 32 + lane;
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16);
#pragma unroll 1
            for (int cb = 16 * ((warp - kEpiWarp0) >> 2); cb < p.BT; cb += 48) {
                uint32_t v[16];
                tc_ld16(taddr + cb, v);
                tc_wait_ld();
#pragma unroll
                for (int j = 0; j < 16; ++j) part[(cb + j) * kWRows] = __uint_as_float(v[j]);
            }
        }
    }
    // ---------------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {   // give copies that may still be in flight time to land before the CTA's memory is released
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
        __syncthreads();
    }
    if (!DOWN && p.split > 1) {
        // Add the ranks' parts in rank order (fixed order: deterministic); rank i finishes tokens i * BT / split ...
        __syncwarp();
        cluster_sync_all();
        pdl_wait();            // every thread stores part of the output below
        if (!*abort_flag && first_tile >= 0 && first_tile < p.n_tiles) {
            const int wt = first_tile / p.n_tok_tiles, tt = first_tile % p.n_tok_tiles;
            const int w0 = wt * kWRows, m0 = tt * p.BT;
            const int tok_per_rank = p.BT / p.split;
            const uint32_t part_addr = smem0;
            uint32_t peer[4];
            for (int rk = 0; rk < 4; ++rk) peer[rk] = map_to_cta(part_addr, (uint32_t)(rk < p.split ? rk : 0));
            // Four weight rows (output columns) at a time, two such pieces per turn: all reads of the peers are under way together (one
            // after the other they took 4900 cycles at 128 tokens).  kThreads is a multiple of 32, so a thread's columns stay the same.
            const int n_e = tok_per_rank * (kWRows / 4), cw = (threadIdx.x % (kWRows / 4)) * 4;
#pragma unroll 1
            for (int e0 = threadIdx.x; e0 < n_e; e0 += 2 * kThreads) {
                float4 x[2][4];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int e = e0 + u * kThreads, t = rank * tok_per_rank + e / (kWRows / 4);
#pragma unroll
                    for (int rk = 0; rk < 4; ++rk)
                        if (rk < p.split && e < n_e) x[u][rk] = ld_cluster_f32x4(peer[rk] + (uint32_t)((t * kWRows + cw) * 4));
                }
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int e = e0 + u * kThreads, t = rank * tok_per_rank + e / (kWRows / 4);
                    if (e >= n_e || m0 + t >= p.M || w0 + cw >= p.C) continue;     // C is a multiple of 8: four columns are all-in or all-out
                    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int rk = 0; rk < 4; ++rk)
                        if (rk < p.split) { v.x += x[u][rk].x; v.y += x[u][rk].y; v.z += x[u][rk].z; v.w += x[u][rk].w; }
                    const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
                    *reinterpret_cast<uint2*>(p.Out + (size_t)(m0 + t) * p.C + w0 + cw) =
                        make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
                }
            }
        }
        __syncwarp();
        cluster_sync_all();   // nobody leaves while a peer may still read its part
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &qres) != cudaSuccess ||
            qres != cudaDriverEntryPointSuccess)
            f = nullptr;
        return (EncodeTiledFn)f;
    }();
    return fn;
}

bool make_map_2d(CUtensorMap* map, CUtensorMapDataType dt, int elem_bytes, const void* base, uint64_t inner, uint64_t outer,
                 uint32_t box_inner, uint32_t box_outer, CUtensorMapSwizzle sw) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {inner, outer};
    cuuint64_t strides[1] = {inner * (uint64_t)elem_bytes};
    cuuint32_t box[2] = {box_inner, box_outer};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, dt, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
              CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Sets a launch's counter pair to zero.  It is launched like the layer kernels (programmatic stream serialization): it
// lets its successor start at once and writes only after its own predecessor -- whose last tile CTAs may still be
// using the pair -- has completed; the kernel behind it touches the pair only after griddepcontrol.wait, i.e. after this
// grid has completed.
__global__ void sync_zero_kernel(unsigned int* sync) {
    pdl_launch_dependents();
    pdl_wait();
    if (threadIdx.x < kSyncWords) sync[threadIdx.x] = 0u;
}

int zero_sync_pair(unsigned int* sync, cudaStream_t st) {
    return launch_pdl(sync_zero_kernel, dim3(1), dim3(kSyncWords), 0, st, 1, sync) == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
}

// Clusters of `width` CTAs, an SM each, that run at a time on the current device (the builds of the kernel differ in nothing that counts here).
int fitting_clusters(int width) {
    static std::mutex mu;
    static int max_clusters_dev[kMaxDevices][5] = {};   // per device, by cluster width
    static SmemLimit limit;
    const int dev = device_ordinal();
    std::lock_guard<std::mutex> lock(mu);
    int& n = max_clusters_dev[dev < 0 ? 0 : dev][width];
    if (n == 0) {
        auto kern = umma_gemm_kernel<4, false, false>;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(sm_count() / width * width));
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = 232448 - 1024;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = (unsigned)width; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        if (!limit.raise(kern, 232448 - 1024) || cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n <= 0) { (void)cudaGetLastError(); n = -1; }
    }
    return n;
}

// (a device that does not tell: its SMs by the cluster's width)
GpuFit gpu_fit() {
    const int sms = sm_count(), c2 = fitting_clusters(2), c4 = fitting_clusters(4);
    return GpuFit{sms, c2 > 0 ? c2 : sms / 2, c4 > 0 ? c4 : sms / 4};
}

// Ldown != NULL: P = In * Ldown is still to be computed.  Where the tile clusters leave room for more clusters on the GPU
// (cudaOccupancyMaxActiveClusters: 33 clusters of 4 fit on 148 SMs, 74 of 2), producer clusters in front of the grid do
// it beside the tiles; else a down-projection launch goes ahead of the kernel.
template <int BITS, bool TRANSPOSED>
int launch_impl(const CUtensorMap& ta, const CUtensorMap& tq, const CUtensorMap& ts, const CUtensorMap& tz, const CUtensorMap& tl, const Params& p_in,
                size_t smem_bytes, int grid, cudaStream_t st, const void* Ldown, unsigned int* sync) {
    if (p_in.down_bytes > 0) {
        static SmemLimit down_limit;
        auto down_kern = umma_gemm_kernel<BITS, TRANSPOSED, true>;
        if (!down_limit.raise(down_kern, 232448 - 1024)) return QLORA_ERR_CUDA;
        return launch_pdl(down_kern, dim3((unsigned)grid), dim3(kThreads), smem_bytes, st, (unsigned)p_in.split, ta, tq, ts, tz, tl, p_in) == cudaSuccess
                   ? QLORA_OK : QLORA_ERR_CUDA;
    }
    static SmemLimit limit;
    auto kern = umma_gemm_kernel<BITS, TRANSPOSED, false>;
    if (!limit.raise(kern, 232448 - 1024)) return QLORA_ERR_CUDA;
    Params p = p_in;
    p.n_prod = 0; p.sync = nullptr; p.wait_limit_us = kWaitLimitUs;
    if (Ldown != nullptr && p.r > 0) {
        const int n_blocks = (p.M + 15) / 16;
        const int idle = fitting_clusters(p.split) - grid / p.split;
        int n_prod = (n_blocks + p.split - 1) / p.split;           // one row block per producer CTA when there is room
        if (n_prod > idle) n_prod = idle;
        const bool fits = p.r <= 16 && n_prod > 0 && n_prod * p.split * 2 >= n_blocks && p.lds_stages >= LDS_MIN_STAGES;
        if (fits && sync != nullptr) {
            p.n_prod = n_prod;
            p.sync = sync;
            grid += n_prod * p.split;
            const int rc = zero_sync_pair(sync, st);
            if (rc != QLORA_OK) return rc;
        } else {
            const int rc = launch_lora_down(p.M, p.T, p.r, !TRANSPOSED, p.In, p.Ldown, p.Pout, st);
            if (rc != QLORA_OK) return rc;
        }
    }
    // one cluster of p.split CTAs per tile when the contraction is split
    return launch_pdl(kern, dim3((unsigned)grid), dim3(kThreads), smem_bytes, st, (unsigned)p.split, ta, tq, ts, tz, tl, p) == cudaSuccess
               ? QLORA_OK : QLORA_ERR_CUDA;
}

#include "umma_pair.cuh"

}  // namespace

int launch_lora_down_stream(int M, int T, int r, bool l_is_A, const void* In, const void* L, float* P, cudaStream_t st, const uint8_t* mask, float out_scale) {
    return launch_lora_down_stream_impl(M, T, r, l_is_A, In, L, P, st, mask, out_scale);
}
bool lora_down_streams_masked(int M, int r) { return lds_masked(M, r); }

bool umma_supported(const qlora_desc& d, int M) {
    if (M < 1) return false;
    if (d.K % 64 != 0 || d.N % 64 != 0) return false;              // contraction steps of 64 in both directions
    // a stage's 64 (forward) or 128 (backward) rows along k hold whole groups, or lie inside one: every 32-code block then has
    // its scale row at the same place in every stage.  (Groups of 32 on the CUDA cores instead: 4210 us for a step of 333 tokens
    // on 11008 -> 4096, against 126 here.)
    if (!(d.group_size == 32 || d.group_size == 64 || d.group_size % 128 == 0)) return false;
    if (d.r > 64) return false;
    return true;
}

// Tiles of a partly filled last wave that are split two ways along the contraction (0: none).  Worth it when at most
// half a wave is left over, so that every left-over tile finds two pairs, and the halves are still long enough.
static int pair_split_tiles(int n_tiles, int steps, int pairs) {
    if (n_tiles <= pairs || steps < 16) return 0;
    const int rem = n_tiles % pairs;
    if (rem == 0 || 2 * rem > pairs || 2 + rem > kSyncWords) return 0;
    return rem;
}

// Workspace the CTA-pair kernel may use to exchange the halves of split tiles, forward or backward (0 when M is too small
// for that kernel or nothing is split).
size_t umma_split_scratch_bytes(const qlora_desc& d, int M) {
    if (M <= 256 || !umma_supported(d, M)) return 0;
    const int pairs = sm_count() / 2;
    const int tok_tiles = (M + 4 * kPairTok - 1) / (4 * kPairTok);
    const int rem_f = pair_split_tiles(tok_tiles * ((d.N + 2 * kPairW - 1) / (2 * kPairW)), d.K / kStepC, pairs);
    const int rem_b = pair_split_tiles(tok_tiles * ((d.K + 2 * kPairW - 1) / (2 * kPairW)), d.N / kStepC, pairs);
    return (size_t)(rem_f > rem_b ? rem_f : rem_b) * kSplitTileBytes;
}

// Workspace with which a backward call of this shape can compute dB on its producer clusters: one [N, r] fp32 part per
// producer CTA (0: the CTA-pair kernel would not take dB on).
size_t umma_db_part_bytes(const qlora_desc& d, int M) {
    return (size_t)2 * umma_db_on_producers(d, M) * (size_t)d.N * d.r * sizeof(float);
}

// CTA-pair kernel: 512 tokens x 256 weight rows per pair of SMs (see prefer_pair_kernel for when it is used).
static int launch_umma_pair(const qlora_desc& d, int M, bool transposed, const void* In, const int32_t* Q, const void* scales,
                            const void* zeros, const void* L, float* Pmat, void* Out, cudaStream_t st, const void* Ldown,
                            unsigned int* sync, void* split_buf, size_t split_bytes, DbFuse* db, bool plan_only = false,
                            const DownExtra* extra = nullptr) {
    // plan_only: nothing is launched and no pointer is looked at; the return value is the number of producer pairs when a
    // backward call with every optional workspace area would form dB on them, else 0
    PairParams p{};
    p.M = M; p.N = d.N; p.K = d.K; p.bits = d.bits; p.g = d.group_size; p.r = d.r; p.lora_lo = keep_lora_low(d.r, d.group_size); p.r_pad = lora_columns(d.r, d.group_size);
    p.C = transposed ? d.K : d.N;
    const int T = transposed ? d.N : d.K;
    p.n_tok_tiles = (M + 4 * kPairTok - 1) / (4 * kPairTok);
    const int n_w_tiles = (p.C + 2 * kPairW - 1) / (2 * kPairW);
    p.n_tiles = p.n_tok_tiles * n_w_tiles;
    p.steps = T / kStepC;
    plan_packed_stage(p, d.bits, d.group_size, transposed);
    p.s = d.r > 0 ? d.alpha / (float)d.r : 0.f;
    p.Pmat = Pmat; p.L = (const __nv_bfloat16*)L; p.Out = (__nv_bfloat16*)Out;

    uint32_t lora_l = (uint32_t)(kPairW * p.r_pad * 2), lora_p = (uint32_t)(2 * kPairTok * p.r_pad * 2);
    if (lora_l + lora_p < 8192) lora_p = 8192 - lora_l;   // the area doubles as the epilogue's staging slices (4 warps x 2 KiB)
    if (!plan_pair_rings(p.packed_slot_bytes, lora_l + lora_p, p.S, p.P)) return QLORA_ERR_UNSUPPORTED;
    p.off_x = 0;
    p.off_w = p.off_x + p.S * kPairXStage;
    p.off_p = p.off_w + p.S * kWStageBytes;
    p.off_lora_l = p.off_p + p.P * p.packed_slot_bytes;
    p.off_lora_p = p.off_lora_l + lora_l;
    p.off_bar = (p.off_lora_p + lora_p + 127u) / 128u * 128u;
    const size_t smem_bytes = (size_t)p.off_bar + 512 + 1024;

    const int pairs = sm_count() / 2;
    p.n_prod = 0; p.T = T; p.sync = nullptr; p.wait_limit_us = kWaitLimitUs;
    p.In = (const __nv_bfloat16*)In; p.Ldown = (const __nv_bfloat16*)Ldown; p.Pout = Pmat;
    p.r_down = extra != nullptr && extra->only_r > 0 ? extra->only_r : d.r;
    p.mask = extra != nullptr ? extra->mask : nullptr;
    p.out_scale = extra != nullptr ? extra->out_scale : 1.0f;
    const int lds_stage = p.mask != nullptr ? LDS_MASKED_STAGE_BYTES : LDS_STAGE_BYTES;
    p.lds_stages = (int)((p.off_bar - LDS_BAR_BYTES) / lds_stage);
    if (p.lds_stages > 6) p.lds_stages = 6;
    const bool ring_fits = p.lds_stages * lds_stage >= LDS_MIN_STAGES * LDS_STAGE_BYTES;    // (the ring also holds the reduction)
    const bool r_fits = p.mask != nullptr ? lds_masked(M, p.r_down) : p.r_down <= 16;       // (the forms that a launch of its own takes too)
    // P = In * Ldown still to be computed (Ldown given): on SM pairs the tiles leave idle when those can take all row
    // blocks (they are then done well before the tiles' contractions are), else by a launch ahead of this one.  Both sum
    // in the same order.  producers(last) = how many pairs would do it when the last wave has `last` items (0: none can).
    const bool want_p = (Ldown != nullptr || plan_only) && p.r_down > 0;
    if (plan_only) { sync = reinterpret_cast<unsigned int*>(sizeof(unsigned int)); split_buf = sync; split_bytes = ~(size_t)0; }   // (never dereferenced)
    const int n_blocks = (M + 15) / 16;
    // Under a mask a producer CTA of several row blocks (48 bytes per row and element instead of 32) has to be through before the first tiles are, or the
    // launch ahead is the shorter way.  Row blocks per CTA and contraction steps at which both were timed, forward, INT4, rank 8 / 16, beside
    // the tiles against ahead: 2 at 8 steps -6 / +4 %, 3 at 18 -15 / -11, 5 at 18 -1 / +5, 5 at 24 -12 / -10, 6 at 24 -7 / -3, 7 at 18 +7 / +12, 7 at 32 -10 / -7.
    auto masked_producers_pay = [&](int n_prod) {
        return p.mask == nullptr || p.steps >= 4 * ((n_blocks + 2 * n_prod - 1) / (2 * n_prod)) + (p.r_down > 8 ? 2 : 0);
    };
    auto producers = [&](int last) {
        // pairs with less to do: no tile at all, or one item fewer than the rest when the last wave is partly filled
        const int idle = p.n_tiles < pairs ? pairs - p.n_tiles : (last ? pairs - last : 0);
        int n_prod = (n_blocks + 3) / 4;                     // four row blocks per producer CTA pair when there is room
        if (n_prod > idle) n_prod = idle;
        const bool fits = want_p && n_prod > 0 && (sync != nullptr || d.r == 0) && r_fits && n_prod * 2 * LDS_MAXB >= n_blocks && ring_fits;
        return fits && masked_producers_pay(n_prod) ? n_prod : 0;
    };
    // A partly filled last wave (more tiles than pairs, at most half a wave left over): each left-over tile goes to two
    // pairs, half of the contraction each, which exchange halves of the result through the workspace -- unless that
    // takes away the idle pairs that would otherwise have computed P beside the tiles (8192 tokens on 4096 x 4096: the
    // down-projection launch it then needs costs what the split wins).  Under a mask the pairs are worth more to the longer product: a short contraction
    // is not split (INT4, rank 8, per cent against neither split nor producers, split / whole: 18 steps, 3000 tokens -> 4096 -1 / -16; 24 steps, 3949 ->
    // 3072 -8 / -15; 32 steps, 2374 -> 4096 -21 / -17).
    constexpr int kMaskedSplitSteps = 28;
    p.n_full = p.n_tiles; p.nsplit = 1; p.split_buf = nullptr;
    const int rem = pair_split_tiles(p.n_tiles, p.steps, pairs);
    if (rem > 0 && sync != nullptr && split_buf != nullptr && (size_t)rem * kSplitTileBytes <= split_bytes &&
        !(p.mask != nullptr && p.steps < kMaskedSplitSteps) && !(want_p && producers(2 * rem) == 0 && producers(p.n_tiles % pairs) > 0)) {
        p.n_full = p.n_tiles - rem; p.nsplit = 2; p.split_buf = static_cast<float4*>(split_buf);
    }
    if (want_p) p.n_prod = producers(p.nsplit > 1 ? 2 * rem : p.n_tiles % pairs);
    // dB on the producers' pass over dY (backward, ranks up to 16): every producer CTA leaves its part in the workspace
    // -- where the producers have a whole tile's time to spare: with a split last wave they are only half a tile ahead of
    // the others, and the extra work then lengthens the kernel (down_proj backward, r = 16: 159 against 140 us)
    const bool db_fits = transposed && p.n_prod > 0 && p.nsplit == 1 && d.r > 0 && d.r <= 16 &&
                         p.n_prod * 2 * (d.r <= 8 ? LDS_MAXB : 3) >= n_blocks;   // (two rank tiles: three row blocks per producer CTA at most)
    if (plan_only) return db_fits ? p.n_prod : 0;
    p.with_db = 0;
    if (db != nullptr && db_fits && db->H != nullptr && db->dB != nullptr && db->part != nullptr &&
        (size_t)2 * p.n_prod * (size_t)T * d.r * sizeof(float) <= db->part_bytes) {
        p.with_db = 1; p.db_accumulate = db->accumulate; p.Hmat = db->H; p.db_part = db->part; p.db_out = db->dB;
        db->done = true;
    }
    CUtensorMap ta, tq, ts, tz;
    if (!make_map_2d(&ta, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, In, (uint64_t)T, (uint64_t)M, 64, (uint32_t)kPairTok, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_2d(&tq, CU_TENSOR_MAP_DATA_TYPE_INT32, 4, Q, (uint64_t)d.N, (uint64_t)(d.K * d.bits / 32), (uint32_t)p.packed_cols, (uint32_t)p.packed_rows, CU_TENSOR_MAP_SWIZZLE_NONE) ||
        !make_map_2d(&ts, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, scales, (uint64_t)d.N, (uint64_t)(d.K / d.group_size), (uint32_t)p.packed_cols, (uint32_t)p.scale_rows, CU_TENSOR_MAP_SWIZZLE_NONE) ||
        !make_map_2d(&tz, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, zeros, (uint64_t)d.N, (uint64_t)(d.K / d.group_size), (uint32_t)p.packed_cols, (uint32_t)p.scale_rows, CU_TENSOR_MAP_SWIZZLE_NONE))
        return QLORA_ERR_CUDA;

    if (want_p && p.n_prod == 0) {
        const int rc = launch_lora_down(M, T, p.r_down, !transposed, In, Ldown, Pmat, st, p.mask, p.out_scale);
        if (rc != QLORA_OK) return rc;
    }
    if ((p.n_prod > 0 && d.r > 0) || p.nsplit > 1) {         // the counters in the workspace are in use: zero them in stream order
        p.sync = sync;
        const int rc = zero_sync_pair(sync, st);
        if (rc != QLORA_OK) return rc;
    }
    const int grid = 2 * (p.n_tiles < pairs ? p.n_tiles + p.n_prod : pairs);
#define QLORA_LAUNCH_PAIR(B)                                                                              \
    return transposed ? launch_pair_impl<B, true>(ta, tq, ts, tz, p, smem_bytes, grid, st)                \
           : p.mask != nullptr && p.n_prod > 0 ? launch_pair_impl<B, false, true>(ta, tq, ts, tz, p, smem_bytes, grid, st) \
                      : launch_pair_impl<B, false>(ta, tq, ts, tz, p, smem_bytes, grid, st)
    switch (d.bits) {
        case 2: QLORA_LAUNCH_PAIR(2);
        case 3: QLORA_LAUNCH_PAIR(3);
        case 4: QLORA_LAUNCH_PAIR(4);
        case 8: QLORA_LAUNCH_PAIR(8);
    }
#undef QLORA_LAUNCH_PAIR
    return QLORA_ERR_UNSUPPORTED;
}

// Between 257 and 1024 tokens either tensor-core kernel may be the faster one: the pair kernel's tiles (512 tokens x 256
// weight rows) leave most SM pairs without one on a 4096-wide layer (42 us against 23 at 512 tokens), but fill a wave
// exactly where the single-CTA kernel's 128 x 256 tiles need two (11008 outputs: 45 against 68 us).  The choice follows
// a small cost model fitted to measurements: waves of tiles times (steps x time per step + fixed part) for each kernel.
// (The constants date from before the single-CTA kernel cut its token tiles in 16s; it has become faster since, so the border lies a
// little too low for it.)
static bool prefer_pair_kernel(const qlora_desc& d, int M, bool transposed) {
    if (M <= 256) return false;
    if (M > 1024) return true;
    const int T = transposed ? d.N : d.K, C = transposed ? d.K : d.N;
    const int steps = T / kStepC, sms = sm_count();
    const int tiles_mid = ((M + 255) / 256) * ((C + kWRows - 1) / kWRows);
    int split = 1;
    for (int sp = 4; sp >= 2; sp /= 2)
        if (tiles_mid * sp <= sms && steps % sp == 0 && steps / sp >= 4) { split = sp; break; }
    const int waves_mid = split > 1 ? 1 : (tiles_mid + sms - 1) / sms;
    const float mid_us = (float)waves_mid * ((float)(steps / split) * 0.29f + 15.0f);
    const int tiles_pair = ((M + 4 * kPairTok - 1) / (4 * kPairTok)) * ((C + 2 * kPairW - 1) / (2 * kPairW));
    const int waves_pair = (tiles_pair + sms / 2 - 1) / (sms / 2);
    const float pair_us = (float)waves_pair * ((float)steps * 0.62f + 4.0f);
    return pair_us < mid_us;
}

// The number of producer pairs on which the backward call of this shape, given its whole workspace, forms dB (on the current
// device: its SM count decides how many pairs the tiles leave idle); 0 when dB goes to the gradient kernels.
int umma_db_on_producers(const qlora_desc& d, int M) {
    if (M <= 256 || d.r == 0 || d.r > 16 || !umma_supported(d, M) || !prefer_pair_kernel(d, M, true)) return 0;
    const int rc = launch_umma_pair(d, M, true, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr,
                                    nullptr, 0, nullptr, true);
    return rc > 0 ? rc : 0;
}

int launch_umma_gemm(const qlora_desc& d, int M, bool transposed, const void* In, const int32_t* Q, const void* scales,
                     const void* zeros, const void* L, float* Pmat, void* Out, cudaStream_t st, const void* Ldown,
                     unsigned int* sync, void* split_buf, size_t split_bytes, DbFuse* db, const DownExtra* extra) {
    if (prefer_pair_kernel(d, M, transposed))
        return launch_umma_pair(d, M, transposed, In, Q, scales, zeros, L, Pmat, Out, st, Ldown, sync, split_buf, split_bytes, db, false, extra);
    if (extra != nullptr && Ldown != nullptr) {              // (not on the single-CTA kernel's spare clusters)
        const int rc = launch_lora_down(M, transposed ? d.N : d.K, extra->only_r > 0 ? extra->only_r : d.r, !transposed, In, Ldown, Pmat, st, extra->mask, extra->out_scale);
        if (rc != QLORA_OK) return rc;
        Ldown = nullptr;
    }
    Params p{};
    p.M = M; p.N = d.N; p.K = d.K; p.bits = d.bits; p.g = d.group_size; p.r = d.r; p.lora_lo = keep_lora_low(d.r, d.group_size); p.r_pad = lora_columns(d.r, d.group_size);
    p.C = transposed ? d.K : d.N;
    const int T = transposed ? d.N : d.K;
    if (!plan_tiles(p, T, transposed, Ldown != nullptr, extra != nullptr, gpu_fit())) return QLORA_ERR_UNSUPPORTED;
    p.s = d.r > 0 ? d.alpha / (float)d.r : 0.f;
    p.Pmat = Pmat; p.L = (const __nv_bfloat16*)L; p.Out = (__nv_bfloat16*)Out;

    const size_t smem_bytes = (size_t)p.off_bar + 512 + 1024;

    CUtensorMap ta, tq, ts, tz, tl{};
    if (!make_map_2d(&ta, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, In, (uint64_t)T, (uint64_t)M, 64, (uint32_t)p.BT, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_2d(&tq, CU_TENSOR_MAP_DATA_TYPE_INT32, 4, Q, (uint64_t)d.N, (uint64_t)(d.K * d.bits / 32), (uint32_t)p.packed_cols, (uint32_t)p.packed_rows, CU_TENSOR_MAP_SWIZZLE_NONE) ||
        !make_map_2d(&ts, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, scales, (uint64_t)d.N, (uint64_t)(d.K / d.group_size), (uint32_t)p.packed_cols, (uint32_t)p.scale_rows, CU_TENSOR_MAP_SWIZZLE_NONE) ||
        !make_map_2d(&tz, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, zeros, (uint64_t)d.N, (uint64_t)(d.K / d.group_size), (uint32_t)p.packed_cols, (uint32_t)p.scale_rows, CU_TENSOR_MAP_SWIZZLE_NONE))
        return QLORA_ERR_CUDA;

    const int grid = p.split > 1 ? p.n_tiles * p.split : (p.n_tiles < sm_count() ? p.n_tiles : sm_count());
    if (p.down_bytes != 0 &&
        !(transposed ? make_map_2d(&tl, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Ldown, (uint64_t)d.r, (uint64_t)T, 8, 64, CU_TENSOR_MAP_SWIZZLE_NONE)
                     : make_map_2d(&tl, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Ldown, (uint64_t)T, (uint64_t)d.r, 64, (uint32_t)d.r, CU_TENSOR_MAP_SWIZZLE_128B)))
        return QLORA_ERR_CUDA;
    p.T = T; p.In = (const __nv_bfloat16*)In; p.Ldown = (const __nv_bfloat16*)Ldown; p.Pout = Pmat; p.wait_limit_us = kWaitLimitUs;
    p.lds_stages = (int)((p.off_bar - LDS_BAR_BYTES) / LDS_STAGE_BYTES);
    if (p.lds_stages > 6) p.lds_stages = 6;
#define QLORA_LAUNCH(B)                                                                              \
    return transposed ? launch_impl<B, true>(ta, tq, ts, tz, tl, p, smem_bytes, grid, st, Ldown, sync)  \
                      : launch_impl<B, false>(ta, tq, ts, tz, tl, p, smem_bytes, grid, st, Ldown, sync)
    switch (d.bits) {
        case 2: QLORA_LAUNCH(2);
        case 3: QLORA_LAUNCH(3);
        case 4: QLORA_LAUNCH(4);
        case 8: QLORA_LAUNCH(8);
    }
#undef QLORA_LAUNCH
    return QLORA_ERR_UNSUPPORTED;
}

namespace {
// The give-up path of the bounded waits, exercised without stalling any real kernel: one thread of one CTA waits with
// the library's own mbar_wait on a barrier in shared memory that nobody ever arrives at, with `limit_us` as the limit.  The
// wait runs out, sets the sticky status word and returns false; the kernel then ends normally (no TMA, no tensor memory).
__global__ void wait_probe_kernel(int limit_us) {
    __shared__ uint64_t bar;
    __shared__ int flag[2];
    if (threadIdx.x == 0) {
        flag[0] = 0; flag[1] = limit_us;
        mbar_init(smem_u32(&bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) (void)mbar_wait(smem_u32(&bar), 0u, flag);
}
}  // namespace

int launch_wait_probe(int limit_us, cudaStream_t st) {
    wait_probe_kernel<<<1, 32, 0, st>>>(limit_us);
    return cudaGetLastError() == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
}

int read_device_status(unsigned int* out, int clear) {
    unsigned int v = 0;
    if (cudaMemcpyFromSymbol(&v, g_device_status, sizeof(v)) != cudaSuccess) return QLORA_ERR_CUDA;
    if (clear && v != 0) {
        const unsigned int zero = 0;
        if (cudaMemcpyToSymbol(g_device_status, &zero, sizeof(zero)) != cudaSuccess) return QLORA_ERR_CUDA;
    }
    *out = v;
    return QLORA_OK;
}

}  // namespace qlora
