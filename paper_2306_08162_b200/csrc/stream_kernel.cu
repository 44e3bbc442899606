// Few-token kernels (M <= 16) of the quantized-linear + LoRA layer, both directions.
//
// With a handful of tokens the layer is bound by reading the packed weights once -- in bytes; in time, by the chain of dependent
// steps of a call (activations arrive, products, exchange of partial sums, store) and by what a thread issues per weight.  So:
//   - a warp loads its packed words straight into registers, 16 bytes per lane, several hundred contraction elements ahead and
//     before the kernel waits for its predecessor in the stream (griddepcontrol.wait); scales and zeros go to shared memory at the
//     same time.  A CTA is 256 threads x 128 registers with at most half an SM's shared memory where the shape allows it, so the
//     CTAs of the NEXT call move in beside those of the current one and have their weights under way when it ends.  Only Q, scales
//     and zeros are touched before the wait: the activations, the adapters (which an optimizer rewrites every step), H / G and the
//     outputs come after it;
//   - the codes go to the warp-level tensor-core instruction (mma.sync m16n8k16, weights as the 16-row operand, tokens as
//     the 8 columns) as RAW integers: a code is ORed into the mantissa of the bf16 constant 128 (one shift + one logic
//     operation per pair of codes), so the operand is 128 + q.  The group scale and the zero-point are applied outside the
//     per-weight path:
//       forward   Y[m,n] = sum_groups s[G,n] * ( sum_{k in G} X[m,k] (128 + q[k,n])  -  (128 + z[G,n]) * sum_{k in G} X[m,k] )
//                 (one accumulator per group segment; the sums of the activations come from the staging pass);
//       backward  dX[m,k] = sum_n dYs[m,n] (128 + q[k,n])  -  sum_n dYs[m,n] (128 + z[G(k),n]),   dYs = bf16(dY[m,n] * s[G(k),n])
//                 (the scale varies along the contraction, so it is folded into a per-group copy of the activation slice,
//                 rounded once to bf16 -- the same relative rounding the dequantised weight would get; the second sum comes from
//                 the staging pass, in fp32).
//     8-bit codes take an fp32 detour (byte -> 2^23 + q -> q -> bf16, exact), offset 0 instead of 128;
//   - backward: the contraction runs across packed columns, so an operand register needs one feature's codes of two columns.  A lane
//     holds the words of the same features for neighbouring columns and merges their halves (one byte permute per eight codes):
//     the register form of the transposition of the packed matrix (Section 3.1, "Implementation Details");
//   - one staging pass after the wait: warps take 32-wide slices of the activations, keep them in the order the products ask for,
//     and feed the LoRA down-projection (H = X A^T, G = dY B, ranks up to 16) from the same registers;
//   - the contraction is split over a cluster of up to 8 CTAs, and inside a CTA over its warps.  A CTA adds its warps' partial sums
//     in order; CTA i of a cluster finishes a slice of the columns: every CTA stores its sums for that slice straight into i's
//     shared memory (distributed shared memory; nothing waits on a remote store), one cluster barrier later i adds them in a fixed
//     order, adds s P L in fp32 and rounds once to bf16.  No workspace, no counters, and the result is the same on every run;
//   - at these sizes a warp has little main loop (two chunks of 128 x 32 weights at 4096 x 4096), so what it issues before and after
//     counts as much: no divisions (the host passes reciprocals and logarithms), loads without per-lane predicates where a whole
//     warp is inside, and only the tokens and ranks that exist are exchanged.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <mutex>

#include "common.cuh"
#include "device_state.h"
#include "launch.h"

namespace qlora {
namespace {

constexpr int ST_WARPS = 8, ST_THREADS = 32 * ST_WARPS;
constexpr int ST_LONG = 16384;                               // contractions up to here are staged whole
constexpr int ST_CHUNK = 128;                                // forward: contraction elements per step of a warp

template <int BITS>
struct Fmt {
    static constexpr float OFF = BITS == 8 ? 0.f : 128.f;   // what the integer operand carries on top of the code
    // forward: a block = KB contraction elements x 32 columns of one warp; lane (g, q) has columns 4g .. 4g+3 of packed row q
    static constexpr int KB = BITS == 2 ? 64 : 32;
    static constexpr int BPC = ST_CHUNK / KB;                // blocks per chunk
    static constexpr int STEPS = KB / 16;                    // k16 MMA steps per block
    static constexpr int NPAIR = 2 * STEPS;                  // bf16 pairs per column and lane
    static constexpr int NLD = (BITS == 3 || BITS == 8) ? 2 : 1;   // 16-byte loads per lane and block
    static constexpr int LPC = BPC * NLD;
    static constexpr int DEPTH = BITS == 2 ? 4 : 2;          // chunks in flight per warp: 32 registers (64 for 3 and 8 bits), 4 KB
};

struct StreamParams {
    int M, K, N, g, r;
    int C;                       // output columns (N forward, K backward)
    int ks, lks;                 // CTAs per cluster = ways the contraction is split, and its log2
    int wc, lwc;                 // warps side by side in a CTA (32 columns forward, 8 FL features backward each), and its log2
    int lwp;                     // log2 of the parts the warps of a CTA split its range of the contraction into (wc << lwp == ST_WARPS)
    int lsl;                     // log2 of the columns a CTA of the cluster finishes
    int pitch;                   // bytes of a staged activation row
    int pass;                    // units of the contraction (128 elements forward, 32 columns backward) a CTA stages at a time
    int range;                   // contraction elements a CTA stages at most
    int ngl;                     // forward: group rows of a CTA's range at most; backward: groups its features span (1 or 2)
    int gd;                      // g / 32, and ceil(2^32 / gd): a group index is a multiplication
    uint32_t gm;
    int fused;                   // H / G is computed here (ranks up to 16) and written to P; else P is an input
    float s;
    const __nv_bfloat16* In;
    const uint32_t* Q;
    const __half* scales;
    const __half* zeros;
    const __nv_bfloat16* Ldown;  // A [r, K] (forward) or B [N, r] (backward): the adapter applied first
    const __nv_bfloat16* Lup;    // B [N, r] (forward) or A [r, K] (backward): the adapter applied second
    float* P;                    // H / G fp32 [M, r]
    __nv_bfloat16* Out;
};

__device__ __forceinline__ uint32_t s_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, int bytes) {   // bytes = 16, or 0 to zero-fill
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// 16 bytes of packed words, kept in program order with griddepcontrol.wait.
__device__ __forceinline__ void ldg_words(uint4& v, const uint32_t* src) {
    asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(src));
}
// Shared memory, where `ok`; otherwise the registers keep what they hold.
__device__ __forceinline__ void lds16(uint32_t& a, uint32_t& b, uint32_t& c, uint32_t& d, uint32_t addr, bool ok) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t@p ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];\n\t}"
                 : "+r"(a), "+r"(b), "+r"(c), "+r"(d) : "r"(addr), "r"((uint32_t)ok) : "memory");
}
__device__ __forceinline__ void lds8(uint32_t& a, uint32_t& b, uint32_t addr, bool ok) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p ld.shared.v2.u32 {%0, %1}, [%2];\n\t}"
                 : "+r"(a), "+r"(b) : "r"(addr), "r"((uint32_t)ok) : "memory");
}
// Group of the u-th 32 rows along k (u < 2^16, gd < 2^16: exact).
__device__ __forceinline__ int st_group(const StreamParams& p, int u) { return p.gd == 1 ? u : (int)__umulhi((uint32_t)u, p.gm); }
__device__ __forceinline__ uint4 ldg16(const void* src, bool ok) {      // plain global load, zero without `ok`
    return ok ? *reinterpret_cast<const uint4*>(src) : make_uint4(0, 0, 0, 0);
}
__device__ __forceinline__ uint32_t ldg32(const void* p) { return *reinterpret_cast<const uint32_t*>(p); }
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

__device__ __forceinline__ uint32_t st_cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t st_map(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void st_cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void st_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void st_mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t st_movm(uint32_t a) {
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}
__device__ __forceinline__ uint32_t st_comp(const uint4& v, int i) { return i == 0 ? v.x : (i == 1 ? v.y : (i == 2 ? v.z : v.w)); }
__device__ __forceinline__ uint32_t st_pack(float a, float b) {
    const __nv_bfloat162 pr = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&pr);
}
__device__ __forceinline__ float st_byte(uint32_t w, int j) {            // byte j as fp32, exact
    return __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7540 + j)) - 8388608.f;
}

// One column's codes of this lane -> bf16 pairs holding OFF + q.  With c_0 .. c_{n-1} the lane's codes in contraction order:
//   2-bit (16 codes): p[t] = (c_t, c_{t+8}), t < 8        3- and 4-bit (8 codes): p[t] = (c_t, c_{t+4}), t < 4
//   8-bit (row q: c_0..3, row q + 4: c_4..7): p = (c_0,c_1), (c_2,c_3), (c_4,c_5), (c_6,c_7)
// (3-bit: w0, w1 are the rows of stream bits 24 q and 24 q + 23 of the block.)
template <int BITS>
__device__ __forceinline__ void st_unpack(uint32_t w0, uint32_t w1, int q, uint32_t (&p)[Fmt<BITS>::NPAIR]) {
    if constexpr (BITS == 4) {
#pragma unroll
        for (int t = 0; t < 4; ++t) p[t] = ((w0 >> (4 * t)) & 0x000F000Fu) | 0x43004300u;
    } else if constexpr (BITS == 2) {
#pragma unroll
        for (int t = 0; t < 8; ++t) p[t] = ((w0 >> (2 * t)) & 0x00030003u) | 0x43004300u;
    } else if constexpr (BITS == 3) {
        const uint32_t v = __funnelshift_r(w0, w1, (24 * q) & 31);        // codes at bits 3 j, j < 8
        const uint32_t m = (v & 0x0000FFFFu) | ((v << 4) & 0xFFFF0000u);  // codes 0..3 at bits 3 j, codes 4..7 at 16 + 3 j
#pragma unroll
        for (int t = 0; t < 4; ++t) p[t] = ((m >> (3 * t)) & 0x00070007u) | 0x43004300u;
    } else {
        p[0] = st_pack(st_byte(w0, 0), st_byte(w0, 1)); p[1] = st_pack(st_byte(w0, 2), st_byte(w0, 3));
        p[2] = st_pack(st_byte(w1, 0), st_byte(w1, 1)); p[3] = st_pack(st_byte(w1, 2), st_byte(w1, 3));
    }
}

__device__ __forceinline__ float st_sum8(const uint4& v) {
    return ((bf16_lo(v.x) + bf16_hi(v.x)) + (bf16_lo(v.y) + bf16_hi(v.y))) + ((bf16_lo(v.z) + bf16_hi(v.z)) + (bf16_lo(v.w) + bf16_hi(v.w)));
}
__device__ __forceinline__ float st_quad_sum(float v) {
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// ---- shared memory ------------------------------------------------------------------------------------------------------
// Everything but the staged activations (which come first) and the staged group parameters (second):
//   sums   forward: [range / 32][TOKS] sums of 32 activations;  backward: [ST_WARPS][2][16] zero-point sums
//   hp     [ST_WARPS][M][16] the warps' parts of H / G (16 ranks)   hfull  [M][16 or r] the whole of it
//   lup    this CTA's slice of the second adapter
//   part   [parts][M][tile_c] the warps' partial sums
//   recv_h [ks][M][16], recv [ks][M][sl]: what the CTAs of the cluster send this one
struct SmemPlan { uint32_t sz, sums, hp, hfull, lup, recv_h, part, recv, total; };
__host__ __device__ inline SmemPlan st_plan(const StreamParams& p, bool transposed, int toks, int tile_c) {
    SmemPlan s;
    const uint32_t rows = (uint32_t)p.M * (transposed ? (uint32_t)p.ngl : 1u);
    s.sz = (rows * (uint32_t)p.pitch + 127u) / 128u * 128u;
    s.sums = s.sz + (transposed ? 4u * (uint32_t)p.ngl * (uint32_t)p.range : 4u * (uint32_t)p.ngl * (uint32_t)tile_c);
    s.hp = s.sums + (transposed ? ST_WARPS * 128u : (uint32_t)(p.range / 32 * toks) * 4u);
    s.hfull = s.hp + (p.fused ? ST_WARPS * 64u * (uint32_t)p.M : 0u);
    s.lup = s.hfull + (p.r > 0 ? (uint32_t)(p.r < 16 ? 16 : p.r) * 4u * (uint32_t)p.M : 0u);
    s.recv_h = s.lup + (((uint32_t)(p.r * 2) << p.lsl) + 15u) / 16u * 16u;
    s.part = s.recv_h + (p.fused ? (uint32_t)p.ks * 64u * (uint32_t)p.M : 0u);
    s.recv = s.part + ((uint32_t)(p.M * tile_c * 4) << p.lwp);
    s.total = s.recv + (p.ks > 1 ? (uint32_t)(p.M * tile_c * 4) : 0u);
    return s;
}

// A warp's partial H / G tile (MMA accumulator layout: rows = ranks, columns = tokens) -> its slot of hp.
// `add`: on top of what the slot holds (a later pass).
template <int NT>
__device__ __forceinline__ void st_store_hp(const StreamParams& p, const float (&ah)[NT][4], float* hp, int warp, int g, int q, bool add) {
    float* mine = hp + warp * 16 * p.M + g;
#pragma unroll
    for (int tt = 0; tt < NT; ++tt)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int tok = 8 * tt + 2 * q + e;
            if (tok < p.M) {
                mine[tok * 16] = ah[tt][e] + (add ? mine[tok * 16] : 0.f);
                mine[tok * 16 + 8] = ah[tt][2 + e] + (add ? mine[tok * 16 + 8] : 0.f);
            }
        }
}

// The CTA's part of H / G: the warps' parts added in order, sent to every CTA of the cluster.
__device__ __forceinline__ void st_share_h(const StreamParams& p, const float* hp, uint32_t recv_h_addr, int rank) {
    const int n = 16 * p.M;
    if ((int)threadIdx.x < n) {
        float h = 0.f;
#pragma unroll
        for (int w = 0; w < ST_WARPS; ++w) h += hp[w * n + threadIdx.x];
#pragma unroll 1
        for (int peer = 0; peer < p.ks; ++peer)
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(st_map(recv_h_addr + (uint32_t)(rank * n + (int)threadIdx.x) * 4u, (uint32_t)peer)), "f"(h) : "memory");
    }
}

// This CTA's slice of the second adapter, and H / G where it is an input.  After griddepcontrol.wait.
template <bool TRANSPOSED>
__device__ __forceinline__ void st_stage_lup(const StreamParams& p, uint8_t* lup, float* hfull, int c_lo) {
    if (p.r == 0) return;
    const int tid = threadIdx.x;
    if (TRANSPOSED) {                                     // A [r, K]: [r][sl]
        const int lc8 = p.lsl - 3;                        // log2 of the 16-byte pieces per rank
        for (int e = tid; e < p.r << lc8; e += ST_THREADS) {
            const int j = e >> lc8, col = c_lo + 8 * (e & ((1 << lc8) - 1));
            cp16(s_u32(lup) + e * 16, col < p.K ? p.Lup + (size_t)j * p.K + col : p.Lup, col < p.K ? 16 : 0);
        }
    } else {                                              // B [N, r]: [sl][r], contiguous
        const int pieces = ((1 << p.lsl) * p.r) >> 3, valid = max(0, p.N - c_lo) * p.r >> 3;
        for (int e = tid; e < pieces; e += ST_THREADS)
            cp16(s_u32(lup) + e * 16, e < valid ? p.Lup + (size_t)c_lo * p.r + 8 * e : p.Lup, e < valid ? 16 : 0);
    }
    if (!p.fused)
        for (int e = tid; e < p.M * p.r; e += ST_THREADS) hfull[e] = p.P[e];
}

// The end of a call, once the warps' partial sums are in `part`: the CTA's sums go to the owners of their columns, one cluster
// barrier later the owner adds them (CTA by CTA, in order), adds s P L, stores bf16.  A CTA alone adds its warps' parts directly.
template <bool TRANSPOSED>
__device__ __forceinline__ void st_finish(const StreamParams& p, uint8_t* smem, const SmemPlan& sp, int c_lo, int rank, bool writes_p) {
    const int tid = threadIdx.x, sl = 1 << p.lsl;
    const float* src = reinterpret_cast<const float*>(smem + sp.part);
    const float* recv_h = reinterpret_cast<const float*>(smem + sp.recv_h);
    float* hfull = reinterpret_cast<float*>(smem + sp.hfull);
    const __nv_bfloat16* lup = reinterpret_cast<const __nv_bfloat16*>(smem + sp.lup);
    int nsrc = 1 << p.lwp;
    __syncthreads();
    if (p.ks > 1) {
        const int ltc = p.lsl + p.lks;                    // log2 of the tile's columns
        const uint32_t recv_addr = s_u32(smem + sp.recv);
#pragma unroll 1
        for (int e = tid; e < p.M << (ltc - 2); e += ST_THREADS) {
            const int c = 4 * (e & ((1 << (ltc - 2)) - 1)), tok = e >> (ltc - 2);
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
            for (int i = 0; i < nsrc; ++i) {
                const float4 x = *reinterpret_cast<const float4*>(src + (((i * p.M + tok) << ltc) + c));
                v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
            }
            const uint32_t off = (uint32_t)(((rank * p.M + tok) << p.lsl) + (c & (sl - 1))) * 4u;
            asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(st_map(recv_addr + off, (uint32_t)(c >> p.lsl))), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
        }
        src = reinterpret_cast<const float*>(smem + sp.recv);
        nsrc = p.ks;
        st_cluster_sync();                                // every CTA's stores into this CTA's shared memory are visible
    }
    const int hs = p.fused ? 16 : p.r;                    // ranks per row of hfull
    if (p.fused) {
        const int n = 16 * p.M;
        if (tid < n) {
            float h = 0.f;
#pragma unroll 4
            for (int rk = 0; rk < p.ks; ++rk) h += recv_h[rk * n + tid];
            hfull[tid] = h;
            const int tok = tid >> 4, j = tid & 15;
            if (writes_p && j < p.r) p.P[(size_t)tok * p.r + j] = h;
        }
        __syncthreads();
    }
#pragma unroll 1
    for (int e = tid; e < p.M << (p.lsl - 1); e += ST_THREADS) {          // two columns per thread
        const int c = 2 * (e & ((sl >> 1) - 1)), tok = e >> (p.lsl - 1), col = c_lo + c;
        float v0 = 0.f, v1 = 0.f, l0 = 0.f, l1 = 0.f;
#pragma unroll 4
        for (int i = 0; i < nsrc; ++i) {
            const float2 x = *reinterpret_cast<const float2*>(src + (((i * p.M + tok) << p.lsl) + c));
            v0 += x.x; v1 += x.y;
        }
#pragma unroll 4
        for (int j = 0; j < p.r; ++j) {
            const float h = hfull[tok * hs + j];
            l0 = fmaf(h, __bfloat162float(TRANSPOSED ? lup[j * sl + c] : lup[c * p.r + j]), l0);
            l1 = fmaf(h, __bfloat162float(TRANSPOSED ? lup[j * sl + c + 1] : lup[(c + 1) * p.r + j]), l1);
        }
        if (p.r > 0) { v0 += p.s * l0; v1 += p.s * l1; }
        if (col < p.C) *reinterpret_cast<uint32_t*>(p.Out + (size_t)tok * p.C + col) = st_pack(v0, v1);   // (C is a multiple of 8)
    }
}

// ------------------------------------------------------------------------------------------------------------
// Forward: Y = X W^T + s H B^T.  CTA (rank, tile): columns [32 wc tile, + 32 wc), contraction chunks [c0, c1) of 128 elements.
// Warp (cg, part): 32 columns and its share of the chunks.  GPC: scale segments per chunk -- 1 for groups that are multiples of
// 128, 2 for multiples of 64, 4 for multiples of 32 (the segment, not the group, is what one accumulator spans).
// MULTI: a contraction whose activations do not fit the shared memory; staging and products take p.pass chunks at a time in turn.
// ------------------------------------------------------------------------------------------------------------
template <int BITS, int NT, int GPC, int PER_SM, bool MULTI>
__global__ void __launch_bounds__(ST_THREADS, PER_SM) stream_fwd_kernel(const StreamParams p) {
    using F = Fmt<BITS>;
    constexpr int TOKS = 8 * NT, SB = 2;                   // SB: slices of the staging pass whose loads a warp has in flight
    pdl_launch_dependents();
    if (p.ks > 1) st_cluster_arrive_relaxed();             // waited for before the first store into a peer's shared memory
    extern __shared__ __align__(128) uint8_t smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, q = lane & 3;
    const int tile_c = 32 * p.wc, cg = warp & (p.wc - 1), part = warp >> p.lwc;
    const int rank = p.ks > 1 ? (int)st_cluster_rank() : 0;
    const int tile_c0 = (int)blockIdx.y * tile_c, c_lo = tile_c0 + (rank << p.lsl);
    const int nch = (p.K + ST_CHUNK - 1) / ST_CHUNK;
    const int c0 = (nch * rank) >> p.lks, c1 = (nch * (rank + 1)) >> p.lks;
    int p0 = c0, p1 = MULTI ? min(c1, c0 + p.pass) : c1;   // the chunks of this pass, and this warp's share of them
    int w0 = p0 + (((p1 - p0) * part) >> p.lwp), w1 = p0 + (((p1 - p0) * (part + 1)) >> p.lwp);
    const SmemPlan sp = st_plan(p, false, TOKS, tile_c);
    uint8_t* xs = smem;                                    // [M][pitch] activations in fragment order
    const __half* sz = reinterpret_cast<const __half*>(smem + sp.sz);       // [group][scales, zeros][tile_c]
    float* xsum = reinterpret_cast<float*>(smem + sp.sums);                 // [slice of 32][TOKS]
    float* hp = reinterpret_cast<float*>(smem + sp.hp);
    float* hfull = reinterpret_cast<float*>(smem + sp.hfull);

    // ---- frozen weights only: in flight while the predecessor finishes ----
    const int rows_total = p.K * BITS / 32;
    const int row_a = BITS == 3 ? (24 * q) >> 5 : q, row_b = BITS == 3 ? (24 * q + 23) >> 5 : q + 4;   // of a block
    const int col = tile_c0 + 32 * cg + 4 * g;
    const uint32_t* qcol = p.Q + (col < p.N ? col : 0);    // (a column beyond the last loads another one's words and is dropped)
    auto load_chunk = [&](uint4 (&w)[F::LPC], int ch) {
        if (ch >= w1) return;
        const int r0 = ch * (4 * BITS), last = rows_total - 1;
        const bool full = (ch + 1) * ST_CHUNK <= p.K;       // (rows beyond the last: any words will do, their activations are zero)
#pragma unroll
        for (int b = 0; b < F::BPC; ++b) {
            int ra = r0 + b * (F::KB * BITS / 32) + row_a;
            if (!full) ra = min(ra, last);
            ldg_words(w[b * F::NLD], qcol + (size_t)ra * p.N);
            if constexpr (F::NLD == 2) {
                int rb = r0 + b * (F::KB * BITS / 32) + row_b;
                if (!full) rb = min(rb, last);
                ldg_words(w[b * F::NLD + 1], qcol + (size_t)rb * p.N);
            }
        }
    };
    uint4 w[F::DEPTH][F::LPC];
#pragma unroll
    for (int d = 0; d < F::DEPTH; ++d) load_chunk(w[d], w0 + d);
    int g_first = 0;
    auto load_sz = [&]() {
        g_first = st_group(p, p0 * (ST_CHUNK / 32));
        const int g_last = p1 > p0 ? st_group(p, min(p1 * (ST_CHUNK / 32), p.K >> 5) - 1) : g_first - 1;
        const int lper = p.lwc + 2, n = (g_last - g_first + 1) << (lper + 1);             // 16-byte pieces
        for (int e = tid; e < n; e += ST_THREADS) {
            const int row = e >> lper, c = tile_c0 + 8 * (e & ((1 << lper) - 1));
            const __half* src = ((row & 1) ? p.zeros : p.scales) + (size_t)(g_first + (row >> 1)) * p.N + c;
            cp16(s_u32(sz) + e * 16, c < p.N ? src : p.scales, c < p.N ? 16 : 0);
        }
    };
    load_sz();
    constexpr int SEG_K = ST_CHUNK / GPC, SEG_B = F::BPC / GPC;             // contraction elements and blocks of a segment
    const int spg = p.gd / (SEG_K / 32);                                    // segments per group
    int gpos = 0;
    const __half* sz_lane = nullptr;
    int k_lo = 0, n_slices = 0, n_valid = 0;
    auto set_pass = [&]() {
        const int g_w0 = st_group(p, w0 * (ST_CHUNK / 32));
        gpos = w0 * GPC - g_w0 * spg;
        sz_lane = sz + (g_w0 - g_first) * 2 * tile_c + 32 * cg + 4 * g;
        k_lo = p0 * ST_CHUNK; n_slices = (p1 - p0) * (ST_CHUNK / 32); n_valid = min(n_slices, (p.K - k_lo) >> 5);
    };
    set_pass();
    {   // ask the lines this CTA will read right after the wait into L2 (nothing is read into the SM): its slices of X, A and B
        const int rows = p.M + (p.fused ? p.r : 0);
        for (int j = warp; j < rows; j += ST_WARPS) {
            const __nv_bfloat16* base = (j < p.M ? p.In + (size_t)j * p.K : p.Ldown + (size_t)(j - p.M) * p.K) + k_lo;
            for (int l = lane; 2 * l < n_valid; l += 32) prefetch_l2(base + 64 * l);
        }
        if (tid * 64 < min(1 << p.lsl, p.N - c_lo) * p.r) prefetch_l2(p.Lup + (size_t)c_lo * p.r + tid * 64);
    }

    pdl_wait();

    const bool tok_ok[2] = {g < p.M, g + 8 < p.M};
    const uint32_t recv_h_addr = s_u32(smem + sp.recv_h);
    float acc[2][NT][4];
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int tt = 0; tt < NT; ++tt) acc[u][tt][0] = acc[u][tt][1] = acc[u][tt][2] = acc[u][tt][3] = 0.f;
#pragma unroll 1
    do {
    // ---- staging: activations into fragment order, their sums, and this CTA's part of H = X A^T ----
    const bool again = MULTI && p0 > c0;
    if (again) {
        __syncthreads();                                   // every warp is done with the pass before
        load_sz();
        set_pass();
    }
    {
        bool first = !again;                               // (every warp stages its share of the second adapter once)
        float hacc[NT][4];
#pragma unroll
        for (int tt = 0; tt < NT; ++tt) hacc[tt][0] = hacc[tt][1] = hacc[tt][2] = hacc[tt][3] = 0.f;
        const __nv_bfloat16* xr = p.In + (size_t)g * p.K + k_lo + 8 * q;
        const __nv_bfloat16* ar = p.Ldown + (size_t)g * p.K + k_lo + 8 * q;
        const bool a_lo = p.fused && g < p.r, a_hi = p.fused && g + 8 < p.r;
#pragma unroll 1
        for (int s0 = warp; s0 < n_slices || first; s0 += SB * ST_WARPS) {
            uint4 xv[SB][NT], al[SB], ah[SB];
#pragma unroll
            for (int s = 0; s < SB; ++s) {
                const int sl = s0 + s * ST_WARPS;
                const bool in = sl < n_valid;              // (slices of a last chunk that is not full are zero)
#pragma unroll
                for (int tt = 0; tt < NT; ++tt) xv[s][tt] = ldg16(xr + 8 * tt * (size_t)p.K + 32 * sl, in && tok_ok[tt]);
                al[s] = ldg16(ar + 32 * sl, in && a_lo);
                ah[s] = ldg16(ar + 8 * (size_t)p.K + 32 * sl, in && a_hi);
            }
            if (first) st_stage_lup<false>(p, smem + sp.lup, hfull, c_lo);   // (with the first loads on their way)
            first = false;
#pragma unroll
            for (int s = 0; s < SB; ++s) {
                const int sl = s0 + s * ST_WARPS;
                if (sl >= n_slices) break;
#pragma unroll
                for (int tt = 0; tt < NT; ++tt) {
                    const uint4 v = xv[s][tt];
                    st_mma(hacc[tt], al[s].x, ah[s].x, al[s].y, ah[s].y, v.x, v.y);
                    st_mma(hacc[tt], al[s].z, ah[s].z, al[s].w, ah[s].w, v.z, v.w);
                    const float sum = st_quad_sum(st_sum8(v));
                    if (q == 0) xsum[sl * TOKS + 8 * tt + g] = sum;
                    uint4 o;
                    if constexpr (BITS == 2) {             // (x0,x8) (x1,x9) ... (x7,x15) of 16 elements = two lanes
                        const uint32_t s0v = (q & 1) ? v.x : v.z, s1v = (q & 1) ? v.y : v.w;
                        const uint32_t r0v = __shfl_xor_sync(0xffffffffu, s0v, 1), r1v = __shfl_xor_sync(0xffffffffu, s1v, 1);
                        const uint32_t a0 = (q & 1) ? r0v : v.x, a1 = (q & 1) ? r1v : v.y, b0 = (q & 1) ? v.z : r0v, b1 = (q & 1) ? v.w : r1v;
                        o = make_uint4(__byte_perm(a0, b0, 0x5410), __byte_perm(a0, b0, 0x7632), __byte_perm(a1, b1, 0x5410), __byte_perm(a1, b1, 0x7632));
                    } else if constexpr (BITS == 8) {
                        o = v;
                    } else {                               // (x0,x4) (x1,x5) (x2,x6) (x3,x7)
                        o = make_uint4(__byte_perm(v.x, v.z, 0x5410), __byte_perm(v.x, v.z, 0x7632), __byte_perm(v.y, v.w, 0x5410), __byte_perm(v.y, v.w, 0x7632));
                    }
                    if (tok_ok[tt]) *reinterpret_cast<uint4*>(xs + (g + 8 * tt) * p.pitch + sl * 64 + q * 16) = o;
                }
            }
        }
        if (p.fused) st_store_hp<NT>(p, hacc, hp, warp, g, q, again);
    }
    cp_wait_all();
    __syncthreads();
    if (!MULTI || p1 == c1) {
        if (p.ks > 1) st_cluster_wait();                   // every CTA of the cluster is running: its shared memory may be written
        if (p.fused) st_share_h(p, hp, recv_h_addr, rank);
    }

    // ---- main loop ----
    const uint32_t xl = s_u32(xs) + (uint32_t)(g * p.pitch + q * (BITS == 2 ? 32 : (BITS == 8 ? 8 : 16)));
    uint32_t xf[NT][F::NPAIR];                             // activation fragments: token g (+ 8), this lane's quarter of a block
#pragma unroll
    for (int tt = 0; tt < NT; ++tt)
#pragma unroll
        for (int i = 0; i < F::NPAIR; ++i) xf[tt][i] = 0u; // (stays zero for tokens that do not exist)
    auto compute = [&](const uint4 (&wd)[F::LPC], int ch) {
        const uint32_t xc = xl + (uint32_t)(ch - p0) * (ST_CHUNK * 2);
        const float* sumc = xsum + (ch - p0) * (ST_CHUNK / 32) * TOKS + 2 * q;
#pragma unroll
        for (int sg = 0; sg < GPC; ++sg) {
            if (GPC > 1 && ch * ST_CHUNK + sg * SEG_K >= p.K) break;        // (a last chunk that is not full: no such group)
            float grp[2][NT][4];
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int tt = 0; tt < NT; ++tt) grp[u][tt][0] = grp[u][tt][1] = grp[u][tt][2] = grp[u][tt][3] = 0.f;
#pragma unroll
            for (int bs = 0; bs < SEG_B; ++bs) {
                const int b = sg * SEG_B + bs;
#pragma unroll
                for (int tt = 0; tt < NT; ++tt) {
                    const uint32_t x = xc + (uint32_t)(8 * tt * p.pitch + b * (F::KB * 2));
                    if constexpr (BITS == 8) {
                        lds8(xf[tt][0], xf[tt][1], x, tok_ok[tt]);
                        lds8(xf[tt][2], xf[tt][3], x + 32, tok_ok[tt]);
                    } else {
#pragma unroll
                        for (int h = 0; h < F::NPAIR / 4; ++h) lds16(xf[tt][4 * h], xf[tt][4 * h + 1], xf[tt][4 * h + 2], xf[tt][4 * h + 3], x + 16 * h, tok_ok[tt]);
                    }
                }
                uint32_t pc[4][F::NPAIR];                  // [column i of the lane's four][pair]
#pragma unroll
                for (int i = 0; i < 4; ++i) st_unpack<BITS>(st_comp(wd[b * F::NLD], i), F::NLD > 1 ? st_comp(wd[b * F::NLD + F::NLD - 1], i) : 0u, q, pc[i]);
                // two tiles of 16 columns: rows g / g + 8 of tile u are columns 4g + 2u / 4g + 2u + 1
#pragma unroll
                for (int s = 0; s < F::STEPS; ++s)
#pragma unroll
                    for (int u = 0; u < 2; ++u)
#pragma unroll
                        for (int tt = 0; tt < NT; ++tt)
                            st_mma(grp[u][tt], pc[2 * u][2 * s], pc[2 * u + 1][2 * s], pc[2 * u][2 * s + 1], pc[2 * u + 1][2 * s + 1], xf[tt][2 * s], xf[tt][2 * s + 1]);
            }
            // end of a segment: scale, correct for offset and zero-point
            const uint2 s2 = *reinterpret_cast<const uint2*>(sz_lane), z2 = *reinterpret_cast<const uint2*>(sz_lane + tile_c);
            const float2 sa = __half22float2(*reinterpret_cast<const __half2*>(&s2.x)), sb = __half22float2(*reinterpret_cast<const __half2*>(&s2.y));
            const float2 za = __half22float2(*reinterpret_cast<const __half2*>(&z2.x)), zb = __half22float2(*reinterpret_cast<const __half2*>(&z2.y));
            const float sc[4] = {sa.x, sa.y, sb.x, sb.y};
            const float oz[4] = {F::OFF + za.x, F::OFF + za.y, F::OFF + zb.x, F::OFF + zb.y};
#pragma unroll
            for (int tt = 0; tt < NT; ++tt) {
                float sx0 = 0.f, sx1 = 0.f;
#pragma unroll
                for (int i = 0; i < SEG_K / 32; ++i) {
                    const float2 v = *reinterpret_cast<const float2*>(sumc + (sg * (SEG_K / 32) + i) * TOKS + 8 * tt);
                    sx0 += v.x; sx1 += v.y;
                }
#pragma unroll
                for (int u = 0; u < 2; ++u)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        acc[u][tt][2 * h] = fmaf(sc[2 * u + h], fmaf(-oz[2 * u + h], sx0, grp[u][tt][2 * h]), acc[u][tt][2 * h]);
                        acc[u][tt][2 * h + 1] = fmaf(sc[2 * u + h], fmaf(-oz[2 * u + h], sx1, grp[u][tt][2 * h + 1]), acc[u][tt][2 * h + 1]);
                    }
            }
            if (++gpos == spg) { gpos = 0; sz_lane += 2 * tile_c; }
        }
    };
#pragma unroll 1
    for (int ch = w0; ch < w1; ch += F::DEPTH) {
#pragma unroll
        for (int d = 0; d < F::DEPTH; ++d) {
            if (ch + d < w1) {
                compute(w[d], ch + d);
                load_chunk(w[d], ch + d + F::DEPTH);
            }
        }
    }
    if (!MULTI || p1 == c1) break;
    p0 = p1; p1 = min(c1, p0 + p.pass);
    w0 = p0 + (((p1 - p0) * part) >> p.lwp); w1 = p0 + (((p1 - p0) * (part + 1)) >> p.lwp);
#pragma unroll
    for (int d = 0; d < F::DEPTH; ++d) load_chunk(w[d], w0 + d);
    } while (true);
    // accumulator element (u, tt, e): column 4g + 2u + (e >> 1) of this warp's 32, token 2q + (e & 1) + 8 tt
    float* mine = reinterpret_cast<float*>(smem + sp.part) + part * p.M * tile_c + 32 * cg + 4 * g;
#pragma unroll
    for (int tt = 0; tt < NT; ++tt)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int tok = 8 * tt + 2 * q + e;
            if (tok < p.M) *reinterpret_cast<float4*>(mine + tok * tile_c) = make_float4(acc[0][tt][e], acc[0][tt][2 + e], acc[1][tt][e], acc[1][tt][2 + e]);
        }
    st_finish<false>(p, smem, sp, c_lo, rank, blockIdx.y == 0 && rank == 0);
}

// ------------------------------------------------------------------------------------------------------------
// Backward: dX = dY W + s G A.  CTA (rank, tile): output features [8 FL wc tile, + 8 FL wc), contraction units [u0, u1) of 32
// packed columns.  Warp (fw, part): 8 FL features (all inside one group) and its share of the units.  Lane (g, q) has features
// FL g .. FL g + FL - 1 of the warp's, columns 4q .. 4q+3 (+ 16) of a unit.  FL = 8, or 4 where groups are not multiples of 64.
// MULTI as forward.
// ------------------------------------------------------------------------------------------------------------
template <int BITS, int FL>
struct BFmt {
    static constexpr int NLD = (BITS == 3 || (BITS == 8 && FL == 8)) ? 2 : 1;   // packed rows a lane reads per column
    static constexpr int DEPTH = 4;                                             // units in flight per warp: 32 or 64 registers, 4 KB
};

// FL features of two neighbouring columns (words a0 / a1 and b0 / b1) -> pairs (column a, column b) of OFF + q per feature.
template <int BITS, int FL>
__device__ __forceinline__ void st_bwd_pairs(uint32_t a0, uint32_t a1, uint32_t b0, uint32_t b1, uint32_t sh, uint32_t sel, uint32_t (&p)[FL]) {
    if constexpr (BITS == 8) {
#pragma unroll
        for (int t = 0; t < FL; ++t) p[t] = st_pack(st_byte(t < 4 ? a0 : a1, t & 3), st_byte(t < 4 ? b0 : b1, t & 3));
    } else {
        constexpr uint32_t M2 = BITS == 2 ? 0x00030003u : (BITS == 3 ? 0x00070007u : 0x000F000Fu);
        uint32_t x, y = 0u;
        if constexpr (BITS == 3) {
            const uint32_t va = __funnelshift_r(a0, a1, sh), vb = __funnelshift_r(b0, b1, sh);
            x = __byte_perm(va, vb, 0x5410);
            if constexpr (FL == 8) y = __byte_perm(va >> 12, vb >> 12, 0x5410);
        } else {
            x = __byte_perm(a0, b0, sel);
            if constexpr (BITS == 4 && FL == 8) y = __byte_perm(a0, b0, 0x7632);
        }
        constexpr int IN_X = BITS == 2 ? 8 : 4;
#pragma unroll
        for (int t = 0; t < FL; ++t) p[t] = (((t < IN_X ? x : y) >> (BITS * (t % IN_X))) & M2) | 0x43004300u;
    }
}

template <int BITS, int NT, int FL, int PER_SM, bool MULTI>
__global__ void __launch_bounds__(ST_THREADS, PER_SM) stream_bwd_kernel(const StreamParams p) {
    using F = Fmt<BITS>;
    using BF = BFmt<BITS, FL>;
    constexpr int TOKS = 8 * NT, SB = MULTI && NT == 1 ? 4 : 2;   // SB: as forward
    pdl_launch_dependents();
    if (p.ks > 1) st_cluster_arrive_relaxed();             // waited for before the first store into a peer's shared memory
    extern __shared__ __align__(128) uint8_t smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, q = lane & 3;
    const int tile_c = 8 * FL * p.wc, fw = warp & (p.wc - 1), part = warp >> p.lwc;
    const int rank = p.ks > 1 ? (int)st_cluster_rank() : 0;
    const int tile_f0 = (int)blockIdx.y * tile_c, c_lo = tile_f0 + (rank << p.lsl), f0 = tile_f0 + 8 * FL * fw;
    const int nun = (p.N + 31) >> 5;
    const int u0 = (nun * rank) >> p.lks, u1 = (nun * (rank + 1)) >> p.lks;
    int p0 = u0, p1 = MULTI ? min(u1, u0 + p.pass) : u1;   // the units of this pass, and this warp's share of them
    int w0 = p0 + (((p1 - p0) * part) >> p.lwp), w1 = p0 + (((p1 - p0) * (part + 1)) >> p.lwp);
    const int gk0 = st_group(p, tile_f0 >> 5), ngroups = st_group(p, p.K >> 5);    // group of the CTA's first feature
    const int copy = min(st_group(p, f0 >> 5) - gk0, p.ngl - 1);
    const SmemPlan sp = st_plan(p, true, TOKS, tile_c);
    uint8_t* ys = smem;                                    // [groups][M][pitch] scaled slices of dY
    const __half* sz = reinterpret_cast<const __half*>(smem + sp.sz);       // [group][scales, zeros][range]
    float* zp = reinterpret_cast<float*>(smem + sp.sums);                   // [ST_WARPS][2][16] zero-point sums, per warp
    float* hp = reinterpret_cast<float*>(smem + sp.hp);
    float* hfull = reinterpret_cast<float*>(smem + sp.hfull);

    // ---- frozen weights only: in flight while the predecessor finishes ----
    const int bitpos = FL * BITS * g, row = f0 * BITS / 32 + (bitpos >> 5);
    const uint32_t sh = (uint32_t)bitpos & 31u;
    const uint32_t byte = sh >> 3;
    const uint32_t sel = BITS == 2 && FL == 4 ? byte * 0x0011u + (byte + 4u) * 0x1100u : (sh ? 0x7632u : 0x5410u);
    const int rows_total = p.K * BITS / 32;
    // (rows and columns beyond the last load other words: their results are dropped, their activations are zero)
    const int row2 = BITS == 8 || (int)sh + FL * BITS > 32 ? row + 1 : row;
    const uint32_t* qrow = p.Q + (size_t)min(row, rows_total - 1) * p.N;
    const uint32_t* qrow2 = p.Q + (size_t)min(row2, rows_total - 1) * p.N;
    auto load_unit = [&](uint4 (&w)[2 * BF::NLD], int un) {
        if (un >= w1) return;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int n = min(32 * un + 16 * h + 4 * q, p.N - 4);
            ldg_words(w[h * BF::NLD], qrow + n);
            if constexpr (BF::NLD == 2) ldg_words(w[h * BF::NLD + 1], qrow2 + n);
        }
    };
    uint4 w[BF::DEPTH][2 * BF::NLD];
#pragma unroll
    for (int d = 0; d < BF::DEPTH; ++d) load_unit(w[d], w0 + d);
    int n_lo = 0, nu = 0;
    auto load_sz = [&]() {
        n_lo = p0 << 5; nu = p1 - p0;
        const int per = nu * 4;                            // 16-byte pieces of a row
        for (int rr = 0; rr < 2 * p.ngl; ++rr) {
            const int gk = gk0 + (rr >> 1);
            const __half* src = ((rr & 1) ? p.zeros : p.scales) + (size_t)min(gk, ngroups - 1) * p.N;
            for (int i = tid; i < per; i += ST_THREADS) {
                const int c = n_lo + 8 * i;
                cp16(s_u32(sz) + (uint32_t)(rr * p.range + 8 * i) * 2u, src + min(c, p.N - 8), c < p.N ? 16 : 0);
            }
        }
    };
    load_sz();
    {   // ask the lines this CTA will read right after the wait into L2 (nothing is read into the SM): its slices of dY, B and A
        const int n = min(32 * nu, p.N - n_lo);
        for (int j = warp; j < p.M; j += ST_WARPS)
            for (int l = lane; 64 * l < n; l += 32) prefetch_l2(p.In + (size_t)j * p.N + n_lo + 64 * l);
        if (p.fused)
            for (int e = tid * 64; e < n * p.r; e += ST_THREADS * 64) prefetch_l2(p.Ldown + (size_t)n_lo * p.r + e);
        if (tid < p.r && c_lo < p.K) prefetch_l2(p.Lup + (size_t)tid * p.K + c_lo);
    }

    pdl_wait();

    const bool tok_ok[2] = {g < p.M, g + 8 < p.M};
    const uint32_t recv_h_addr = s_u32(smem + sp.recv_h);
    float acc[FL / 2][NT][4], z_sub[NT][2];
#pragma unroll
    for (int i = 0; i < FL / 2; ++i)
#pragma unroll
        for (int tt = 0; tt < NT; ++tt) acc[i][tt][0] = acc[i][tt][1] = acc[i][tt][2] = acc[i][tt][3] = 0.f;
#pragma unroll 1
    do {
    const bool again = MULTI && p0 > u0;
    if (again) {
        __syncthreads();                                   // every warp is done with the pass before
        load_sz();
    }
    // ---- staging: slices of dY, scaled by each group's scales (one rounding); the zero-point sums; this CTA's part of G = dY B ----
    {
        float hacc[NT][4], zacc[2][NT];
#pragma unroll
        for (int tt = 0; tt < NT; ++tt) {
            hacc[tt][0] = hacc[tt][1] = hacc[tt][2] = hacc[tt][3] = 0.f;
            zacc[0][tt] = zacc[1][tt] = 0.f;
        }
        const __nv_bfloat16* yr = p.In + (size_t)g * p.N + n_lo + 8 * q;
        const int n_left = p.N - n_lo - 8 * q;             // columns from this lane's first on
        bool staged = false;
#pragma unroll 1
        for (int s0 = warp; s0 < nu || !staged; s0 += SB * ST_WARPS) {
            uint4 yv[SB][NT];
            uint32_t bl[SB][4], bh[SB][4];
#pragma unroll
            for (int s = 0; s < SB; ++s) {
                const int sl = s0 + s * ST_WARPS;
                const bool in = sl < nu && 32 * sl < n_left;               // (N is a multiple of 8)
#pragma unroll
                for (int tt = 0; tt < NT; ++tt) yv[s][tt] = ldg16(yr + 8 * tt * (size_t)p.N + 32 * sl, in && tok_ok[tt]);
                // row rho of 8 x 8 tile t <-> column 8 (rho / 2) + rho % 2 + 2 t
                const int n8 = n_lo + 32 * sl + 8 * (g >> 1);
                const bool on = p.fused && sl < nu && n8 < p.N;
                const __nv_bfloat16* src = p.Ldown + (size_t)(n8 + (g & 1)) * p.r + 2 * q;
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    bl[s][t] = on ? ldg32(src + 2 * t * p.r) : 0u;
                    bh[s][t] = on && p.r > 8 ? ldg32(src + 2 * t * p.r + 8) : 0u;
                }
            }
            if (!staged) {                                 // (with the first loads on their way: every warp comes here once)
                if (!again) st_stage_lup<true>(p, smem + sp.lup, hfull, c_lo);
                cp_wait_all();
                __syncthreads();                           // the group parameters are staged
                staged = true;
            }
#pragma unroll
            for (int s = 0; s < SB; ++s) {
                const int sl = s0 + s * ST_WARPS;
                if (sl >= nu) break;
                if (p.fused) {
                    uint32_t a[4], b[4];
#pragma unroll
                    for (int t = 0; t < 4; ++t) { a[t] = st_movm(bl[s][t]); b[t] = p.r > 8 ? st_movm(bh[s][t]) : 0u; }
#pragma unroll
                    for (int tt = 0; tt < NT; ++tt) {
                        st_mma(hacc[tt], a[0], b[0], a[1], b[1], yv[s][tt].x, yv[s][tt].y);
                        st_mma(hacc[tt], a[2], b[2], a[3], b[3], yv[s][tt].z, yv[s][tt].w);
                    }
                }
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    if (c >= p.ngl) break;
                    const uint4 s8 = *reinterpret_cast<const uint4*>(sz + (2 * c) * p.range + 32 * sl + 8 * q);
                    const uint4 z8 = *reinterpret_cast<const uint4*>(sz + (2 * c + 1) * p.range + 32 * sl + 8 * q);
#pragma unroll
                    for (int tt = 0; tt < NT; ++tt) {
                        const uint4 v = yv[s][tt];
                        uint32_t o[4];
                        float zs = 0.f;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const uint32_t vi = st_comp(v, i), si = st_comp(s8, i), zi = st_comp(z8, i);
                            const float2 sf = __half22float2(*reinterpret_cast<const __half2*>(&si)), zf = __half22float2(*reinterpret_cast<const __half2*>(&zi));
                            o[i] = st_pack(bf16_lo(vi) * sf.x, bf16_hi(vi) * sf.y);
                            zs = fmaf(bf16_lo(o[i]), F::OFF + zf.x, zs);
                            zs = fmaf(bf16_hi(o[i]), F::OFF + zf.y, zs);
                        }
                        zacc[c][tt] += zs;
                        if (tok_ok[tt])
                            *reinterpret_cast<uint4*>(ys + (size_t)(c * p.M + g + 8 * tt) * p.pitch + sl * 64 + q * 16) = make_uint4(o[0], o[1], o[2], o[3]);
                    }
                }
            }
        }
        if (p.fused) st_store_hp<NT>(p, hacc, hp, warp, g, q, again);
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int tt = 0; tt < 2; ++tt) {
                const float z = tt < NT ? st_quad_sum(zacc[c][tt < NT ? tt : 0]) : 0.f;
                if (q == 0) zp[warp * 32 + c * 16 + 8 * tt + g] = z + (again ? zp[warp * 32 + c * 16 + 8 * tt + g] : 0.f);
            }
    }
    __syncthreads();
    if (!MULTI || p1 == u1) {
        if (p.ks > 1) st_cluster_wait();                   // every CTA of the cluster is running: its shared memory may be written
        if (p.fused) st_share_h(p, hp, recv_h_addr, rank);
        // zero-point sums of the CTA's whole range, warps added in order; part 0 alone subtracts them
#pragma unroll
        for (int tt = 0; tt < NT; ++tt) z_sub[tt][0] = z_sub[tt][1] = 0.f;
        if (part == 0) {
#pragma unroll
            for (int tt = 0; tt < NT; ++tt)
#pragma unroll
                for (int wv = 0; wv < ST_WARPS; ++wv) {
                    const float2 z = *reinterpret_cast<const float2*>(zp + wv * 32 + copy * 16 + 8 * tt + 2 * q);
                    z_sub[tt][0] += z.x; z_sub[tt][1] += z.y;
                }
        }
    }

    if (again) {                                           // (registers: they would lie idle during the staging)
#pragma unroll
        for (int d = 0; d < BF::DEPTH; ++d) load_unit(w[d], w0 + d);
    }

    // ---- main loop ----
    const uint32_t yl = s_u32(ys) + (uint32_t)((copy * p.M + g) * p.pitch + 8 * q);
    uint32_t xv[NT][2];
#pragma unroll
    for (int tt = 0; tt < NT; ++tt) xv[tt][0] = xv[tt][1] = 0u;            // (stays zero for tokens that do not exist)
#pragma unroll 1
    for (int un = w0; un < w1; un += BF::DEPTH) {
#pragma unroll
        for (int d = 0; d < BF::DEPTH; ++d) {
            if (un + d < w1) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint4& wa = w[d][h * BF::NLD];
                    const uint4& wb = w[d][h * BF::NLD + BF::NLD - 1];
                    uint32_t pa[FL], pb[FL];
                    st_bwd_pairs<BITS, FL>(wa.x, wb.x, wa.y, wb.y, sh, sel, pa);
                    st_bwd_pairs<BITS, FL>(wa.z, wb.z, wa.w, wb.w, sh, sel, pb);
#pragma unroll
                    for (int tt = 0; tt < NT; ++tt) {
                        lds8(xv[tt][0], xv[tt][1], yl + (uint32_t)(8 * tt * p.pitch + (un + d - p0) * 64 + 32 * h), tok_ok[tt]);
#pragma unroll
                        for (int i = 0; i < FL / 2; ++i) st_mma(acc[i][tt], pa[2 * i], pa[2 * i + 1], pb[2 * i], pb[2 * i + 1], xv[tt][0], xv[tt][1]);
                    }
                }
                load_unit(w[d], un + d + BF::DEPTH);
            }
        }
    }
    if (!MULTI || p1 == u1) break;
    p0 = p1; p1 = min(u1, p0 + p.pass);
    w0 = p0 + (((p1 - p0) * part) >> p.lwp); w1 = p0 + (((p1 - p0) * (part + 1)) >> p.lwp);
    } while (true);
    // accumulator element (i, tt, e): feature FL g + 2 i + (e >> 1) of the warp's, token 2q + (e & 1) + 8 tt
    float* mine = reinterpret_cast<float*>(smem + sp.part) + part * p.M * tile_c + 8 * FL * fw + FL * g;
#pragma unroll
    for (int tt = 0; tt < NT; ++tt)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int tok = 8 * tt + 2 * q + e;
            if (tok < p.M) {
#pragma unroll
                for (int j = 0; j < FL / 4; ++j)
                    *reinterpret_cast<float4*>(mine + tok * tile_c + 4 * j) = make_float4(acc[2 * j][tt][e] - z_sub[tt][e], acc[2 * j][tt][2 + e] - z_sub[tt][e],
                                                                                        acc[2 * j + 1][tt][e] - z_sub[tt][e], acc[2 * j + 1][tt][2 + e] - z_sub[tt][e]);
            }
        }
    st_finish<true>(p, smem, sp, c_lo, rank, blockIdx.y == 0 && rank == 0);
}

// Three CTAs per SM (80 registers) exist where the kernels spill 24 bytes at most: up to 8 tokens, 4 bits, and 2 bits backward.
// (Of the builds with 128 registers, those for 9 .. 16 tokens spill up to 80 bytes at 3 bits and 72 at 8 bits, the others none; the multi-pass
// ones up to 650, all of it around the staging.)
constexpr bool st_has_three(int bits, int nt, bool transposed) { return nt == 1 && (bits == 4 || (bits == 2 && transposed)); }

int fwd_kb(int bits) { return bits == 2 ? 64 : 32; }

constexpr int ST_MAX_DEVICES = kMaxDevices;
__global__ void __launch_bounds__(ST_THREADS, 2) st_probe_kernel() {}

// SM count, and how many clusters of 2 / 4 / 8 CTAs that share an SM two by two can run at once, per device ordinal.
struct DeviceFacts { int sms = 0; int clusters[9] = {}; };

const DeviceFacts& device_facts() {
    static std::mutex mu;
    static DeviceFacts facts[ST_MAX_DEVICES];
    static const DeviceFacts fallback{148, {0, 296, 148, 0, 72, 0, 0, 0, 34}};
    const int dev = device_ordinal();
    if (dev < 0) return fallback;
    std::lock_guard<std::mutex> lock(mu);
    DeviceFacts& f = facts[dev];
    if (f.sms == 0) {
        const int sms = sm_count();
        f.clusters[1] = 2 * sms;
        (void)cudaFuncSetAttribute(st_probe_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
        for (int cs = 2; cs <= 8; cs *= 2) {
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = dim3((unsigned)cs, (unsigned)sms);
            cfg.blockDim = dim3(ST_THREADS);
            cfg.dynamicSmemBytes = 100 * 1024;
            cudaLaunchAttribute attr;
            attr.id = cudaLaunchAttributeClusterDimension;
            attr.val.clusterDim.x = (unsigned)cs; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
            cfg.attrs = &attr;
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, st_probe_kernel, &cfg) != cudaSuccess || n <= 0) { (void)cudaGetLastError(); n = 2 * sms / cs; }
            f.clusters[cs] = n;
        }
        f.sms = sms;
    }
    return f;
}

// How a shape is cut: warps side by side (wc), CTAs per cluster (ks).  Every candidate that fits is costed in cycles, with the times
// read off stamped kernels (4096 x 4096 and the MLP shapes, 1 and 16 tokens):
//   products  a warp's own units of the contraction, 1400 cycles per chunk forward and 650 per unit backward whatever else the SM
//             does, up to a fifth more when a second CTA shares it: the chain of one warp, not the SM's throughput, sets the pace, so
//             the best cut is usually the one with about 256 CTAs;
//   staging   a warp's slices of the CTA's range, two in flight per round trip to L2;
//   exchange  the cluster barriers and the adding up;
// and the whole repeats when the CTAs exceed what the GPU holds at once (two per SM up to half an SM's shared memory).  Three per SM, with
// 80 registers, take 1.28 times as long for the same cut (4096 x 4096: 8.1 against 6.3 us) and are for cuts that two would need a second
// wave for, one INT4 token: K = 4096, N = 11008 forward, 344 CTAs, 15.9 -> 13.1 us; K = 11008, N = 4096 backward, 17.4 -> 14.7.
// (4096 x 4096, INT4, one token: 128 columns x 8 CTAs 6.3 us, 64 x 4 6.7, 32 x 2 8.2, 256 x 8 8.7, 128 x 4 9.3, 64 x 8 9.5.)
struct StreamPlan { StreamParams p; int tiles, tile_c, per_sm, nt; SmemPlan sm; bool multi, ok; };

template <int BITS, int NT, int V, bool TRANSPOSED, int PER_SM, bool MULTI>   // V: GPC forward, FL backward
int st_launch_as(const StreamPlan& plan, cudaStream_t st) {
    static SmemLimit limit;
    const dim3 grid((unsigned)plan.p.ks, (unsigned)plan.tiles);
    void (*kern)(const StreamParams);
    if constexpr (TRANSPOSED) kern = stream_bwd_kernel<BITS, NT, V, PER_SM, MULTI>;
    else kern = stream_fwd_kernel<BITS, NT, V, PER_SM, MULTI>;
    if (!limit.raise(kern, 227 * 1024)) return QLORA_ERR_CUDA;
    return launch_pdl(kern, grid, dim3(ST_THREADS), plan.sm.total, st, (unsigned)plan.p.ks, plan.p) == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
}

template <int BITS, int NT, int V, bool TRANSPOSED>
int st_launch(const StreamPlan& plan, cudaStream_t st) {
    if constexpr (st_has_three(BITS, NT, TRANSPOSED))
        if (plan.per_sm == 3) return st_launch_as<BITS, NT, V, TRANSPOSED, 3, false>(plan, st);
    if (plan.multi) return st_launch_as<BITS, NT, V, TRANSPOSED, 2, true>(plan, st);
    return st_launch_as<BITS, NT, V, TRANSPOSED, 2, false>(plan, st);
}

StreamPlan st_cut(StreamParams p, int bits, bool transposed) {
    StreamPlan best{};
    best.ok = false;
    float best_cost = 0.f;
    const DeviceFacts& gpu = device_facts();
    const int sms = gpu.sms;
    const int fl = p.g % 64 == 0 ? 8 : 4;
    p.gd = p.g / 32;
    p.gm = (uint32_t)(((1ull << 32) + p.gd - 1) / p.gd);
    const int T = transposed ? p.N : p.K;
    const int unit = transposed ? 32 : ST_CHUNK, units = (T + unit - 1) / unit;
    for (int lwc = 0; lwc <= 3; ++lwc) {
        p.wc = 1 << lwc; p.lwc = lwc; p.lwp = 3 - lwc;
        const int tile_c = (transposed ? 8 * fl : 32) * p.wc, tiles = (p.C + tile_c - 1) / tile_c;
        if (lwc > 0 && tile_c / 2 >= p.C) break;                       // (half the warps would have no column)
        if (tiles > 65535) continue;
        int groups = 1;                                                // backward: groups the features of a CTA span
        if (transposed && p.g % tile_c != 0) groups = tile_c % p.g == 0 ? tile_c / p.g : (tile_c - 1) / p.g + 2;
        if (groups > 2) continue;
        for (int lks = 0; lks <= 3; ++lks) {
            p.ks = 1 << lks; p.lks = lks;
            const int sl = tile_c >> lks;
            if (sl < 8) break;
            p.lsl = 0;
            while ((1 << p.lsl) < sl) ++p.lsl;
            const int per_cta = (units + p.ks - 1) / p.ks, parts = 1 << p.lwp;
            // the whole range in one pass, or in passes that leave room for two CTAs per SM, or for one
            for (int mode = 0; mode < (T > ST_LONG ? 3 : 1); ++mode) {
                const int nt = p.M > 8 ? 2 : 1, toks = 8 * nt;
                SmemPlan sm{};
                for (p.pass = per_cta;;) {
                    p.range = p.pass * unit;
                    p.ngl = transposed ? groups : (p.range + p.g - 1) / p.g + 1;
                    // rows far enough apart that the fragment loads of neighbouring tokens meet different banks
                    const int want = transposed ? 32 : (bits == 2 ? 16 : (bits == 8 ? 32 : 64));
                    p.pitch = p.range * 2;
                    p.pitch += (want - p.pitch % 128 + 128) % 128;
                    sm = st_plan(p, transposed, toks, tile_c);
                    if (mode == 0 || p.pass == 1 || sm.total <= (mode == 1 ? 113u * 1024 : 227u * 1024 - 1024)) break;
                    p.pass = p.pass > 16 ? p.pass * 7 / 8 : p.pass - 1;
                }
                if (sm.total > 227 * 1024 - 1024 || (mode > 0 && p.pass == per_cta)) continue;
                const int passes = (per_cta + p.pass - 1) / p.pass, per_warp = (p.pass + parts - 1) / parts * passes;
                const float step = (transposed ? 650.f + 150.f * (nt - 1) : 1400.f + 450.f * (nt - 1)) * (bits == 8 ? 1.3f : 1.f) * (tiles * p.ks > sms ? 1.2f : 1.f);
                const float rounds = (float)((p.pass * (unit / 32) + 2 * ST_WARPS - 1) / (2 * ST_WARPS) * passes);
                const float round = transposed ? 2500.f * nt : 900.f + 1100.f * nt;
                const float once = (float)per_warp * step + rounds * round + 1500.f + 500.f * (float)lks + 1000.f * (float)(passes - 1);
                for (int per_sm = 2; per_sm <= (mode == 0 && st_has_three(bits, nt, transposed) && sm.total <= 74 * 1024 ? 3 : 2); ++per_sm) {
                    const int occ = sm.total <= 113 * 1024 ? per_sm : 1;
                    const float fill = (float)(tiles * 2) / (float)(gpu.clusters[p.ks] * occ);     // of what the GPU holds at once
                    const float waves = fill <= 1.f ? 1.f : 0.5f * (fill + ceilf(fill));
                    const float cost = waves * once * (per_sm == 3 ? 1.28f : 1.f);
                    if (!best.ok || cost < best_cost) { best = StreamPlan{p, tiles, tile_c, per_sm, nt, sm, mode > 0, true}; best_cost = cost; }
                }
            }
        }
    }
    return best;
}

}  // namespace

bool stream_supported(const qlora_desc& d, int M, bool transposed) {
    if (M < 1 || M > 16) return false;
    if (d.K < 32 || d.N < 8 || d.K > (1 << 20)) return false;   // (the group index's reciprocal is exact up to there)
    if (!transposed && d.group_size % fwd_kb(d.bits) != 0) return false;
    const int T = transposed ? d.N : d.K;
    if (T <= ST_LONG) return true;                          // eight ways split, such a range always fits the shared memory
    // More than 8 tokens on a longer one, backward: 16 scaled copies of it are staged, in as many passes as they need, and the tensor-core kernel
    // is the faster one where it takes the shape (N = 128256: 206 against 302 us).
    if (transposed && M > 8 && umma_supported(d, M)) return false;
    StreamParams p{};
    p.M = M; p.K = d.K; p.N = d.N; p.g = d.group_size; p.r = d.r; p.C = transposed ? d.K : d.N;
    p.fused = d.r > 0 && d.r <= 16 ? 1 : 0;
    return st_cut(p, d.bits, transposed).ok;
}

int launch_stream_gemm(const qlora_desc& d, int M, bool transposed, const void* In, const int32_t* Q, const void* scales,
                       const void* zeros, const void* Ldown, const void* Lup, float* P, bool p_is_input, void* Out,
                       cudaStream_t st) {
    StreamParams p{};
    p.M = M; p.K = d.K; p.N = d.N; p.g = d.group_size; p.r = d.r;
    p.C = transposed ? d.K : d.N;
    p.s = d.r > 0 ? d.alpha / (float)d.r : 0.f;
    p.In = (const __nv_bfloat16*)In; p.Q = (const uint32_t*)Q; p.scales = (const __half*)scales; p.zeros = (const __half*)zeros;
    p.Ldown = (const __nv_bfloat16*)Ldown; p.Lup = (const __nv_bfloat16*)Lup; p.P = P; p.Out = (__nv_bfloat16*)Out;
    p.fused = (d.r > 0 && !p_is_input) ? 1 : 0;
    if (p.fused && d.r > 16) return QLORA_ERR_INVALID_ARG;
    const StreamPlan plan = st_cut(p, d.bits, transposed);
    if (!plan.ok) return QLORA_ERR_UNSUPPORTED;
#define QLORA_ST(B, NT)                                                                                                          \
    if (transposed)                                                                                                              \
        return d.group_size % 64 == 0 ? st_launch<B, NT, 8, true>(plan, st)                                                      \
                                      : st_launch<B, NT, 4, true>(plan, st);                                                     \
    if (d.group_size % 128 == 0) return st_launch<B, NT, 1, false>(plan, st);                                                    \
    if (d.group_size % 64 == 0) return st_launch<B, NT, 2, false>(plan, st);                                                     \
    if constexpr (B != 2) return st_launch<B, NT, 4, false>(plan, st);                                                           \
    else return QLORA_ERR_UNSUPPORTED
#define QLORA_ST_BITS(NT)           \
    switch (d.bits) {               \
        case 2: { QLORA_ST(2, NT); }    \
        case 3: { QLORA_ST(3, NT); }    \
        case 4: { QLORA_ST(4, NT); }    \
        case 8: { QLORA_ST(8, NT); }    \
    }
    if (plan.nt == 1) { QLORA_ST_BITS(1) } else { QLORA_ST_BITS(2) }
#undef QLORA_ST_BITS
#undef QLORA_ST
    return QLORA_ERR_UNSUPPORTED;
}

}  // namespace qlora
