// CUDA-core kernels of the quantized-linear + LoRA layer.  They are correct for every shape the library accepts
// and serve (a) shapes the tensor-core kernels do not tile, and (b) the skinny LoRA products, which are bound by
// HBM traffic rather than by arithmetic (Figure 1 of the paper: the green "MM" blocks and their gradients).
#include "common.cuh"
#include "device_state.h"
#include "launch.h"
#include "lora_down.cuh"

#include <type_traits>

namespace qlora {

// ------------------------------------------------------------------------------------------------------------
// Generic tiled product with on-the-fly dequantisation.
//   forward        : Out[m, n] = sum_k In[m, k] W[n, k] + s sum_j P[m, j] B[n, j]        (T = K, C = N)
//   backward-input : Out[m, k] = sum_n In[m, n] W[n, k] + s sum_j P[m, j] A[j, k]        (T = N, C = K)
// 64 x 64 output tile, contraction step 16, 256 threads, 4 x 4 outputs per thread, fp32 accumulation.
// ------------------------------------------------------------------------------------------------------------
constexpr int SG_BM = 64, SG_BC = 64, SG_BT = 16;

template <bool TRANSPOSED>
__global__ void __launch_bounds__(256)
simt_gemm_kernel(int bits, int g, int K, int N, int r, float s, int M, const __nv_bfloat16* __restrict__ In,
                 const uint32_t* __restrict__ Q, const __half* __restrict__ scales, const __half* __restrict__ zeros,
                 const __nv_bfloat16* __restrict__ L, const float* __restrict__ P, __nv_bfloat16* __restrict__ Out) {
    pdl_launch_dependents();
    pdl_wait();
    const int T = TRANSPOSED ? N : K;   // contraction length
    const int C = TRANSPOSED ? K : N;   // output columns
    __shared__ float sIn[SG_BT][SG_BM + 4];
    __shared__ float sW[SG_BT][SG_BC + 4];
    const int tid = threadIdx.x;
    const int m0 = blockIdx.y * SG_BM, c0 = blockIdx.x * SG_BC;
    const int ty = tid / 16, tx = tid % 16;
    float acc[4][4] = {};

    for (int t0 = 0; t0 < T; t0 += SG_BT) {
        {   // activations: 64 rows x 16 contraction values, 4 consecutive t per thread
            const int mi = tid / 4, tq = (tid % 4) * 4;
            const int m = m0 + mi;
            float v[4] = {0.f, 0.f, 0.f, 0.f};
            if (m < M && t0 + tq < T) {   // T is a multiple of 8, so a group of 4 is all-in or all-out
                const uint2 raw = *reinterpret_cast<const uint2*>(In + (size_t)m * T + t0 + tq);
                v[0] = bf16_lo(raw.x); v[1] = bf16_hi(raw.x); v[2] = bf16_lo(raw.y); v[3] = bf16_hi(raw.y);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) sIn[tq + i][mi] = v[i];
        }
        {   // weights: 16 contraction values x 64 output columns, 4 per thread
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int e = tid + i * 256;
                const int ti = e / 64, ci = e % 64;   // ti: contraction offset, ci: output offset (fastest across threads)
                const int t = t0 + ti, c = c0 + ci;
                float w = 0.f;
                if (t < T && c < C) {
                    const int k = TRANSPOSED ? c : t, n = TRANSPOSED ? t : c;
                    const size_t gi = (size_t)(k / g) * N + n;
                    w = __bfloat162float(dequant_one(load_code(Q, N, bits, k, n), scales[gi], zeros[gi]));
                }
                sW[ti][ci] = w;
            }
        }
        __syncthreads();
#pragma unroll
        for (int t = 0; t < SG_BT; ++t) {
            const float4 a = *reinterpret_cast<const float4*>(&sIn[t][ty * 4]);
            const float4 b = *reinterpret_cast<const float4*>(&sW[t][tx * 4]);
            const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
        __syncthreads();
    }

#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + ty * 4 + i;
        if (m >= M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = c0 + tx * 4 + j;
            if (c >= C) continue;
            float lo = 0.f;
            for (int q = 0; q < r; ++q) {
                const float l = TRANSPOSED ? __bfloat162float(L[(size_t)q * K + c])    // A[j, k]
                                           : __bfloat162float(L[(size_t)c * r + q]);   // B[n, j]
                lo = fmaf(P[(size_t)m * r + q], l, lo);
            }
            Out[(size_t)m * C + c] = __float2bfloat16_rn(acc[i][j] + s * lo);
        }
    }
}

int launch_simt_gemm(const qlora_desc& d, int M, bool transposed, const void* In, const int32_t* Q,
                     const void* scales, const void* zeros, const void* L, const float* P, void* Out,
                     cudaStream_t st) {
    const int C = transposed ? d.K : d.N;
    if (M == 0 || C == 0) return QLORA_OK;
    const float s = d.r > 0 ? d.alpha / (float)d.r : 0.f;
    dim3 grid((C + SG_BC - 1) / SG_BC, (M + SG_BM - 1) / SG_BM);
    cudaError_t err;
    if (transposed)
        err = launch_pdl(simt_gemm_kernel<true>, grid, dim3(256), 0, st, 1, d.bits, d.group_size, d.K, d.N, d.r, s, M,
            (const __nv_bfloat16*)In, (const uint32_t*)Q, (const __half*)scales, (const __half*)zeros,
            (const __nv_bfloat16*)L, P, (__nv_bfloat16*)Out);
    else
        err = launch_pdl(simt_gemm_kernel<false>, grid, dim3(256), 0, st, 1, d.bits, d.group_size, d.K, d.N, d.r, s, M,
            (const __nv_bfloat16*)In, (const uint32_t*)Q, (const __half*)scales, (const __half*)zeros,
            (const __nv_bfloat16*)L, P, (__nv_bfloat16*)Out);
    return err == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
}

// ------------------------------------------------------------------------------------------------------------
// LoRA down-projections: H = X A^T (contraction over K) and G = dY B (contraction over N), fp32 [M, r].
// Skinny products bound by reading the activations once.  Up to 256 rows, rank 8, no mask: a block owns 16 token rows
// (lora_down.cuh has the method; few blocks, so that the kernel behind this one can set itself up on the other SMs meanwhile: 160 rows
// forward, 16.2 us, against 18.7 with the clusters below).
// ------------------------------------------------------------------------------------------------------------
constexpr int LD_WARPS = 32;

template <bool L_IS_A>
__global__ void __launch_bounds__(LD_WARPS * 32)
lora_down_kernel(int M, int T, int r, const __nv_bfloat16* __restrict__ In, const __nv_bfloat16* __restrict__ L, float* __restrict__ P) {
    __shared__ float red[LD_WARPS * 128];
    pdl_launch_dependents();
    pdl_wait();
    lora_down_rows<L_IS_A, 1, 1, L_IS_A ? 4 : 2>(M, T, r, In, L, P, (int)blockIdx.x * 16, 0, LD_WARPS, red);   // (64 registers; no spills)
}

// thread-block cluster helpers
__device__ __forceinline__ uint32_t lg_map_to_cta(const void* smem_ptr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(smem_ptr)), "r"(rank));
    return r;
}
__device__ __forceinline__ float4 lg_ld_cluster_f32x4(uint32_t cluster_addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(cluster_addr) : "memory");
    return v;
}
__device__ __forceinline__ void lg_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Ranks above 8 (above 16 with many rows), or a dropout mask (with many rows, ranks above 16): 16 token rows per cluster, the contraction split over its 1 << lcs CTAs and their eight warps.
// Bound by the latency of the adapter and activation loads (the adapter's share of the loads grows with the rank), so a warp issues
// all loads of DEPTH 32-wide steps together, and the cluster is as wide as keeps two CTAs per SM: 2048 tokens x 4096, rank 32,
// inputs from DRAM: 18 -> 10 us (blocks of eight warps that waited for every step's adapter words before).
// Fragments as in lora_down.cuh, except that a lane reads its 2 NT neighbouring ranks of a row of B in 16-byte pieces where the rank
// fills the tiles: column c of tile i is then rank 2 NT (c / 2) + 2 i + c % 2.  Partial tiles: the warps' in order, then the CTAs' in
// order, each CTA for a part of the elements: the same bits on every run.
constexpr int LS_WARPS = 8;

template <bool L_IS_A, int NT, bool MASKED>
__global__ void __launch_bounds__(LS_WARPS * 32, 2)
lora_down_split_kernel(int M, int T, int r, int lcs, const __nv_bfloat16* __restrict__ In, const __nv_bfloat16* __restrict__ L,
                       float* __restrict__ P, const uint8_t* __restrict__ mask, float out_scale) {
    constexpr int DEPTH = NT <= 2 ? 4 : (NT <= 4 ? 2 : 1), ELEMS = NT * 128;
    __shared__ float red[LS_WARPS * ELEMS];
    __shared__ float recv[ELEMS];                              // [CTA of the cluster][this CTA's share of the elements]
    pdl_launch_dependents();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    const int cs = 1 << lcs, rank = (int)blockIdx.x & (cs - 1), m_base = ((int)blockIdx.x >> lcs) * 16;
    const int steps = (T + 31) >> 5, s0 = (steps * rank) >> lcs, s1 = (steps * (rank + 1)) >> lcs;
    const int r0 = m_base + g, r1 = r0 + 8;
    const bool v0 = r0 < M, v1 = r1 < M, packed = r == 8 * NT;
    const __nv_bfloat16* row0 = In + (size_t)r0 * T;
    const __nv_bfloat16* row1 = In + (size_t)r1 * T;
    float acc[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.f;
    const uint4 zero4 = make_uint4(0, 0, 0, 0);
    pdl_wait();
#pragma unroll 1
    for (int st = s0 + warp; st < s1; st += LS_WARPS * DEPTH) {
        uint4 xlo[DEPTH], xhi[DEPTH], l[DEPTH][NT];            // B: l[u][i] = tile i's words of the four 8 x 8 row tiles
        uint2 mlo[DEPTH], mhi[DEPTH];
#pragma unroll
        for (int u = 0; u < DEPTH; ++u) {
            const int k0 = (st + u * LS_WARPS) * 32, k = k0 + q * 8;
            const bool in = st + u * LS_WARPS < s1 && k < T;   // T is a multiple of 8: 8 elements are all-in or all-out
            xlo[u] = v0 && in ? __ldg(reinterpret_cast<const uint4*>(row0 + k)) : zero4;
            xhi[u] = v1 && in ? __ldg(reinterpret_cast<const uint4*>(row1 + k)) : zero4;
            if constexpr (MASKED) {
                mlo[u] = v0 && in ? __ldg(reinterpret_cast<const uint2*>(mask + (size_t)r0 * T + k)) : make_uint2(0, 0);
                mhi[u] = v1 && in ? __ldg(reinterpret_cast<const uint2*>(mask + (size_t)r1 * T + k)) : make_uint2(0, 0);
            }
            if constexpr (L_IS_A) {
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
                    l[u][nt] = in && nt * 8 + g < r ? __ldg(reinterpret_cast<const uint4*>(L + (size_t)(nt * 8 + g) * T + k)) : zero4;
            } else {
                const int nb = k0 + 8 * (g >> 1) + (g & 1);    // tile t's row g <-> contraction index nb + 2 t
                const bool on = st + u * LS_WARPS < s1 && nb < T;   // (T a multiple of 8: the four rows are all-in or all-out)
                const __nv_bfloat16* src = L + (size_t)nb * r;
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) l[u][nt] = zero4;
                if (on) {
                    if (packed && NT % 4 == 0) {
#pragma unroll
                        for (int h = 0; h < NT / 4; ++h) {
                            const uint4 t0 = __ldg(reinterpret_cast<const uint4*>(src + 2 * NT * q + 8 * h));
                            const uint4 t1 = __ldg(reinterpret_cast<const uint4*>(src + 2 * r + 2 * NT * q + 8 * h));
                            const uint4 t2 = __ldg(reinterpret_cast<const uint4*>(src + 4 * r + 2 * NT * q + 8 * h));
                            const uint4 t3 = __ldg(reinterpret_cast<const uint4*>(src + 6 * r + 2 * NT * q + 8 * h));
                            l[u][(4 * h) % NT] = make_uint4(t0.x, t1.x, t2.x, t3.x);
                            l[u][(4 * h + 1) % NT] = make_uint4(t0.y, t1.y, t2.y, t3.y);
                            l[u][(4 * h + 2) % NT] = make_uint4(t0.z, t1.z, t2.z, t3.z);
                            l[u][(4 * h + 3) % NT] = make_uint4(t0.w, t1.w, t2.w, t3.w);
                        }
                    } else {
                        const int lane_r = packed ? 2 * NT * q : 2 * q, tile_r = packed ? 2 : 8;
#pragma unroll
                        for (int nt = 0; nt < NT; ++nt)
                            if (nt * 8 < r) {
                                const __nv_bfloat16* t = src + lane_r + tile_r * nt;
                                l[u][nt] = make_uint4(__ldg(reinterpret_cast<const uint32_t*>(t)), __ldg(reinterpret_cast<const uint32_t*>(t + 2 * r)),
                                                      __ldg(reinterpret_cast<const uint32_t*>(t + 4 * r)), __ldg(reinterpret_cast<const uint32_t*>(t + 6 * r)));
                            }
                    }
                }
            }
        }
#pragma unroll
        for (int u = 0; u < DEPTH; ++u) {
            if (st + u * LS_WARPS >= s1) break;                // warp-uniform
            if constexpr (MASKED) { xlo[u] = mask_eight(xlo[u], mlo[u]); xhi[u] = mask_eight(xhi[u], mhi[u]); }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                uint4 lv = l[u][nt];
                if constexpr (!L_IS_A) lv = make_uint4(movmatrix_trans(lv.x), movmatrix_trans(lv.y), movmatrix_trans(lv.z), movmatrix_trans(lv.w));
                mma_bf16_16816(acc[nt], xlo[u].x, xhi[u].x, xlo[u].y, xhi[u].y, lv.x, lv.y);
                mma_bf16_16816(acc[nt], xlo[u].z, xhi[u].z, xlo[u].w, xhi[u].w, lv.z, lv.w);
            }
        }
    }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int c = 0; c < 4; ++c) red[warp * ELEMS + (nt * 4 + c) * 32 + lane] = acc[nt][c];
    __syncthreads();
    const int share = ELEMS >> lcs;                            // elements a CTA finishes (a multiple of 16)
    if (lcs > 0) lg_cluster_sync();                            // every CTA of the cluster is running: its shared memory may be written
    for (int e = threadIdx.x; e < ELEMS; e += LS_WARPS * 32) {
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < LS_WARPS; ++w) v += red[w * ELEMS + e];
        const int owner = e / share;
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(lg_map_to_cta(recv + rank * share + (e - owner * share), (uint32_t)owner)), "f"(v) : "memory");
    }
    if (lcs > 0) lg_cluster_sync();                            // everyone's sums for this CTA's elements have arrived
    else __syncthreads();
    for (int i = threadIdx.x; i < share; i += LS_WARPS * 32) {
        float v = 0.f;
        for (int rk = 0; rk < cs; ++rk) v += recv[rk * share + i];
        const int e = rank * share + i, nt = e >> 7, c = (e >> 5) & 3, ln = e & 31;
        const int row = m_base + (ln >> 2) + ((c & 2) ? 8 : 0);
        const int col = !L_IS_A && packed ? 2 * NT * (ln & 3) + 2 * nt + (c & 1) : nt * 8 + (ln & 3) * 2 + (c & 1);
        if (row < M && col < r) P[(size_t)row * r + col] = v * out_scale;
    }
}

int launch_lora_down(int M, int T, int r, bool l_is_A, const void* In, const void* L, float* P, cudaStream_t st,
                     const uint8_t* mask, float out_scale) {
    if (M == 0 || r == 0) return QLORA_OK;
    const bool plain = mask == nullptr && out_scale == 1.0f && r <= 16;
    // Many rows, low rank: the streaming kernel (also the form that runs inside the CTA-pair kernel, so H / G have the
    // same bits whichever call produced them).
    if ((plain && M > 256) || (mask != nullptr && l_is_A && lora_down_streams_masked(M, r))) return launch_lora_down_stream(M, T, r, l_is_A, In, L, P, st, mask, out_scale);
    const unsigned blocks = (unsigned)((M + 15) / 16);
    const __nv_bfloat16* in = (const __nv_bfloat16*)In;
    const __nv_bfloat16* l = (const __nv_bfloat16*)L;
    const int nt = (r + 7) / 8;
    cudaError_t err = cudaSuccess;
    if (plain && r <= 8) {
        if (l_is_A) err = launch_pdl(lora_down_kernel<true>, dim3(blocks), dim3(LD_WARPS * 32), 0, st, 1, M, T, r, in, l, P);
        else        err = launch_pdl(lora_down_kernel<false>, dim3(blocks), dim3(LD_WARPS * 32), 0, st, 1, M, T, r, in, l, P);
        return err == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
    }
    // clusters as wide as leave two CTAs per SM, while a CTA keeps a step for each of its warps
    int lcs = 0;
    while (lcs < 3 && (blocks << (lcs + 1)) <= 2u * (unsigned)sm_count() && (T >> (lcs + 1)) >= 32 * LS_WARPS) ++lcs;
    const dim3 grid(blocks << lcs), block(LS_WARPS * 32);
#define QLORA_LS(NTV)                                                                                                             \
    do {                                                                                                                          \
        if (!l_is_A)      err = launch_pdl(lora_down_split_kernel<false, NTV, false>, grid, block, 0, st, 1u << lcs, M, T, r, lcs, in, l, P, (const uint8_t*)nullptr, out_scale); \
        else if (mask)    err = launch_pdl(lora_down_split_kernel<true, NTV, true>, grid, block, 0, st, 1u << lcs, M, T, r, lcs, in, l, P, mask, out_scale);   \
        else              err = launch_pdl(lora_down_split_kernel<true, NTV, false>, grid, block, 0, st, 1u << lcs, M, T, r, lcs, in, l, P, mask, out_scale);  \
    } while (0)
    if (!l_is_A && mask != nullptr) return QLORA_ERR_INVALID_ARG;   // (a mask is on the input of the first adapter only)
    if (nt <= 1) QLORA_LS(1);
    else if (nt <= 2) QLORA_LS(2);
    else if (nt <= 4) QLORA_LS(4);
    else QLORA_LS(8);
#undef QLORA_LS
    return err == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
}

// ------------------------------------------------------------------------------------------------------------
// LoRA gradients: Out(c, j) = s * sum_m In[m, c] * P[m, j]   (dB: In = dY, P = H, C = N;  dA: In = X, P = G, C = K).
// Bound by reading X and dY once.  Pass 1 (one launch for both gradients): a block owns 256 columns and one slice of
// the token rows; a warp owns 32 of the columns and runs mma.sync m16n8k16 with the ranks as the MMA's M side:
//   D[j, c] += sum_m P^T[j, m] In[m, c]
// The P^T fragments come from a bf16 copy of the slice's P rows staged (transposed) in shared memory; the In fragments
// need pairs of consecutive m for a fixed column, so the 16-byte row loads (8 columns per lane) are transposed across
// the warp with movmatrix.  This permutes which column each accumulator element belongs to (lane (g, q), tile c,
// element e  <->  column 8q + 2c + e of the warp's 32), which the write-out undoes.  The block writes its tile to
// scratch[slice]; pass 2 adds the slices in index order, scales by s and writes (or adds to) dA / dB.
// Nothing depends on scheduling: the result is bitwise reproducible.
// ------------------------------------------------------------------------------------------------------------
constexpr int LG_COLS = 256;          // columns per block (32 per warp)
constexpr int LG_WARPS = 8;
constexpr int LG_UNROLL = 4;          // 16-row steps whose loads are issued together
constexpr int LG_MAX_SLICES = 64;

struct GradPlan { int slices, rows_per_slice; };

static GradPlan lora_grad_plan(int M, int K, int N) {
    int col_blocks = (K + LG_COLS - 1) / LG_COLS + (N + LG_COLS - 1) / LG_COLS;
    if (col_blocks < 1) col_blocks = 1;                          // (K = N = 0: a layer without elements)
    int slices = (2 * 148) / col_blocks;                         // two blocks fit an SM (registers): aim for one wave of a 148-SM part
    if (slices > LG_MAX_SLICES) slices = LG_MAX_SLICES;
    if (slices < 1) slices = 1;
    int rows = (M + slices - 1) / slices;
    rows = (rows + 63) / 64 * 64;                                // whole 16-row MMA steps; keeps the staged P^T conflict-free
    if (rows < 64) rows = 64;
    if (rows > 1024) rows = 1024;                                // bounds the staged P^T (64 ranks x 1032 x 2 B = 129 KiB at most)
    GradPlan g;
    g.rows_per_slice = rows;
    g.slices = M > 0 ? (M + rows - 1) / rows : 1;
    return g;
}

size_t lora_grad_scratch_bytes(int M, int K, int N, int r) {
    return (size_t)lora_grad_plan(M, K, N).slices * (size_t)(K + N) * (size_t)r * sizeof(float);
}

struct GradSide {
    const __nv_bfloat16* In;   // [M, C]
    const float* P;            // [M, r]
    float* partial;            // [slices][C][r]
    float* Out;
    int C;
    const uint8_t* mask;       // [M, C] dropout mask on In (non-zero = keep), or NULL
    float scale;               // s (times the dropout keep scale on the masked side)
    int out_is_dB;             // Out is dB [C, r] (else dA [r, C])
};

// A 16-byte load that stays where it is written: ahead of the products of the round before.
__device__ __forceinline__ void lg_load(uint4& v, const void* p) {
    asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
}

// CL == 0: grid (column blocks, slices, 2 sides); the block writes its partial tile to scratch for lora_grad_reduce_kernel.
// CL >= 1: one launch does it all.  grid (column blocks * CL, 1, 2 sides) in clusters of CL CTAs along x; the CTAs of a
//   cluster take the CL row slices of one column block, leave their partial tiles in shared memory, and after a cluster
//   barrier CTA i adds them in slice order (distributed shared memory, fixed order) for its 256 / CL columns, scales
//   and writes (or adds to) dA / dB.
// MASKED: side 1 (dA) has a dropout mask on its activations; the mask bytes travel with the loads of their round and are applied when
// the round's turn comes (applied as they were loaded they made every round wait for memory: 29 against 13.7 us at 1800 tokens).
// (Two blocks per SM for ranks up to 32; with 104 registers, up to 16, they leave room for a block of the reduction launch, which starts early.
// The masked form with two rank tiles spills 48 bytes for it, and gains: 1800 tokens, rank 32, 21.7 us against 27.7 with 140 registers and one
// block; in clusters, where there are few blocks anyway, it has the 140: 200 tokens 8.8 -> 7.4.)
template <int RT, int CL, bool MASKED>   // rank tiles of 16; cluster width (0 = two-launch form)
__global__ void __launch_bounds__(LG_WARPS * 32) __maxnreg__(RT == 1 && !MASKED ? 104 : (RT == 1 || (RT == 2 && !(MASKED && CL > 0)) ? 128 : 184))
lora_grad_partial_kernel(int M, int r, int rows_per_slice, GradSide side0, GradSide side1, int accumulate) {
    extern __shared__ __align__(16) uint8_t lg_smem[];
    pdl_launch_dependents();
    pdl_wait();
    __nv_bfloat16* Pt = reinterpret_cast<__nv_bfloat16*>(lg_smem);   // [RT * 16][rows_per_slice + 8]
    const GradSide& sd = blockIdx.z == 0 ? side0 : side1;
    const int C = sd.C;
    const int cb = (CL > 0 ? (int)blockIdx.x / CL : (int)blockIdx.x) * LG_COLS;
    if (cb >= C) return;                                       // (the whole cluster returns: same column block)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, q = lane & 3;
    const int slice = CL > 0 ? (int)blockIdx.x % CL : (int)blockIdx.y;
    const int m_begin = slice * rows_per_slice;
    const int stride = rows_per_slice + 8;                     // in bf16: (stride / 2) % 32 == 4 -> conflict-free fragment loads
    constexpr int RP = RT * 16;
    auto stage_p = [&]() {   // P^T (bf16) of this slice: rows beyond M and ranks beyond r are zero
        for (int e = threadIdx.x; e < rows_per_slice * RP; e += LG_WARPS * 32) {
            const int ml = e / RP, j = e % RP;
            const int m = m_begin + ml;
            const float v = (m < M && j < r) ? __ldg(sd.P + (size_t)m * r + j) : 0.f;
            Pt[j * stride + ml] = __float2bfloat16_rn(v);
        }
        __syncthreads();
    };
    if constexpr (RT > 1) stage_p();

    const int c0 = cb + warp * 32 + q * 8;                     // this lane loads columns c0 .. c0 + 7
    const bool live = c0 < C;                                  // C is a multiple of 8
    const __nv_bfloat16* src = sd.In + c0;
    float acc[RT][4][4];
#pragma unroll
    for (int rt = 0; rt < RT; ++rt)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[rt][c][0] = acc[rt][c][1] = acc[rt][c][2] = acc[rt][c][3] = 0.f;
    const uint4 zero4 = make_uint4(0, 0, 0, 0);
    const int m_stop = min(M, m_begin + rows_per_slice);
    // two register sets: the loads of the next round of 16-row steps are in flight while this round is transposed and multiplied
    uint4 n0[LG_UNROLL], n1[LG_UNROLL];
    uint2 k0[MASKED ? LG_UNROLL : 1], k1[MASKED ? LG_UNROLL : 1];
    const bool masked = MASKED && sd.mask != nullptr;
    auto load_round = [&](int mm) {
#pragma unroll
        for (int u = 0; u < LG_UNROLL; ++u) {
            const int ma = mm + 16 * u + g, mb = ma + 8;
            n0[u] = zero4; n1[u] = zero4;
            if (live && ma < m_stop) lg_load(n0[u], src + (size_t)ma * C);
            if (live && mb < m_stop) lg_load(n1[u], src + (size_t)mb * C);
            if constexpr (MASKED) {
                if (masked) {
                    if (live && ma < m_stop) k0[u] = __ldg(reinterpret_cast<const uint2*>(sd.mask + (size_t)ma * C + c0));
                    if (live && mb < m_stop) k1[u] = __ldg(reinterpret_cast<const uint2*>(sd.mask + (size_t)mb * C + c0));
                }
            }
        }
    };
    load_round(m_begin);
    // One rank tile has the registers to keep the first round under way while P is staged: 64 tokens, 4096 x 4096, 3.28 -> 2.90 us (3.25
    // before the loads were made volatile); 1024 tokens 8.8 -> 8.5.
    if constexpr (RT == 1) stage_p();
    for (int mm = m_begin; mm < m_stop; mm += 16 * LG_UNROLL) {
        uint4 x0[LG_UNROLL], x1[LG_UNROLL];
#pragma unroll
        for (int u = 0; u < LG_UNROLL; ++u) {
            x0[u] = n0[u]; x1[u] = n1[u];
            if constexpr (MASKED) {
                if (masked) { x0[u] = mask_eight(x0[u], k0[u]); x1[u] = mask_eight(x1[u], k1[u]); }   // (rows beyond the last are zero anyway)
            }
        }
        if (mm + 16 * LG_UNROLL < m_stop) load_round(mm + 16 * LG_UNROLL);
#pragma unroll
        for (int u = 0; u < LG_UNROLL; ++u) {
            const int ml = mm + 16 * u - m_begin;              // warp-uniform
            if (ml >= rows_per_slice || mm + 16 * u >= m_stop) break;
            uint32_t b0[4], b1[4];
            b0[0] = movmatrix_trans(x0[u].x); b0[1] = movmatrix_trans(x0[u].y);
            b0[2] = movmatrix_trans(x0[u].z); b0[3] = movmatrix_trans(x0[u].w);
            b1[0] = movmatrix_trans(x1[u].x); b1[1] = movmatrix_trans(x1[u].y);
            b1[2] = movmatrix_trans(x1[u].z); b1[3] = movmatrix_trans(x1[u].w);
#pragma unroll
            for (int rt = 0; rt < RT; ++rt) {
                const __nv_bfloat16* pa = Pt + (rt * 16 + g) * stride + ml + 2 * q;
                const uint32_t a0 = *reinterpret_cast<const uint32_t*>(pa);
                const uint32_t a1 = *reinterpret_cast<const uint32_t*>(pa + 8 * stride);
                const uint32_t a2 = *reinterpret_cast<const uint32_t*>(pa + 8);
                const uint32_t a3 = *reinterpret_cast<const uint32_t*>(pa + 8 * stride + 8);
#pragma unroll
                for (int c = 0; c < 4; ++c) mma_bf16_16816(acc[rt][c], a0, a1, a2, a3, b0[c], b1[c]);
            }
        }
    }
    // accumulator element (rt, c, i): rank rt*16 + g (+8 for i >= 2), column 8q + 2c + (i & 1) of the warp's 32
    if constexpr (CL > 0) {
        __syncthreads();                                       // every warp is done with the staged P^T: the tile takes its place
        float* tile = reinterpret_cast<float*>(lg_smem);       // [256 columns][RP] fp32
#pragma unroll
        for (int rt = 0; rt < RT; ++rt)
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    tile[(warp * 32 + q * 8 + 2 * c + (i & 1)) * RP + rt * 16 + g + ((i & 2) ? 8 : 0)] = acc[rt][c][i];
        __syncthreads();
        lg_cluster_sync();                                     // all CL partial tiles are written
        constexpr int COLS_PER = LG_COLS / CL;
        uint32_t peer[CL];
#pragma unroll
        for (int k = 0; k < CL; ++k) peer[k] = lg_map_to_cta(tile, (uint32_t)k);
        const bool is_dB = sd.out_is_dB != 0;
        for (int e = threadIdx.x; e < COLS_PER * (RP / 4); e += LG_WARPS * 32) {
            const int cl = slice * COLS_PER + e / (RP / 4), j = (e % (RP / 4)) * 4;     // column inside the block, first of four ranks
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int k = 0; k < CL; ++k) {                     // slice order
                const float4 x = lg_ld_cluster_f32x4(peer[k] + (uint32_t)((cl * RP + j) * 4));
                v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
            }
            const int col = cb + cl;
            if (col >= C || j >= r) continue;                  // r is a multiple of 8: four ranks are all-in or all-out
            v.x *= sd.scale; v.y *= sd.scale; v.z *= sd.scale; v.w *= sd.scale;
            if (is_dB) {                                       // dB [C, r]
                float4* dst = reinterpret_cast<float4*>(sd.Out + (size_t)col * r + j);
                if (accumulate) { const float4 o = *dst; v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w; }
                *dst = v;
            } else {                                           // dA [r, C]
                float* dst = sd.Out + (size_t)j * C + col;
                if (accumulate) { v.x += dst[0]; v.y += dst[C]; v.z += dst[2 * (size_t)C]; v.w += dst[3 * (size_t)C]; }
                dst[0] = v.x; dst[C] = v.y; dst[2 * (size_t)C] = v.z; dst[3 * (size_t)C] = v.w;
            }
        }
        lg_cluster_sync();                                     // nobody leaves while a peer may still read its tile
        return;
    }
    float* part = sd.partial + (size_t)slice * C * r;
#pragma unroll
    for (int rt = 0; rt < RT; ++rt)
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int j = rt * 16 + g + ((i & 2) ? 8 : 0);
                const int col = cb + warp * 32 + q * 8 + 2 * c + (i & 1);
                if (col < C && j < r) part[(size_t)col * r + j] = acc[rt][c][i];
            }
}

// Adds the slices' partial sums in slice order.  Two forms; of the blocks the first are dB's, the others dA's.
//   reduce4: a thread takes four ranks of one column, neighbouring threads the next ranks of dB [N, r] (stored as it lies in scratch), the
//   next columns of dA [r, K] (its four stores are contiguous across the warp; its loads are not).
//   reduce: one element per thread as it lies in scratch, or four where there are plenty (2^18), dA stored through shared memory, a
//   block's columns of one rank together.
// The scattered loads are few at rank 8, where two threads share a sector, and at rank 16 while there are few slices; the line lies there.
// Gradient call, reduce4 / reduce by one / by four: 4096 x 4096, 2048 tokens, rank 8 12.65 / 12.97 / 13.7 us, rank 16 14.0 / 14.3 / 13.9,
// rank 32 19.0 / 16.7 / 17.2, rank 64 38.9 / 36.3 / 36.0; 4096 x 11008, 512 tokens, rank 64 23.3 / 24.8 / 22.8; 1024 x 1024, 1024 tokens
// (16 slices), rank 16 8.5 / 6.2 / 7.8.
constexpr int LR_THREADS = 256, LR4_MAX_SLICES = 9;

__device__ __forceinline__ float4 lg_add(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float lg_add(float a, float b) { return a + b; }
__device__ __forceinline__ float4 lg_scaled(float4 a, float s) { return make_float4(a.x * s, a.y * s, a.z * s, a.w * s); }
__device__ __forceinline__ float lg_scaled(float a, float s) { return a * s; }

// The sum over the slices, eight independent loads in flight.
template <typename V>
__device__ __forceinline__ V lg_slice_sum(const V* src, size_t step, int slices) {
    V v{};
    int sl = 0;
    for (; sl + 8 <= slices; sl += 8) {
        V x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = src[(sl + i) * step];
#pragma unroll
        for (int i = 0; i < 8; ++i) v = lg_add(v, x[i]);
    }
    if (sl + 4 <= slices) {
        V x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = src[(sl + i) * step];
#pragma unroll
        for (int i = 0; i < 4; ++i) v = lg_add(v, x[i]);
        sl += 4;
    }
    for (; sl < slices; ++sl) v = lg_add(v, src[sl * step]);
    return v;
}

template <int THREADS>
__global__ void __launch_bounds__(THREADS) lora_grad_reduce4_kernel(int r, int slices, int accumulate, int blocks_dB, GradSide dB_side, GradSide dA_side) {
    pdl_launch_dependents();
    const bool is_dB = (int)blockIdx.x < blocks_dB;
    const GradSide& sd = is_dB ? dB_side : dA_side;
    const int e = ((int)blockIdx.x - (is_dB ? 0 : blocks_dB)) * THREADS + (int)threadIdx.x, r4 = r >> 2;
    const int j = 4 * (is_dB ? e % r4 : e / sd.C), c = is_dB ? e / r4 : e % sd.C;
    pdl_wait();
    if (e >= sd.C * r4) return;
    const size_t C = (size_t)sd.C;
    float4 v = lg_scaled(lg_slice_sum(reinterpret_cast<const float4*>(sd.partial + (size_t)c * r + j), C * r / 4, slices), sd.scale);
    if (is_dB) {
        float4* dst = reinterpret_cast<float4*>(sd.Out + (size_t)c * r + j);
        if (accumulate) v = lg_add(*dst, v);
        *dst = v;
    } else {
        float* dst = sd.Out + (size_t)j * C + c;
        if (accumulate) { v.x = dst[0] + v.x; v.y = dst[C] + v.y; v.z = dst[2 * C] + v.z; v.w = dst[3 * C] + v.w; }
        dst[0] = v.x; dst[C] = v.y; dst[2 * C] = v.z; dst[3 * C] = v.w;
    }
}

template <int W>   // ranks per thread: 1 or 4
__global__ void __launch_bounds__(LR_THREADS / W) lora_grad_reduce_kernel(int r, int slices, int accumulate, int blocks_dB, GradSide dB_side, GradSide dA_side) {
    using V = std::conditional_t<W == 4, float4, float>;
    __shared__ __align__(16) float tile[LR_THREADS];           // dA: [column of the block][rank]
    pdl_launch_dependents();
    const bool is_dB = (int)blockIdx.x < blocks_dB;
    const GradSide& sd = is_dB ? dB_side : dA_side;
    const int cols = LR_THREADS / r, tid = threadIdx.x;        // columns of a block (threads beyond cols * r have no part)
    const int c0 = ((int)blockIdx.x - (is_dB ? 0 : blocks_dB)) * cols, n = min(cols, sd.C - c0) * r;
    const size_t e = (size_t)c0 * r + W * tid;
    pdl_wait();
    if (W * tid < n) {
        V v = lg_scaled(lg_slice_sum(reinterpret_cast<const V*>(sd.partial + e), (size_t)sd.C * r / W, slices), sd.scale);
        if (is_dB) {
            V* dst = reinterpret_cast<V*>(sd.Out + e);
            *dst = accumulate ? lg_add(*dst, v) : v;
        } else {
            *reinterpret_cast<V*>(tile + W * tid) = v;
        }
    }
    if (is_dB) return;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < W; ++i) {
        const int t = tid + i * (LR_THREADS / W), j = t / cols, cl = t - j * cols;
        if (j < r && cl * r < n) {
            float* dst = sd.Out + (size_t)j * sd.C + c0 + cl;
            const float v = tile[cl * r + j];
            *dst = accumulate ? *dst + v : v;
        }
    }
}

int launch_lora_grads(int M, int K, int N, int r, float s, const void* X, const void* dY, const float* H, const float* G,
                      float* dA, float* dB, int accumulate, void* scratch, cudaStream_t st, const uint8_t* x_mask, float keep_scale,
                      int sides) {
    if (r == 0) return QLORA_OK;
    const bool want_dB = (sides & 1) != 0 && N > 0, want_dA = (sides & 2) != 0 && K > 0;   // (a gradient without elements: nothing to do)
    if (!want_dB && !want_dA) return QLORA_OK;
    if (M == 0) {   // empty sums: dA = dB = 0 unless accumulating
        if (!accumulate) {
            if (want_dA && cudaMemsetAsync(dA, 0, (size_t)r * K * sizeof(float), st) != cudaSuccess) return QLORA_ERR_CUDA;
            if (want_dB && cudaMemsetAsync(dB, 0, (size_t)N * r * sizeof(float), st) != cudaSuccess) return QLORA_ERR_CUDA;
        }
        return QLORA_OK;
    }
    const int n_sides = (want_dB ? 1 : 0) + (want_dA ? 1 : 0);
    const int cols = want_dB && want_dA ? (N > K ? N : K) : (want_dB ? N : K);
    const int col_blocks = (cols + LG_COLS - 1) / LG_COLS;
    const int rt = (r + 15) / 16;
    const bool masked = want_dA && x_mask != nullptr;
    cudaError_t err = cudaSuccess;
    // Up to 256 tokens: one launch; the (at most four) 64-row slices of a column block form a cluster and reduce through
    // distributed shared memory.  (With more tokens, clusters of eight slices measured slower than free-floating blocks
    // plus a reduction launch: 19.6 against 13.4 us at 2048 tokens.)
    int cl = 4;
    while (cl > 1 && M <= 64 * (cl / 2)) cl /= 2;
    const int rows_cl = ((M + cl - 1) / cl + 63) / 64 * 64;
    if (M <= 256) {
        GradSide sB{(const __nv_bfloat16*)dY, H, nullptr, dB, N, nullptr, s, 1};
        GradSide sA{(const __nv_bfloat16*)X, G, nullptr, dA, K, x_mask, x_mask ? s * keep_scale : s, 0};
        if (!want_dB) sB = sA;                                  // one side only: it is the first (and only) z-slice of the grid
        const size_t pt_bytes = (size_t)rt * 16 * (rows_cl + 8) * sizeof(__nv_bfloat16), tile_bytes = (size_t)LG_COLS * rt * 16 * sizeof(float);
        const size_t smem = pt_bytes > tile_bytes ? pt_bytes : tile_bytes;
        const dim3 grid((unsigned)(col_blocks * cl), 1, (unsigned)n_sides);
#define QLORA_LGC_M(RTV, CLV, MK)                                                                              \
    do {                                                                                                       \
        static SmemLimit limit;                                                                                \
        if (!limit.raise(lora_grad_partial_kernel<RTV, CLV, MK>, (size_t)RTV * 16 * (1024 + 8) * 2)) return QLORA_ERR_CUDA; \
        err = launch_pdl(lora_grad_partial_kernel<RTV, CLV, MK>, grid, dim3(LG_WARPS * 32), smem, st, CLV, M, r, rows_cl, sB, sA, accumulate); \
    } while (0)
#define QLORA_LGC(RTV, CLV)                                                                                    \
    do { if (masked) QLORA_LGC_M(RTV, CLV, true); else QLORA_LGC_M(RTV, CLV, false); } while (0)
#define QLORA_LGC_RT(CLV)                                                                                      \
    switch (rt) {                                                                                              \
        case 1: QLORA_LGC(1, CLV); break;                                                                      \
        case 2: QLORA_LGC(2, CLV); break;                                                                      \
        case 3: QLORA_LGC(3, CLV); break;                                                                      \
        default: QLORA_LGC(4, CLV); break;                                                                     \
    }
        switch (cl) {
            case 4: QLORA_LGC_RT(4); break;
            case 2: QLORA_LGC_RT(2); break;
            default: QLORA_LGC_RT(1); break;
        }
#undef QLORA_LGC_RT
#undef QLORA_LGC
#undef QLORA_LGC_M
        return err == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
    }
    // More tokens: partial sums per row slice to scratch, then a reduction launch.
    GradPlan plan = lora_grad_plan(M, K, N);
    if (n_sides == 1) {
        // one gradient only: its column blocks alone would leave most SMs without a block, so the rows are cut finer -- as
        // fine as the scratch sized for both gradients allows
        const size_t room = (size_t)plan.slices * (size_t)(K + N);
        const int C1 = want_dB ? N : K;
        GradPlan one = lora_grad_plan(M, want_dB ? 0 : K, want_dB ? N : 0);
        while ((size_t)one.slices * C1 > room && one.rows_per_slice < 1024) {
            one.rows_per_slice += 64;
            one.slices = (M + one.rows_per_slice - 1) / one.rows_per_slice;
        }
        if ((size_t)one.slices * C1 <= room) plan = one;
    }
    float* part_dB = (float*)scratch;
    float* part_dA = n_sides == 1 ? part_dB : part_dB + (size_t)plan.slices * N * r;   // (alone, it starts at the base)
    GradSide sB{(const __nv_bfloat16*)dY, H, part_dB, dB, N, nullptr, s, 1};
    GradSide sA{(const __nv_bfloat16*)X, G, part_dA, dA, K, x_mask, x_mask ? s * keep_scale : s, 0};
    GradSide none{};                                         // C = 0: no elements for the reduction
    if (!want_dB) sB = sA;
    dim3 grid(col_blocks, plan.slices, (unsigned)n_sides);
    const size_t smem = (size_t)rt * 16 * (plan.rows_per_slice + 8) * sizeof(__nv_bfloat16);
#define QLORA_LG_M(RTV, MK)                                                                                    \
    do {                                                                                                       \
        static SmemLimit limit;                                                                                \
        if (!limit.raise(lora_grad_partial_kernel<RTV, 0, MK>, (size_t)RTV * 16 * (1024 + 8) * 2)) return QLORA_ERR_CUDA; \
        err = launch_pdl(lora_grad_partial_kernel<RTV, 0, MK>, grid, dim3(LG_WARPS * 32), smem, st, 1, M, r, plan.rows_per_slice, sB, sA, accumulate); \
    } while (0)
#define QLORA_LG(RTV)                                                                                          \
    do { if (masked) QLORA_LG_M(RTV, true); else QLORA_LG_M(RTV, false); } while (0)
    switch (rt) {
        case 1: QLORA_LG(1); break;
        case 2: QLORA_LG(2); break;
        case 3: QLORA_LG(3); break;
        default: QLORA_LG(4); break;
    }
#undef QLORA_LG
#undef QLORA_LG_M
    if (err != cudaSuccess) return QLORA_ERR_CUDA;
    const GradSide& rB = want_dB ? sB : none;
    const GradSide& rA = want_dA ? sA : none;
    const bool four = r == 8 || (r == 16 && plan.slices <= LR4_MAX_SLICES), wide = (size_t)(rB.C + rA.C) * r > (1u << 18);
    const int threads = four ? (r == 8 ? 64 : LR_THREADS) : (wide ? LR_THREADS / 4 : LR_THREADS), per = LR_THREADS / r;
    auto blocks = [&](int C) { return four ? (int)(((size_t)C * (r / 4) + threads - 1) / threads) : (C + per - 1) / per; };
    const dim3 red_grid((unsigned)(blocks(rB.C) + blocks(rA.C))), red_block((unsigned)threads);
    auto reduce = four ? (r == 8 ? lora_grad_reduce4_kernel<64> : lora_grad_reduce4_kernel<LR_THREADS>) : (wide ? lora_grad_reduce_kernel<4> : lora_grad_reduce_kernel<1>);
    err = launch_pdl(reduce, red_grid, red_block, 0, st, 1, r, plan.slices, accumulate, blocks(rB.C), rB, rA);
    return err == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
}

// ------------------------------------------------------------------------------------------------------------
// LoRA dropout, backward through the branch input: dX[m, k] += mask[m, k] * c * sum_j G[m, j] A[j, k]   (c = s * keep scale).
// The tensor-core kernels add the LoRA term inside the accumulator, where a per-element mask cannot be applied, so with
// dropout they run without the branch and this elementwise pass adds the masked term (dX is read and rounded once more).
// Bound by reading and writing dX and reading the mask (5 bytes per element).  One thread = 8 consecutive k of LU_ROWS token rows: A is
// read once for all of them (row by row it came from L2 64 KB at a time, 118 MB in all at 1800 tokens x 4096, rank 8: 16 us; now
// 12 us), and the loads of dX and the mask are all under way before the products.
// ------------------------------------------------------------------------------------------------------------
constexpr int LU_ROWS = 4;

__global__ void __launch_bounds__(256)
lora_masked_update_kernel(int M, int K, int r, float c, const float* __restrict__ G, const __nv_bfloat16* __restrict__ A,
                          const uint8_t* __restrict__ mask, __nv_bfloat16* __restrict__ dX) {
    pdl_launch_dependents();
    pdl_wait();
    const int kc = (int)(blockIdx.x * blockDim.x + threadIdx.x), k = kc * 8, m0 = (int)blockIdx.y * LU_ROWS;
    if (k >= K) return;
    uint4 xv[LU_ROWS];
    uint2 mb[LU_ROWS];
    float acc[LU_ROWS][8];
#pragma unroll
    for (int i = 0; i < LU_ROWS; ++i) {
        const bool in = m0 + i < M;
        xv[i] = in ? *reinterpret_cast<const uint4*>(dX + (size_t)(m0 + i) * K + k) : make_uint4(0, 0, 0, 0);
        mb[i] = in ? __ldg(reinterpret_cast<const uint2*>(mask + (size_t)(m0 + i) * K + k)) : make_uint2(0, 0);
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[i][e] = 0.f;
    }
    for (int j = 0; j < r; j += 4) {                           // (r is a multiple of 8)
        uint4 av[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) av[t] = __ldg(reinterpret_cast<const uint4*>(A + (size_t)(j + t) * K + k));
#pragma unroll
        for (int i = 0; i < LU_ROWS; ++i) {
            const float4 g4 = __ldg(reinterpret_cast<const float4*>(G + (size_t)min(m0 + i, M - 1) * r + j));
            const float g[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                acc[i][0] = fmaf(g[t], bf16_lo(av[t].x), acc[i][0]); acc[i][1] = fmaf(g[t], bf16_hi(av[t].x), acc[i][1]);
                acc[i][2] = fmaf(g[t], bf16_lo(av[t].y), acc[i][2]); acc[i][3] = fmaf(g[t], bf16_hi(av[t].y), acc[i][3]);
                acc[i][4] = fmaf(g[t], bf16_lo(av[t].z), acc[i][4]); acc[i][5] = fmaf(g[t], bf16_hi(av[t].z), acc[i][5]);
                acc[i][6] = fmaf(g[t], bf16_lo(av[t].w), acc[i][6]); acc[i][7] = fmaf(g[t], bf16_hi(av[t].w), acc[i][7]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < LU_ROWS; ++i) {
        if (m0 + i >= M || (mb[i].x | mb[i].y) == 0u) continue;
        const uint32_t xin[4] = {xv[i].x, xv[i].y, xv[i].z, xv[i].w}, mbytes[2] = {mb[i].x, mb[i].y};
        uint32_t o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const uint32_t m2 = mbytes[e >> 1] >> (16 * (e & 1));
            const float lo = bf16_lo(xin[e]) + ((m2 & 0xFFu) ? c * acc[i][2 * e] : 0.f);
            const float hi = bf16_hi(xin[e]) + ((m2 & 0xFF00u) ? c * acc[i][2 * e + 1] : 0.f);
            const __nv_bfloat162 pr = __floats2bfloat162_rn(lo, hi);
            o[e] = *reinterpret_cast<const uint32_t*>(&pr);
        }
        *reinterpret_cast<uint4*>(dX + (size_t)(m0 + i) * K + k) = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

int launch_lora_masked_update(int M, int K, int r, float c, const float* G, const void* A, const uint8_t* mask, void* dX,
                              cudaStream_t st) {
    if (M == 0 || K == 0 || r == 0) return QLORA_OK;
    cudaError_t err = cudaSuccess;
    for (int m = 0; m < M && err == cudaSuccess; m += 65535 * LU_ROWS) {       // (the grid's height has a limit)
        const int rows = M - m < 65535 * LU_ROWS ? M - m : 65535 * LU_ROWS;
        err = launch_pdl(lora_masked_update_kernel, dim3((unsigned)((K / 8 + 255) / 256), (unsigned)((rows + LU_ROWS - 1) / LU_ROWS)), dim3(256), 0, st, 1,
                         rows, K, r, c, G + (size_t)m * r, (const __nv_bfloat16*)A, mask + (size_t)m * K, (__nv_bfloat16*)dX + (size_t)m * K);
    }
    return err == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
}

}  // namespace qlora
