// LoRA down-projection of one or two blocks of 16 token rows, as a device function shared by the stand-alone kernel for up to 256
// rows (simt_kernels.cu) and by the single-CTA tensor-core kernel, whose spare clusters run it beside the main tiles.
//   P[m, j] = sum_t In[m, t] * L(j, t)     l_is_A: L = A [r, T] (contraction-contiguous), else L = B [T, r].
// mma.sync m16n8k16 (bf16 in, fp32 accumulate) fed straight from 16-byte row loads: the warps of the block stride over
// the contraction in steps of 32 and keep UNROLL steps of loads in flight, the adapter's among them.  The 32 contraction indices of a step are
// assigned to the fragments in a permuted order (lane q of a quad owns indices 8q..8q+7); activation and adapter fragments
// use the same permutation, so the sum is unchanged.  A is contraction-contiguous and loads directly; B is rank-contiguous,
// so its 8 x 8 fragment tiles are loaded row-wise and transposed across the warp with movmatrix.  The per-warp partial
// tiles are added in warp order through shared memory (fixed order: deterministic for a given number of warps).
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

namespace qlora {

__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                               uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// LoRA dropout: keep the bf16 pair elements whose mask byte is non-zero (mask bytes m0, m1 in the low two bytes of `mb`).
__device__ __forceinline__ uint32_t mask_pair(uint32_t pair, uint32_t mb) {
    return pair & (((mb & 0xFFu) ? 0x0000FFFFu : 0u) | ((mb & 0xFF00u) ? 0xFFFF0000u : 0u));
}
// Eight bf16 (uint4) against eight mask bytes (uint2).
__device__ __forceinline__ uint4 mask_eight(uint4 x, uint2 m) {
    return make_uint4(mask_pair(x.x, m.x), mask_pair(x.y, m.x >> 16), mask_pair(x.z, m.y), mask_pair(x.w, m.y >> 16));
}
// Transpose an 8 x 8 matrix of 16-bit elements held across the warp (lane l: row l / 4, elements 2 (l % 4), +1).
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t a) {
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}

// Rows m_base .. m_base + 15 and, with NB = 2, the block of rows `block_stride` further on (beside the first: the same adapter words serve
// both).  Called by all `nwarps` warps of a block (it synchronises the block twice); `red` is shared memory for nwarps * NB * NT * 128
// floats.  L is read through the read-only path, and so is In.  UNROLL: as many steps as the registers hold, 8 NB + 4 NT of them each
// (with 1024 threads, four steps at NT = 2 spilled 150 bytes and took 1.3 to 1.8 times as long).
template <bool L_IS_A, int NT, int NB, int UNROLL>
__device__ __forceinline__ void lora_down_rows(int M, int T, int r, const __nv_bfloat16* __restrict__ In,
                                               const __nv_bfloat16* __restrict__ L, float* __restrict__ P, int m_base, int block_stride, int nwarps,
                                               float* red) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, q = lane & 3;
    float acc[NB][NT][4];
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) acc[b][nt][0] = acc[b][nt][1] = acc[b][nt][2] = acc[b][nt][3] = 0.f;
    const uint4 zero4 = make_uint4(0, 0, 0, 0);
    const int wstride = nwarps * 32;
#pragma unroll 1
    for (int kk = warp * 32; kk < T; kk += wstride * UNROLL) {
        uint4 xlo[NB][UNROLL], xhi[NB][UNROLL], l[UNROLL][NT];
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {                 // all loads of the unrolled steps first
            const int k0 = kk + u * wstride, k = k0 + q * 8;  // T is a multiple of 8: 8 elements are all-in or all-out
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const int r0 = m_base + b * block_stride + g, r1 = r0 + 8;
                xlo[b][u] = (r0 < M && k < T) ? __ldg(reinterpret_cast<const uint4*>(In + (size_t)r0 * T + k)) : zero4;
                xhi[b][u] = (r1 < M && k < T) ? __ldg(reinterpret_cast<const uint4*>(In + (size_t)r1 * T + k)) : zero4;
            }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                uint4 lv = zero4;
                if (L_IS_A) {
                    const int j = nt * 8 + g;                  // rank index of this lane's adapter fragment
                    if (k < T && j < r) lv = __ldg(reinterpret_cast<const uint4*>(L + (size_t)j * T + k));   // A[j, k..k+7]
                } else if (nt * 8 < r) {
                    // tile t: row rho (0..7) <-> n = k0 + 8 (rho / 2) + (rho % 2) + 2 t, columns = ranks 8 nt .. 8 nt + 7
                    const int n = k0 + 8 * (g >> 1) + (g & 1);
                    if (n < T) {
                        const __nv_bfloat16* src = L + (size_t)n * r + nt * 8 + 2 * q;
                        lv = make_uint4(__ldg(reinterpret_cast<const uint32_t*>(src)), __ldg(reinterpret_cast<const uint32_t*>(src + 2 * r)),
                                        __ldg(reinterpret_cast<const uint32_t*>(src + 4 * r)), __ldg(reinterpret_cast<const uint32_t*>(src + 6 * r)));
                    }
                }
                l[u][nt] = lv;
            }
        }
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
            if (kk + u * wstride >= T) break;                  // warp-uniform
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                uint4 lv = l[u][nt];
                // after the transpose lane (g, q) holds B[k0 + 8q + 2t, 8nt + g], B[k0 + 8q + 2t + 1, 8nt + g]
                if (!L_IS_A) lv = make_uint4(movmatrix_trans(lv.x), movmatrix_trans(lv.y), movmatrix_trans(lv.z), movmatrix_trans(lv.w));
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    mma_bf16_16816(acc[b][nt], xlo[b][u].x, xhi[b][u].x, xlo[b][u].y, xhi[b][u].y, lv.x, lv.y);
                    mma_bf16_16816(acc[b][nt], xlo[b][u].z, xhi[b][u].z, xlo[b][u].w, xhi[b][u].w, lv.z, lv.w);
                }
            }
        }
    }
    // red[warp][b][nt][c][lane]
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int c = 0; c < 4; ++c) red[(((warp * NB + b) * NT + nt) * 4 + c) * 32 + lane] = acc[b][nt][c];
    __syncthreads();
    for (int idx = threadIdx.x; idx < NB * NT * 128; idx += wstride) {
        const int b = idx / (NT * 128), nt = (idx >> 7) % NT, c = (idx >> 5) & 3, ln = idx & 31;
        float v = 0.f;
        for (int w = 0; w < nwarps; ++w) v += red[(((w * NB + b) * NT + nt) * 4 + c) * 32 + ln];
        const int row = m_base + b * block_stride + (ln >> 2) + ((c & 2) ? 8 : 0);
        const int col = nt * 8 + (ln & 3) * 2 + (c & 1);
        if (row < M && col < r) P[(size_t)row * r + col] = v;
    }
    __syncthreads();   // `red` may be rewritten by the next call
}

}  // namespace qlora
