// Fused LREC training loss (Section 3.2, Eq. 1-2 of the paper): per token, with student logits z (the quantized model with
// its LoRA pairs) and cached teacher logits t (the frozen full-precision model),
//     loss = lambda_KL * KL(softmax(z) || softmax(t)) + lambda_CE * ( -log softmax(z)[label] )
// and its gradient with respect to z, in one pass over the two [T, V] logit matrices:
//     d KL / d z_j = p_j * ((log p_j - log q_j) - KL),      d CE / d z_j = p_j - [j == label]        (p = softmax(z), q = softmax(t))
// Bound by HBM traffic (read 2 * V * 2 bytes, write V * 2 bytes per token), so a token row is read once: a block holds both rows
// entirely in registers (CH chunks of 8 bf16 per thread and matrix) and writes the gradient from the same registers.
// What the SM has to do per logit pair has to stay below the time of its 6 bytes (a row of 32000: 4.3 us per SM at the copy rate),
// so:
//   - exponentials use the hardware ex2 path (relative error ~2^-22 on the arguments <= 0 that occur here) and the KL sum shares the
//     exp-sum pass: three per logit pair, 3.1 us a row, the special-function unit's share;
//   - fp32 arithmetic on pairs (f32x2), maxima on bf16 pairs as they lie in memory;
//   - every warp sums relative to ITS OWN maxima, so a row has one block-wide exchange (maxima and sums together, one
//     barrier) instead of five, and the warps of a block drift: some load and exponentiate the next row while others store;
//   - 1024 threads per SM in as many blocks as the row length allows (grid_plan).
// One SM's worth of rows fills the register file; to keep HBM busy meanwhile, every thread prefetches ITS OWN chunks of the block's
// next row into shared memory with cp.async (thread-private slots: no barrier is involved, the thread just waits for its own
// copies) and moves them to registers when the row's turn comes.
// T = 2048, V = 32000: 111 -> 89 us (4.4 TB/s, 0.68 of the measured copy bandwidth).
#include "common.cuh"
#include "device_state.h"
#include "launch.h"

namespace qlora {

constexpr int LL_MAX_THREADS = 1024;

// 2^x on the special-function unit (relative error about 2^-22; results below the normal range flush to zero).
__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Two fp32 values in a register pair.
struct f2 { uint64_t v; };
__device__ __forceinline__ f2 make_f2(float lo, float hi) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float lo_of(f2 a) { return __uint_as_float((uint32_t)a.v); }
__device__ __forceinline__ float hi_of(f2 a) { return __uint_as_float((uint32_t)(a.v >> 32)); }
__device__ __forceinline__ f2 unpack_bf16(uint32_t w) { return make_f2(bf16_lo(w), bf16_hi(w)); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 exp2_2(f2 a) { return make_f2(fast_exp2(lo_of(a)), fast_exp2(hi_of(a))); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}

template <int CH>   // 16-byte chunks (8 bf16) per thread and matrix
__global__ void __launch_bounds__(LL_MAX_THREADS, 1)
lrec_loss_kernel(int T, int V, const __nv_bfloat16* __restrict__ Z, const __nv_bfloat16* __restrict__ Tt,
                 const int32_t* __restrict__ labels, float lambda_kl, float lambda_ce, float grad_scale,
                 float* __restrict__ loss_tokens, __nv_bfloat16* __restrict__ dZ) {
    __shared__ float part[2][5][32];                            // per warp: max z, max t, sum e_z, sum e_t, sum e_z (z - t); two rows' worth
    extern __shared__ __align__(16) uint8_t ll_smem[];          // [2][CH][threads] uint4: next row of Z and of Tt
    const int threads = blockDim.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = threads >> 5;
    uint4* stage_z = reinterpret_cast<uint4*>(ll_smem) + threadIdx.x;
    uint4* stage_t = stage_z + CH * threads;
    pdl_launch_dependents();
    pdl_wait();
    const int chunks = V / 8;
    auto prefetch = [&](int row) {                              // this thread's chunks of `row` -> its shared-memory slots
        const uint4* zr = reinterpret_cast<const uint4*>(Z + (size_t)row * V);
        const uint4* tr = reinterpret_cast<const uint4*>(Tt + (size_t)row * V);
#pragma unroll
        for (int c = 0; c < CH; ++c) {
            const int ci = c * threads + threadIdx.x;
            if (ci < chunks) {
                const uint32_t dz = (uint32_t)__cvta_generic_to_shared(stage_z + c * threads), dt = (uint32_t)__cvta_generic_to_shared(stage_t + c * threads);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dz), "l"(zr + ci) : "memory");
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dt), "l"(tr + ci) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    constexpr float kLog2e = 1.4426950408889634f, kAzScale = 0x1p-16f;   // (a row has 2^15 terms)
    const f2 log2e2 = make_f2(kLog2e, kLog2e), scale2 = make_f2(kAzScale, kAzScale), minus1 = make_f2(-1.f, -1.f);
    if ((int)blockIdx.x < T) prefetch(blockIdx.x);
    // Gradient: what grad_scale * lambda_kl has above 1 goes into the exponent of p_j as a power of two; on a masked logit's z - t it would
    // overflow, and p_j = 0 must give 0.
    const float g_all = grad_scale * lambda_kl;
    const int n_up = fabsf(g_all) > 1.f ? min(ilogbf(g_all), 125) + 1 : 0;
    const float up_inv = __uint_as_float((uint32_t)(127 - n_up) << 23), gkl = g_all * up_inv;
    int buf = 0;
    for (int row = blockIdx.x; row < T; row += gridDim.x, buf ^= 1) {
        uint4 zc[CH], tc[CH];
        const uint4 neg = make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u);   // bf16 -inf pairs: padding
        const int label = labels != nullptr ? __ldg(labels + row) : -1;
        asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
        for (int c = 0; c < CH; ++c) {
            const int ci = c * threads + threadIdx.x;
            zc[c] = ci < chunks ? stage_z[c * threads] : neg;
            tc[c] = ci < chunks ? stage_t[c * threads] : neg;
        }
        if (row + (int)gridDim.x < T) prefetch(row + gridDim.x);   // overlaps everything below
        // this warp's maxima (exact in bf16)
        __nv_bfloat162 mz2v = *reinterpret_cast<const __nv_bfloat162*>(&neg.x), mt2v = mz2v;
#pragma unroll
        for (int c = 0; c < CH; ++c) {
            const uint32_t zw[4] = {zc[c].x, zc[c].y, zc[c].z, zc[c].w}, tw[4] = {tc[c].x, tc[c].y, tc[c].z, tc[c].w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                mz2v = __hmax2(mz2v, *reinterpret_cast<const __nv_bfloat162*>(&zw[i]));
                mt2v = __hmax2(mt2v, *reinterpret_cast<const __nv_bfloat162*>(&tw[i]));
            }
        }
        __nv_bfloat162 mzt = __hmax2(__lows2bfloat162(mz2v, mt2v), __highs2bfloat162(mz2v, mt2v));   // (max z, max t)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mzt = __hmax2(mzt, __shfl_xor_sync(0xFFFFFFFFu, mzt, o));
        const float mz_w = __low2float(mzt), mt_w = __high2float(mzt);
        // One pass gives both exp-sums and the KL numerator: with e_j = exp(z_j - mz) and sz = sum e_j,
        //   KL = sum_j (e_j / sz) ((z_j - lz) - (t_j - lt)) = (sum_j e_j (z_j - t_j)) / sz - lz + lt        (lz = mz + log sz, ...)
        // (padding: z = t = -inf would give 0 * nan, so padded chunks are skipped rather than relied on to vanish)
        // Masked logits (finfo.min, -1e30) can be all that a warp holds.  From 2^16 on two different bf16 lie 256 or more apart, so
        // exp(z - mz) is 1 or 0 in any base, and in base 2 the difference is exact, where mz log2(e) would be rounded by more than 2^-8 or
        // overflow.  Their z - t times a weight of 1 (relative to the warp's own maximum) is summed scaled, so that it stays finite.
        // (No branch for them: one in this place kept the gradient's first steps from moving up between the shuffles, 86 -> 88 us.)
        const float kz = fabsf(mz_w) < 65536.f ? kLog2e : 1.f, kt = fabsf(mt_w) < 65536.f ? kLog2e : 1.f;
        const float rz = mz_w == -INFINITY ? 0.f : -mz_w * kz, rt = mt_w == -INFINITY ? 0.f : -mt_w * kt;   // (a warp with nothing finite)
        const f2 kz2 = make_f2(kz, kz), kt2 = make_f2(kt, kt), rz2 = make_f2(rz, rz), rt2 = make_f2(rt, rt);
        f2 sz2 = make_f2(0.f, 0.f), st2 = sz2, az2 = sz2;
#pragma unroll
        for (int c = 0; c < CH; ++c) {
            if (c * threads + (int)threadIdx.x < chunks) {
                const uint32_t zw[4] = {zc[c].x, zc[c].y, zc[c].z, zc[c].w}, tw[4] = {tc[c].x, tc[c].y, tc[c].z, tc[c].w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const f2 z = unpack_bf16(zw[i]), t = unpack_bf16(tw[i]);
                    const f2 e = exp2_2(fma2(z, kz2, rz2));
                    sz2 = add2(sz2, e);
                    az2 = fma2(mul2(e, scale2), fma2(t, minus1, z), az2);
                    st2 = add2(st2, exp2_2(fma2(t, kt2, rt2)));
                }
            }
        }
        const float sz_w = warp_sum(lo_of(sz2) + hi_of(sz2)), st_w = warp_sum(lo_of(st2) + hi_of(st2)), az_w = warp_sum(lo_of(az2) + hi_of(az2));
        if (lane == 0) {
            part[buf][0][warp] = mz_w; part[buf][1][warp] = mt_w;
            part[buf][2][warp] = sz_w; part[buf][3][warp] = st_w; part[buf][4][warp] = az_w;
        }
        __syncthreads();                                        // (the next row uses the other buffer: one barrier a row)
        // every warp combines the partial results in the same order: lane l takes warp l's
        const bool has = lane < nwarps;
        const float pz = has ? part[buf][0][lane] : -INFINITY, pt = has ? part[buf][1][lane] : -INFINITY;
        const float mz = warp_max(pz), mt = warp_max(pt);
        const float fz = pz == -INFINITY ? 0.f : fast_exp2((pz - mz) * kLog2e), ft = pt == -INFINITY ? 0.f : fast_exp2((pt - mt) * kLog2e);
        const float sz = warp_sum(has ? part[buf][2][lane] * fz : 0.f), st = warp_sum(has ? part[buf][3][lane] * ft : 0.f);
        const float az = warp_sum(has ? part[buf][4][lane] * fz : 0.f);
        const float lz = mz + logf(sz), lt = mt + logf(st);       // log-partition functions: log p_j = z_j - lz
        const float kl = az / sz * (1.f / kAzScale) - lz + lt;
        const bool has_label = label >= 0 && label < V;
        const int label_chunk = has_label ? label >> 3 : -1;
        if (!has_label && threadIdx.x == 0) loss_tokens[row] = lambda_kl * kl;
        uint4* dr = dZ != nullptr ? reinterpret_cast<uint4*>(dZ + (size_t)row * V) : nullptr;
        // g_j = p_j (lambda_kl ((z_j - t_j) - (lz - lt) - KL) + lambda_ce) - lambda_ce [j == label], times grad_scale
        const float nshift = -((lz - lt) + kl), nlz = fmaf(-lz, kLog2e, (float)n_up), gce = has_label ? grad_scale * lambda_ce : 0.f, gce_n = gce * up_inv;
        const f2 nshift2 = make_f2(nshift, nshift), nlz2 = make_f2(nlz, nlz), gkl2 = make_f2(gkl, gkl), gce2 = make_f2(gce_n, gce_n);
#pragma unroll
        for (int c = 0; c < CH; ++c) {
            const int ci = c * threads + threadIdx.x;
            const uint32_t zw[4] = {zc[c].x, zc[c].y, zc[c].z, zc[c].w}, tw[4] = {tc[c].x, tc[c].y, tc[c].z, tc[c].w};
            if (ci == label_chunk) {                            // the thread that holds the label's logit: -log p_label = lz - z_label
                const int wi = (label >> 1) & 3;
                const uint32_t w = wi == 0 ? zw[0] : (wi == 1 ? zw[1] : (wi == 2 ? zw[2] : zw[3]));
                loss_tokens[row] = lambda_kl * kl + lambda_ce * (lz - ((label & 1) ? bf16_hi(w) : bf16_lo(w)));
            }
            if (dr != nullptr && ci < chunks) {
                uint32_t o[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const f2 z = unpack_bf16(zw[i]), t = unpack_bf16(tw[i]);
                    const f2 pj = exp2_2(fma2(z, log2e2, nlz2));
                    f2 gr = mul2(pj, fma2(gkl2, add2(fma2(t, minus1, z), nshift2), gce2));
                    if (ci == label_chunk && i == ((label >> 1) & 3)) gr = add2(gr, (label & 1) ? make_f2(0.f, -gce) : make_f2(-gce, 0.f));
                    const __nv_bfloat162 pr = __floats2bfloat162_rn(lo_of(gr), hi_of(gr));
                    o[i] = *reinterpret_cast<const uint32_t*>(&pr);
                }
                __stcs(dr + ci, make_uint4(o[0], o[1], o[2], o[3]));
            }
        }
    }
}

// Chunks per thread (1 .. 4) and threads per block for rows of `chunks` chunks.  More rows than SMs: the register file holds 1024 threads of
// this kernel, so the choice is the one with the most blocks per SM, then the one with the most threads.  Fewer: the most threads, a
// row is done soonest (64 rows of 8192: 5.9 us with 256 threads, 4.1 with 1024).
static void grid_plan(int T, int chunks, int sms, int& ch, int& threads, int& per_sm) {
    ch = 4; threads = 0; per_sm = 0;
    for (int c = 4; c >= 1; --c) {
        const int t = (chunks + 32 * c - 1) / (32 * c) * 32;
        if (t > LL_MAX_THREADS) break;
        int n = LL_MAX_THREADS / t;
        if (n > 16) n = 16;
        if (T <= sms || n >= per_sm) { ch = c; threads = t; per_sm = n; }
    }
}

int launch_lrec_loss(int T, int V, const void* Z, const void* Tt, const int32_t* labels, float lambda_kl, float lambda_ce,
                     float grad_scale, float* loss_tokens, void* dZ, cudaStream_t st) {
    if (T == 0) return QLORA_OK;
    int ch, threads, per_sm;
    const int sms = sm_count();
    grid_plan(T, V / 8, sms, ch, threads, per_sm);
    if (threads == 0) return QLORA_ERR_UNSUPPORTED;
    const int slots = sms * per_sm;
    const unsigned grid = (unsigned)(T < slots ? T : slots);     // persistent over the rows
    const size_t smem = (size_t)2 * ch * threads * 16;
    cudaError_t err;
#define QLORA_LL(CHV)                                                                                                  \
    {                                                                                                                  \
        static SmemLimit limit;                                                                                        \
        if (!limit.raise(lrec_loss_kernel<CHV>, (size_t)2 * CHV * LL_MAX_THREADS * 16)) return QLORA_ERR_CUDA;         \
    }                                                                                                                  \
    err = launch_pdl(lrec_loss_kernel<CHV>, dim3(grid), dim3((unsigned)threads), smem, st, 1, T, V, (const __nv_bfloat16*)Z, \
                     (const __nv_bfloat16*)Tt, labels, lambda_kl, lambda_ce, grad_scale, loss_tokens, (__nv_bfloat16*)dZ)
    if (ch == 1) { QLORA_LL(1); }
    else if (ch == 2) { QLORA_LL(2); }
    else if (ch == 3) { QLORA_LL(3); }
    else { QLORA_LL(4); }
#undef QLORA_LL
    return err == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
}

}  // namespace qlora
