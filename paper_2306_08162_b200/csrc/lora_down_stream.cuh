// Streaming form of the LoRA down-projection for many token rows (included by umma_kernel.cu, inside its anonymous
// namespace, after the mbarrier helpers):
//   P[m, j] = sum_t In[m, t] * L(j, t)      L_IS_A: L = A [r, T] (contraction-contiguous), else L = B [T, r].
// A CTA of 15 warps owns up to LDS_MAXB blocks of 16 token rows.  The last warp streams the activation rows
// into a deep shared-memory ring with bulk copies (one per row and chunk of LDS_TC contraction elements, ~200 KB in
// flight per SM: the product is bound by the latency of cold reads, not by arithmetic); 14 consumer warps run
// mma.sync m16n8k16 on them.  The chunks are visited chunk-major, so a warp loads its adapter fragments once per chunk
// (from L2) and reuses them for all of the CTA's row blocks, whose accumulators it keeps in registers until the end;
// then the warps' partial tiles are added in warp order through shared memory.  The summation order of a row block
// depends on nothing but T, so every launch shape gives the same bits.
// Used (a) by the producer clusters of the CTA-pair kernel and (b) by lora_down_stream_kernel, the stand-alone launch
// ahead of the tensor-core kernels when they cannot host it (under a mask: lora_down_masked_kernel).

constexpr int LDS_TC = 1024;                              // contraction elements per ring stage
constexpr int LDS_ROW_BYTES = LDS_TC * 2 + 64;            // padded: rows 16 words apart (mod 32) -> conflict-free 16-byte fragment loads
constexpr int LDS_STAGE_BYTES = 16 * LDS_ROW_BYTES;       // 33 KiB
constexpr int LDS_MAXB = 8;                               // row blocks per CTA
constexpr int LDS_CWARPS = 14;                            // consumer warps (warp 14 issues the copies)
constexpr int LDS_STEPS = (LDS_TC / 32 + LDS_CWARPS - 1) / LDS_CWARPS;   // 32-wide contraction steps per warp and chunk
constexpr int LDS_BAR_BYTES = 256;                        // full[S] + empty[S] barriers behind the ring (S <= 16)
// Under dropout a stage carries the mask bytes of its rows behind them (rows 8 words apart (mod 32): conflict-free 8-byte loads).
constexpr int LDS_MASK_ROW_BYTES = LDS_TC + 32;
constexpr int LDS_MASKED_STAGE_BYTES = LDS_STAGE_BYTES + 16 * LDS_MASK_ROW_BYTES;

__device__ __forceinline__ void bulk_copy_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// Ring stages that the cross-warp reduction, which reuses the ring, takes.
constexpr int LDS_MIN_STAGES = (LDS_CWARPS * LDS_MAXB * 2 * 128 * 4 + LDS_STAGE_BYTES - 1) / LDS_STAGE_BYTES;   // room for the reduction

// Row blocks first_block, first_block + block_stride, ... (at most LDS_MAXB of them below ceil(M / 16)).
// Called by all threads of the CTA (15 warps or more; the first 15 work); `smem` is 128-byte aligned and holds `stages` ring stages with LDS_BAR_BYTES behind
// them; the ring is as large as LDS_MIN_STAGES plain stages at least.  Returns with no copy in flight (every issued stage has been waited for)
// unless the kernel is aborting.
// WITH_DB (backward only: In = dY [M, T = N], L = B): the rows that pass through for G = dY B also give this CTA's part of
//   dB[n, j] = sum_m dY[m, n] H[m, j]   (H fp32 [M, r], the forward's down-projection; the scale s is applied by whoever adds the parts up)
// as a second product per fragment: the tokens are now the contraction, so the 8 x 8 blocks of the dY fragments are
// transposed across the warp (movmatrix) into the 16-row operand and H supplies the 8-column one.  A warp owns the columns
// n of its own contraction steps, so nothing is summed across warps; its accumulators live for one chunk and are then
// written to dBpart [T, r] (fp32, this CTA's own: every n below T is written exactly once, provided the CTA has a row block).
// MASKED: `mask` (uint8 [M, T], non-zero = keep) is applied to In, and P is multiplied by out_scale (LoRA dropout).
template <bool L_IS_A, int NT, bool WITH_DB = false, int MAXB = LDS_MAXB, bool MASKED = false>   // MAXB: row blocks this instantiation keeps accumulators for
__device__ __forceinline__ void lora_down_stream(int M, int T, int r, const __nv_bfloat16* __restrict__ In,
                                                 const __nv_bfloat16* __restrict__ L, float* __restrict__ P, int first_block,
                                                 int block_stride, uint8_t* smem, int stages, volatile int* abort_flag,
                                                 const float* __restrict__ Hm = nullptr, float* __restrict__ dBpart = nullptr,
                                                 const uint8_t* __restrict__ mask = nullptr, float out_scale = 1.f) {
    static_assert(!(WITH_DB && L_IS_A), "dB rides on the backward's pass over dY");
    constexpr int STAGE = MASKED ? LDS_MASKED_STAGE_BYTES : LDS_STAGE_BYTES;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, q = lane & 3;
    const uint32_t ring = smem_u32(smem);
    const uint32_t bar_full = ring + (uint32_t)stages * STAGE;
    const uint32_t bar_empty = bar_full + 8u * (uint32_t)stages;
    const int n_blocks = (M + 15) / 16;
    int nb = first_block < n_blocks ? (n_blocks - first_block + block_stride - 1) / block_stride : 0;
    if (nb > MAXB) nb = MAXB;
    const int n_chunks = (T + LDS_TC - 1) / LDS_TC;

    if (threadIdx.x == 0) {
        for (int i = 0; i < stages; ++i) {
            mbar_init(bar_full + 8 * i, 1);
            mbar_init(bar_empty + 8 * i, LDS_CWARPS);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    float acc[MAXB][NT][4];
#pragma unroll
    for (int b = 0; b < MAXB; ++b)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) acc[b][nt][0] = acc[b][nt][1] = acc[b][nt][2] = acc[b][nt][3] = 0.f;

    if (warp == LDS_CWARPS) {
        // ---------------------------------------------------------------- copy issuer: lane 0 waits for the slot and posts
        // the byte count, then lane `row` issues the copy of that row (one thread issuing all 16 was the bottleneck)
        uint32_t slot = 0, phase = 0;
        bool live = true;
        for (int c = 0; c < n_chunks && live; ++c) {
            const int t0 = c * LDS_TC;
            const uint32_t row_bytes = (uint32_t)((T - t0 < LDS_TC ? T - t0 : LDS_TC) * 2);   // T % 8 == 0: a multiple of 16
            for (int b = 0; b < nb; ++b) {
                const int m0 = (first_block + b * block_stride) * 16;
                const int rows = M - m0 < 16 ? M - m0 : 16;
                uint32_t ok = 1;
                if (lane == 0) {
                    ok = mbar_wait(bar_empty + 8 * slot, phase ^ 1u, abort_flag) ? 1u : 0u;
                    if (ok) mbar_expect_tx(bar_full + 8 * slot, (MASKED ? row_bytes + row_bytes / 2 : row_bytes) * (uint32_t)rows);
                }
                ok = __shfl_sync(0xFFFFFFFFu, ok, 0);
                if (!ok) { live = false; break; }
                if (lane < rows) {
                    bulk_copy_g2s(ring + slot * STAGE + lane * LDS_ROW_BYTES, In + (size_t)(m0 + lane) * T + t0, row_bytes, bar_full + 8 * slot);
                    if constexpr (MASKED)
                        bulk_copy_g2s(ring + slot * STAGE + LDS_STAGE_BYTES + lane * LDS_MASK_ROW_BYTES, mask + (size_t)(m0 + lane) * T + t0,
                                      row_bytes / 2, bar_full + 8 * slot);
                }
                if (++slot == (uint32_t)stages) { slot = 0; phase ^= 1u; }
            }
        }
    } else if (warp < LDS_CWARPS) {
        // ---------------------------------------------------------------- consumers (warps beyond the issuer's have no part)
        uint32_t slot = 0, phase = 0;
        const uint4 zero4 = make_uint4(0, 0, 0, 0);
        bool live = true;
        for (int c = 0; c < n_chunks && live; ++c) {
            const int t0 = c * LDS_TC;
            const int chunk_len = T - t0 < LDS_TC ? T - t0 : LDS_TC;
            // this warp's adapter fragments of the chunk (steps warp, warp + 14, ...), reused for every row block
            uint4 lf[LDS_STEPS][NT];
#pragma unroll
            for (int i = 0; i < LDS_STEPS; ++i) {
                const int k0 = t0 + (warp + i * LDS_CWARPS) * 32;          // warp-uniform
                const int k = k0 + q * 8;
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    uint4 lv = zero4;
                    if ((warp + i * LDS_CWARPS) * 32 < chunk_len) {
                        if (L_IS_A) {
                            const int j = nt * 8 + g;
                            if (k < T && j < r) lv = __ldg(reinterpret_cast<const uint4*>(L + (size_t)j * T + k));
                        } else {
                            // 8 x 8 tiles of B loaded row-wise and transposed across the warp (see lora_down.cuh)
                            uint32_t w[4];
#pragma unroll
                            for (int t = 0; t < 4; ++t) {
                                const int n = k0 + 8 * (g >> 1) + (g & 1) + 2 * t;
                                uint32_t v = 0;
                                if (n < T && nt * 8 < r) v = __ldg(reinterpret_cast<const uint32_t*>(L + (size_t)n * r + nt * 8 + 2 * q));
                                w[t] = movmatrix_trans(v);
                            }
                            lv = make_uint4(w[0], w[1], w[2], w[3]);
                        }
                    }
                    lf[i][nt] = lv;
                }
            }
            float dbacc[WITH_DB ? LDS_STEPS : 1][2][NT][4];
            if constexpr (WITH_DB) {
#pragma unroll
                for (int i = 0; i < LDS_STEPS; ++i)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int nt = 0; nt < NT; ++nt) dbacc[i][h][nt][0] = dbacc[i][h][nt][1] = dbacc[i][h][nt][2] = dbacc[i][h][nt][3] = 0.f;
            }
#pragma unroll
            for (int b = 0; b < MAXB; ++b) {
                if (b < nb && live) {
                    uint32_t hb[NT][2];                                    // H rows of the block as the 8-column operand (tokens = contraction)
                    if constexpr (WITH_DB) {
                        const int mh = (first_block + b * block_stride) * 16 + 2 * q;
#pragma unroll
                        for (int nt = 0; nt < NT; ++nt) {
                            const int j = nt * 8 + g;
                            float h0 = 0.f, h1 = 0.f, h2 = 0.f, h3 = 0.f;
                            if (j < r) {
                                if (mh < M) h0 = Hm[(size_t)mh * r + j];
                                if (mh + 1 < M) h1 = Hm[(size_t)(mh + 1) * r + j];
                                if (mh + 8 < M) h2 = Hm[(size_t)(mh + 8) * r + j];
                                if (mh + 9 < M) h3 = Hm[(size_t)(mh + 9) * r + j];
                            }
                            const __nv_bfloat162 p0 = __floats2bfloat162_rn(h0, h1), p1 = __floats2bfloat162_rn(h2, h3);
                            hb[nt][0] = *reinterpret_cast<const uint32_t*>(&p0);
                            hb[nt][1] = *reinterpret_cast<const uint32_t*>(&p1);
                        }
                    }
                    if (!warp_wait(bar_full + 8 * slot, phase, abort_flag, lane)) { live = false; break; }
                    const int m0 = (first_block + b * block_stride) * 16;
                    const bool v0 = m0 + g < M, v1 = m0 + g + 8 < M;       // rows beyond M were not copied
                    const uint8_t* st = smem + slot * STAGE;
#pragma unroll
                    for (int i = 0; i < LDS_STEPS; ++i) {
                        const int kl = (warp + i * LDS_CWARPS) * 32;       // warp-uniform
                        if (kl < chunk_len) {
                            const int k = kl + q * 8;                      // chunk_len % 8 == 0: 8 elements are all-in or all-out
                            uint4 xlo = (v0 && k < chunk_len) ? *reinterpret_cast<const uint4*>(st + g * LDS_ROW_BYTES + k * 2) : zero4;
                            uint4 xhi = (v1 && k < chunk_len) ? *reinterpret_cast<const uint4*>(st + (g + 8) * LDS_ROW_BYTES + k * 2) : zero4;
                            if constexpr (MASKED) {
                                const uint8_t* ms = st + LDS_STAGE_BYTES + k;   // (bytes that were not copied meet a zero)
                                xlo = mask_eight(xlo, *reinterpret_cast<const uint2*>(ms + g * LDS_MASK_ROW_BYTES));
                                xhi = mask_eight(xhi, *reinterpret_cast<const uint2*>(ms + (g + 8) * LDS_MASK_ROW_BYTES));
                            }
#pragma unroll
                            for (int nt = 0; nt < NT; ++nt) {
                                mma_bf16_16816(acc[b][nt], xlo.x, xhi.x, xlo.y, xhi.y, lf[i][nt].x, lf[i][nt].y);
                                mma_bf16_16816(acc[b][nt], xlo.z, xhi.z, xlo.w, xhi.w, lf[i][nt].z, lf[i][nt].w);
                            }
                            if constexpr (WITH_DB) {
                                // transposed 8 x 8 blocks: lane (g, q) then holds tokens 2q, 2q + 1 (+ 8) of column
                                // kl + 8 (g >> 1) + (g & 1) + {0, 2, 4, 6} -- the rows of the two products below
                                const uint32_t t0x = movmatrix_trans(xlo.x), t0y = movmatrix_trans(xlo.y), t1x = movmatrix_trans(xhi.x), t1y = movmatrix_trans(xhi.y);
                                const uint32_t t0z = movmatrix_trans(xlo.z), t0w = movmatrix_trans(xlo.w), t1z = movmatrix_trans(xhi.z), t1w = movmatrix_trans(xhi.w);
#pragma unroll
                                for (int nt = 0; nt < NT; ++nt) {
                                    mma_bf16_16816(dbacc[i][0][nt], t0x, t0y, t1x, t1y, hb[nt][0], hb[nt][1]);
                                    mma_bf16_16816(dbacc[i][1][nt], t0z, t0w, t1z, t1w, hb[nt][0], hb[nt][1]);
                                }
                            }
                        }
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_empty + 8 * slot);
                    if (++slot == (uint32_t)stages) { slot = 0; phase ^= 1u; }
                }
            }
            if constexpr (WITH_DB) {
                // accumulator (i, h, nt): rows g / g + 8 = columns n and n + 2, n = step base + 4 h + 8 (g >> 1) + (g & 1); ranks 2q, 2q + 1
                if (live && nb > 0) {
#pragma unroll
                    for (int i = 0; i < LDS_STEPS; ++i) {
                        const int kl = (warp + i * LDS_CWARPS) * 32;
                        if (kl < chunk_len) {
#pragma unroll
                            for (int h = 0; h < 2; ++h)
#pragma unroll
                                for (int nt = 0; nt < NT; ++nt) {
                                    const int n = t0 + kl + 4 * h + 8 * (g >> 1) + (g & 1), j = nt * 8 + 2 * q;
                                    if (j < r) {
                                        if (n < T) *reinterpret_cast<float2*>(dBpart + (size_t)n * r + j) = make_float2(dbacc[i][h][nt][0], dbacc[i][h][nt][1]);
                                        if (n + 2 < T) *reinterpret_cast<float2*>(dBpart + (size_t)(n + 2) * r + j) = make_float2(dbacc[i][h][nt][2], dbacc[i][h][nt][3]);
                                    }
                                }
                        }
                    }
                }
            }
        }
    }
    __syncthreads();   // every stage has landed and been read: the ring is free for the reduction
    if (*abort_flag) return;
    float* red = reinterpret_cast<float*>(smem);   // [warp][b][nt][c][lane]
    if (warp < LDS_CWARPS) {
#pragma unroll
        for (int b = 0; b < MAXB; ++b)
            if (b < nb)
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int c = 0; c < 4; ++c) red[(((warp * LDS_MAXB + b) * NT + nt) * 4 + c) * 32 + lane] = acc[b][nt][c];
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < nb * NT * 128; idx += blockDim.x) {
        const int b = idx / (NT * 128), nt = (idx >> 7) % NT, c = (idx >> 5) & 3, ln = idx & 31;
        float v = 0.f;
        for (int w = 0; w < LDS_CWARPS; ++w) v += red[(((w * LDS_MAXB + b) * NT + nt) * 4 + c) * 32 + ln];
        const int row = (first_block + b * block_stride) * 16 + (ln >> 2) + ((c & 2) ? 8 : 0);
        const int col = nt * 8 + (ln & 3) * 2 + (c & 1);
        if (row < M && col < r) P[(size_t)row * r + col] = MASKED ? v * out_scale : v;
    }
    __syncthreads();
}

// Under a dropout mask the streaming order is taken from this many tokens on -- wherever the product is formed, so that saved and recomputed H have
// the same bits.  1800 tokens, 4096 x 4096, INT4, against a launch of lora_down_split_kernel ahead of the layer: dropout forward 58.9 -> 51.5 us
// (and backward, G beside the tiles, 71.0 -> 58.0).  Below, where the single-CTA kernel mostly runs and cannot host it, the split kernel is
// the shorter launch.  Ranks 17 to 32, seven warps per 16 of them, were timed and taken out: beside the tiles X A^T came to 57.9 -> 51.5 us at
// rank 32, but as a launch of its own (H recomputed for the gradients, 33 -> 43 us) the form is slower than the split kernel.
constexpr int LDS_MASKED_TOKENS = 1025;
static bool lds_masked(int M, int r) { return M >= LDS_MASKED_TOKENS && r <= 16; }

struct LdsParams {
    int M, T, r, stages, wait_limit_us;
    const uint8_t* mask;
    float out_scale;
    const __nv_bfloat16* In;
    const __nv_bfloat16* L;
    float* P;
};

template <bool L_IS_A>
__global__ void __launch_bounds__(kThreads, 1) lora_down_stream_kernel(const LdsParams p) {
    extern __shared__ uint8_t lds_raw[];
    __shared__ int abort_flag_s[2];   // [0] set when a wait gave up, [1] the wait limit in microseconds
    pdl_launch_dependents();
    uint8_t* smem = lds_raw + ((128u - (smem_u32(lds_raw) & 127u)) & 127u);
    if (threadIdx.x == 0) { abort_flag_s[0] = 0; abort_flag_s[1] = p.wait_limit_us; }
    __syncthreads();
    pdl_wait();
    const int first = (int)blockIdx.x, stride = (int)gridDim.x;
    if (p.r <= 8) {
        lora_down_stream<L_IS_A, 1>(p.M, p.T, p.r, p.In, p.L, p.P, first, stride, smem, p.stages, abort_flag_s);
    } else {
        lora_down_stream<L_IS_A, 2>(p.M, p.T, p.r, p.In, p.L, p.P, first, stride, smem, p.stages, abort_flag_s);
    }
    if (abort_flag_s[0]) {   // give copies that may still be in flight time to land before the CTA's memory is released
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
        __syncthreads();
    }
}

// The same product under a mask, as a launch of its own, bit for bit: the 14 partial sums of a row block are those of the ring form's warps, step by
// step, and are added in their order.  But that form has one CTA of 15 warps per row block or more, which waits for its first rows, for the adapter words
// of every chunk and for the slowest warp, and leaves SMs idle below 2368 tokens.  Here a warp loads DEPTH steps at a time straight into registers,
// and a row block's sums are spread as wide as keeps two CTAs of seven warps per SM: over two CTAs, eight rows to each pair of them (ROWS = 8) or
// sixteen; with more row blocks than SMs over one CTA, two sums to a warp (SUMS = 2).
// Gradients that recompute H, INT4, rank 8, microseconds -- lora_down_split_kernel (other bits) / the ring form / this: 4096 x 4096, 1100 tokens 15.1 / 19.7 /
// 15.9, 1800 tokens 23.1 / 25.3 / 23.6, 4096 tokens 39.0 / 46.4 / 39.3; 11008 -> 4096, 2048 tokens 41.3 / 52.9 / 42.2, 8192 tokens 134 / 203 / 142.
constexpr int LDO_WARPS = LDS_CWARPS / 2;

__device__ __forceinline__ float ld_cluster_f32(uint32_t cluster_addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(cluster_addr) : "memory");
    return v;
}

template <int NT, int SUMS, int ROWS>
__global__ void __launch_bounds__(LDO_WARPS * 32, 2)
lora_down_masked_kernel(const LdsParams p) {
    constexpr int DEPTH = NT == 1 ? 6 : 4, ELEMS = NT * 128, CTAS = 2 / SUMS;
    __shared__ float red[SUMS * LDO_WARPS * ELEMS];
    pdl_launch_dependents();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    const int rank = (int)blockIdx.x % CTAS, m_base = (int)blockIdx.x / CTAS * ROWS;
    const int steps = p.T >> 5;                                     // (K is a multiple of 32)
    const int r0 = m_base + g, r1 = r0 + 8;
    const bool v0 = r0 < p.M, v1 = ROWS > 8 && r1 < p.M;
    const size_t at0 = (size_t)r0 * p.T + q * 8, at1 = (size_t)r1 * p.T + q * 8;
    const __nv_bfloat16* l0 = p.L + (size_t)g * p.T + q * 8;
    const uint4 zero4 = make_uint4(0, 0, 0, 0);
    const uint2 zero2 = make_uint2(0, 0);
    float acc[SUMS][NT][4];
    int next[SUMS], left[SUMS], skip[SUMS];                         // per sum: its next step; steps left in the chunk; from its last step in a chunk to the next one's first
#pragma unroll
    for (int v = 0; v < SUMS; ++v) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) acc[v][nt][0] = acc[v][nt][1] = acc[v][nt][2] = acc[v][nt][3] = 0.f;
        next[v] = (SUMS == 2 ? v : rank) * LDO_WARPS + warp;        // the ring form's consumer warp: steps w, w + 14, w + 28 of every chunk of 32
        left[v] = (LDS_TC / 32 - next[v] + LDS_CWARPS - 1) / LDS_CWARPS;
        skip[v] = LDS_TC / 32 - (left[v] - 1) * LDS_CWARPS;
    }
    int per_chunk[SUMS];
#pragma unroll
    for (int v = 0; v < SUMS; ++v) per_chunk[v] = left[v];
    pdl_wait();
#pragma unroll 1
    while (next[0] < steps || next[SUMS - 1] < steps) {
        uint4 xlo[DEPTH], xhi[DEPTH], l[DEPTH][NT];
        uint2 mlo[DEPTH], mhi[DEPTH];
        uint32_t in = 0;                                            // bit u: step u exists (warp-uniform)
#pragma unroll
        for (int u = 0; u < DEPTH; ++u) {
            const int v = u % SUMS, k = next[v] * 32;
            const bool ok = next[v] < steps;
            if (ok) in |= 1u << u;
            xlo[u] = v0 && ok ? __ldg(reinterpret_cast<const uint4*>(p.In + at0 + k)) : zero4;
            xhi[u] = v1 && ok ? __ldg(reinterpret_cast<const uint4*>(p.In + at1 + k)) : zero4;
            mlo[u] = v0 && ok ? __ldg(reinterpret_cast<const uint2*>(p.mask + at0 + k)) : zero2;
            mhi[u] = v1 && ok ? __ldg(reinterpret_cast<const uint2*>(p.mask + at1 + k)) : zero2;
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) l[u][nt] = ok && nt * 8 < p.r ? __ldg(reinterpret_cast<const uint4*>(l0 + (size_t)nt * 8 * p.T + k)) : zero4;
            const bool last = --left[v] == 0;
            next[v] += last ? skip[v] : LDS_CWARPS;
            if (last) left[v] = per_chunk[v];
        }
#pragma unroll
        for (int u = 0; u < DEPTH; ++u) {
            if (!(in >> u & 1u)) continue;
            xlo[u] = mask_eight(xlo[u], mlo[u]);
            xhi[u] = mask_eight(xhi[u], mhi[u]);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                mma_bf16_16816(acc[u % SUMS][nt], xlo[u].x, xhi[u].x, xlo[u].y, xhi[u].y, l[u][nt].x, l[u][nt].y);
                mma_bf16_16816(acc[u % SUMS][nt], xlo[u].z, xhi[u].z, xlo[u].w, xhi[u].w, l[u][nt].z, l[u][nt].w);
            }
        }
    }
#pragma unroll
    for (int v = 0; v < SUMS; ++v)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int c = 0; c < 4; ++c) red[(v * LDO_WARPS + warp) * ELEMS + (nt * 4 + c) * 32 + lane] = acc[v][nt][c];
    __syncwarp();
    if (CTAS == 2) cluster_sync_all();
    else __syncthreads();
    const uint32_t part0 = CTAS == 2 ? map_to_cta(smem_u32(red), 0) : 0u, part1 = CTAS == 2 ? map_to_cta(smem_u32(red), 1) : 0u;
    for (int e = rank * (ELEMS / CTAS) + (int)threadIdx.x; e < (rank + 1) * (ELEMS / CTAS); e += LDO_WARPS * 32) {
        float x[LDS_CWARPS], y = 0.f;
#pragma unroll
        for (int w = 0; w < LDS_CWARPS; ++w)
            x[w] = CTAS == 2 ? ld_cluster_f32((w < LDO_WARPS ? part0 : part1) + (uint32_t)((w % LDO_WARPS) * ELEMS + e) * 4u) : red[(w % (SUMS * LDO_WARPS)) * ELEMS + e];
#pragma unroll
        for (int w = 0; w < LDS_CWARPS; ++w) y += x[w];
        const int nt = e >> 7, c = (e >> 5) & 3, ln = e & 31;
        const int row = m_base + (ln >> 2) + ((c & 2) ? 8 : 0), col = nt * 8 + (ln & 3) * 2 + (c & 1);
        if (row < p.M && col < p.r && (ROWS > 8 || c < 2)) p.P[(size_t)row * p.r + col] = y * p.out_scale;
    }
    if (CTAS == 2) {
        __syncwarp();
        cluster_sync_all();                                         // nobody leaves while its peer may still read its parts
    }
}

template <int NT>
cudaError_t launch_lora_down_masked(const LdsParams& p, cudaStream_t st) {
    const unsigned sms = (unsigned)sm_count(), eights = (unsigned)((p.M + 7) / 8), blocks = (unsigned)((p.M + 15) / 16);
    const dim3 block(LDO_WARPS * 32);
    if (eights <= sms) return launch_pdl(lora_down_masked_kernel<NT, 1, 8>, dim3(2 * eights), block, 0, st, 2, p);
    if (blocks <= sms) return launch_pdl(lora_down_masked_kernel<NT, 1, 16>, dim3(2 * blocks), block, 0, st, 2, p);
    return launch_pdl(lora_down_masked_kernel<NT, 2, 16>, dim3(blocks), block, 0, st, 1, p);
}

// Stand-alone launch (r <= 16): one CTA per SM at most, each with up to LDS_MAXB row blocks; under a mask the kernel above.
int launch_lora_down_stream_impl(int M, int T, int r, bool l_is_A, const void* In, const void* L, float* P, cudaStream_t st, const uint8_t* mask,
                                 float out_scale) {
    if (M == 0 || r == 0) return QLORA_OK;
    const int n_blocks = (M + 15) / 16;
    int grid = n_blocks < sm_count() ? n_blocks : sm_count();
    if ((n_blocks + grid - 1) / grid > LDS_MAXB) grid = (n_blocks + LDS_MAXB - 1) / LDS_MAXB;   // several waves of CTAs
    LdsParams p{};
    p.M = M; p.T = T; p.r = r; p.stages = 6; p.wait_limit_us = kWaitLimitUs;
    p.In = (const __nv_bfloat16*)In; p.L = (const __nv_bfloat16*)L; p.P = P;
    p.mask = mask; p.out_scale = out_scale;
    if (mask != nullptr) {
        const cudaError_t err = r <= 8 ? launch_lora_down_masked<1>(p, st) : launch_lora_down_masked<2>(p, st);
        return err == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
    }
    constexpr size_t smem_bytes = 6 * LDS_STAGE_BYTES + LDS_BAR_BYTES + 128;
    static SmemLimit limit_a, limit_b;
    if (!limit_a.raise(lora_down_stream_kernel<true>, smem_bytes) || !limit_b.raise(lora_down_stream_kernel<false>, smem_bytes)) return QLORA_ERR_CUDA;
    const cudaError_t err = l_is_A ? launch_pdl(lora_down_stream_kernel<true>, dim3((unsigned)grid), dim3(kThreads), smem_bytes, st, 1, p)
                                   : launch_pdl(lora_down_stream_kernel<false>, dim3((unsigned)grid), dim3(kThreads), smem_bytes, st, 1, p);
    return err == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
}
