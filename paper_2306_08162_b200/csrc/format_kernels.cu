// Pack / unpack / full dequantisation of the bit-packed INT32 weight matrix (Section 3.1 of the paper:
// "bit-packed, compact INT32 datatype matrix").  Integer work, bit-exact by construction.
#include "common.cuh"
#include "device_state.h"
#include "launch.h"

namespace qlora {

// One thread builds one packed word: it gathers the (up to 17) codes whose bits fall into stream bits
// [32*row, 32*row+32) of column n.  Consecutive threads own consecutive n, so both the byte reads of codes[k, n]
// and the word writes are coalesced.
__global__ void pack_kernel(int bits, int rows, int N, const uint8_t* __restrict__ codes, uint32_t* __restrict__ Q) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)rows * N) return;
    const int row = (int)(idx / N), n = (int)(idx % N);
    const uint32_t mask = (1u << bits) - 1u;
    const int first_bit = row * 32;
    const int k_first = first_bit / bits;                 // first code with bits in this word
    const int k_last = (first_bit + 31) / bits;           // last one
    uint32_t word = 0;
    for (int k = k_first; k <= k_last; ++k) {
        const uint32_t q = codes[(size_t)k * N + n] & mask;
        const int pos = k * bits - first_bit;             // may be negative (code started in the previous word)
        word |= (pos >= 0) ? (q << pos) : (q >> (-pos));  // bits shifted past 31 fall off
    }
    Q[idx] = word;
}

__global__ void unpack_kernel(int bits, int K, int N, const uint32_t* __restrict__ Q, uint8_t* __restrict__ codes) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)K * N) return;
    const int k = (int)(idx / N), n = (int)(idx % N);
    codes[idx] = (uint8_t)load_code(Q, N, bits, k, n);
}

// Full dequantisation.  One thread turns the 32 consecutive-k codes of one column (BITS words) into 32 bf16 with the same
// routine the tensor-core kernel uses, and writes them as 64 contiguous bytes of row n of W.
template <int BITS>
__global__ void dequant_kernel(int g, int K, int N, const uint32_t* __restrict__ Q, const __half* __restrict__ scales,
                               const __half* __restrict__ zeros, __nv_bfloat16* __restrict__ W) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int blocks = K / 32;
    if (idx >= (size_t)blocks * N) return;
    const int kb = (int)(idx / N), n = (int)(idx % N);
    uint32_t w[BITS];
#pragma unroll
    for (int i = 0; i < BITS; ++i) w[i] = __ldg(Q + (size_t)(kb * BITS + i) * N + n);
    const size_t gi = (size_t)((kb * 32) / g) * N + n;
    const GroupParams gp = group_params(scales[gi], zeros[gi]);
    uint32_t out[16];
    dequant32<BITS>(w, gp, out);
    uint4* dst = reinterpret_cast<uint4*>(W + (size_t)n * K + (size_t)kb * 32);
#pragma unroll
    for (int c = 0; c < 4; ++c) dst[c] = make_uint4(out[4 * c], out[4 * c + 1], out[4 * c + 2], out[4 * c + 3]);
}

// Column gather out[m, j] = in[m, perm[j]] for 2- or 4-byte elements: the per-call step of the activation-order format
// (Appendix A: GPTQ "activation order" leaves the input features of a group scattered; permuting the packed rows once so
// that groups become contiguous, and gathering the activation columns with the same permutation, gives the same layer).
// Two forms.  Few rows (an adapter), or rows that are not whole 16-byte pieces: one element per thread.  Many rows (activations): a
// block brings GC_ROWS whole rows into shared memory with 16-byte loads, and a thread gathers 16 bytes of output at a time from
// there with one set of column numbers for all of them -- bound by the shared-memory reads, a few columns per bank and cycle.
// (333 x 11008 bf16: 18 us with one 2-byte global read and a 64-bit division per element, 8.6 us now.)
template <typename T>
__global__ void __launch_bounds__(256) gather_columns_kernel(int rows, int cols, const T* __restrict__ in, const int32_t* __restrict__ perm, T* __restrict__ out) {
    pdl_wait();
    const int j = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (j >= cols) return;
    const int src = __ldg(perm + j);
    for (int m = (int)blockIdx.y; m < rows; m += (int)gridDim.y) out[(size_t)m * cols + j] = in[(size_t)m * cols + src];
}

constexpr int GC_ROWS = 2, GC_THREADS = 512, GC_NARROW_THREADS = 128, GC_NARROW = 2048;   // GC_NARROW: bytes of a row

template <typename T, int THREADS>
__global__ void __launch_bounds__(THREADS) gather_rows_kernel(int rows, int cols, const T* __restrict__ in, const int32_t* __restrict__ perm, T* __restrict__ out) {
    constexpr int V = 16 / (int)sizeof(T);
    extern __shared__ __align__(16) uint8_t gc_smem[];
    T* row = reinterpret_cast<T*>(gc_smem);                      // [GC_ROWS][cols]
    const int m0 = (int)blockIdx.x * GC_ROWS, n = min(GC_ROWS, rows - m0);
    pdl_wait();
    const uint4* src = reinterpret_cast<const uint4*>(in + (size_t)m0 * cols);
    for (int e = threadIdx.x; e < n * (cols / V); e += THREADS) reinterpret_cast<uint4*>(gc_smem)[e] = src[e];
    __syncthreads();
    for (int c = threadIdx.x; c < cols / V; c += THREADS) {
        int idx[V];
#pragma unroll
        for (int v = 0; v < V; v += 4) {
            const int4 q = __ldg(reinterpret_cast<const int4*>(perm + c * V + v));
            idx[v] = q.x; idx[v + 1] = q.y; idx[v + 2] = q.z; idx[v + 3] = q.w;
        }
#pragma unroll
        for (int r = 0; r < GC_ROWS; ++r) {
            if (r >= n) break;
            __align__(16) T o[V];
#pragma unroll
            for (int v = 0; v < V; ++v) o[v] = row[r * cols + idx[v]];
            *reinterpret_cast<uint4*>(out + (size_t)(m0 + r) * cols + c * V) = *reinterpret_cast<const uint4*>(o);
        }
    }
}

// Asymmetric min-max round-to-nearest quantizer (the "RTN" of the paper's comparisons, and how the benchmark layers get
// their codes).  A block of 8 warps owns one group index and 32 consecutive output rows n of W [N, K]:
//   1. warp w takes rows 4w .. 4w+3 in turn: its lanes read the group's g weights (coalesced along k), min and max go
//      through shuffles, and every lane derives the same scale / zero-point -- in float32, with IEEE division, the scale
//      rounded to fp16 first and halves rounded to even, so the integers are those of the CPU statement of the method;
//   2. per 32 consecutive k: each warp quantizes its four rows (lane = k) into shared memory, then thread (word i, row n)
//      assembles word i of the 32-code block of row n from the bit-stream definition of the format and stores it;
//      neighbouring threads own neighbouring n, so the word stores are coalesced.
// Integer results: bit-exact by construction.
constexpr int QZ_ROWS = 32;

template <int BITS>
__global__ void __launch_bounds__(256) quantize_rtn_kernel(int g, int K, int N, const float* __restrict__ W, uint32_t* __restrict__ Q,
                                                            __half* __restrict__ scales, __half* __restrict__ zeros) {
    __shared__ float s_scale[QZ_ROWS], s_zero[QZ_ROWS];
    __shared__ uint8_t s_code[QZ_ROWS][36];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gi = blockIdx.y, n0 = blockIdx.x * QZ_ROWS;
    const float qmax = (float)((1 << BITS) - 1);
    for (int j = 0; j < 4; ++j) {
        const int n = n0 + 4 * warp + j;
        float lo = 0.f, hi = 0.f;
        if (n < N) {
            const float* row = W + (size_t)n * K + (size_t)gi * g;
            for (int k = lane; k < g; k += 32) { const float w = row[k]; lo = fminf(lo, w); hi = fmaxf(hi, w); }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o)); hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o)); }
        __half sc16 = __float2half_rn(__fdiv_rn(hi - lo, qmax));
        if (__half2float(sc16) == 0.f) sc16 = __float2half_rn(1.f);
        const float sc = __half2float(sc16);
        const float z = fminf(fmaxf(rintf(__fdiv_rn(-lo, sc)), 0.f), qmax) + 0.f;
        if (lane == 0 && n < N) {
            s_scale[4 * warp + j] = sc; s_zero[4 * warp + j] = z;
            scales[(size_t)gi * N + n] = sc16;
            zeros[(size_t)gi * N + n] = __float2half_rn(z);
        }
    }
    __syncthreads();
    for (int kb = 0; kb < g / 32; ++kb) {
        const int k0 = gi * g + kb * 32;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int r = 4 * warp + j, n = n0 + r;
            uint8_t c = 0;
            if (n < N) {
                const float w = W[(size_t)n * K + k0 + lane];
                c = (uint8_t)fminf(fmaxf(rintf(__fdiv_rn(w, s_scale[r])) + s_zero[r], 0.f), qmax);
            }
            s_code[r][lane] = c;
        }
        __syncthreads();
        if (threadIdx.x < BITS * QZ_ROWS) {
            const int i = threadIdx.x / QZ_ROWS, r = threadIdx.x % QZ_ROWS;   // word i of the block's BITS words, row r
            const int k_first = (32 * i) / BITS, k_last = (32 * i + 31) / BITS;
            uint32_t word = 0;
            for (int k = k_first; k <= k_last; ++k) {
                const uint32_t q = s_code[r][k];
                const int pos = k * BITS - 32 * i;                        // negative: the code started in the previous word
                word |= pos >= 0 ? (q << pos) : (q >> (-pos));
            }
            if (n0 + r < N) Q[(size_t)((k0 / 32) * BITS + i) * N + n0 + r] = word;
        }
        __syncthreads();
    }
}

// The same quantizer for groups of 32, 64 and 128 in one pass over W.  Bound by reading W (fp32) once; the kernel above reads it
// twice, one dependent load -> reduce -> divide chain per row.  Here a block of 8 warps owns 32 output rows x 128 k: a warp holds its
// four rows in registers (a float4 per lane and row, all four loads in flight together), so a group is 8, 16 or 32 neighbouring
// lanes.
//   - min and max of the four rows (max(w, 0) and max(-w, 0)) are eight values per lane: three halving exchanges (4 + 2 + 1
//     shuffles) leave lane 2 j + kind with value `kind` of row j, instead of ten shuffles per row; the scale and zero-point of
//     a row are then computed once per eight lanes and handed back with two shuffles.
//   - a code is rint(RN(w / scale)): the product with the reciprocal differs from the quotient by less than 2^-23 |w / scale| <
//     2^-13 (|w / scale| <= 2 qmax), so wherever it lies further than 2^-12 from a tie both round to the same integer; only the others
//     (and NaN) take the division.
//   - four consecutive codes of a lane are one piece of 4 BITS bits, stored to shared memory by row and read back by column as words
//     (odd pitch: no bank conflicts), so the word stores cover 32 neighbouring columns.
// Consecutive blocks walk along k, i.e. along the rows of W in memory.
// 4096 x 11008, 4 bits, group 128: 131 -> 47 us (4.3 TB/s of W + Q, 0.66 of the measured copy bandwidth).
constexpr int QF_K = 128;

template <int BITS> struct QfPiece { using type = uint16_t; };
template <> struct QfPiece<2> { using type = uint8_t; };
template <> struct QfPiece<8> { using type = uint32_t; };

template <int BITS, int GL>   // GL: lanes per group (group size / 4)
__global__ void __launch_bounds__(256) quantize_rtn_fast_kernel(int K, int N, const float* __restrict__ W, uint32_t* __restrict__ Q,
                                                                __half* __restrict__ scales, __half* __restrict__ zeros) {
    using Piece = typename QfPiece<BITS>::type;
    constexpr int PITCH = 8 * (int)sizeof(Piece) + 1;             // 32-bit words per row of pieces
    constexpr int GROUPS = 32 / GL;
    constexpr float QMAX = (float)((1 << BITS) - 1);
    __shared__ uint32_t s_piece[QZ_ROWS * PITCH];
    __shared__ uint32_t s_sz[GROUPS][QZ_ROWS];                    // scale | zero << 16, fp16 bits
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k0 = blockIdx.x * QF_K, n0 = blockIdx.y * QZ_ROWS;
    const int k = k0 + 4 * lane;                                  // (K is a multiple of the group: a group's lanes are all in or all out)
    float4 w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int n = n0 + 4 * warp + j;
        w[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (n < N && k < K) w[j] = __ldcs(reinterpret_cast<const float4*>(W + (size_t)n * K + k));
    }
    float hi[4], nlo[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        hi[j] = fmaxf(fmaxf(fmaxf(fmaxf(0.f, w[j].x), w[j].y), w[j].z), w[j].w);
        nlo[j] = fmaxf(fmaxf(fmaxf(fmaxf(0.f, -w[j].x), -w[j].y), -w[j].z), -w[j].w);
    }
    float v4[4], v2[2], v;
#pragma unroll
    for (int j = 0; j < 4; ++j) {                                 // odd lanes keep -min, even lanes max
        const float send = (lane & 1) ? hi[j] : nlo[j], keep = (lane & 1) ? nlo[j] : hi[j];
        v4[j] = fmaxf(keep, __shfl_xor_sync(0xffffffffu, send, 1));
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {                                 // lane bit 1 picks the row's low bit
        const float send = (lane & 2) ? v4[2 * j] : v4[2 * j + 1], keep = (lane & 2) ? v4[2 * j + 1] : v4[2 * j];
        v2[j] = fmaxf(keep, __shfl_xor_sync(0xffffffffu, send, 2));
    }
    {
        const float send = (lane & 4) ? v2[0] : v2[1], keep = (lane & 4) ? v2[1] : v2[0];
        v = fmaxf(keep, __shfl_xor_sync(0xffffffffu, send, 4));
    }
    if constexpr (GL >= 16) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 8));
    if constexpr (GL >= 32) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 16));
    const float other = __shfl_xor_sync(0xffffffffu, v, 1);
    const float mx = (lane & 1) ? other : v, nmn = (lane & 1) ? v : other;
    __half sc16 = __float2half_rn(__fdiv_rn(mx + nmn, QMAX));
    if (__half2float(sc16) == 0.f) sc16 = __float2half_rn(1.f);
    const float my_sc = __half2float(sc16);
    const float my_z = fminf(fmaxf(rintf(__fdiv_rn(nmn, my_sc)), 0.f), QMAX) + 0.f;
    const uint32_t my_sz = (uint32_t)__half_as_ushort(sc16) | ((uint32_t)__half_as_ushort(__float2half_rn(my_z)) << 16);
    if ((lane & 1) == 0 && (lane & (GL - 1)) < 8) s_sz[lane / GL][4 * warp + ((lane >> 1) & 3)] = my_sz;

    constexpr float MAGIC = 12582912.f;                           // 1.5 * 2^23: adding it rounds to an integer, half to even
    constexpr float BASE = 8388608.f;                             // 2^23: an integer below it sits in the low mantissa bits
    Piece* pieces = reinterpret_cast<Piece*>(s_piece);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t sz = __shfl_sync(0xffffffffu, my_sz, (lane & ~7) | (j << 1));
        const float sc = __half2float(__ushort_as_half((unsigned short)(sz & 0xFFFFu)));
        const float zb = BASE + __half2float(__ushort_as_half((unsigned short)(sz >> 16)));
        const float inv = __frcp_rn(sc);
        const float wj[4] = {w[j].x, w[j].y, w[j].z, w[j].w};
        float q[4], worst = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            q[i] = __fmaf_rn(wj[i], inv, MAGIC) - MAGIC;
            const float d = fabsf(__fmaf_rn(wj[i], inv, -q[i]));
            worst = d < 0.5f - 0x1p-12f ? worst : 1.f;            // (a NaN fails the comparison)
        }
        if (worst != 0.f) {
#pragma unroll
            for (int i = 0; i < 4; ++i) q[i] = rintf(__fdiv_rn(wj[i], sc));
        }
        uint32_t u[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) u[i] = __float_as_uint(fminf(fmaxf(q[i] + zb, BASE), BASE + QMAX));   // code in the low bits
        uint32_t piece;
        if constexpr (BITS == 8) piece = __byte_perm(__byte_perm(u[0], u[1], 0x0040), __byte_perm(u[2], u[3], 0x0040), 0x5410);
        else piece = u[0] + (u[1] << BITS) + (u[2] << (2 * BITS)) + (u[3] << (3 * BITS));                 // (BASE's bits stay above 23)
        pieces[(4 * warp + j) * PITCH * (4 / (int)sizeof(Piece)) + lane] = (Piece)piece;
    }
    __syncthreads();
    const int r = lane, n = n0 + r;
    if (n < N) {
#pragma unroll
        for (int i = warp; i < 4 * BITS; i += 8) {                // word i of the 128 k: 32-code block i / BITS
            const uint32_t* row = s_piece + r * PITCH;
            uint32_t word;
            if constexpr (BITS == 3) {
                const int b = i / 3, part = i % 3;
                const uint32_t x = row[4 * b + part], y = row[4 * b + part + 1];   // pieces 2 part, +1 and 2 part + 2, +3 (12 bits each)
                if (part == 0)      word = (x & 0xFFFFu) | ((x >> 16) << 12) | (y << 24);
                else if (part == 1) word = ((x & 0xFFFFu) >> 8) | ((x >> 16) << 4) | ((y & 0xFFFFu) << 16) | ((y >> 16) << 28);
                else                word = (x >> 20) | ((y & 0xFFFFu) << 8) | ((y >> 16) << 20);
            } else {
                word = row[i];
            }
            if (k0 + 32 * (i / BITS) < K) Q[(size_t)(k0 / 32 * BITS + i) * N + n] = word;
        }
        if (warp < GROUPS && k0 + warp * 4 * GL < K) {
            const uint32_t sz = s_sz[warp][r];
            const size_t gi = (size_t)(k0 / (4 * GL) + warp) * N + n;
            scales[gi] = __ushort_as_half((unsigned short)(sz & 0xFFFFu));
            zeros[gi] = __ushort_as_half((unsigned short)(sz >> 16));
        }
    }
}

template <int BITS>
static void launch_quantize_fast(const qlora_desc& d, const float* W, uint32_t* q, __half* s, __half* z, cudaStream_t st) {
    const dim3 grid((unsigned)((d.K + QF_K - 1) / QF_K), (unsigned)((d.N + QZ_ROWS - 1) / QZ_ROWS));
    if (d.group_size == 32) quantize_rtn_fast_kernel<BITS, 8><<<grid, 256, 0, st>>>(d.K, d.N, W, q, s, z);
    else if (d.group_size == 64) quantize_rtn_fast_kernel<BITS, 16><<<grid, 256, 0, st>>>(d.K, d.N, W, q, s, z);
    else quantize_rtn_fast_kernel<BITS, 32><<<grid, 256, 0, st>>>(d.K, d.N, W, q, s, z);
}

int launch_quantize_rtn(const qlora_desc& d, const float* W, int32_t* Q, void* scales, void* zeros, cudaStream_t st) {
    if (d.K == 0 || d.N == 0) return QLORA_OK;
    const dim3 grid((unsigned)((d.N + QZ_ROWS - 1) / QZ_ROWS), (unsigned)(d.K / d.group_size));
    uint32_t* q = (uint32_t*)Q;
    __half* s = (__half*)scales;
    __half* z = (__half*)zeros;
    // groups that are whole lanes of one 128-wide strip: one pass; other sizes (96, 256, K, ...) reduce in a loop, in the first kernel
    if ((d.group_size == 32 || d.group_size == 64 || d.group_size == 128) && (d.N + QZ_ROWS - 1) / QZ_ROWS <= 65535) {
        switch (d.bits) {
            case 2: launch_quantize_fast<2>(d, W, q, s, z, st); break;
            case 3: launch_quantize_fast<3>(d, W, q, s, z, st); break;
            case 4: launch_quantize_fast<4>(d, W, q, s, z, st); break;
            case 8: launch_quantize_fast<8>(d, W, q, s, z, st); break;
            default: return QLORA_ERR_UNSUPPORTED;
        }
        return cudaGetLastError() == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
    }
    switch (d.bits) {
        case 2: quantize_rtn_kernel<2><<<grid, 256, 0, st>>>(d.group_size, d.K, d.N, W, q, s, z); break;
        case 3: quantize_rtn_kernel<3><<<grid, 256, 0, st>>>(d.group_size, d.K, d.N, W, q, s, z); break;
        case 4: quantize_rtn_kernel<4><<<grid, 256, 0, st>>>(d.group_size, d.K, d.N, W, q, s, z); break;
        case 8: quantize_rtn_kernel<8><<<grid, 256, 0, st>>>(d.group_size, d.K, d.N, W, q, s, z); break;
        default: return QLORA_ERR_UNSUPPORTED;
    }
    return cudaGetLastError() == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
}

template <typename T>
static cudaError_t launch_gather(int rows, int cols, const void* in, const int32_t* perm, void* out, cudaStream_t st) {
    const size_t smem = (size_t)GC_ROWS * cols * sizeof(T);
    // from 64 rows on the whole-row blocks cover enough SMs (below, an element per thread is the faster); two blocks fit an SM
    if (rows >= 64 && (size_t)cols * sizeof(T) % 16 == 0 && smem <= 100 * 1024) {
        const dim3 grid((unsigned)((rows + GC_ROWS - 1) / GC_ROWS));
        // narrow rows, more of them than the SMs hold at 512 threads a block: fewer threads, of which more have a piece (8192 rows of 256 floats:
        // 9.5 us by elements, 11.4 with 512 threads, 5.6 with 128; 200 rows of 512 floats 1.9 with 512, 2.1 with 128)
        if ((size_t)cols * sizeof(T) <= GC_NARROW && rows > GC_ROWS * 4 * sm_count())
            return launch_pdl(gather_rows_kernel<T, GC_NARROW_THREADS>, grid, dim3(GC_NARROW_THREADS), smem, st, 1, rows, cols, (const T*)in, perm, (T*)out);
        static SmemLimit limit;
        if (!limit.raise(gather_rows_kernel<T, GC_THREADS>, 100 * 1024)) return cudaErrorUnknown;
        return launch_pdl(gather_rows_kernel<T, GC_THREADS>, grid, dim3(GC_THREADS), smem, st, 1, rows, cols, (const T*)in, perm, (T*)out);
    }
    return launch_pdl(gather_columns_kernel<T>, dim3((unsigned)((cols + 255) / 256), (unsigned)(rows < 65535 ? rows : 65535)), dim3(256), 0, st, 1, rows, cols, (const T*)in, perm, (T*)out);
}

// (Launched so that it may start while its predecessor ends; it does not let its own dependents start early.)
int launch_gather_columns(int elem_bytes, int rows, int cols, const void* in, const int32_t* perm, void* out, cudaStream_t st) {
    if (rows == 0 || cols == 0) return QLORA_OK;
    if (elem_bytes != 2 && elem_bytes != 4) return QLORA_ERR_UNSUPPORTED;
    const cudaError_t err = elem_bytes == 2 ? launch_gather<uint16_t>(rows, cols, in, perm, out, st) : launch_gather<uint32_t>(rows, cols, in, perm, out, st);
    return err == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
}

int launch_pack(int bits, int K, int N, const uint8_t* codes, int32_t* Q, cudaStream_t st) {
    const int rows = K * bits / 32;
    const size_t total = (size_t)rows * N;
    if (total == 0) return QLORA_OK;
    pack_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(bits, rows, N, codes, (uint32_t*)Q);
    return cudaGetLastError() == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
}

int launch_unpack(int bits, int K, int N, const int32_t* Q, uint8_t* codes, cudaStream_t st) {
    const size_t total = (size_t)K * N;
    if (total == 0) return QLORA_OK;
    unpack_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(bits, K, N, (const uint32_t*)Q, codes);
    return cudaGetLastError() == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
}

int launch_dequant(const qlora_desc& d, const int32_t* Q, const void* scales, const void* zeros, void* W,
                   cudaStream_t st) {
    if (d.K == 0 || d.N == 0) return QLORA_OK;
    const size_t total = (size_t)(d.K / 32) * d.N;
    const unsigned grid = (unsigned)((total + 255) / 256);
    const uint32_t* q = (const uint32_t*)Q;
    const __half* s = (const __half*)scales;
    const __half* z = (const __half*)zeros;
    __nv_bfloat16* w = (__nv_bfloat16*)W;
    switch (d.bits) {
        case 2: dequant_kernel<2><<<grid, 256, 0, st>>>(d.group_size, d.K, d.N, q, s, z, w); break;
        case 3: dequant_kernel<3><<<grid, 256, 0, st>>>(d.group_size, d.K, d.N, q, s, z, w); break;
        case 4: dequant_kernel<4><<<grid, 256, 0, st>>>(d.group_size, d.K, d.N, q, s, z, w); break;
        case 8: dequant_kernel<8><<<grid, 256, 0, st>>>(d.group_size, d.K, d.N, q, s, z, w); break;
        default: return QLORA_ERR_UNSUPPORTED;
    }
    return cudaGetLastError() == cudaSuccess ? QLORA_OK : QLORA_ERR_CUDA;
}

}  // namespace qlora
