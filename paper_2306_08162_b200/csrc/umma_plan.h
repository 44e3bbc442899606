// How the tensor-core kernels cut a layer call: token tiles, ranks per tile, ring lengths and the layout of shared memory.  Host code without
// CUDA, so that its rules can be checked over all shapes on the CPU.
#pragma once
#include <stdint.h>

namespace qlora {

constexpr int kWRows = 128;          // weight rows (MMA M) per tile: n in forward, k in backward
constexpr int kStepC = 64;           // contraction elements per pipeline stage
constexpr int kWStageBytes = kWRows * kStepC * 2;   // 16 KiB of bf16 per stage
constexpr int kPairTok = 128;                          // CTA-pair kernel: token rows per CTA per accumulator
constexpr int kPairW = 128;                            // weight rows per CTA (256 per pair tile)
constexpr int kPairXSub = kPairTok * kStepC * 2;       // 16 KiB: one 128-token sub-tile of a stage
constexpr int kPairXStage = 2 * kPairXSub;             // two accumulators' sub-tiles
constexpr int kDequantGroups = 2, kDownGroups = 3;     // dequant groups, and in the DOWN build
constexpr uint32_t kSmemBudget = 232448 - 1024 /*alignment slack*/ - 2048 /*static, barriers, padding*/;
constexpr int kMaxDownTokens = 128;

// Whether `groups` dequant groups that take the stages of a tile in turn may run on an operand ring of S stages and a packed ring of P slots.
// A group tells the laps of a slot apart by one parity bit, so whoever waits for lap l must know that lap l - 1 is over.  A group that is about to
// take step t has seen the MMAs of step t - groups - S through (it waited for that stage to be free), hence of all steps before it:
//   - the stage of step t was last but one used by step t - 2 S, which is over when S >= groups;
//   - the slot of step t was last filled for step t - P: over when P >= S + groups, or when that step was this very group's (P a multiple of groups).
// Else a wait may return a lap early, on codes that have not landed.
inline bool rings_sound(int S, int P, int groups) { return S >= groups && (P % groups == 0 || P >= S + groups); }

// Rows of scales / zeros that go with the k range of one pipeline stage (64 rows of W forward, 128 backward).
inline int scale_rows_per_stage(int g, bool transposed) {
    const int k_rows = transposed ? kWRows : kStepC;
    return g >= k_rows ? 1 : k_rows / g;
}

// lora_lo and r_pad (see TilePlan).
inline int keep_lora_low(int r, int g) { return r == 8 || g == 32 ? 1 : 0; }
inline int lora_columns(int r, int g) { return ((keep_lora_low(r, g) ? 2 : 1) * r + 15) / 16 * 16; }

// A pipeline stage of packed codes and group parameters (Plan: TilePlan or the CTA-pair kernel's parameters).
template <class Plan>
inline void plan_packed_stage(Plan& p, int bits, int g, bool transposed) {
    p.packed_cols = transposed ? 64 : 128;
    p.packed_rows = (transposed ? 128 : 64) * bits / 32;
    p.scale_rows = scale_rows_per_stage(g, transposed);
    p.words_bytes = (uint32_t)(p.packed_rows * p.packed_cols * 4);
    p.scale_bytes = (uint32_t)(p.scale_rows * p.packed_cols * 2);
    p.packed_slot_bytes = (p.words_bytes + 2 * p.scale_bytes + 127u) / 128u * 128u;
}

// Single-CTA kernel.  Offsets count from the 1024-byte aligned base of shared memory.  (The head of the kernel's parameters.  With the
// fields in another order the smallest calls took 1 to 3 % longer: 512 x 512, 17 tokens, rank 8 4.98 -> 5.12 us.)
struct TilePlan {
    int M, N, K, bits, g, r, r_pad;
    // r_pad: columns of the LoRA operands, a multiple of 16.  lora_lo: ranks [r, 2r) hold, beside the finite ones of the same adapter
    // elements again, what the rounding of s * P to bf16 left over, so that the update has 16 significant bits of P's 24: for r == 8,
    // where half an MMA's contraction is padding otherwise, and for groups of 32, whose products the CUDA-core kernel gave from fp32
    // (the error of Y and dX against 64 bits is the same with it: that of the weights' and outputs' bf16).
    int lora_lo;
    int C;               // output columns (N forward, K backward)
    int BT;              // token rows per tile (MMA N): a multiple of 16, 32 .. 256
    int n_tok_tiles, n_tiles, steps;   // steps: of one rank
    int split;           // CTAs per cluster sharing one tile, each taking `steps` consecutive steps of the contraction (1 = no cluster)
    int S, P;            // stages of the activation/weight ring and of the packed ring
    int packed_cols;     // 128 forward, 64 backward
    int packed_rows;     // int32 rows per stage
    int scale_rows;      // group rows per stage
    uint32_t words_bytes, scale_bytes, packed_slot_bytes, x_stage_bytes;
    uint32_t off_x, off_w, off_l, off_p, off_lora_a, off_lora_p, off_bar;
    uint32_t down_bytes;             // DOWN: bytes per stage of the adapter applied first (else 0)
};

// What runs at a time: SMs, and clusters of two and of four CTAs with an SM to each (148 SMs: 74 and 33, not 37, as a cluster stays in one group of SMs).
// 34 to 37 tiles on clusters of four are two waves: two ranks per tile instead are 20 to 50 % faster (4352 outputs, rank 8, 64 tokens, T = 512 11.5 -> 6.4 us,
// 4096 20.6 -> 14.6; 4736, 256 tokens, 11008 long 60.6 -> 45.3).
struct GpuFit {
    int sms, clusters2, clusters4;
    int clusters(int width) const { return width == 4 ? clusters4 : width == 2 ? clusters2 : sms; }
};

// Whether ranks of `steps` contraction steps form P themselves (DOWN; rank 8 or 16, up to 128 tokens).  Their MMAs cost some 250 cycles per step and P's
// parts go through the exchange; the producer clusters cost a launch, a counter and a chain that grows with the rank and is longer in the
// backward; and DOWN has a third dequant group, which INT3 gains the most from.  Two ranks have twice as much to exchange.  Microseconds without / with,
// INT4, forward: two ranks of five steps, 128 tokens, 512 wide 8.88 / 8.20, 8192 wide 9.26 / 9.56; of seven, 6016 wide, 64 tokens 8.57 / 8.22, 128 tokens
// 9.37 / 9.91.  Four ranks, rank 8, 2048 wide: eight steps, 64 tokens 9.04 / 8.00; 16 steps, 48 tokens 10.27 / 10.04, 64 tokens 10.50 / 10.89, backward
// 96 tokens 12.19 / 11.79, 128 tokens 12.76 / 13.22, INT3, 96 tokens 13.00 / 12.12.  Rank 16: 14 steps, 128 tokens 13.32 / 12.64; 16 steps, 112
// tokens 12.94 / 12.71, 128 tokens 13.32 / 13.67; 24 steps, 96 tokens 15.10 / 15.00, 128 tokens 15.59 / 16.62, backward 17.17 / 16.70; 32 steps, 32 tokens
// 14.77 / 14.76, 64 tokens 15.52 / 16.72; 43 steps, 512 wide, 64 tokens 19.25 / 20.47.  Where the producers would take the last clusters or find none
// (4096 wide: 32 tiles), 43 steps, 128 tokens 32.4 / 25.7; rank 8, 16 steps, 96 tokens 13.63 / 13.15.
inline bool down_pays(const TilePlan& p, int split, int steps, bool transposed, const GpuFit& fit) {
    if (split == 2) return steps <= 5 ? p.BT <= 96 || 4 * p.n_tiles * split <= 3 * fit.sms : steps <= 8 && p.BT <= 168 - 12 * steps;
    if (p.r == 8 && steps > 16) return false;
    if (p.bits == 3 || fit.clusters(split) - p.n_tiles <= ((p.M + 15) / 16 + split - 1) / split) return true;
    const int most = p.r == 16 ? (steps <= 14 ? 128 : steps <= 20 ? 112 : steps <= 24 ? 96 : steps <= 32 ? 48 : 32) : (steps <= 14 ? 128 : 48);
    return p.BT <= most + (transposed ? 48 : 0);
}

// Contraction steps that a rank of a split tile of this plan has at least.  Up to 128 tokens the DOWN build takes two (512 x 512, rank 8: four ranks of
// two steps against two of four 5.1 / 5.7 us at 17 tokens; what the ranks exchange grows with the tokens: 11.8 / 10.6 at 256).  Without it there is
// the chain of a down-projection or nothing to hide more ranks behind, and they pay up to 16 ranks only, with two steps up to 64 tokens, with three
// up to 128, while the clusters leave room for the CTAs of the launch behind; under dropout (`dropout`: other launches of the call go before and
// after) that matters less.  INT4, microseconds, four ranks of two or three steps / two of four or six: rank 0, 512 -> 2048, 64 tokens 5.51 / 5.81,
// 128 tokens 6.83 / 6.65; 512 -> 4096, 64 tokens 6.83 / 5.89; 768 -> 2048, 17 tokens 5.12 / 5.77, 128 tokens 7.06 / 7.18; rank 32, 768 -> 2048,
// 64 tokens 9.87 / 9.91, 128 tokens 11.49 / 10.81; dropout forward, rank 16, 512 -> 2048, 17 tokens 7.88 / 8.12, 128 tokens 9.98 / 9.54, rank 8,
// 768 -> 4096, 64 tokens 8.45 / 9.26; dropout backward (rank 0 in this kernel), 512 long, 17 tokens, 4096 wide 8.64 / 9.74, 48 tokens 12.34 / 11.33 (3072 wide 9.25 / 9.74).
inline int min_split_steps(const TilePlan& p, int split, bool down, bool dropout, const GpuFit& fit) {
    if (p.BT > kMaxDownTokens) return 4;
    if (down) return 2;
    const int ctas = p.n_tiles * split, most = !dropout || p.BT > 64 ? fit.sms / 2 : p.BT > 32 ? fit.sms * 2 / 3 : fit.sms;
    if (p.r > 16 || (p.r == 0 && ctas > most)) return 4;
    return p.BT <= 64 ? 2 : 3;
}

// Rings and layout for `split` ranks per tile, `total_steps` steps among them; with_down: the DOWN build.  False: does not fit.
inline bool plan_rings(TilePlan& p, int split, int total_steps, bool with_down) {
    p.split = split;
    p.steps = total_steps / split;
    p.down_bytes = with_down ? (uint32_t)p.r * 128u : 0u;
    const uint32_t lora_a = (uint32_t)(kWRows * p.r_pad * 2), lora_p = (uint32_t)(p.BT * p.r_pad * 2);
    const uint32_t per_stage = p.x_stage_bytes + kWStageBytes + p.down_bytes;
    // With few tokens the kernel is bound by the latency of streaming cold packed weights through a handful of CTAs, so the packed ring is
    // deep (bytes in flight), at the cost of one or two operand stages; it gives way until three of those fit (two, at four slots and below).
    // Lengths are even: three slots beside two stages are none that two groups may use (rings_sound).  Only INT8 with groups of 32 at rank 64 ever had them:
    // with two, 250 tokens on 4096 x 4096 49.6 -> 52.7 us forward, 50.1 -> 55.6 backward, in the CTA-pair kernel nothing.
    uint32_t S = 0;
    for (p.P = p.BT <= 128 ? 16 : 8;; p.P -= p.P > 4 ? 4 : 2) {
        const uint32_t fixed = lora_a + lora_p + p.P * p.packed_slot_bytes + 512;
        S = kSmemBudget > fixed ? (kSmemBudget - fixed) / per_stage : 0;
        if (S >= (p.P > 4 ? 3u : 2u) || p.P == 2) break;
    }
    if (S > 8) S = 8;
    p.S = (int)S;
    p.off_x = 0;
    p.off_w = p.off_x + S * p.x_stage_bytes;
    p.off_l = p.off_w + S * kWStageBytes;
    p.off_p = p.off_l + S * p.down_bytes;
    p.off_lora_a = p.off_p + p.P * p.packed_slot_bytes;
    p.off_lora_p = p.off_lora_a + lora_a;
    p.off_bar = (p.off_lora_p + lora_p + 127u) / 128u * 128u;
    // a split tile's fp32 parts (and those of P) meet in the operand ring
    return rings_sound(p.S, p.P, with_down ? kDownGroups : kDequantGroups) &&
           (split == 1 || (uint32_t)(p.BT * (kWRows + (with_down ? p.r : 0)) * 4) <= p.off_p);
}

// For the shape in M .. C and a contraction of T elements.  wants_p: P = In * Ldown is still to be computed; dropout: see min_split_steps.  False: does not fit.
inline bool plan_tiles(TilePlan& p, int T, bool transposed, bool wants_p, bool dropout, const GpuFit& fit) {
    plan_packed_stage(p, p.bits, p.g, transposed);
    // The tokens in as few tiles as 256 columns allow, cut evenly: a multiple of 16 (the MMA's N), not the next power of two, so that
    // neither products nor the exchange between the ranks are made for tokens that do not exist (333: two tiles of 176, not 256).
    p.n_tok_tiles = (p.M + 255) / 256;
    p.BT = ((p.M + p.n_tok_tiles - 1) / p.n_tok_tiles + 15) / 16 * 16;
    if (p.BT < 32) p.BT = 32;
    p.n_tok_tiles = (p.M + p.BT - 1) / p.BT;
    p.n_tiles = p.n_tok_tiles * ((p.C + kWRows - 1) / kWRows);
    p.x_stage_bytes = (uint32_t)(p.BT * 128);
    // Few tiles (few tokens): split each tile's contraction over a cluster of 2 or 4 CTAs so that the whole GPU streams
    // the weights.  Needs one tile per cluster, an even split of the steps, and room for the fp32 parts in the operand ring.
    const int steps = T / kStepC;
    for (int sp = 4; sp >= 2; sp /= 2) {
        if (p.n_tiles > fit.clusters(sp) || steps % sp != 0 || p.BT % sp != 0) continue;
        const bool down = wants_p && (p.r == 8 || p.r == 16) && p.BT <= kMaxDownTokens && down_pays(p, sp, steps / sp, transposed, fit);
        if (steps / sp < min_split_steps(p, sp, down, dropout, fit)) continue;
        if (down && plan_rings(p, sp, steps, true)) return true;
        if (plan_rings(p, sp, steps, false)) return true;
    }
    return plan_rings(p, 1, steps, false);
}

// CTA-pair kernel: the lengths of its rings beside `lora_bytes` of LoRA operands.  False: does not fit.
inline bool plan_pair_rings(uint32_t packed_slot_bytes, uint32_t lora_bytes, int& S, int& P) {
    for (P = 4; P >= 2; P -= 2) {                              // (the packed ring gives way where the LoRA operands are at their largest)
        S = (int)((kSmemBudget - (lora_bytes + P * packed_slot_bytes + 512)) / (kPairXStage + kWStageBytes));
        if (S > 8) S = 8;
        if (rings_sound(S, P, kDequantGroups)) return true;
    }
    return false;
}

}  // namespace qlora
