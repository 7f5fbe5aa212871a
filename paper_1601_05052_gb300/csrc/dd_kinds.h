// dd_kinds.h -- the forward kernel kinds and their CTA shapes, shared by the
// host code that builds a variant's tables and the kernels that run it.
//
// kind 0: lane-strided accumulation from the staged channel windows;
// kind 1: register windows; kind 2: sub-band partial series (groups of four
// channels) with a producer warp; kind 3: kind 2 with warp-specialised
// builders; kind 4: kind 2 in CTAs of up to 16 trial warps; kind 5: kind 0
// with operand reuse between trials (equal delays, or register windows); kind 6:
// kind 4 with one partial-sum slot and up to 8 groups per chunk, which lets
// FP32 input stage 32 channels at a time.
#pragma once

#include <cuda_runtime.h>

namespace dd {

// Builder warps of kind 3.
constexpr int kWsBuilders = 4;

// Warps a CTA has beyond its warps_dm * warps_time trial warps.
__host__ __device__ constexpr int extra_warps(int kind) {
    return kind == 3 ? kWsBuilders : ((kind == 2 || kind == 4 || kind == 6) ? 1 : 0);
}
// Sub-band kinds (partial series per channel group).
__host__ __device__ constexpr bool is_subband(int kind) {
    return kind == 2 || kind == 3 || kind == 4 || kind == 6;
}
// Register-window form of kind 5 (see dd_fwd_tile.cuh): 2 * odd samples per
// thread in two runs of consecutive samples.
__host__ __device__ constexpr bool is_window(int kind, int spt) {
    return kind == 5 && spt % 4 == 2;
}
// Byte-quad form of kind 0 (8-bit input only): 20 consecutive samples per
// thread, read as 32-bit words.
__host__ __device__ constexpr bool is_quad(int kind, int spt) { return kind == 0 && spt == 20; }
// Forms of float input that sum groups of four consecutive channels before they
// add to the accumulators, in the sub-bands' order: the sub-bands themselves and
// the lane-strided 2 x 4, 4 x 2 and 4 x 8. Their rounding error over C channels
// grows like that of a chain of C / 4 terms, the other forms' like C terms.
__host__ __device__ constexpr bool sums_groups(int kind, int dpt, int spt) {
    return is_subband(kind) || (kind == 0 && (dpt * spt == 8 || (dpt == 4 && spt == 8)));
}
// Kernels whose CTAs may have 16 trial warps and stage 1 or 2 channels at a time:
// the register windows, the byte quads and the lane-strided 8 x 8 form.
__host__ __device__ constexpr bool is_wide(int kind, int dpt, int spt) {
    return is_window(kind, spt) || is_quad(kind, spt) || (kind == 0 && dpt == 8 && spt == 8);
}
// Codes of the delay steps a register window serves: steps (s1, s2, s3)
// between a thread's four trials with every step in {b, b + 1} are code 7 b +
// (s1 - b) + 2 (s2 - b) + 4 (s3 - b), b < kWinBands (so all steps equal to b +
// 1 are code 7 (b + 1)). Other steps: kWinNone.
constexpr int kWinBands = 5;
constexpr int kWinNone = 7 * kWinBands + 1;
// Largest trial-warp count of a CTA.
__host__ __device__ constexpr int max_trial_warps(int kind, int dpt, int spt) {
    return (kind == 4 || kind == 6 || is_wide(kind, dpt, spt)) ? 16 : 8;
}
// Launch bounds of the forward kernels: threads per CTA and resident CTAs
// per SM that the register allocation must allow (the lane-strided 4 x 8 form's
// grouped sums would take 140 registers instead of 128, one CTA of four warps
// fewer per SM).
__host__ __device__ constexpr int fwd_max_threads(int kind, int dpt, int spt) {
    return 32 * (max_trial_warps(kind, dpt, spt) + extra_warps(kind));
}
__host__ __device__ constexpr int fwd_min_blocks(int kind, int dpt, int spt) {
    if (kind == 0 && dpt == 4 && spt == 8) return 2;
    return kind == 2 ? (dpt * spt <= 16 ? 3 : 2) : (kind == 3 ? 2 : 1);
}

}  // namespace dd
