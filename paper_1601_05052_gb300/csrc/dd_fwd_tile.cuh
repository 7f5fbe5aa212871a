// dd_fwd_tile.cuh -- the per-tile body of the forward dedispersion kernel,
// shared by the one-shot and the persistent batched kernels (dd_kernels.cu).
//
// A tile is (beam b, DM tile of Dt trials, time tile of Ts output samples)
// and computes out[b][d][t] = sum_c w[c] * in[b][c][t + shift[d][c]] for its
// trials and samples (Algorithm 1, Section III-A, with weights; the 2-D
// work-group decomposition of Section III-B). Each trial warp owns DPT
// trials by 32*SPT samples; a thread accumulates DPT x SPT outputs in
// registers.
//
// Staging (Section III-B's shared "local memory"): channels are taken in
// chunks. Per chunk the tile's shifted input windows are copied, one 1-D TMA
// bulk copy per lane, into a pipeline slot, together with the chunk's tables
// and weights; the slot's `full` mbarrier counts the bytes. A tile's first
// chunks are issued by all warps together, later ones by one warp each: the
// trial warps in turn (kinds 0, 1 and 5) or a producer or builder warp
// (sub-bands). Copy lists are read ahead, so the copies go out without waiting
// on global memory.
//
// Ways to turn a staged window into sums (the `kind` of a variant):
//  kind 0, lane-strided: lane l owns samples l, l+32, ...; every add reads
//    its operand from shared memory (conflict-free, one word per add).
//    Slots are recycled through `empty` mbarriers (one arrival per warp).
//    Three float forms sum groups of four channels first (see GroupedLanes).
//    8-bit input with 20 samples per thread reads words (see Quads).
//  kind 1, register window: a thread owns SPT (odd) consecutive samples;
//    per channel it loads its warp's union window into registers once and
//    serves every trial from it through a warp-uniform switch on the
//    trial's relative delay (0..15); wider groups take a direct path.
//  kind 2, sub-band partial sums: channels form groups of 4; inside a DM
//    tile the trials of a group share few distinct relative delay patterns,
//    so the CTA builds each pattern's weighted 4-channel partial series in
//    shared memory once per chunk and the lane-strided trial loop adds one
//    partial value per group instead of one input value per channel (the
//    same sums, associated per group). A dedicated producer warp stages the
//    chunks; the compute warps meet at one named barrier per chunk.
//  kind 4, wide sub-band: kind 2 in CTAs of up to 16 trial warps (one
//    resident CTA per SM), for DM tiles of 128 trials.
//  kind 3, warp-specialised sub-band: kind 2's arithmetic with 4 extra
//    builder warps; mbarriers on the staging slots and on 3 partial-sum
//    slots replace every CTA-wide barrier.
//  kind 5, shared operands: kind 0, but operands in registers serve several
//    trials: those whose delay in the channel equals the previous trial's, or
//    (2 * odd samples per thread, see Window) every trial of the thread whose
//    delay lies within a window of consecutive samples.
//  kind 6, one-slot wide sub-band: kind 4 with a single partial-sum slot
//    (one more barrier per chunk) and up to 8 groups per chunk, so that
//    FP32 input fits 32-channel chunks.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cstdint>
#include <type_traits>

#include "dd_kinds.h"
#include "dd_ptx.cuh"

// The compiled forward kernels: X(kind, dm_per_thread, samples_per_thread).
// Kind 4 is kind 2 in CTAs of up to 16 trial warps (one CTA per SM), so a
// DM tile can span 128 trials and amortise each partial series over more of them.
#define DD_FWD_KEYS(X)                                                                    \
    X(0, 2, 4) X(0, 4, 2) X(0, 4, 4) X(0, 8, 2) X(0, 8, 4) X(0, 4, 8) X(1, 8, 9) X(2, 4, 4) \
        X(2, 4, 8) X(2, 8, 4) X(2, 8, 2) X(3, 8, 4) X(3, 4, 8) X(3, 8, 2) X(4, 8, 4) X(4, 4, 8) \
            X(5, 4, 8) X(5, 8, 4) X(6, 4, 8) X(0, 4, 16) X(5, 4, 14) X(5, 4, 18) X(5, 4, 22) \
                X(0, 8, 8) X(0, 4, 20)

namespace dd {

// Whether a key has a kernel for an input type (the byte quads: 8-bit only).
template <typename T>
constexpr bool key_has_type(int kind, int spt) {
    return !is_quad(kind, spt) || sizeof(T) == 1;
}

// Largest relative delay inside a warp's trial group served from registers.
constexpr int kRwRmax = 15;
// Channels per group and patterns per group of the sub-band kinds; builder
// warps and partial-sum slots of kind 3.
constexpr int kSbG = 4;
constexpr int kSbP = 8;
constexpr int kWsPSlots = 3;
// Chunks whose channel descriptors a producer warp holds in registers ahead
// of issuing their copies.
constexpr int kDescAhead = 4;

template <typename T>
struct Elem;
template <>
struct Elem<float> {
    using Acc = float;
    using W = float;
    __device__ static float val(float x) { return x; }
};
template <>
struct Elem<__half> {
    using Acc = float;
    using W = float;
    __device__ static float val(__half x) { return __half2float(x); }
};
template <>
struct Elem<__nv_bfloat16> {
    using Acc = float;
    using W = float;
    __device__ static float val(__nv_bfloat16 x) { return __bfloat162float(x); }
};
template <>
struct Elem<uint8_t> {
    using Acc = int;
    using W = int;
    __device__ static int val(uint8_t x) { return int(x); }
};

// Everything a tile needs about one plan and one set of buffers.
struct FwdArgs {
    const void *in;
    const void *w;
    void *out;
    int C, D;
    long long S, stride;
    int Dt, Ts, C_pad, cch, stages, warps_dm;
    int stage_data_bytes, stage_offs_bytes;
    int n_dtiles, n_ttiles, B;
    // One-shot launches cover DM tiles [dtile0, dtile0 + grid_dt) by time
    // tiles [ttile0, ttile0 + grid_tt); CTA x of the launch takes them with
    // the DM tile fastest (time_major 0) or the time tile fastest (1).
    int ttile0, dtile0, grid_tt, grid_dt, time_major;
    const int4 *copies;  // staging copies [n_dtiles][n_chunks][n_copies]
    int n_copies;
    int copies_ahead;  // a slot holds a later chunk's copies (kinds 0, 1 and 5)
    const uint16_t *offs;
    const int4 *bdesc;  // sub-band kinds: build blocks [n_dtiles][n_chunks][n_blocks]
    int n_blocks;       // sub-band kinds
    const uint32_t *codes;  // register windows: [n_dtiles][n_chunks][warps_dm][cch]
    int p_elems;        // sub-band kinds
    // [n_dtiles][n_ttiles] {first, end} range of the chunks whose staged
    // windows reach the input's nonzero columns, for plans that declare zero
    // input borders (the adjoint's transposed gather); chunks outside it only
    // add zeros. Read only by kernels compiled with LIVE; null otherwise.
    const int2 *live;
    int *err;
};

// The chunks a tile stages and sums: all of them, or (kernels compiled with
// LIVE, launched for plans that have a live table) the live range.
template <bool LIVE>
__device__ __forceinline__ int2 chunk_range(const FwdArgs &a, int dtile, int ttile) {
    if constexpr (LIVE) return a.live[(size_t)dtile * a.n_ttiles + ttile];
    return make_int2(0, (a.C + a.cch - 1) / a.cch);
}

// Loads the DPT uint16 smem offsets of this warp's trials with one vector
// load (4/8/16-byte aligned by construction of the tables).
template <int DPT>
__device__ __forceinline__ void load_offsets(const uint16_t *p, int (&o)[DPT]) {
    if constexpr (DPT == 8) {
        const uint4 v = *reinterpret_cast<const uint4 *>(p);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            o[2 * i] = int(w[i] & 0xffffu);
            o[2 * i + 1] = int(w[i] >> 16);
        }
    } else if constexpr (DPT == 4) {
        const uint2 v = *reinterpret_cast<const uint2 *>(p);
        o[0] = int(v.x & 0xffffu);
        o[1] = int(v.x >> 16);
        o[2] = int(v.y & 0xffffu);
        o[3] = int(v.y >> 16);
    } else {
        static_assert(DPT == 2, "DPT must be 2, 4 or 8");
        const uint32_t v = *reinterpret_cast<const uint32_t *>(p);
        o[0] = int(v & 0xffffu);
        o[1] = int(v >> 16);
    }
}

// Barrier over the first n threads of the CTA (named barrier 1): the
// compute warps of a kind-2 CTA synchronise without the producer warp.
__device__ __forceinline__ void compute_barrier(int n) {
    asm volatile("bar.sync 1, %0;" ::"r"(n) : "memory");
}

// The same barrier, returning whether any of the threads came with `p` set.
__device__ __forceinline__ bool compute_barrier_or(int n, bool p) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred a, b;\n\t"
        "setp.ne.u32 a, %1, 0;\n\t"
        "bar.red.or.pred b, 1, %2, a;\n\t"
        "selp.u32 %0, 1, 0, b;\n\t}"
        : "=r"(r)
        : "r"(uint32_t(p)), "r"(n)
        : "memory");
    return r != 0;
}

// Packed FP32 pair arithmetic of sm_100-class GPUs (one instruction for two
// lanes' worth of adds / fmas, each rounded to nearest like the scalar
// forms): a += b and d = a * b + d element-wise.
__device__ __forceinline__ void add2(float &a0, float &a1, float b0, float b1) {
    const float2 r = __fadd2_rn(make_float2(a0, a1), make_float2(b0, b1));
    a0 = r.x;
    a1 = r.y;
}
__device__ __forceinline__ void fma2(float &d0, float &d1, float a0, float a1, float b0, float b1) {
    const float2 r = __ffma2_rn(make_float2(a0, a1), make_float2(b0, b1), make_float2(d0, d1));
    d0 = r.x;
    d1 = r.y;
}

// ------------------------------------------------------------------ staging

// Per-tile staging context. Layout of a slot: [window data: stage_data_bytes]
// [tables: tab_bytes][weights: 16-byte rounded cch words][kinds 0, 1 and 5:
// the staging copies of the chunk `ahead` chunks on].
template <typename T>
struct Stager {
    const FwdArgs &a;
    const T *in_b;
    long long t0;
    const int4 *copies_k;  // this DM tile's staging copies
    const void *tab_k;    // kind 0/1: trial offsets; sub-band kinds: group offsets
    const void *tab2_k;   // second table: sub-band build blocks or window codes
    uint32_t tab_bytes;   // per chunk, both tables
    uint32_t tab1_bytes;  // per chunk, first table
    unsigned char *stage0;
    int stage_bytes;
    bool subband;
    int kc0;  // chunk k of the tile's loop is chunk kc0 + k of the plan

    // Bytes of a slot's weights.
    __device__ __forceinline__ int weight_bytes() const { return (a.cch * 4 + 15) & ~15; }

    // This lane's first staging copy of chunk k (copy `lane`; zero if none).
    __device__ __forceinline__ int4 desc(int k, int lane) const {
        return lane < a.n_copies ? copies_k[(size_t)(kc0 + k) * a.n_copies + lane]
                                 : make_int4(0, 0, 0, 0);
    }

    // Bytes copy d moves (a window may reach past the row's padded end only
    // in the last time tile; it is cut there, on a 16-byte boundary).
    __device__ __forceinline__ uint32_t copy_bytes(int4 d) const {
        return d.y ? uint32_t(min((long long)d.y, a.stride - (t0 + d.x))) * uint32_t(sizeof(T))
                   : 0u;
    }

    __device__ __forceinline__ void copy(unsigned char *sb, int c0, int4 d, uint64_t *full) const {
        const uint32_t bytes = copy_bytes(d);
        if (bytes)
            bulk_g2s(sb + (size_t)d.z * sizeof(T),
                     in_b + (long long)(c0 + d.w) * a.stride + t0 + d.x, bytes, full);
    }

    // Warp-cooperative: announces chunk k's bytes on `full` and, if told so,
    // issues its window copies (lane l copy l; at most 32 per chunk; `dsc`
    // preloaded); lane 0 copies the tables and weights. All 32 lanes of one
    // warp must call it. `ahead`: chunk k + ahead's staging copies come with
    // chunk k (0: none do).
    __device__ __forceinline__ void issue(int k, int slot, int4 dsc, uint64_t *full, int lane,
                                          int ahead = 0, bool windows = true) const {
        unsigned char *sb = stage0 + slot * stage_bytes;
        const int c0 = (kc0 + k) * a.cch;
        const int nch = min(a.cch, a.C - c0);
        uint32_t total = copy_bytes(dsc);
#pragma unroll
        for (int m = 16; m >= 1; m >>= 1) total += __shfl_xor_sync(0xffffffffu, total, m);
        // the chunk's weights, from a 16-byte boundary on
        const int w0 = c0 & ~3;
        const uint32_t w_bytes = uint32_t(((c0 - w0 + nch) * 4 + 15) & ~15);
        const uint32_t d_bytes = ahead ? uint32_t(a.n_copies) * 16u : 0u;
        if (lane == 0) mbar_arrive_expect_tx(full, total + tab_bytes + w_bytes + d_bytes);
        __syncwarp();
        fence_proxy_async_smem();
        if (windows) copy(sb, c0, dsc, full);
        if (lane == 0) {
            unsigned char *tb = sb + a.stage_data_bytes;
            if (!subband) {
                bulk_g2s(tb, static_cast<const uint16_t *>(tab_k) + (size_t)c0 * a.Dt, tab1_bytes,
                         full);
            } else {
                const int g0i = c0 / kSbG;
                bulk_g2s(tb, static_cast<const uint16_t *>(tab_k) + (size_t)g0i * a.Dt,
                         tab1_bytes, full);
            }
            if (tab_bytes > tab1_bytes) {
                const uint32_t b2 = tab_bytes - tab1_bytes;
                bulk_g2s(tb + tab1_bytes,
                         static_cast<const unsigned char *>(tab2_k) + (size_t)(kc0 + k) * b2, b2,
                         full);
            }
            // a 16-byte granule never crosses a page, so rounding the last
            // chunk up stays inside the weight buffer's page
            bulk_g2s(tb + tab_bytes, static_cast<const uint32_t *>(a.w) + w0, w_bytes, full);
            if (d_bytes)
                bulk_g2s(tb + tab_bytes + weight_bytes(),
                         copies_k + (size_t)(kc0 + k + ahead) * a.n_copies, d_bytes, full);
        }
    }

    // All warps of the CTA together: stage a tile's first chunks (n <= S of
    // them, into slots `slot`, slot + 1, ... modulo S, which nothing reads or
    // fills any more). Warp w issues copies w, w + n_warps, ... of every chunk;
    // one warp per chunk also announces the bytes (a copy may complete before
    // that: the barrier's phase still waits for the announcing arrival). One
    // warp alone takes 30-60 clocks per copy, which nothing hides at a tile's
    // start: 64 channels x 64 trials x 4096 samples, one tile per CTA, 7.5 ->
    // 6.1 us a launch. (The register windows' registers leave no room for this
    // form: 114.6 -> 116.9 us for 96 such beams; there warp 0 issues all.)
    __device__ __forceinline__ void issue_first(int n, int slot, int S, uint64_t *full, int warp,
                                                int n_warps, int lane, int ahead, int n_chunks) const {
        const int m = warp + lane * n_warps;
        fence_proxy_async_smem();
        for (int k = 0; k < n; ++k) {
            if (m < a.n_copies)
                copy(stage0 + slot * stage_bytes, (kc0 + k) * a.cch,
                     copies_k[(size_t)(kc0 + k) * a.n_copies + m], &full[slot]);
            if (warp == k % n_warps)
                issue(k, slot, desc(k, lane), &full[slot], lane,
                      ahead && k + ahead < n_chunks ? ahead : 0, false);
            if (++slot == S) slot = 0;
        }
    }
};

template <typename T>
__device__ __forceinline__ Stager<T> make_stager(const FwdArgs &a, int dtile, int b, long long t0,
                                                 unsigned char *stage0, bool subband, int kc0) {
    const int gpc = a.cch / kSbG;
    const int g_pad = a.C_pad / kSbG;
    Stager<T> s{a,
                static_cast<const T *>(a.in) + (long long)b * a.C * a.stride,
                t0,
                a.copies + (size_t)dtile * ((a.C + a.cch - 1) / a.cch) * a.n_copies,
                subband ? static_cast<const void *>(a.offs + (size_t)dtile * g_pad * a.Dt)
                        : static_cast<const void *>(a.offs + (size_t)dtile * a.C_pad * a.Dt),
                subband ? static_cast<const void *>(
                              a.bdesc + (size_t)dtile * ((a.C + a.cch - 1) / a.cch) * a.n_blocks)
                        : static_cast<const void *>(a.codes + (size_t)dtile * a.C_pad * a.warps_dm),
                subband ? uint32_t(gpc) * a.Dt * 2 + uint32_t(a.n_blocks) * 16
                        : uint32_t(a.cch) * (a.Dt * 2 + (a.codes ? a.warps_dm * 4 : 0)),
                subband ? uint32_t(gpc) * a.Dt * 2 : uint32_t(a.cch) * a.Dt * 2,
                stage0,
                a.stage_data_bytes + a.stage_offs_bytes,
                subband,
                kc0};
    return s;
}

// Stores a thread's accumulators (lane-strided sample mapping).
template <typename Acc, int DPT, int SPT>
__device__ __forceinline__ void store_lane_strided(const FwdArgs &a, const Acc (&acc)[DPT][SPT],
                                                   int dtile, int b, long long t0, int wd, int lb) {
    Acc *out = static_cast<Acc *>(a.out);
#pragma unroll
    for (int i = 0; i < DPT; ++i) {
        const int d = dtile * a.Dt + wd * DPT + i;
        if (d >= a.D) continue;
        Acc *orow = out + ((long long)b * a.D + d) * a.S + t0 + lb;
        const long long tmax = a.S - t0 - lb;
#pragma unroll
        for (int j = 0; j < SPT; ++j)
            if (32 * j < tmax) orow[32 * j] = acc[i][j];
    }
}

// Stores a thread's accumulators where it owns RUNS runs of consecutive
// samples (register windows: 2, sample j of run r in acc[i][2 j + r]; byte
// quads: 1): each warp turns one trial at a time around in its own 32 * SPT
// words of shared memory (the staging slots, which nothing reads any more once
// every warp has passed the barrier), so that the lanes' stores to global
// memory are coalesced. (An odd run length keeps the turn free of conflicts;
// the quads' 20 collide four ways, 0.3 % of their time at 256 channels.)
template <int RUNS, typename Acc, int DPT, int SPT>
__device__ __forceinline__ void store_runs(const FwdArgs &a, const Acc (&acc)[DPT][SPT], int dtile,
                                           int b, long long t0, int wd, int wt, int lane, int warp,
                                           volatile int *gave_up, unsigned char *stage0) {
    constexpr int M = SPT / RUNS;
    __syncthreads();
    if (!*gave_up) {
        Acc *buf = reinterpret_cast<Acc *>(stage0) + warp * 32 * SPT;
#pragma unroll
        for (int i = 0; i < DPT; ++i) {
            const int d = dtile * a.Dt + wd * DPT + i;
            if (d >= a.D) break;
#pragma unroll
            for (int j = 0; j < M; ++j)
#pragma unroll
                for (int r = 0; r < RUNS; ++r)
                    buf[32 * M * r + lane * M + j] = acc[i][RUNS * j + r];
            __syncwarp();
            Acc *orow = static_cast<Acc *>(a.out) + ((long long)b * a.D + d) * a.S + t0 +
                        wt * 32 * SPT + lane;
            const long long tmax = a.S - t0 - wt * 32 * SPT - lane;
#pragma unroll
            for (int j = 0; j < SPT; ++j)
                if (32 * j < tmax) orow[32 * j] = buf[32 * j + lane];
            __syncwarp();
        }
    }
    fence_proxy_async_smem();  // before the next tile's copies into these slots
}

// ------------------------------------------------------------------ kinds 0 and 1

// kind 0: lane-strided samples, one shared-memory read per add. kind 5
// (REUSE): the same, but a trial whose delay in the channel equals the
// previous trial's adds the operands already loaded for it; adjacent trials
// often share a channel's delay at low DMs and high frequencies, so this
// saves shared-memory reads there (it is a separate kernel because the test
// and branch slow down setups where no trials share a delay).
template <typename T, int DPT, int SPT, bool REUSE = false>
struct LaneStrided {
    using Acc = typename Elem<T>::Acc;
    using Wt = typename Elem<T>::W;
    __device__ static int sample_of(int j) { return 32 * j; }
    __device__ static int lane_base(int wt, int lane) { return wt * 32 * SPT + lane; }
    __device__ static void channel(Acc (&acc)[DPT][SPT], const T *sdata, int lane_base,
                                   const int (&o)[DPT], Wt wc) {
        const T *s = sdata + lane_base;
        if constexpr (REUSE) {
            Acc v[SPT];
#pragma unroll
            for (int i = 0; i < DPT; ++i) {
                if (i == 0 || o[i] != o[i - 1]) {
                    const T *src = s + o[i];
#pragma unroll
                    for (int j = 0; j < SPT; ++j) v[j] = Elem<T>::val(src[32 * j]);
                }
#pragma unroll
                for (int j = 0; j < SPT; ++j) acc[i][j] += wc * v[j];
            }
        } else {
#pragma unroll
            for (int i = 0; i < DPT; ++i) {
                const T *src = s + o[i];
#pragma unroll
                for (int j = 0; j < SPT; ++j) acc[i][j] += wc * Elem<T>::val(src[32 * j]);
            }
        }
    }
};

// Grouped sums (float input, 2 x 4, 4 x 2 and 4 x 8 outputs per thread): four
// channels' products of an output are summed first and then added to its
// accumulator, a sub-band kernel's operations in the same order, so that both
// give the same bits and a plan may take either. The reads stay one shared word
// per add, which bounds the loop as before: 0.97 to 1.04 of the single chain's
// speed per tile shape, in the geometric mean over 27 setups of 4 to 101 trials
// (384 beams x 64 channels x 4 trials x 4096 samples, FP32: 72.9 -> 72.0 us,
// largest error 1.7e-7 -> 8.2e-8 of the largest output; one beam, 64 trials: 6.6
// -> 6.4). Two groups are unrolled in the small tiles (2 x 4, 16-bit, one beam:
// 5.9 -> 5.7 us).
template <typename T, int DPT, int SPT>
struct GroupedLanes {
    static constexpr int U = DPT * SPT > 8 ? 1 : 2;  // groups with their loads in flight at once

    // A chunk's nch channels; `offs` the warp's trial offsets, Dt apart.
    static __device__ __forceinline__ void chunk(float (&acc)[DPT][SPT], const T *s,
                                                 const uint16_t *offs, int Dt, const float *sw,
                                                 int nch) {
        int cc = 0;
#pragma unroll U
        for (; cc + kSbG <= nch; cc += kSbG) {
            const float4 w = *reinterpret_cast<const float4 *>(sw + cc);
            int o[kSbG][DPT];
#pragma unroll
            for (int q = 0; q < kSbG; ++q) load_offsets<DPT>(offs + (cc + q) * Dt, o[q]);
#pragma unroll
            for (int i = 0; i < DPT; ++i) {
                float v[SPT];
#pragma unroll
                for (int j = 0; j < SPT; ++j)
                    v[j] = __fmul_rn(w.x, Elem<T>::val(s[o[0][i] + 32 * j]));
#pragma unroll
                for (int q = 1; q < kSbG; ++q) {
                    const float wq = q == 1 ? w.y : (q == 2 ? w.z : w.w);
                    const T *t = s + o[q][i];
#pragma unroll
                    for (int j = 0; j < SPT; j += 2)
                        fma2(v[j], v[j + 1], wq, wq, Elem<T>::val(t[32 * j]),
                             Elem<T>::val(t[32 * j + 32]));
                }
#pragma unroll
                for (int j = 0; j < SPT; j += 2) add2(acc[i][j], acc[i][j + 1], v[j], v[j + 1]);
            }
        }
        if (cc < nch) {  // the plan's last group may hold fewer channels
#pragma unroll
            for (int i = 0; i < DPT; ++i) {
                float v[SPT];
                const T *t = s + offs[cc * Dt + i];
#pragma unroll
                for (int j = 0; j < SPT; ++j) v[j] = __fmul_rn(sw[cc], Elem<T>::val(t[32 * j]));
#pragma unroll 1
                for (int c = cc + 1; c < nch; ++c) {
                    t = s + offs[c * Dt + i];
#pragma unroll
                    for (int j = 0; j < SPT; ++j)
                        v[j] = __fmaf_rn(sw[c], Elem<T>::val(t[32 * j]), v[j]);
                }
#pragma unroll
                for (int j = 0; j < SPT; ++j) acc[i][j] = __fadd_rn(acc[i][j], v[j]);
            }
        }
    }
};

// kind 1: thread-contiguous samples served from a register window.
template <typename T, int DPT, int SPT>
struct RegWindow {
    using Acc = typename Elem<T>::Acc;
    using Wt = typename Elem<T>::W;
    static_assert(SPT % 2 == 1, "odd samples_per_thread keeps window loads conflict-free");
    static constexpr int R = kRwRmax;
    __device__ static int sample_of(int j) { return j; }
    __device__ static int lane_base(int wt, int lane) { return wt * 32 * SPT + lane * SPT; }

    template <int RR>
    __device__ static __forceinline__ void add_shifted(Acc (&a)[SPT], const Acc (&win)[SPT + R],
                                                       Wt wc) {
#pragma unroll
        for (int j = 0; j < SPT; ++j) a[j] += wc * win[RR + j];
    }

    __device__ static void channel(Acc (&acc)[DPT][SPT], const T *sdata, int lane_base,
                                   const int (&o)[DPT], Wt wc) {
        int gb = o[0], gm = o[0];
#pragma unroll
        for (int i = 1; i < DPT; ++i) {
            gb = min(gb, o[i]);
            gm = max(gm, o[i]);
        }
        const int span = gm - gb;  // warp-uniform
        const T *src = sdata + lane_base + gb;
        if (span <= R) {
            Acc win[SPT + R];
#pragma unroll
            for (int k = 0; k < SPT; ++k) win[k] = Elem<T>::val(src[k]);
#pragma unroll
            for (int k = SPT; k < SPT + R; ++k)
                win[k] = (k < SPT + span) ? Elem<T>::val(src[k]) : Acc(0);
#pragma unroll
            for (int i = 0; i < DPT; ++i) {
                switch (o[i] - gb) {
#define DD_RW_CASE(RR) \
    case RR: add_shifted<RR>(acc[i], win, wc); break;
                    DD_RW_CASE(0) DD_RW_CASE(1) DD_RW_CASE(2) DD_RW_CASE(3) DD_RW_CASE(4)
                    DD_RW_CASE(5) DD_RW_CASE(6) DD_RW_CASE(7) DD_RW_CASE(8) DD_RW_CASE(9)
                    DD_RW_CASE(10) DD_RW_CASE(11) DD_RW_CASE(12) DD_RW_CASE(13) DD_RW_CASE(14)
                    default: add_shifted<15>(acc[i], win, wc); break;
#undef DD_RW_CASE
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < DPT; ++i) {
                const T *s = src + (o[i] - gb);
#pragma unroll
                for (int j = 0; j < SPT; ++j) acc[i][j] += wc * Elem<T>::val(s[j]);
            }
        }
    }
};

// Register windows (kind 5 with 2 * odd samples per thread). Lane l of a warp
// owns two runs of M = SPT / 2 consecutive samples, [l M, l M + M) and the
// same 32 M samples later, for the DPT = 4 trials of its warp. Per channel it
// loads the union window of its trials, M + (delay span) words per run, once
// into registers and serves all four trials from it; which register holds a
// trial's sample depends on the delay steps between the trials, so every
// combination of steps within a band {b, b + 1} (all that an evenly spaced
// DM grid produces) is a case of its own with compile-time positions,
// entered by one warp-uniform jump per channel. The two runs make the
// operands of the packed pair arithmetic: samples j of both runs sit in one
// register pair whatever the delay. M is odd, so the lanes' loads are
// conflict-free at every offset. Channels whose steps fit no case read one
// word per add, like kind 0. Bound by issue slots and the shared-memory pipe
// about equally (122 instructions per channel for 88 adds a thread at M = 11,
// the pipe 68 % busy); two CTAs of 8 warps hide a tile's start and end better
// than one of 16 (survey scale: 2.39 against 2.50 ms). Measured, FP32: 96 beams
// x 64 channels x 64 trials x 4096 samples 0.187 ms (kind 5, equal delays) ->
// 0.115; 16 beams x 512 channels x 1024 trials x 8192 samples 3.84 (kind 6) ->
// 3.60 ms; survey scale 2.39 against kind 6's 2.34 ms.
template <typename T, int SPT>
struct Window {
    using Acc = typename Elem<T>::Acc;
    using Wt = typename Elem<T>::W;
    static constexpr int DPT = 4, M = SPT / 2, H = 32 * M;

    static __device__ __forceinline__ void add(Acc &a0, Acc &a1, Wt w, Acc x0, Acc x1) {
        if constexpr (std::is_same<Acc, float>::value) {
            fma2(a0, a1, w, w, x0, x1);
        } else {
            a0 += w * x0;
            a1 += w * x1;
        }
    }

    // acc[i][2 j + r] += w * s[d_i + j + r H], d = (0, S1, S1 + S2, S1 + S2 + S3)
    template <int S1, int S2, int S3>
    static __device__ __forceinline__ void serve(Acc (&acc)[DPT][SPT], const T *s, Wt w) {
        constexpr int d[DPT] = {0, S1, S1 + S2, S1 + S2 + S3};
#pragma unroll
        for (int k = 0; k < M + d[DPT - 1]; ++k) {
            const Acc x0 = Elem<T>::val(s[k]), x1 = Elem<T>::val(s[k + H]);
#pragma unroll
            for (int i = 0; i < DPT; ++i) {
                const int j = k - d[i];
                if (j >= 0 && j < M) add(acc[i][2 * j], acc[i][2 * j + 1], w, x0, x1);
            }
        }
    }

    static __device__ __forceinline__ void channel(Acc (&acc)[DPT][SPT], const T *sl, uint32_t code,
                                                   const uint16_t *offs, Wt w) {
        const T *s = sl + (code & 0xffffu);
        switch (code >> 16) {
#define DD_WIN_CASE(B_, K_)                                                          \
    case 7 * B_ + K_:                                                                \
        serve<B_ + (K_ & 1), B_ + ((K_ >> 1) & 1), B_ + ((K_ >> 2) & 1)>(acc, s, w); \
        break;
#define DD_WIN_BAND(B_)                                                         \
    DD_WIN_CASE(B_, 0) DD_WIN_CASE(B_, 1) DD_WIN_CASE(B_, 2) DD_WIN_CASE(B_, 3) \
    DD_WIN_CASE(B_, 4) DD_WIN_CASE(B_, 5) DD_WIN_CASE(B_, 6)
            DD_WIN_BAND(0) DD_WIN_BAND(1) DD_WIN_BAND(2) DD_WIN_BAND(3) DD_WIN_BAND(4)
            DD_WIN_CASE(4, 7)
#undef DD_WIN_BAND
#undef DD_WIN_CASE
            case kWinNone: {
                int o[DPT];
                load_offsets<DPT>(offs, o);
#pragma unroll
                for (int i = 0; i < DPT; ++i) {
                    const T *t = sl + o[i];
#pragma unroll
                    for (int j = 0; j < M; ++j)
                        add(acc[i][2 * j], acc[i][2 * j + 1], w, Elem<T>::val(t[j]),
                            Elem<T>::val(t[j + H]));
                }
                break;
            }
            default: __builtin_unreachable();
        }
    }
};

// Byte quads (kind 0 with 20 samples per thread, 8-bit input). Lane l of a
// warp owns M = 20 consecutive samples, M / 4 = 5 words apart from its
// neighbours' (an odd number: the lanes' word loads are conflict-free), and
// takes the channels two at a time. Per trial and channel it reads the M / 4 +
// 1 words that hold its samples, 0.3 words per add where kind 0's byte loads
// read one, shifts them by the delay's two low bits, interleaves the two
// channels' bytes and adds both channels' products with one 16-bit by 8-bit
// dot product per sample. Weights beyond 16 bits take byte extracts and
// multiply-adds. Whole numbers: the sums are the same bits in any order. Bound
// by issue slots (1.8 per add at 0.74 a clock; shared-memory pipe 51 %, integer
// pipe 59 % busy). 32 beams x 256 channels over 120-180 MHz x 2000 trials x
// 10000 samples: 17.8 ms (kind 0, 8 x 8) -> 10.2 ms; survey scale 2.65 against
// the sub-bands' 2.25 ms. (Four channels at a time would halve the dot
// products of weights below 256 but needs a byte transpose, as many integer
// instructions more.)
template <int SPT>
struct Quads {
    static constexpr int DPT = 4, Q = SPT / 4;

    // acc += (wc.lo, wc.hi) . two bytes of b: bytes 0, 1 or bytes 2, 3
    static __device__ __forceinline__ void dot_lo(int &acc, uint32_t wc, uint32_t b) {
        asm("dp2a.lo.s32.u32 %0, %1, %2, %0;" : "+r"(acc) : "r"(wc), "r"(b));
    }
    static __device__ __forceinline__ void dot_hi(int &acc, uint32_t wc, uint32_t b) {
        asm("dp2a.hi.s32.u32 %0, %1, %2, %0;" : "+r"(acc) : "r"(wc), "r"(b));
    }
    // the thread's samples of a channel for a trial at byte offset o
    static __device__ __forceinline__ void words(uint32_t (&v)[Q], const uint8_t *sl, int o) {
        const uint32_t *p = reinterpret_cast<const uint32_t *>(sl + (o & ~3));
        const uint32_t sh = uint32_t(o) << 3;  // the funnel shift takes it modulo 32
        uint32_t r[Q + 1];
#pragma unroll
        for (int k = 0; k <= Q; ++k) r[k] = p[k];
#pragma unroll
        for (int k = 0; k < Q; ++k) v[k] = __funnelshift_r(r[k], r[k + 1], sh);
    }
    // Two channels: offsets oa and ob, weights wa and wb (NARROW: both fit 16
    // bits).
    template <bool NARROW>
    static __device__ __forceinline__ void channels(int (&acc)[DPT][SPT], const uint8_t *sl,
                                                    const int (&oa)[DPT], const int (&ob)[DPT],
                                                    int wa, int wb) {
        const uint32_t wc = __byte_perm(uint32_t(wa), uint32_t(wb), 0x5410);
#pragma unroll
        for (int i = 0; i < DPT; ++i) {
            uint32_t a[Q], b[Q];
            words(a, sl, oa[i]);
            words(b, sl, ob[i]);
#pragma unroll
            for (int k = 0; k < Q; ++k) {
                if constexpr (NARROW) {
                    const uint32_t lo = __byte_perm(a[k], b[k], 0x5140);
                    const uint32_t hi = __byte_perm(a[k], b[k], 0x7362);
                    dot_lo(acc[i][4 * k], wc, lo);
                    dot_hi(acc[i][4 * k + 1], wc, lo);
                    dot_lo(acc[i][4 * k + 2], wc, hi);
                    dot_hi(acc[i][4 * k + 3], wc, hi);
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        acc[i][4 * k + j] += wa * int(a[k] >> (8 * j) & 0xffu) +
                                             wb * int(b[k] >> (8 * j) & 0xffu);
                }
            }
        }
    }

    // A chunk's nch channels; `offs` the warp's trial offsets, Dt apart.
    template <bool NARROW>
    static __device__ __forceinline__ void chunk(int (&acc)[DPT][SPT], const uint8_t *sl,
                                                 const uint16_t *offs, int Dt, const int *sw,
                                                 int nch) {
#pragma unroll 1
        for (int cc = 0; cc < nch; cc += 2) {
            // an odd last channel is paired with itself at weight 0
            const int cb = min(cc + 1, nch - 1);
            int oa[DPT], ob[DPT];
            load_offsets<DPT>(offs + cc * Dt, oa);
            load_offsets<DPT>(offs + cb * Dt, ob);
            channels<NARROW>(acc, sl, oa, ob, sw[cc], cb > cc ? sw[cb] : 0);
        }
    }
};

// Barriers: every kind uses full[s] = bars[s] (producer arrival + bytes) and
// empty[s] = bars[8 + s]: one arrival per warp for kinds 0/1, one per chunk
// for kind 2 (after its compute barrier), one per builder warp for kind 3,
// which also uses
// bars[4..6] / bars[12..14] for its partial-sum slots and counts builder
// warps on the staging slots' empty barriers.
template <int KIND>
__device__ __forceinline__ void fwd_init_barriers(uint64_t *bars, int stages) {
    if (threadIdx.x == 0) {
        const int n_warps = int(blockDim.x >> 5);
        const int releasers = KIND == 3 ? kWsBuilders : (is_subband(KIND) ? 1 : n_warps);
        for (int s = 0; s < stages; ++s) {
            mbar_init(&bars[s], 1);
            mbar_init(&bars[8 + s], uint32_t(releasers));
        }
        *reinterpret_cast<volatile int *>(&bars[7]) = 0;  // the CTA's give-up flag
        if (KIND == 3) {
            for (int q = 0; q < kWsPSlots; ++q) {
                mbar_init(&bars[4 + q], uint32_t(kWsBuilders));
                mbar_init(&bars[12 + q], uint32_t(n_warps - kWsBuilders));
            }
        }
        fence_barrier_init();
    }
    __syncthreads();
}

// Kinds 0, 1 and 5. `kbase` counts the chunks this CTA has already pushed
// through its slots; chunk kg uses slot kg % stages, and the n-th completion
// of a slot's full/empty barrier belongs to chunk slot + n * stages, so the
// phase parities carry over from tile to tile without re-initialisation.
template <int KIND, typename T, int DPT, int SPT, bool LIVE>
__device__ __forceinline__ void fwd_tile(const FwdArgs &a, int dtile, int ttile, int b,
                                         uint64_t *bars, unsigned char *stage0,
                                         uint32_t &kbase) {
    using P = typename std::conditional<
        KIND == 1, RegWindow<T, DPT, SPT>, LaneStrided<T, DPT, SPT, KIND == 5>>::type;
    using Acc = typename Elem<T>::Acc;
    using Wt = typename Elem<T>::W;
    constexpr bool WIN = is_window(KIND, SPT), QUAD = is_quad(KIND, SPT);
    constexpr bool GROUPS = sums_groups(KIND, DPT, SPT) && std::is_same<Acc, float>::value;
    // With two slots, a refill at the end of a chunk leaves no copy in flight
    // during the next one; the kernels with the largest tiles, whose slots
    // leave no room for a third, refill before they sum a chunk (LOFAR, 8
    // trials x 4096 samples, two channels per slot: 2.94 -> 2.07 ms). The
    // others keep the one place: a second copy of the staging code slows them
    // (register windows at the survey scale: 2.41 -> 2.58 ms).
    constexpr bool EARLY = KIND == 0 && DPT * SPT == 64;
    uint64_t *full = bars, *empty = bars + 8;
    volatile int *gave_up = reinterpret_cast<volatile int *>(&bars[7]);
    const uint32_t S = uint32_t(a.stages);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wd = warp % a.warps_dm, wt = warp / a.warps_dm;
    const long long t0 = (long long)ttile * a.Ts;
    const int2 kr = chunk_range<LIVE>(a, dtile, ttile);
    const int n_chunks = kr.y - kr.x;
    const Stager<T> st = make_stager<T>(a, dtile, b, t0, stage0, false, kr.x);

    // Staging: all warps (windows: warp 0) issue the first S chunks; chunk kn >= S is issued by the
    // warps in turn, at the end of their chunk kn - S + 1, once every warp has
    // released chunk kn - S (one chunk of slack for slower warps). Issuing a
    // chunk's copies takes one warp 1-2 thousand clocks; with warp 0 issuing
    // every chunk, the whole CTA waited for it. Chunk kn's copy list comes with
    // chunk kn - S + 1, so that no global load stands before them. Kind 0 at
    // 1024 channels x 2048 trials x 20000 samples, FP32, 32-trial tiles: 5.56
    // -> 4.71 ms; 64 channels x 64 trials x 4096 samples: 18.4 -> 15.1 us.
    const int n_warps = int(blockDim.x >> 5);
    auto ahead = [&](int k) {
        return a.copies_ahead && k + int(S) - 1 < n_chunks ? int(S) - 1 : 0;
    };
    int slot = int(kbase % S), turn = 0;
    uint32_t parity = (kbase / S) & 1u;
    // the slots' earlier chunks were released by every warp before this tile
    if constexpr (WIN) {
        if (warp == 0)
            for (int k = 0, sl = slot; k < min(int(S), n_chunks); ++k) {
                st.issue(k, sl, st.desc(k, lane), &full[sl], lane, ahead(k));
                if (++sl == int(S)) sl = 0;
            }
    } else {
        st.issue_first(min(int(S), n_chunks), slot, int(S), full, warp, n_warps, lane,
                       a.copies_ahead ? int(S) - 1 : 0, n_chunks);
    }

    Acc acc[DPT][SPT];
#pragma unroll
    for (int i = 0; i < DPT; ++i)
#pragma unroll
        for (int j = 0; j < SPT; ++j) acc[i][j] = Acc(0);
    const int lb = WIN    ? wt * 32 * SPT + lane * (SPT / 2)
                   : QUAD ? wt * 32 * SPT + lane * SPT
                          : P::lane_base(wt, lane);

    // stages the chunk that goes into chunk k - 1's slot (sb: chunk k's slot)
    auto refill = [&](int k, const unsigned char *sb) {
        const int kn = k - 1 + int(S);
        if (k < 1 || kn >= n_chunks || warp != turn) return;
        int4 dsc = make_int4(0, 0, 0, 0);
        if (!a.copies_ahead)
            dsc = st.desc(kn, lane);
        else if (lane < a.n_copies)
            dsc = reinterpret_cast<const int4 *>(sb + a.stage_data_bytes + st.tab_bytes +
                                                 st.weight_bytes())[lane];
        const int prev = slot ? slot - 1 : int(S) - 1;
        // chunk k - 1's release: the same phase as its full barrier's
        const uint32_t par = slot ? parity : parity ^ 1u;
        const bool ok = mbar_wait_bounded(&empty[prev], par, a.err, kWaitBudgetNs, gave_up);
        if (__all_sync(0xffffffffu, ok))
            st.issue(kn, prev, dsc, &full[prev], lane, ahead(kn));
    };
    for (int k = 0; k < n_chunks; ++k) {
        // A failed wait (or one that finds the CTA's give-up flag set) ends
        // the tile: the slot may hold a stale chunk, so nothing more is
        // summed, released or stored.
        if (!__all_sync(0xffffffffu,
                        mbar_wait_bounded(&full[slot], parity, a.err, kWaitBudgetNs, gave_up)))
            break;
        const unsigned char *sb = stage0 + slot * st.stage_bytes;
        const T *sdata = reinterpret_cast<const T *>(sb);
        const uint16_t *soffs =
            reinterpret_cast<const uint16_t *>(sb + a.stage_data_bytes) + wd * DPT;
        const int c0 = (kr.x + k) * a.cch, nch = min(a.cch, a.C - c0);
        const Wt *sw =
            reinterpret_cast<const Wt *>(sb + a.stage_data_bytes + st.tab_bytes) + (c0 & 3);
        if (EARLY && S == 2) refill(k, sb);
        if constexpr (WIN) {
            const uint32_t *codes =
                reinterpret_cast<const uint32_t *>(sb + a.stage_data_bytes + st.tab1_bytes) +
                wd * a.cch;
            uint32_t code = codes[0];
            Wt wc = sw[0];
#pragma unroll 1
            for (int cc = 0; cc < nch; ++cc) {
                // read one channel ahead, never past the chunk's last channel
                const int cn = min(cc + 1, nch - 1);
                const uint32_t code_next = codes[cn];
                const Wt w_next = sw[cn];
                Window<T, SPT>::channel(acc, sdata + lb, code, soffs + cc * a.Dt, wc);
                code = code_next;
                wc = w_next;
            }
        } else if constexpr (QUAD) {
            const int wl = lane < nch ? sw[lane] : 0;  // nch <= 32
            if (__all_sync(0xffffffffu, wl == int(short(wl))))
                Quads<SPT>::template chunk<true>(acc, sdata + lb, soffs, a.Dt, sw, nch);
            else
                Quads<SPT>::template chunk<false>(acc, sdata + lb, soffs, a.Dt, sw, nch);
        } else if constexpr (GROUPS) {
            GroupedLanes<T, DPT, SPT>::chunk(acc, sdata + lb, soffs, a.Dt, sw, nch);
        } else {
            for (int cc = 0; cc < nch; ++cc) {
                int o[DPT];
                load_offsets<DPT>(soffs + cc * a.Dt, o);
                P::channel(acc, sdata, lb, o, sw[cc]);
            }
        }
        if (!(EARLY && S == 2)) refill(k, sb);
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[slot]);
        if (k >= 1 && ++turn == n_warps) turn = 0;
        if (++slot == int(S)) {
            slot = 0;
            parity ^= 1u;
        }
    }
    kbase += uint32_t(n_chunks);
    if constexpr (WIN || QUAD) {
        store_runs<WIN ? 2 : 1, Acc, DPT, SPT>(a, acc, dtile, b, t0, wd, wt, lane, warp, gave_up,
                                               stage0);
        return;
    }
    if (*gave_up) return;

    Acc *out = static_cast<Acc *>(a.out);
#pragma unroll
    for (int i = 0; i < DPT; ++i) {
        const int d = dtile * a.Dt + wd * DPT + i;
        if (d >= a.D) continue;
        Acc *orow = out + ((long long)b * a.D + d) * a.S + t0 + lb;
        const long long tmax = a.S - t0 - lb;
#pragma unroll
        for (int j = 0; j < SPT; ++j) {
            const int off = P::sample_of(j);
            if (off < tmax) orow[off] = acc[i][j];
        }
    }
}

// ------------------------------------------------------------------ kinds 2 and 3

// Builds this worker's share of a chunk's partial series from the chunk's
// build blocks. A block covers up to 4 sub-blocks of 32 consecutive
// elements of one series: {dst, r0, (r1-r0) | (r2-r0) << 16, (r3-r0) |
// group << 16 | channels << 20 | sub-blocks << 24}, and lane l of sub-block s
// writes P[dst + 32 s + l] = sum_{j < channels} w[4 group + j] *
// raw[r_j + 32 s + l]. Worker `part` of `parts` takes blocks part, part +
// parts, ...; the next block's descriptor is loaded while the current one is
// built, and all of a block's operand loads are issued before its
// arithmetic. Blocks with 0 sub-blocks are capacity padding; they sit after
// every real block of the chunk, so a worker stops at its first one.
template <typename T>
__device__ __forceinline__ void sb_build_blocks(typename Elem<T>::Acc *P, const T *raw,
                                                const int4 *blk, const typename Elem<T>::W *sw,
                                                int n_blocks, int part, int parts, int lane) {
    using Acc = typename Elem<T>::Acc;
    using Wt = typename Elem<T>::W;
    static_assert(sizeof(Wt) == 4, "weights are 4-byte words");
    int b = part;
    int4 d = b < n_blocks ? blk[b] : make_int4(0, 0, 0, 0);
    while (b < n_blocks) {
        const int bn = b + parts;
        const int4 dn = bn < n_blocks ? blk[bn] : make_int4(0, 0, 0, 0);
        const int nsub = (d.w >> 24) & 7;
        if (!nsub) break;
        {
            const int g = (d.w >> 16) & 7, gn = (d.w >> 20) & 7;
            const int4 wv = *reinterpret_cast<const int4 *>(sw + 4 * g);
            const Wt w[4] = {__builtin_bit_cast(Wt, wv.x), __builtin_bit_cast(Wt, wv.y),
                             __builtin_bit_cast(Wt, wv.z), __builtin_bit_cast(Wt, wv.w)};
            const int r0 = d.y + lane;
            const int r[4] = {r0, r0 + int(short(d.z & 0xffff)), r0 + (d.z >> 16),
                              r0 + int(short(d.w & 0xffff))};
            Acc x[4][4];  // [sub-block][channel]
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (q < nsub) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) x[q][j] = Elem<T>::val(raw[r[j] + 32 * q]);
                }
            Acc v[4];
            if (gn == kSbG) {
                if constexpr (std::is_same<Acc, float>::value) {
#pragma unroll
                    for (int q = 0; q < 4; q += 2) {
                        v[q] = w[0] * x[q][0];
                        v[q + 1] = w[0] * x[q + 1][0];
#pragma unroll
                        for (int j = 1; j < 4; ++j)
                            fma2(v[q], v[q + 1], w[j], w[j], x[q][j], x[q + 1][j]);
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        v[q] = w[0] * x[q][0] + w[1] * x[q][1] + w[2] * x[q][2] + w[3] * x[q][3];
                }
            } else {  // the last group of a plan may hold fewer channels
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    v[q] = w[0] * x[q][0];
#pragma unroll
                    for (int j = 1; j < kSbG; ++j)
                        if (j < gn) v[q] += w[j] * x[q][j];
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (q < nsub) P[d.x + 32 * q + lane] = v[q];
        }
        d = dn;
        b = bn;
    }
}

// The packed 16-bit offsets of all the chunk's groups are loaded first, so
// their shared-memory latency is paid once per chunk rather than per group.
template <int DPT>
struct OffWords {
    uint32_t w[DPT / 2];
};
template <int DPT>
__device__ __forceinline__ OffWords<DPT> load_offwords(const uint16_t *p) {
    OffWords<DPT> r;
    if constexpr (DPT == 8) {
        const uint4 v = *reinterpret_cast<const uint4 *>(p);
        r.w[0] = v.x, r.w[1] = v.y, r.w[2] = v.z, r.w[3] = v.w;
    } else if constexpr (DPT == 4) {
        const uint2 v = *reinterpret_cast<const uint2 *>(p);
        r.w[0] = v.x, r.w[1] = v.y;
    } else {
        r.w[0] = *reinterpret_cast<const uint32_t *>(p);
    }
    return r;
}

template <typename Acc, int DPT, int SPT>
__device__ __forceinline__ void sb_trials4(Acc (&acc)[DPT][SPT], const Acc *Pl,
                                           const uint16_t *poffs, int Dt, int ng) {
    OffWords<DPT> ow[4];
#pragma unroll
    for (int g = 0; g < 4; ++g)
        if (g < ng) ow[g] = load_offwords<DPT>(poffs + g * Dt);
#pragma unroll
    for (int g = 0; g < 4; ++g) {  // up to 4 groups (16 channels) at a time
        if (g < ng) {
            int o[DPT];
#pragma unroll
            for (int i = 0; i < DPT / 2; ++i) {
                o[2 * i] = int(ow[g].w[i] & 0xffffu);
                o[2 * i + 1] = int(ow[g].w[i] >> 16);
            }
            // trials of a thread that share the group's series and offset
            // (same pattern, same base delay) reuse the loaded values
            Acc v[SPT];
#pragma unroll
            for (int i = 0; i < DPT; ++i) {
                const Acc *src = Pl + o[i];
                if constexpr (std::is_same<Acc, float>::value && SPT % 2 == 0) {
                    if (i == 0 || o[i] != o[i - 1]) {
#pragma unroll
                        for (int j = 0; j < SPT; ++j) v[j] = src[32 * j];
                    }
#pragma unroll
                    for (int j = 0; j < SPT; j += 2)
                        add2(acc[i][j], acc[i][j + 1], v[j], v[j + 1]);
                } else {
#pragma unroll
                    for (int j = 0; j < SPT; ++j) acc[i][j] += src[32 * j];
                }
            }
        }
    }
}

// The trial loop over a chunk's ng groups, four at a time. PASSES: 1 = at
// most 4 groups (16 channels); 2 = up to 8 (32 channels) as two inlined
// passes; 0 = up to 8 as a loop over one copy of the pass. Which form is
// fastest depends on the kernel (GB300, survey scale): the FP32 kinds 2-4
// keep one pass (a second one, even never taken, cost 5.7 %); 8-bit input
// takes two inlined passes (2.26 against 2.32 ms as a loop); 16-bit input
// and kind 6 take the loop (16-bit kind 4: 2.37 against 2.44 ms; FP32 kind
// 6: 2.34 against 2.55 ms, where the inlined form spills).
template <int PASSES, typename Acc, int DPT, int SPT>
__device__ __forceinline__ void sb_trials(Acc (&acc)[DPT][SPT], const Acc *Pl,
                                          const uint16_t *poffs, int Dt, int ng) {
    if constexpr (PASSES == 1) {
        sb_trials4<Acc, DPT, SPT>(acc, Pl, poffs, Dt, ng);
    } else if constexpr (PASSES == 2) {
        sb_trials4<Acc, DPT, SPT>(acc, Pl, poffs, Dt, min(ng, 4));
        if (ng > 4) sb_trials4<Acc, DPT, SPT>(acc, Pl, poffs + 4 * Dt, Dt, ng - 4);
    } else {
#pragma unroll 1
        for (int g0 = 0; g0 < ng; g0 += 4)
            sb_trials4<Acc, DPT, SPT>(acc, Pl, poffs + g0 * Dt, Dt, min(ng - g0, 4));
    }
}

// The trial-loop form of a sub-band kernel (see sb_trials).
template <typename T, bool ONE_SLOT>
__host__ __device__ constexpr int sb_passes() {
    return sizeof(T) == 1 ? 2 : ((ONE_SLOT || sizeof(T) == 2) ? 0 : 1);
}

// kind 2: sub-band partial sums with a producer warp. Warps [0, NC) compute;
// warp NC only stages chunks, running up to `stages` chunks ahead and
// throttled by the slots' empty barriers (one arrival per chunk, made after
// the compute warps' build barrier). Per chunk the compute warps build the
// partial series (and copy the chunk's trial offsets next to them), meet at
// a named barrier, release the staging slot and run the trial loop.
// Partial-sum slots alternate by global chunk parity, so a chunk's build
// never overwrites what slower warps still read. (Replacing the barrier by
// per-warp mbarrier hand-offs, so that a warp builds chunk k+1 before its
// trials on chunk k, measured slower on GB300.)
// ONE_SLOT (kind 6): a single partial-sum slot, so that FP32 input fits
// 32-channel chunks; a second barrier per chunk then keeps the next build
// from overwriting series that slower warps still read.
template <typename T, int DPT, int SPT, bool LIVE, bool ONE_SLOT = false>
__device__ __forceinline__ void fwd_tile_sb(const FwdArgs &a, int dtile, int ttile, int b,
                                            uint64_t *bars, unsigned char *stage0,
                                            uint32_t &kbase) {
    using Acc = typename Elem<T>::Acc;
    using Wt = typename Elem<T>::W;
    uint64_t *full = bars, *empty = bars + 8;
    volatile int *gave_up = reinterpret_cast<volatile int *>(&bars[7]);
    const uint32_t S = uint32_t(a.stages);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nc = int(blockDim.x >> 5) - 1;  // compute warps; warp nc produces
    const long long t0 = (long long)ttile * a.Ts;
    const int2 kr = chunk_range<LIVE>(a, dtile, ttile);
    const int n_chunks = kr.y - kr.x;
    const Stager<T> st = make_stager<T>(a, dtile, b, t0, stage0, true, kr.x);
    const uint32_t poffs_bytes = st.tab1_bytes;
    const int pslot_bytes = a.p_elems * int(sizeof(Acc)) + int(poffs_bytes);
    unsigned char *pslot0 = stage0 + S * st.stage_bytes;
    // the slots' earlier chunks were released before this tile
    st.issue_first(min(int(S), n_chunks), int(kbase % S), int(S), full, warp, nc + 1, lane, 0,
                   n_chunks);

    if (warp == nc) {
        // ---------------- producer warp
        // Channel descriptors are loaded kDescAhead chunks before their copy
        // is issued, so the issue rate is not bound by one global-memory
        // latency per chunk.
        // The ring is indexed by compile-time positions (the loop over j is
        // unrolled), so a descriptor is loaded into the register it is
        // consumed from kDescAhead chunks later, with no move that would wait
        // for the load.
        int4 q[kDescAhead];
#pragma unroll
        for (int j = 0; j < kDescAhead; ++j)
            q[j] = int(S) + j < n_chunks ? st.desc(int(S) + j, lane) : make_int4(0, 0, 0, 0);
        for (int k0 = int(S); k0 < n_chunks; k0 += kDescAhead) {
#pragma unroll
            for (int j = 0; j < kDescAhead; ++j) {
                const int k = k0 + j;
                if (k < n_chunks) {
                    const uint32_t kg = kbase + uint32_t(k);
                    const int slot = int(kg % S);
                    const bool ok = mbar_wait_bounded(&empty[slot], ((kg / S) - 1u) & 1u, a.err,
                                                      kWaitBudgetNs, gave_up);
                    if (__all_sync(0xffffffffu, ok)) st.issue(k, slot, q[j], &full[slot], lane);
                    q[j] = k + kDescAhead < n_chunks ? st.desc(k + kDescAhead, lane)
                                                     : make_int4(0, 0, 0, 0);
                }
            }
        }
        kbase += uint32_t(n_chunks);
        return;
    }

    // ---------------- compute warps
    const int wd = warp % a.warps_dm, wt = warp / a.warps_dm;
    Acc acc[DPT][SPT];
#pragma unroll
    for (int i = 0; i < DPT; ++i)
#pragma unroll
        for (int j = 0; j < SPT; ++j) acc[i][j] = Acc(0);
    const int lb = wt * 32 * SPT + lane;

    // Slot and phase of a chunk are counted on (a division by the run-time
    // number of slots takes about 150 clocks, which every warp waits for), and
    // a lost wait travels with the barrier instead of being read from shared
    // memory after it. Survey scale: FP32 (kind 6) 2.328 -> 2.280 ms, 8-bit
    // 2.250 -> 2.232 ms. (16-bit input with two slots keeps the flag: with the
    // barrier's answer the 4 x 8 kernels of kinds 2 and 4 take 1.05 to 1.12 times
    // as long on each of 26 setups, the 4 x 4 and 8 x 4 ones the same.)
    uint32_t slot = kbase % S, parity = (kbase / S) & 1u;
    for (int k = 0; k < n_chunks; ++k) {
        // A failed wait in any warp is known to all of them after the barrier;
        // the chunk's trials are then skipped.
        const bool ok = __all_sync(
            0xffffffffu, mbar_wait_bounded(&full[slot], parity, a.err, kWaitBudgetNs, gave_up));
        const unsigned char *sb = stage0 + slot * st.stage_bytes;
        const T *raw = reinterpret_cast<const T *>(sb);
        const int4 *bd = reinterpret_cast<const int4 *>(sb + a.stage_data_bytes + poffs_bytes);
        const Wt *sw = reinterpret_cast<const Wt *>(sb + a.stage_data_bytes + st.tab_bytes);
        unsigned char *pb =
            pslot0 + (ONE_SLOT ? 0u : ((kbase + uint32_t(k)) & 1u)) * pslot_bytes;
        Acc *P = reinterpret_cast<Acc *>(pb);
        uint16_t *poffs = reinterpret_cast<uint16_t *>(pb + a.p_elems * int(sizeof(Acc)));
        const int ng = (min(a.cch, a.C - (kr.x + k) * a.cch) + kSbG - 1) / kSbG;

        if (ok) {
            sb_build_blocks<T>(P, raw, bd, sw, a.n_blocks, warp, nc, lane);
            // the chunk's trial offsets move next to its partial sums
            const uint32_t *src = reinterpret_cast<const uint32_t *>(sb + a.stage_data_bytes);
            uint32_t *dst = reinterpret_cast<uint32_t *>(poffs);
            for (int i = tid; i < int(poffs_bytes / 4); i += nc * 32) dst[i] = src[i];
        }
        bool lost;
        if constexpr (sizeof(T) == 2 && !ONE_SLOT) {
            compute_barrier(nc * 32);
            lost = *gave_up;
        } else {
            lost = compute_barrier_or(nc * 32, !ok);
        }
        // nothing reads this staging slot any more (a lost chunk's is not
        // released: the producer's next wait fails too)
        if (tid == 0 && !lost) mbar_arrive(&empty[slot]);
        if (++slot == S) {
            slot = 0;
            parity ^= 1u;
        }
        if constexpr (ONE_SLOT) {
            if (!lost)
                sb_trials<sb_passes<T, true>(), Acc, DPT, SPT>(acc, P + lb, poffs + wd * DPT, a.Dt,
                                                               ng);
            compute_barrier(nc * 32);
        } else {
            if (lost) continue;
            sb_trials<sb_passes<T, false>(), Acc, DPT, SPT>(acc, P + lb, poffs + wd * DPT, a.Dt,
                                                            ng);
        }
    }
    kbase += uint32_t(n_chunks);
    if (!*gave_up) store_lane_strided<Acc, DPT, SPT>(a, acc, dtile, b, t0, wd, lb);
}

// kind 3: warp-specialised sub-band. Warps [0, NC) are trial warps (as in
// kind 2), warps [NC, NC + 4) builders. Barriers: full/empty of the staging
// slots at bars[0..3] / bars[8..11], full/empty of the partial-sum slots at
// bars[4..6] / bars[12..14]. A partial-sum slot holds the chunk's partial
// series followed by its per-group trial offsets (copied out of the staging
// slot so that slot can be refilled as soon as the builders are done).
template <typename T, int DPT, int SPT, bool LIVE>
__device__ __forceinline__ void fwd_tile_ws(const FwdArgs &a, int dtile, int ttile, int b,
                                            uint64_t *bars, unsigned char *stage0,
                                            uint32_t &kbase) {
    using Acc = typename Elem<T>::Acc;
    using Wt = typename Elem<T>::W;
    uint64_t *full_r = bars, *empty_r = bars + 8, *full_p = bars + 4, *empty_p = bars + 12;
    volatile int *gave_up = reinterpret_cast<volatile int *>(&bars[7]);
    const uint32_t S = uint32_t(a.stages), Q = uint32_t(kWsPSlots);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nc = int(blockDim.x >> 5) - kWsBuilders;  // trial warps
    const long long t0 = (long long)ttile * a.Ts;
    const int2 kr = chunk_range<LIVE>(a, dtile, ttile);
    const int n_chunks = kr.y - kr.x;
    const Stager<T> st = make_stager<T>(a, dtile, b, t0, stage0, true, kr.x);
    const uint32_t poffs_bytes = st.tab1_bytes;
    const int pslot_bytes = a.p_elems * int(sizeof(Acc)) + int(poffs_bytes);
    unsigned char *pslot0 = stage0 + S * st.stage_bytes;

    if (warp >= nc) {
        // ---------------- builder warps
        const int bw = warp - nc;
        auto issue = [&](int k, int4 dsc) {  // builder warp 0
            const uint32_t kg = kbase + uint32_t(k);
            const int slot = int(kg % S);
            bool ok = true;
            if (kg >= S)
                ok = mbar_wait_bounded(&empty_r[slot], ((kg / S) - 1u) & 1u, a.err, kWaitBudgetNs,
                                       gave_up);
            if (__all_sync(0xffffffffu, ok && !*gave_up))
                st.issue(k, slot, dsc, &full_r[slot], lane);
        };
        if (bw == 0) {
            const int pro = min(int(S), n_chunks);
            for (int k = 0; k < pro; ++k) issue(k, st.desc(k, lane));
        }
        for (int k = 0; k < n_chunks; ++k) {
            const uint32_t kg = kbase + uint32_t(k);
            const int rs = int(kg % S), ps = int(kg % Q);
            const int kn = k - 1 + int(S);
            int4 pre = make_int4(0, 0, 0, 0);
            if (bw == 0 && k >= 1 && kn < n_chunks) pre = st.desc(kn, lane);
            bool ok = mbar_wait_bounded(&full_r[rs], (kg / S) & 1u, a.err, kWaitBudgetNs, gave_up);
            if (ok && kg >= Q)
                ok = mbar_wait_bounded(&empty_p[ps], ((kg / Q) - 1u) & 1u, a.err, kWaitBudgetNs,
                                       gave_up);
            if (!__all_sync(0xffffffffu, ok)) break;  // a lost hand-off ends the tile
            const unsigned char *sb = stage0 + rs * st.stage_bytes;
            const T *raw = reinterpret_cast<const T *>(sb);
            const int4 *bd =
                reinterpret_cast<const int4 *>(sb + a.stage_data_bytes + poffs_bytes);
            const Wt *sw = reinterpret_cast<const Wt *>(sb + a.stage_data_bytes + st.tab_bytes);
            unsigned char *pb = pslot0 + ps * pslot_bytes;
            sb_build_blocks<T>(reinterpret_cast<Acc *>(pb), raw, bd, sw, a.n_blocks, bw,
                               kWsBuilders, lane);
            if (bw == 0) {  // the trial offsets travel with the partial sums
                const uint32_t *src = reinterpret_cast<const uint32_t *>(sb + a.stage_data_bytes);
                uint32_t *dsto = reinterpret_cast<uint32_t *>(pb + a.p_elems * int(sizeof(Acc)));
                for (int i = lane; i < int(poffs_bytes / 4); i += 32) dsto[i] = src[i];
            }
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&full_p[ps]);
                mbar_arrive(&empty_r[rs]);
            }
            // refill the staging slot of the previous chunk (one chunk of slack)
            if (bw == 0 && k >= 1 && kn < n_chunks) issue(kn, pre);
        }
        kbase += uint32_t(n_chunks);
        return;
    }

    // ---------------- trial warps
    const int wd = warp % a.warps_dm, wt = warp / a.warps_dm;
    Acc acc[DPT][SPT];
#pragma unroll
    for (int i = 0; i < DPT; ++i)
#pragma unroll
        for (int j = 0; j < SPT; ++j) acc[i][j] = Acc(0);
    const int lb = wt * 32 * SPT + lane;
    for (int k = 0; k < n_chunks; ++k) {
        const uint32_t kg = kbase + uint32_t(k);
        const int ps = int(kg % Q);
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(&full_p[ps], (kg / Q) & 1u, a.err,
                                                       kWaitBudgetNs, gave_up)))
            break;
        const unsigned char *pb = pslot0 + ps * pslot_bytes;
        const uint16_t *poffs =
            reinterpret_cast<const uint16_t *>(pb + a.p_elems * int(sizeof(Acc))) + wd * DPT;
        const int ng = (min(a.cch, a.C - (kr.x + k) * a.cch) + kSbG - 1) / kSbG;
        sb_trials<sb_passes<T, false>(), Acc, DPT, SPT>(
            acc, reinterpret_cast<const Acc *>(pb) + lb, poffs, a.Dt, ng);
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty_p[ps]);
    }
    kbase += uint32_t(n_chunks);
    if (!*gave_up) store_lane_strided<Acc, DPT, SPT>(a, acc, dtile, b, t0, wd, lb);
}

// Dispatches a tile to the kind's body.
template <int KIND, typename T, int DPT, int SPT, bool LIVE = false>
__device__ __forceinline__ void fwd_tile_any(const FwdArgs &a, int dtile, int ttile, int b,
                                             uint64_t *bars, unsigned char *stage0,
                                             uint32_t &kbase) {
    if constexpr (KIND == 2 || KIND == 4)
        fwd_tile_sb<T, DPT, SPT, LIVE>(a, dtile, ttile, b, bars, stage0, kbase);
    else if constexpr (KIND == 6)
        fwd_tile_sb<T, DPT, SPT, LIVE, true>(a, dtile, ttile, b, bars, stage0, kbase);
    else if constexpr (KIND == 3)
        fwd_tile_ws<T, DPT, SPT, LIVE>(a, dtile, ttile, b, bars, stage0, kbase);
    else
        fwd_tile<KIND, T, DPT, SPT, LIVE>(a, dtile, ttile, b, bars, stage0, kbase);
}

}  // namespace dd
