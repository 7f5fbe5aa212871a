// dd_default.cpp -- the variant a plan (or batch) starts with: a time model
// of the candidate variants, from the plan's sizes, type and delay steps.
//
// One tile of a variant takes, with r CTAs resident on its SM,
//     max(r * warps * C * (a (W + G) + s P + b + 10 k / cch), C (10 l + 100 m / cch)) + 1000 o
// clocks: its share of the SM's shared-memory pipe and issue slots, or the
// latency of one channel after the other when too few warps are resident,
// plus a tile's start and end. W is the shared-memory words a warp reads per
// channel, G the staged words, P the sub-bands' partial-series words, cch the
// channels per stage. The tiles run in rounds of the CTAs that are resident at
// once; staged bytes (L2) and compulsory bytes (HBM) bound the sum from below.
// (Lane-strided with two small slots: latency s more, as no copy is in flight
// while a chunk is summed.)
// The constants of each kernel family were fitted on a GB300 to 75700 timings
// (44 variants, where they fit, on 3550 setups: 2036 drawn from five bands, 1 to
// 384 beams, 16 to 1024 channels, 4 to 2048 trials, all input types, some
// gradients' transposed tables; 403 at steps of up to 1.5 samples; 1111
// transposed tables at 120-180 and 138-144 MHz), then adjusted, on four fifths
// of the setups, to what the choice costs. Residuals 9 % (quads) to 21 % (kind
// 2). The choice, among the variants that keep a plan's channel groups
// (dd_plan.cpp), takes 1.018 times the best one's time in the geometric mean
// (1.018 on the last fifth too), 1.11 at the 95th percentile and 1.63 at worst.
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "dd_internal.h"

namespace dd {

namespace {

struct Candidate {
    dd_variant v;
    bool time_major;
};

// The variants worth starting with: the best of them takes 1.003 times the best
// of all 44 in the geometric mean.
const Candidate kCandidates[] = {
    // sub-bands: long Eq. 1 grids whose channel groups share delay patterns
    {{6, 4, 8, 16, 1, 32, 2}, false},
    {{4, 4, 8, 16, 1, 32, 2}, false},
    {{4, 4, 8, 16, 1, 16, 2}, false},
    {{6, 4, 8, 8, 2, 32, 2}, false},
    {{4, 4, 8, 8, 2, 16, 2}, false},
    {{4, 4, 8, 8, 1, 32, 2}, false},
    {{2, 4, 8, 8, 1, 16, 2}, false},
    {{2, 4, 4, 8, 1, 16, 2}, false},
    // register windows: delays that move by up to five samples per trial
    {{5, 4, 22, 8, 1, 8, 3}, false},
    {{5, 4, 22, 4, 1, 8, 3}, false},
    {{5, 4, 18, 8, 1, 8, 3}, false},
    {{5, 4, 18, 4, 1, 8, 3}, false},
    {{5, 4, 14, 8, 1, 8, 3}, false},
    {{5, 4, 14, 4, 1, 8, 3}, false},
    // byte quads: 8-bit input whose channel groups share few patterns
    {{0, 4, 20, 4, 2, 16, 3}, false},
    {{0, 4, 20, 8, 1, 16, 3}, false},
    {{0, 4, 20, 4, 1, 16, 3}, false},
    {{0, 4, 20, 2, 2, 16, 3}, false},
    {{0, 4, 20, 1, 4, 4, 3}, true},
    // lane-strided: few trials, little work, or delays far apart
    {{0, 8, 8, 1, 8, 4, 3}, false},
    {{0, 8, 8, 2, 4, 8, 3}, false},
    {{0, 8, 8, 2, 4, 4, 4}, false},
    {{0, 8, 8, 4, 2, 8, 3}, false},
    {{0, 8, 8, 1, 16, 2, 2}, true},
    {{0, 8, 8, 1, 8, 2, 3}, true},
    {{0, 4, 8, 1, 4, 4, 3}, false},
    {{0, 4, 8, 1, 8, 4, 3}, false},
    {{0, 4, 8, 4, 1, 8, 3}, false},
    {{0, 4, 8, 2, 4, 8, 3}, false},
    {{0, 4, 8, 2, 2, 8, 3}, false},
    {{0, 4, 4, 4, 1, 16, 4}, false},
    {{0, 4, 2, 4, 2, 32, 2}, false},
    {{0, 2, 4, 4, 1, 32, 3}, false},
    {{0, 2, 4, 2, 4, 16, 3}, false},
    {{5, 4, 8, 4, 1, 16, 3}, false},
};

// Fitted constants of a kernel family.
struct Fit {
    double a, b, k, l, o, s, m;
};
constexpr Fit kLane{1.02, 1.2, 1.31, 2.56, 6.08, 129.99, 14.66};
constexpr Fit kQuad{1.09, 19.26, 3.89, 25.72, 9.8, 0, 12.39};
constexpr Fit kWindow{1.08, 4.28, 8.06, 25.66, 8.62, 0, 23.07};
constexpr Fit kReuse{0.63, 14.59, 1.64, 24.87, 8.86, 0, 15.3};
constexpr Fit kSub2{0.96, 0.35, 11.67, 19.14, 8.39, 6.37, 20.33};
constexpr Fit kSub4{0.69, 6.59, 2.42, 20.76, 7.41, 6.88, 3.37};
constexpr Fit kSub6{1.33, 0.7, 0.47, 18.82, 7.66, 8.78, 5.21};

// Registers per thread of the candidates' one-shot kernels, as ptxas reports
// them (asking the runtime would load every candidate's code at plan time).
int registers(dd_dtype t, const dd_variant &v) {
    const int n = v.dm_per_thread * v.samples_per_thread;
    if (v.kind == 2) return n <= 16 ? 72 : 96;
    if (v.kind == 4 || v.kind == 6) return 96;
    if (is_window(v.kind, v.samples_per_thread) || is_quad(v.kind, v.samples_per_thread))
        return 128;
    if (v.kind == 5) return 88;
    if (n <= 8) return t == DD_F32 ? 118 : 96;
    if (n <= 16) return 96;
    return n <= 32 && t == DD_U8 ? 106 : 128;
}

}  // namespace

DelaySteps delay_steps(const dd_plan_s *p) {
    DelaySteps s;
    const int K = std::min(p->D - 1, 16);  // trials of a small tile
    std::vector<int32_t> lo(p->shifts.begin(), p->shifts.begin() + p->C), hi = lo;
    int32_t span = 0;
    for (int d = 1; d < p->D; ++d) {
        const int32_t *row = &p->shifts[size_t(d) * p->C];
        const int32_t *back = d >= K ? row - size_t(K) * p->C : row;
        for (int c = 0; c < p->C; ++c) {
            lo[size_t(c)] = std::min(lo[size_t(c)], row[c]);
            hi[size_t(c)] = std::max(hi[size_t(c)], row[c]);
            span = std::max(span, std::abs(row[c] - back[c]));
        }
    }
    for (int c = 0; c < p->C; ++c) {
        const double x = double(hi[size_t(c)] - lo[size_t(c)]) / std::max(1, p->D - 1);
        s.mean += x / p->C;
        s.max = std::max(s.max, x);
    }
    s.widest = double(span) / std::max(1, K);
    return s;
}

// Modelled time of one forward launch in microseconds.
double model_us(const dd_plan_s *p, const DelaySteps &st, const dd_variant &v) {
    const bool sb = is_subband(v.kind), win = is_window(v.kind, v.samples_per_thread);
    const bool quad = is_quad(v.kind, v.samples_per_thread);
    const Fit &f = quad          ? kQuad
                   : v.kind == 0 ? kLane
                   : win         ? kWindow
                   : v.kind == 5 ? kReuse
                   : v.kind == 2 ? kSub2
                   : v.kind == 4 ? kSub4
                                 : kSub6;
    const double elt = elt_bytes(p->dtype), C = p->C, cch = v.chans_per_stage;
    const int Dt = v.dm_per_thread * v.warps_dm, nw = v.warps_dm * v.warps_time;
    const double Ts = 32.0 * v.samples_per_thread * v.warps_time, De = std::min(Dt, p->D);
    const double tiles = std::ceil(double(p->D) / Dt) * std::ceil(double(p->S) / Ts) * p->B;
    // window of a channel for the tile's trials, in a mean and the widest channel
    const double len = std::min(Ts + (De - 1) * st.mean, De * Ts);
    const double widest = std::min(Ts + (De - 1) * st.widest, De * Ts);
    // resident CTAs per SM
    const double slot = std::min(cch, C) * widest * elt + cch * (2 * Dt + 20);
    double smem = 1152 + v.stages * slot;
    if (sb) {  // partial series, at five patterns per group
        const double series = cch / 4 * 5 * (Ts + De * st.widest) * 4 * 1.15;
        smem += v.kind == 6 ? series : 2 * series;
    }
    const int threads = 32 * (nw + extra_warps(v.kind));
    const double r_max = std::max(
        1.0, std::floor(std::min({double(p->smem_optin + 1024) / smem,
                                  65536.0 / ((registers(p->dtype, v) + 7) / 8 * 8 * threads),
                                  2048.0 / threads, 32.0})));
    // Words per warp and channel. Shared operands: steps taken as spread
    // evenly over [0, 2 mean], `same` of adjacent trials share a delay.
    const double x = 2 * st.mean, same = x <= 1 ? 1 - x / 2 : 1 / (2 * x);
    double W = v.dm_per_thread * v.samples_per_thread, P = 0;
    if (quad)
        W = v.dm_per_thread * (v.samples_per_thread / 4 + 1);
    else if (win && st.max <= kWinBands + 0.5)
        W = 2 * (v.samples_per_thread / 2 + 3 * st.mean);
    else if (v.kind == 5 && !win)
        W *= 1 - same * (v.dm_per_thread - 1) / v.dm_per_thread;
    else if (sb)
        W = W / 4 * (1 - same / 2), P = (Ts + De * st.mean) / (32 * nw);
    const double per = C * (f.a * (W + len * elt / 128 / nw) + f.s * P + f.b + 10 * f.k / cch);
    // two small slots leave no copy in flight while a chunk is summed
    const bool bare = v.kind == 0 && v.stages == 2 && v.dm_per_thread * v.samples_per_thread < 64;
    const double lat = C * (10 * f.l + 100 * f.m / cch + (bare ? f.s : 0));
    auto tile = [&](double r) { return std::max(r * nw * per, lat) + 1000 * f.o; };
    const double slots = r_max * p->sm_count, full = std::floor(tiles / slots);
    const double rest = tiles - full * slots;
    double clk = full * tile(r_max);
    if (rest > 0) clk += tile(std::ceil(rest / p->sm_count));
    double us = clk / 2070.0;
    us = std::max(us, tiles * C * len * elt / 7.5e6);
    us = std::max(us, (p->B * C * double(p->stride) * elt + 4.0 * p->B * p->D * double(p->S)) / 5.5e6);
    // Narrow input: one partial-sum slot comes after two of the same size, for
    // where those do not fit (survey scale, 8-bit: kind 4 2.26 ms, kind 6 2.38;
    // 439 channels x 287 trials x 19105 samples, FP16: kind 6 203 us, kind 4 with
    // 16 channels per chunk 225).
    if (v.kind == 6 && v.warps_dm == 16 && p->dtype != DD_F32)
        us = std::max(us, 1.0001 * model_us(p, st, {4, 4, 8, 16, 1, 32, 2}));
    return us;
}

// How much longer the persistent form of a variant's kernel runs than its
// one-shot form's model says (other registers, spills; one launch for all
// plans): the geometric means over 587 batches of two setups, every candidate
// that fits both. With them the choice takes 1.03 times the best candidate's
// time, without 1.10.
double batch_factor(dd_dtype t, const dd_variant &v) {
    const int n = v.dm_per_thread * v.samples_per_thread, i = t == DD_F32 ? 0 : (t == DD_U8 ? 2 : 1);
    using Row = const double[3];  // FP32, 16-bit, 8-bit
    static Row sub{1.05, 1.3, 1.37}, reuse{1.04, 1.22, 0.96}, lane8{1, 1.06, 1},
        lane16{1.12, 1.22, 1.02}, lane32{0.9, 1.05, 0.97}, lane64{1.1, 1.36, 1.16};
    if (is_subband(v.kind)) return sub[i];
    if (is_quad(v.kind, v.samples_per_thread)) return 1.17;
    if (is_window(v.kind, v.samples_per_thread))  // FP32 only
        return v.samples_per_thread == 14 ? 1.14 : (v.samples_per_thread == 18 ? 1.5 : 1.8);
    if (v.kind == 5) return reuse[i];
    return n <= 8 ? lane8[i] : (n <= 16 ? lane16[i] : (n <= 32 ? lane32[i] : lane64[i]));
}

std::vector<RankedVariant> ranked_variants(const dd_plan_s *p) {
    const DelaySteps st = delay_steps(p);
    std::vector<RankedVariant> r;
    for (const Candidate &c : kCandidates) {
        if (is_quad(c.v.kind, c.v.samples_per_thread) && p->dtype != DD_U8) continue;
        // Windows want 32-bit samples (narrower ones at odd strides collide in
        // the banks: 64 channels x 64 trials, 8-bit, 22.6 against 9.4 us).
        if (is_window(c.v.kind, c.v.samples_per_thread) && p->dtype != DD_F32) continue;
        r.push_back(RankedVariant{c.v, c.time_major, model_us(p, st, c.v)});
    }
    // 8-bit sums at nearly constant delays: sub-bands first, whose few series
    // per group the model does not count (204 setups of 32 to 1024 channels and
    // up to 1.5 samples per trial: choice 1.067 times the best, 1.05 with lines
    // from 0.2 to 0.5, 1.061 at 0.8; floats do better without: 1.027 to 1.036).
    const bool smooth = p->dtype == DD_U8 && p->D >= 24 && st.max <= 0.3;
    std::stable_sort(r.begin(), r.end(), [&](const RankedVariant &a, const RankedVariant &b) {
        if (smooth && is_subband(a.v.kind) != is_subband(b.v.kind)) return is_subband(a.v.kind);
        return a.us < b.us;
    });
    return r;
}

}  // namespace dd
