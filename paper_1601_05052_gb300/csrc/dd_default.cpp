// dd_default.cpp -- the variant a plan (or batch) starts with: a time model
// of the candidate variants, from the plan's sizes, type and delay steps.
//
// One tile of a variant takes, with r CTAs resident on its SM,
//     max(r * warps * C * (a (W + G) + b + 10 k / cch), C (10 l + 100 m / cch)) + 1000 o
// clocks: its share of the SM's shared-memory pipe and issue slots, or the
// latency of one channel after the other when too few warps are resident,
// plus a tile's start and end. W is the shared-memory words a warp reads per
// channel, G the staged words, cch the channels per stage. The tiles run in
// rounds of the CTAs that are resident at once; staged bytes (L2) and
// compulsory bytes (HBM) bound the sum from below. The constants of each
// kernel family were fitted on a GB300 to timings of 272 setups drawn from
// five bands (64-channel L-band, Apertif, 300 MHz L-band, 120-180 MHz, LOFAR;
// 1 to 384 beams, 16 to 1024 channels, 4 to 2048 trials, all four input types),
// each with every candidate that fits it. Residual 6 % (quads) and 10 %
// (lane-strided, windows) to 15 % (sub-bands, whose patterns are not counted). Over
// those setups the model's choice took 1.03 times the best candidate's time in
// the geometric mean (1.31 at worst); the fixed preference list it replaced,
// 1.39 times (5.2 at worst, LOFAR).
#include <algorithm>
#include <cmath>

#include "dd_internal.h"

namespace dd {

namespace {

struct Candidate {
    dd_variant v;
    bool time_major;
};

// The variants worth starting with: of 45 timed, these were within 0.3 % of
// the best in the geometric mean.
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
    {{0, 4, 4, 4, 1, 16, 4}, false},
    {{0, 4, 2, 4, 2, 32, 2}, false},
    {{0, 2, 4, 4, 1, 32, 3}, false},
    {{0, 2, 4, 2, 4, 16, 3}, false},
    {{5, 4, 8, 4, 1, 16, 3}, false},
};

// Fitted constants {a, b, k, l, o, s, m}; s: sub-band build words.
struct Fit {
    double a, b, k, l, o, s, m;
};
constexpr Fit kLane{0.95, 3.82, 1.55, 4.97, 6.49, 0, 13.84};
constexpr Fit kQuad{1.3, 15.7, 2.84, 41.3, 6.12, 0, 7.05};
constexpr Fit kWindow{1.21, 8.26, 0, 32.3, 9.1, 0, 8.41};
constexpr Fit kReuse{0.58, 11.6, 11.2, 22.9, 3.93, 0, 34.8};
constexpr Fit kSub2{1.03, 4.96, 0.73, 34.8, 1.84, 10.8, 3.44};
constexpr Fit kSub4{0.28, 10.9, 2.17, 19.5, 2.02, 27.6, 15.7};
constexpr Fit kSub6{0.06, 9.76, 8.19, 24.1, 2.69, 148, 3.01};

// Registers per thread of the kernels with 2x4 .. 8x8 outputs per thread.
int registers(const dd_variant &v) {
    if (v.kind == 2) return v.dm_per_thread * v.samples_per_thread <= 16 ? 72 : 80;
    if (v.kind == 4 || v.kind == 6) return 96;
    if (is_window(v.kind, v.samples_per_thread) || is_quad(v.kind, v.samples_per_thread))
        return 128;
    if (v.kind == 5) return 90;
    const int n = v.dm_per_thread * v.samples_per_thread;
    return n <= 8 ? 40 : (n <= 16 ? 56 : (n <= 32 ? 76 : 126));
}

}  // namespace

DelaySteps delay_steps(const dd_plan_s *p) {
    DelaySteps s;
    std::vector<int32_t> lo(p->shifts.begin(), p->shifts.begin() + p->C), hi = lo;
    for (int d = 1; d < p->D; ++d) {
        const int32_t *row = &p->shifts[size_t(d) * p->C];
        for (int c = 0; c < p->C; ++c) {
            lo[size_t(c)] = std::min(lo[size_t(c)], row[c]);
            hi[size_t(c)] = std::max(hi[size_t(c)], row[c]);
        }
    }
    for (int c = 0; c < p->C; ++c) {
        const double x = double(hi[size_t(c)] - lo[size_t(c)]) / std::max(1, p->D - 1);
        s.mean += x / p->C;
        s.max = std::max(s.max, x);
    }
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
    const double widest = std::min(Ts + (De - 1) * st.max, De * Ts);
    // resident CTAs per SM
    const double slot = std::min(cch, C) * widest * elt + cch * (2 * Dt + 20);
    double smem = 1152 + v.stages * slot;
    if (sb) {  // partial series, at five patterns per group
        const double P = cch / 4 * 5 * (Ts + De * st.max) * 4 * 1.15;
        smem += v.kind == 6 ? P : 2 * P;
    }
    const int threads = 32 * (nw + extra_warps(v.kind));
    const double r_max = std::max(
        1.0, std::floor(std::min({233000.0 / smem,
                                  65536.0 / ((registers(v) + 7) / 8 * 8 * threads),
                                  2048.0 / threads, 32.0})));
    // Words per warp and channel. Shared operands: steps taken as spread
    // evenly over [0, 2 mean], `same` of adjacent trials share a delay.
    const double x = 2 * st.mean, same = x <= 1 ? 1 - x / 2 : 1 / (2 * x);
    double W = v.dm_per_thread * v.samples_per_thread;
    if (quad)
        W = v.dm_per_thread * (v.samples_per_thread / 4 + 1);
    else if (win && st.max <= kWinBands + 0.5)
        W = 2 * (v.samples_per_thread / 2 + 3 * st.mean);
    else if (v.kind == 5 && !win)
        W *= 1 - same * (v.dm_per_thread - 1) / v.dm_per_thread;
    else if (sb)
        W = W / 4 * (1 - same / 2) + f.s * (Ts + De * st.mean) / (32 * nw);
    const double per = C * (f.a * (W + len * elt / 128 / nw) + f.b + 10 * f.k / cch);
    const double lat = C * (10 * f.l + 100 * f.m / cch);
    auto tile = [&](double r) { return std::max(r * nw * per, lat) + 1000 * f.o; };
    const double slots = r_max * p->sm_count, full = std::floor(tiles / slots);
    const double rest = tiles - full * slots;
    double clk = full * tile(r_max);
    if (rest > 0) clk += tile(std::ceil(rest / p->sm_count));
    double us = clk / 2070.0;
    us = std::max(us, tiles * C * len * elt / 7.5e6);
    us = std::max(us, (p->B * C * double(p->stride) * elt + 4.0 * p->B * p->D * double(p->S)) / 5.5e6);
    return us;
}

// Long float chains whose delays move by 12 to 32 samples per trial (adjoints
// at survey bands; low bands start at 39): sub-bands round less there too, but
// the model does not order them well enough (gradients of 3 x 268 channels x
// 1886 trials x 10382 samples: its choice 5.8 ms, the preference list's 4.5;
// windows 3.6 at twice the error).
bool by_preference(const dd_plan_s *p) {
    if (p->dtype == DD_U8 || p->C <= 128 || p->D < 24) return false;
    const double steps = delay_steps(p).max;
    return steps > 12 && steps <= 32;
}

std::vector<RankedVariant> ranked_variants(const dd_plan_s *p) {
    const DelaySteps st = delay_steps(p);
    std::vector<RankedVariant> r;
    for (const Candidate &c : kCandidates) {
        if (is_quad(c.v.kind, c.v.samples_per_thread) && p->dtype != DD_U8) continue;
        // Windows want 32-bit samples (narrower ones at odd strides collide in
        // the banks: 64 channels x 64 trials, 8-bit, 22.6 against 9.4 us).
        if (is_window(c.v.kind, c.v.samples_per_thread) && p->dtype != DD_F32) continue;
        // One partial-sum slot only where two do not fit (survey scale, 8-bit:
        // kind 4 2.26 ms, kind 6 2.38; FP32 fits 32 channels in kind 6 alone).
        if (c.v.kind == 6 && c.v.warps_dm == 16 && p->dtype != DD_F32) continue;
        // Where no channel moves by more than 0.8 samples per trial, a
        // thread's trials mostly share a sub-band's series and offset, which
        // the model does not see (500 channels x 1000 trials x 10000 samples,
        // FP32: sub-bands 0.51 ms, windows 0.59, lane-strided 1.2). And a
        // float chain over more than 128 channels rounds more than the
        // sub-bands' groups of four, so smooth delays keep those: 473 channels
        // x 788 trials x 4406 samples, gradients, 5.2e-7 of the largest output
        // against 2.8e-7, and 0.69 ms against 0.55.
        if (p->D >= 24 && !is_subband(c.v.kind) &&
            (st.max <= 0.8 || (p->dtype != DD_U8 && p->C > 128 && st.max <= 12)))
            continue;
        // Near ties go to the wide sub-bands, whose grouped sums are also the
        // more accurate (500 channels x 1000 trials, FP32: 0.54 ms where the
        // model has 0.61, windows 0.615 where it has 0.56).
        const double tie = is_subband(c.v.kind) && c.v.warps_dm == 16 ? 1.0 : 1.04;
        r.push_back(RankedVariant{c.v, c.time_major, tie * model_us(p, st, c.v)});
    }
    std::stable_sort(r.begin(), r.end(),
                     [](const RankedVariant &a, const RankedVariant &b) { return a.us < b.us; });
    return r;
}

}  // namespace dd
