// cls_case.h -- host-side case set-up shared by every entry point that takes
// case parameters (cls_create / cls_batch_create and cls_run_noalloc): the
// parameter check and the derived quantities the kernels read (CaseParams).
#pragma once

#include <algorithm>
#include <cmath>
#include <cstring>

#include "../../include/cls.h"
#include "cls_fixed.h"
#include "cls_internal.h"

namespace cls {

constexpr int kMaxBins = 4096;

// (sigma0, sigma1, lambda0, lambda1, c0, c1, L, d, nbins): Sigma_i >= 0 and
// finite, Lambda_i > 0 and finite, 0 <= c_i <= 1 (c_i = Sigma_s,i / Sigma_i,
// paper Sec. 2), L > 0, a known geometry code, 1 <= nbins <= kMaxBins.
inline int validate_case(const double *p) {
    const double s0 = p[0], s1 = p[1], l0 = p[2], l1 = p[3], c0 = p[4], c1 = p[5], L = p[6];
    const double d = p[7], nb = p[8];
    auto finite = [](double v) { return std::isfinite(v); };
    if (!(finite(s0) && s0 >= 0 && finite(s1) && s1 >= 0)) return CLS_E_INVAL;
    if (!(finite(l0) && l0 > 0 && finite(l1) && l1 > 0)) return CLS_E_INVAL;
    if (!(c0 >= 0 && c0 <= 1 && c1 >= 0 && c1 <= 1)) return CLS_E_INVAL;
    if (!(finite(L) && L > 0)) return CLS_E_INVAL;
    if (!(d == 1.0 || d == 2.0 || d == 3.0 || d == 11.0 || d == 13.0)) return CLS_E_INVAL;
    if (!(nb >= 1 && nb <= kMaxBins && nb == std::floor(nb))) return CLS_E_INVAL;
    return CLS_OK;
}

// Rough events-per-history estimate, used only to order cases largest first:
// flights per unit path length times an estimate of the path length, which
// grows with the number of scatterings ~ 1/(1 - c) and with the size L.
inline double cost_estimate(const CaseParams &c) {
    const double p0 = c.p0, p1 = 1.0 - c.p0;
    const double sig = p0 * c.sigma[0] + p1 * c.sigma[1];
    const double rate = sig + p0 / c.lambda[0] + p1 / c.lambda[1];
    const double cbar = sig > 0 ? (p0 * c.c[0] * c.sigma[0] + p1 * c.c[1] * c.sigma[1]) / sig : 0.0;
    const double tau = sig * c.L;
    const double ncol = std::min(1.0 / std::max(1.0 - cbar, 1e-6), 1.0 + tau * tau);
    const double path = std::min(c.L, 1.0 / std::max(sig, 1e-12)) * (1.0 + ncol * std::min(1.0, tau));
    return 1.0 + rate * path;
}

// Runs of up to this many histories for each warp of the narrow walk go to it
// alone (LaunchArgs::narrow).  Measured, us in the tracker / the narrow walk.
// FP64, 8 a warp (14,000): 3D case 3a 848 / 670, box L = 10 1239 / 1224, extruded
// 448 / 582 (at 4000: 410 / 324), case 1b, of 4 events, 84 / 174 (at 1000: 68 /
// 50); slab 146 / 108, rod 204 / 168.  FP32, 22 a warp (40,000): 3D case 3a 310 /
// 264, extruded 218 / 212, rod 168 / 151, case 1b 83 / 101 (at 20,000: 69 / 61).
// The crossing follows the longest history's length over the mean's, which
// no estimate here knows, so the line is where most cases cross.
inline double narrow_histories(bool fp32, int geom) {
    return fp32 ? 24.0 : geom == 1 || geom == 11 || geom == 13 ? 14.0 : 8.0;
}

// Estimated events per history: about cost^(3/4) (the cost estimate is within a
// factor of two for short histories and several times too high for scattering media).
inline double estimated_events(double cost) { return std::pow(std::max(cost, 1.0), 0.75); }

// Warps of a launch hand their last histories over to the narrow walk, which
// walks a history two to four times as fast, but only one per warp: the last
// kHandOver where histories average kHandOverEvents or more by the estimate,
// else the last two, except in the FP64 walks with two or three axes, whose
// draws cost the narrow walk most.  Measured, none / 2 / 4 handed over: diffusive
// box (153 events) 1e6 in FP32 20.4 / 14.7 / 13.3 ms, 1e5 10.1 / 8.3 / 6.3 ms; box
// L = 10 (47 events) in FP32 1e6 1.74 / 1.57 / 1.56 ms, 1e5 781 / 678 / 665 us, in
// FP64 1e5 2.15 / 2.25 / 2.45 ms; slab 1e5 in FP64 275 / 233 / 234 us.
constexpr double kHandOverEvents = 128.0;

inline int hand_over_for(double events, bool fp32, int geom) {
    if (events >= kHandOverEvents) return kHandOver;
    return fp32 || geom == 1 || geom == 11 || geom == 13 ? 2 : 0;
}

// How a history-tracker launch of n histories in each of `nruns` run entries is
// claimed (LaunchArgs): pieces of whole statistics batches, at most max_pieces
// of them; as many warps start on a piece as it takes to employ all; and the
// least a warp claims is 32 histories, a warp's lanes, or where that would not
// go round, a power of two below.  may_narrow: whether a run small enough goes to
// the narrow walk, whose launch shape is `narrow`.
inline void plan_pieces(LaunchArgs &a, uint64_t n, uint64_t batch_len, double mean_cost, int geom, int sm_count, bool fp32,
                        uint64_t max_pieces, bool may_narrow, const NarrowShape &narrow) {
    const double total = (double)n * a.nruns;
    const double narrow_warps = (double)sm_count * narrow.blocks * narrow.warps;
    a.narrow = may_narrow && total <= narrow_histories(fp32, geom) * narrow_warps;
    const double warps = a.narrow ? std::min(total, narrow_warps) : sm_count * (fp32 ? 28.0 : 20.0);
    const uint64_t used = (n + batch_len - 1) / batch_len;  // batches
    const uint64_t per_run = std::max<uint64_t>(1, std::min<uint64_t>(std::min<uint64_t>(used, 64), max_pieces / a.nruns));
    const uint64_t batches = (used + per_run - 1) / per_run;
    a.piece_len = batches * batch_len;
    a.pieces_per_run = (uint32_t)((used + batches - 1) / batches);
    a.team = (uint32_t)std::ceil(warps / ((double)a.pieces_per_run * a.nruns));
    a.hand_over = hand_over_for(estimated_events(mean_cost), fp32, geom);
    a.chunk = a.narrow ? 1 : 32;
    while (a.chunk > 1 && (double)a.chunk > total / warps) a.chunk >>= 1;
}

// Blocks of the narrow walk: as many as the run has histories for its warps.
inline int narrow_grid(const LaunchArgs &a, const NarrowShape &narrow, uint64_t n, int sm_count) {
    const int full = sm_count * narrow.blocks;
    return a.narrow ? (int)std::min((double)full, std::ceil((double)n * a.nruns / narrow.warps)) : full;
}

// Claim limit and refill threshold of a run entry (RunCase), from the
// estimated cost of its histories and of all histories of the launch.  A claim
// takes at most 1/8 of a warp's share of the launch by that estimate (a sweep's
// longest cases have a hundred times its shortest's events), and at most 32
// times the chunk option.
inline void plan_claims(RunCase &r, const CaseParams &c, double launch_cost, int sm_count, uint32_t chunk,
                        uint32_t option) {
    const double share = launch_cost / (8.0 * 24.0 * sm_count * std::max(c.cost, 1.0) * chunk);  // 24: about the warps of an SM
    const double most = std::min(share, 32.0 * option / chunk);
    int bits = 0;
    while (bits < 40 && std::ldexp(1.0, bits + 1) <= most) ++bits;
    r.claim_bits = (uint16_t)bits;
    // lanes die 32 / events per step, and waiting idles half of refill_min of them.  Measured, 2 / 4 / 8 / 12 / 16
    // lanes: box L = 10 (47 events, FP32, 1e8) 101 / 97 / 100 / 107 / 118 ms; sweep (5 events, 256 x 1e6) 50.8 /
    // 49.4 / 47.3 / 46.5 / 47.1 ms; by this rule 46.2 ms, with 5.2 and at most 12 lanes 46.8
    const double wait = std::floor(6.5 * std::sqrt(32.0 / estimated_events(c.cost)) + 0.5);
    r.refill_min = (uint16_t)std::min(16.0, std::max(2.0, wait));
}

// The kernels' view of one validated case: p_0 = Lambda_0 / (Lambda_0 +
// Lambda_1) (paper Sec. 2), the mesh width, FP32 copies, reciprocals and the
// integer thresholds of the draw comparisons.  Case k of a launch draws with
// Philox counter word 3 = case_id.
inline CaseParams make_case(const double *p, uint32_t case_id) {
    CaseParams c;
    std::memset(&c, 0, sizeof(c));
    for (int i = 0; i < 2; ++i) {
        c.sigma[i] = p[i];
        c.inv_sigma[i] = p[i] > 0 ? 1.0 / p[i] : 0.0;
        c.lambda[i] = p[2 + i];
        c.c[i] = p[4 + i];
        c.sigma_f[i] = (float)p[i];
        c.inv_sigma_f[i] = p[i] > 0 ? (float)(1.0 / p[i]) : 0.0f;
        c.lambda_f[i] = (float)p[2 + i];
        c.c_f[i] = (float)p[4 + i];
    }
    c.L = p[6];
    c.d = (int32_t)p[7];
    c.nbins = (int32_t)p[8];
    c.p0 = c.lambda[0] / (c.lambda[0] + c.lambda[1]);
    c.dx = c.L / c.nbins;
    c.inv_dx = c.nbins / c.L;
    c.L_f = (float)c.L;
    c.p0_f = (float)c.p0;
    c.dx_f = (float)c.dx;
    c.inv_dx_f = (float)c.inv_dx;
    c.case_id = case_id;
    for (int i = 0; i < 2; ++i) {
        c.thr_c53[i] = unit_threshold(c.c[i], 53);
        c.thr_c24[i] = (uint32_t)unit_threshold((double)c.c_f[i], 24);
    }
    c.thr_p053 = unit_threshold(c.p0, 53);
    c.thr_p024 = (uint32_t)unit_threshold((double)c.p0_f, 24);
    // products of these in FP32 neither overflow nor lose bits
    auto moderate = [](double v) { return v >= 0x1p-60 && v <= 0x1p60; };
    c.filter = moderate(c.L) && moderate(c.lambda[0]) && moderate(c.lambda[1]) &&
               (p[0] == 0 || moderate(1.0 / p[0])) && (p[1] == 0 || moderate(1.0 / p[1]));
    c.fix_bits = fixed_bits(c.dx, c.sigma, c.lambda);
    c.fix_unit = std::ldexp(c.dx, -c.fix_bits);
    c.cost = cost_estimate(c);
    return c;
}

}  // namespace cls
