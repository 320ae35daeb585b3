// Which plan of the grouped INT4 second kernels (w4a4_gemm.cu, w4a4_narrow.cu) a call takes.  Plain C++, so that the rule can be checked without a device.
#pragma once
#include <initializer_list>

namespace dirotq {

// A plan is named by the value of dirotq_set_gemm_tile that forces it: output columns per tile, + 2 with 256 token rows per tile (130 in one CTA, 258 in a
// pair of CTAs); 66: 64 columns, the K-groups cut over a cluster where that applies.
inline bool w4a4_plan_exists(int plan) {
    for (const int p : {32, 64, 66, 128, 130, 192, 256, 258})
        if (p == plan) return true;
    return false;
}

// What dirotq_set_gemm_tile(knob) means for these kernels: a plan of theirs, 0 where the kernel chooses for itself (512 names a plan of the
// NVFP4 and W4A8 kernels), -1 for a value that names nothing.
inline int w4a4_forced_plan(int knob) { return knob == 0 || knob == 512 ? 0 : w4a4_plan_exists(knob) ? knob : -1; }

// The plan with the shortest schedule: turns of the SMs (or of the pairs of SMs) x what one tile of the plan costs.  Costs relative to a pair's tile,
// from 4608 x 3072 -> 9216 (a turn of pairs: 26.2 us with groups of 64, 17.0 with groups of 128), whose clusters cost a call 0.9 us more.  Over 110
// shapes of 16 to 17816 rows, 512 to 11776 coefficients and 512 to 12240 columns what is chosen is within 3 % of the fastest plan, in the mean
// within 0.5 % (one call of 7 us: 5 %).
inline int choose_w4a4_plan(int M, int N, int K_lp, int G, int sms) {
    struct Candidate { int plan, rows, columns, ctas; double cost64, cost128; };
    static constexpr Candidate kPlans[] = {{32, 128, 32, 1, 0.25, 0.0}, {64, 128, 64, 1, 0.295, 0.38}, {128, 128, 128, 1, 0.615, 0.73}, {192, 128, 192, 1, 0.846, 0.957},
                                           {130, 256, 128, 1, 1.02, 1.03}, {256, 128, 256, 1, 1.068, 1.21}, {258, 256, 256, 2, 1.0, 1.0}};
    int plan = 0;
    double best = 0.0;
    for (const Candidate& c : kPlans) {
        if (c.plan == 32 && (G != 64 || (M + 127L) / 128 * ((N + 31) / 32) > sms / 2)) continue;  // (see w4a4_narrow.cu)
        const long tiles = (static_cast<long>(M) + c.rows - 1) / c.rows * ((N + c.columns - 1) / c.columns), slots = sms / c.ctas;
        const double t = static_cast<double>((tiles + slots - 1) / slots) * (G == 64 ? c.cost64 : c.cost128) + (c.ctas == 2 ? 100.0 / K_lp : 0.0);
        if (plan == 0 || t < best) {
            plan = c.plan;
            best = t;
        }
    }
    return plan;
}

}  // namespace dirotq
