// Estimated time of a J/K part (a launch over one angular class) for each kernel shape that computes it,
// and the choice between the shapes.  Host only.
//
// The parts of a build run side by side, so a shape is charged for the share of the GPU it takes as well
// as for its latency, in the way the autotuner measures it: the time of JK_COPIES launches together.
//   latency    = t0 + it (a fp + a1) + b fix     the serial chain of one quartet: its longest lane's `it`
//                                                primitive quartets, then sums, HRR and digestion
//   throughput = quartets (it G (c fp + c1) + d fix G + e)       the instructions of every quartet
//   time       = (latency^3 + (JK_COPIES throughput)^3)^(1/3)
// with fp the algorithmic flops of a primitive quartet, h those of the HRR and the sums, g those of the
// digestion, fix = h + g, and where G lanes deal out the digestion h + g / G (G = 1 for the team kernels).
// The constants (microseconds) are fitted by least squares on the logarithm to 4000 such timings on one
// GB300: every class and shape, 1 to 13 million quartets, 1 to 420 primitive quartets each, from one water
// in STO-3G to (H2O)_32 in 6-31G*; one timing was estimated within 12 to 33 % (one standard deviation).
// The timings are of the kernels before the bra runs (MESS_RUN_MIN), the finer FP32 Boys rows, the double-float sums
// normalised once per expression (8 to 23 % faster) and the split of primitive quartets over blocks (prim_split). The
// estimate has no terms for runs and that split: a part in runs (up to 3.3 times faster) is ordered and put on a stream by
// the time of one thread per quartet. With the kernels of the fit, summed over the parts of a build,
// the chosen shapes took 541, 5669, 2293, 3019 and 27880 us for C2H6 and (H2O)_8 (FP64), (H2O)_8, C7H16 and (H2O)_32
// (mixed), where the best shape of every part, found by timing them all, took 527, 5515, 2204, 2882 and 27223 us.
// Against fixed thresholds on quartets and primitives, whole builds: one water 251 -> 115 us, (H2O)_8 6.8 -> 4.8 ms
// (FP64), (H2O)_8 1.48 -> 1.03, C7H16 1.19 -> 0.94 and (H2O)_32 16.3 -> 16.0 ms (mixed).
#pragma once
#include <math.h>

#include "eri_launch.h"

constexpr double JK_COPIES = 8.0;

struct JkShape { int G, team, mode; };   // lanes per quartet, team kernel (0..3), arithmetic (MESS_MODE_*)
struct JkWork { double fp, h, g, quartets, prims; };

struct JkCost { double a, a1, b, t0, c, c1, d, e; };

// one thread per quartet in straight-line code, or running the op program; G lanes; a warp, a block, a
// block with split primitives per quartet
enum { JK_LINE = 0, JK_PROGRAM = 1, JK_LANES = 2, JK_WARP = 3, JK_BLOCK = 4, JK_SPLIT = 5 };

inline const JkCost& jk_cost(int mode, int family)
{
    static const JkCost fp64[6] = {{0.02, 2.39, 0.0613, 28.4, 2.11e-6, 1.58e-5, 1.32e-6, 1.55e-4},
                                   {0.0571, 0, 0.115, 210.0, 1.04e-5, 0, 0, 0},
                                   {0.016, 2.81, 0.0447, 24.2, 1.65e-6, 1.3e-5, 1.09e-6, 5.82e-4},
                                   {2.2e-3, 3.36, 1.44e-3, 63.5, 5.69e-6, 3.1e-3, 1.2e-6, 1.25e-3},
                                   {0, 4.72, 0, 62.3, 5.33e-6, 0.0119, 0, 3.89e-3},
                                   {2.62e-3, 3.11, 1.61e-4, 41.4, 1.43e-5, 0.0131, 0, 0}};
    static const JkCost df32[6] = {{0, 1.05, 0.18, 19.7, 3.47e-7, 0, 2.71e-6, 0},
                                   {0.0438, 0, 0.114, 80.4, 1.16e-6, 0, 3.52e-6, 0},
                                   {7.97e-3, 0.563, 0.143, 22.4, 3.4e-7, 0, 1.89e-6, 6.4e-5},
                                   {1.62e-3, 1.64, 7.99e-4, 66.3, 1.22e-6, 8.81e-4, 1.9e-6, 1.31e-3},
                                   {0, 2.23, 0, 56.8, 1.99e-6, 3.29e-3, 6.65e-7, 5.09e-3},
                                   {0, 2.17, 2.92e-3, 44.9, 5.38e-6, 2.73e-3, 2.14e-6, 4.1e-3}};
    // FP32 (the op program, never the best, by the double-float constants; FP32 with FP64 Boys as FP32)
    static const JkCost fp32[6] = {{0, 0.271, 5.27e-3, 30.0, 3.31e-8, 0, 3.69e-7, 5.79e-5},
                                   {0.0438, 0, 0.114, 80.4, 1.16e-6, 0, 3.52e-6, 0},
                                   {0, 0.185, 0, 23.4, 2.57e-8, 2.81e-6, 3.78e-7, 1.38e-4},
                                   {3.13e-4, 1.06, 5.45e-4, 72.5, 5.54e-7, 3.16e-4, 5.91e-7, 4.26e-4},
                                   {1.66e-4, 1.5, 8.19e-4, 35.3, 7.07e-7, 1.16e-3, 3.16e-7, 1.4e-3},
                                   {3.47e-4, 1.31, 3.86e-3, 27.6, 2.24e-6, 1.11e-3, 4.68e-7, 9.51e-4}};
    return (mode == MESS_MODE_FP64 ? fp64 : mode == MESS_MODE_DF32 ? df32 : fp32)[family];
}

inline double jk_time(const mess_qclass_info& c, const JkShape& v, const JkWork& w)
{
    const int line = v.mode == MESS_MODE_FP64 ? 2 : v.mode == MESS_MODE_DF32 ? 4 : 1;
    const int family = v.team ? JK_WARP + v.team - 1 : v.G > 1 ? JK_LANES : (c.line & line) ? JK_LINE : JK_PROGRAM;
    const JkCost& k = jk_cost(v.mode, family);
    const double avg = w.quartets > 0.0 ? w.prims / w.quartets : 0.0;
    const double it = family == JK_LANES ? ceil(avg / v.G) : family == JK_SPLIT ? ceil(avg / MESS_TEAM_WARPS) : avg;
    const double lanes = family == JK_LANES ? v.G : 1.0, fix = w.h + w.g / lanes;
    const double lat = k.t0 + it * (k.a * w.fp + k.a1) + k.b * fix;
    const double thr = JK_COPIES * w.quartets * (it * lanes * (k.c * w.fp + k.c1) + k.d * fix * lanes + k.e);
    return cbrt(lat * lat * lat + thr * thr * thr);
}

// the shape with the smallest estimated time among those that exist for the class
inline JkShape jk_choose(const mess_qclass_info& c, int mode, const JkWork& w)
{
    JkShape best{1, 0, mode};
    double least = 1e300;
    auto consider = [&](int G, int team) {
        const JkShape v{G, team, mode};
        const double t = jk_time(c, v, w);
        if (t < least) { least = t; best = v; }
    };
    consider(1, 0);
    if (c.straight)
        for (int G : {4, 8, 32}) consider(G, 0);
    if (c.team)
        for (int team : {1, 2, 3}) consider(1, team);
    return best;
}
