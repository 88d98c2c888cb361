// Plain-data layouts shared by the host code and the kernels (no torch types anywhere).
#pragma once
#include <stdint.h>

// Boys-function values reported by mess_boys_grid: rows k = 0..MESS_BOYS_NROW-1 at T_k = k *
// MESS_BOYS_DT; columns n = 0..NF-1 hold F_n(T_k) and column NF holds exp(-T_k).  The kernels expand
// around finer grids of the same routine (below), whose steps FP32 and FP64 hold exactly.
#define MESS_BOYS_DT 0.1
#define MESS_BOYS_TMAX64 48.0     // FP64: Taylor expansion below this
#define MESS_BOYS_TMAXDF 36.0     // double-float, and the FP64 Boys function of FP32 quartets
#define MESS_BOYS_TMAX32 36.0     // FP32
#define MESS_BOYS_TMAX32_L5 30.0  // FP32, highest order up to 5
#define MESS_BOYS_NF 16
#define MESS_BOYS_NCOL (MESS_BOYS_NF + 1)
#define MESS_BOYS_NROW 362
#define MESS_BOYS_NL 9            // orders L = 0..8 of the FP32 Taylor rows (L = la+lb+lc+ld <= 8)
// FP64 rows: step 1/32 (|T_k - T| <= 1/64, so order 6 leaves 5e-17), per order L and row 64 bytes:
// F_{L+j}(T_k) / j! for j = 0..6, exp(-T_k).  Double-float rows: step 1/64 (order 5: 3e-16), 48 bytes:
// the coefficients of j = 0..3 as hi, lo, of j = 4, 5 (whose terms are below 2e-10) as FP32, exp(-T_k)
// as hi, lo.  With 1/j! in the coefficients a term is one FMA.
#define MESS_BOYS64_INV_DT 32.0
#define MESS_BOYS64_NROW 1538
#define MESS_BOYSDF_INV_DT 64.0
#define MESS_BOYSDF_NROW 2306
// FP32 rows: step 1/128, which FP32 holds exactly (T_k - T is then exact; a step of 0.1 or 0.05 rounded to
// FP32 shifts x by up to 5e-7 at the far end of the grid, a one-signed error of up to 1e-7 in F_L).
// F_L, F_L+1, F_L+2 / 2 and exp(-T_k) in one 16-byte row: order 2 leaves at most 8e-9 of F_L, of both signs.
// L = 0, which needs no exp(-T): F_0, F_1, F_2 / 2, F_3 / 6 at a step of 1/32 (order 3 leaves 3e-10).
#define MESS_BOYS32_INV_DT 128.0
#define MESS_BOYS32_INV_DT0 32.0
#define MESS_BOYS32_NROW 4610

#define MESS_PRIM_EPS 1e-18       // primitive pairs below this weight bound are left out (build_pairs)

#define MESS_LMAX 2               // s, p, Cartesian d
#define MESS_NUM_PCLASS 6         // pair classes (la,lb): ss ps pp ds dp dd
#define MESS_NGROUP 3             // primitive-pair count groups: <= 3, 4..12, >= 13
// pair lists: per class, primitive group and whether the pair has an extra shell (a raised or lowered
// shell of a derivative basis; none elsewhere)
#define MESS_NLIST (2 * MESS_NUM_PCLASS * MESS_NGROUP)
#define MESS_LIST(extra, pclass, group) (((extra) * MESS_NUM_PCLASS + (pclass)) * MESS_NGROUP + (group))
#define MESS_TEAM_WARPS 4         // warps (one shell quartet each) per block of the large-class kernels

// One primitive pair: zeta, PAx, PAy, PAz (P - A, P the Gaussian product centre), K, 1/(2 zeta), and
// two padding slots: 32 bytes in FP32 (one sector per record), 64 in FP64 and double-float.
template <typename R> struct alignas(32) PrimPairRec { R v[8]; };

// Everything a J/K kernel reads about the ket pair of a quartet, in one 112-byte record (seven 16-byte
// loads at most; the arithmetic reads only the ones it needs).  Stored per pair (pair order) and per
// class list (list order, so that the consecutive kets of consecutive lanes are adjacent).
//   [0]   pp_off, pp_n, fa | fb << 16 (first functions within the molecule), same | mol << 1
//   [16]  C (centre of the pair's first shell) and A - B, FP64
//   [64]  C as FP32 hi[3], lo[3]; A - B in FP32; the pair id
struct alignas(16) KetRec {
    int pp_off, pp_n, fab, flags;
    double C[3], AB[3];
    float Cf[6], ABf[3];
    int pair;
};

// One launch over a class bin (a contiguous range of quartets of one angular class).
struct BinLaunch {
    const int* bra;          // [nbra] pair ids, Q descending
    const int* ket;          // ket list (pair ids, Q descending)
    const KetRec* ketrec;    // the ket list's records, same order
    const long long* offs;   // [nbra + 1] exclusive prefix of ket counts
    const int* kbeg;         // [nbra] first ket index of each bra
    const int* seg;          // [ceil(total / 32)] bra of quartet 32 k (narrows the bra search)
    int nbra;
    long long total;
};

// A bin's bras in runs that share their first shell (FP32 parts, see k_jk_run_*): one thread per (run,
// ket), ket ranges as the union over the run's bras.
#define MESS_RUN_MAX 8            // bras per run at most
// A part is laid out in runs when it has many shell quartets (a run takes an eighth of the threads) with few
// primitive quartets each (with more, the primitives bound it, and the registers that hold the run's sums cost
// warps).  One thread per quartet -> runs, (H2O)_32 / 6-31G* and (H2O)_64 / STO-3G, 13 M (ps|ss) quartets of 4
// primitive quartets 1830 -> 548 us, 3.7 M (ds|ps) of 3 1487 -> 457, 3.2 M (ps|ss) of 13 354 -> 290, 1.9 M of 14
// 182 -> 188; of 46: 12 M (ss|ss) 1555 -> 1548, 1.5 M (pp|ss) 353 -> 455, 0.7 M (pp|ps) 343 -> 485.  16 bras per
// run instead of 8: 0 to 20 % slower.
#define MESS_RUN_MIN (1LL << 19)
#define MESS_RUN_PRIM 16
struct RunLaunch {
    const int4* run;         // [nrun] first bra, number of bras, first ket, 0
    const long long* offs;   // [nrun + 1] exclusive prefix of the runs' ket counts
    const int* seg;          // [ceil(total / 32)] run of thread 32 k
    int nrun;
    long long total;         // threads
};
