// Host-side launch interface of the generated per-class ERI kernels.
#pragma once
#include <algorithm>

#include <cuda_runtime.h>

#include "df32.cuh"
#include "eri_classes.h"
#include "mess_device.h"

template <typename R> struct PairTable;

enum { MESS_KIND_JK = 0, MESS_KIND_STORE = 1, MESS_KIND_SCHWARZ = 2 };
// kernel modes: FP64; FP32 recursion with FP64 Boys at small T; FP32 recursion with FP32 Boys;
// double-float (FP32 pairs) recursion and Boys
enum { MESS_MODE_FP64 = 0, MESS_MODE_MIXED = 1, MESS_MODE_FP32 = 2, MESS_MODE_DF32 = 3 };

struct ClassLaunchArgs {
    int kind;                    // MESS_KIND_*
    int mode;                    // MESS_MODE_* (JK only)
    int G;                       // JK: lanes per shell quartet (1, 4, 8 or 32)
    int team;                    // JK: 1 = one warp per shell quartet (level-scheduled program)
    int split;                   // JK: blocks that share a quartet's primitive quartets (G = 32, team 3; 0: one)
    BinLaunch bin;               // JK / STORE
    const RunLaunch* runs;       // JK: the FP32 one-thread kernel goes by bra runs (null: by quartets)
    const int* pairs;            // SCHWARZ: pair ids of one diagonal class
    int npairs;
    const PairTable<double>* P64_ptr;
    const PairTable<float>* P32_ptr;
    const PairTable<df32>* Pdf_ptr;
    const double* D;             // device, n x n
    const float* D32;            // D rounded to FP32 (FP32 kernels)
    const float2* Ddf;           // D as double-float hi, lo (double-float kernels)
    double* J;                   // device, n x n accumulators
    double* K;
    double* out;                 // STORE: n^4 tensor; SCHWARZ: Q per pair
    int n;
    cudaStream_t stream;
};

template <typename R> inline const typename DElem<R>::T* dmat(const ClassLaunchArgs& a);
template <> inline const double* dmat<double>(const ClassLaunchArgs& a) { return a.D; }
template <> inline const float* dmat<float>(const ClassLaunchArgs& a) { return a.D32; }
template <> inline const float2* dmat<df32>(const ClassLaunchArgs& a) { return a.Ddf; }

// Threads per block of the straight-line J/K kernels: one warp while the warps are fewer than eight per
// SM, so that they spread over the SMs (the FP64 pipe of an SM serves one warp instruction in 16 cycles
// and is full with one block of four warps), else four warps (MESS_THREADS).
inline int jk_block_threads(long long threads) { return threads < 152LL * 8 * 32 ? 32 : 128; }

// Lanes per pair of the Schwarz kernels: as few as still give the FP64 pipes four warps per SM (more
// lanes repeat the per-pair part of the work), 32 where there are too few pairs for that.
inline int schwarz_lanes(int npairs)
{
    const long long fill = 152LL * 4 * 32;
    return npairs >= fill ? 1 : (8LL * npairs >= fill ? 8 : 32);
}

// Blocks over which the primitive quartets of a part's shell quartets are split (the J/K digestion is linear in
// the integrals, so each block adds its share's): the quartets of a part on a warp (G = 32) or a block
// (team 3) each run their primitive quartets as one chain, which a part of fewer quartets than SMs
// leaves on a few of them.  At most two blocks per SM, a full pass of lanes each, and kMaxBlocks per quartet: each
// block adds to K, so more of them round more often (one water / 6-31G, mean error of K against extended precision
// over 48 densities: 5.9e-16 before the split and the fitted shapes, 6.4e-16 with four blocks, 7.0e-16 with up to 304; two blocks 107 us per
// call, three or more 98).  Only where the whole build
// has few quartets: otherwise the other parts fill the SMs, and the repeated HRR and digestion cost more
// (kMaxBuild lies between one water / 6-31G, 1,035 quartets, 98 -> 76 us, and C2H6 / 6-31G*, 45,000, 352 -> 367).
// One water / STO-3G in FP64: (pp|pp), one quartet of 81 primitive quartets, 80 -> 45 us, (pp|ps) 31 -> 18, the
// whole call 115 -> 80.
inline int prim_split(long long quartets, long long prim_quartets, int G, int team, long long build_quartets)
{
    constexpr long long kMaxBuild = 16384, kMaxBlocks = 4;
    if (build_quartets > kMaxBuild) return 1;
    const int lanes = team == 3 ? MESS_TEAM_WARPS : (G == 32 && !team ? 32 : 0);
    if (!lanes || quartets <= 0 || quartets > 152) return 1;
    const long long passes = (prim_quartets / quartets + lanes - 1) / lanes;
    return (int)std::max(1LL, std::min({passes, 2 * 152 / quartets, kMaxBlocks}));
}

typedef cudaError_t (*mess_class_launcher)(const ClassLaunchArgs&);
extern const mess_class_launcher MESS_CLASS_LAUNCHERS[MESS_NUM_QCLASS];

// Launch of a warp-per-quartet kernel with its dynamic shared memory (opt-in above 48 KB, set
// once per kernel).
template <typename R, int BMODE, typename Kern>
cudaError_t mess_team_launch(Kern kern, dim3 grid, size_t smem, const ClassLaunchArgs& a, const PairTable<R>& P,
                             int* configured /* per kernel: 0 until the attribute is set on this device */)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!configured[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        configured[dev] = 1;
    }
    kern<<<grid, 32 * MESS_TEAM_WARPS, smem, a.stream>>>(a.bin, P, dmat<R>(a), a.J, a.K, a.n);
    return cudaGetLastError();
}
