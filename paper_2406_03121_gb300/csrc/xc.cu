// Exchange-correlation part of the Kohn-Sham energy functional (paper Sec. 5.1: the Hamiltonian's
// xc_method "lda" or "pbe"): the density of a closed-shell density matrix on a molecular quadrature
// grid, the functional's energy and its matrix V_xc,mn = dE_xc / dD_mn.
//
// Grid (per atom, then Becke's fuzzy-cell partition between the atoms of each molecule):
//   radial: Gauss-Chebyshev of the second kind, x_i = cos(i pi / (N + 1)), i = 1..N, weight
//           pi / (N + 1) sin^2(i pi / (N + 1)) / sqrt(1 - x_i^2), mapped by r = R (1 + x) / (1 - x)
//           (Jacobian 2 R / (1 - x)^2, times r^2); R = 0.35 angstrom for H (its Bragg-Slater
//           radius), half the Bragg-Slater radius otherwise (C 0.35, N 0.325, O 0.30 angstrom);
//           N = 50 for H, 75 otherwise;
//   angular: Gauss-Legendre nodes in cos(theta) (16) times 32 equally spaced phi, weight
//           w_theta * 2 pi / 32;
//   partition: w_A(r) = P_A(r) / sum_B P_B(r), P_A = prod_{B != A} s(mu_AB), mu_AB = (|r - R_A| -
//           |r - R_B|) / |R_A - R_B|, s(mu) = (1 - f(f(f(mu)))) / 2, f(mu) = 3/2 mu - 1/2 mu^3.
// Functionals (closed shell): LDA = Slater exchange + Perdew-Wang 1992 correlation; PBE (Perdew,
// Burke & Ernzerhof 1996) on top of the same PW92 correlation.  Derivatives are written out
// analytically below.
#include <math.h>

#include <algorithm>
#include <vector>

#include "mess_internal.h"

namespace {

constexpr double kAngstrom = 1.0 / 0.52917721092;
constexpr int kNTheta = 16, kNPhi = 32;
constexpr int kFuncThreads = 128;                   // points per block of the functional
constexpr int kVxcThreads = 256, kVxcTile = 64;     // threads and function tile of the V_xc reduction
constexpr int kVxcMaxEl = kVxcTile * kVxcTile / kVxcThreads;   // elements per thread at most
constexpr int kSmallN = 4;                            // functions up to which V_xc is summed by the functional
constexpr int kLogBins = 128;                       // entries of the logarithm table
constexpr double kRhoMin = 1e-14;   // points with less density carry no exchange-correlation energy

double radius_of(int Z)
{
    switch (Z) {
    case 1: return 0.35;
    case 6: return 0.35;
    case 7: return 0.325;
    case 8: return 0.30;
    default: return 0.35;
    }
}

// Gauss-Legendre nodes and weights on [-1, 1]: Newton's method on P_n from the Chebyshev guesses
// cos(pi (i + 3/4) / (n + 1/2)), P_n and P_n' by the three-term recurrence.
void gauss_legendre(int n, std::vector<double>& x, std::vector<double>& w)
{
    x.assign(n, 0.0);
    w.assign(n, 0.0);
    for (int i = 0; i < n; ++i) {
        double z = cos(M_PI * (i + 0.75) / (n + 0.5)), dp = 0.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = z;
            for (int k = 2; k <= n; ++k) {
                const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            dp = n * (z * p1 - p0) / (z * z - 1.0);
            const double dz = p1 / dp;
            z -= dz;
            if (fabs(dz) < 1e-16) break;
        }
        x[n - 1 - i] = z;
        w[n - 1 - i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
}

// ------------------------------------------------------------------------------------------ kernels
// Points and weights before the partition, one thread per point.  tab (after the table of log_1p): the
// angular table (cos theta, sin theta, weight for kNTheta; cos phi, sin phi for kNPhi), then per radial grid its radii and weights.
// (Tabulated on the host and copied, the 3.3 million points of 64 H2 took about 70 ms of a call; here 0.05.)
constexpr int kAngular = kNTheta * kNPhi, kAngularAt = 2 * kLogBins, kAngularTab = kAngularAt + 3 * kNTheta + 2 * kNPhi;
constexpr int kRadialMax = 75, kGridThreads = 256, kBlocksPerAtom = kRadialMax * kAngular / kGridThreads;
static_assert(kRadialMax * kAngular % kGridThreads == 0, "whole blocks per atom");

__global__ void __launch_bounds__(kGridThreads) k_grid(const double* __restrict__ tab, const int* __restrict__ radial_at,
                                                       const int* __restrict__ radial_n, const long long* __restrict__ abase,
                                                       const double* __restrict__ xyz, double* __restrict__ pts,
                                                       double* __restrict__ w, int* __restrict__ atom)
{
    const int A = blockIdx.x / kBlocksPerAtom;
    const int t = (blockIdx.x % kBlocksPerAtom) * kGridThreads + threadIdx.x;
    const int i = t / kAngular, th = t % kAngular / kNPhi, ph = t % kNPhi, nr = radial_n[A];
    if (i >= nr) return;
    const double* rad = tab + radial_at[A];
    const double* ang = tab + kAngularAt;
    const double r = rad[i], st = ang[kNTheta + th];
    const long long p = abase[A] + t;
    pts[3 * p] = xyz[3 * A] + r * st * ang[3 * kNTheta + ph];
    pts[3 * p + 1] = xyz[3 * A + 1] + r * st * ang[3 * kNTheta + kNPhi + ph];
    pts[3 * p + 2] = xyz[3 * A + 2] + r * ang[th];
    w[p] = rad[nr + i] * ang[2 * kNTheta + th] * 2.0 * M_PI / kNPhi;
    atom[p] = A;
}

struct GridArgs {
    const double* pts;       // [npts][3]
    double* w;               // [npts] radial x angular weight, times the partition after k_becke
    const int* atom;         // [npts] global atom index of the point's atomic grid
    const int* atom_mol;     // [natom]
    const int* atom_off;     // [nmol] first atom of each molecule
    const int* atom_n;       // [nmol]
    const double* xyz;       // [natom][3]
    long long npts;
};

__global__ void k_becke(GridArgs g)
{
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= g.npts) return;
    const int own = g.atom[p], m = g.atom_mol[own], a0 = g.atom_off[m], na = g.atom_n[m];
    if (na == 1) return;
    const double x = g.pts[3 * p], y = g.pts[3 * p + 1], z = g.pts[3 * p + 2];
    double sum = 0.0, mine = 0.0;
    for (int A = a0; A < a0 + na; ++A) {
        const double* RA = g.xyz + 3 * A;
        const double dA = sqrt((x - RA[0]) * (x - RA[0]) + (y - RA[1]) * (y - RA[1]) + (z - RA[2]) * (z - RA[2]));
        double P = 1.0;
        for (int B = a0; B < a0 + na; ++B) {
            if (B == A) continue;
            const double* RB = g.xyz + 3 * B;
            const double dB = sqrt((x - RB[0]) * (x - RB[0]) + (y - RB[1]) * (y - RB[1]) + (z - RB[2]) * (z - RB[2]));
            const double RAB = sqrt((RA[0] - RB[0]) * (RA[0] - RB[0]) + (RA[1] - RB[1]) * (RA[1] - RB[1]) +
                                    (RA[2] - RB[2]) * (RA[2] - RB[2]));
            double f = (dA - dB) / RAB;
            for (int k = 0; k < 3; ++k) f = 1.5 * f - 0.5 * f * f * f;
            P *= 0.5 * (1.0 - f);
        }
        sum += P;
        if (A == own) mine = P;
    }
    g.w[p] *= sum > 0.0 ? mine / sum : 0.0;
}

struct AoArgs {
    const double* pts;
    const int* atom;         // [npts]
    const int* atom_mol;     // [natom]
    long long npts;
    const int* shell_off;    // [nmol] first shell of the molecule
    const int* shell_n;      // [nmol]
    const int* shell_l;
    const int* shell_K;
    const int* shell_poff;   // first primitive of the shell
    const int* shell_fl;     // first function of the shell within its molecule
    const double* shell_R;   // [nshell][3]
    const double* alpha;
    const double* coef;
    const double* fscale;    // per global function: component normalisation
    const int* fbase;        // [nmol] global index of the molecule's first function
    const long long* pbase;  // [nmol + 1]
    const long long* aobase; // [nmol] offset of the molecule's [n_m][npts_m] block
    const int* mn;           // [nmol] functions of the molecule
    double* phi;             // values
    double* dphi;            // gradients: three blocks [3][n_m][npts_m] from 3 * aobase[m]
};

// value and gradient of every basis function of the point's molecule at the point.  Stored function by
// function, so that here and in every later pass the threads of a warp (consecutive points) touch
// consecutive addresses.
__global__ void k_ao(AoArgs a)
{
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.npts) return;
    const int m = a.atom_mol[a.atom[p]], n = a.mn[m];
    const long long lp = p - a.pbase[m], np_ = a.pbase[m + 1] - a.pbase[m];
    double* ph = a.phi + a.aobase[m] + lp;
    double* dx = a.dphi + 3 * a.aobase[m] + lp;
    double* dy = dx + np_ * n;
    double* dz = dy + np_ * n;
    const double x = a.pts[3 * p], y = a.pts[3 * p + 1], z = a.pts[3 * p + 2];
    for (int s = a.shell_off[m]; s < a.shell_off[m] + a.shell_n[m]; ++s) {
        const double X = x - a.shell_R[3 * s], Y = y - a.shell_R[3 * s + 1], Z = z - a.shell_R[3 * s + 2];
        const double r2 = X * X + Y * Y + Z * Z;
        double g = 0.0, gd = 0.0;   // sum c e^{-a r^2}, sum -2 a c e^{-a r^2}
        for (int k = 0; k < a.shell_K[s]; ++k) {
            const double al = a.alpha[a.shell_poff[s] + k];
            const double e = a.coef[a.shell_poff[s] + k] * exp(-al * r2);
            g += e;
            gd -= 2.0 * al * e;
        }
        const int l = a.shell_l[s], f0 = a.shell_fl[s];
        int k = 0;
        for (int lx = l; lx >= 0; --lx)
            for (int ly = l - lx; ly >= 0; --ly, ++k) {
                const int lz = l - lx - ly;
                const double px = lx == 0 ? 1.0 : (lx == 1 ? X : X * X);
                const double py = ly == 0 ? 1.0 : (ly == 1 ? Y : Y * Y);
                const double pz = lz == 0 ? 1.0 : (lz == 1 ? Z : Z * Z);
                const double dpx = lx == 0 ? 0.0 : (lx == 1 ? 1.0 : 2.0 * X);
                const double dpy = ly == 0 ? 0.0 : (ly == 1 ? 1.0 : 2.0 * Y);
                const double dpz = lz == 0 ? 0.0 : (lz == 1 ? 1.0 : 2.0 * Z);
                const double sc = a.fscale[a.fbase[m] + f0 + k];
                const double poly = px * py * pz;
                const long long at = (long long)(f0 + k) * np_;
                ph[at] = sc * poly * g;
                dx[at] = sc * (dpx * py * pz * g + poly * gd * X);
                dy[at] = sc * (px * dpy * pz * g + poly * gd * Y);
                dz[at] = sc * (px * py * dpz * g + poly * gd * Z);
            }
    }
}

// Roots, reciprocals and logarithms of the functional in few FP64 instructions (each takes 16 cycles of an
// SM; the library's log1p, rcbrt, sqrt and division took most of an LDA point's): an FP32 estimate and the first
// terms of the series in what it leaves, e.  Reciprocal and reciprocal root: e below 4e-7 (the roundings to FP32 and
// the estimate's), and the next term, in e^3, below 1e-19.  Cube root, by exp2 of a third of log2 x, which is rounded in
// proportion to its size (up to 100): e below 1e-5 at the ends of the range and 3e-6 about x = 1, next term 2e-16 and 1e-17.
// x^(-1/3) for 1e-14 <= x (an FP32 number): (1 - e)^(-1/3) = 1 + e/3 + 2/9 e^2, e = 1 - x y^3
__device__ __forceinline__ double inv_cbrt(double x)
{
    if (x > 1e30) return rcbrt(x);
    const double y = f2d_alu(exp2f(log2f(d2f_alu(x)) * (-1.0f / 3.0f)));
    const double e = fma(-x, y * y * y, 1.0);
    return fma(y * e, fma(e, 2.0 / 9.0, 1.0 / 3.0), y);
}
// x^(1/2) = x x^(-1/2), (1 - e)^(-1/2) = 1 + e/2 + 3/8 e^2, e = 1 - x y^2
__device__ __forceinline__ double fast_sqrt(double x)
{
    const float f = d2f_alu(x);
    if (f < 1e-30f) return sqrt(x);
    const double y = f2d_alu(rsqrtf(f));
    const double e = fma(-x * y, y, 1.0);
    return x * fma(y * e, fma(e, 0.375, 0.5), y);
}
// 1 / x: (1 - e)^(-1) = 1 + e + e^2, e = 1 - x y
__device__ __forceinline__ double fast_inv(double x)
{
    const float f = d2f_alu(x);
    if (f < 1e-30f) return 1.0 / x;
    const double y = f2d_alu(__frcp_rn(f));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
// log(1 + y), y >= 0: 1 + y = 2^k m, m c = 1 + w with c about 1/m from a table of 128 (c, -log c) over the
// leading bits of m (c = 1 in the first, so that small y keep their relative accuracy), and the series of
// log(1 + w) to w^8 (|w| <= 1/128).  What 1 + y rounds off goes into w.
__device__ __forceinline__ double log_1p(double y, const double2* __restrict__ tab)
{
    const double z = 1.0 + y, lost = y - (z - 1.0);
    const int hi = __double2hiint(z), k = (hi >> 20) - 1023;
    const double m = __hiloint2double((hi & 0xfffff) | 0x3ff00000, __double2loint(z));
    const double2 t = __ldg(tab + ((hi >> 13) & (kLogBins - 1)));
    const double w = fma(lost * __hiloint2double((1023 - k) << 20, 0), t.x, fma(m, t.x, -1.0));
    double p = 1.0 / 7 - w * (1.0 / 8);
    p = -1.0 / 6 + w * p;
    p = 1.0 / 5 + w * p;
    p = -1.0 / 4 + w * p;
    p = 1.0 / 3 + w * p;
    p = -1.0 / 2 + w * p;
    p = w + w * w * p;
    const double kd = __hiloint2double(0x43300000, k ^ (int)0x80000000) - 4503601774854144.0;   // k without I2F
    return y < 1e300 ? fma(kd, M_LN2, t.y + p) : log1p(y);
}

// Perdew-Wang 1992 correlation energy per electron (closed shell) and its derivative in rs, from rs
// and 1 / rs.  One division: log(1 + 1/Q) and dQ / (Q (Q + 1)) share 1 / (Q (Q + 1)).
__device__ __forceinline__ void pw92(double rs, double irs, const double2* __restrict__ logs, double& ec, double& dec)
{
    const double A = 0.031091, a1 = 0.21370, b1 = 7.5957, b2 = 3.5876, b3 = 1.6382, b4 = 0.49294;
    const double srs = fast_sqrt(rs);
    const double Q = 2.0 * A * srs * (b1 + srs * (b2 + srs * (b3 + srs * b4)));
    const double dQ = 2.0 * A * (0.5 * b1 * srs * irs + b2 + 1.5 * b3 * srs + 2.0 * b4 * rs);
    const double r = fast_inv(Q * (Q + 1.0));
    const double L = log_1p((Q + 1.0) * r, logs);
    ec = -2.0 * A * (1.0 + a1 * rs) * L;
    dec = -2.0 * A * a1 * L + 2.0 * A * (1.0 + a1 * rs) * dQ * r;
}

struct FuncArgs {
    const double* phi;
    const double* dphi;
    const double* D;         // packed density
    const long long* mbase;  // [nmol] offset of the molecule's n x n block
    const long long* pbase;
    const long long* aobase;
    const int* mn;
    const double* w;
    double* vrho;            // [npts] w * d e / d rho
    double* vgrad;           // [npts][3] w * 2 d e / d sigma * grad rho (PBE)
    const double2* logs;     // table of log_1p
    double* Exc;             // [nmol] accumulated
    double* V;               // packed, accumulated (N > 0)
    int ppt;                 // points per thread
};

// density, its gradient, and the functional at every point of a molecule (grid.y = molecule, ppt points
// per thread); E_xc accumulated per molecule.  N > 0: the molecules have at most N functions, and the
// kernel adds V_xc as well (see k_vxc): a point's phi and v_rho are in its registers already, and N (N + 1) / 2
// sums per thread fit there.  N = 0: v_rho and v_sigma grad rho go to memory for k_vxc.
// Bound: the FP64 pipe (two FMA lanes per SM and clock): n^2 FMAs per point for D phi and about 80
// (LDA) to 170 (PBE) instructions of the functional.  So the memory side only has to stay out of the
// way: phi function by function (coalesced, re-read from L1), D as warp-uniform loads, four rows of D
// per pass so that four accumulation chains hide the FMA latency.  The functional works from
// rho^(-1/3) and multiplies where it can.  CH4 / 6-31G / PBE (17 functions, 140,800 points): 231 -> 155 us
// (167 with the library's roots and logarithms); 64 H2 (51,200 points each), LDA: 729 -> 445 us (546).
// With V_xc in it (N = 2), 480 us instead of 445 and k_vxc's 148; minimisation of 64 H2, 128 steps: STO-3G 95.0 ->
// 79.6 ms in LDA, 187 -> 177 in PBE; 6-31G (N = 4) 124 -> 104 and 224 -> 218.  Beyond four functions the sums of
// a thread outgrow its registers in PBE.
template <int KIND, int N>
__global__ void __launch_bounds__(kFuncThreads) k_functional(FuncArgs f)
{
    constexpr int NS = 1 + N * (N + 1) / 2;             // sums of a thread: E_xc, V_ij (i <= j)
    __shared__ double red[kFuncThreads / 32][NS];
    const int m = blockIdx.y, n = f.mn[m];
    const long long np_ = f.pbase[m + 1] - f.pbase[m];
    const long long first = (long long)blockIdx.x * kFuncThreads * f.ppt;
    if (first >= np_) return;
    double sum[NS], Dr[N > 0 ? N * N : 1];
#pragma unroll
    for (int k = 0; k < NS; ++k) sum[k] = 0.0;
#pragma unroll
    for (int k = 0; k < N * N; ++k) Dr[k] = k / N < n && k % N < n ? __ldg(f.D + f.mbase[m] + k / N * n + k % N) : 0.0;
    for (int pt = 0; pt < f.ppt; ++pt) {
        const long long lp = first + pt * kFuncThreads + threadIdx.x;
        if (lp >= np_) break;
        double e = 0.0, pv[N > 0 ? N : 1], dv[KIND == 2 && N > 0 ? 3 * N : 1];
        const double* ph = f.phi + f.aobase[m] + lp;
        const double* dx = f.dphi + 3 * f.aobase[m] + lp;
        const double* dy = dx + np_ * n;
        const double* dz = dy + np_ * n;
        const double* D = f.D + f.mbase[m];
        double rho = 0.0, gx = 0.0, gy = 0.0, gz = 0.0;
        auto row_done = [&](int i, double t) {
            rho += t * ph[i * np_];
            if (KIND == 2) {
                gx += 2.0 * t * dx[i * np_];
                gy += 2.0 * t * dy[i * np_];
                gz += 2.0 * t * dz[i * np_];
            }
        };
#pragma unroll
        for (int k = 0; k < N; ++k) {
            pv[k] = k < n ? ph[k * np_] : 0.0;
            if (KIND == 2) {
                dv[3 * k] = k < n ? dx[k * np_] : 0.0;
                dv[3 * k + 1] = k < n ? dy[k * np_] : 0.0;
                dv[3 * k + 2] = k < n ? dz[k * np_] : 0.0;
            }
        }
#pragma unroll
        for (int k = 0; k < N; ++k) {
            double t = 0.0;
#pragma unroll
            for (int j = 0; j < N; ++j) t += Dr[k * N + j] * pv[j];
            rho += t * pv[k];
            if (KIND == 2) {
                gx += 2.0 * t * dv[3 * k];
                gy += 2.0 * t * dv[3 * k + 1];
                gz += 2.0 * t * dv[3 * k + 2];
            }
        }
        int i = N > 0 ? n : 0;
        for (; i + 4 <= n; i += 4) {
            const double* D0 = D + (long long)i * n;
            double t0 = 0.0, t1 = 0.0, t2 = 0.0, t3 = 0.0;
            for (int j = 0; j < n; ++j) {
                const double pj = ph[j * np_];
                t0 += __ldg(D0 + j) * pj;
                t1 += __ldg(D0 + n + j) * pj;
                t2 += __ldg(D0 + 2 * n + j) * pj;
                t3 += __ldg(D0 + 3 * n + j) * pj;
            }
            row_done(i, t0);
            row_done(i + 1, t1);
            row_done(i + 2, t2);
            row_done(i + 3, t3);
        }
        for (; i < n; ++i) {
            double t = 0.0;
            for (int j = 0; j < n; ++j) t += __ldg(D + (long long)i * n + j) * ph[j * np_];
            row_done(i, t);
        }
        double vr = 0.0, vs = 0.0;
        if (rho > kRhoMin) {
            const double ic = inv_cbrt(rho), c13 = rho * ic * ic;    // rho^(-1/3), rho^(1/3)
            const double cx = 0.7385587663820224;    // (3/4)(3/pi)^(1/3)
            const double ex = -cx * rho * c13;
            const double vx = -(4.0 / 3.0) * cx * c13;
            const double k_rs = 0.6203504908994001;       // (3/(4 pi))^(1/3)
            const double rs = k_rs * ic;
            double ec, dec;
            pw92(rs, c13 * (1.0 / k_rs), f.logs, ec, dec);
            const double rdec = -(1.0 / 3.0) * dec * rs;   // rho d ec / d rho
            if (KIND == 1) {
                e = ex + rho * ec;
                vr = vx + ec + rdec;
            } else {
                const double sigma = gx * gx + gy * gy + gz * gz;
                const double kf = 3.0936677262801355;          // kF = (3 pi^2 rho)^(1/3) = kf rho^(1/3)
                const double kappa = 0.804, beta = 0.06672455060314922;
                const double mu = beta * M_PI * M_PI / 3.0, gamma = (1.0 - M_LN2) / (M_PI * M_PI);
                const double ir = ic * ic * ic, ir2 = ir * ir;  // 1 / rho, 1 / rho^2
                // exchange: ex F(s^2), s^2 = sigma / (2 kF rho)^2 (d s^2 / d rho = -8/3 s^2 / rho)
                const double ds2 = ic * ic * ir2 * (1.0 / (4.0 * kf * kf));
                const double s2 = sigma * ds2;
                const double rden = 1.0 / (1.0 + (mu / kappa) * s2);
                const double F = 1.0 + kappa - kappa * rden;
                const double dF = mu * rden * rden;
                const double dex_drho = vx * F + ex * dF * (-8.0 / 3.0) * s2 * ir;
                const double dex_dsig = ex * dF * ds2;
                // correlation: rho (ec + H), u = t^2 = sigma pi / (16 kF rho^2) (d u / d rho = -7/3 u / rho),
                // H = gamma log(1 + N/M), N = (beta/gamma) u (1 + A u), M = 1 + A u + (A u)^2
                const double du = ic * ir2 * (M_PI / (16.0 * kf));
                const double u = sigma * du;
                const double bg = beta / gamma;
                const double E1 = expm1(ec * (-1.0 / gamma));
                const double A = bg / E1;
                const double dA_dec = A * A * (E1 + 1.0) * (1.0 / beta);
                const double au = A * u;
                const double M = 1.0 + au + au * au;
                const double N = bg * u * (1.0 + au);
                const double rMN = 1.0 / (M * (M + N));        // dH/dy / M^2 = gamma rMN
                const double H = gamma * log_1p(N * (M + N) * rMN, f.logs);
                const double dH_du = gamma * rMN * bg * (1.0 + 2.0 * au);
                const double dH_dA = -gamma * rMN * bg * u * u * u * A * (2.0 + au);
                e = ex * F + rho * (ec + H);
                vr = dex_drho + ec + H + rdec + dH_dA * dA_dec * rdec - (7.0 / 3.0) * dH_du * u;
                vs = dex_dsig + rho * dH_du * du;
            }
        }
        const long long p = f.pbase[m] + lp;
        const double w = f.w[p];
        sum[0] += e * w;
        if (N > 0) {
            double a[N > 0 ? N : 1];                    // LDA: w v_rho phi; PBE: half of it, and the gradient's part
            const double ws = w * 2.0 * vs, wr = (KIND == 2 ? 0.5 : 1.0) * w * vr;
#pragma unroll
            for (int k = 0; k < N; ++k) {
                a[k] = wr * pv[k];
                if (KIND == 2) a[k] += ws * (gx * dv[3 * k] + gy * dv[3 * k + 1] + gz * dv[3 * k + 2]);
            }
#pragma unroll
            for (int c = 0; c < N; ++c)
#pragma unroll
                for (int r = 0; r <= c; ++r) {
                    double& v = sum[1 + c * (c + 1) / 2 + r];
                    v += a[r] * pv[c];
                    if (KIND == 2) v += pv[r] * a[c];
                }
        } else {
            f.vrho[p] = w * vr;
            if (KIND == 2) {
                f.vgrad[3 * p] = w * 2.0 * vs * gx;
                f.vgrad[3 * p + 1] = w * 2.0 * vs * gy;
                f.vgrad[3 * p + 2] = w * 2.0 * vs * gz;
            }
        }
    }
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        for (int o = 16; o > 0; o >>= 1) sum[k] += __shfl_xor_sync(0xffffffffu, sum[k], o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][k] = sum[k];
    }
    __syncthreads();
    const int k = threadIdx.x;
    if (k < NS) {
        double t = 0.0;
        for (int g = 0; g < kFuncThreads / 32; ++g) t += red[g][k];
        if (k == 0) {
            atomicAdd(f.Exc + m, t);
        } else {
            int c = 0;
            while ((c + 1) * (c + 2) / 2 <= k - 1) ++c;
            const int r = k - 1 - c * (c + 1) / 2;
            if (c < n) {
                double* V = f.V + f.mbase[m];
                atomicAdd(V + (long long)r * n + c, t);
                if (r != c) atomicAdd(V + (long long)c * n + r, t);
            }
        }
    }
}

struct VxcArgs {
    const double* phi;
    const double* dphi;
    const double* vrho;
    const double* vgrad;
    const long long* pbase;
    const long long* aobase;
    const long long* mbase;
    const int* mn;
    int chunk;               // points per block
    int tp;                  // points staged at a time
    double* V;               // packed, accumulated
};

// (molecules of more than kSmallN functions)
// V_mn += sum over a chunk of the molecule's points of a_m phi_n + phi_m a_n, a = (1/2) w v_rho phi +
// w 2 v_sigma grad rho . grad phi (vgrad holds w 2 v_sigma grad rho); LDA: of w v_rho phi_m phi_n; grid (chunks, tile pairs, nmol).
// A block owns the elements m <= n of one pair of kVxcTile x kVxcTile function tiles.  It stages phi and
// a of tp points at a time in shared memory (a is formed once per function and point) and every thread
// sums its elements over the points.  Where a tile pair has fewer elements than threads (H2: 3), groups
// of threads take different points and are summed at the end.
// Bound: FP64 FMAs (n^2 per point at two lanes per SM and clock); each FMA needs two 8-byte
// shared-memory reads, a quarter of what shared memory delivers in that time, so elements are not
// blocked in registers.  CH4 / 6-31G / PBE (17 functions, 140,800 points): 5448 -> 122 us; 64 H2 (2
// functions, 51,200 points each), LDA: 2249 -> 147 us, before with one thread per element that looped
// over 2048 points in global memory.
template <int KIND>
__global__ void __launch_bounds__(kVxcThreads) k_vxc(VxcArgs v)
{
    extern __shared__ double sm[];
    const int m = blockIdx.z, n = v.mn[m];
    // tile pair: blockIdx.y = J (J + 1) / 2 + I, I <= J
    int J = 0;
    while ((J + 1) * (J + 2) / 2 <= (int)blockIdx.y) ++J;
    const int I = (int)blockIdx.y - J * (J + 1) / 2;
    const int i0 = I * kVxcTile, j0 = J * kVxcTile;
    const long long np_ = v.pbase[m + 1] - v.pbase[m];
    const long long c0 = (long long)blockIdx.x * v.chunk;
    if (j0 >= n || c0 >= np_) return;
    const long long c1 = min(np_, c0 + v.chunk);
    const int ni = min(kVxcTile, n - i0), nj = min(kVxcTile, n - j0);
    const int rows = I == J ? nj : ni + nj;             // staged functions: tile I, then (I != J) tile J
    const int rj = I == J ? 0 : ni;                     // first staged row of tile J
    const int nel = I == J ? nj * (nj + 1) / 2 : ni * nj;
    const int ngrp = max(1, kVxcThreads / nel);
    const int pitch = v.tp + 1;                         // odd (tp is even): lanes on different rows hit different banks
    double* sphi = sm;
    double* sa = sm + rows * pitch;
    const int grp = nel >= kVxcThreads ? 0 : (int)threadIdx.x / nel;
    const int e0 = nel >= kVxcThreads ? (int)threadIdx.x : (int)threadIdx.x % nel;
    int ri[kVxcMaxEl], rjj[kVxcMaxEl];
    double acc[kVxcMaxEl];
#pragma unroll
    for (int k = 0; k < kVxcMaxEl; ++k) {
        const int e = e0 + k * kVxcThreads;
        acc[k] = 0.0;
        ri[k] = rjj[k] = -1;
        if (e < nel && grp < ngrp) {
            if (I == J) {                               // e = j (j + 1) / 2 + i, i <= j
                int j = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
                while (j * (j + 1) / 2 > e) --j;
                while ((j + 1) * (j + 2) / 2 <= e) ++j;
                ri[k] = e - j * (j + 1) / 2;
                rjj[k] = j;
            } else {
                ri[k] = e / nj;
                rjj[k] = rj + e % nj;
            }
        }
    }
    const double* ph = v.phi + v.aobase[m];
    const double* dx = v.dphi + 3 * v.aobase[m];
    const double* dy = dx + np_ * n;
    const double* dz = dy + np_ * n;
    const long long gp = v.pbase[m];
    for (long long p0 = c0; p0 < c1; p0 += v.tp) {
        const int cnt = (int)min((long long)v.tp, c1 - p0);
        __syncthreads();
        for (int t = threadIdx.x; t < rows * v.tp; t += kVxcThreads) {
            const int r = t / v.tp, p = t % v.tp;
            double fv = 0.0, av = 0.0;
            if (p < cnt) {
                const long long at = (long long)(r < ni ? i0 + r : j0 + r - rj) * np_ + p0 + p;
                fv = ph[at];
                av = (KIND == 2 ? 0.5 : 1.0) * v.vrho[gp + p0 + p] * fv;
                if (KIND == 2) {
                    const double* g = v.vgrad + 3 * (gp + p0 + p);
                    av += g[0] * dx[at] + g[1] * dy[at] + g[2] * dz[at];
                }
            }
            sphi[r * pitch + p] = fv;
            sa[r * pitch + p] = av;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kVxcMaxEl; ++k) {
            if (ri[k] < 0) break;
            const double *fi = sphi + ri[k] * pitch, *fj = sphi + rjj[k] * pitch;
            const double *ai = sa + ri[k] * pitch, *aj = sa + rjj[k] * pitch;
            double s0 = 0.0, s1 = 0.0;
            for (int p = grp; p < cnt; p += ngrp) {
                s0 += ai[p] * fj[p];
                if (KIND == 2) s1 += fi[p] * aj[p];      // (LDA: the same as s0, in a)
            }
            acc[k] += s0 + s1;
        }
    }
    if (ngrp > 1) {                                     // sum the groups (at most one element per thread)
        __syncthreads();
        if (ri[0] >= 0) sm[grp * nel + e0] = acc[0];
        __syncthreads();
        if (grp == 0)
            for (int g = 1; g < ngrp; ++g) acc[0] += sm[g * nel + e0];
        else
            ri[0] = -1;
    }
#pragma unroll
    for (int k = 0; k < kVxcMaxEl; ++k) {
        if (ri[k] < 0) break;
        const int i = i0 + ri[k], j = j0 + rjj[k] - rj;
        atomicAdd(v.V + v.mbase[m] + (long long)i * n + j, acc[k]);
        if (i != j) atomicAdd(v.V + v.mbase[m] + (long long)j * n + i, acc[k]);
    }
}

}  // namespace

// ------------------------------------------------------------------------------------------ host
void mess_free_xc(mess_basis* b)
{
    XcState& x = b->xc;
    x.pts.free(); x.w.free(); x.atom.free(); x.atom_mol.free(); x.tab.free(); x.radial_at.free(); x.radial_n.free();
    x.abase.free(); x.pbase.free(); x.phi.free(); x.dphi.free();
    x.aobase.free(); x.vrho.free(); x.vgrad.free(); x.fbase.free(); x.shell_off.free(); x.shell_n.free();
    x.shell_fl.free();
    x.npts = 0;
    x.ready = false;
}

mess_status mess_xc_prepare(mess_basis* b, cudaStream_t s)
{
    XcState& X = b->xc;
    if (X.ready) return MESS_OK;
    // table of log_1p, angular table, then the radial grid of every element present
    std::vector<double> tab((size_t)kAngularTab);
    for (int i = 0; i < kLogBins; ++i) {
        const double c = i ? 1.0 / (1.0 + (i + 0.5) / kLogBins) : 1.0;
        tab[2 * i] = c;
        tab[2 * i + 1] = -log(c);
    }
    {
        std::vector<double> ct, wt;
        gauss_legendre(kNTheta, ct, wt);
        double* ang = tab.data() + kAngularAt;
        for (int t = 0; t < kNTheta; ++t) {
            ang[t] = ct[t];
            ang[kNTheta + t] = sqrt(1.0 - ct[t] * ct[t]);
            ang[2 * kNTheta + t] = wt[t];
        }
        for (int k = 0; k < kNPhi; ++k) {
            ang[3 * kNTheta + k] = cos(2.0 * M_PI * k / kNPhi);
            ang[3 * kNTheta + kNPhi + k] = sin(2.0 * M_PI * k / kNPhi);
        }
    }
    std::vector<int> at_of_z(128, -1), radial_at(b->natom), radial_n(b->natom), atom_mol(b->natom);
    std::vector<long long> pbase(1, 0), aobase, abase(b->natom);
    long long ao = 0, np = 0;
    for (int m = 0; m < b->nmol; ++m) {
        const long long start = np;
        for (int A = b->mol_atom_off[m]; A < b->mol_atom_off[m] + b->mol_atom_n[m]; ++A) {
            const int Z = b->Z[A], nr = Z == 1 ? 50 : kRadialMax;
            if (at_of_z[Z] < 0) {
                at_of_z[Z] = (int)tab.size();
                const double R = radius_of(Z) * kAngstrom;
                std::vector<double> rw;
                for (int i = 1; i <= nr; ++i) {
                    const double th = i * M_PI / (nr + 1);
                    const double xr = cos(th);
                    const double wx = M_PI / (nr + 1) * sin(th) * sin(th) / sqrt(1.0 - xr * xr);
                    const double r = R * (1.0 + xr) / (1.0 - xr);
                    tab.push_back(r);
                    rw.push_back(wx * r * r * 2.0 * R / ((1.0 - xr) * (1.0 - xr)));
                }
                tab.insert(tab.end(), rw.begin(), rw.end());
            }
            radial_at[A] = at_of_z[Z];
            radial_n[A] = nr;
            atom_mol[A] = m;
            abase[A] = np;
            np += (long long)nr * kAngular;
        }
        pbase.push_back(np);
        aobase.push_back(ao);
        ao += (np - start) * b->mol_nbf[m];
    }
    std::vector<int> fbase(b->nmol, 0), shell_fl;
    for (int m = 1; m < b->nmol; ++m) fbase[m] = fbase[m - 1] + b->mol_nbf[m - 1];
    for (const HostShell& sh : b->shells) shell_fl.push_back(sh.fl);
    X.npts = np;
    X.ao = ao;
    X.mol_npts_max = 0;
    for (int m = 0; m < b->nmol; ++m) X.mol_npts_max = std::max(X.mol_npts_max, pbase[m + 1] - pbase[m]);
    MESS_CUDA_TRY(X.tab.upload(tab));
    MESS_CUDA_TRY(X.radial_at.upload(radial_at));
    MESS_CUDA_TRY(X.radial_n.upload(radial_n));
    MESS_CUDA_TRY(X.atom_mol.upload(atom_mol));
    MESS_CUDA_TRY(X.abase.upload(abase));
    MESS_CUDA_TRY(X.pts.alloc((size_t)np * 3));
    MESS_CUDA_TRY(X.w.alloc((size_t)np));
    MESS_CUDA_TRY(X.atom.alloc((size_t)np));
    MESS_CUDA_TRY(X.pbase.upload(pbase));
    MESS_CUDA_TRY(X.aobase.upload(aobase));
    MESS_CUDA_TRY(X.fbase.upload(fbase));
    MESS_CUDA_TRY(X.shell_off.upload(b->mol_shell_off));
    MESS_CUDA_TRY(X.shell_n.upload(b->mol_shell_n));
    MESS_CUDA_TRY(X.shell_fl.upload(shell_fl));
    MESS_CUDA_TRY(X.phi.alloc((size_t)ao));
    MESS_CUDA_TRY(X.dphi.alloc((size_t)ao * 3));
    MESS_CUDA_TRY(X.vrho.alloc((size_t)X.npts));
    MESS_CUDA_TRY(X.vgrad.alloc((size_t)X.npts * 3));
    const int T = 256;
    const unsigned blocks = (unsigned)((X.npts + T - 1) / T);
    k_grid<<<(unsigned)(b->natom * kBlocksPerAtom), kGridThreads, 0, s>>>(X.tab.p, X.radial_at.p, X.radial_n.p, X.abase.p,
                                                                          b->d_xyz.p, X.pts.p, X.w.p, X.atom.p);
    MESS_CUDA_TRY(cudaGetLastError());
    GridArgs g{X.pts.p, X.w.p, X.atom.p, X.atom_mol.p, b->d_mol_atom_off.p, b->d_mol_atom_n.p, b->d_xyz.p, X.npts};
    k_becke<<<blocks, T, 0, s>>>(g);
    MESS_CUDA_TRY(cudaGetLastError());
    AoArgs a{X.pts.p, X.atom.p, X.atom_mol.p, X.npts, X.shell_off.p, X.shell_n.p, b->d_shell_l.p, b->d_shell_K.p, b->d_shell_poff.p,
             X.shell_fl.p, b->d_shell_R.p, b->d_shell_alpha.p, b->d_shell_coef.p, b->d_fscale.p, X.fbase.p, X.pbase.p,
             X.aobase.p, b->d_mol_n.p, X.phi.p, X.dphi.p};
    k_ao<<<blocks, T, 0, s>>>(a);
    MESS_CUDA_TRY(cudaGetLastError());
    X.ready = true;
    return MESS_OK;
}

mess_status mess_xc_eval(mess_basis* b, int kind, const double* dD, double* dV, double* dExc, cudaStream_t s)
{
    if (kind != 1 && kind != 2) { mess_set_error("exchange-correlation: unknown functional %d", kind); return MESS_EINVAL; }
    XcState& X = b->xc;
    if (!X.ready) { mess_set_error("exchange-correlation grid not prepared"); return MESS_EINVAL; }
    MESS_CUDA_TRY(cudaMemsetAsync(dExc, 0, sizeof(double) * b->nmol, s));
    MESS_CUDA_TRY(cudaMemsetAsync(dV, 0, sizeof(double) * b->packed, s));
    if (X.npts == 0) return MESS_OK;
    FuncArgs f{X.phi.p, X.dphi.p, dD, b->d_mol_base.p, X.pbase.p, X.aobase.p, b->d_mol_n.p, X.w.p, X.vrho.p, X.vgrad.p,
               reinterpret_cast<const double2*>(X.tab.p), dExc, dV, 1};
    // sixteen blocks per SM before a thread takes more points (fewer sums over a block's threads)
    f.ppt = (int)std::clamp<long long>(X.npts / (152LL * 16 * kFuncThreads), 1, 8);
    const dim3 fgrid((unsigned)((X.mol_npts_max + (long long)kFuncThreads * f.ppt - 1) / ((long long)kFuncThreads * f.ppt)), (unsigned)b->nmol);
    typedef void (*Kernel)(FuncArgs);
    static const Kernel kernels[2][kSmallN + 1] = {
        {k_functional<1, 0>, k_functional<1, 1>, k_functional<1, 2>, k_functional<1, 3>, k_functional<1, 4>},
        {k_functional<2, 0>, k_functional<2, 1>, k_functional<2, 2>, k_functional<2, 3>, k_functional<2, 4>}};
    const int small_n = b->max_nbf <= kSmallN ? b->max_nbf : 0;
    kernels[kind - 1][small_n]<<<fgrid, kFuncThreads, 0, s>>>(f);
    MESS_CUDA_TRY(cudaGetLastError());
    if (small_n) return MESS_OK;
    // V_xc: function tiles of the largest molecule; points staged per pass so that phi and a of the
    // staged functions take at most about 40 KB (16 to 256 points, fewer where functions are many);
    // about eight blocks per SM over all molecules and tile pairs, each with enough points to pay for
    // its atomics
    const int tiles = (b->max_nbf + kVxcTile - 1) / kVxcTile;
    const int rows = tiles > 1 ? 2 * kVxcTile : b->max_nbf;
    int tp = 256;
    while (tp > 16 && 2 * rows * (tp + 1) > 5120) tp /= 2;
    const long long want = std::max<long long>(1, X.npts * (tiles * (tiles + 1) / 2) / (152 * 8));
    const int chunk = (int)std::max<long long>(tp, std::min<long long>(2048, (want + tp - 1) / tp * tp));
    const size_t smem = sizeof(double) * (size_t)std::max(2 * rows * (tp + 1), kVxcThreads);
    VxcArgs v{X.phi.p, X.dphi.p, X.vrho.p, X.vgrad.p, X.pbase.p, X.aobase.p, b->d_mol_base.p, b->d_mol_n.p, chunk, tp, dV};
    const dim3 vgrid((unsigned)((X.mol_npts_max + chunk - 1) / chunk), (unsigned)(tiles * (tiles + 1) / 2), (unsigned)b->nmol);
    if (kind == 2) k_vxc<2><<<vgrid, kVxcThreads, smem, s>>>(v);
    else k_vxc<1><<<vgrid, kVxcThreads, smem, s>>>(v);
    MESS_CUDA_TRY(cudaGetLastError());
    return MESS_OK;
}

extern "C" mess_status mess_xc(const mess_basis* bc, int xc, const double* D, double* Exc, double* V, long long* npts)
{
    mess_basis* b = const_cast<mess_basis*>(bc);
    if (!b || !D) { mess_set_error("null argument"); return MESS_EINVAL; }
    if (xc != 1 && xc != 2) { mess_set_error("mess_xc: functional must be 1 (LDA) or 2 (PBE)"); return MESS_EINVAL; }
    { const mess_status gs = mess_basis_gpu(b); if (gs != MESS_OK) return gs; }
    mess_status st = mess_xc_prepare(b, 0);
    if (st != MESS_OK) return st;
    const size_t nn = (size_t)b->packed;
    DevBuf<double> d;
    MESS_CUDA_TRY(d.alloc(2 * nn + b->nmol));
    cudaError_t e = cudaMemcpy(d.p, D, nn * sizeof(double), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        st = mess_xc_eval(b, xc, d.p, d.p + nn, d.p + 2 * nn, 0);
        if (st == MESS_OK) {
            e = cudaDeviceSynchronize();
            if (e == cudaSuccess && V) e = cudaMemcpy(V, d.p + nn, nn * sizeof(double), cudaMemcpyDeviceToHost);
            if (e == cudaSuccess && Exc) e = cudaMemcpy(Exc, d.p + 2 * nn, b->nmol * sizeof(double), cudaMemcpyDeviceToHost);
        }
    }
    d.free();
    if (st != MESS_OK) return st;
    if (e != cudaSuccess) { mess_set_error("mess_xc: %s", cudaGetErrorString(e)); return MESS_ECUDA; }
    if (npts) *npts = b->xc.npts;
    return MESS_OK;
}
