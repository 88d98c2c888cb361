// One-electron integrals S, T, V over contracted Cartesian shells (Obara-Saika recursions), FP64.
//   overlap (1-D):  s_{i+1,j} = X_PA s_ij + (i s_{i-1,j} + j s_{i,j-1}) / (2p),
//                   s_{i,j+1} = X_PB s_ij + (i s_{i-1,j} + j s_{i,j-1}) / (2p),  s_00 = 1
//   kinetic:        T = 1/2 <grad a | grad b>, with d/dx (x_A^i e^{-a x_A^2}) = i x_A^{i-1} - 2a x_A^{i+1}
//   nuclear:        [e|0]^(m) by the VRR
//                   [e+1_i|0]^(m) = PA_i [e|0]^(m) - PC_i [e|0]^(m+1)
//                                   + e_i/(2p) ([e-1_i|0]^(m) - [e-1_i|0]^(m+1)),
//                   [0|0]^(m) = 2 pi/p exp(-ab/p |AB|^2) F_m(p |PC|^2), summed over the nuclei and
//                   the primitive pairs, then the HRR (a|b+1_i) = (a+1_i|b) + AB_i (a|b) once per shell pair.
//
// One warp per canonical shell pair writes both (m, n) and (n, m) blocks.  The work is V: one VRR per
// (primitive pair, nucleus), so the lanes split those, each with its own sums of [e|0] (la <= |e| <= la +
// lb) in registers; the recursion is unrolled for every class.  V reads the screened primitive pairs of
// the repulsion integrals (a dropped pair's weight is below MESS_PRIM_EPS of the heaviest); S and T
// take every primitive.  Bound: the FP64 pipe, about 40 (ss) to 300 (dd) instructions per primitive pair
// and nucleus.  (H2O)_32 / 6-31G* (52,000 pairs, 96 nuclei): 20.3 -> 1.29 ms; the
// 256 alkanes of an STO-3G batch: 23.5 -> 5.0 ms, before with one thread per shell pair.
#include <math.h>

#include <utility>

#include "mess_internal.h"

namespace {

constexpr int kPairsPerBlock = 4;   // warps per block

__host__ __device__ constexpr int n_cart(int l) { return (l + 1) * (l + 2) / 2; }

// component c of cart(L): x^i y^j z^k with i descending, then j descending
__host__ __device__ constexpr int comp_x(int L, int c)
{
    int x = L;
    while (c >= L - x + 1) { c -= L - x + 1; --x; }
    return x;
}
__host__ __device__ constexpr int comp_z(int L, int c)
{
    int x = L;
    while (c >= L - x + 1) { c -= L - x + 1; --x; }
    return c;
}
__host__ __device__ constexpr int comp(int L, int c, int d)
{
    return d == 0 ? comp_x(L, c) : (d == 2 ? comp_z(L, c) : L - comp_x(L, c) - comp_z(L, c));
}
__host__ __device__ constexpr int comp_id(int x, int y, int z) { return (y + z) * (y + z + 1) / 2 + z; }
// direction in which component c of cart(L) is lowered: one with exponent 1 if there is one (its
// recursion has no third term)
__host__ __device__ constexpr int low_dir(int L, int c)
{
    for (int d = 0; d < 3; ++d) if (comp(L, c, d) == 1) return d;
    for (int d = 0; d < 3; ++d) if (comp(L, c, d) > 0) return d;
    return 0;
}
__host__ __device__ constexpr int lowered(int L, int c, int d, int k)
{
    return comp_id(comp(L, c, 0) - (d == 0 ? k : 0), comp(L, c, 1) - (d == 1 ? k : 0), comp(L, c, 2) - (d == 2 ? k : 0));
}

// f(std::integral_constant<int, 0>) .. f(<N - 1>): loops whose index has to be a constant, so that every
// array in them stays in registers
template <class F, int... I> __device__ __forceinline__ void unrolled(F&& f, std::integer_sequence<int, I...>)
{
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F> __device__ __forceinline__ void unrolled(F&& f)
{
    unrolled(f, std::make_integer_sequence<int, N>{});
}

// offset of the sums of |e| = L within a lane's sums (which start at |e| = LA)
template <int LA> __host__ __device__ constexpr int sums_at(int L)
{
    int o = 0;
    for (int k = LA; k < L; ++k) o += n_cart(k);
    return o;
}

// one level of the VRR: cart(L) x (LAB - L + 1) values from the two levels below, added to the sums
// where L >= LA, then the next level
template <int LA, int LAB, int L> struct Vrr {
    static __device__ __forceinline__ void run(const double (&p1)[n_cart(L - 1)][LAB - L + 2],
                                               const double (&p2)[n_cart(L > 1 ? L - 2 : 0)][LAB - L + 3],
                                               const double (&PA)[3], const double (&PC)[3], double o2p,
                                               double (&sums)[sums_at<LA>(LAB + 1)])
    {
        double t[n_cart(L)][LAB - L + 1];
        unrolled<n_cart(L)>([&](auto ci) {
            constexpr int c = decltype(ci)::value, d = low_dir(L, c), c1 = lowered(L, c, d, 1), k = comp(L, c, d) - 1;
#pragma unroll
            for (int m = 0; m <= LAB - L; ++m) {
                double v = PA[d] * p1[c1][m] - PC[d] * p1[c1][m + 1];
                if constexpr (k > 0) {
                    constexpr int c2 = lowered(L, c, d, 2);
                    v += k * o2p * (p2[c2][m] - p2[c2][m + 1]);
                }
                t[c][m] = v;
            }
            if constexpr (L >= LA) sums[sums_at<LA>(L) + c] += t[c][0];
        });
        if constexpr (L < LAB) Vrr<LA, LAB, L + 1>::run(t, p1, PA, PC, o2p, sums);
    }
};

__host__ __device__ constexpr int binom(int n, int k) { return k == 0 || k == n ? 1 : (k == 1 ? n : n * (n - 1) / 2); }
template <int N> __device__ __forceinline__ double ipow(double x) { return N == 0 ? 1.0 : (N == 1 ? x : x * x); }

struct Seg { const int* list; int count, block0, la, lb; };   // pairs of one class and primitive group
constexpr int kMaxSeg = MESS_NLIST;

struct OneEArgs {
    Seg seg[kMaxSeg];
    int nseg;
    PairTable<double> P;
    const int *pair_a, *pair_b;   // shells of a pair
    const int *K, *f0, *poff;     // per shell: primitives, first (global) function, first primitive
    const double *alpha, *coef, *R, *fscale;
    const int* Z;
    const double* xyz;
    const int* atom_off;          // [nmol] first atom of the molecule
    const int* atom_n;            // [nmol] atoms of the molecule
    double *S, *T, *V;
};

// the (m, n) and (n, m) elements of a block from the lanes that own them: element k in lane k mod 32,
// its value in own[k / 32].  In the block of a shell with itself both orders of a pair of functions are there, as sums
// of the same terms in different orders: the lower triangle's gives both elements.
template <int NA, int NB, int NOWN>
__device__ __forceinline__ void store_block(double* __restrict__ M, const double (&own)[NOWN], const OneEArgs& s, int fa, int fb,
                                            int la0, int lb0, int n, int lane)
{
#pragma unroll
    for (int o = 0; o < NOWN; ++o) {
        const int k = lane + 32 * o;
        const int i = k / NB, j = k % NB;
        if (k < NA * NB && (fa != fb || i >= j)) {
            const double v = s.fscale[fa + i] * s.fscale[fb + j] * own[o];
            M[(size_t)(la0 + i) * n + lb0 + j] = v;
            M[(size_t)(lb0 + j) * n + la0 + i] = v;
        }
    }
}

template <int LA, int LB> __device__ __forceinline__ void one_e_pair(const OneEArgs& s, int pair, int lane)
{
    constexpr int NA = n_cart(LA), NB = n_cart(LB), LAB = LA + LB, NOWN = (NA * NB + 31) / 32;
    const int A = s.pair_a[pair], B = s.pair_b[pair];
    const double Rx[3] = {s.R[3 * A], s.R[3 * A + 1], s.R[3 * A + 2]};
    const double AB[3] = {s.P.AB[3 * pair], s.P.AB[3 * pair + 1], s.P.AB[3 * pair + 2]};
    const int fa = s.f0[A], fb = s.f0[B], la0 = s.P.fa[pair], lb0 = s.P.fb[pair];
    const int mol = s.P.mol[pair], n = s.P.mn[mol];
    const long long base = s.P.mbase[mol];
    if (s.V) {
        constexpr int NS = sums_at<LA>(LAB + 1);
        double sums[NS];
#pragma unroll
        for (int k = 0; k < NS; ++k) sums[k] = 0.0;
        const int at0 = s.atom_off[mol], na = s.atom_n[mol];
        const int items = s.P.pp_n[pair] * na, pp0 = s.P.pp_off[pair];
        int ip = lane / na, C = lane % na;
        const int dip = 32 / na, dC = 32 % na;
        for (int it = lane; it < items; it += 32) {
            const PrimPair<double> q = s.P.load(pp0 + ip);
            const double* X = s.xyz + 3 * (at0 + C);
            const double PA[3] = {q.PAx, q.PAy, q.PAz};
            const double PC[3] = {q.PAx + (Rx[0] - X[0]), q.PAy + (Rx[1] - X[1]), q.PAz + (Rx[2] - X[2])};
            // 2 pi/p c_a c_b exp(..) = K sqrt(2) pi^(-1/4), K the record's prefactor
            const double pre = -1.0622519320271969 * (double)s.Z[at0 + C] * q.K;
            double t0[1][LAB + 1];
            boys_eval<double, LAB, 0>(q.zeta * (PC[0] * PC[0] + PC[1] * PC[1] + PC[2] * PC[2]), pre, t0[0], s.P);
            if (LA == 0) sums[0] += t0[0][0];
            if constexpr (LAB > 0) {
                double none[1][LAB + 2];
                Vrr<LA, LAB, 1>::run(t0, none, PA, PC, q.oo2z, sums);
            }
            ip += dip;
            C += dC;
            if (C >= na) { C -= na; ++ip; }
        }
#pragma unroll
        for (int k = 0; k < NS; ++k) sums[k] = warp_sum(sums[k]);
        double own[NOWN] = {};
        unrolled<NA * NB>([&](auto ki) {
            // (a|b) = sum_t C(b, t) AB^(b - t) (a + t|0), t over the (bx + 1)(by + 1)(bz + 1) shifts
            constexpr int k = decltype(ki)::value, i = k / NB, j = k % NB;
            constexpr int bx = comp(LB, j, 0), by = comp(LB, j, 1), bz = comp(LB, j, 2);
            double v = 0.0;
            unrolled<(bx + 1) * (by + 1) * (bz + 1)>([&](auto ti) {
                constexpr int t = decltype(ti)::value;
                constexpr int tz = t % (bz + 1), ty = t / (bz + 1) % (by + 1), tx = t / (bz + 1) / (by + 1);
                constexpr int at = sums_at<LA>(LA + tx + ty + tz)
                                   + comp_id(comp(LA, i, 0) + tx, comp(LA, i, 1) + ty, comp(LA, i, 2) + tz);
                v += binom(bx, tx) * binom(by, ty) * binom(bz, tz) * ipow<bx - tx>(AB[0]) * ipow<by - ty>(AB[1])
                     * ipow<bz - tz>(AB[2]) * sums[at];
            });
            if (lane == k % 32) own[k / 32] = v;
        });
        store_block<NA, NB>(s.V + base, own, s, fa, fb, la0, lb0, n, lane);
    }
    if (!s.S && !s.T) return;
    const double ab2 = AB[0] * AB[0] + AB[1] * AB[1] + AB[2] * AB[2];
    const int KB = s.K[B], nprim = s.K[A] * KB;
    double ownS[NOWN], ownT[NOWN];
#pragma unroll
    for (int o = 0; o < NOWN; ++o) ownS[o] = ownT[o] = 0.0;
    for (int q0 = 0; q0 < nprim; q0 += 32) {            // 32 primitive pairs at a time, one per lane
        const int q = min(q0 + lane, nprim - 1);
        const double a = s.alpha[s.poff[A] + q / KB], b = s.alpha[s.poff[B] + q % KB];
        const double c = q0 + lane < nprim ? s.coef[s.poff[A] + q / KB] * s.coef[s.poff[B] + q % KB] : 0.0;
        const double rp = 1.0 / (a + b), o2p = 0.5 * rp;
        const double u = M_PI * rp;
        const double s00 = c * u * sqrt(u) * exp(-a * b * rp * ab2);
        double s1[3][LA + 2][LB + 2];                   // 1-D overlaps, i <= la + 1, j <= lb + 1
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            const double PA = -b * rp * AB[x], PB = a * rp * AB[x];
#pragma unroll
            for (int i = 0; i <= LA + 1; ++i)
#pragma unroll
                for (int j = 0; j <= LB + 1; ++j) {
                    double v = 1.0;
                    if (i > 0) {
                        v = PA * s1[x][i - 1][j];
                        if (i > 1) v += (i - 1) * o2p * s1[x][i > 1 ? i - 2 : 0][j];
                        if (j > 0) v += j * o2p * s1[x][i - 1][j > 0 ? j - 1 : 0];
                    } else if (j > 0) {
                        v = PB * s1[x][0][j - 1];
                        if (j > 1) v += (j - 1) * o2p * s1[x][0][j > 1 ? j - 2 : 0];
                    }
                    s1[x][i][j] = v;
                }
        }
        const double ab4 = 4.0 * a * b, a2 = 2.0 * a, b2 = 2.0 * b;
        unrolled<NA * NB>([&](auto ki) {
            constexpr int k = decltype(ki)::value, i = k / NB, j = k % NB;
            double sx[3], dx[3];
            unrolled<3>([&](auto xi) {
                constexpr int x = decltype(xi)::value, e = comp(LA, i, x), f = comp(LB, j, x);
                sx[x] = s1[x][e][f];
                double g = ab4 * s1[x][e + 1][f + 1];
                if constexpr (e > 0) g -= b2 * e * s1[x][e - 1][f + 1];
                if constexpr (f > 0) g -= a2 * f * s1[x][e + 1][f - 1];
                if constexpr (e > 0 && f > 0) g += (double)(e * f) * s1[x][e - 1][f - 1];
                dx[x] = g;
            });
            const double vS = warp_sum(s00 * sx[0] * sx[1] * sx[2]);
            const double vT = warp_sum(0.5 * s00 * (dx[0] * sx[1] * sx[2] + sx[0] * (dx[1] * sx[2] + sx[1] * dx[2])));
            if (lane == k % 32) {
                ownS[k / 32] += vS;
                ownT[k / 32] += vT;
            }
        });
    }
    if (s.S) store_block<NA, NB>(s.S + base, ownS, s, fa, fb, la0, lb0, n, lane);
    if (s.T) store_block<NA, NB>(s.T + base, ownT, s, fa, fb, la0, lb0, n, lane);
}

__global__ void __launch_bounds__(32 * kPairsPerBlock) k_one_e(const __grid_constant__ OneEArgs s)
{
    int g = 0;
    while (g + 1 < s.nseg && s.seg[g + 1].block0 <= (int)blockIdx.x) ++g;
    const int t = ((int)blockIdx.x - s.seg[g].block0) * kPairsPerBlock + (int)(threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (t >= s.seg[g].count) return;
    const int pair = s.seg[g].list[t];
    switch (s.seg[g].la * 3 + s.seg[g].lb) {
    case 0: one_e_pair<0, 0>(s, pair, lane); break;
    case 3: one_e_pair<1, 0>(s, pair, lane); break;
    case 4: one_e_pair<1, 1>(s, pair, lane); break;
    case 6: one_e_pair<2, 0>(s, pair, lane); break;
    case 7: one_e_pair<2, 1>(s, pair, lane); break;
    default: one_e_pair<2, 2>(s, pair, lane); break;
    }
}

}  // namespace

cudaError_t mess_launch_one_e(const mess_basis* b, double* dS, double* dT, double* dV, cudaStream_t st)
{
    static const int cls[MESS_NUM_PCLASS][2] = {{0, 0}, {1, 0}, {1, 1}, {2, 0}, {2, 1}, {2, 2}};
    OneEArgs s{};
    int blocks = 0;
    // the longest pairs first: dd to ss, many primitives to few
    for (int c = MESS_NUM_PCLASS - 1; c >= 0; --c)
        for (int g = 2 * MESS_NGROUP - 1; g >= 0; --g) {
            const DevBuf<int>& l = b->d_class_list[MESS_LIST(g / MESS_NGROUP, c, g % MESS_NGROUP)];
            if (l.n == 0) continue;
            s.seg[s.nseg++] = Seg{l.p, (int)l.n, blocks, cls[c][0], cls[c][1]};
            blocks += ((int)l.n + kPairsPerBlock - 1) / kPairsPerBlock;
        }
    if (blocks == 0) return cudaSuccess;
    s.P = b->P64;
    s.pair_a = b->d_pair_a.p; s.pair_b = b->d_pair_b.p;
    s.K = b->d_shell_K.p; s.f0 = b->d_shell_f0.p; s.poff = b->d_shell_poff.p;
    s.alpha = b->d_shell_alpha.p; s.coef = b->d_shell_coef.p; s.R = b->d_shell_R.p; s.fscale = b->d_fscale.p;
    s.Z = b->d_Z.p; s.xyz = b->d_xyz.p;
    s.atom_off = b->d_mol_atom_off.p; s.atom_n = b->d_mol_atom_n.p;
    s.S = dS; s.T = dT; s.V = dV;
    k_one_e<<<blocks, 32 * kPairsPerBlock, 0, st>>>(s);
    return cudaGetLastError();
}
