// Device-side building blocks shared by the generated per-class ERI code and the kernels:
// primitive-pair tables, the Boys function F_m(T), and J/K accumulation helpers.
#pragma once
#include <type_traits>
#include <cuda_runtime.h>
#include <stdint.h>

#include "df32.cuh"
#include "mess_device.h"

// ------------------------------------------------------------------------------------------
// Primitive-pair record (Gaussian product theorem): for primitives alpha on A, beta on B,
//   zeta = alpha + beta,  P = (alpha A + beta B)/zeta,  PA = P - A,
//   K = sqrt(2) pi^{5/4} c_a c_b exp(-alpha beta/zeta |AB|^2) / zeta   (so that K_ab K_cd / sqrt(zeta+eta)
//       is the 2 pi^{5/2}/(zeta eta sqrt(zeta+eta)) prefactor of [00|00]^(m)),
//   oo2z = 1/(2 zeta).
// ------------------------------------------------------------------------------------------
template <typename R> struct PrimPair { R zeta, PAx, PAy, PAz, K, oo2z; };

template <typename R> struct PairTable;

// Conversions between FP64 and FP32 done on the integer ALU: on this GPU the FP64 pipe (which also
// executes F2F / I2F conversions) runs at 1/64 of the FP32 rate, so FP32 kernels avoid it entirely,
// including in rarely taken branches (the compiler predicates them, and a predicated-off FP64-pipe
// instruction still issues).  d2f: round to nearest with ties away from zero, results below 2^-126
// flush to signed zero, overflow and infinities give signed infinity, NaN stays NaN.  f2d: exact; FP32 subnormals flush to zero.
__device__ __forceinline__ float d2f_alu(double d)
{
    const unsigned long long o = (unsigned long long)__double_as_longlong(d);
    const unsigned long long b = o + (1ull << 28);
    const unsigned ohi = (unsigned)(o >> 32);
    const unsigned sign = ohi & 0x80000000u;
    const unsigned hi = (unsigned)(b >> 32);
    const int fe = (int)((hi >> 20) & 0x7ffu) - 896;
    const unsigned mant = (unsigned)((b >> 29) & 0x7fffffu);
    unsigned bits = sign | ((unsigned)fe << 23) | mant;
    bits = fe <= 0 ? sign : bits;
    bits = fe >= 255 ? (sign | 0x7f800000u) : bits;
    bits = ((ohi >> 20) & 0x7ffu) == 0x7ffu ? (sign | 0x7f800000u | ((o << 12) ? 0x400000u : 0u)) : bits;
    return __uint_as_float(bits);
}

__device__ __forceinline__ double f2d_alu(float f)
{
    const unsigned u = __float_as_uint(f);
    const unsigned e = (u >> 23) & 0xffu;
    const unsigned m = u & 0x7fffffu;
    const unsigned sign = u & 0x80000000u;
    unsigned hi = sign | ((e + 896u) << 20) | (m >> 3);
    hi = e == 0u ? sign : hi;
    hi = e == 0xffu ? (sign | 0x7ff00000u | (m >> 3)) : hi;
    const unsigned lo = (e == 0u) ? 0u : (m << 29);
    return __hiloint2double((int)hi, (int)lo);
}

// small non-negative integer to float without I2F: 2^23 + k as bits, minus 2^23 (0 <= k < 2^22)
__device__ __forceinline__ float int_to_f32_alu(int k) { return __int_as_float(0x4B000000 | k) - 8388608.0f; }

template <typename R> __device__ __forceinline__ R small_int(int k);
template <> __device__ __forceinline__ double small_int<double>(int k) { return (double)k; }
template <> __device__ __forceinline__ float small_int<float>(int k) { return int_to_f32_alu(k); }
template <> __device__ __forceinline__ df32 small_int<df32>(int k) { return df32(int_to_f32_alu(k), 0.f); }

// a generated per-integral scale (double with float hi / lo copies) in R
template <typename R> __device__ __forceinline__ R gen_scale(const double* d, const float* hi, const float* lo, int k);
template <> __device__ __forceinline__ double gen_scale<double>(const double* d, const float*, const float*, int k) { return __ldg(d + k); }
template <> __device__ __forceinline__ float gen_scale<float>(const double*, const float* hi, const float*, int k) { return __ldg(hi + k); }
template <> __device__ __forceinline__ df32 gen_scale<df32>(const double*, const float* hi, const float* lo, int k)
{ return df32(__ldg(hi + k), __ldg(lo + k)); }

// double -> double-float: hi rounded to nearest, lo the rounded remainder (one FP64 subtraction)
__device__ __forceinline__ df32::df32(double v)
{
    hi = d2f_alu(v);
    lo = d2f_alu(v - f2d_alu(hi));
}

// density elements: the FP32 and double-float kernels read copies of D converted once per build
__device__ __forceinline__ double ldD(const double* p) { return __ldg(p); }
__device__ __forceinline__ float ldD(const float* p) { return __ldg(p); }
__device__ __forceinline__ df32 ldD(const float2* p) { const float2 v = __ldg(p); return df32(v.x, v.y); }
__device__ __forceinline__ double to_f64(double v) { return v; }
__device__ __forceinline__ double to_f64(float v) { return f2d_alu(v); }
__device__ __forceinline__ double to_f64(df32 v) { return f2d_alu(v.hi) + f2d_alu(v.lo); }

template <typename R> struct PairTable {
    const PrimPairRec<R>* __restrict__ pp;   // [npp]
    const int* __restrict__ pp_off;          // [npair]
    const int* __restrict__ pp_n;            // [npair]
    const double* __restrict__ AB;           // [npair][3]  A - B
    const int* __restrict__ fa;              // [npair] first function of A
    const int* __restrict__ fb;              // [npair] first function of B
    const int* __restrict__ same;            // [npair] 1 if A == B (same shell)
    const double* __restrict__ C;            // [npair][3] centre of the pair's first shell A
    const float* __restrict__ Cf;            // [npair][6] the same as FP32 hi[3], lo[3] (C = hi + lo)
    const float* __restrict__ ABf;           // [npair][3] A - B in FP32
    const int* __restrict__ mol;             // [npair] molecule of the pair (batched bases)
    const long long* __restrict__ mbase;     // [nmol] offset of the molecule's n x n block (packed matrices)
    const int* __restrict__ mn;              // [nmol] basis functions of the molecule (row stride)
    const double* __restrict__ boys64;       // FP64 Boys rows per order L (mess_device.h)
    const float4* __restrict__ boys32v;      // FP32 rows per order L: [L][row] {F_L, F_L+1, F_L+2 / 2, exp(-T_k)}; L = 0: F_3 / 6 last
    const float4* __restrict__ boysdf;       // double-float rows per order L
    // per molecule: 0 = left the computation (a converged molecule of a batched SCF): its quartets
    // are skipped by the J/K kernels.  Null: every molecule takes part.
    const unsigned char* __restrict__ active = nullptr;
    // Density-weighted screening of a build (null dmax: none): a shell quartet is skipped when
    // Q_ab Q_cd max(dmax_ab, dmax_cd) < dtau, with dmax_p the largest |D_mn| over the rows m of the
    // two shells of pair p.  Every density element a quartet's J/K terms read lies in one of those
    // rows, so each skipped contribution is below dtau (the incremental Fock builds of an SCF, whose
    // density changes shrink as it converges).
    const KetRec* __restrict__ rec = nullptr;   // per pair (pair order)
    const float* __restrict__ Qf = nullptr;     // Schwarz factor per pair (FP32)
    const float* __restrict__ dmax = nullptr;
    float dtau = 0.f;

    __device__ __forceinline__ bool live(int pair) const { return !active || __ldg(active + __ldg(mol + pair)) != 0; }
    __device__ __forceinline__ bool dens_ok(int bp, int kp) const
    {
        return !dmax || __ldg(Qf + bp) * __ldg(Qf + kp) * fmaxf(__ldg(dmax + bp), __ldg(dmax + kp)) >= dtau;
    }

    __device__ __forceinline__ PrimPair<R> load(int i) const
    {
        const PrimPairRec<R>& r = pp[i];
        PrimPair<R> o;
        o.zeta = r.v[0]; o.PAx = r.v[1]; o.PAy = r.v[2]; o.PAz = r.v[3];
        o.K = r.v[4]; o.oo2z = r.v[5];
        return o;
    }
};

// A - C between the first shells of two pairs, and A - B of one pair, in R.  FP32 forms the
// difference from hi/lo parts, so it is accurate relative to |A - C|, not to |A|.
__device__ __forceinline__ double pair_ac(const PairTable<double>& P, int bp, int kp, int x)
{
    return P.C[3 * bp + x] - P.C[3 * kp + x];
}
__device__ __forceinline__ float pair_ac(const PairTable<float>& P, int bp, int kp, int x)
{
    return (__ldg(P.Cf + 6 * bp + x) - __ldg(P.Cf + 6 * kp + x)) + (__ldg(P.Cf + 6 * bp + 3 + x) - __ldg(P.Cf + 6 * kp + 3 + x));
}
__device__ __forceinline__ df32 pair_ac(const PairTable<df32>& P, int bp, int kp, int x)
{
    const df32 h = df_two_sum(__ldg(P.Cf + 6 * bp + x), -__ldg(P.Cf + 6 * kp + x));
    const df32 l = df_two_sum(__ldg(P.Cf + 6 * bp + 3 + x), -__ldg(P.Cf + 6 * kp + 3 + x));
    return h + l;
}
__device__ __forceinline__ double pair_ab(const PairTable<double>& P, int p, int x) { return P.AB[3 * p + x]; }
__device__ __forceinline__ df32 pair_ab(const PairTable<df32>& P, int p, int x) { return df32(P.AB[3 * p + x]); }
__device__ __forceinline__ float pair_ab(const PairTable<float>& P, int p, int x) { return __ldg(P.ABf + 3 * p + x); }

// The ket side of a quartet as the recursion needs it: its primitive range, A - C (bra first centre
// minus ket first centre, formed as in pair_ac) and C - D, from the ket's record.
template <typename R> struct KetView {
    int k0, nk;
    R AC[3], CD[3];
};

__device__ __forceinline__ int4 ket_hdr(const KetRec* r) { return __ldg(reinterpret_cast<const int4*>(r)); }

__device__ __forceinline__ KetView<double> ket_view(const PairTable<double>& P, int bp, const KetRec* r, int4 h)
{
    KetView<double> v;
    v.k0 = h.x;
    v.nk = h.y;
    const double2 c01 = __ldg(reinterpret_cast<const double2*>(r) + 1);
    const double2 c2a0 = __ldg(reinterpret_cast<const double2*>(r) + 2);
    const double2 a12 = __ldg(reinterpret_cast<const double2*>(r) + 3);
    v.AC[0] = __ldg(P.C + 3 * bp) - c01.x;
    v.AC[1] = __ldg(P.C + 3 * bp + 1) - c01.y;
    v.AC[2] = __ldg(P.C + 3 * bp + 2) - c2a0.x;
    v.CD[0] = c2a0.y; v.CD[1] = a12.x; v.CD[2] = a12.y;
    return v;
}
__device__ __forceinline__ KetView<float> ket_view(const PairTable<float>& P, int bp, const KetRec* r, int4 h)
{
    KetView<float> v;
    v.k0 = h.x;
    v.nk = h.y;
    const float4 f0 = __ldg(reinterpret_cast<const float4*>(r) + 4);   // Cf hi x y z, lo x
    const float4 f1 = __ldg(reinterpret_cast<const float4*>(r) + 5);   // lo y z, ABf x y
    const float4 f2 = __ldg(reinterpret_cast<const float4*>(r) + 6);   // ABf z, pair
    const float* cb = P.Cf + 6 * bp;
    v.AC[0] = (__ldg(cb) - f0.x) + (__ldg(cb + 3) - f0.w);
    v.AC[1] = (__ldg(cb + 1) - f0.y) + (__ldg(cb + 4) - f1.x);
    v.AC[2] = (__ldg(cb + 2) - f0.z) + (__ldg(cb + 5) - f1.y);
    v.CD[0] = f1.z; v.CD[1] = f1.w; v.CD[2] = f2.x;
    return v;
}
__device__ __forceinline__ KetView<df32> ket_view(const PairTable<df32>& P, int bp, const KetRec* r, int4 h)
{
    KetView<df32> v;
    v.k0 = h.x;
    v.nk = h.y;
    const float4 f0 = __ldg(reinterpret_cast<const float4*>(r) + 4);
    const float4 f1 = __ldg(reinterpret_cast<const float4*>(r) + 5);
    const float* cb = P.Cf + 6 * bp;
    const float kh[3] = {f0.x, f0.y, f0.z}, kl[3] = {f0.w, f1.x, f1.y};
#pragma unroll
    for (int x = 0; x < 3; ++x) {
        const df32 hi = df_two_sum(__ldg(cb + x), -kh[x]);
        const df32 lo = df_two_sum(__ldg(cb + 3 + x), -kl[x]);
        v.AC[x] = hi + lo;
    }
    const double2 c2a0 = __ldg(reinterpret_cast<const double2*>(r) + 2);
    const double2 a12 = __ldg(reinterpret_cast<const double2*>(r) + 3);
    v.CD[0] = df32(c2a0.y); v.CD[1] = df32(a12.x); v.CD[2] = df32(a12.y);
    return v;
}
__device__ __forceinline__ int ket_pair(const KetRec* r) { return __ldg(&r->pair); }

// ------------------------------------------------------------------------------------------
// Boys function F_m(T) = int_0^1 t^{2m} exp(-T t^2) dt, m = 0..L, times a factor (the primitive
// quartet's prefactor).
//   small T: Taylor expansion about the nearest grid point, F_n(T) = sum_j F_{n+j}(T_k) x^j / j!,
//            x = T_k - T, for the highest order L, then the stable downward recursion
//            F_{m-1} = (2 T F_m + exp(-T)) / (2m - 1);
//   large T: F_0 = (1/2) sqrt(pi/T) (erf(sqrt T) = 1 to working precision there) and the upward
//            recursion F_{m+1} = ((2m+1) F_m - exp(-T)) / (2T), stable for large T.
// The FP64 and double-float forms are bound by instruction count (an FP64 instruction takes 16 cycles of
// an SM, a double-float operation 7 to 11 instructions), so the grids are fine and their rows hold the
// Taylor coefficients themselves: 13 FP64 instructions before the recursion, where a step of 0.1 and
// plain values took 30; 130 FP32 instructions instead of 420 in double-float.
// BMODE 0: everything in FP64.  BMODE 1: FP64 for T < MESS_BOYS_TMAXDF (small-T Taylor + downward
// recursion), FP32 asymptote above it.  BMODE 2: everything in FP32.
// ------------------------------------------------------------------------------------------
template <int L> __device__ __forceinline__ void boys_small_f64(double T, double pref, double* F, const double* __restrict__ tab)
{
    // nearest grid index without conversion instructions (they run on the FP64 pipe): adding 1.5 * 2^52
    // rounds 32 T to an integer held in the low mantissa bits
    const double r = fma(T, MESS_BOYS64_INV_DT, 6755399441055744.0);
    const int k = __double2loint(r);
    const double x = fma(r - 6755399441055744.0, 1.0 / MESS_BOYS64_INV_DT, -T);
    const double2* row = reinterpret_cast<const double2*>(tab) + (size_t)(L * MESS_BOYS64_NROW + k) * 4;
    const double2 a = __ldg(row), b = __ldg(row + 1), c = __ldg(row + 2), d = __ldg(row + 3);
    const double s = a.x + x * (a.y + x * (b.x + x * (b.y + x * (c.x + x * (c.y + x * d.x)))));
    F[L] = pref * s;
    if (L == 0) return;
    // exp(-T) = exp(-T_k) exp(x) (|x| <= 1/64)
    const double ex = 1.0 + x * (1.0 + x * (1.0 / 2 + x * (1.0 / 6 + x * (1.0 / 24 + x * (1.0 / 120 + x * (1.0 / 720))))));
    const double e = pref * d.y * ex;
    const double t2 = 2.0 * T;
#pragma unroll
    for (int m = L; m >= 1; --m) F[m - 1] = m == 1 ? t2 * F[m] + e : (t2 * F[m] + e) * (1.0 / (2 * m - 1));
}

// T >= MESS_BOYS_TMAX64: exp(-T) is below 2e-21 there and enters F_8 (4e-11) at 5e-13 of its value, so
// an FP32 exponential carries it
template <int L> __device__ __forceinline__ void boys_large_f64(double T, double pref, double* F)
{
    const double rt = rsqrt(T);
    F[0] = 0.886226925452758014 * rt * pref;   // sqrt(pi)/2 / sqrt(T)
    if (L > 0) {
        const double e = (double)__expf(-(float)T) * pref;
        const double h = 0.5 * rt * rt;
#pragma unroll
        for (int m = 0; m < L; ++m) F[m + 1] = ((2 * m + 1) * F[m] - e) * h;
    }
}

template <int L> __device__ __forceinline__ void boys_large_f32(float T, float* F)
{
    const float rt = rsqrt_ftz(T);
    F[0] = 0.886226925f * rt;
    if (L > 0) {
        const float e = __expf(-T);
        const float h = 0.5f * rt * rt;
#pragma unroll
        for (int m = 0; m < L; ++m) F[m + 1] = ((2 * m + 1) * F[m] - e) * h;
    }
}

// v c for a constant c that FP32 does not hold: rounded, 1/3 or sqrt(pi)/2 would move every integral to the same side, and
// J and K sum that up.  (hi and lo are compile-time constants: one multiplication more.)
__device__ __forceinline__ float mul_const(float v, double c)
{
    const float hi = (float)c, lo = (float)(c - (double)hi);
    return fmaf(v, hi, v * lo);
}

// FP32.  The lanes of a warp lie on both sides of the grid's end, and the two sides of a branch would run one after
// the other: the asymptote is formed for every lane and replaced below the end.  It leaves out exp(-T), at most 1e-8 of 2 T F_L
// at the end: T = 30 up to L = 5, 36 above (the asymptote, one root, carries fewer roundings than the recursion).
// For L <= 1 the lanes above it skip the rest, since the gather of rows fills the L1 data
// pipe there (95 % for (ss|ss)); for the longer recursions the selection is 1 to 8 % faster.  Instructions, not
// loads, bound those, so a row holds what order 2 at a step of 1/128 needs (three FMAs, where order 4 at 1/16
// took the upward recursion for two of its terms and a division).
// Batch of 256 alkanes / STO-3G, per three builds: (ps|ss) 15.9 -> 12.6 ms, (ps|ps) 6.7 -> 5.8, (pp|ss) 3.3 -> 2.6,
// (ss|ss) 10.8 -> 10.3; (H2O)_32 / 6-31G*, (ss|ss) 894 -> 733 us, (ps|ss) 1349 -> 1253.
// Error of J and K of mixed builds against FP64, as a share of the error with the rows at 1/16 (24 geometries and densities
// each): with the constants rounded and every end at 36, (H2O)_8 / 6-31G* 1.02 and 1.03, C7H16 / 6-31G 0.99 and 1.04;
// as here 0.74 and 0.99, 0.93 and 1.03 (0.74 and 0.96, 0.93 and 0.95 with the lanes' sums rounded once, lane_sum).
// Times of the builds and the batch within 0.6 % of each other.
template <int L> __device__ __forceinline__ void boys_f32(float T, float* F, const float4* __restrict__ tabv)
{
    const bool far = !(T < (L <= 5 ? (float)MESS_BOYS_TMAX32_L5 : (float)MESS_BOYS_TMAX32));
    const float rt = rsqrt_ftz(T), h = 0.5f * rt * rt;
    F[0] = mul_const(rt, 0.886226925452758014);   // sqrt(pi)/2 / sqrt(T)
#pragma unroll
    for (int m = 0; m < L; ++m) F[m + 1] = F[m] * ((float)(2 * m + 1) * h);
    if (L <= 1 && far) return;
    const float Tc = fminf(T, (float)MESS_BOYS_TMAX32);
    // nearest grid index without F2I / I2F conversions (those issue on the slow FP64 pipe): adding
    // 1.5 * 2^23 rounds T / dT to an integer held in the low mantissa bits (0 <= T / dT < 2^22)
    constexpr float inv_dt = L > 0 ? (float)MESS_BOYS32_INV_DT : (float)MESS_BOYS32_INV_DT0;
    const float r = fmaf(Tc, inv_dt, 12582912.0f);
    const int k = __float_as_int(r) - 0x4B400000;
    const float x = fmaf(r - 12582912.0f, 1.0f / inv_dt, -Tc);    // T_k - T (exact)
    const float4 a = __ldg(tabv + (size_t)L * MESS_BOYS32_NROW + k);
    float d = fmaf(x, fmaf(x, L > 0 ? a.z : fmaf(x, a.w, a.z), a.y), a.x);
    F[L] = far ? F[L] : d;
    if (L == 0) return;
    // exp(-T) = exp(-T_k) exp(x), exp(x) to third order (the next term is below 1e-11)
    const float e = a.w * fmaf(x, fmaf(x, fmaf(x, 1.0f / 6, 0.5f), 1.0f), 1.0f);
    const float t2 = 2.0f * T;
#pragma unroll
    for (int m = L; m >= 1; --m) {
        d = fmaf(t2, d, e);
        if (m > 1) d = mul_const(d, 1.0 / (2 * m - 1));
        F[m - 1] = far ? F[m - 1] : d;
    }
}

// double-float Boys: the same scheme; terms too small to need it are FP32.  Above the grid F_0 =
// sqrt(pi)/2 T^-1/2 and the upward recursion, whose exp(-T) term (below 3e-16 there) is FP32.
__device__ __forceinline__ df32 df_inv_int(int j)   // 1/j as double-float
{
    const float h = 1.0f / (float)j;
    return df32(h, fmaf(-h, (float)j, 1.0f) / (float)j);
}

template <int L> __device__ __forceinline__ void boys_small_df(df32 T, df32 pref, df32* F, const float4* __restrict__ tab)
{
    const float r = fmaf(T.hi, (float)MESS_BOYSDF_INV_DT, 12582912.0f);
    const int k = __float_as_int(r) - 0x4B400000;
    // T_k - T.hi is exact (T_k is a short number within 1/128 of T.hi)
    const float xh = (r - 12582912.0f) * (1.0f / (float)MESS_BOYSDF_INV_DT) - T.hi;
    const df32 x = df_fast_two_sum(xh, -T.lo);
    const float4* row = tab + (size_t)(L * MESS_BOYSDF_NROW + k) * 3;
    const float4 a = __ldg(row), b = __ldg(row + 1), c = __ldg(row + 2);
    df32 s = df_fast_two_sum(b.z, fmaf(x.hi, fmaf(x.hi, c.y, c.x), b.w));
    s = df_add_smaller(df32(b.x, b.y), x * s);
    s = df_add_smaller(df32(a.z, a.w), x * s);
    s = df_add_smaller(df32(a.x, a.y), x * s);
    F[L] = pref * s;
    if (L == 0) return;
    // exp(x) = 1 + x + x^2/2 + x^3/6 in double-float, x^4/24 + x^5/120 (below 2e-10) in FP32
    const df32 x2 = x * x, h2 = df32(0.5f * x2.hi, 0.5f * x2.lo);
    df32 u = df_inv_int(6) * x;
    u.lo = fmaf(x2.hi, fmaf(x.hi, 1.0f / 120, 1.0f / 24), u.lo);
    u = df_add_smaller(h2, x2 * df_fast_two_sum(u.hi, u.lo));
    u = df_add_smaller(x, u);
    const df32 e = pref * (df32(c.z, c.w) * df_add_smaller(df32(1.0f, 0.f), u));
    const df32 t2 = df32(2.0f * T.hi, 2.0f * T.lo);
#pragma unroll
    for (int m = L; m >= 1; --m) F[m - 1] = m == 1 ? t2 * F[m] + e : (t2 * F[m] + e) * df_inv_int(2 * m - 1);
}

template <int L> __device__ __forceinline__ void boys_large_df(df32 T, df32 pref, df32* F)
{
    const df32 rt = df_rsqrt(T);
    F[0] = df32(0.8862269520759583f, -2.6623199644859596e-08f) * rt * pref;   // sqrt(pi)/2 = 0.88622692545275801 as hi + lo
    if (L > 0) {
        const df32 e = df32(__expf(-T.hi), 0.f) * pref;
        df32 h = rt * rt;
        h = df32(0.5f * h.hi, 0.5f * h.lo);
#pragma unroll
        for (int m = 0; m < L; ++m) F[m + 1] = (df32((float)(2 * m + 1), 0.f) * F[m] - e) * h;
    }
}

// F_0..F_L times pref
template <typename R, int L, int BMODE> struct BoysEval;
template <int L> struct BoysEval<double, L, 0> {
    static __device__ __forceinline__ void run(double T, double pref, double* F, const PairTable<double>& P)
    { if (T < MESS_BOYS_TMAX64) boys_small_f64<L>(T, pref, F, P.boys64); else boys_large_f64<L>(T, pref, F); }
};
template <int L> struct BoysEval<float, L, 1> {
    static __device__ __forceinline__ void run(float T, float pref, float* F, const PairTable<float>& P)
    {
        if (T < (float)MESS_BOYS_TMAXDF) {
            double Fd[L + 1];
            boys_small_f64<L>((double)T, 1.0, Fd, P.boys64);
#pragma unroll
            for (int m = 0; m <= L; ++m) F[m] = (float)Fd[m];
        } else {
            boys_large_f32<L>(T, F);
        }
#pragma unroll
        for (int m = 0; m <= L; ++m) F[m] *= pref;
    }
};
template <int L> struct BoysEval<float, L, 2> {
    static __device__ __forceinline__ void run(float T, float pref, float* F, const PairTable<float>& P)
    {
        boys_f32<L>(T, F, P.boys32v);
#pragma unroll
        for (int m = 0; m <= L; ++m) F[m] *= pref;
    }
};
template <int L> struct BoysEval<df32, L, 3> {
    static __device__ __forceinline__ void run(df32 T, df32 pref, df32* F, const PairTable<df32>& P)
    { if (T < MESS_BOYS_TMAXDF) boys_small_df<L>(T, pref, F, P.boysdf); else boys_large_df<L>(T, pref, F); }
};
template <typename R, int L, int BMODE>
__device__ __forceinline__ void boys_eval(R T, R pref, R* F, const PairTable<R>& P) { BoysEval<R, L, BMODE>::run(T, pref, F, P); }

// 1/(zeta + eta) and its square root (the prefactor's 1/sqrt(zeta + eta)): one reciprocal square root and
// its square, instead of a division and a root (FP64: 8 instructions of the FP64 pipe instead of about 20)
__device__ __forceinline__ void recip_and_sqrt(double s, double& rz, double& sq) { sq = rsqrt(s); rz = sq * sq; }
__device__ __forceinline__ void recip_and_sqrt(float s, float& rz, float& sq) { sq = rsqrt_ftz(s); rz = sq * sq; }
__device__ __forceinline__ void recip_and_sqrt(df32 s, df32& rz, df32& sq) { sq = df_rsqrt(s); rz = sq * sq; }

// primitive loops of the straight-line FP32 kernels run two primitive quartets per iteration (more
// independent loads in flight); FP64 and double-float keep one (register pressure)
template <typename R> struct PrimUnroll { static constexpr int value = 1; };
template <> struct PrimUnroll<float> { static constexpr int value = 2; };


// ------------------------------------------------------------------------------------------
// J/K accumulation.  For a unique shell quartet (ab|cd) (pair ab >= pair cd, a >= b, c >= d by
// the canonical pair order) with degeneracy weight s = (1/2)^{[a=b] + [c=d] + [ab=cd]}:
//   Jacc_ab += s sum_cd I D_cd,   Jacc_cd += s sum_ab I D_ab,
//   Kacc_ac += s sum_bd I D_bd,   Kacc_ad += s sum_bc I D_bc,
//   Kacc_bc += s sum_ad I D_ad,   Kacc_bd += s sum_ac I D_ac,
// and afterwards J = 2 (Jacc + Jacc^T), K = Kacc + Kacc^T.  This visits each of the 8 index
// permutations of every function quartet exactly once for a symmetric D.
// ------------------------------------------------------------------------------------------
template <typename R> struct DigestCtx {
    const typename DElem<R>::T* __restrict__ D;
    double* __restrict__ J;
    double* __restrict__ K;
    int n;
    int fa, fb, fc, fd;
    bool warp_reduce_ab;   // all 32 lanes share the bra pair: reduce J_ab across the warp first
};

__device__ __forceinline__ float shfl_xor(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ double shfl_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ df32 shfl_xor(df32 v, int o) { return df_shfl_xor(v, o); }

// a + b of two lanes, and the rounding of a whole sum.  FP32 values are summed as hi + lo and rounded once: log2 G roundings
// at the size of the sum move K more than a lane's whole chain of primitives does.  Error of K of C7H16 / 6-31G below
// the split, all classes with 32 lanes, 2.85e-10 -> 2.44e-10 (8 lanes 2.85 -> 2.51, 4 lanes 2.78 -> 2.52, one thread 2.57);
// mixed builds take 0 to 0.7 % longer.
__device__ __forceinline__ df32 lane_sum(float a, float b) { return df_two_sum(a, b); }
__device__ __forceinline__ df32 lane_sum(df32 a, df32 b) { return a + b; }
__device__ __forceinline__ double lane_sum(double a, double b) { return a + b; }
__device__ __forceinline__ void lane_store(float& x, float v) { x = v; }
__device__ __forceinline__ void lane_store(float& x, df32 v) { x = v.hi + v.lo; }
__device__ __forceinline__ void lane_store(df32& x, df32 v) { x = v; }
__device__ __forceinline__ void lane_store(double& x, double v) { x = v; }

// Sums of acc[0..N) over the G lanes of a group into the group's shared array sh.  Each halving of the
// group also halves what a lane carries on (it keeps one half and sends the other), so the whole costs
// about N additions per lane; an all-lanes butterfly of every value takes N log2 G.
template <int O, int N> struct GroupSums {
    template <typename R, typename S> static __device__ __forceinline__ void run(const R (&acc)[N], int g, int off, int len, S* sh)
    {
        constexpr int H = (N + 1) / 2;
        const bool up = (g & O) != 0;
        decltype(lane_sum(acc[0], acc[0])) t[H];
#pragma unroll
        for (int k = 0; k < H; ++k) {
            const R lo = acc[k], hi = k + H < N ? acc[k + H < N ? k + H : 0] : R(0);
            t[k] = lane_sum(up ? hi : lo, shfl_xor(up ? lo : hi, O));
        }
        GroupSums<O / 2, H>::run(t, g, up ? off + H : off, up ? max(len - H, 0) : min(len, H), sh);
    }
};
template <int N> struct GroupSums<0, N> {
    template <typename R, typename S> static __device__ __forceinline__ void run(const R (&acc)[N], int, int off, int len, S* sh)
    {
#pragma unroll
        for (int k = 0; k < N; ++k)
            if (k < len) lane_store(sh[off + k], acc[k]);
    }
};

template <typename R> __device__ __forceinline__ R warp_sum(R v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += shfl_xor(v, o);
    return v;
}

template <typename R>
__device__ __forceinline__ void jk_add(double* __restrict__ M, size_t idx, R v, bool warp_reduce)
{
    if (warp_reduce) {
        v = warp_sum(v);
        if ((threadIdx.x & 31) == 0) atomicAdd(M + idx, to_f64(v));
    } else {
        if (v != R(0)) atomicAdd(M + idx, to_f64(v));
    }
}
__device__ __forceinline__ void jk_add(double* __restrict__ M, size_t idx, df32u v, bool warp_reduce)
{
    jk_add<df32>(M, idx, v, warp_reduce);
}

// ------------------------------------------------------------------------------------------
// Work decomposition of one class bin: bra pairs i (sorted by Q descending), each with a
// contiguous ket range [kbeg[i], kbeg[i] + offs[i+1] - offs[i]) of the ket list.  A flat quartet
// index q maps to (i, j) by a binary search over offs.
// ------------------------------------------------------------------------------------------
// the largest i < n with offs[i] <= q, searched between the entries of seg for q / 32 and q / 32 + 1 (a
// few steps instead of a search over all)
__device__ __forceinline__ int find_segment(const int* __restrict__ seg, const long long* __restrict__ offs, int n,
                                            long long total, long long q)
{
    const long long k = q >> 5;
    int lo = __ldg(seg + k);
    int hi = ((k + 1) << 5) < total ? __ldg(seg + k + 1) : n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(offs + mid) <= q) lo = mid; else hi = mid - 1;
    }
    return lo;
}
// bra of flat quartet q
__device__ __forceinline__ int find_bra(const BinLaunch& b, long long q) { return find_segment(b.seg, b.offs, b.nbra, b.total, q); }

__device__ __forceinline__ bool warp_uniform_int(int v)
{
    const int v0 = __shfl_sync(0xffffffffu, v, 0);
    return __all_sync(0xffffffffu, v == v0);
}

#define MESS_THREADS 128

// Digestion of one quartet by TW threads (this one `lane`): the outputs are dealt out, the integrals are
// read from shared memory.
template <typename R, int TW, int NA, int NB, int NC, int ND>
__device__ __forceinline__ void team_digest(const R* I, const DigestCtx<R>& x, R s, int lane)
{
    const typename DElem<R>::T* __restrict__ D = x.D;
    double* __restrict__ J = x.J;
    double* __restrict__ K = x.K;
    const size_t nn = (size_t)x.n;
    const int fa = x.fa, fb = x.fb, fc = x.fc, fd = x.fd;
#define MESS_I(a_, b_, c_, d_) I[(((a_) * NB + (b_)) * NC + (c_)) * ND + (d_)]
    for (int o = lane; o < NA * NB; o += TW) {          // J_ab = sum_cd I D_cd
        const int a = o / NB, bb = o % NB;
        R t = R(0);
        for (int c = 0; c < NC; ++c)
            for (int d = 0; d < ND; ++d) t += MESS_I(a, bb, c, d) * ldD(D + (fc + c) * nn + fd + d);
        atomicAdd(J + (fa + a) * nn + fb + bb, to_f64(s * t));
    }
    for (int o = lane; o < NC * ND; o += TW) {          // J_cd = sum_ab I D_ab
        const int c = o / ND, d = o % ND;
        R t = R(0);
        for (int a = 0; a < NA; ++a)
            for (int bb = 0; bb < NB; ++bb) t += MESS_I(a, bb, c, d) * ldD(D + (fa + a) * nn + fb + bb);
        atomicAdd(J + (fc + c) * nn + fd + d, to_f64(s * t));
    }
    for (int o = lane; o < NA * NC; o += TW) {          // K_ac = sum_bd I D_bd
        const int a = o / NC, c = o % NC;
        R t = R(0);
        for (int bb = 0; bb < NB; ++bb)
            for (int d = 0; d < ND; ++d) t += MESS_I(a, bb, c, d) * ldD(D + (fb + bb) * nn + fd + d);
        atomicAdd(K + (fa + a) * nn + fc + c, to_f64(s * t));
    }
    for (int o = lane; o < NA * ND; o += TW) {          // K_ad = sum_bc I D_bc
        const int a = o / ND, d = o % ND;
        R t = R(0);
        for (int bb = 0; bb < NB; ++bb)
            for (int c = 0; c < NC; ++c) t += MESS_I(a, bb, c, d) * ldD(D + (fb + bb) * nn + fc + c);
        atomicAdd(K + (fa + a) * nn + fd + d, to_f64(s * t));
    }
    for (int o = lane; o < NB * NC; o += TW) {          // K_bc = sum_ad I D_ad
        const int bb = o / NC, c = o % NC;
        R t = R(0);
        for (int a = 0; a < NA; ++a)
            for (int d = 0; d < ND; ++d) t += MESS_I(a, bb, c, d) * ldD(D + (fa + a) * nn + fd + d);
        atomicAdd(K + (fb + bb) * nn + fc + c, to_f64(s * t));
    }
    for (int o = lane; o < NB * ND; o += TW) {          // K_bd = sum_ac I D_ac
        const int bb = o / ND, d = o % ND;
        R t = R(0);
        for (int a = 0; a < NA; ++a)
            for (int c = 0; c < NC; ++c) t += MESS_I(a, bb, c, d) * ldD(D + (fa + a) * nn + fc + c);
        atomicAdd(K + (fb + bb) * nn + fd + d, to_f64(s * t));
    }
#undef MESS_I
}

// Lanes that share a quartet (G > 1) also share its digestion, through shared memory, where that costs
// fewer instructions than one lane digesting from registers while the others wait: always in FP64 and
// double-float (16 cycles or 7 to 11 instructions per operation against about five of addressing and
// loads), in FP32 from 8 lanes on.
template <typename R, int G> constexpr bool shared_digest() { return G > 1 && (sizeof(R) == 8 || G >= 8); }
// shared memory of a group, in elements: its sums, then its integrals; odd, so that groups start in
// different banks
constexpr int group_pitch(int nacc, int nint) { return (nacc > nint ? nacc : nint) | 1; }

// JK kernel of one class: G consecutive lanes per shell quartet of the bin (G = 1: one thread).
#define MESS_DEFINE_CLASS_KERNELS(TAG, NA, NB, NC, ND, NACC)                                       \
    template <typename R, int BMODE, int G>                                                         \
    __global__ void __launch_bounds__(MESS_THREADS)                                                 \
    k_jk_##TAG(const BinLaunch b, const PairTable<R> P, const typename DElem<R>::T* __restrict__ D,            \
               double* __restrict__ J, double* __restrict__ K, int n)                               \
    {                                                                                               \
        constexpr int NINT_ = (NA) * (NB) * (NC) * (ND), PITCH_ = group_pitch(NACC, NINT_);         \
        __shared__ __align__(16) unsigned char sh_[G > 1 ? MESS_THREADS / G * PITCH_ * sizeof(R) : 16]; \
        R* sh = reinterpret_cast<R*>(sh_) + (G > 1 ? (int)threadIdx.x / G * PITCH_ : 0);            \
        const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;                     \
        const long long q0 = t0 / G;                                                                \
        const int g = (int)(t0 % G);                                                                \
        const bool valid = q0 < b.total;                                                            \
        const long long q = valid ? q0 : b.total - 1;                                               \
        const int i = find_bra(b, q);                                                  \
        const int j = __ldg(b.kbeg + i) + (int)(q - __ldg(b.offs + i));                            \
        const int bp = __ldg(b.bra + i);                                                            \
        const KetRec* kr = b.ketrec + j;                                                            \
        const int4 kh = ket_hdr(kr);                                                                \
        const int kp = ket_pair(kr);                                                                \
        /* quartets past the end or of a molecule that has left: no work; a warp without any    */ \
        /* quartet to do leaves (lanes of a group share the quartet, so groups leave together)  */ \
        const bool live = valid && P.live(bp) && P.dens_ok(bp, kp);                                 \
        if (__all_sync(0xffffffffu, !live)) return;                                                 \
        R I[NINT_];                                                                                 \
        eri_##TAG<R, BMODE, G>(P, bp, ket_view(P, bp, kr, kh), g, I, live, sh);                    \
        DigestCtx<R> c;                                                                              \
        {                                                                                           \
            const int m_ = __ldg(P.mol + bp);                                                       \
            const long long o_ = __ldg(P.mbase + m_);                                               \
            c.D = D + o_; c.J = J + o_; c.K = K + o_; c.n = __ldg(P.mn + m_);                       \
        }                                                                                           \
        (void)n;                                                                                    \
        c.fa = __ldg(P.fa + bp); c.fb = __ldg(P.fb + bp);                                           \
        c.fc = kh.z & 0xffff; c.fd = kh.z >> 16;                                                    \
        R s = live ? R(1) : R(0);                                                                   \
        if (__ldg(P.same + bp)) s *= R(0.5);                                                        \
        if (kh.w & 1) s *= R(0.5);                                                                  \
        if (bp == kp) s *= R(0.5);                                                                  \
        if (G == 1) {                                                                               \
            c.warp_reduce_ab = warp_uniform_int(bp);                                                \
            digest_##TAG<R>(I, c, s);                                                               \
        } else if constexpr (shared_digest<R, G>()) {                                               \
            _Pragma("unroll") for (int k = 0; k < NINT_; ++k)                                       \
                if (k % G == g) sh[k] = I[k];                                                       \
            __syncwarp();                                                                           \
            if (live) team_digest<R, G, NA, NB, NC, ND>(sh, c, s, g);                               \
        } else if (g == 0) {                                                                        \
            c.warp_reduce_ab = false;                                                               \
            digest_##TAG<R>(I, c, s);                                                               \
        }                                                                                           \
    }                                                                                               \
    /* every integral of the bin written to a dense n^4 tensor, all 8 index permutations */         \
    __global__ void __launch_bounds__(MESS_THREADS)                                                 \
    k_store_##TAG(const BinLaunch b, const PairTable<double> P, double* __restrict__ G, int n)      \
    {                                                                                               \
        const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;                      \
        if (q >= b.total) return;                                                                   \
        const int i = find_bra(b, q);                                                  \
        const int j = b.kbeg[i] + (int)(q - b.offs[i]);                                             \
        const int bp = b.bra[i], kp = b.ket[j];                                                     \
        double I[(NA) * (NB) * (NC) * (ND)];                                                        \
        eri_##TAG<double, 0, 1>(P, bp, ket_view(P, bp, P.rec + kp, ket_hdr(P.rec + kp)), 0, I);     \
        const int fa = P.fa[bp], fb = P.fb[bp], fc = P.fa[kp], fd = P.fb[kp];                       \
        const size_t nn = (size_t)n;                                                                \
        for (int ia = 0; ia < (NA); ++ia)                                                           \
            for (int ib = 0; ib < (NB); ++ib)                                                       \
                for (int ic = 0; ic < (NC); ++ic)                                                   \
                    for (int id = 0; id < (ND); ++id) {                                             \
                        const double v = I[((ia * (NB) + ib) * (NC) + ic) * (ND) + id];             \
                        const size_t a = fa + ia, bb = fb + ib, c = fc + ic, d = fd + id;           \
                        G[((a * nn + bb) * nn + c) * nn + d] = v;                                   \
                        G[((bb * nn + a) * nn + c) * nn + d] = v;                                   \
                        G[((a * nn + bb) * nn + d) * nn + c] = v;                                   \
                        G[((bb * nn + a) * nn + d) * nn + c] = v;                                   \
                        G[((c * nn + d) * nn + a) * nn + bb] = v;                                   \
                        G[((d * nn + c) * nn + a) * nn + bb] = v;                                   \
                        G[((c * nn + d) * nn + bb) * nn + a] = v;                                   \
                        G[((d * nn + c) * nn + bb) * nn + a] = v;                                   \
                    }                                                                               \
    }

// hi + lo += v (error-free sum of the leading parts)
__device__ __forceinline__ void sum_exact(df32& acc, float v)
{
    const df32 t = df_two_sum(acc.hi, v);
    acc.hi = t.hi;
    acc.lo += t.lo;
}
__device__ __forceinline__ void flush_exact(double* __restrict__ M, size_t idx, df32 v)
{
    if (v.hi != 0.f || v.lo != 0.f) atomicAdd(M + idx, f2d_alu(v.hi) + f2d_alu(v.lo));
}

// FP32 J/K kernel of one class over bra runs: one thread takes a ket cd through up to MESS_RUN_MAX bras
// ab, ab', ... with the same first shell a.  J_cd, K_ac and K_ad then go to memory once per run instead of
// once per quartet (summed exactly in hi + lo FP32 pairs), D_cd, D_ac and D_ad are loaded once, and so is
// the ket.  Per quartet there remain K_bc, K_bd and the warp's sum for J_ab.  The one-thread-per-quartet
// kernels are bound by exactly that traffic (FP64 reductions at 110 to 140 G sectors/s, 60 to 70 % of the
// L1 and L2 throughput).  (H2O)_32 / 6-31G*, launches one at a time: (ps|ss) 2.70 -> 1.36 ms,
// (ds|ps) 1.78 -> 0.75, (ds|ss) 1.45 -> 0.69, (ps|ps) 1.36 -> 0.61, all J/K kernels 21.6 -> 16.7.
#define MESS_DEFINE_RUN_KERNEL(TAG, NA, NB, NC, ND)                                                 \
    __global__ void __launch_bounds__(MESS_THREADS)                                                 \
    k_jk_run_##TAG(const BinLaunch b, const RunLaunch r, const PairTable<float> P, const float* __restrict__ D, \
                   double* __restrict__ J, double* __restrict__ K)                                  \
    {                                                                                               \
        const long long q0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;                     \
        const bool valid = q0 < r.total;                                                            \
        const long long q = valid ? q0 : r.total - 1;                                               \
        const int i = find_segment(r.seg, r.offs, r.nrun, r.total, q);                              \
        const int4 run = __ldg(r.run + i);                                                          \
        const int j = run.z + (int)(q - __ldg(r.offs + i));                                         \
        const KetRec* kr = b.ketrec + j;                                                            \
        const int4 kh = ket_hdr(kr);                                                                \
        const int kp = ket_pair(kr);                                                                \
        const int bp0 = __ldg(b.bra + run.x);                                                       \
        const bool live = valid && P.live(bp0);                                                     \
        if (__all_sync(0xffffffffu, !live)) return;                                                 \
        const KetView<float> kv = ket_view(P, bp0, kr, kh);   /* (A is the run's) */                \
        const int m_ = __ldg(P.mol + bp0);                                                          \
        const long long o_ = __ldg(P.mbase + m_);                                                   \
        RunCtx<NA, NC, ND> c;                                                                       \
        c.D = D + o_; c.J = J + o_; c.K = K + o_; c.n = __ldg(P.mn + m_);                           \
        c.fa = __ldg(P.fa + bp0); c.fc = kh.z & 0xffff; c.fd = kh.z >> 16;                          \
        c.uniform = warp_uniform_int(i);                                                            \
        c.load();                                                                                   \
        const int nb = c.uniform ? run.y : __reduce_max_sync(0xffffffffu, run.y);                   \
        _Pragma("unroll 1") for (int t = 0; t < nb; ++t) {                                          \
            const int bi = run.x + min(t, run.y - 1);                                               \
            const int k0 = __ldg(b.kbeg + bi), bp = __ldg(b.bra + bi);                              \
            const int k1 = k0 + (int)(__ldg(b.offs + bi + 1) - __ldg(b.offs + bi));                 \
            const bool act = live && t < run.y && j >= k0 && j < k1 && P.dens_ok(bp, kp);           \
            if (!__any_sync(0xffffffffu, act)) continue;                                            \
            float I[(NA) * (NB) * (NC) * (ND)];                                                     \
            eri_##TAG<float, 2, 1>(P, bp, kv, 0, I, act);                                           \
            float s = act ? 1.0f : 0.0f;                                                            \
            if (__ldg(P.same + bp)) s *= 0.5f;                                                      \
            if (kh.w & 1) s *= 0.5f;                                                                \
            if (bp == kp) s *= 0.5f;                                                                \
            digest_run_##TAG(I, c, s, __ldg(P.fb + bp));                                            \
        }                                                                                           \
        c.flush();                                                                                  \
    }

// what a thread of a run keeps: the density blocks and sums that do not depend on b
template <int NA, int NC, int ND> struct RunCtx {
    const float* __restrict__ D;
    double* __restrict__ J;
    double* __restrict__ K;
    int n, fa, fc, fd;
    bool uniform;            // every lane of the warp is in the same run: reduce J_ab across the warp
    float Dcd[NC * ND], Dac[NA * NC], Dad[NA * ND];
    df32 Jcd[NC * ND], Kac[NA * NC], Kad[NA * ND];

    __device__ __forceinline__ void load()
    {
        block<NC, ND>(Dcd, Jcd, fc, fd);
        block<NA, NC>(Dac, Kac, fa, fc);
        block<NA, ND>(Dad, Kad, fa, fd);
    }
    __device__ __forceinline__ void flush() const
    {
        store<NC, ND>(J, Jcd, fc, fd);
        store<NA, NC>(K, Kac, fa, fc);
        store<NA, ND>(K, Kad, fa, fd);
    }
private:
    template <int M, int N> __device__ __forceinline__ void block(float* d, df32* sum, int r0, int c0)
    {
#pragma unroll
        for (int i = 0; i < M; ++i)
#pragma unroll
            for (int j = 0; j < N; ++j) {
                d[i * N + j] = ldD(D + (size_t)(r0 + i) * n + c0 + j);
                sum[i * N + j] = df32(0.f, 0.f);
            }
    }
    template <int M, int N> __device__ __forceinline__ void store(double* X, const df32* sum, int r0, int c0) const
    {
#pragma unroll
        for (int i = 0; i < M; ++i)
#pragma unroll
            for (int j = 0; j < N; ++j) flush_exact(X, (size_t)(r0 + i) * n + c0 + j, sum[i * N + j]);
    }
};

// Schwarz factors Q_ab = sqrt(max_{m in a, n in b} |(mn|mn)|) for a list of pairs of one class, G lanes
// per pair: the primitive quartets of a diagonal quartet number the square of the pair's primitive
// pairs (81 in STO-3G, up to 1296 in 6-31G*), so one thread per pair leaves a small molecule waiting for
// one serial loop.  Lane counts: see schwarz_lanes.  C2H6 / 6-31G's derivative basis, one thread per pair
// (pp|pp) 13.4 -> 0.43 ms, (ss|ss) 2.1 -> 0.07 ms.
#define MESS_DEFINE_SCHWARZ_KERNEL(TAG, NA, NB, NACC)                                              \
    template <int G>                                                                                \
    __global__ void __launch_bounds__(MESS_THREADS)                                                 \
    k_schwarz_##TAG(const int* __restrict__ pairs, int npairs, const PairTable<double> P,           \
                    double* __restrict__ Q)                                                         \
    {                                                                                               \
        constexpr int PITCH_ = group_pitch(NACC, 0);                                                \
        __shared__ double sh[G > 1 ? MESS_THREADS / G * PITCH_ : 1];                                \
        const int t = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) / G);               \
        const int g = (int)(threadIdx.x % G);                                                       \
        if (__all_sync(0xffffffffu, t >= npairs)) return;                                           \
        const int p = pairs[min(t, npairs - 1)];                                                    \
        double I[(NA) * (NB) * (NA) * (NB)];                                                        \
        eri_##TAG<double, 0, G>(P, p, ket_view(P, p, P.rec + p, ket_hdr(P.rec + p)), g, I, t < npairs, \
                               sh + (G > 1 ? (int)threadIdx.x / G * PITCH_ : 0));                   \
        double m = 0.0;                                                                             \
        for (int ia = 0; ia < (NA); ++ia)                                                           \
            for (int ib = 0; ib < (NB); ++ib)                                                       \
                m = fmax(m, fabs(I[((ia * (NB) + ib) * (NA) + ia) * (NB) + ib]));                   \
        if (t < npairs && g == 0) Q[p] = sqrt(m);                                                   \
    }

// ------------------------------------------------------------------------------------------
// Op-program evaluation of one shell quartet (large angular classes).  The program is the same
// VRR / HRR sequence as the straight-line code, with values packed into NV / NH slots:
//   VRR op (uint4): x = kind | dir<<2 | m1<<4 | m2<<8 | target<<16, y = s1 | s2<<16,
//                   z = s3 | s4<<16, w = s5
//     kind 0: V[t] = F[s1] (base [00|00]^(m), prefactor included)
//     kind 1: V[t] = PA_d V[s1] + WP_d V[s2] + m1/(2 zeta) (V[s3] - rho/zeta V[s4])
//     kind 2: V[t] = QC_d V[s1] + WQ_d V[s2] + m1/(2 eta) (V[s3] - rho/eta V[s4])
//                    + m2/(2(zeta+eta)) V[s5]
//     kind 3: H[s1] += V[t]  (contraction into [e0|f0])
//   HRR op (uint2): x = target | dir<<16 | side<<18, y = s1 | s2<<16:
//     H[t] = H[s1] + X_d H[s2],  X = A - B (side 0) or C - D (side 1)
//   I[k] = fscale[k] * H[fslot[k]]  (per-component normalisation)
// Every thread runs the same op sequence, so the kind / direction branches are warp-uniform.
// ------------------------------------------------------------------------------------------
template <typename R> __device__ __forceinline__ R pick3(int d, R x, R y, R z)
{
    return d == 0 ? x : (d == 1 ? y : z);
}

template <typename R, int BMODE, int L, int NV, int NH, int NACC, int NVOPS, int NHOPS, int NINT>
__device__ __forceinline__ void eri_program(const PairTable<R>& P, int bp, const KetView<R>& kv,
                                            const uint4* __restrict__ vprog, const uint2* __restrict__ hprog,
                                            const int* __restrict__ fslot, const double* __restrict__ fscale,
                                            const float* __restrict__ fscale_hi, const float* __restrict__ fscale_lo,
                                            R* I, bool live)
{
    R V[NV];
    R H[NH];
#pragma unroll 1
    for (int k = 0; k < NACC; ++k) H[k] = R(0);
    const int b0 = P.pp_off[bp], b1 = b0 + (live ? P.pp_n[bp] : 0);
    const int k0 = kv.k0, k1 = k0 + kv.nk;
    const R ACx = kv.AC[0], ACy = kv.AC[1], ACz = kv.AC[2];
    // ket primitives outside (per-lane records read once), bra primitives inside (the same for the warp)
#pragma unroll 1
    for (int ik = k0; ik < (live ? k1 : k0); ++ik) {
        const PrimPair<R> pk = P.load(ik);
#pragma unroll 1
        for (int ib = b0; ib < b1; ++ib) {
            const PrimPair<R> pb = P.load(ib);
            R rz, srz;
            recip_and_sqrt(pb.zeta + pk.zeta, rz, srz);
            const R roz = pk.zeta * rz, roe = pb.zeta * rz, oo2ze = R(0.5) * rz;
            const R PQx = pb.PAx - pk.PAx + ACx, PQy = pb.PAy - pk.PAy + ACy, PQz = pb.PAz - pk.PAz + ACz;
            const R WPx = -roz * PQx, WPy = -roz * PQy, WPz = -roz * PQz;
            const R WQx = roe * PQx, WQy = roe * PQy, WQz = roe * PQz;
            const R T = pb.zeta * roz * (PQx * PQx + PQy * PQy + PQz * PQz);
            const R pref = pb.K * pk.K * srz;
            R F[L + 1];
            boys_eval<R, L, BMODE>(T, pref, F, P);
#pragma unroll 1
            for (int o = 0; o < NVOPS; ++o) {
                const uint4 w = __ldg(vprog + o);
                const int kind = w.x & 3, d = (w.x >> 2) & 3;
                const int m1 = (w.x >> 4) & 15, m2 = (w.x >> 8) & 15, t = w.x >> 16;
                const int s1 = w.y & 0xffff, s2 = w.y >> 16;
                if (kind == 0) {
                    R f = F[0];
#pragma unroll
                    for (int m = 1; m <= L; ++m) f = (s1 == m) ? F[m] : f;
                    V[t] = f;
                } else if (kind == 3) {
                    H[s1] += V[t];
                } else {
                    R v;
                    if (kind == 1) {
                        v = pick3(d, pb.PAx, pb.PAy, pb.PAz) * V[s1] + pick3(d, WPx, WPy, WPz) * V[s2];
                        if (m1) v += small_int<R>(m1) * pb.oo2z * (V[w.z & 0xffff] - roz * V[w.z >> 16]);
                    } else {
                        v = pick3(d, pk.PAx, pk.PAy, pk.PAz) * V[s1] + pick3(d, WQx, WQy, WQz) * V[s2];
                        if (m1) v += small_int<R>(m1) * pk.oo2z * (V[w.z & 0xffff] - roe * V[w.z >> 16]);
                        if (m2) v += small_int<R>(m2) * oo2ze * V[w.w];
                    }
                    V[t] = v;
                }
            }
        }
    }
    const R ABx = pair_ab(P, bp, 0), ABy = pair_ab(P, bp, 1), ABz = pair_ab(P, bp, 2);
    const R CDx = kv.CD[0], CDy = kv.CD[1], CDz = kv.CD[2];
#pragma unroll 1
    for (int o = 0; o < NHOPS; ++o) {
        const uint2 w = __ldg(hprog + o);
        const int t = w.x & 0xffff, d = (w.x >> 16) & 3, side = (w.x >> 18) & 1;
        const R X = side ? pick3(d, CDx, CDy, CDz) : pick3(d, ABx, ABy, ABz);
        H[t] = H[w.y & 0xffff] + X * H[w.y >> 16];
    }
#pragma unroll 1
    for (int k = 0; k < NINT; ++k) I[k] = gen_scale<R>(fscale, fscale_hi, fscale_lo, k) * H[__ldg(fslot + k)];
}


// ------------------------------------------------------------------------------------------
// Warp-per-quartet J/K kernel for the large classes: the 32 lanes of a warp run the independent
// ops of one dependency level of the level-scheduled program in parallel (values in shared
// memory, __syncwarp between levels), then split the digestion outputs between them.
// ------------------------------------------------------------------------------------------

// TW threads share one shell quartet: 32 (a warp, MESS_TEAM_WARPS quartets per block) or
// 32 * MESS_TEAM_WARPS (the whole block on one quartet, for parts with very few quartets)
template <int TW> __device__ __forceinline__ void team_sync()
{
    if (TW == 32) __syncwarp();
    else __syncthreads();
}

// PS (with TW = the block): the block's warps split the quartet's primitive quartets, each warp
// accumulating into its own copy of the contracted values, summed before the HRR.
// Evaluates the quartet (bra pair bp, ket view kv) with its TW threads and leaves its integrals in the
// returned shared-memory array (synchronised).
template <typename R, int BMODE, int TW, int PS, int L, int NVI, int NH, int NACC, int NVL, int NHL, int NINT,
          int NA, int NB, int NC, int ND>
__device__ __forceinline__ const R* team_eri(const PairTable<R>& P, int bp, const KetView<R>& kv,
                                             const uint4* __restrict__ vprog, const int* __restrict__ vlev,
                                             const uint2* __restrict__ hprog, const int* __restrict__ hlev,
                                             const int* __restrict__ fslot, const double* __restrict__ fscale,
                                             const float* __restrict__ fscale_hi, const float* __restrict__ fscale_lo,
                                             R* __restrict__ sm)
{
    static_assert(TW == 32 || TW == 32 * MESS_TEAM_WARPS, "a warp or the whole block per quartet");
    static_assert(!PS || TW == 32 * MESS_TEAM_WARPS, "the primitive split spans the block");
    constexpr int TP = PS ? 32 : TW;                // threads of one primitive-loop group
    const int slot = threadIdx.x / TW, lane = threadIdx.x % TW;
    const int pslot = PS ? (int)(threadIdx.x >> 5) : slot, plane = threadIdx.x % TP;
    R* V = sm + (size_t)slot * (NVI + NH);
    R* H = V + NVI;
    R* Vp = sm + (size_t)pslot * (NVI + NH);        // the group's own values and contracted sums
    R* Hp = Vp + NVI;
    for (int k = plane; k < NACC; k += TP) Hp[k] = R(0);
    team_sync<TP>();
    const int b0 = P.pp_off[bp], nbp = P.pp_n[bp];
    const int k0 = kv.k0, nkp = kv.nk;
    const R ACx = kv.AC[0], ACy = kv.AC[1], ACz = kv.AC[2];
#pragma unroll 1
    for (int ip = PS ? pslot + MESS_TEAM_WARPS * (int)blockIdx.y : 0; ip < nbp * nkp; ip += PS ? MESS_TEAM_WARPS * (int)gridDim.y : 1) {
        const int ib = b0 + ip / nkp, ik = k0 + ip % nkp;
        const PrimPair<R> pb = P.load(ib);
        {
            const PrimPair<R> pk = P.load(ik);
            R rz, srz;
            recip_and_sqrt(pb.zeta + pk.zeta, rz, srz);
            const R roz = pk.zeta * rz, roe = pb.zeta * rz, oo2ze = R(0.5) * rz;
            const R PQx = pb.PAx - pk.PAx + ACx, PQy = pb.PAy - pk.PAy + ACy, PQz = pb.PAz - pk.PAz + ACz;
            const R WPx = -roz * PQx, WPy = -roz * PQy, WPz = -roz * PQz;
            const R WQx = roe * PQx, WQy = roe * PQy, WQz = roe * PQz;
            const R T = pb.zeta * roz * (PQx * PQx + PQy * PQy + PQz * PQz);
            const R pref = pb.K * pk.K * srz;
            R F[L + 1];
            boys_eval<R, L, BMODE>(T, pref, F, P);
#pragma unroll 1
            for (int lv = 0; lv < NVL; ++lv) {
                const int oend = __ldg(vlev + lv + 1);
#pragma unroll 1
                for (int o = __ldg(vlev + lv) + plane; o < oend; o += TP) {
                    const uint4 w = __ldg(vprog + o);
                    const int kind = w.x & 3, d = (w.x >> 2) & 3;
                    const int m1 = (w.x >> 4) & 15, m2 = (w.x >> 8) & 15, t = w.x >> 16;
                    const int s1 = w.y & 0xffff, s2 = w.y >> 16;
                    if (kind == 0) {
                        R f = F[0];
#pragma unroll
                        for (int m = 1; m <= L; ++m) f = (s1 == m) ? F[m] : f;
                        Vp[t] = f;
                    } else if (kind == 3) {
                        Hp[s1] += Vp[t];
                    } else if (kind == 1) {
                        R v = pick3(d, pb.PAx, pb.PAy, pb.PAz) * Vp[s1] + pick3(d, WPx, WPy, WPz) * Vp[s2];
                        if (m1) v += small_int<R>(m1) * pb.oo2z * (Vp[w.z & 0xffff] - roz * Vp[w.z >> 16]);
                        Vp[t] = v;
                    } else {
                        R v = pick3(d, pk.PAx, pk.PAy, pk.PAz) * Vp[s1] + pick3(d, WQx, WQy, WQz) * Vp[s2];
                        if (m1) v += small_int<R>(m1) * pk.oo2z * (Vp[w.z & 0xffff] - roe * Vp[w.z >> 16]);
                        if (m2) v += small_int<R>(m2) * oo2ze * Vp[w.w];
                        Vp[t] = v;
                    }
                }
                team_sync<TP>();
            }
        }
    }
    if (PS) {
        __syncthreads();
        for (int k = threadIdx.x; k < NACC; k += TW) {
            R acc = H[k];
#pragma unroll
            for (int w = 1; w < MESS_TEAM_WARPS; ++w) acc += sm[(size_t)w * (NVI + NH) + NVI + k];
            H[k] = acc;
        }
        __syncthreads();
    }
    const R ABx = pair_ab(P, bp, 0), ABy = pair_ab(P, bp, 1), ABz = pair_ab(P, bp, 2);
    const R CDx = kv.CD[0], CDy = kv.CD[1], CDz = kv.CD[2];
#pragma unroll 1
    for (int lv = 0; lv < NHL; ++lv) {
        const int oend = __ldg(hlev + lv + 1);
#pragma unroll 1
        for (int o = __ldg(hlev + lv) + lane; o < oend; o += TW) {
            const uint2 w = __ldg(hprog + o);
            const int t = w.x & 0xffff, d = (w.x >> 16) & 3, side = (w.x >> 18) & 1;
            const R X = side ? pick3(d, CDx, CDy, CDz) : pick3(d, ABx, ABy, ABz);
            H[t] = H[w.y & 0xffff] + X * H[w.y >> 16];
        }
        team_sync<TW>();
    }
    for (int k = lane; k < NINT; k += TW) V[k] = gen_scale<R>(fscale, fscale_hi, fscale_lo, k) * H[__ldg(fslot + k)];
    team_sync<TW>();
    return V;
}

template <typename R, int BMODE, int TW, int PS, int L, int NVI, int NH, int NACC, int NVL, int NHL, int NINT,
          int NA, int NB, int NC, int ND>
__device__ __forceinline__ void jk_team_body(const BinLaunch& b, const PairTable<R>& P, const typename DElem<R>::T* __restrict__ D,
                                             double* __restrict__ J, double* __restrict__ K, int n,
                                             const uint4* __restrict__ vprog, const int* __restrict__ vlev,
                                             const uint2* __restrict__ hprog, const int* __restrict__ hlev,
                                             const int* __restrict__ fslot, const double* __restrict__ fscale,
                                             const float* __restrict__ fscale_hi, const float* __restrict__ fscale_lo,
                                             R* __restrict__ sm)
{
    const int slot = threadIdx.x / TW, lane = threadIdx.x % TW;
    const long long q = (long long)blockIdx.x * (32 * MESS_TEAM_WARPS / TW) + slot;
    if (q >= b.total) return;                       // the quartet's threads leave together
    const int i = find_bra(b, q);
    const int j = __ldg(b.kbeg + i) + (int)(q - __ldg(b.offs + i));
    const int bp = __ldg(b.bra + i);
    const KetRec* kr = b.ketrec + j;
    const int4 kh = ket_hdr(kr);
    const int kp = ket_pair(kr);
    if (!P.live(bp) || !P.dens_ok(bp, kp)) return;   // the quartet's threads leave together
    const R* I = team_eri<R, BMODE, TW, PS, L, NVI, NH, NACC, NVL, NHL, NINT, NA, NB, NC, ND>(
        P, bp, ket_view(P, bp, kr, kh), vprog, vlev, hprog, hlev, fslot, fscale, fscale_hi, fscale_lo, sm);
    R s = R(1);
    if (__ldg(P.same + bp)) s *= R(0.5);
    if (kh.w & 1) s *= R(0.5);
    if (bp == kp) s *= R(0.5);
    const int mol_ = __ldg(P.mol + bp);
    const long long off_ = __ldg(P.mbase + mol_);
    (void)n;
    const DigestCtx<R> c{D + off_, J + off_, K + off_, __ldg(P.mn + mol_), __ldg(P.fa + bp), __ldg(P.fb + bp),
                         kh.z & 0xffff, kh.z >> 16, false};
    team_digest<R, TW, NA, NB, NC, ND>(I, c, s, lane);
}

#define MESS_DEFINE_TEAM_KERNEL_IMPL(TAG, ...)                                                      \
    template <typename R> constexpr size_t team_smem_##TAG()                                        \
    {                                                                                               \
        return team_smem_bytes<R, __VA_ARGS__>();                                                   \
    }                                                                                               \
    template <typename R, int BMODE, int TW, int PS>                                                \
    __global__ void __launch_bounds__(32 * MESS_TEAM_WARPS)                                         \
    k_jk_team_##TAG(const BinLaunch b, const PairTable<R> P, const typename DElem<R>::T* __restrict__ D,          \
                    double* __restrict__ J, double* __restrict__ K, int n)                          \
    {                                                                                               \
        extern __shared__ __align__(16) unsigned char mess_team_smem[];                             \
        jk_team_body<R, BMODE, TW, PS, __VA_ARGS__>(b, P, D, J, K, n, MESS_TEAM_PROG_##TAG,         \
                                            reinterpret_cast<R*>(mess_team_smem));                  \
    }
#define MESS_DEFINE_TEAM_KERNEL(TAG) MESS_DEFINE_TEAM_KERNEL_IMPL(TAG, MESS_TEAM_ARGS_##TAG)

// Schwarz factors of the op-program classes: one block per pair, its warps splitting the primitive
// quartets of the diagonal quartet.  Latency-bound (81 primitive quartets, one dependency level at a
// time); C2H6 / 6-31G's derivative basis: (dd|dd) 118.8 -> 1.0 ms, (dp|dp) 106.0 -> 1.4 ms against one
// thread per pair.
template <int L, int NVI, int NH, int NACC, int NVL, int NHL, int NINT, int NA, int NB, int NC, int ND>
__device__ __forceinline__ void schwarz_team_body(const int* __restrict__ pairs, const PairTable<double>& P, double* __restrict__ Q,
                                                  const uint4* __restrict__ vprog, const int* __restrict__ vlev,
                                                  const uint2* __restrict__ hprog, const int* __restrict__ hlev,
                                                  const int* __restrict__ fslot, const double* __restrict__ fscale,
                                                  const float* __restrict__ fscale_hi, const float* __restrict__ fscale_lo,
                                                  double* __restrict__ sm)
{
    __shared__ double red[MESS_TEAM_WARPS];
    const int p = pairs[blockIdx.x];
    const double* I = team_eri<double, 0, 32 * MESS_TEAM_WARPS, 1, L, NVI, NH, NACC, NVL, NHL, NINT, NA, NB, NC, ND>(
        P, p, ket_view(P, p, P.rec + p, ket_hdr(P.rec + p)), vprog, vlev, hprog, hlev, fslot, fscale, fscale_hi, fscale_lo, sm);
    double m = 0.0;
    for (int o = threadIdx.x; o < NA * NB; o += 32 * MESS_TEAM_WARPS) m = fmax(m, fabs(I[o * (NC * ND) + o]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, shfl_xor(m, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < MESS_TEAM_WARPS; ++w) m = fmax(m, red[w]);
        Q[p] = sqrt(m);
    }
}

#define MESS_DEFINE_TEAM_SCHWARZ_KERNEL_IMPL(TAG, ...)                                              \
    __global__ void __launch_bounds__(32 * MESS_TEAM_WARPS)                                         \
    k_schwarz_team_##TAG(const int* __restrict__ pairs, const PairTable<double> P, double* __restrict__ Q) \
    {                                                                                               \
        extern __shared__ __align__(16) unsigned char mess_team_smem[];                             \
        schwarz_team_body<__VA_ARGS__>(pairs, P, Q, MESS_TEAM_PROG_##TAG,                           \
                                       reinterpret_cast<double*>(mess_team_smem));                  \
    }
#define MESS_DEFINE_TEAM_SCHWARZ_KERNEL(TAG) MESS_DEFINE_TEAM_SCHWARZ_KERNEL_IMPL(TAG, MESS_TEAM_ARGS_##TAG)

template <typename R, int L, int NVI, int NH, int NACC, int NVL, int NHL, int NINT, int NA, int NB, int NC, int ND>
constexpr size_t team_smem_bytes()
{
    return (size_t)MESS_TEAM_WARPS * (NVI + NH) * sizeof(R);
}
