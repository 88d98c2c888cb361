// Tabulation of the Boys function: the grids that the kernels expand around, one copy per device, and
// the values reported by mess_boys_grid.
//   tab[k][n] = F_n(T_k), T_k = k * MESS_BOYS_DT, n = 0..MESS_BOYS_NF-1;  tab[k][MESS_BOYS_NF] = exp(-T_k).
// F_{NF-1}(T) comes from the positive series exp(-T) sum_i (2T)^i / ((2n+1)(2n+3)...(2n+2i+1)) in
// long double; the lower orders follow from the downward recursion F_{n-1} = (2T F_n + e^{-T})/(2n-1),
// which is stable in that direction.
#include <math.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "mess_internal.h"

void mess_boys_table(std::vector<double>& tab, int nrow, double dt)
{
    tab.assign((size_t)nrow * MESS_BOYS_NCOL, 0.0);
    for (int k = 0; k < nrow; ++k) {
        const long double T = (long double)k * (long double)dt;
        const long double eT = expl(-T);
        const int top = MESS_BOYS_NF - 1;
        long double term = 1.0L / (2 * top + 1), sum = term;
        for (int i = 1; i < 10000; ++i) {
            term *= 2.0L * T / (long double)(2 * top + 2 * i + 1);
            sum += term;
            if (term < sum * 1e-21L) break;
        }
        long double F[MESS_BOYS_NF];
        F[top] = eT * sum;
        for (int n = top; n >= 1; --n) F[n - 1] = (2.0L * T * F[n] + eT) / (long double)(2 * n - 1);
        for (int n = 0; n < MESS_BOYS_NF; ++n) tab[(size_t)k * MESS_BOYS_NCOL + n] = (double)F[n];
        tab[(size_t)k * MESS_BOYS_NCOL + MESS_BOYS_NF] = (double)eT;
    }
}

// The kernels' tables (mess_device.h): constants, the same for every basis, so one copy per device in the
// library's image, filled when the first basis of the device builds its data (2.5 MB; tabulating them
// for every basis took 6 ms of host time each).
static __device__ __align__(256) double g_boys64[MESS_BOYS_NL * MESS_BOYS64_NROW * 8];
static __device__ __align__(256) float4 g_boys32[MESS_BOYS_NL * MESS_BOYS32_NROW];
static __device__ __align__(256) float4 g_boysdf[MESS_BOYS_NL * MESS_BOYSDF_NROW * 3];

mess_status mess_boys_device(MessBoysTables* out)
{
    static std::mutex mu;
    static MessBoysTables ready[64];
    int dev = 0;
    MESS_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) { mess_set_error("device index %d out of range", dev); return MESS_EINVAL; }
    std::lock_guard<std::mutex> lk(mu);
    if (!ready[dev].b64) {
        static std::vector<double> h64;
        static std::vector<float4> h32, hdf;
        if (h64.empty()) {
            // one table at the finest step (1/128); the others take every second and every fourth row
            static_assert(MESS_BOYS32_INV_DT == 2 * MESS_BOYSDF_INV_DT && MESS_BOYS32_INV_DT == 4 * MESS_BOYS64_INV_DT, "steps");
            const int nrow = std::max({4 * MESS_BOYS64_NROW, 2 * MESS_BOYSDF_NROW, MESS_BOYS32_NROW});
            std::vector<double> t;
            mess_boys_table(t, nrow, 1.0 / MESS_BOYS32_INV_DT);
            const double fact[7] = {1.0, 1.0, 2.0, 6.0, 24.0, 120.0, 720.0};
            std::vector<float4> df((size_t)MESS_BOYS_NL * MESS_BOYSDF_NROW * 3);
            for (int L = 0; L < MESS_BOYS_NL; ++L)
                for (int k = 0; k < MESS_BOYSDF_NROW; ++k) {
                    const double* row = t.data() + (size_t)(2 * k) * MESS_BOYS_NCOL;
                    float hi[7], lo[7];
                    for (int j = 0; j < 7; ++j) {
                        const double c = j < 6 ? row[L + j] / fact[j] : row[MESS_BOYS_NF];
                        hi[j] = (float)c;
                        lo[j] = (float)(c - (double)hi[j]);
                    }
                    float4* o = df.data() + ((size_t)L * MESS_BOYSDF_NROW + k) * 3;
                    o[0] = make_float4(hi[0], lo[0], hi[1], lo[1]);
                    o[1] = make_float4(hi[2], lo[2], hi[3], lo[3]);
                    o[2] = make_float4(hi[4], hi[5], hi[6], lo[6]);
                }
            std::vector<float4> f32((size_t)MESS_BOYS_NL * MESS_BOYS32_NROW);
            for (int L = 0; L < MESS_BOYS_NL; ++L)
                for (int k = 0; k < MESS_BOYS32_NROW; ++k) {
                    const double* row = t.data() + (size_t)k * MESS_BOYS_NCOL;
                    if (L == 0) {
                        constexpr int step = (int)(MESS_BOYS32_INV_DT / MESS_BOYS32_INV_DT0);
                        if (k % step == 0) f32[k / step] = make_float4((float)row[0], (float)row[1], (float)(row[2] / 2), (float)(row[3] / 6));
                        continue;
                    }
                    f32[(size_t)L * MESS_BOYS32_NROW + k] =
                        make_float4((float)row[L], (float)row[L + 1], (float)(0.5 * row[L + 2]), (float)row[MESS_BOYS_NF]);
                }
            std::vector<double> f64((size_t)MESS_BOYS_NL * MESS_BOYS64_NROW * 8);
            for (int L = 0; L < MESS_BOYS_NL; ++L)
                for (int k = 0; k < MESS_BOYS64_NROW; ++k) {
                    const double* row = t.data() + (size_t)(4 * k) * MESS_BOYS_NCOL;
                    double* o = f64.data() + ((size_t)L * MESS_BOYS64_NROW + k) * 8;
                    for (int j = 0; j < 7; ++j) o[j] = row[L + j] / fact[j];
                    o[7] = row[MESS_BOYS_NF];
                }
            hdf.swap(df);
            h32.swap(f32);
            h64.swap(f64);
        }
        void *p64 = nullptr, *p32 = nullptr, *pdf = nullptr;
        MESS_CUDA_TRY(cudaGetSymbolAddress(&p64, g_boys64));
        MESS_CUDA_TRY(cudaGetSymbolAddress(&p32, g_boys32));
        MESS_CUDA_TRY(cudaGetSymbolAddress(&pdf, g_boysdf));
        MESS_CUDA_TRY(cudaMemcpy(p64, h64.data(), h64.size() * sizeof(double), cudaMemcpyHostToDevice));
        MESS_CUDA_TRY(cudaMemcpy(p32, h32.data(), h32.size() * sizeof(float4), cudaMemcpyHostToDevice));
        MESS_CUDA_TRY(cudaMemcpy(pdf, hdf.data(), hdf.size() * sizeof(float4), cudaMemcpyHostToDevice));
        MESS_CUDA_TRY(cudaDeviceSynchronize());
        ready[dev] = MessBoysTables{static_cast<double*>(p64), static_cast<float4*>(p32), static_cast<float4*>(pdf)};
    }
    *out = ready[dev];
    return MESS_OK;
}

extern "C" mess_status mess_boys_grid(double* out, int max_values, int* nrows, int* ncols, double* dT)
{
    if (nrows) *nrows = MESS_BOYS_NROW;
    if (ncols) *ncols = MESS_BOYS_NCOL;
    if (dT) *dT = MESS_BOYS_DT;
    if (!out) return MESS_OK;
    if (max_values < MESS_BOYS_NROW * MESS_BOYS_NCOL) {
        mess_set_error("mess_boys_grid: %d values needed, max_values = %d", MESS_BOYS_NROW * MESS_BOYS_NCOL, max_values);
        return MESS_EINVAL;
    }
    std::vector<double> tab;
    mess_boys_table(tab, MESS_BOYS_NROW, MESS_BOYS_DT);
    for (size_t i = 0; i < tab.size(); ++i) out[i] = tab[i];
    return MESS_OK;
}
