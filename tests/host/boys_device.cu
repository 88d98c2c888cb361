// The kernels' Boys function and its tables, as compiled into them, for arguments of the caller's.
#include "boys_table.cu"

void mess_set_error(const char*, ...) {}

template <typename R, int L, int BMODE> __global__ void k_eval(const double* T, int n, PairTable<R> P, double* out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    R F[L + 1];
    boys_eval<R, L, BMODE>(R(T[i]), R(1), F, P);
    for (int m = 0; m <= L; ++m) out[(size_t)i * (L + 1) + m] = F[m];
}

template <typename R, int BMODE, int L> cudaError_t eval(int l, const double* T, int n, const MessBoysTables& t, double* out)
{
    if constexpr (L >= MESS_BOYS_NL) {
        return cudaErrorInvalidValue;
    } else {
        if (l != L) return eval<R, BMODE, L + 1>(l, T, n, t, out);
        PairTable<R> P{};
        P.boys64 = t.b64;
        P.boys32v = t.b32;
        k_eval<R, L, BMODE><<<(n + 127) / 128, 128>>>(T, n, P, out);
        return cudaGetLastError();
    }
}

// F_0..F_L of n arguments into out[n][L + 1]; mode 0 FP64, 1 FP32 with the FP64 function, 2 FP32
extern "C" int boys_device(int mode, int L, int n, const double* T, double* out)
{
    MessBoysTables t;
    if (n <= 0 || mess_boys_device(&t) != MESS_OK) return 1;
    DevBuf<double> dT, dF;
    if (dT.alloc(n) != cudaSuccess || dF.alloc((size_t)n * (L + 1)) != cudaSuccess) return 2;
    if (cudaMemcpy(dT.p, T, sizeof(double) * n, cudaMemcpyHostToDevice) != cudaSuccess) return 3;
    const cudaError_t e = mode == 0 ? eval<double, 0, 0>(L, dT.p, n, t, dF.p) : mode == 1 ? eval<float, 1, 0>(L, dT.p, n, t, dF.p)
                                                                                 : eval<float, 2, 0>(L, dT.p, n, t, dF.p);
    if (e != cudaSuccess) return 4;
    return cudaMemcpy(out, dF.p, sizeof(double) * n * (L + 1), cudaMemcpyDeviceToHost) == cudaSuccess ? 0 : 5;
}
