// The part of the CUDA runtime that the library's host code uses, over malloc, with kernels that do nothing and
// allocations that can be made to fail one at a time: host programs link it in place of libcudart.  No GPU.
#include <cstdlib>
#include <cstring>
#include <set>

long fake_fail_in = -1;      // allocations until one fails (-1: none)
long fake_null_copies = 0;   // copies and fills that met a null pointer
static int last_error = 0;   // as the runtime keeps it: until someone asks
static std::set<void*>& live() { static std::set<void*> s; return s; }
size_t fake_live() { return live().size(); }

enum { ok = 0, invalid_value = 1, memory_allocation = 2 };
struct Dim { unsigned x, y, z; };

extern "C" {
int cudaMalloc(void** p, size_t n)
{
    if (fake_fail_in >= 0 && fake_fail_in-- == 0) { *p = nullptr; return last_error = memory_allocation; }
    *p = malloc(n);
    live().insert(*p);
    return ok;
}
int cudaFree(void* p) { live().erase(p); free(p); return ok; }
int cudaMemcpy(void* d, const void* s, size_t n, int)
{
    if (!d || !s) { ++fake_null_copies; return last_error = invalid_value; }
    memmove(d, s, n);
    return ok;
}
int cudaMemcpyAsync(void* d, const void* s, size_t n, int k, void*) { return cudaMemcpy(d, s, n, k); }
int cudaMemset(void* d, int v, size_t n)
{
    if (!d) { ++fake_null_copies; return last_error = invalid_value; }
    memset(d, v, n);
    return ok;
}
int cudaMemsetAsync(void* d, int v, size_t n, void*) { return cudaMemset(d, v, n); }
int cudaGetLastError() { const int e = last_error; last_error = ok; return e; }
const char* cudaGetErrorString(int) { return "error"; }
int cudaDeviceSynchronize() { return ok; }
int cudaStreamSynchronize(void*) { return ok; }
int cudaLaunchKernel(const void*, Dim, Dim, void**, size_t, void*) { return ok; }
int __cudaGetKernel(void** k, const void* f) { *k = const_cast<void*>(f); return ok; }
int __cudaLaunchKernel(void*, Dim, Dim, void**, size_t, void*) { return ok; }
unsigned __cudaPushCallConfiguration(Dim, Dim, size_t, void*) { return 0; }
int __cudaPopCallConfiguration(Dim*, Dim*, size_t*, void*) { return ok; }
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
}
