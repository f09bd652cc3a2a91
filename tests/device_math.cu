// Entry points for tests/test_gpu_device_math.py: the device helpers of
// fvm_device.cuh beside the instructions they replace, one value per thread.
#include "fvm_device.cuh"

using namespace fvm;

namespace {

template <typename F>
__global__ void k_each(long long n, F f) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) f(i);
}

template <typename F>
int each(long long n, F f) {
  k_each<<<(unsigned)((n + 255) / 256), 256>>>(n, f);
  const cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? (int)e : (int)cudaDeviceSynchronize();
}

}  // namespace

extern "C" int dm_clamp01(long long n, const double* a, double* out) {
  return each(n, [=] __device__(long long i) { out[i] = clamp01(a[i]); });
}

extern "C" int dm_root(long long n, const double* a, double* out) {
  return each(n, [=] __device__(long long i) { out[i] = root(a[i]); });
}

extern "C" int dm_quotient(long long n, const double* a, const double* b, double* out) {
  return each(n, [=] __device__(long long i) { out[i] = quotient(a[i], b[i]); });
}

// the plain division, root and conversion on the device
extern "C" int dm_divide(long long n, const double* a, const double* b, double* out) {
  return each(n, [=] __device__(long long i) { out[i] = a[i] / b[i]; });
}
extern "C" int dm_sqrt(long long n, const double* a, double* out) {
  return each(n, [=] __device__(long long i) { out[i] = sqrt(a[i]); });
}

extern "C" int dm_narrow(long long n, const double* a, float* out) {
  return each(n, [=] __device__(long long i) { out[i] = narrow<float>(a[i]); });
}
extern "C" int dm_to_float(long long n, const double* a, float* out) {
  return each(n, [=] __device__(long long i) { out[i] = (float)a[i]; });
}

// counts the float bit patterns whose widen() is not the conversion's
extern "C" int dm_widen_all(unsigned long long* differ) {
  return each(1LL << 32, [=] __device__(long long i) {
    const float f = __uint_as_float((unsigned)i);
    if (__double_as_longlong(widen(f)) != __double_as_longlong((double)f)) atomicAdd(differ, 1ULL);
  });
}
