// The library's float64 functions evaluated over arrays, for
// test_gpu_float64_functions.py.
#include "sdpd_rand64.cuh"

using namespace sdpd;

enum { kRcp, kSqrt, kRsqrt, kExpm1, kLog1p, kPairR, kPairR2, kPairRinv, kUnitLog, kUnitCos, kUnitSin, kUnitValue,
       kCudaExpm1, kCudaLog1p };

__global__ void k_eval(int fn, int64_t n, const double* x, double* y) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = x[i];
  const uint64_t u = (uint64_t)__double_as_longlong(v);  // unit_*: the bits of x
  double a = 0.0, b = 0.0;
  int k, j;
  switch (fn) {
    case kRcp: a = f64::rcp(v); break;
    case kSqrt: a = f64::sqrt_(v); break;
    case kRsqrt: a = f64::rsqrt_(v); break;
    case kExpm1: a = f64::expm1(v); break;
    case kLog1p: a = f64::log1p(v); break;
    case kPairR: a = pair_r64(v); break;
    case kPairR2: a = pair_r64(v, b); break;
    case kPairRinv: pair_r64(v, a); break;
    case kUnitLog: a = f64::unit_log(u); break;
    case kUnitCos: f64::unit_cossin(u, a, b); break;
    case kUnitSin: f64::unit_cossin(u, b, a); break;
    case kCudaExpm1: a = ::expm1(v); break;
    case kCudaLog1p: a = ::log1p(v); break;
    case kUnitValue: a = f64::unit_value(u, k, j, b); break;
  }
  y[i] = a;
}

extern "C" int eval(int fn, int64_t n, const double* x, double* y) {
  k_eval<<<(unsigned)((n + 255) / 256), 256>>>(fn, n, x, y);
  return (int)cudaDeviceSynchronize();
}
