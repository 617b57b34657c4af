// Activations and the fused epilogues of the FP64 path's GEMMs (the SIMT ones
// and the tensor-core ones): each is called once per output (row, column).
#pragma once
#include <cuda_runtime.h>

#include <cstddef>

namespace dino {
namespace {

template <typename T>
__device__ __forceinline__ T act_fn(int kind, T z) {
  if (kind == 1) return tanh(z);
  if (kind == 2) return T(0.5) * z * (T(1) + erf(z * T(0.70710678118654752440)));
  return z;
}

template <typename T>
__device__ __forceinline__ T act_deriv(int kind, T z) {
  if (kind == 1) {
    const T t = tanh(z);
    return T(1) - t * t;
  }
  if (kind == 2)
    return T(0.5) * (T(1) + erf(z * T(0.70710678118654752440))) +
           z * exp(T(-0.5) * z * z) * T(0.39894228040143267794);
  return T(1);
}

template <typename T>
struct EpiStore {
  T *out;
  int ldo;
  __device__ void operator()(int r, int c, T v) const { out[(size_t)r * ldo + c] = v; }
};

template <typename T>
struct EpiBiasAct {
  const T *bias;
  int act;
  T *out, *der;
  int ldo;
  __device__ void operator()(int r, int c, T v) const {
    const T z = v + bias[c];
    out[(size_t)r * ldo + c] = act_fn(act, z);
    if (der) der[(size_t)r * ldo + c] = act_deriv(act, z);
  }
};

template <typename T>
struct EpiScaleGroup {
  const T *scale;
  int lds, group;
  T *out;
  int ldo;
  __device__ void operator()(int r, int c, T v) const {
    out[(size_t)r * ldo + c] = v * scale[(size_t)(r / group) * lds + c];
  }
};

template <typename T>
struct EpiCoef {
  const double *coef;
  int ldc;
  double cs;
  T *out;
  int ldo;
  __device__ void operator()(int r, int c, T v) const {
    out[(size_t)r * ldo + c] = (T)(coef[(size_t)r * ldc + c] - cs * (double)v);
  }
};

template <typename T>
struct EpiField {
  const int *acc;
  double s, cs;
  T *m;
  const T *Mf;
  int ldm;
  __device__ void operator()(int r, int c, T v) const {
    if (!acc[r]) return;
    const size_t o = (size_t)r * ldm + c;
    m[o] = (T)(s * (double)m[o] + cs * (double)Mf[o]) + v;
  }
};

// Newton-Schulz: P = (3 I - S) / 2 from S = X^T X, and the largest |S - I| (as the
// bits of a nonnegative double; a NaN is larger than every number) where res is
// given
struct EpiPoly {
  double *P;
  int ld;
  unsigned long long *res;
  __device__ void operator()(int r, int c, double v) const {
    const double e = v - (r == c ? 1.0 : 0.0);
    P[(size_t)r * ld + c] = (r == c ? 1.0 : 0.0) - 0.5 * e;
    if (res) atomicMax(res, (unsigned long long)__double_as_longlong(fabs(e)));
  }
};

// ... and the new Y = X^T = P X^T, kept both ways
struct EpiBoth {
  double *Y, *X;
  int ld;
  __device__ void operator()(int r, int c, double v) const {
    Y[(size_t)r * ld + c] = v;
    X[(size_t)c * ld + r] = v;
  }
};

}  // namespace
}  // namespace dino
