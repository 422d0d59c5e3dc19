// Complex arithmetic on interleaved float2/double2 values (re = .x, im = .y).
#pragma once
#include <cuda_runtime.h>

namespace hh {

__host__ __device__ __forceinline__ float2 cmk(float a, float b) {
  return make_float2(a, b);
}
__host__ __device__ __forceinline__ double2 cmk(double a, double b) {
  return make_double2(a, b);
}

template <typename C> __host__ __device__ __forceinline__ C czero() {
  C z;
  z.x = 0;
  z.y = 0;
  return z;
}

template <typename C> __device__ __forceinline__ C cadd(C a, C b) {
  return cmk(a.x + b.x, a.y + b.y);
}
template <typename C> __device__ __forceinline__ C csub(C a, C b) {
  return cmk(a.x - b.x, a.y - b.y);
}
template <typename C> __device__ __forceinline__ C cneg(C a) {
  return cmk(-a.x, -a.y);
}
template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
  return cmk(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a * b + c
template <typename C> __device__ __forceinline__ C cfma(C a, C b, C c) {
  return cmk(c.x + a.x * b.x - a.y * b.y, c.y + a.x * b.y + a.y * b.x);
}
template <typename C, typename R> __device__ __forceinline__ C cscale(C a, R s) {
  return cmk(a.x * s, a.y * s);
}
template <typename C> __device__ __forceinline__ auto cabs2(C a) {
  return a.x * a.x + a.y * a.y;
}
// a / b = a conj(b) / |b|^2 (the operands here are O(1)..O(1e10) in
// modulus, far from overflow in either precision).
template <typename C> __device__ __forceinline__ C cdiv(C a, C b) {
  const auto d = b.x * b.x + b.y * b.y;
  return cmk((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}
// fused multiply-add a * b + c in the operands' precision
__device__ __forceinline__ float fmaf_any(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmaf_any(double a, double b, double c) { return fma(a, b, c); }
// 1 / b (one real division)
template <typename C> __device__ __forceinline__ C crcp(C b) {
  const auto s = decltype(b.x)(1) / (b.x * b.x + b.y * b.y);
  return cmk(b.x * s, -b.y * s);
}

// c - a b
template <typename C> __device__ __forceinline__ C cfnma(C a, C b, C c) {
  return cmk(c.x - a.x * b.x + a.y * b.y, c.y - a.x * b.y - a.y * b.x);
}
// d - beta k2.  In complex128 a uniform branch leaves out the imaginary part of a real
// beta (the finest level's); in complex64 a branch costs more than it saves.
template <typename C, typename R> __device__ __forceinline__ C diag_less(C d, C beta, R k2) {
  d.x = fmaf_any(-beta.x, k2, d.x);
  if (sizeof(R) == 4 || beta.y != R(0)) d.y = fmaf_any(-beta.y, k2, d.y);
  return d;
}
// omega / D: one real division (omega is real in all but the ablation)
template <typename C> __device__ __forceinline__ C jacobi_weight(C omega, C D) {
  if (sizeof(D.x) == 8 && omega.y == decltype(D.x)(0)) {
    const auto s = omega.x / (D.x * D.x + D.y * D.y);
    return cmk(D.x * s, -D.y * s);
  }
  return cmul(omega, crcp(D));
}

// f - (D u - the neighbours' part) of a 5-point row with its own coefficients.
// complex128 counts FP64 instructions: one chain of multiply-adds; complex64, whose
// small levels wait for the chain, two shorter ones and an addition.
template <typename C>
__device__ __forceinline__ C resid_row(C f, C D, C u, C lx, C uw, C ux, C ue, C ly, C un, C uy, C us) {
  if (sizeof(f.x) == 8) {
    C r = cfnma(D, u, f);
    r = cfma(lx, uw, r);
    r = cfma(ux, ue, r);
    r = cfma(ly, un, r);
    return cfma(uy, us, r);
  }
  C nb = cmul(lx, uw);
  nb = cfma(ux, ue, nb);
  nb = cfma(ly, un, nb);
  nb = cfma(uy, us, nb);
  return cadd(csub(f, cmul(D, u)), nb);
}

}  // namespace hh
