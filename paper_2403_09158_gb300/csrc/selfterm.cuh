// Sums of the self-term table over the half spectrum, shared by the sum over stored spectra
// (defects.cu) and the sum inside the pencil pass (solve_fast.cu).
#pragma once

#include "okmc_internal.cuh"

namespace okmc {

// Per-thread accumulators of the self-term sums: compensated FP32 pairs for FP32
// spectra, plain FP64 for FP64 spectra.
template <class T> struct WAcc;
template <> struct WAcc<float> {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float t = s + x;
    const float bp = t - s;
    c += (s - (t - bp)) + (x - bp);
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};
template <> struct WAcc<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double x) { s += x; }
  __device__ __forceinline__ double value() const { return s; }
};

// The FP32 sums with their roundings fixed, so that every kernel that forms them forms the
// same ones: the compiler contracts products and sums differently from kernel to kernel, and a
// table off by 1e-7 eV moves the kinetic clock by 1e-6.  Products of phases: the real part as
// fma(a.x, b.x, -(a.y b.y)), the imaginary part with either product rounded first.
__device__ __forceinline__ C2<float> st_mul(C2<float> a, C2<float> b) {
  return C2<float>{__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.y, b.x, __fmul_rn(a.x, b.y))};
}
__device__ __forceinline__ C2<float> st_mul_last(C2<float> a, C2<float> b) { return cmul_rn(a, b); }
__device__ __forceinline__ C2<double> st_mul(C2<double> a, C2<double> b) { return a * b; }
__device__ __forceinline__ C2<double> st_mul_last(C2<double> a, C2<double> b) { return a * b; }

// exp(i xi.d) for the eight d in {-1, 0}^3 (bit 2: x, 1: y, 0: z; clear means -1, a factor
// conj(e_axis)) from the conjugate phases of the axes
template <class T>
__device__ __forceinline__ void selfterm_phases(C2<T> ax, C2<T> ay, C2<T> az, C2<T>* ph) {
  ph[7] = C2<T>{T(1), T(0)};
  ph[6] = az;
  ph[5] = ay;
  ph[4] = st_mul(ay, az);
  ph[3] = ax;
  ph[2] = st_mul(ax, az);
  ph[1] = st_mul(ax, ay);
  ph[0] = st_mul_last(ph[1], az);
}

// a + the term whose sum with a value z is sum(z), compensated
template <class F>
__device__ __forceinline__ void st_add(WAcc<float>& a, const F& sum) {
  const float t = sum(a.s), bp = __fsub_rn(t, a.s);
  a.c = __fadd_rn(a.c, __fadd_rn(__fsub_rn(a.s, __fsub_rn(t, bp)), sum(-bp)));
  a.s = t;
}

// One frequency of one defect: q |w0|^2, q |w1|^2 and q Re(conj(w1) w0 ph[s]), products in
// the spectrum precision (the first two enter their sums unrounded)
__device__ __forceinline__ void selfterm_add(WAcc<float>* acc, C2<float> w0, C2<float> w1, float q, const C2<float>* ph) {
  const float n0 = __fmaf_rn(w0.x, w0.x, __fmul_rn(w0.y, w0.y)), n1 = __fmaf_rn(w1.x, w1.x, __fmul_rn(w1.y, w1.y));
  st_add(acc[0], [&](float z) { return __fmaf_rn(q, n0, z); });
  st_add(acc[1], [&](float z) { return __fmaf_rn(q, n1, z); });
  // conj(w1) * w0
  const float qr = __fmul_rn(q, __fmaf_rn(w1.x, w0.x, __fmul_rn(w1.y, w0.y)));
  const float qi = __fmul_rn(q, __fmaf_rn(w1.x, w0.y, -__fmul_rn(w1.y, w0.x)));
#pragma unroll
  for (int s = 0; s < 7; ++s) {
    const float x = __fmaf_rn(qr, ph[s].x, -__fmul_rn(qi, ph[s].y));
    st_add(acc[2 + s], [&](float z) { return __fadd_rn(x, z); });
  }
  st_add(acc[9], [&](float z) { return __fadd_rn(qr, z); });
}
__device__ __forceinline__ void selfterm_add(WAcc<double>* acc, C2<double> w0, C2<double> w1, double q, const C2<double>* ph) {
  acc[0].add(q * (w0.x * w0.x + w0.y * w0.y));
  acc[1].add(q * (w1.x * w1.x + w1.y * w1.y));
  const double qr = q * (w1.x * w0.x + w1.y * w0.y), qi = q * (w1.x * w0.y - w1.y * w0.x);
#pragma unroll
  for (int s = 0; s < 8; ++s) acc[2 + s].add(qr * ph[s].x - qi * ph[s].y);
}

}  // namespace okmc
