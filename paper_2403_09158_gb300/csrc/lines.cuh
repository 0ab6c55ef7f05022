// Line passes: the solve of Sec. 3.2 for grids of any edges that okmc_grid_create takes,
// FP32 or FP64 fields, as five kernels that each transform lines along one axis.
//
//   x_fwd  : tiles of RB rows of a (component, z) plane: real rows of nx as complex rows
//            of H = nx/2, untangling, stored transposed (kx-major, RB consecutive y).
//   y      : lines of ny consecutive complex values, in place (forward or inverse).
//   pencil : tiles of TW consecutive ky at one kx, every kz, six components: forward z
//            transform, Green operator, inverse z transform.
//   x_inv  : tiles of RB rows: untangling from the kx-major plane, inverse rows, stress.
//
// A line of L = R1 R2 values is transformed in registers in two steps (Cooley-Tukey, n =
// n1 + R1 n2, k = k2 + R2 k1) with one exchange through shared memory between them.
//
// Why five passes and not the three of the cluster kernels: an x or y pass needs one
// tile of 16 rows or lines in shared memory whatever the plane's size, so it runs at
// several CTAs per SM without clusters, at every edge; the price is 240 N instead of
// 144 N bytes of traffic per FP32 solve (the x passes' output is re-read from L2 or HBM).
// What bounds them: FP64 fields, the FP64 pipe (two lanes per clock and SM): at 128^3 a full
// solve has about 0.97 G FP64 operations, 1.6 ms at that rate.  FP32 fields, memory and
// latency.  Against the shared-memory Stockham passes of solve.cu, which they replace here
// (GB300, us per pass, x and y | pencil | y and x): 128^3 FP64 1773 | 1312 | 1495 -> forward
// pass of the few planes of a moved defect 90 | 940 | 539; 512^3 FP32 8808 | 13195 | 15090 ->
// 438 (moved planes) | 2800 | 2790; 96x64x160 FP32 70 | 89 | 82 -> 19 | 28 | 25.
#pragma once

#include <type_traits>
#include <utility>

#include "fft_reg.cuh"

namespace okmc {

// ---------------------------------------------------------------- compile-time angles
__host__ __device__ constexpr double ct_sin_taylor(double x) {
  double t = x, s = x;
  for (int k = 1; k < 20; ++k) {
    t *= -x * x / ((2.0 * k) * (2.0 * k + 1.0));
    s += t;
  }
  return s;
}
__host__ __device__ constexpr double ct_cos_taylor(double x) {
  double t = 1.0, s = 1.0;
  for (int k = 1; k < 20; ++k) {
    t *= -x * x / ((2.0 * k - 1.0) * (2.0 * k));
    s += t;
  }
  return s;
}
// sin and tan(theta/2) of theta = 2 pi num / den, |theta| <= pi/2
__host__ __device__ constexpr double ct_sin(int num, int den) { return ct_sin_taylor(2.0 * kPi * num / den); }
__host__ __device__ constexpr double ct_tan_half(int num, int den) {
  return ct_sin_taylor(kPi * num / den) / ct_cos_taylor(kPi * num / den);
}

__device__ __forceinline__ C2<double> lift(C2<double> v, double t, double s) {
  const double x1 = fma(-t, v.y, v.x);
  const double y1 = fma(s, x1, v.y);
  const double x2 = fma(-t, y1, x1);
  return C2<double>{x2, y1};
}

// v * exp(-+2 pi i e / R) (minus sign forward): quarter turns exactly, any other angle as a
// rotation by three shears (three fma; a complex multiplication takes four operations)
template <class T, int R, bool INV, int E>
__device__ __forceinline__ C2<T> rotc(C2<T> v) {
  constexpr int e = E % R;
  if constexpr (e == 0) return v;
  else if constexpr (4 * e == R) return rot<T, INV>(v);
  else if constexpr (2 * e == R) return C2<T>{-v.x, -v.y};
  else if constexpr (4 * e == 3 * R) return rot<T, !INV>(v);
  else {
    constexpr int j0 = 2 * e > R ? R - e : -e;              // forward angle in units of 2 pi / R, within half a turn
    constexpr bool neg = 4 * (j0 < 0 ? -j0 : j0) > R;       // beyond a quarter turn: half a turn less, sign flipped
    constexpr int jn2 = neg ? (j0 > 0 ? 2 * j0 - R : 2 * j0 + R) : 2 * j0;  // in units of pi / R
    constexpr int j = INV ? -jn2 : jn2;
    constexpr double t = ct_tan_half(j, 2 * R), s = ct_sin(j, 2 * R);
    const C2<T> r = lift(v, T(t), T(s));
    return neg ? C2<T>{-r.x, -r.y} : r;
  }
}

// ---------------------------------------------------------------- register DFTs, FP32 or FP64
template <int R> struct GSplit;
template <> struct GSplit<6> { static constexpr int P = 2, Q = 3; };
template <> struct GSplit<8> { static constexpr int P = 2, Q = 4; };
template <> struct GSplit<10> { static constexpr int P = 2, Q = 5; };
template <> struct GSplit<12> { static constexpr int P = 4, Q = 3; };
template <> struct GSplit<16> { static constexpr int P = 4, Q = 4; };
template <> struct GSplit<18> { static constexpr int P = 3, Q = 6; };
template <> struct GSplit<20> { static constexpr int P = 4, Q = 5; };
template <> struct GSplit<24> { static constexpr int P = 8, Q = 3; };
template <> struct GSplit<32> { static constexpr int P = 4, Q = 8; };

template <bool INV> __device__ __forceinline__ void ddft3(C2<double>* v) {
  const double s = INV ? 0.86602540378443864676 : -0.86602540378443864676;  // sin(2 pi / 3)
  const C2<double> a = v[1] + v[2], b = v[1] - v[2];
  const C2<double> m{fma(-0.5, a.x, v[0].x), fma(-0.5, a.y, v[0].y)};
  v[0] = v[0] + a;
  v[1] = C2<double>{fma(-s, b.y, m.x), fma(s, b.x, m.y)};
  v[2] = C2<double>{fma(s, b.y, m.x), fma(-s, b.x, m.y)};
}

template <class T, int R, bool INV> __device__ __forceinline__ void gdft(C2<T>* v);

template <class T, int R, bool INV, int N1, int... K>
__device__ __forceinline__ void gdft_twiddle(C2<T>* y, const C2<T>* a, std::integer_sequence<int, K...>) {
  constexpr int Q = GSplit<R>::Q;
  ((y[N1 * Q + K] = rotc<T, R, INV, N1 * K>(a[K])), ...);
}
template <class T, int R, bool INV, int... N1>
__device__ __forceinline__ void gdft_rows(C2<T>* y, const C2<T>* v, std::integer_sequence<int, N1...>) {
  constexpr int P = GSplit<R>::P, Q = GSplit<R>::Q;
  auto row = [&](auto n1c) {
    constexpr int n1 = decltype(n1c)::value;
    C2<T> a[Q];
#pragma unroll
    for (int n2 = 0; n2 < Q; ++n2) a[n2] = v[n1 + P * n2];
    gdft<T, Q, INV>(a);
    gdft_twiddle<T, R, INV, n1>(y, a, std::make_integer_sequence<int, Q>{});
  };
  (row(std::integral_constant<int, N1>{}), ...);
}
template <class T, int R, bool INV>
__device__ __forceinline__ void gdft_composite(C2<T>* v) {
  constexpr int P = GSplit<R>::P, Q = GSplit<R>::Q;
  C2<T> y[R];
  gdft_rows<T, R, INV>(y, v, std::make_integer_sequence<int, P>{});
#pragma unroll
  for (int k2 = 0; k2 < Q; ++k2) {
    C2<T> b[P];
#pragma unroll
    for (int n1 = 0; n1 < P; ++n1) b[n1] = y[n1 * Q + k2];
    gdft<T, P, INV>(b);
#pragma unroll
    for (int k1 = 0; k1 < P; ++k1) v[k2 + Q * k1] = b[k1];
  }
}
// X_k = sum_n x_n exp(-+2 pi i n k / R), minus sign forward
template <class T, int R, bool INV>
__device__ __forceinline__ void gdft(C2<T>* v) {
  if constexpr (R == 1) return;
  else if constexpr (sizeof(T) == 4) {
    if constexpr (R == 2) pdft2<INV>(v);
    else if constexpr (R == 3) pdft3<INV>(v);
    else if constexpr (R == 4) pdft4<INV>(v);
    else if constexpr (R == 5) pdft5<INV>(v);
    else if constexpr (R == 8) pdft8<INV>(v);
    else if constexpr (R == 16) dft16<INV>(v);
    else gdft_composite<T, R, INV>(v);
  } else {
    if constexpr (R == 2) dft2<T, INV>(v);
    else if constexpr (R == 3) ddft3<INV>(v);
    else if constexpr (R == 4) dft4<T, INV>(v);
    else if constexpr (R == 5) dft5<T, INV>(v);
    else gdft_composite<T, R, INV>(v);
  }
}

// ---------------------------------------------------------------- line plans
// L = R1 R2 for every line length of the grids (edges 16..512 and half edges 8..256)
#define OKMC_LINE_PLANS(X)                                                                                          \
  X(8, 2, 4) X(16, 4, 4) X(24, 4, 6) X(32, 4, 8) X(40, 5, 8) X(48, 6, 8) X(64, 8, 8) X(72, 6, 12) X(80, 8, 10)     \
  X(96, 8, 12) X(120, 10, 12) X(128, 8, 16) X(144, 12, 12) X(160, 10, 16) X(192, 12, 16) X(200, 10, 20)            \
  X(216, 12, 18) X(240, 12, 20) X(256, 16, 16) X(288, 16, 18) X(320, 16, 20) X(384, 16, 24) X(400, 20, 20)         \
  X(432, 18, 24) X(480, 20, 24) X(512, 16, 32)
// the lengths met along x (half edges) and along y or z (edges)
#define OKMC_HALF_EDGES(X) \
  X(8) X(16) X(24) X(32) X(40) X(48) X(64) X(72) X(80) X(96) X(120) X(128) X(144) X(160) X(192) X(200) X(216) X(240) X(256)
#define OKMC_EDGES(X)                                                                                                 \
  X(16) X(32) X(48) X(64) X(80) X(96) X(128) X(144) X(160) X(192) X(240) X(256) X(288) X(320) X(384) X(400) X(432) X(480) \
  X(512)
template <int L> struct GPlan;
#define OKMC_PLAN(l, a, b) \
  template <> struct GPlan<l> { static constexpr int R1 = a, R2 = b, M = a > b ? a : b; static_assert(a * b == l, ""); };
OKMC_LINE_PLANS(OKMC_PLAN)
#undef OKMC_PLAN
// (R1, R2) of a line length known at run time; false if it has no plan
inline bool line_split(int L, int& R1, int& R2) {
  switch (L) {
#define OKMC_CASE(l, a, b) \
  case l: R1 = a; R2 = b; return true;
    OKMC_LINE_PLANS(OKMC_CASE)
#undef OKMC_CASE
    default: return false;
  }
}

__host__ __device__ constexpr int round32(int x) { return (x + 31) / 32 * 32; }

// Rows per tile of the x passes: 128 bytes of consecutive y in the kx-major plane
template <class T> __host__ __device__ constexpr int x_rows() { return 128 / (2 * (int)sizeof(T)); }
template <class T, int H> __host__ __device__ constexpr int x_threads() { return round32(x_rows<T>() * GPlan<H>::M); }
// Exchange slots of a line: (n1, k2) at k2 (R1 + 1) + n1 for even R1 (an odd stride: both
// steps meet distinct banks), and the row must also hold the H + 1 values of a half row.
template <int L> __host__ __device__ constexpr int xch_stride() { return GPlan<L>::R1 | 1; }
template <int L> __host__ __device__ constexpr int xch_size() { return GPlan<L>::R2 * xch_stride<L>(); }
template <int H> __host__ __device__ constexpr int x_pitch() { return (xch_size<H>() > H + 1 ? xch_size<H>() : H + 1) | 1; }
template <class T, int H> __host__ __device__ constexpr size_t x_smem() { return sizeof(C2<T>) * x_rows<T>() * x_pitch<H>(); }
// Lines per CTA of the y pass (about 256 threads in FP32; 128 in FP64, whose line step
// holds twice the registers)
template <class T, int L> __host__ __device__ constexpr int y_lines() {
  return (sizeof(T) == 4 ? 256 : 128) / GPlan<L>::M < 1 ? 1 : (sizeof(T) == 4 ? 256 : 128) / GPlan<L>::M;
}
template <class T, int L> __host__ __device__ constexpr int y_threads() { return round32(y_lines<T, L>() * GPlan<L>::M); }
// lines R1 slots apart modulo 16, so that the lines of a half-warp fall on distinct banks
template <int L> __host__ __device__ constexpr int y_pitch() {
  int p = xch_size<L>();
  while (GPlan<L>::R1 < 16 && p % 16 != GPlan<L>::R1 % 16) ++p;
  return p;
}
template <class T, int L> __host__ __device__ constexpr size_t y_smem() { return sizeof(C2<T>) * y_lines<T, L>() * y_pitch<L>(); }
// Pencil tile: slot s (0 <= s < L) of a line in row s + s / R1, rows of TW complex values
template <int L> __host__ __device__ constexpr int z_rows() { return L + GPlan<L>::R2; }
// TW: FP32 eight ky (64-byte rows) while two CTAs fit an SM, else four; FP64 four (64-byte
// rows too: the FP64 pipe bounds the pass, so more and smaller tiles cost nothing)
__host__ __device__ constexpr int z_width(int rows, int tsize) { return tsize == 4 && 8 * 6 * rows * 8 <= 112 * 1024 ? 8 : 4; }
template <class T, int L> __host__ __device__ constexpr int z_tw() { return z_width(z_rows<L>(), (int)sizeof(T)); }
// the same for a line length known at run time
inline int z_tile_width(int L, size_t tsize) {
  int R1 = 0, R2 = 0;
  return line_split(L, R1, R2) ? z_width(L + R2, (int)tsize) : 4;
}
template <class T, int L> __host__ __device__ constexpr size_t z_smem() { return sizeof(C2<T>) * 6 * z_rows<L>() * z_tw<T, L>(); }

// ---------------------------------------------------------------- fixed-point and real rows
template <class Q> struct Pair;
template <> struct Pair<int32_t> { using V = int2; };
template <> struct Pair<int64_t> { using V = longlong2; };
template <> struct Pair<float> { using V = float2; };
__device__ __forceinline__ C2<float> to_real(int2 v, float q) { return {__int2float_rn(v.x) * q, __int2float_rn(v.y) * q}; }
__device__ __forceinline__ C2<float> to_real(float2 v, float q) { return {v.x * q, v.y * q}; }
// |v| < 2^51: the integer added to the mantissa of 1.5 * 2^52, then one FP64 subtraction;
// larger values (an eigenstrain above 2^11) by the conversion
__device__ __forceinline__ double ll_to_double(long long v) {
  if ((unsigned long long)(v + (1ll << 51)) < (1ull << 52))
    return __longlong_as_double(v + 0x4338000000000000ll) - 6755399441055744.0;
  return __ll2double_rn(v);
}
__device__ __forceinline__ C2<double> to_real(longlong2 v, double q) { return {ll_to_double(v.x) * q, ll_to_double(v.y) * q}; }

// ---------------------------------------------------------------- x, forward
template <class T, class Q, int H>
__global__ void __launch_bounds__((x_threads<T, H>())) k_x_fwd(const Q* __restrict__ eps, C2<T>* __restrict__ spec, PassCfg c) {
  using G = GPlan<H>;
  constexpr int R1 = G::R1, R2 = G::R2, RB = x_rows<T>(), NT = x_threads<T, H>(), S1 = xch_stride<H>(), PITCH = x_pitch<H>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2<T>* buf = reinterpret_cast<C2<T>*>(smem_raw);  // [RB][PITCH]
  const int plane = plane_of(c.zin, c.nzin, c.nz, blockIdx.y);
  if (plane < 0 || (c.dirty && c.dirty[plane] == 0)) return;
  const int tid = threadIdx.x, y0 = blockIdx.x * RB;
  const C2<T>* __restrict__ tw = reinterpret_cast<const C2<T>*>(c.lwH);
  {
    const int r = tid / R1, n1 = tid % R1;
    if (r < RB) {
      const typename Pair<Q>::V* row = reinterpret_cast<const typename Pair<Q>::V*>(eps + ((size_t)plane * c.ny + y0 + r) * (2 * H));
      C2<T> v[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) v[n2] = to_real(__ldg(row + n1 + R1 * n2), T(c.q));
      gdft<T, R2, false>(v);
      C2<T>* x = buf + r * PITCH + n1;
      x[0] = v[0];
#pragma unroll
      for (int k2 = 1; k2 < R2; ++k2) x[k2 * S1] = v[k2] * tw[k2 * R1 + n1];
    }
  }
  __syncthreads();
  {
    const int r = tid / R2, k2 = tid % R2;
    C2<T> v[R1];
    if (r < RB) {
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) v[n1] = buf[r * PITCH + k2 * S1 + n1];
    }
    __syncthreads();
    if (r < RB) {
      gdft<T, R1, false>(v);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) buf[r * PITCH + k2 + R2 * k1] = v[k1];
    }
  }
  __syncthreads();
  // X[k] = (A + B)/2 - (i/2) w^k (A - B), X[H-k] = conj((A + B)/2 + (i/2) w^k (A - B)) from
  // A = Z[k], B = conj Z[H-k]; consecutive threads take consecutive rows
  const C2<T>* __restrict__ wu = reinterpret_cast<const C2<T>*>(c.lwU);
  C2<T>* out = spec + (size_t)plane * (H + 1) * c.ny + y0;
  for (int i = tid; i < RB * (H / 2 + 1); i += NT) {
    const int r = i % RB, k = i / RB;
    const C2<T> A = buf[r * PITCH + k];
    if (k == 0) {
      out[r] = C2<T>{A.x + A.y, T(0)};
      out[(size_t)H * c.ny + r] = C2<T>{A.x - A.y, T(0)};
      continue;
    }
    const C2<T> B = conjg(buf[r * PITCH + H - k]);
    const C2<T> s = T(0.5) * (A + B), d = wu[k] * (T(0.5) * (A - B));
    out[(size_t)k * c.ny + r] = C2<T>{s.x + d.y, s.y - d.x};
    if (2 * k != H) out[(size_t)(H - k) * c.ny + r] = C2<T>{s.x - d.y, -s.y - d.x};
  }
}

// ---------------------------------------------------------------- x, inverse
template <class T, int H>
__global__ void __launch_bounds__((x_threads<T, H>())) k_x_inv(const C2<T>* __restrict__ spec, T* __restrict__ sig, PassCfg c) {
  using G = GPlan<H>;
  constexpr int R1 = G::R1, R2 = G::R2, RB = x_rows<T>(), NT = x_threads<T, H>(), S1 = xch_stride<H>(), PITCH = x_pitch<H>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2<T>* buf = reinterpret_cast<C2<T>*>(smem_raw);
  const int plane = plane_of(c.zout, c.nzout, c.nz, blockIdx.y);
  if (plane < 0) return;
  const int tid = threadIdx.x, y0 = blockIdx.x * RB;
  const C2<T>* __restrict__ tw = reinterpret_cast<const C2<T>*>(c.lwH);
  const C2<T>* __restrict__ wu = reinterpret_cast<const C2<T>*>(c.lwU);
  const C2<T>* in = spec + (size_t)plane * (H + 1) * c.ny + y0;
  // Z[k] = E + i O, E = X[k] + conj X[H-k], O = (X[k] - conj X[H-k]) exp(+2 pi i k / nx);
  // Z[H-k] = conj(E - i O)
#pragma unroll 4
  for (int i = tid; i < RB * (H / 2 + 1); i += NT) {
    const int r = i % RB, k = i / RB;
    const C2<T> A = in[(size_t)k * c.ny + r];
    const C2<T> B = conjg(in[(size_t)(H - k) * c.ny + r]);
    const C2<T> E = A + B, O = (A - B) * conjg(wu[k]);
    buf[r * PITCH + k] = C2<T>{E.x - O.y, E.y + O.x};
    if (k != 0 && 2 * k != H) buf[r * PITCH + H - k] = C2<T>{E.x + O.y, O.x - E.y};
  }
  __syncthreads();
  {
    const int r = tid / R1, n1 = tid % R1;
    C2<T> v[R2];
    if (r < RB) {
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) v[n2] = buf[r * PITCH + n1 + R1 * n2];
    }
    __syncthreads();
    if (r < RB) {
      gdft<T, R2, true>(v);
      C2<T>* x = buf + r * PITCH + n1;
      x[0] = v[0];
#pragma unroll
      for (int k2 = 1; k2 < R2; ++k2) x[k2 * S1] = v[k2] * conjg(tw[k2 * R1 + n1]);
    }
  }
  __syncthreads();
  {
    const int r = tid / R2, k2 = tid % R2;
    if (r < RB) {
      C2<T> v[R1];
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) v[n1] = buf[r * PITCH + k2 * S1 + n1];
      gdft<T, R1, true>(v);
      C2<T>* row = reinterpret_cast<C2<T>*>(sig + ((size_t)plane * c.ny + y0 + r) * (2 * H));
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) row[k2 + R2 * k1] = v[k1];
    }
  }
}

// ---------------------------------------------------------------- y, in place
template <class T, int L, bool INV>
__global__ void __launch_bounds__((y_threads<T, L>())) k_y(C2<T>* __restrict__ spec, PassCfg c, int nlines) {
  using G = GPlan<L>;
  constexpr int R1 = G::R1, R2 = G::R2, LB = y_lines<T, L>(), S1 = xch_stride<L>(), PITCH = y_pitch<L>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2<T>* buf = reinterpret_cast<C2<T>*>(smem_raw);  // [LB][PITCH]
  const C2<T>* __restrict__ tw = reinterpret_cast<const C2<T>*>(c.lwY);
  // line l of this CTA, or nullptr: past the end, past the plane list, or a clean plane
  auto line = [&](int l) -> C2<T>* {
    const int id = blockIdx.x * LB + l;
    if (l >= LB || id >= nlines) return nullptr;
    const int vp = id / (c.H + 1), kx = id - vp * (c.H + 1);
    const int plane = plane_of(INV ? c.zout : c.zin, INV ? c.nzout : c.nzin, c.nz, vp);
    if (plane < 0 || (!INV && c.dirty && c.dirty[plane] == 0)) return nullptr;
    return spec + ((size_t)plane * (c.H + 1) + kx) * L;
  };
  {
    const int l = threadIdx.x / R1, n1 = threadIdx.x % R1;
    const C2<T>* in = line(l);
    if (in) {
      C2<T> v[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) v[n2] = in[n1 + R1 * n2];
      gdft<T, R2, INV>(v);
      C2<T>* x = buf + l * PITCH + n1;
      x[0] = v[0];
#pragma unroll
      for (int k2 = 1; k2 < R2; ++k2) {
        const C2<T> w = tw[k2 * R1 + n1];
        x[k2 * S1] = v[k2] * (INV ? conjg(w) : w);
      }
    }
  }
  __syncthreads();
  {
    const int l = threadIdx.x / R2, k2 = threadIdx.x % R2;
    C2<T>* out = line(l);
    if (out) {
      C2<T> v[R1];
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) v[n1] = buf[l * PITCH + k2 * S1 + n1];
      gdft<T, R1, INV>(v);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) out[k2 + R2 * k1] = v[k1];
    }
  }
}

// ---------------------------------------------------------------- pencil
// FP64 Green operator at slot frequencies q (the signed frequency over the edge, from
// tables): the operator of sigma_of with the frequency-only factors formed first.  The
// FP64 pipe of this GPU issues two lanes per clock and SM, so the count of FP64
// operations is what the pass costs.
__device__ __forceinline__ void green_apply(const C2<double>* e, double q0, double q1, double q2, const GreenC<double>& C,
                                            const GreenC<double>& Cs, C2<double>* s) {
  using Z = C2<double>;
  auto mul = [](double a, Z b) { return Z{a * b.x, a * b.y}; };
  auto mad = [](double a, Z b, Z c) { return Z{fma(a, b.x, c.x), fma(a, b.y, c.y)}; };
  const double ds = Cs.C11 - Cs.C12, gs = 2.0 * Cs.C44;
  const Z tr = e[0] + e[1] + e[2];
  const Z ct = mul(Cs.C12, tr);
  const Z t0 = mad(ds, e[0], ct), t1 = mad(ds, e[1], ct), t2 = mad(ds, e[2], ct);
  const Z t3 = mul(gs, e[3]), t4 = mul(gs, e[4]), t5 = mul(gs, e[5]);
  const Z v0 = mad(q2, t4, mad(q1, t5, mul(q0, t0)));
  const Z v1 = mad(q2, t3, mad(q1, t1, mul(q0, t5)));
  const Z v2 = mad(q2, t2, mad(q1, t3, mul(q0, t4)));
  const double B = C.C12 + C.C44, AB = C.C11 - C.C44;
  const double a0 = q0 * q0, a1 = q1 * q1, a2 = q2 * q2;
  const double cq = C.C44 * (a0 + a1 + a2);
  const double k00 = fma(AB, a0, cq), k11 = fma(AB, a1, cq), k22 = fma(AB, a2, cq);
  const double b0 = B * q0, k01 = b0 * q1, k02 = b0 * q2, k12 = B * (q1 * q2);
  auto dif = [](double a, double b, double c, double d) { return fma(a, b, -(c * d)); };
  const double i00 = dif(k11, k22, k12, k12), i01 = dif(k02, k12, k01, k22), i02 = dif(k01, k12, k02, k11);
  const double i11 = dif(k00, k22, k02, k02), i12 = dif(k01, k02, k00, k12), i22 = dif(k00, k11, k01, k01);
  const double rd = __drcp_rn(fma(k02, i02, fma(k01, i01, k00 * i00)));
  const Z w0 = mul(rd, mad(i02, v2, mad(i01, v1, mul(i00, v0))));
  const Z w1 = mul(rd, mad(i12, v2, mad(i11, v1, mul(i01, v0))));
  const Z w2 = mul(rd, mad(i22, v2, mad(i12, v1, mul(i02, v0))));
  const Z qw = mad(q2, w2, mad(q1, w1, mul(q0, w0)));
  const double d = C.C11 - C.C12;
  s[0] = mad(d * q0, w0, Z{fma(C.C12, qw.x, -t0.x), fma(C.C12, qw.y, -t0.y)});
  s[1] = mad(d * q1, w1, Z{fma(C.C12, qw.x, -t1.x), fma(C.C12, qw.y, -t1.y)});
  s[2] = mad(d * q2, w2, Z{fma(C.C12, qw.x, -t2.x), fma(C.C12, qw.y, -t2.y)});
  const double g0 = C.C44 * q0, g1 = C.C44 * q1, g2 = C.C44 * q2;
  s[3] = mad(g1, w2, Z{fma(g2, w1.x, -t3.x), fma(g2, w1.y, -t3.y)});
  s[4] = mad(g0, w2, Z{fma(g2, w0.x, -t4.x), fma(g2, w0.y, -t4.y)});
  s[5] = mad(g0, w1, Z{fma(g1, w0.x, -t5.x), fma(g1, w0.y, -t5.y)});
}
__device__ __forceinline__ void green_line(C2<double>* e, int kx, int ky, int kz, const PassCfg& c, double scale) {
  const double q0 = c.fq[kx], q1 = c.fq[c.H + 1 + ky], q2 = c.fq[c.H + 1 + c.ny + kz];
  if (kx == 0 && ky == 0 && kz == 0) {
    green_point<double>(e, kx, ky, kz, c, scale);
    return;
  }
  const GreenC<double> C{c.C11, c.C12, c.C44}, Cs{c.C11 * scale, c.C12 * scale, c.C44 * scale};
  C2<double> s[6];
  green_apply(e, q0, q1, q2, C, Cs, s);
  // on the Nyquist planes the average over the sign of the Nyquist components (green_point)
  const bool nx_ = (kx == c.H), ny_ = (2 * ky == c.ny), nz_ = (2 * kz == c.nz);
  if (nx_ || ny_ || nz_) {
    C2<double> s2[6];
    green_apply(e, nx_ ? -q0 : q0, ny_ ? -q1 : q1, nz_ ? -q2 : q2, C, Cs, s2);
#pragma unroll
    for (int a = 0; a < 6; ++a) s[a] = 0.5 * (s[a] + s2[a]);
  }
#pragma unroll
  for (int a = 0; a < 6; ++a) e[a] = s[a];
}
__device__ __forceinline__ void green_line(C2<float>* e, int kx, int ky, int kz, const PassCfg& c, float scale) {
  green_point<float>(e, kx, ky, kz, c, scale);
}

constexpr int kZThreads = 256;

__device__ __forceinline__ void cp16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem) : "memory");
}

// One tile of TW consecutive ky at one kx: the lines stay in their slots throughout, so
// neither step needs a second buffer.  The forward transform leaves frequency kz = k2 +
// R2 k1 in slot k1 + R1 k2, where the Green operator reads it and the inverse starts from
// it (first over k1, then over k2), back to natural order.  in and out may be one buffer.
template <class T, int L>
__global__ void __launch_bounds__(kZThreads, sizeof(T) == 4 ? 2 : 1) k_z(const C2<T>* in, C2<T>* out, PassCfg c) {
  using G = GPlan<L>;
  constexpr int R1 = G::R1, R2 = G::R2, TW = z_tw<T, L>(), ROWS = z_rows<L>(), V = 16 / (int)sizeof(C2<T>);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2<T>* tile = reinterpret_cast<C2<T>*>(smem_raw);  // [6][ROWS][TW]
  auto row = [](int s) { return s + s / R1; };
  const int tid = threadIdx.x;
  const size_t P = (size_t)(c.H + 1) * c.ny;
  const size_t p0 = (size_t)blockIdx.x * TW;
  const int kx = (int)(p0 / c.ny), ky0 = (int)(p0 % c.ny);
  const int nc = c.ncomp;
  // planes whose transforms the x and y passes have renewed are clean now
  if (c.dirty && blockIdx.x == 0)
    for (int i = tid; i < nc * L; i += kZThreads)
      if (!c.zin || c.zin[1 + L + i % L]) c.dirty[i] = 0;
  for (int i = tid; i < nc * L * (TW / V); i += kZThreads) {
    const int t = (i % (TW / V)) * V, z = (i / (TW / V)) % L, a = i / ((TW / V) * L);
    C2<T>* dst = tile + (a * ROWS + row(z)) * TW + t;
    if (!c.zin || c.zin[1 + L + z]) cp16(dst, in + ((size_t)a * L + z) * P + p0 + t);
    else *reinterpret_cast<float4*>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);  // no eigenstrain in that plane
  }
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
  __syncthreads();
  const C2<T>* __restrict__ tw = reinterpret_cast<const C2<T>*>(c.lwZ);
#pragma unroll 1
  for (int i = tid; i < nc * R1 * TW; i += kZThreads) {
    const int t = i % TW, n1 = (i / TW) % R1, a = i / (TW * R1);
    C2<T>* x = tile + (a * ROWS + n1) * TW + t;
    C2<T> v[R2];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) v[n2] = x[n2 * (R1 + 1) * TW];
    gdft<T, R2, false>(v);
    x[0] = v[0];
#pragma unroll
    for (int k2 = 1; k2 < R2; ++k2) x[k2 * (R1 + 1) * TW] = v[k2] * tw[k2 * R1 + n1];
  }
  __syncthreads();
#pragma unroll 1
  for (int i = tid; i < nc * R2 * TW; i += kZThreads) {
    const int t = i % TW, k2 = (i / TW) % R2, a = i / (TW * R2);
    C2<T>* x = tile + (a * ROWS + k2 * (R1 + 1)) * TW + t;
    C2<T> v[R1];
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) v[n1] = x[n1 * TW];
    gdft<T, R1, false>(v);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) x[k1 * TW] = v[k1];
  }
  __syncthreads();
  if (c.forward_only) {  // frequencies in natural order
    for (int i = tid; i < nc * L * TW; i += kZThreads) {
      const int t = i % TW, kz = (i / TW) % L, a = i / (TW * L);
      const int s = kz / R2 + R1 * (kz % R2);
      out[((size_t)a * L + kz) * P + p0 + t] = tile[(a * ROWS + row(s)) * TW + t];
    }
    return;
  }
  const T scale = T(1) / (T(c.nx) * T(c.ny) * T(c.nz));
#pragma unroll 1
  for (int i = tid; i < L * TW; i += kZThreads) {
    const int t = i % TW, s = i / TW;
    C2<T>* x = tile + row(s) * TW + t;
    C2<T> e[6];
#pragma unroll
    for (int a = 0; a < 6; ++a) e[a] = x[a * ROWS * TW];
    green_line(e, kx, ky0 + t, s / R1 + R2 * (s % R1), c, scale);
#pragma unroll
    for (int a = 0; a < 6; ++a) x[a * ROWS * TW] = e[a];
  }
  __syncthreads();
#pragma unroll 1
  for (int i = tid; i < 6 * R2 * TW; i += kZThreads) {
    const int t = i % TW, k2 = (i / TW) % R2, a = i / (TW * R2);
    C2<T>* x = tile + (a * ROWS + k2 * (R1 + 1)) * TW + t;
    C2<T> v[R1];
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) v[k1] = x[k1 * TW];
    gdft<T, R1, true>(v);
    x[0] = v[0];
#pragma unroll
    for (int n1 = 1; n1 < R1; ++n1) x[n1 * TW] = v[n1] * conjg(tw[k2 * R1 + n1]);
  }
  __syncthreads();
#pragma unroll 1
  for (int i = tid; i < 6 * R1 * TW; i += kZThreads) {
    const int t = i % TW, n1 = (i / TW) % R1, a = i / (TW * R1);
    C2<T>* x = tile + (a * ROWS + n1) * TW + t;
    C2<T> v[R2];
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) v[k2] = x[k2 * (R1 + 1) * TW];
    gdft<T, R2, true>(v);
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) x[n2 * (R1 + 1) * TW] = v[n2];
  }
  __syncthreads();
  for (int i = tid; i < 6 * L * (TW / V); i += kZThreads) {
    const int t = (i % (TW / V)) * V, z = (i / (TW / V)) % L, a = i / ((TW / V) * L);
    if (!c.zout || c.zout[1 + L + z])
      *reinterpret_cast<float4*>(out + ((size_t)a * L + z) * P + p0 + t) =
          *reinterpret_cast<const float4*>(tile + (a * ROWS + row(z)) * TW + t);
  }
}

// ---------------------------------------------------------------- launches
template <class K, class... Args>
inline cudaError_t launch_lines(K k, dim3 grid, int threads, size_t smem, cudaStream_t st, Args... args) {
  cudaError_t e = smem > 48 * 1024 ? cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) : cudaSuccess;
  if (e != cudaSuccess) return e;
  k<<<grid, threads, smem, st>>>(args...);
  return cudaGetLastError();
}

}  // namespace okmc
