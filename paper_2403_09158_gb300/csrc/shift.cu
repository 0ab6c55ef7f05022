// The paper's own evaluation of a defect's interaction energy at continuous positions
// (Sec. 3.3, Eq. shift; Sec. 2 Eq. interaction_energy3 in its elastic-strain form):
//
//   E_i(X) = kappa int sigma^(-i) : eps^e_i(. - X) dV
//          = kappa (h^3 / N) Re sum_xi conj(sigma^(-i)_hat(xi)) : eps^e_ref_hat(xi) exp(-i xi.X)
//
// eps^e_ref is the elastic strain C^-1 : sigma_ref of defect i alone with its class-0
// stencil placed at the origin (its centre at X0 = 0), moved to X by the phase factor of
// the shift theorem and summed by Parseval over the discrete frequencies of Sec. 3.4.
// sigma^(-i) is the stress of everything on the grid except defect i at its current site.
//
// Both spectra come from the Green operator per frequency:
//   sigma^(-i)_hat = G(eps*_hat - alpha_c e W_c(xi) exp(-i xi.b h)),
//   sigma_ref_hat  = G(alpha_0 e W_0(xi)),
// with eps*_hat the transformed eigenstrain of the grid, W_c the transformed count field
// of defect i's class-c stencil at the origin and b its current base voxel.  On the
// stored half spectrum the full sum is, per stored frequency: the kx = 0 and kx = nx/2
// planes once with their own phase; 0 < kx < nx/2 twice, with the phase averaged over the
// sign of the y and z Nyquist components (flipped together), which is the mirror
// frequency's contribution under the Hermitian symmetry of both spectra.
//
// A(xi) = conj(sigma^(-i)_hat) : eps^e_ref_hat does not depend on X and exp(-i xi.X) is a
// product over the axes, so a call forms A once (k_shift_spectrum, over the spectrum it was
// given), tabulates the phases of every axis and position (k_shift_phases), and contracts A
// over ky for all positions at once (k_shift_sum).  The contraction takes the frequencies ky
// and -ky together: with S = A(ky) + A(-ky) and D = A(ky) - A(-ky) the pair contributes
// S cos - i D sin, four real FP64 fma for both.  The FP64 pipe (two lanes per clock and SM)
// bounds the call: 128^3, 121 positions, GB300: 0.26 G fma, 0.44 ms at that rate.  (One pass
// over the spectrum per eight positions, with A and a sincospi per frequency and position
// formed in each, took 16 x 1853 us; the four kernels here take 750 us.)
#include "okmc_internal.cuh"

namespace okmc {

constexpr int kShiftMax = 128;  // positions per pass of the contraction (its threads)

namespace {

constexpr int kShiftThreads = 256;
constexpr int kShiftLines = 8;  // (kx, kz) lines per CTA of the contraction: their sums share a phase load

template <class T>
__device__ __forceinline__ C2<T> scale_c(T s, C2<T> a) {
  return C2<T>{s * a.x, s * a.y};
}

// A(xi) in place of component 0 (FP64: both parts) or components 0 (real part) and 1
// (imaginary part; FP32: a double has the size of a complex value) of the spectrum
template <class T>
__device__ __forceinline__ void put_a(C2<T>* spec, size_t idx, size_t total, double re, double im) {
  if constexpr (sizeof(T) == 8) {
    spec[idx] = C2<T>{re, im};
  } else {
    reinterpret_cast<double*>(spec)[idx] = re;
    reinterpret_cast<double*>(spec + total)[idx] = im;
  }
}
template <class T>
__device__ __forceinline__ double2 get_a(const C2<T>* spec, size_t idx, size_t total) {
  if constexpr (sizeof(T) == 8) return make_double2(spec[idx].x, spec[idx].y);
  else return make_double2(reinterpret_cast<const double*>(spec)[idx], reinterpret_cast<const double*>(spec + total)[idx]);
}

template <class T>
__global__ void __launch_bounds__(kShiftThreads) k_shift_spectrum(C2<T>* spec_e, const C2<T>* __restrict__ spec_w, PassCfg c,
                                                                  const okmc_defect* __restrict__ def,
                                                                  const DefGeo* __restrict__ G,
                                                                  const double* __restrict__ alpha, int i) {
  // exp(-2 pi i (k b mod n) / n) of the current base voxel b, per axis
  __shared__ double2 root[3][512];
  const size_t P = (size_t)(c.H + 1) * c.ny;
  const size_t total = P * c.nz;
  const int pos[3] = {def[i].pos[0], def[i].pos[1], def[i].pos[2]};
  const int cls = pos[0] & 1;
  const int nn[3] = {c.nx, c.ny, c.nz}, cnt[3] = {c.H + 1, c.ny, c.nz};
  for (int a = 0; a < 3; ++a)
    for (int k = threadIdx.x; k < cnt[a]; k += blockDim.x) {
      double s, co;
      sincospi(2.0 * (double)(((long long)k * floor_div2(pos[a])) % nn[a]) / nn[a], &s, &co);
      root[a][k] = make_double2(co, -s);
    }
  __syncthreads();
  const DefGeo g = G[i];
  const T a0 = (T)alpha[2 * i], ac = (T)alpha[2 * i + cls];
  const double C11 = c.C11, C12 = c.C12, C44 = c.C44;
  const double den = (C11 - C12) * (C11 + 2.0 * C12);
  const double S11 = (C11 + C12) / den, S12 = -C12 / den, S44h = 0.5 / C44;  // tensor shear strain = s / (2 C44)
  auto mul = [](double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); };
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total; idx += (size_t)gridDim.x * blockDim.x) {
    const int kz = (int)(idx / P);
    const int p = (int)(idx % P);
    const int kx = p / c.ny, ky = p % c.ny;
    const C2<T> w0 = spec_w[idx];
    const C2<T> wc = spec_w[(size_t)cls * total + idx];
    const double2 r = mul(mul(root[0][kx], root[1][ky]), root[2][kz]);
    const C2<T> wcb{(T)((double)wc.x * r.x - (double)wc.y * r.y), (T)((double)wc.y * r.x + (double)wc.x * r.y)};
    C2<T> ex[6], er[6];
#pragma unroll
    for (int a = 0; a < 6; ++a) {
      const C2<T> e = spec_e[(size_t)a * total + idx];
      const T ea = (T)g.e6[a];
      ex[a] = e - scale_c(ac * ea, wcb);
      er[a] = scale_c(a0 * ea, w0);
    }
    green_point<T>(ex, kx, ky, kz, c, T(1));  // sigma^(-i)_hat
    green_point<T>(er, kx, ky, kz, c, T(1));  // sigma_ref_hat
    // eps^e_ref = C^-1 : sigma_ref (tensor components), then A = conj(sigma^(-i)) : eps^e_ref
    double Ar = 0.0, Ai = 0.0;
#pragma unroll
    for (int a = 0; a < 6; ++a) {
      double erx, ery;
      if (a < 3) {
        const int a1 = (a + 1) % 3, a2 = (a + 2) % 3;
        erx = S11 * er[a].x + S12 * ((double)er[a1].x + er[a2].x);
        ery = S11 * er[a].y + S12 * ((double)er[a1].y + er[a2].y);
      } else {
        erx = 2.0 * S44h * er[a].x;  // factor 2: the off-diagonal pair of a : b
        ery = 2.0 * S44h * er[a].y;
      }
      Ar += (double)ex[a].x * erx + (double)ex[a].y * ery;
      Ai += (double)ex[a].x * ery - (double)ex[a].y * erx;
    }
    put_a(spec_e, idx, total, Ar, Ai);
  }
}

// (cos, sin) of 2 pi f x / n for f = 0 .. n/2 along x, then y, then z, row (axis, f) of
// kShiftMax positions
__global__ void __launch_bounds__(kShiftThreads) k_shift_phases(const double* __restrict__ X, int m, double h, int3 n,
                                                                double2* __restrict__ tab) {
  const int rx = n.x / 2 + 1, ry = n.y / 2 + 1, rz = n.z / 2 + 1;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < (rx + ry + rz) * kShiftMax; i += gridDim.x * blockDim.x) {
    const int k = i % kShiftMax, row = i / kShiftMax;
    const int a = row < rx ? 0 : row < rx + ry ? 1 : 2, f = row - (a == 0 ? 0 : a == 1 ? rx : rx + ry);
    if (k >= m) continue;
    double s, c;
    sincospi(2.0 * ((double)f * (X[3 * k + a] / h) / (a == 0 ? n.x : a == 1 ? n.y : n.z)), &s, &c);
    tab[i] = make_double2(c, s);
  }
}

// partial[CTA][position]: the weighted real parts of kShiftLines lines (kx, kz), one thread
// per position.  Shared memory: S and D of every pair of each line.
template <class T>
__global__ void __launch_bounds__(kShiftMax) k_shift_sum(const C2<T>* __restrict__ spec, PassCfg c, int m,
                                                         const double2* __restrict__ tab, double* __restrict__ partial) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* S = reinterpret_cast<double2*>(smem_raw);  // [ny/2 + 1][kShiftLines]: pairs 1 .. ny/2 - 1; row 0: A(0), row ny/2: A(ny/2)
  const int hy = c.ny / 2;
  double2* D = S + (size_t)(hy + 1) * kShiftLines;
  const size_t P = (size_t)(c.H + 1) * c.ny, total = P * c.nz;
  const int nl = (c.H + 1) * c.nz, l0 = blockIdx.x * kShiftLines;
  for (int i = threadIdx.x; i < (hy + 1) * kShiftLines; i += blockDim.x) {
    const int q = i / (hy + 1), j = i % (hy + 1);
    double2 s = make_double2(0.0, 0.0), d = s;
    if (l0 + q < nl) {  // line l = kz (H + 1) + kx starts at l ny
      const size_t at = (size_t)(l0 + q) * c.ny;
      s = get_a(spec, at + j, total);
      if (j > 0 && j < hy) {
        const double2 b = get_a(spec, at + c.ny - j, total);
        d = make_double2(s.x - b.x, s.y - b.y);
        s = make_double2(s.x + b.x, s.y + b.y);
      }
    }
    S[j * kShiftLines + q] = s;
    D[j * kShiftLines + q] = d;
  }
  __syncthreads();
  const int k = threadIdx.x;
  if (k >= m) return;
  const double2 *tx = tab + k, *ty = tx + (size_t)(c.H + 1) * kShiftMax, *tz = ty + (size_t)(hy + 1) * kShiftMax;
  double2 acc[kShiftLines];
#pragma unroll
  for (int q = 0; q < kShiftLines; ++q) acc[q] = S[q];
#pragma unroll 2
  for (int j = 1; j < hy; ++j) {
    const double2 w = ty[(size_t)j * kShiftMax];
#pragma unroll
    for (int q = 0; q < kShiftLines; ++q) {
      const double2 s = S[j * kShiftLines + q], d = D[j * kShiftLines + q];
      acc[q].x = fma(d.y, w.y, fma(s.x, w.x, acc[q].x));
      acc[q].y = fma(-d.x, w.y, fma(s.y, w.x, acc[q].y));
    }
  }
  auto mul = [](double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); };
  const double2 wn = ty[(size_t)hy * kShiftMax];
  double v = 0.0;
#pragma unroll
  for (int q = 0; q < kShiftLines; ++q) {
    const int l = l0 + q;
    if (l >= nl) break;
    const int kz = l / (c.H + 1), kx = l % (c.H + 1);
    const bool inner = kx > 0 && kx < c.H, zn = 2 * kz == c.nz;
    // exp(-i theta) with the signed frequency (Nyquist: -n/2)
    double2 px = tx[(size_t)kx * kShiftMax], pz = tz[(size_t)(2 * kz < c.nz ? kz : c.nz - kz) * kShiftMax];
    px.y = kx < c.H ? -px.y : px.y;
    pz.y = 2 * kz < c.nz ? -pz.y : pz.y;
    const double2 an = S[hy * kShiftLines + q];
    double2 t;
    if (!inner) {
      t = mul(an, wn);  // exp(-i theta) at f = -ny/2 is cos + i sin
      t = mul(make_double2(acc[q].x + t.x, acc[q].y + t.y), pz);
    } else if (!zn) {  // averaged over the sign of the y Nyquist component: cos
      t = mul(make_double2(fma(an.x, wn.x, acc[q].x), fma(an.y, wn.x, acc[q].y)), pz);
    } else {  // y and z Nyquist components flip together: the real part of the product of phases
      const double cz = pz.x, cn = wn.x * pz.x - wn.y * pz.y;
      t = make_double2(fma(an.x, cn, acc[q].x * cz), fma(an.y, cn, acc[q].y * cz));
    }
    const double r = t.x * px.x - t.y * px.y;
    v += inner ? 2.0 * r : r;
  }
  partial[(size_t)blockIdx.x * kShiftMax + k] = v;
}

// one block per position: a fixed-order sum over the CTAs
__global__ void __launch_bounds__(kShiftThreads) k_shift_final(const double* __restrict__ partial, int nblocks, double scale,
                                                               double* __restrict__ E) {
  __shared__ double sh[kShiftThreads];
  double t = 0.0;
  for (int b = threadIdx.x; b < nblocks; b += kShiftThreads) t += partial[(size_t)b * kShiftMax + blockIdx.x];
  sh[threadIdx.x] = t;
  __syncthreads();
  for (int w = kShiftThreads / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) E[blockIdx.x] = scale * sh[0];
}

size_t phase_rows(const PassCfg& c) { return (size_t)(c.H + 1) + c.ny / 2 + 1 + c.nz / 2 + 1; }
int sum_blocks(const PassCfg& c) { return ((c.H + 1) * c.nz + kShiftLines - 1) / kShiftLines; }

}  // namespace

// Scratch of launch_shift_energies: the phase tables and the partial sums of one pass.  Less
// than a half spectrum of six FP32 components at every grid (16^3: 74 of 110 KB).
size_t shift_scratch_bytes(const PassCfg& c) {
  return phase_rows(c) * kShiftMax * sizeof(double2) + (size_t)sum_blocks(c) * kShiftMax * sizeof(double);
}

// Energies at m positions X (nm, device).  spec_e is overwritten.
template <class T>
cudaError_t launch_shift_energies(C2<T>* spec_e, const C2<T>* spec_w, const PassCfg& c, const okmc_defect* def, const DefGeo* G,
                                  const double* alpha, int i, const double* X, int m, double h, void* scratch, double* E,
                                  cudaStream_t st) {
  const int3 n = make_int3(c.nx, c.ny, c.nz);
  double2* tab = static_cast<double2*>(scratch);
  double* partial = reinterpret_cast<double*>(tab + phase_rows(c) * kShiftMax);
  k_shift_spectrum<T><<<1216, kShiftThreads, 0, st>>>(spec_e, spec_w, c, def, G, alpha, i);
  cudaError_t e = cudaGetLastError();
  const size_t smem = 2 * sizeof(double2) * (size_t)(c.ny / 2 + 1) * kShiftLines;
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_shift_sum<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  const double scale = kKappa * h * h * h / ((double)c.nx * c.ny * c.nz);
  for (int k0 = 0; k0 < m && e == cudaSuccess; k0 += kShiftMax) {
    const int mk = m - k0 < kShiftMax ? m - k0 : kShiftMax;
    k_shift_phases<<<304, kShiftThreads, 0, st>>>(X + 3 * (size_t)k0, mk, h, n, tab);
    k_shift_sum<T><<<sum_blocks(c), (mk + 31) / 32 * 32, smem, st>>>(spec_e, c, mk, tab, partial);
    k_shift_final<<<mk, kShiftThreads, 0, st>>>(partial, sum_blocks(c), scale, E + k0);
    e = cudaGetLastError();
  }
  return e;
}

template cudaError_t launch_shift_energies<float>(C2<float>*, const C2<float>*, const PassCfg&, const okmc_defect*, const DefGeo*,
                                                  const double*, int, const double*, int, double, void*, double*, cudaStream_t);
template cudaError_t launch_shift_energies<double>(C2<double>*, const C2<double>*, const PassCfg&, const okmc_defect*,
                                                   const DefGeo*, const double*, int, const double*, int, double, void*,
                                                   double*, cudaStream_t);

}  // namespace okmc
