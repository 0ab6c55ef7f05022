// Plane passes of the FP32 register-FFT path by tiles: the x and y transforms of all planes in
// one persistent kernel, whose CTAs take x tiles (RB rows of a plane) and y tiles (GL
// columns) in an order in which the second kind follows the first some planes behind, so
// that what passes between them stays in L2.
//
// The cluster kernels of solve_fast.cu move every plane through the shared memory of a
// cluster: two CTAs per SM, barriers between the phases, three quarters of the column
// values over distributed shared memory.  A tile needs about 40 KB and 64 registers a thread
// (80 with DFTs of 20 and 24 points), so four CTAs (three) share an SM at independent
// phases.  DRAM traffic is the same 48 N bytes per pass: the forward x tiles write the
// columns where the y tiles transform them in place; the inverse y tiles write into the
// stress plane itself, tile by tile (RB y values of one kx in a row, an x tile's share of the
// plane contiguous and exactly as large as its stress rows), and the x tiles replace it in
// place.  What bounds it (256^3): 0.54 of the copy bandwidth; barriers and shared-memory latency
// of the steps, with the L2 round trip between the kinds of tile.
// Measured (GB300, every plane, us, cluster kernels' best -> tiles): forward 160^3 96 -> 93,
// 192^3 171 -> 126, 256^3 306 -> 217, 320^3 1041 -> 438; inverse 160^3 93 -> 94, 192^3 160 ->
// 126, 256^3 279 -> 221, 320^3 886 -> 470.  Where a plane fits one CTA (up to 128^3) the cluster
// kernels' single launch stays ahead (128^3 40 against 43): the tuner chooses.
// A form with two buffers per CTA (the next tile's input copied during the current one, three
// tickets ahead, 80 registers) took 560 us at 256^3: its acquire loads and fences stood on
// the path of every tile.
//
// Every line is transformed by the same register DFTs, twiddles and roundings as in the
// cluster kernels (fft_reg.cuh), and column 0 carries (X[0], X[nx/2]) packed as there, so
// results are bitwise the same.
#include "fft_reg.cuh"

namespace okmc {

namespace {

constexpr int kTileThreads = 256;
constexpr unsigned long long kTileWaitNs = 500000000ull;  // 0.5 s: a tile that late has failed

template <int H, int NY>
struct Tiles {
  static constexpr int R1H = RegPlan<H>::R1, R2H = RegPlan<H>::R2, R1Y = RegPlan<NY>::R1, R2Y = RegPlan<NY>::R2;
  static constexpr int RB = NY % 32 == 0 ? 32 : 16;  // rows of an x tile
  static constexpr int TX = NY / RB;
  // columns of a y tile: a line per R1 threads, and no more than an x tile's bytes
  static constexpr int GL = kTileThreads / R1Y * NY <= 4096 || R1Y == 16 ? kTileThreads / R1Y : kTileThreads / R1Y / 2;
  static constexpr int TY = (H + GL - 1) / GL;
  // lines R1 slots apart modulo 16, so that the lines of a half-warp fall on distinct banks
  static constexpr int apart(int p, int r1) {
    while (r1 < 16 && p % 16 != r1 % 16) ++p;
    return p;
  }
  // Exchange slots (n1, k2).  Forward x: slot k2 R1 + n1, rows 34 (18) slots wide: step 1
  // writes along n1 and two rows, step 2 reads along the rows.  Inverse x: slot n1 R2 + k2, 33
  // (17) wide: step 1 writes along the rows, step 2 reads along k2.  y: k2 S + n1, S
  // odd.  No bank is met twice in a half-warp.
  static constexpr int WF = RB + 2, WI = RB + 1;
  static constexpr int SY = R1Y | 1, PY = apart(R2Y * SY, R1Y);
  static constexpr int max(int x, int y) { return x > y ? x : y; }
  static constexpr int BUF = H * WF > GL * PY ? H * WF : GL * PY;
  static constexpr int TAB = tw2_size<H>() + tw2_size<NY>() + H + 1;
  static constexpr size_t SMEM = sizeof(C2<float>) * ((size_t)TAB + BUF + NY);
  // CTAs per SM: four at 64 registers a thread, three at 80 for DFTs of 20 and 24 points
  static constexpr int MINB = R2H > 16 || R2Y > 16 || 4 * (SMEM + 1024) > 228 * 1024 ? 3 : 4;
  static_assert(RB * R1H <= kTileThreads && R2H % 2 == 0 && R1H % 2 == 0, "");
};

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// The planes of a launch: all of them, those of a list (count, planes), or every component's
// planes of a z list.
struct PlaneSet {
  const int* list;
  const int* zl;
  int n, nz;
  __device__ __forceinline__ PlaneSet(const PassCfg& c, const int* plist, const int* z) {
    list = plist;
    zl = plist ? nullptr : z;
    nz = c.nz;
    n = list ? list[0] : zl ? c.ncomp * zl[0] : c.ncomp * c.nz;
  }
  __device__ __forceinline__ int at(int j) const {
    if (list) return list[1 + j];
    if (!zl) return j;
    const int k = zl[0];
    return j / k * nz + zl[1 + j % k];
  }
};

// Tickets.  ctr[0] counts tickets taken, ctr[1] CTAs that have left, ctr[2 + plane] the tiles
// of a plane that are done.  Ticket t stands for tile t % (NA + NB) of plane slot t / (NA +
// NB): the first NA tiles belong to that plane, the others to the plane lag slots before.  A
// tile waits only for tiles of smaller tickets.  A CTA works on the smallest ticket it holds, so
// the smallest unfinished ticket of all is always being worked on and the waits end, whatever
// the number of resident CTAs.  The counters are back at zero when the kernel ends: a plane's
// last tile clears its count, the last CTA to leave the first two.  Only a wait that gave up
// leaves counts of unfinished planes behind, with which the next launch's second tiles could run
// before their inputs are there: the host clears the counters wherever it clears the error
// (clear_error; by the last CTA, behind a fence of every CTA, it took 1.5 us of a 256^3 step).
struct Tile {
  int plane, i;  // plane -1: nothing to do; i counts within its kind
  bool second;
};
template <int NA, int NB>
__device__ __forceinline__ Tile tile_of(int t, int total, int lag, const PlaneSet& ps) {
  if (t >= total) return Tile{-1, 0, false};
  const int j = t / (NA + NB), i = t % (NA + NB);
  const bool second = i >= NA;
  const int slot = second ? j - lag : j;
  return Tile{slot >= 0 && slot < ps.n ? ps.at(slot) : -1, second ? i - NA : i, second};
}
// true once the plane's first NA tiles are done
__device__ __forceinline__ bool wait_tiles(const int* done, int want) {
  if (ld_acquire(done) >= want) return true;
  const unsigned long long t0 = now_ns();
  for (unsigned it = 0; it < (1u << 26); ++it) {
    if (ld_acquire(done) >= want) return true;
    __nanosleep(64);
    if ((it & 63) == 63 && now_ns() - t0 > kTileWaitNs) break;
  }
  return false;
}
template <int H, int NY>
__device__ __forceinline__ void load_tables(C2<float>* twH, C2<float>* twY, C2<float>* untw, const PassCfg& c) {
  fill_tw2<H>(twH, reinterpret_cast<const C2<float>*>(c.ftwH));
  fill_tw2<NY>(twY, reinterpret_cast<const C2<float>*>(c.ftwY));
  const C2<float>* gU = reinterpret_cast<const C2<float>*>(c.ftwU);
  for (int i = threadIdx.x; i <= H; i += kTileThreads) untw[i] = gU[i];
}

// Step 1 of a line's thread n1: the R2-point DFT of v and the twiddles, each value to at(k2)
template <bool INV, int L, class At>
__device__ __forceinline__ void step1(C2<float>* v, const At& at, const C2<float>* tw2, int n1) {
  constexpr int R2 = RegPlan<L>::R2;
  dft_reg<R2, INV>(v);
  *at(0) = v[0];
#pragma unroll
  for (int k2 = 1; k2 < R2; ++k2) {
    C2<float> w = tw2[n1 * (R2 + 1) + k2];
    if (INV) w.y = -w.y;
    *at(k2) = cmul_rn(v[k2], w);
  }
}

// ---------------------------------------------------------------- tiles
// Each tile: step 1 of every line from global memory, the exchange, a barrier, step 2 to
// global memory.
//
// Forward x: step 1 with consecutive threads along a row; step 2 with consecutive threads on
// consecutive rows (the columns' order in memory), each thread taking the frequencies k2 and
// R2 - k2 of its row, which are each other's partners in the untangling, so that the
// untangling happens in registers.
template <int H, int NY>
__device__ __forceinline__ void fwd_x_tile(const int32_t* __restrict__ eps, C2<float>* __restrict__ spec, float q, int plane,
                                           int tile, C2<float>* buf, const C2<float>* twH, const C2<float>* untw) {
  using T = Tiles<H, NY>;
  constexpr int R1 = T::R1H, R2 = T::R2H, RB = T::RB, W = T::WF;
  const int tid = threadIdx.x;
  if (tid < RB * R1) {
    const int r = tid / R1, n1 = tid % R1;
    const int2* row = reinterpret_cast<const int2*>(eps + ((size_t)plane * NY + (size_t)tile * RB + r) * (2 * H)) + n1;
    C2<float> v[R2];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) {
      const int2 e = __ldg(row + R1 * n2);
      v[n2] = C2<float>{__int2float_rn(e.x) * q, __int2float_rn(e.y) * q};
    }
    step1<false, H>(v, [&](int k2) { return buf + (k2 * R1 + n1) * W + r; }, twH, n1);
  }
  __syncthreads();
  C2<float>* col = spec + (size_t)plane * (H + 1) * NY + (size_t)tile * RB;
#pragma unroll 1
  for (int i = tid; i < RB * (R2 / 2); i += kTileThreads) {
    const int r = i % RB, a = i / RB, b = a == 0 ? R2 / 2 : R2 - a;
    C2<float> u[R1], w[R1];
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) u[n1] = buf[(a * R1 + n1) * W + r];
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) w[n1] = buf[(b * R1 + n1) * W + r];
    dft_reg<R1, false>(u);
    dft_reg<R1, false>(w);
    // X[k] = (A + B)/2 - (i/2) w^k (A - B), X[H-k] its mirror, from A = Z[k], B = conj Z[H-k], k <= H/2
    auto put = [&](int k, C2<float> A, C2<float> Zm) {
      const C2<float> B = conjg(Zm);
      const C2<float> sum = A + B, d1 = cmul_rn(untw[k], A - B);
      col[(size_t)k * NY + r] = C2<float>{0.5f * (sum.x + d1.y), 0.5f * (sum.y - d1.x)};
      if (2 * k != H) {
        const C2<float> d2 = conjg(d1);
        col[(size_t)(H - k) * NY + r] = C2<float>{0.5f * (sum.x + d2.y), 0.5f * (-sum.y - d2.x)};
      }
    };
    if (a == 0) {
      col[r] = C2<float>{u[0].x + u[0].y, u[0].x - u[0].y};  // (X[0], X[nx/2])
#pragma unroll
      for (int k1 = 1; k1 < R1 / 2; ++k1) put(R2 * k1, u[k1], u[R1 - k1]);
      put(H / 2, u[R1 / 2], u[R1 / 2]);
#pragma unroll
      for (int k1 = 0; k1 < R1 / 2; ++k1) put(R2 / 2 + R2 * k1, w[k1], w[R1 - 1 - k1]);
    } else {
#pragma unroll
      for (int k1 = 0; k1 < R1 / 2; ++k1) {
        put(a + R2 * k1, u[k1], w[R1 - 1 - k1]);
        put(b + R2 * k1, w[k1], u[R1 - 1 - k1]);
      }
    }
  }
}

// y: columns kx0 .. kx0 + GL - 1 of a plane.  Forward in place (column 0 unpacks into columns 0
// and H); inverse from columns 0 and H packed, into the plane's stress memory: value (kx, y)
// at (y / RB * H + kx) * RB + y % RB.  pk: NY values, the packed column's transform.
template <int H, int NY, bool INV>
__device__ __forceinline__ void y_tile(const C2<float>* in0, C2<float>* base, int tile, C2<float>* buf, C2<float>* pk,
                                       const C2<float>* twY) {
  using T = Tiles<H, NY>;
  constexpr int R1 = T::R1Y, R2 = T::R2Y, GL = T::GL, PY = T::PY, RB = T::RB;
  const int tid = threadIdx.x, kx0 = tile * GL;
  {
    const int l = tid / R1, n1 = tid % R1;
    if (l < GL && kx0 + l < H) {
      const C2<float>* in = in0 + (size_t)(kx0 + l) * NY + n1;
      C2<float> v[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) v[n2] = in[R1 * n2];
      if (INV && kx0 + l == 0) {  // A + i B, columns 0 and H
        const C2<float>* nyq = in0 + (size_t)H * NY + n1;
#pragma unroll
        for (int n2 = 0; n2 < R2; ++n2) {
          const C2<float> B = nyq[R1 * n2];
          v[n2] = C2<float>{v[n2].x - B.y, v[n2].y + B.x};
        }
      }
      step1<INV, NY>(v, [&](int k2) { return buf + l * PY + k2 * T::SY + n1; }, twY, n1);
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int i = tid; i < GL * R2; i += kTileThreads) {
    const int l = i / R2, k2 = i % R2, kx = kx0 + l;
    if (kx >= H) break;
    C2<float> u[R1];
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) u[n1] = buf[l * PY + k2 * T::SY + n1];
    dft_reg<R1, INV>(u);
    if constexpr (INV) {
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) {
        const int y = k2 + R2 * k1;
        base[((size_t)(y / RB) * H + kx) * RB + y % RB] = u[k1];
      }
    } else {
      C2<float>* out = kx == 0 ? pk : base + (size_t)kx * NY;
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) out[k2 + R2 * k1] = u[k1];
    }
  }
  if (!INV && kx0 == 0) {
    __syncthreads();
    // P = A + i B, A and B the spectra of the real columns X[0] and X[nx/2]
    for (int k = tid; k < NY; k += kTileThreads) {
      const C2<float> Pk = pk[k], Pm = conjg(pk[k == 0 ? 0 : NY - k]);
      const C2<float> s = Pk + Pm, d = Pk - Pm;
      base[k] = C2<float>{0.5f * s.x, 0.5f * s.y};
      base[(size_t)H * NY + k] = C2<float>{0.5f * d.y, -0.5f * d.x};
    }
  }
}

// Inverse x, in place in the plane's stress memory: step 1 with consecutive threads on
// consecutive rows (the y tiles' order), step 2 along the rows.
template <int H, int NY>
__device__ __forceinline__ void inv_x_tile(float* __restrict__ sig, int plane, int tile, C2<float>* buf, const C2<float>* twH,
                                           const C2<float>* untw) {
  using T = Tiles<H, NY>;
  constexpr int R1 = T::R1H, R2 = T::R2H, RB = T::RB, W = T::WI;
  const int tid = threadIdx.x;
  C2<float>* rows = reinterpret_cast<C2<float>*>(sig) + ((size_t)plane * NY + (size_t)tile * RB) * H;
  {
    const int r = tid % RB, n1 = tid / RB;
    if (n1 < R1) {
      const C2<float>* x = rows + r;
      C2<float> v[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) {
        const int k = n1 + R1 * n2;
        const C2<float> Xk = x[k * RB];
        if (k == 0) {
          v[n2] = C2<float>{Xk.x + Xk.y, Xk.x - Xk.y};
        } else {
          const C2<float> Xc = conjg(x[(H - k) * RB]);
          const C2<float> E = Xk + Xc;
          const C2<float> O = cmul_rn(conjg(untw[k]), Xk - Xc);
          v[n2] = C2<float>{E.x - O.y, E.y + O.x};
        }
      }
      step1<true, H>(v, [&](int k2) { return buf + (n1 * R2 + k2) * W + r; }, twH, n1);
    }
  }
  __syncthreads();  // every thread has read its share: the rows may be overwritten
#pragma unroll 1
  for (int i = tid; i < RB * R2; i += kTileThreads) {
    const int rr = i / R2, k2 = i % R2;
    C2<float> u[R1];
#pragma unroll
    for (int m = 0; m < R1; ++m) u[m] = buf[(m * R2 + k2) * W + rr];
    dft_reg<R1, true>(u);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) rows[(size_t)rr * H + k2 + R2 * k1] = u[k1];
  }
}

// ---------------------------------------------------------------- the persistent kernels
// Thread 0 holds one ticket ahead, so that the atomic's latency is not waited for, and
// reports a finished tile behind the barrier that starts the next one: the fence runs while
// the other warps load.
template <int H, int NY, bool INV>
__global__ void __launch_bounds__(kTileThreads, (Tiles<H, NY>::MINB))
    k_plane_tiles(const void* __restrict__ in, void* out, PassCfg c, const int* __restrict__ plist, int* __restrict__ ctr) {
  using T = Tiles<H, NY>;
  constexpr int NA = INV ? T::TY : T::TX, NB = INV ? T::TX : T::TY;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_next;
  C2<float>* twH = reinterpret_cast<C2<float>*>(smem_raw);
  C2<float>* twY = twH + tw2_size<H>();
  C2<float>* untw = twY + tw2_size<NY>();
  C2<float>* buf = twH + T::TAB;
  C2<float>* pk = buf + T::BUF;
  const int tid = threadIdx.x;
  load_tables<H, NY>(twH, twY, untw, c);
  const PlaneSet ps(c, plist, INV ? c.zout : c.zin);
  // enough slots behind that the tickets all resident CTAs hold lie between the two kinds
  const int lag = min(ps.n, (2 * (int)gridDim.x + NA + NB - 1) / (NA + NB) + 4);
  const int total = (ps.n + lag) * (NA + NB);
  int rel = -1;  // the plane of a finished tile not yet reported (thread 0)
  auto report = [&] {
    if (tid == 0 && rel >= 0) {
      __threadfence();
      if (atomicAdd(ctr + 2 + rel, 1) == NA + NB - 1) ctr[2 + rel] = 0;  // the plane's last tile
      rel = -1;
    }
  };
  if (tid == 0) s_next = atomicAdd(ctr, 1);
  __syncthreads();
  int t = s_next;
  bool ok = true;
  while (t < total) {
    const Tile k = tile_of<NA, NB>(t, total, lag, ps);
    int next = 0;
    if (tid == 0) next = atomicAdd(ctr, 1);  // arrives while the tile is worked on
    report();
    if (k.plane >= 0) {
      if (k.second) {
        ok = __syncthreads_and(tid == 0 ? wait_tiles(ctr + 2 + k.plane, NA + c.tile_extra) : true);
        if (!ok) break;
      }
      if constexpr (INV) {
        float* plane = (float*)out + (size_t)k.plane * NY * (2 * H);
        if (k.second) inv_x_tile<H, NY>((float*)out, k.plane, k.i, buf, twH, untw);
        else y_tile<H, NY, true>((const C2<float>*)in + (size_t)k.plane * (H + 1) * NY, (C2<float>*)plane, k.i, buf, pk, twY);
      } else {
        C2<float>* plane = (C2<float>*)out + (size_t)k.plane * (H + 1) * NY;
        if (k.second) y_tile<H, NY, false>(plane, plane, k.i, buf, pk, twY);
        else fwd_x_tile<H, NY>((const int32_t*)in, (C2<float>*)out, (float)c.q, k.plane, k.i, buf, twH, untw);
      }
      rel = k.plane;
    }
    __syncthreads();  // the tile's stores, the end of its use of the buffer, every thread's read of s_next
    if (tid == 0) s_next = next;
    __syncthreads();
    t = s_next;
  }
  report();
  if (tid == 0) {
    if (!ok) atomicExch(c.err, 6);
    if (atomicAdd(ctr + 1, 1) == (int)gridDim.x - 1) {
      ctr[0] = 0;
      ctr[1] = 0;
    }
  }
}

// The dirty planes (within the z list, if there is one) in increasing order: count, planes.
// Their flags are cleared: the forward tiles transform exactly these.
__global__ void __launch_bounds__(1024) k_dirty_list(int* __restrict__ dirty, const int* __restrict__ zl, int nplanes, int nz,
                                                     int* __restrict__ out) {
  __shared__ int wsum[32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  int base = 0;
  for (int p0 = 0; p0 < nplanes; p0 += 1024) {
    const int p = p0 + tid;
    const bool f = p < nplanes && dirty[p] != 0 && (!zl || zl[1 + nz + p % nz]);
    const unsigned bal = __ballot_sync(0xffffffffu, f);
    if (lane == 0) wsum[w] = __popc(bal);
    __syncthreads();
    int pre = base;
    for (int q = 0; q < 32; ++q) {
      if (q < w) pre += wsum[q];
      base += wsum[q];
    }
    if (f) {
      out[1 + pre + __popc(bal & ((1u << lane) - 1u))] = p;
      dirty[p] = 0;
    }
    __syncthreads();
  }
  if (tid == 0) out[0] = base;
}

template <int H, int NY, bool INV>
cudaError_t launch_tiles_of(const void* in, void* out, const PassCfg& c, const int* plist, int* ctr, cudaStream_t st) {
  using T = Tiles<H, NY>;
  auto* k = k_plane_tiles<H, NY, INV>;
  // CTAs resident on the device at once (the persistent grid), looked up once
  static const int resident = [&] {
    int dev = 0, sms = 0, per = 0;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T::SMEM) != cudaSuccess ||
        cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, kTileThreads, T::SMEM) != cudaSuccess || per < 1) {
      (void)cudaGetLastError();
      return 152;
    }
    return sms * per;
  }();
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T::SMEM);
  if (e != cudaSuccess) return e;
  const int tiles = c.ncomp * (INV ? c.nzout : c.nzin) * (T::TX + T::TY);
  k<<<resident < tiles ? resident : tiles, kTileThreads, T::SMEM, st>>>(in, out, c, plist, ctr);
  return cudaGetLastError();
}

}  // namespace

// The forward (spec from eps) or inverse (sig from spec) plane pass by tiles.  With dirty
// flags the forward pass takes the dirty planes, listed first by a launch of its own.
cudaError_t launch_plane_tiles(bool inverse, const void* in, void* out, const PassCfg& c, cudaStream_t st) {
  const int* plist = nullptr;
  if (!inverse && c.dirty) {
    k_dirty_list<<<1, 1024, 0, st>>>(c.dirty, c.zin, c.ncomp * c.nz, c.nz, c.plist);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    plist = c.plist;
  }
  switch (c.ny) {
#define OKMC_CASE(n, h)                                                                  \
  case n:                                                                                \
    return inverse ? launch_tiles_of<h, n, true>(in, out, c, plist, c.tile_ctr, st)      \
                   : launch_tiles_of<h, n, false>(in, out, c, plist, c.tile_ctr, st);
    OKMC_CASE(32, 16) OKMC_CASE(48, 24) OKMC_CASE(64, 32) OKMC_CASE(96, 48) OKMC_CASE(128, 64) OKMC_CASE(160, 80)
    OKMC_CASE(192, 96) OKMC_CASE(256, 128) OKMC_CASE(320, 160)
#undef OKMC_CASE
    default: return cudaErrorInvalidConfiguration;
  }
}

}  // namespace okmc
