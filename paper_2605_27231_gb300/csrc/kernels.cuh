// Device kernels of the lattice SIGW path, templated on the working precision T
// (float or double) and the lattice size N.  Included by one translation unit per
// precision, which instantiates them and defines the sigw::Ops launchers.
//
// Layouts (b = realisation in the batch, H = N/2, NH = N/2 + 1):
//   real       R[b][a0][a1][a2]                      N^3 values
//   standard   X[b][k0][k1][k2], k2 = 0..H           the usual half spectrum (Phi~ is kept this way)
//   packed     Y[b][a0|k0][a1|k1][c], c = 0..H-1     column 0 holds (k2 = 0) + i (k2 = H); this is
//              exact because both planes are transforms of real 2-D fields, and it makes every
//              strided pass run over exactly H columns.
// Lattice wave numbers: index k -> n = k for k <= H, k - N otherwise (index H is +N/2).
// The derivative factor uses n^D = 0 on the Nyquist index H.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <type_traits>

#include "fft.cuh"
#include "noise.cuh"
#include "ops.h"

namespace sigw {

__device__ __forceinline__ int wrapn(int k, int N) { return k <= (N >> 1) ? k : k - N; }
__device__ __forceinline__ int derivn(int k, int N) { return k == (N >> 1) ? 0 : wrapn(k, N); }

// ---------------------------------------------------------------- shapes
template <typename T, int N> struct Shape {
  static constexpr int H = N / 2;
  // strided passes: E values per thread, TC columns per CTA
  static constexpr int ES = (sizeof(T) == 4) ? (N >= 256 ? 16 : (N >= 16 ? 8 : 4)) : (N >= 16 ? 8 : 4);
  static constexpr int PS = N / ES;
  static constexpr int TC0 = 256 / PS;
  static constexpr int TC = TC0 < 1 ? 1 : (TC0 > H ? H : TC0);
  // row passes: E values per thread, RPC rows per CTA
  static constexpr int ER = (N >= 16) ? 8 : 4;
  static constexpr int PR = N / ER;
  static constexpr int RPC0 = 256 / PR;
  static constexpr int RPC = RPC0 > (N * N / 2) ? (N * N / 2) : RPC0;
  // forward-a0 + TT pass keeps six spectra per thread: fewer values per thread
  static constexpr int E3 = (sizeof(T) == 4) ? (N >= 16 ? 8 : 4) : 4;
  static constexpr int P3 = N / E3;
  static constexpr int TC3_0 = 256 / P3;
  static constexpr int TC3_1 = TC3_0 < 1 ? 1 : (TC3_0 > 8 ? 8 : TC3_0);
  static constexpr int TC3 = TC3_1 * P3 < 32 ? 32 / P3 : TC3_1;  // whole warps (the partial sum uses shuffles)
};

// Alternative radix of the first strided inverse pass (variant bit 1): FP32, N >= 128 only.  At N = 512 the alternative
// is radix 32 (two stages, one exchange, 16-column tiles) instead of radix 16 (three stages).
template <typename T, int N> struct AltStrided {
  static constexpr bool exists = sizeof(T) == 4 && N >= 128;
  static constexpr int E = N == 512 ? 32 : (Shape<T, N>::ES == 16 ? 8 : 16);
  static constexpr int P = N / E;
  static constexpr int TC0 = 256 / P;
  static constexpr int TC = TC0 > N / 2 ? N / 2 : TC0;
};

// Column-tile exchange layout of the strided passes: one buffer when E >= 32 (a radix-32 pencil of 512
// points would otherwise need 128 KB for a 16-column tile).
template <typename T, int N, int TC, int E> using StridedLay = ColLayout<T, N, TC, E, (E >= 32)>;

// Second strided pass: E values per thread and TCL columns per CTA.  TCL is also the column tile of the first pass's
// output T[b][term][a0][column tile][k1][TCL], so that a CTA's input is one contiguous block (one bulk copy).
template <typename T, int N> struct Pass2 {
  static constexpr int E = sizeof(T) == 4 && N == 128 ? 16 : Shape<T, N>::ES;
  static constexpr int TCL = Shape<T, N>::TC;
  static constexpr int THREADS = TCL * (N / E);
  // a field's first transform waits for the second in tensor memory (FP32, N >= 128)
  static constexpr bool ZTM = sizeof(T) == 4 && E == 16;
};
// Place of (k1, cc) in a plane a0 of T.
template <typename T, int N> __device__ __forceinline__ int t_index(int k1, int cc) {
  constexpr int TCL = Pass2<T, N>::TCL;
  return (cc / TCL) * (N * TCL) + k1 * TCL + cc % TCL;
}

template <int P> struct RowSync { using type = SyncWarp; };
template <> struct RowSync<64> { using type = SyncBlock; };
template <> struct RowSync<128> { using type = SyncBlock; };

// ================================================================ synthesis chain
// Two real rows (2q, 2q+1) share one complex FFT: z = x1 + i x2, Z = DFT z,
// X1(k) = (Z(k) + Z*(N-k))/2, X2(k) = -i/2 (Z(k) - Z*(N-k)).
// MODE 0: rows from R;  MODE 1: Philox noise;  MODE 2: R through the NG map;  MODE 3: R squared.
// The non-local map (kind 3) also reads lap(zeta_g) from R2 and lap(zeta_g^2) from R3 (same layout as R).
template <typename T, int N, int MODE>
__global__ void __launch_bounds__(256) k_rows_r2c(const T* __restrict__ R, cx<T>* __restrict__ Y,
                                                  const cx<T>* __restrict__ tw, const uint64_t* __restrict__ seeds,
                                                  const MapArgs* __restrict__ maps, const double* __restrict__ mean,
                                                  unsigned long long* __restrict__ hits, const T* __restrict__ R2,
                                                  const T* __restrict__ R3) {
  using SH = Shape<T, N>;
  constexpr int E = SH::ER, P = SH::PR, H = N / 2;
  constexpr int PPC = SH::RPC;  // row pairs per CTA
  using Sync = typename RowSync<P>::type;
  using Lay = RowLayout<T, N>;
  extern __shared__ __align__(16) unsigned char smraw[];
  const Lay L{reinterpret_cast<cx<T>*>(smraw) + (threadIdx.x / P) * Lay::SIZE};
  const int j = threadIdx.x % P;
  const int b = blockIdx.y;
  const long pair = (long)blockIdx.x * PPC + threadIdx.x / P;
  const bool live = pair < (long)N * N / 2;
  const long row0 = 2 * pair;
  cx<T> v[E];
  unsigned long long myhits = 0;
  double mu = 0.0;
  MapArgs map{0, 0.0, 0.0, 0.0};
  if (MODE == 2) {
    mu = mean[b];
    map = maps[b];
  }
#pragma unroll
  for (int r = 0; r < E; ++r) {
    const int x = j + r * P;
    T x1 = 0, x2 = 0;
    if (live) {
      if (MODE == 1) {
        const uint64_t sd = seeds[b];
        if constexpr (sizeof(T) == 4) {
          x1 = gauss_draw_f32((uint32_t)(row0 * N + x), sd);
          x2 = gauss_draw_f32((uint32_t)((row0 + 1) * N + x), sd);
        } else {
          x1 = gauss_draw((uint32_t)(row0 * N + x), sd);
          x2 = gauss_draw((uint32_t)((row0 + 1) * N + x), sd);
        }
      } else {
        const long ro = ((long)b * N * N + row0) * N;
        const T* rb = R + ro;
        x1 = rb[x];
        x2 = rb[N + x];
        if (MODE == 3) {
          x1 = x1 * x1;
          x2 = x2 * x2;
        }
        if (MODE == 2) {
          T z[2] = {x1, x2};
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const T g = z[q];
            if (map.kind == 1) {
              z[q] = g + (T)map.F * (g * g - (T)mu) + (T)map.G * g * g * g;
            } else if (map.kind == 3) {
              const long o = ro + (long)q * N + x;
              z[q] = g + (T)map.F * R3[o] + (T)map.G * g * R2[o];
            } else if (map.kind == 2) {
              T arg = (T)1 - (T)3 * g;
              if (arg < (T)map.floor) {
                ++myhits;
                arg = (T)map.floor;
              }
              z[q] = -log(arg) / (T)3;
            }
          }
          x1 = z[0];
          x2 = z[1];
        }
      }
    }
    v[r] = mk<T>(x1, x2);
  }
  if (MODE == 2 && map.kind == 2) {
    // warp-reduce the hit count, one atomic per warp
    for (int o = 16; o > 0; o >>= 1) myhits += __shfl_down_sync(0xffffffffu, myhits, o);
    if ((threadIdx.x & 31) == 0 && myhits) atomicAdd(hits + b, myhits);
  }
  fft_pencil<T, N, E, -1, Lay, Sync>(v, j, L, tw, Sync());
  cx<T>* zb = L.buf(0);
#pragma unroll
  for (int r = 0; r < E; ++r) zb[L.idx(j + r * P)] = v[r];
  Sync()();
  if (live) {
    cx<T>* y1 = Y + ((long)b * N * N + row0) * H;
    cx<T>* y2 = y1 + H;
#pragma unroll
    for (int r = 0; r < E / 2; ++r) {
      const int c = j + r * P;
      if (c == 0) {
        const cx<T> z0 = zb[L.idx(0)];
        const cx<T> zh = zb[L.idx(H)];
        y1[0] = mk<T>(z0.x, zh.x);
        y2[0] = mk<T>(z0.y, zh.y);
      } else {
        const cx<T> zc = zb[L.idx(c)];
        const cx<T> zm = conjg<T>(zb[L.idx(N - c)]);
        y1[c] = mk<T>((T)0.5 * (zc.x + zm.x), (T)0.5 * (zc.y + zm.y));
        y2[c] = mk<T>((T)0.5 * (zc.y - zm.y), (T)-0.5 * (zc.x - zm.x));
      }
    }
  }
}

// Packed half rows -> real rows (two rows per complex inverse FFT), scaled by `scale`.
// With SQ, per-CTA FP64 partial sums of the squared outputs go to sq_partial[b][blockIdx.x].
template <typename T, int N, bool SQ>
__global__ void __launch_bounds__(256) k_rows_c2r(const cx<T>* __restrict__ Y, T* __restrict__ R, T scale,
                                                  double* __restrict__ sq_partial, const cx<T>* __restrict__ tw) {
  using SH = Shape<T, N>;
  constexpr int E = SH::ER, P = SH::PR, H = N / 2;
  constexpr int PPC = SH::RPC;
  using Sync = typename RowSync<P>::type;
  using Lay = RowLayout<T, N>;
  extern __shared__ __align__(16) unsigned char smraw[];
  const Lay L{reinterpret_cast<cx<T>*>(smraw) + (threadIdx.x / P) * Lay::SIZE};
  __shared__ double red[32];
  const int j = threadIdx.x % P;
  const int b = blockIdx.y;
  const long pair = (long)blockIdx.x * PPC + threadIdx.x / P;
  const bool live = pair < (long)N * N / 2;
  const long row0 = 2 * pair;
  const cx<T>* y1 = Y + ((long)b * N * N + row0) * H;
  const cx<T>* y2 = y1 + H;
  cx<T> v[E];
#pragma unroll
  for (int r = 0; r < E; ++r) {
    const int k = j + r * P;
    cx<T> a = mk<T>(0, 0), c = mk<T>(0, 0);
    if (live) {
      if (k == 0) {
        a = mk<T>(y1[0].x, 0);
        c = mk<T>(y2[0].x, 0);
      } else if (k == H) {
        a = mk<T>(y1[0].y, 0);
        c = mk<T>(y2[0].y, 0);
      } else if (k < H) {
        a = y1[k];
        c = y2[k];
      } else {
        a = conjg<T>(y1[N - k]);
        c = conjg<T>(y2[N - k]);
      }
    }
    v[r] = mk<T>(a.x - c.y, a.y + c.x);  // a + i c
  }
  fft_pencil<T, N, E, +1, Lay, Sync>(v, j, L, tw, Sync());
  double sq = 0.0;
  if (live) {
    T* r1 = R + ((long)b * N * N + row0) * N;
#pragma unroll
    for (int r = 0; r < E; ++r) {
      const int x = j + r * P;
      const T u = v[r].x * scale, w = v[r].y * scale;
      r1[x] = u;
      r1[N + x] = w;
      if (SQ) sq += (double)u * (double)u + (double)w * (double)w;
    }
  }
  if (SQ) {
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_down_sync(0xffffffffu, sq, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sq;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < (int)(blockDim.x + 31) / 32; ++w) t += red[w];
      sq_partial[(long)b * gridDim.x + blockIdx.x] = t;
    }
  }
}

// In-place C2C transforms along axis 0 (AX = 0, stride N*H) or axis 1 (AX = 1, stride H) of a packed array.
template <typename T, int N, int DIR, int AX>
__global__ void __launch_bounds__(256) k_pass(cx<T>* __restrict__ Y, const cx<T>* __restrict__ tw) {
  using SH = Shape<T, N>;
  constexpr int E = SH::ES, P = SH::PS, TC = SH::TC, H = N / 2;
  using Lay = ColLayout<T, N, TC, E, true>;  // one exchange buffer: more CTAs share an SM
  extern __shared__ __align__(16) unsigned char smraw[];
  const int c = threadIdx.x % TC, j = threadIdx.x / TC;
  const Lay L{reinterpret_cast<cx<T>*>(smraw), c};
  const int col = blockIdx.x * TC + c;
  const int o = blockIdx.y;
  const int b = blockIdx.z;
  const long stride = AX == 0 ? (long)N * H : (long)H;
  const long ostride = AX == 0 ? (long)H : (long)N * H;
  cx<T>* base = Y + (long)b * N * N * H + o * ostride + col;
  cx<T> v[E];
#pragma unroll
  for (int r = 0; r < E; ++r) v[r] = base[(j + r * P) * stride];
  fft_pencil<T, N, E, DIR, Lay, SyncBlock, false>(v, j, L, tw, SyncBlock());
#pragma unroll
  for (int r = 0; r < E; ++r) base[(j + r * P) * stride] = v[r];
}

// Packed -> standard.  MODE 0 (synthesis): times amp[|n|^2] * factor, zero on k = 0 and the Nyquist planes.
// MODE 1: times factor.
template <typename T, int MODE>
__global__ void k_unpack(const cx<T>* __restrict__ Y, cx<T>* __restrict__ X, int N, const T* __restrict__ amp,
                         long amp_bstride, T factor, long total) {
  const int H = N / 2, NH = H + 1;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
    const int k2 = (int)(i % NH);
    const long q = i / NH;
    const int k1 = (int)(q % N);
    const long q2 = q / N;
    const int k0 = (int)(q2 % N);
    const long b = q2 / N;
    cx<T> val;
    if (k2 >= 1 && k2 < H) {
      val = Y[((b * N + k0) * N + k1) * H + k2];
    } else {
      const cx<T> yk = Y[((b * N + k0) * N + k1) * H];
      const cx<T> ym = Y[((b * N + ((N - k0) & (N - 1))) * N + ((N - k1) & (N - 1))) * H];
      if (k2 == 0)
        val = mk<T>((T)0.5 * (yk.x + ym.x), (T)0.5 * (yk.y - ym.y));
      else
        val = mk<T>((T)0.5 * (yk.y + ym.y), (T)-0.5 * (yk.x - ym.x));
    }
    if (MODE == 0) {
      const int n0 = wrapn(k0, N), n1 = wrapn(k1, N);
      const int msq = n0 * n0 + n1 * n1 + k2 * k2;
      const bool zero = (k0 == H) || (k1 == H) || (k2 == H) || msq == 0;
      const T a = zero ? (T)0 : amp[b * amp_bstride + msq] * factor;
      val = mk<T>(val.x * a, val.y * a);
    } else {
      val = mk<T>(val.x * factor, val.y * factor);
    }
    X[i] = val;
  }
}

// Inverse C2C transforms along axis 0 from the standard half spectrum X into the packed array Y: column 0 takes
// X(k2 = 0) + i X(k2 = H).  With LAP each value is first multiplied by -lap |n|^2 (the spectral Laplacian for
// lap = k_f^2; a Nyquist index counts as n = +N/2, which is exact for the second derivative).  (A pass of its own for the
// packing read and wrote the whole spectrum once more: inverse transform at 256^3 FP32 105 us, now 78 to 84.)
template <typename T, int N, bool LAP>
__global__ void __launch_bounds__(256) k_pass_pack(const cx<T>* __restrict__ X, cx<T>* __restrict__ Y, double lap,
                                                   const cx<T>* __restrict__ tw) {
  using SH = Shape<T, N>;
  constexpr int E = SH::ES, P = SH::PS, TC = SH::TC, H = N / 2, NH = H + 1;
  using Lay = ColLayout<T, N, TC, E, true>;  // one exchange buffer: more CTAs share an SM
  extern __shared__ __align__(16) unsigned char smraw[];
  const int c = threadIdx.x % TC, j = threadIdx.x / TC;
  const Lay L{reinterpret_cast<cx<T>*>(smraw), c};
  const int col = blockIdx.x * TC + c;
  const int k1 = blockIdx.y;
  const long b = blockIdx.z;
  const cx<T>* src = X + ((b * N + j) * N + k1) * NH + col;  // + r P N NH
  cx<T> v[E];
#pragma unroll
  for (int r = 0; r < E; ++r) v[r] = src[(long)r * P * N * NH];
  const int n1 = wrapn(k1, N);
  if (LAP) {
#pragma unroll
    for (int r = 0; r < E; ++r) {
      const int n0 = wrapn(j + r * P, N);
      v[r] = scale<T>(v[r], (T)(-lap * (double)(n0 * n0 + n1 * n1 + col * col)));
    }
  }
  if (col == 0) {
#pragma unroll
    for (int r = 0; r < E; ++r) {
      cx<T> h = src[(long)r * P * N * NH + H];
      if (LAP) {
        const int n0 = wrapn(j + r * P, N);
        h = scale<T>(h, (T)(-lap * (double)(n0 * n0 + n1 * n1 + H * H)));
      }
      v[r] = mk<T>(v[r].x - h.y, v[r].y + h.x);
    }
  }
  fft_pencil<T, N, E, +1, Lay, SyncBlock, false>(v, j, L, tw, SyncBlock());
  cx<T>* dst = Y + ((b * N + j) * N + k1) * H + col;
#pragma unroll
  for (int r = 0; r < E; ++r) dst[(long)r * P * N * H] = v[r];
}

#ifdef SIGW_COMMON_KERNELS
__global__ void k_reduce_mean(const double* __restrict__ part, int nblk, double* __restrict__ mean, double inv) {
  const int b = blockIdx.x;
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < nblk; ++i) t += part[(long)b * nblk + i];
    mean[b] = t * inv;
  }
}
#endif

// ================================================================ hot path
// P1: first inverse pass along axis 0 for a tile of TC packed columns at fixed k1.
//   V_a(n) = phi_a(cell(|n|^2)) Phi~(n)          (column 0: V(k2=0) + i V(k2=H), each with its own cell)
//   Ta_a = IDFT_0[V_a],  Tb_a = IDFT_0[i n0^D V_a]
// The nb terms of a launch are split over nag CTAs per tile (blockIdx.z = b * nag + group), see p1_groups.  With
// swz = 8 the column index is stored as cc ^ (8 (k1 mod 2)) (the fused second and last pass reads it that way).
template <typename T, int N, int E_ = Shape<T, N>::ES, int TC_ = Shape<T, N>::TC>
__global__ void __launch_bounds__(256) k_p1(const cx<T>* __restrict__ phi, cx<T>* __restrict__ Ta,
                                            cx<T>* __restrict__ Tb, const int16_t* __restrict__ lut,
                                            const T* __restrict__ phitab, int nm1, int alpha0, int nb, int nag,
                                            int swz, const cx<T>* __restrict__ tw) {
  constexpr int E = E_, P = N / E_, TC = TC_, H = N / 2, NH = H + 1;
  using Lay = StridedLay<T, N, TC, E>;
  extern __shared__ __align__(16) unsigned char smraw[];
  cx<T>* sm_nyq = reinterpret_cast<cx<T>*>(smraw) + Lay::SIZE;  // N values (column 0 only)
  int* sm_cn = reinterpret_cast<int*>(sm_nyq + N);              // N cells
  T* sm_tab = reinterpret_cast<T*>(sm_cn + N);                  // (terms of this CTA) * nm1
  const int c = threadIdx.x % TC, j = threadIdx.x / TC;
  const Lay L{reinterpret_cast<cx<T>*>(smraw), c};
  const int cc = blockIdx.x * TC + c;
  const int k1 = blockIdx.y;
  const int b = blockIdx.z / nag, ag = blockIdx.z % nag;
  const int alo = (int)((long)nb * ag / nag), ahi = (int)((long)nb * (ag + 1) / nag);  // terms of this CTA
  const int n1 = wrapn(k1, N);
  for (int i = threadIdx.x; i < (ahi - alo) * nm1; i += blockDim.x) sm_tab[i] = phitab[(long)(alpha0 + alo) * nm1 + i];
  const cx<T>* pb = phi + ((long)b * N * N + k1) * NH;  // + k0 * N * NH + k2
  if (blockIdx.x == 0) {
    for (int k0 = threadIdx.x; k0 < N; k0 += blockDim.x) {
      const int n0 = wrapn(k0, N);
      sm_nyq[k0] = pb[(long)k0 * N * NH + H];
      sm_cn[k0] = lut[n0 * n0 + n1 * n1 + H * H];
    }
  }
  cx<T> ph[E];
  int cell[E];
#pragma unroll
  for (int r = 0; r < E; ++r) {
    const int k0 = j + r * P;
    const int n0 = wrapn(k0, N);
    ph[r] = pb[(long)k0 * N * NH + cc];
    cell[r] = lut[n0 * n0 + n1 * n1 + cc * cc];
  }
  __syncthreads();
  const long fstride = (long)N * N * H;  // one field
  const T fj = (T)j;
  const int cs = cc ^ ((k1 & 1) * swz);
  for (int a = alo; a < ahi; ++a) {
    const T* tab = sm_tab + (a - alo) * nm1;
    // D = 0: V_a; D = 1: i n0 V_a.  V_a is formed again for the second transform instead of being kept,
    // so only one value array is live next to the Phi~ tile.
#pragma unroll 1
    for (int D = 0; D < 2; ++D) {
      cx<T> v[E];
#pragma unroll
      for (int r = 0; r < E; ++r) {
        const T f = tab[cell[r]];
        cx<T> x = mk<T>(f * ph[r].x, f * ph[r].y);
        if (cc == 0) {
          const int k0 = j + r * P;
          const T fn = tab[sm_cn[k0]];
          const cx<T> yn = sm_nyq[k0];
          x = mk<T>(x.x - fn * yn.y, x.y + fn * yn.x);
        }
        if (D) {  // n^D(k0) for k0 = j + r P: j < P, so k0 < N/2 exactly when r < E/2 (Nyquist: r = E/2, j = 0)
          const T nd = r < E / 2 ? fj + (T)(r * P) : ((r == E / 2 && j == 0) ? (T)0 : fj + (T)(r * P - N));
          x = mk<T>(-nd * x.y, nd * x.x);
        }
        v[r] = x;
      }
      fft_pencil<T, N, E, +1, Lay, SyncBlock>(v, j, L, tw, SyncBlock());
      cx<T>* dst = (D ? Tb : Ta) + ((long)b * nb + a) * fstride + t_index<T, N>(k1, cs);
#pragma unroll
      for (int r = 0; r < E; ++r) dst[(long)(j + r * P) * N * H] = v[r];
    }
  }
}

// Rows handed from the second to the last inverse pass: for term pair (a, a + 1) and every (a0, a1) three full complex
// rows over k2, the inputs of the last pass's three complex transforms:
//   f = 0: g2^a + i g1^a      f = 1: the same of a + 1      f = 2: g0^a + i g0^{a+1}       W[b][pair][f][a0][a1][N]
// Element c < N/2 of a row is the value at k2 = c, element N - 1 - c the one at k2 = -c; element N - 1 is the value at
// k2 = N/2.  All rows carry a common factor -1 (the products do not see it), which saves sign changes in k_p2.
// With 64-bit values at N = 128 the index is xor-ed with 8 on odd rows: a half warp of the radix-16 last pass reads two
// rows there, and they then fall into different banks (see k_p3_tm).
template <typename T, int N> struct ZRow {
  static constexpr int SWZ = sizeof(T) == 4 && N == 128 ? 8 : 0;
};

// ---------------------------------------------------------------- bulk-copy pipeline helpers
// cp.async.bulk (TMA, 1-D) global -> shared with mbarrier completion.  Waits are bounded: after `limit` clock
// cycles (about a second by default) the wait sets *err and gives up, so a lost copy can never hang the GPU.
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// With the default limit the wait uses try_wait, which may suspend the thread for a while inside the instruction;
// with a shorter limit (a test's) it polls with the non-blocking test_wait and looks at the clock first, so that a tiny
// limit gives up however soon the copy lands.  The default looks at the barrier first: a thread that was switched out for
// longer than the limit finds its copy.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int* err, int bit,
                                          long long limit = kDefaultWaitLimit) {
  const uint32_t a = smem_u32(bar);
  const long long t0 = clock64();
  const bool poll = limit < kDefaultWaitLimit;
  while (true) {
    uint32_t done;
    if (poll) {
      if (clock64() - t0 > limit) break;
      asm volatile(
          "{ .reg .pred p; mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
          : "=r"(done)
          : "r"(a), "r"(parity)
          : "memory");
    } else {
      asm volatile(
          "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
          : "=r"(done)
          : "r"(a), "r"(parity)
          : "memory");
    }
    if (done) return true;
    if (!poll && clock64() - t0 > limit) break;
  }
  atomicOr(err, bit);
  return false;
}

template <typename T, int N, int E_ = ((N >= 16) ? 8 : 4)> struct P3Cfg {
  static constexpr int H = N / 2;
  static constexpr int E = E_;
  static constexpr int P = N / E;
  static constexpr int STAGES = 2;
  using Lay = RowLayout<T, N, true, 4>;  // single exchange buffer per row
  static constexpr size_t smem_for(int rpc) {
    return (size_t)STAGES * 6 * rpc * H * sizeof(cx<T>) + (size_t)rpc * Lay::SIZE * sizeof(cx<T>) +
           STAGES * sizeof(uint64_t);
  }
  // A 32 KB bulk copy per row block.  On the small lattices 64 threads: a realisation at N = 32 then has 64 CTAs (times
  // seven groups of term pairs) instead of 16 or 8 (FP64, 50 terms: 976 -> 131 us).
  static constexpr int RPC0 = N <= 32 ? 64 / P : 16384 / (H * (int)sizeof(cx<T>));
  static constexpr int RPC1 = RPC0 > N * N ? N * N : RPC0;
  static constexpr int RPC = smem_for(RPC1) <= 227 * 1024 ? RPC1 : RPC1 / 2;
  static constexpr int THREADS = RPC * P;
  static constexpr int STAGE_ELEMS = 3 * RPC * N;  // the three row blocks of a term pair
  static constexpr size_t SMEM = smem_for(RPC);
  static_assert(SMEM <= 227 * 1024, "shared memory");
};

// Radix-16 alternative of the last inverse pass (autotuner variant bit 2), FP32.  N = 128, 256: one
// shared-memory exchange per transform instead of two.  N = 512: two exchanges either way, but a row is one
// warp (P = 32), so the exchanges need warp barriers only (the radix-8 form uses 64 threads and block barriers).
template <typename T, int N> struct AltP3 {
  static constexpr bool exists = sizeof(T) == 4 && (N == 128 || N == 256 || N == 512);
  static constexpr int E = 16;
};

// Transform input k = j + r P (0 <= j < P, r unrolled) of a row written by k_p2; par: the row's parity.
template <typename T, int N, int E>
__device__ __forceinline__ cx<T> zrow(const cx<T>* row, int j, int r, int par) {
  constexpr int P = N / E, SWZ = ZRow<T, N>::SWZ;
  const bool hz = (r == E / 2) && (j == 0);  // k = N/2
  if constexpr (SWZ == 0) {
    return row[r < E / 2 ? j + r * P : (hz ? N - 1 : j + r * P - 1)];
  } else if constexpr (P == 8) {  // the xor moves by one register index: constant offsets from two bases
    const int sx = (r & 1) ? -8 * par : 8 * par;
    if (r < E / 2) return row[j + sx + r * P];
    return row[hz ? N - 1 - 8 * par : j - 1 + (j == 0 ? -sx : sx) + r * P];
  } else {
    return row[(r < E / 2 ? j + r * P : (hz ? N - 1 : j + r * P - 1)) ^ (SWZ * par)];
  }
}
// One term's contribution sigma g_i g_j to the six product components at one point, with zz = (g2, g1):
// a0 = s_00, a21 = (s_22, s_11), a43 = (s_02, s_01), a5 = s_12.  PAIRED (FP32, N <= 256) uses paired (FP32x2)
// multiply-adds; at N = 512 their aligned register pairs made the radix-16 last pass spill, so it stays scalar.
template <typename T, bool PAIRED>
__device__ __forceinline__ void accum6(T sa, T g0, cx<T> zz, T& a0, cx<T>& a21, cx<T>& a43, T& a5) {
  const T s0 = sa * g0;
  const cx<T> t = mk<T>(sa * zz.x, sa * zz.y);
  a21 = mk<T>(fma(t.x, zz.x, a21.x), fma(t.y, zz.y, a21.y));
  a43 = mk<T>(fma(s0, zz.x, a43.x), fma(s0, zz.y, a43.y));
  a0 = fma(s0, g0, a0);
  a5 = fma(t.y, zz.x, a5);
}
template <>
__device__ __forceinline__ void accum6<float, true>(float sa, float g0, float2 zz, float& a0, float2& a21,
                                                    float2& a43, float& a5) {
  const float s0 = sa * g0;
  const float2 t = __fmul2_rn(zz, make_float2(sa, sa));
  a21 = __ffma2_rn(t, zz, a21);
  a43 = __ffma2_rn(make_float2(s0, s0), zz, a43);
  a0 = __fmaf_rn(s0, g0, a0);
  a5 = __fmaf_rn(t.y, zz.x, a5);
}

// P3: last inverse pass (axis 2, C2R) of all terms for RPC consecutive rows, the product
//   s_ij(x) = sum_a sigma_a g^a_i(x) g^a_j(x)  (six components in registers),
// then the forward R2C of s_ij along axis 2 keeping k2 = 0..n_c, written to F[b][comp][a0][a1][k2].
// Term pair (a, a+1) uses three complex transforms: (g2^a + i g1^a), (g0^a + i g0^{a+1}), (g2^{a+1} + i g1^{a+1}),
// whose inputs are the rows of W.  The rows of a term pair stream into a STAGES-deep shared-memory ring by cp.async.bulk,
// issued STAGES-1 pairs ahead by thread 0.  Bounded waits: the main loop's waits give up after wait_limit cycles
// (normally kDefaultWaitLimit; a test passes a tiny limit, so that waits give up while the copies still land).
// A thread whose wait gave up sets *err, stops waiting and (thread 0) stops issuing copies; before the CTA exits,
// thread 0 waits, with the default limit, for the last copy issued into each stage, so no bulk copy can still be
// writing into the CTA's shared memory after it has exited.  The results of a launch that set *err are invalid.
template <typename T, int N, int E_ = ((N >= 16) ? 8 : 4)>
__global__ void __launch_bounds__(P3Cfg<T, N, E_>::THREADS, 1) k_p3(const cx<T>* __restrict__ W,
                                                                   const T* __restrict__ sigma, int n_alpha,
                                                                   cx<T>* __restrict__ F, long fgstride, int n_c,
                                                                   const cx<T>* __restrict__ tw,
                                                                   int* __restrict__ err, long long wait_limit) {
  using CF = P3Cfg<T, N, E_>;
  constexpr int E = CF::E, P = CF::P, H = N / 2, RPC = CF::RPC, STAGES = CF::STAGES;
  using Sync = typename RowSync<P>::type;
  using Lay = typename CF::Lay;
  extern __shared__ __align__(128) unsigned char smraw[];
  cx<T>* ring = reinterpret_cast<cx<T>*>(smraw);
  cx<T>* xch = ring + STAGES * CF::STAGE_ELEMS;
  uint64_t* bars = reinterpret_cast<uint64_t*>(xch + RPC * Lay::SIZE);
  const int rr = threadIdx.x / P, j = threadIdx.x % P;
  const Lay L{xch + rr * Lay::SIZE};
  const long row0 = (long)blockIdx.x * RPC;
  const long row = row0 + rr;
  const int b = blockIdx.y;
  const long fstride = (long)N * N * N;
  // term pairs pr0 .. pr0 + npairs - 1 (blockIdx.z of gridDim.z groups; each group writes its own partial F)
  const int allpairs = (n_alpha + 1) / 2;
  const int pr0 = allpairs * (int)blockIdx.z / (int)gridDim.z;
  const int npairs = allpairs * ((int)blockIdx.z + 1) / (int)gridDim.z - pr0;
  F += (long)blockIdx.z * fgstride;
  constexpr uint32_t COPY = RPC * N * sizeof(cx<T>);
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) mbar_init(bars + s, 1);
    mbar_init_fence();
  }
  __syncthreads();
  auto issue = [&](int pr) {  // thread 0: the row blocks of term pair pr into stage pr % STAGES
    const int s = pr % STAGES;
    const bool two = 2 * (pr0 + pr) + 1 < n_alpha;
    cx<T>* dst = ring + s * CF::STAGE_ELEMS;
    fence_proxy_async();
    mbar_expect_tx(bars + s, (two ? 3u : 2u) * COPY);
    for (int f = 0; f < 3; ++f)
      if (f != 1 || two)
        bulk_g2s(dst + f * RPC * N, W + (((long)b * allpairs + pr0 + pr) * 3 + f) * fstride + row0 * N, COPY, bars + s);
  };
  if (threadIdx.x == 0)
    for (int pr = 0; pr < STAGES - 1 && pr < npairs; ++pr) issue(pr);
  T a0[E], a5[E];
  cx<T> a21[E], a43[E];
#pragma unroll
  for (int r = 0; r < E; ++r) {
    a0[r] = a5[r] = (T)0;
    a21[r] = a43[r] = mk<T>((T)0, (T)0);
  }
  const int par = (int)(row & 1);
  bool ok = true;
  int issued = STAGES - 1 < npairs ? STAGES - 1 : npairs;  // term pairs whose copies thread 0 has issued
  for (int pr = 0; pr < npairs; ++pr) {
    const int s = pr % STAGES;
    if (threadIdx.x == 0 && ok && pr + STAGES - 1 < npairs) {
      issue(pr + STAGES - 1);
      issued = pr + STAGES;
    }
    if (ok) ok = mbar_wait(bars + s, (uint32_t)((pr / STAGES) & 1), err, kWaitLast, wait_limit);
    const int a = 2 * (pr0 + pr);
    const bool two = a + 1 < n_alpha;
    const cx<T>* z0 = ring + s * CF::STAGE_ELEMS + rr * N;  // f = 0, 1, 2 follow RPC rows apart
    // (g0^a + i g0^{a+1}) first; its two real parts are kept while the other two transforms run
    cx<T> zB[E], z[E];
#pragma unroll
    for (int r = 0; r < E; ++r) zB[r] = zrow<T, N, E>(z0 + 2 * RPC * N, j, r, par);
    fft_pencil<T, N, E, +1, Lay, Sync>(zB, j, L, tw, Sync());
    const T sa = sigma[a];
#pragma unroll
    for (int r = 0; r < E; ++r) z[r] = zrow<T, N, E>(z0, j, r, par);
    fft_pencil<T, N, E, +1, Lay, Sync>(z, j, L, tw, Sync());
#pragma unroll
    for (int r = 0; r < E; ++r) accum6<T, (sizeof(T) == 4 && N <= 256)>(sa, zB[r].x, z[r], a0[r], a21[r], a43[r], a5[r]);
    if (two) {  // uniform across the CTA
      const T sb = sigma[a + 1];
#pragma unroll
      for (int r = 0; r < E; ++r) z[r] = zrow<T, N, E>(z0 + RPC * N, j, r, par);
      fft_pencil<T, N, E, +1, Lay, Sync>(z, j, L, tw, Sync());
#pragma unroll
      for (int r = 0; r < E; ++r) accum6<T, (sizeof(T) == 4 && N <= 256)>(sb, zB[r].y, z[r], a0[r], a21[r], a43[r], a5[r]);
    }
    __syncthreads();  // stage s fully read before it is refilled
  }
  if (threadIdx.x == 0) {
    // The last copy issued into each stage has landed before the CTA may exit (immediate when every wait
    // succeeded; after a wait gave up, the copies still in flight are waited for with the default limit).
    for (int s = 0; s < STAGES && s < issued; ++s) {
      const int last = s + ((issued - 1 - s) / STAGES) * STAGES;
      mbar_wait(bars + s, (uint32_t)((last / STAGES) & 1), err, kWaitLast);
    }
  }
  // forward R2C of the six real rows (00, 11 | 22, 01 | 02, 12), two per complex transform
  cx<T>* zb = L.buf(0);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    cx<T> z[E];
#pragma unroll
    for (int r = 0; r < E; ++r)
      z[r] = q == 0 ? mk<T>(a0[r], a21[r].y) : (q == 1 ? mk<T>(a21[r].x, a43[r].y) : mk<T>(a43[r].x, a5[r]));
    fft_pencil<T, N, E, -1, Lay, Sync>(z, j, L, tw, Sync());
#pragma unroll
    for (int r = 0; r < E; ++r) zb[L.idx(j + r * P)] = z[r];
    Sync()();
    const int ncp = n_c + 1;
    cx<T>* f1 = F + (((long)b * 6 + 2 * q) * N * N + row) * ncp;
    cx<T>* f2 = F + (((long)b * 6 + 2 * q + 1) * N * N + row) * ncp;
    for (int k = j; k <= n_c; k += P) {
      const cx<T> zk = zb[L.idx(k)];
      const cx<T> zm = conjg<T>(zb[L.idx((N - k) & (N - 1))]);
      f1[k] = mk<T>((T)0.5 * (zk.x + zm.x), (T)0.5 * (zk.y + zm.y));
      f2[k] = mk<T>((T)0.5 * (zk.y - zm.y), (T)-0.5 * (zk.x - zm.x));
    }
    Sync()();
  }
}

// ---------------------------------------------------------------- tensor memory (TMEM) helpers
// A CTA allocates NCOLS 32-bit columns of the SM's tensor memory (128 lanes x 512 columns) with one warp, keeps
// per-thread values in its own lane (warp w may access lanes 32 (w mod 4) .. 32 (w mod 4) + 31), and frees them
// with the same warp before it exits.  No tensor-core instruction is involved: the memory is used as storage.
__device__ __forceinline__ void tmem_alloc(uint32_t* dst_smem, uint32_t ncols) {  // whole warp
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {  // whole warp
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// 16 consecutive columns of this thread's lane into registers; the load and its completion wait are one
// statement, so no use of the values can be scheduled before the wait.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16};" ::"r"(taddr),
      "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
      "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])),
      "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
      "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])), "r"(__float_as_uint(v[15]))
      : "memory");
}
// 32 consecutive columns of this thread's lane into registers (one wait).
__device__ __forceinline__ void tmem_ld32(uint32_t t0, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(t0)
      : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const float (&v)[32]) {
  uint32_t r[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(v[i]);
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
      "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
      "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}

__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Two-stage inverse pencil transform of N = 16 R points (R = 8, 16: N = 128, 256), radix 16 then radix R, with the
// last stage's twiddles held in tensor memory.  Thread j of a pencil needs the same NB (R - 1) twiddles
// W^{-r k}, k = (j + t P) mod 16 (t < NB = 16 / R, 0 < r < R), in every transform of a launch; tw_tm_store writes
// them once into 32 columns of its lane (twiddle q = t (R - 1) + r - 1 in columns 2q, 2q + 1), and
// fft_pencil_tw_tm reads them with two tensor-memory loads instead of NB (R - 1) table loads.  Its first stage
// writes an exchange row in 16-byte pairs where the layout has them (RowLayoutV).  Same arithmetic, in the same order, as
// fft_pencil<float, N, 16, +1>.
template <int N> struct TwTm {
  static constexpr int E = 16, P = N / E, R = N / E, NB = E / R;
  static_assert(R >= 2 && R <= E && NB * (R - 1) <= 16, "two stages, at most 16 twiddles");
};
template <int N>
__device__ __forceinline__ void tw_tm_store(uint32_t taddr, int j, const float2* __restrict__ tw) {
  using C = TwTm<N>;
  float w[2][16];
#pragma unroll
  for (int i = 0; i < 16; ++i) w[0][i] = w[1][i] = 0.f;
#pragma unroll
  for (int t = 0; t < C::NB; ++t) {
    const int k = (j + t * C::P) & 15;
#pragma unroll
    for (int r = 1; r < C::R; ++r) {
      const int q = t * (C::R - 1) + r - 1;
      const float2 x = conjg<float>(__ldg(tw + r * k));  // stride N / (16 R) = 1
      w[q >> 3][2 * (q & 7)] = x.x;
      w[q >> 3][2 * (q & 7) + 1] = x.y;
    }
  }
  tmem_st16(taddr, w[0]);
  tmem_st16(taddr + 16, w[1]);
}
template <int N, typename Lay, typename Sync>
__device__ __forceinline__ void fft_pencil_tw_tm(float2 (&v)[16], int j, const Lay& L, uint32_t tw_taddr, Sync sync) {
  using C = TwTm<N>;
  constexpr int E = C::E, P = C::P, R = C::R, NB = C::NB;
  static_assert(Lay::SINGLE, "one exchange buffer");
  float2* x = L.buf(0);
  dftR<float, +1, E>(v);
  if constexpr (Lay::VEC) {
#pragma unroll
    for (int m = 0; m < E / 2; ++m)
      *reinterpret_cast<float4*>(x + L.idx(j * E + 2 * m)) =
          make_float4(v[2 * m].x, v[2 * m].y, v[2 * m + 1].x, v[2 * m + 1].y);
  } else {
#pragma unroll
    for (int r = 0; r < E; ++r) x[L.idx(j * E + r)] = v[r];
  }
  sync();
  float w[32];
  tmem_ld32(tw_taddr, w);
#pragma unroll
  for (int t = 0; t < NB; ++t) {
    const int jj = j + t * P;
    float2 a[R];
#pragma unroll
    for (int r = 0; r < R; ++r) a[r] = x[L.idx(jj + r * (N / R))];
#pragma unroll
    for (int r = 1; r < R; ++r) {
      const int q = t * (R - 1) + r - 1;
      a[r] = mul<float>(a[r], make_float2(w[2 * q], w[2 * q + 1]));
    }
    dftR<float, +1, R>(a);
#pragma unroll
    for (int r = 0; r < R; ++r) v[t + r * NB] = a[r];
  }
  sync();  // the row may be rewritten at once
}
// As fft_pencil<float, N, 16, +1> for a two-stage transform, with the first 8 of the thread's last-stage twiddles
// (q = t (R - 1) + r - 1 < 8, same order as TwTm) taken from 16 columns of its tensor-memory lane (written once by
// tw8_tm_store) and the others from the table.  Any exchange layout.
template <int N>
__device__ __forceinline__ void tw8_tm_store(uint32_t taddr, int j, const float2* __restrict__ tw) {
  using C = TwTm<N>;
  float w[16];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int t = q / (C::R - 1), r = q % (C::R - 1) + 1;
    const float2 x = conjg<float>(__ldg(tw + r * ((j + t * C::P) & 15)));
    w[2 * q] = x.x;
    w[2 * q + 1] = x.y;
  }
  tmem_st16(taddr, w);
}
template <int N, typename Lay, typename Sync>
__device__ __forceinline__ void fft_pencil_tw8_tm(float2 (&v)[16], int j, const Lay& L, const float2* __restrict__ tw,
                                                  uint32_t tw_taddr, Sync sync) {
  using C = TwTm<N>;
  constexpr int E = C::E, P = C::P, R = C::R, NB = C::NB;
  float2* x = L.buf(0);
  dftR<float, +1, E>(v);
#pragma unroll
  for (int r = 0; r < E; ++r) x[L.idx(j * E + r)] = v[r];
  sync();
  float w[16];
  tmem_ld16(tw_taddr, w);
#pragma unroll
  for (int t = 0; t < NB; ++t) {
    const int jj = j + t * P;
    const int k = jj & 15;
    float2 a[R];
#pragma unroll
    for (int r = 0; r < R; ++r) a[r] = x[L.idx(jj + r * (N / R))];
#pragma unroll
    for (int r = 1; r < R; ++r) {
      const int q = t * (R - 1) + r - 1;
      const float2 wr = q < 8 ? make_float2(w[2 * q], w[2 * q + 1]) : twiddle<float, +1>(tw, r * k);
      a[r] = mul<float>(a[r], wr);
    }
    dftR<float, +1, R>(a);
#pragma unroll
    for (int r = 0; r < R; ++r) v[t + r * NB] = a[r];
  }
  sync();  // the exchange buffer may be rewritten at once
}

// P2: second inverse pass along axis 1 at fixed a0, for one term pair.  Two column transforms give a field's two rows:
//   f = 0, 1:  B = IDFT_1[n1^D Ta], A = IDFT_1[Ta]      (G1 = i B, G2 = i n2 A)
//              U = -(G2 + i G1) at k2 >= 0,              V = -conj(G2 - i G1), the same at -k2
//   f = 2:     A = IDFT_1[Tb^a], B = IDFT_1[Tb^{a+1}]:   U = -(A + i B),   V = -conj(A - i B)
// i.e. six column transforms for six half spectra, as if the fields themselves were stored; the last pass then
// reads each transform input with one access and no arithmetic.  It is bound by its shared-memory accesses, this pass
// by HBM: storing the fields and assembling there cost 96 instead of 48 reads a thread and pair (four realisations at
// 256^3, 50 terms: last pass 6.94 -> 6.04 ms, this pass 10.2 ms either way, 6.6 TB/s).  The first transform
// of a field waits in tensor memory (FP32, N >= 128) or in the shared memory of its tile.
//
// A CTA takes the pairs of one of nag groups for its tile of columns.  Its input tiles (N rows x TCL columns of a field,
// contiguous) come through a ring of two by bulk copy.  A tile is read from shared memory for both transforms that need
// it, and its slot is refilled as soon as it is free, at least one transform (2.6 us at 256^3) before the new tile is
// needed: with both tiles of f = 2 used by one transform the next pair's first copy was waited for (11.3 ms).  FP32, N = 128 and 256: the last-stage twiddles sit in tensor memory.
// Bounded waits, error flag and the drain before exit as in k_p3.
template <typename T, int N> struct P2Cfg {
  static constexpr int E = Pass2<T, N>::E, TC = Pass2<T, N>::TCL, THREADS = Pass2<T, N>::THREADS;
  using Lay = ColLayout<T, N, TC, E, true>;  // one exchange buffer
  static constexpr int TILE = N * TC;
  static constexpr size_t SMEM = (size_t)(Lay::SIZE + 2 * TILE) * sizeof(cx<T>) + 32;
  static constexpr int CTAS = THREADS > 128 ? 2 : 4;
  static constexpr bool FSPLIT = N <= 32;  // few tiles: the three fields of a pair go to three CTAs
  static constexpr bool TWTM = sizeof(T) == 4 && E == 16 && (N == 128 || N == 256);
  static constexpr bool ZTM = Pass2<T, N>::ZTM;
  static constexpr uint32_t NCOLS = 64 * ((THREADS + 127) / 128);  // a warp's share: 32 for each of the two
};

template <typename T, int N>
__global__ void __launch_bounds__(P2Cfg<T, N>::THREADS, P2Cfg<T, N>::CTAS) k_p2(
    const cx<T>* __restrict__ Ta, const cx<T>* __restrict__ Tb, cx<T>* __restrict__ W, int npairs, int alpha0, int nb,
    int nag, const cx<T>* __restrict__ tw, int* __restrict__ err, long long wait_limit) {
  using CF = P2Cfg<T, N>;
  constexpr int E = CF::E, P = N / E, TC = CF::TC, H = N / 2, SWZ = ZRow<T, N>::SWZ;
  constexpr uint32_t COPY = CF::TILE * sizeof(cx<T>);
  using Lay = typename CF::Lay;
  extern __shared__ __align__(128) unsigned char smraw[];
  cx<T>* const ring = reinterpret_cast<cx<T>*>(smraw);
  cx<T>* const xch = ring + 2 * CF::TILE;
  uint64_t* const bars = reinterpret_cast<uint64_t*>(xch + Lay::SIZE);
  uint32_t* const tslot = reinterpret_cast<uint32_t*>(bars + 2);
  const int c = threadIdx.x % TC, j = threadIdx.x / TC;
  const Lay L{xch, c};
  const int cc = blockIdx.x * TC + c;
  const int a0 = blockIdx.y;
  const int b = blockIdx.z / nag, g = CF::FSPLIT ? blockIdx.z % nag / 3 : blockIdx.z % nag;
  const int fs = CF::FSPLIT ? blockIdx.z % nag % 3 : 0;  // the one field of this CTA
  const int npl = (nb + 1) / 2;  // pairs of this launch (alpha0 is even)
  const int p0 = CF::FSPLIT ? g : npl * g / nag, p1 = CF::FSPLIT ? g + 1 : npl * (g + 1) / nag;
  const int nt = min(2 * p1, nb) - 2 * p0;  // terms of this CTA
  if (CF::FSPLIT && fs == 1 && nt == 1) return;
  const long fstride = (long)N * N * H;
  const T n2 = (T)cc, fj = (T)j;
  const int sw = SWZ * (j & 1);  // P is even: the parity of the row a1 = j + r P (and of N - a1)
  // input tiles in order of use: Ta^a, Ta^{a+1}, Tb^a, Tb^{a+1} of every pair (Ta^a, Tb^a of a single last term)
  const int ntiles = !CF::FSPLIT ? 2 * nt : (fs == 2 ? nt : 1);
  const long toff = ((long)b * nb + 2 * p0) * fstride + (long)a0 * N * H + (long)blockIdx.x * CF::TILE;
  auto issue = [&](int q) {  // thread 0: tile q into slot q % 2
    const bool pair = nt - 2 * (q >> 2) >= 2;
    const int e = q & 3, term = CF::FSPLIT ? (fs == 2 ? q : fs) : 2 * (q >> 2) + (pair ? (e & 1) : 0);
    const bool isa = CF::FSPLIT ? fs < 2 : (pair ? e < 2 : e < 1);
    fence_proxy_async();
    mbar_expect_tx(bars + (q & 1), COPY);
    bulk_g2s(ring + (q & 1) * CF::TILE, (isa ? Ta : Tb) + toff + term * fstride, COPY, bars + (q & 1));
  };
  uint32_t twt = 0;
  if (threadIdx.x == 0) {
    mbar_init(bars, 1);
    mbar_init(bars + 1, 1);
    mbar_init_fence();
    issue(0);
    if (ntiles > 1) issue(1);
  }
  if constexpr (CF::ZTM) {
    const int warp = threadIdx.x >> 5;
    if (warp == 0) tmem_alloc(tslot, CF::NCOLS);
    tmem_fence_before_sync();
    __syncthreads();
    tmem_fence_after_sync();
    twt = *tslot + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(64 * (warp >> 2));
    if constexpr (CF::TWTM) {
      tw_tm_store<N>(twt, j, tw);
      tmem_wait_st();
    }
  } else {
    __syncthreads();
  }
  int issued = ntiles > 1 ? 2 : 1;  // tiles thread 0 has issued
  bool ok = true;
  int q = 0;  // tiles used up
  for (int lp = 0; 2 * lp < nt; ++lp) {
    const bool two = nt - 2 * lp >= 2;
    cx<T>* const w0 = W + (((long)b * npairs + alpha0 / 2 + p0 + lp) * 3 * N + a0) * (long)N * N;
    cx<T> hold[E];  // without tensor memory: the first transform of a field until its stash is free
#pragma unroll 1
    for (int t = 0; t < 6; ++t) {
      const int f = t >> 1, s = t & 1;
      if (!two && (f == 1 || t == 5)) continue;
      if (CF::FSPLIT && f != fs) continue;
      const bool last = s == 1 || !two && f == 2;  // this transform completes the field's two rows
      if (s == 0 || f == 2)                        // its tile has arrived
        if (ok) ok = mbar_wait(bars + (q & 1), (uint32_t)((q >> 1) & 1), err, kWaitSecond, wait_limit);
      cx<T>* const x0 = ring + (q & 1) * CF::TILE + j * TC + c;
      cx<T> v[E];
#pragma unroll
      for (int r = 0; r < E; ++r) v[r] = x0[r * P * TC];
      if (f < 2 && s == 0) {
#pragma unroll
        for (int r = 0; r < E; ++r) {
          const T nd = r < E / 2 ? fj + (T)(r * P) : ((r == E / 2 && j == 0) ? (T)0 : fj + (T)(r * P - N));
          v[r] = scale<T>(v[r], nd);
        }
      }
      // the stash of a thread without tensor memory: its own places of the field's first tile, read for the last time
      cx<T>* const stash = ring + ((f == 2 ? q - 1 : q) & 1) * CF::TILE + j * TC + c;
      if constexpr (!CF::ZTM) {
        if (s == 1) {
#pragma unroll
          for (int r = 0; r < E; ++r) stash[r * P * TC] = hold[r];
        }
      }
      if constexpr (CF::TWTM) fft_pencil_tw_tm<N, Lay, SyncBlock>(v, j, L, twt, SyncBlock());
      else fft_pencil<T, N, E, +1, Lay, SyncBlock>(v, j, L, tw, SyncBlock());
      if (CF::ZTM && (s == 1 || f == 2)) {  // every thread has read this tile: refill its slot
        if (threadIdx.x == 0 && ok && q + 2 < ntiles) {
          issue(q + 2);
          issued = q + 3;
        }
        ++q;
      }
      cx<T> h[E];  // the field's first transform
      if constexpr (CF::ZTM) {
        float w[32];
        if (!last) {
#pragma unroll
          for (int r = 0; r < E; ++r) {
            w[2 * r] = v[r].x;
            w[2 * r + 1] = v[r].y;
          }
          tmem_st32(twt + 32, w);
          tmem_wait_st();
          continue;
        }
        if (s == 1) {
          tmem_ld32(twt + 32, w);
#pragma unroll
          for (int r = 0; r < E; ++r) h[r] = make_float2(w[2 * r], w[2 * r + 1]);
        }
      } else {
        if (!last) {
#pragma unroll
          for (int r = 0; r < E; ++r) hold[r] = v[r];
          if (f == 2) ++q;
          continue;
        }
        if (s == 1) {
#pragma unroll
          for (int r = 0; r < E; ++r) h[r] = stash[r * P * TC];
        }
      }
      if (s == 0) {  // a single last term: Tb^{a+1} = 0
#pragma unroll
        for (int r = 0; r < E; ++r) {
          h[r] = v[r];
          v[r] = mk<T>((T)0, (T)0);
        }
      }
      cx<T>* const o = w0 + (long)f * N * N * N + j * N;
      const int pu = cc ^ sw, pv = (N - 1 - cc) ^ sw;
      if (cc == 0) {  // packed column, k2 = 0 and k2 = N/2 (n2^D = 0 on both)
        if (f < 2) {
#pragma unroll
          for (int r = 0; r < E; ++r) {
            o[r * P * N + pu] = mk<T>((T)0, h[r].y);
            o[r * P * N + pv] = mk<T>((T)0, -h[r].x);
          }
        } else {
#pragma unroll
          for (int r = 0; r < E; ++r) {
            o[r * P * N + pu] = mk<T>(-h[r].x, -v[r].x);
            o[r * P * N + pv] = mk<T>(-h[r].y, -v[r].y);
          }
        }
      } else if (f < 2) {
#pragma unroll
        for (int r = 0; r < E; ++r) {
          o[r * P * N + pu] = mk<T>(n2 * v[r].y + h[r].x, h[r].y - n2 * v[r].x);
          o[r * P * N + pv] = mk<T>(n2 * v[r].y - h[r].x, h[r].y + n2 * v[r].x);
        }
      } else {
#pragma unroll
        for (int r = 0; r < E; ++r) {
          o[r * P * N + pu] = mk<T>(v[r].y - h[r].x, -h[r].y - v[r].x);
          o[r * P * N + pv] = mk<T>(-h[r].x - v[r].y, h[r].y - v[r].x);
        }
      }
      if constexpr (!CF::ZTM) {  // every thread has read its stash: refill the field's slots
        __syncthreads();
        const int q0 = (f == 2 && two) ? q - 1 : q;
        ++q;
        if (threadIdx.x == 0 && ok)
          for (int u = q0; u < q; ++u)
            if (u + 2 < ntiles) {
              issue(u + 2);
              issued = u + 3;
            }
      }
    }
  }
  if (threadIdx.x == 0) {  // the last copy issued into each slot has landed before the CTA may exit
    mbar_wait(bars + ((issued - 1) & 1), (uint32_t)(((issued - 1) >> 1) & 1), err, kWaitSecond);
    if (issued > 1) mbar_wait(bars + ((issued - 2) & 1), (uint32_t)(((issued - 2) >> 1) & 1), err, kWaitSecond);
  }
  if constexpr (CF::ZTM) {
    tmem_fence_before_sync();
    __syncthreads();
    tmem_fence_after_sync();
    if (threadIdx.x < 32) tmem_dealloc(*tslot, CF::NCOLS);
  }
}


// P3 with its accumulators in tensor memory (autotuner variant bit 8; FP32, radix 16, N = 128, 256, 512).  The last pass
// above keeps the six product components of its 16 points per thread in registers (96 of its 254), which holds
// it to one CTA of 8 warps per SM.  Here they live in TMEM, in the thread's lane: s00 in columns 0-15, s12 in
// 16-31, (s22, s11) interleaved in 32-63 and (s02, s01) interleaved in 64-95, so a thread needs ~170 registers and
// three CTAs of 128 threads (4 warps; 16, 8 or 4 rows) share an SM.  At N <= 256 (two-stage transforms) columns
// 96-127 hold the thread's last-stage twiddles, and the exchange rows take 16-byte first-stage stores (RowLayoutV).
// One ring stage per CTA: the three transforms' inputs of a term pair are read into registers, the stage is
// refilled for the next pair while the transforms run, and the other CTAs of the SM cover the copy.
// Bounded waits, error flag and the drain before exit as in k_p3.
// What bounds it: HBM at 256^3 (6.8 TB/s of rows, four realisations).  Before the rows came ready-made from k_p2 its
// shared-memory path did (80 % of its cycles at 128^3 with a third of them bank conflicts, 88 % at 512^3), and 50 terms
// took 284 us at 128^3 (one realisation; now 219), 6.94 ms at 256^3 (four; now 6.04), 15.9 ms at 512^3 (40 terms; now 14.3,
// still bound by the exchanges of its three-stage transform).
template <int N>
struct P3TCfg {
  static constexpr int H = N / 2, E = 16, P = N / E, RPC = 128 / P, THREADS = RPC * P;  // 16 / 8 / 4 rows at N = 128 / 256 / 512
  static_assert(THREADS == 128 && P <= 32, "one warp per TMEM lane quarter; a row inside one warp");
  // two-stage transforms (N <= 256): twiddles in TMEM columns 96-127 and 16-byte exchange stores
  static constexpr bool TWTM = N <= 256;
  using Lay = std::conditional_t<TWTM, RowLayoutV<float, N>, RowLayout<float, N, true, 4>>;
  static constexpr int STAGE_ELEMS = 3 * RPC * N;  // the three row blocks of a term pair
  static constexpr uint32_t NCOLS = 128;           // TMEM columns per CTA (96, or 128 with the twiddles)
  static constexpr size_t SMEM = (size_t)STAGE_ELEMS * 8 + (size_t)RPC * Lay::SIZE * 8 + 16;
};

template <int N>
__global__ void __launch_bounds__(P3TCfg<N>::THREADS, 3) k_p3_tm(const float2* __restrict__ W,
                                                                  const float* __restrict__ sigma, int n_alpha,
                                                                  float2* __restrict__ F, int n_c,
                                                                  const float2* __restrict__ tw,
                                                                  int* __restrict__ err, long long wait_limit) {
  using CF = P3TCfg<N>;
  constexpr int E = CF::E, P = CF::P, RPC = CF::RPC;
  using Sync = typename RowSync<P>::type;
  using Lay = typename CF::Lay;
  extern __shared__ __align__(128) unsigned char smraw[];
  float2* ring = reinterpret_cast<float2*>(smraw);
  float2* xch = ring + CF::STAGE_ELEMS;
  uint64_t* bar = reinterpret_cast<uint64_t*>(xch + RPC * Lay::SIZE);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 1);
  const int rr = threadIdx.x / P, j = threadIdx.x % P;
  const Lay L{xch + rr * Lay::SIZE};
  const long row0 = (long)blockIdx.x * RPC;
  const long row = row0 + rr;
  const int b = blockIdx.y;
  const long fstride = (long)N * N * N;
  const int npairs = (n_alpha + 1) / 2;
  constexpr uint32_t COPY = RPC * N * sizeof(float2);
  const int warp = threadIdx.x >> 5;
  if (warp == 0) tmem_alloc(tslot, CF::NCOLS);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    mbar_init_fence();
  }
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  const uint32_t tbase = *tslot + ((uint32_t)(32 * (warp & 3)) << 16);  // this warp's lane quarter
  auto tcol = [&](int c) { return tbase + (uint32_t)(16 * c); };
  {
    float z0[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) z0[i] = 0.f;
#pragma unroll
    for (int c = 0; c < 6; ++c) tmem_st16(tcol(c), z0);
    if constexpr (CF::TWTM) tw_tm_store<N>(tcol(6), j, tw);
    tmem_wait_st();
  }
  auto issue = [&](int pr) {  // thread 0: the row blocks of term pair pr into the stage
    const bool two = 2 * pr + 1 < n_alpha;
    fence_proxy_async();
    mbar_expect_tx(bar, (two ? 3u : 2u) * COPY);
    for (int f = 0; f < 3; ++f)
      if (f != 1 || two)
        bulk_g2s(ring + f * RPC * N, W + (((long)b * npairs + pr) * 3 + f) * fstride + row0 * N, COPY, bar);
  };
  if (threadIdx.x == 0) issue(0);
  int issued = 1;  // term pairs whose copies thread 0 has issued
  const int par = (int)(row & 1);
  const float2* zin = ring + rr * N;  // rows f = 0, 1, 2 follow RPC rows apart
  bool ok = true;
  for (int pr = 0; pr < npairs; ++pr) {
    if (ok) ok = mbar_wait(bar, (uint32_t)(pr & 1), err, kWaitLast, wait_limit);
    const int a = 2 * pr;
    const bool two = a + 1 < n_alpha;
    // inputs of the three transforms: (g0^a + i g0^{a+1}), (g2^a + i g1^a), (g2^{a+1} + i g1^{a+1})
    float2 zB[E], za[E], zb[E];
#pragma unroll
    for (int r = 0; r < E; ++r) zB[r] = zrow<float, N, E>(zin + 2 * RPC * N, j, r, par);
#pragma unroll
    for (int r = 0; r < E; ++r) za[r] = zrow<float, N, E>(zin, j, r, par);
    if (two) {  // all but an odd last pair
#pragma unroll
      for (int r = 0; r < E; ++r) zb[r] = zrow<float, N, E>(zin + RPC * N, j, r, par);
    } else {
#pragma unroll
      for (int r = 0; r < E; ++r) zb[r] = make_float2(0.f, 0.f);
    }
    __syncthreads();  // the stage has been read: refill it for the next pair while the transforms run
    if (threadIdx.x == 0 && ok && pr + 1 < npairs) {
      issue(pr + 1);
      issued = pr + 2;
    }
    if constexpr (CF::TWTM) {
      fft_pencil_tw_tm<N, Lay, Sync>(zB, j, L, tcol(6), Sync());
      fft_pencil_tw_tm<N, Lay, Sync>(za, j, L, tcol(6), Sync());
      fft_pencil_tw_tm<N, Lay, Sync>(zb, j, L, tcol(6), Sync());
    } else {
      fft_pencil<float, N, E, +1, Lay, Sync>(zB, j, L, tw, Sync());
      fft_pencil<float, N, E, +1, Lay, Sync>(za, j, L, tw, Sync());
      fft_pencil<float, N, E, +1, Lay, Sync>(zb, j, L, tw, Sync());
    }
    const float sa = sigma[a], sb = two ? sigma[a + 1] : 0.f;
    // za = (g2a, g1a), zb = (g2b, g1b), zB = (g0a, g0b).  Chunks: s00 and s12 (16 columns each), (s22, s11) and
    // (s02, s01) interleaved (32 columns each), so the pair updates are paired (FP32x2) multiply-adds.
    {
      float u[16];
      tmem_ld16(tcol(0), u);  // s00 += sa g0a^2 + sb g0b^2
#pragma unroll
      for (int r = 0; r < E; ++r) u[r] = fmaf(sb * zB[r].y, zB[r].y, fmaf(sa * zB[r].x, zB[r].x, u[r]));
      tmem_st16(tcol(0), u);
      tmem_ld16(tcol(1), u);  // s12 += sa g1a g2a + sb g1b g2b
#pragma unroll
      for (int r = 0; r < E; ++r) u[r] = fmaf(sb * zb[r].y, zb[r].x, fmaf(sa * za[r].y, za[r].x, u[r]));
      tmem_st16(tcol(1), u);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {  // points 8 h .. 8 h + 7 of the interleaved chunks
      float u[16], w[16];
      tmem_ld16(tcol(2) + 16 * h, u);  // (s22, s11) += sa (g2a, g1a)^2 + sb (g2b, g1b)^2
      tmem_ld16(tcol(4) + 16 * h, w);  // (s02, s01) += sa g0a (g2a, g1a) + sb g0b (g2b, g1b)
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int r = 8 * h + i;
        float2 c = make_float2(u[2 * i], u[2 * i + 1]);
        c = __ffma2_rn(__fmul2_rn(za[r], make_float2(sa, sa)), za[r], c);
        c = __ffma2_rn(__fmul2_rn(zb[r], make_float2(sb, sb)), zb[r], c);
        u[2 * i] = c.x;
        u[2 * i + 1] = c.y;
        float2 d = make_float2(w[2 * i], w[2 * i + 1]);
        const float t0a = sa * zB[r].x, t0b = sb * zB[r].y;
        d = __ffma2_rn(make_float2(t0a, t0a), za[r], d);
        d = __ffma2_rn(make_float2(t0b, t0b), zb[r], d);
        w[2 * i] = d.x;
        w[2 * i + 1] = d.y;
      }
      tmem_st16(tcol(2) + 16 * h, u);
      tmem_st16(tcol(4) + 16 * h, w);
    }
    tmem_wait_st();
  }
  if (threadIdx.x == 0 && issued > 0) mbar_wait(bar, (uint32_t)((issued - 1) & 1), err, kWaitLast);  // drain the last copy
  // forward R2C of the six real rows, two per complex transform: (s00, s11), (s22, s01), (s02, s12)
  float2* zo = L.buf(0);
#pragma unroll 1
  for (int q = 0; q < 3; ++q) {
    float2 z[E];
    {
      float u[16], w[16];
      if (q == 0) {  // s00 and the odd columns of (s22, s11)
        tmem_ld16(tcol(0), u);
#pragma unroll
        for (int r = 0; r < E; ++r) z[r].x = u[r];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          tmem_ld16(tcol(2) + 16 * h, w);
#pragma unroll
          for (int i = 0; i < 8; ++i) z[8 * h + i].y = w[2 * i + 1];
        }
      } else if (q == 1) {  // the even columns of (s22, s11) and the odd ones of (s02, s01)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          tmem_ld16(tcol(2) + 16 * h, u);
          tmem_ld16(tcol(4) + 16 * h, w);
#pragma unroll
          for (int i = 0; i < 8; ++i) z[8 * h + i] = make_float2(u[2 * i], w[2 * i + 1]);
        }
      } else {  // the even columns of (s02, s01) and s12
        tmem_ld16(tcol(1), u);
#pragma unroll
        for (int r = 0; r < E; ++r) z[r].y = u[r];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          tmem_ld16(tcol(4) + 16 * h, w);
#pragma unroll
          for (int i = 0; i < 8; ++i) z[8 * h + i].x = w[2 * i];
        }
      }
    }
    fft_pencil<float, N, E, -1, Lay, Sync>(z, j, L, tw, Sync());
#pragma unroll
    for (int r = 0; r < E; ++r) zo[L.idx(j + r * P)] = z[r];
    Sync()();
    const int ncp = n_c + 1;
    const int c1 = q == 0 ? 0 : (q == 1 ? 2 : 4), c2 = q == 0 ? 1 : (q == 1 ? 3 : 5);
    // stored component order of F: (00, 11, 22, 01, 02, 12) = c = 0..5
    float2* f1 = F + (((long)b * 6 + c1) * N * N + row) * ncp;
    float2* f2 = F + (((long)b * 6 + c2) * N * N + row) * ncp;
    for (int k = j; k <= n_c; k += P) {
      const float2 zk = zo[L.idx(k)];
      const float2 zm = conjg<float>(zo[L.idx((N - k) & (N - 1))]);
      f1[k] = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y + zm.y));
      f2[k] = make_float2(0.5f * (zk.y - zm.y), -0.5f * (zk.x - zm.x));
    }
    Sync()();
  }
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  if (warp == 0) tmem_dealloc(*tslot, CF::NCOLS);
}

// ---------------------------------------------------------------- two transforms side by side
// c2 holds one point of two transforms A and B that use the same roots: r = (Re A, Re B), i = (Im A, Im B).  Every complex
// operation is then two or four paired (FP32x2) instructions for both, and a multiplication by i costs nothing.  SC:
// the outputs of a last butterfly layer come from scalar instructions, so that (Re A, Im A) and (Re B, Im B) can be
// stored as they are without moves.
struct c2 {
  float2 r, i;
};
template <bool SC> __device__ __forceinline__ float2 add2(float2 a, float2 b) {
  if constexpr (SC) return make_float2(a.x + b.x, a.y + b.y);
  else return __fadd2_rn(a, b);
}
template <bool SC> __device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  if constexpr (SC) return make_float2(a.x - b.x, a.y - b.y);
  else return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
}
template <bool SC> __device__ __forceinline__ float2 fma2(float s, float2 u, float2 a) {  // s u + a
  if constexpr (SC) return make_float2(fmaf(s, u.x, a.x), fmaf(s, u.y, a.y));
  else return __ffma2_rn(u, make_float2(s, s), a);
}
// inverse DFTs (roots e^{+2 pi i / R})
template <bool SC> __device__ __forceinline__ void idft2c(c2& a, c2& b) {
  const c2 t = a;
  a = {add2<SC>(t.r, b.r), add2<SC>(t.i, b.i)};
  b = {sub2<SC>(t.r, b.r), sub2<SC>(t.i, b.i)};
}
// (e + i o, e - i o)
template <bool SC> __device__ __forceinline__ void bfly_i(const c2& e, const c2& o, c2& p, c2& m) {
  p = {sub2<SC>(e.r, o.i), add2<SC>(e.i, o.r)};
  m = {add2<SC>(e.r, o.i), sub2<SC>(e.i, o.r)};
}
// (e + s u, e - s u) with separate signs of the real and imaginary parts
template <bool SC> __device__ __forceinline__ void bfly_s(const c2& e, const c2& u, float sr, float si, c2& p, c2& m) {
  p = {fma2<SC>(sr, u.r, e.r), fma2<SC>(si, u.i, e.i)};
  m = {fma2<SC>(-sr, u.r, e.r), fma2<SC>(-si, u.i, e.i)};
}
template <bool SC> __device__ __forceinline__ void idft4c(c2* v) {
  c2 s0 = v[0], d0 = v[2], s1 = v[1], d1 = v[3];
  idft2c<false>(s0, d0);
  idft2c<false>(s1, d1);
  idft2c<SC>(s0, s1);
  v[0] = s0;
  v[2] = s1;
  bfly_i<SC>(d0, d1, v[1], v[3]);
}
template <bool SC> __device__ __forceinline__ void idft8c(c2* v) {
  const float h = 0.70710678118654752440f;
  c2 e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
  idft4c<false>(e);
  idft4c<false>(o);
  idft2c<SC>(e[0], o[0]);
  v[0] = e[0];
  v[4] = o[0];
  c2 u = {sub2<false>(o[1].r, o[1].i), add2<false>(o[1].r, o[1].i)};  // o1 (1 + i)
  bfly_s<SC>(e[1], u, h, h, v[1], v[5]);
  bfly_i<SC>(e[2], o[2], v[2], v[6]);
  u = {add2<false>(o[3].r, o[3].i), sub2<false>(o[3].r, o[3].i)};  // o3 (-1 + i) = (-(r + i), r - i)
  bfly_s<SC>(e[3], u, -h, h, v[3], v[7]);
}
__device__ __forceinline__ void idft16c(c2* v) {
  const float h = 0.70710678118654752440f, c = cos_pi_8<float>(), t = 0.41421356237309504880f;  // cos, tan (pi/8)
  c2 e[8], o[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) { e[k] = v[2 * k]; o[k] = v[2 * k + 1]; }
  idft8c<false>(e);
  idft8c<false>(o);
  idft2c<false>(e[0], o[0]);
  v[0] = e[0];
  v[8] = o[0];
  // o_k times e^{i k pi / 8}, the cosine of the octant taken out
  c2 u = {fma2<false>(-t, o[1].i, o[1].r), fma2<false>(t, o[1].r, o[1].i)};
  bfly_s<false>(e[1], u, c, c, v[1], v[9]);
  u = {sub2<false>(o[2].r, o[2].i), add2<false>(o[2].r, o[2].i)};
  bfly_s<false>(e[2], u, h, h, v[2], v[10]);
  u = {fma2<false>(-t, o[3].r, o[3].i), fma2<false>(t, o[3].i, o[3].r)};
  bfly_s<false>(e[3], u, -c, c, v[3], v[11]);
  bfly_i<false>(e[4], o[4], v[4], v[12]);
  u = {fma2<false>(t, o[5].r, o[5].i), fma2<false>(-t, o[5].i, o[5].r)};
  bfly_s<false>(e[5], u, -c, c, v[5], v[13]);
  u = {add2<false>(o[6].r, o[6].i), sub2<false>(o[6].r, o[6].i)};
  bfly_s<false>(e[6], u, -h, h, v[6], v[14]);
  u = {fma2<false>(t, o[7].i, o[7].r), fma2<false>(-t, o[7].r, o[7].i)};
  bfly_s<false>(e[7], u, -c, -c, v[7], v[15]);
}
template <int R, bool SC> __device__ __forceinline__ void idftc(c2* v) {
  if constexpr (R == 4) idft4c<SC>(v);
  else idft8c<SC>(v);
}
// Times a root given to both transforms as w = (wx, wx, wy, wy), n = (-wy, -wy).
__device__ __forceinline__ c2 mulc(const c2& z, const float4& w, const float2& n) {
  return {__ffma2_rn(z.i, n, __fmul2_rn(z.r, make_float2(w.x, w.y))),
          __ffma2_rn(z.i, make_float2(w.x, w.y), __fmul2_rn(z.r, make_float2(w.z, w.w)))};
}

// P1 with its two transforms side by side (autotuner variant bit 16; FP32, N = 64 and 128): Ta and Tb of a term are the
// transforms of f Phi~ and i n0 f Phi~ with the same roots, so they run as one c2 transform.  Against one after the other
// that is one filter lookup and Phi~ read instead of two, one exchange (16-byte elements) and about 0.6 of the
// instructions.  A thread's 16 Phi~ values and cells sit in its tensor-memory lane for all the terms of a launch (columns
// 0-31: Phi~ as (re, im) pairs, 32-47: cells); the roots of the last stage are in shared memory in the form mulc wants.
// Four CTAs of 128 threads share an SM (with two of 256 threads the barriers of a CTA left it idle: 128^3, 50 terms of one
// realisation 207 us, now 173; the transforms one after the other 219).  Eight realisations at 64^3: 198 -> 161 us.  From
// 256^3 on k_p1_tm is faster: rows of 128 bytes need 256 threads here, and 16 warps a SM then leave more latency open
// than its 24 (50 terms of four realisations 5.80 ms against 5.33).
template <int N>
struct P1ACfg {
  static constexpr int H = N / 2, E = 16, P = N / E;
  static constexpr int THREADS = 128, CTAS = 4, TC = THREADS / P;  // 32 and 16 columns
  static constexpr int RL = N / 16, NB = 16 / RL;                  // last stage: radix, butterflies per thread
  static constexpr int ROOTS = NB * (RL - 1) * P;                  // its roots [t][r - 1][j]
  static constexpr uint32_t NCOLS = 64;
  static size_t smem(int nb, int nm1) {
    return (size_t)N * TC * 16 + (size_t)ROOTS * 24 + (size_t)N * 8 + (size_t)N * 4 + (size_t)nb * nm1 * 4 + 16;
  }
};

template <int N>
__global__ void __launch_bounds__(P1ACfg<N>::THREADS, P1ACfg<N>::CTAS) k_p1_ab(
    const float2* __restrict__ phi, float2* __restrict__ Ta, float2* __restrict__ Tb, const int16_t* __restrict__ lut,
    const float* __restrict__ phitab, int nm1, int alpha0, int nb, int nag, int swz,
    const float2* __restrict__ tw) {
  using CF = P1ACfg<N>;
  constexpr int E = CF::E, P = CF::P, TC = CF::TC, H = CF::H, NH = H + 1, RL = CF::RL, NB = CF::NB;
  extern __shared__ __align__(16) unsigned char smraw[];
  float4* const xch = reinterpret_cast<float4*>(smraw);           // [N][TC]
  float4* const rw = xch + N * TC;                                // roots
  float2* const rn = reinterpret_cast<float2*>(rw + CF::ROOTS);
  float2* const sm_nyq = rn + CF::ROOTS;                          // N values (column 0 only)
  int* const sm_cn = reinterpret_cast<int*>(sm_nyq + N);          // N cells
  float* const sm_tab = reinterpret_cast<float*>(sm_cn + N);      // (terms of this CTA) * nm1
  const int b = blockIdx.z / nag, ag = blockIdx.z % nag;
  const int alo = (int)((long)nb * ag / nag), ahi = (int)((long)nb * (ag + 1) / nag);  // terms of this CTA
  uint32_t* const tslot = reinterpret_cast<uint32_t*>(sm_tab + (ahi - alo) * nm1);
  const int c = threadIdx.x % TC, j = threadIdx.x / TC;
  const int cc = blockIdx.x * TC + c;
  const int k1 = blockIdx.y;
  const int n1 = wrapn(k1, N);
  const int warp = threadIdx.x >> 5;
  if (warp == 0) tmem_alloc(tslot, CF::NCOLS);
  for (int i = threadIdx.x; i < (ahi - alo) * nm1; i += CF::THREADS) sm_tab[i] = phitab[(long)(alpha0 + alo) * nm1 + i];
  for (int i = threadIdx.x; i < CF::ROOTS; i += CF::THREADS) {
    const int jj = i % P, q = i / P, t = q / (RL - 1), r = q % (RL - 1) + 1;
    const int e = r * ((jj + t * P) & 15);  // exponent of e^{+2 pi i / N}
    const float2 w = __ldg(tw + e);  // e^{-2 pi i e / N}
    rw[i] = make_float4(w.x, w.x, -w.y, -w.y);
    rn[i] = make_float2(w.y, w.y);
  }
  const float2* pb = phi + ((long)b * N * N + k1) * NH;  // + k0 * N * NH + k2
  if (blockIdx.x == 0) {
    for (int k0 = threadIdx.x; k0 < N; k0 += CF::THREADS) {
      const int n0 = wrapn(k0, N);
      sm_nyq[k0] = pb[(long)k0 * N * NH + H];
      sm_cn[k0] = lut[n0 * n0 + n1 * n1 + H * H];
    }
  }
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  const uint32_t tbase = *tslot + ((uint32_t)(32 * warp) << 16);
  {
    float u[16];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float2 v = pb[(long)(j + (8 * h + i) * P) * N * NH + cc];
        u[2 * i] = v.x;
        u[2 * i + 1] = v.y;
      }
      tmem_st16(tbase + 16 * h, u);
    }
#pragma unroll
    for (int r = 0; r < E; ++r) {
      const int n0 = wrapn(j + r * P, N);
      u[r] = __int_as_float((int)lut[n0 * n0 + n1 * n1 + cc * cc]);
    }
    tmem_st16(tbase + 32, u);
    tmem_wait_st();
  }
  const long fstride = (long)N * N * H;  // one field
  const float fj = (float)j;
  const int cs = cc ^ ((k1 & 1) * swz);
  const long toff = ((long)b * nb) * fstride + t_index<float, N>(k1, cs) + (long)j * N * H;
  float4* const xw = xch + 16 * j * TC + c;  // first-stage outputs 16 j + r
  float4* const xr = xch + j * TC + c;       // points j + ...
  auto put = [](const c2& z) { return make_float4(z.r.x, z.r.y, z.i.x, z.i.y); };
  auto get = [](const float4& x) { return c2{make_float2(x.x, x.y), make_float2(x.z, x.w)}; };
#pragma unroll 1
  for (int a = alo; a < ahi; ++a) {
    const float* tab = sm_tab + (a - alo) * nm1;
    c2 v[E];
    {
      float fl[16], u[32];
      tmem_ld16(tbase + 32, fl);
#pragma unroll
      for (int r = 0; r < E; ++r) fl[r] = tab[__float_as_int(fl[r])];
      tmem_ld32(tbase, u);
      // the pair (V, i n0^D V): n0^D of k0 = j + r P (k0 < N/2 exactly when r < E/2; zero on the Nyquist index r = E/2,
      // j = 0).  NYQ: the CTA holds packed column 0, whose thread c = 0 adds i V(k2 = N/2) with its own cell.
      auto fill = [&](auto nyq) {
#pragma unroll
        for (int r = 0; r < E; ++r) {
          const float nd = r < E / 2 ? fj + (float)(r * P) : ((r == E / 2 && j == 0) ? 0.f : fj + (float)(r * P - N));
          float x = fl[r] * u[2 * r], y = fl[r] * u[2 * r + 1];
          if (decltype(nyq)::value && cc == 0) {
            const float fn = tab[sm_cn[j + r * P]];
            const float2 yn = sm_nyq[j + r * P];
            x = x - fn * yn.y;
            y = y + fn * yn.x;
          }
          v[r] = {make_float2(x, -nd * y), make_float2(y, nd * x)};
        }
      };
      if (blockIdx.x == 0) fill(std::true_type{});
      else fill(std::false_type{});
    }
    idft16c(v);
    __syncthreads();  // the exchange of the term before has been read
#pragma unroll
    for (int r = 0; r < E; ++r) xw[r * TC] = put(v[r]);
    __syncthreads();
    float2* const da = Ta + toff + a * fstride;
    float2* const db = Tb + toff + a * fstride;
#pragma unroll
    for (int t = 0; t < NB; ++t) {
      c2 z[RL];
#pragma unroll
      for (int r = 0; r < RL; ++r) {
        z[r] = get(xr[(t * P + r * (N / RL)) * TC]);
        if (r) {
          const int i = (t * (RL - 1) + r - 1) * P + j;
          z[r] = mulc(z[r], rw[i], rn[i]);
        }
      }
      idftc<RL, true>(z);
#pragma unroll
      for (int r = 0; r < RL; ++r) {  // point j + t P + r N / RL
        da[(long)(t * P + r * (N / RL)) * N * H] = make_float2(z[r].r.x, z[r].i.x);
        db[(long)(t * P + r * (N / RL)) * N * H] = make_float2(z[r].r.y, z[r].i.y);
      }
    }
  }
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  if (warp == 0) tmem_dealloc(*tslot, CF::NCOLS);
}

// P1 with its Phi~ tile and cell indices in tensor memory (autotuner variant bit 16; FP32, N = 256 and 512, radix 16,
// 256 threads per CTA: 16 or 8 columns).  k_p1 keeps each thread's 16 Phi~ values and cells in registers for all the terms of a launch
// (125 registers: two CTAs of 8 warps per SM, latency-bound).  Here they sit in the thread's TMEM lane (columns
// 0-31: Phi~ as (re, im) pairs, 32-47: cells; warps w and w + 4 share a lane quarter, the latter at column 64) and are read back for every transform;
// with a single exchange buffer (free for a two-stage transform; a three-stage
// one syncs between a stage's reads and writes) three CTAs share an SM at 80 registers (measured faster than four at
// 64).  At N = 256, 8 of each thread's 15 last-stage twiddles also sit in its lane (columns 48-63).  Same arithmetic
// as k_p1.
template <int N>
struct P1TCfg {
  static constexpr int H = N / 2, E = 16, P = N / E, TC = 256 / P, THREADS = TC * P;  // 16 / 8 columns
  static constexpr int CTAS = 3;
  static_assert(THREADS == 256, "two warps per TMEM lane quarter");
  using Lay = ColLayout<float, N, TC, E, true>;
  static constexpr uint32_t NCOLS = 128;  // per warp group: Phi~ 0-31, cells 32-47, 8 twiddles 48-63 (N <= 256)
  static size_t smem(int nb, int nm1) {
    return (size_t)Lay::SIZE * 8 + (size_t)N * 8 + (size_t)N * 4 + (size_t)nb * nm1 * 4 + 16;
  }
};

template <int N>
__global__ void __launch_bounds__(P1TCfg<N>::THREADS, 3) k_p1_tm(const float2* __restrict__ phi, float2* __restrict__ Ta,
                                                                  float2* __restrict__ Tb, const int16_t* __restrict__ lut,
                                                                  const float* __restrict__ phitab, int nm1, int alpha0,
                                                                  int nb, int nag,
                                                                  const float2* __restrict__ tw) {
  using CF = P1TCfg<N>;
  constexpr int E = CF::E, P = CF::P, TC = CF::TC, H = CF::H, NH = H + 1;
  using Lay = typename CF::Lay;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* sm_nyq = reinterpret_cast<float2*>(smraw) + Lay::SIZE;  // N values (column 0 only)
  int* sm_cn = reinterpret_cast<int*>(sm_nyq + N);                // N cells
  float* sm_tab = reinterpret_cast<float*>(sm_cn + N);            // (terms of this CTA) * nm1
  const int b = blockIdx.z / nag, ag = blockIdx.z % nag;
  const int alo = (int)((long)nb * ag / nag), ahi = (int)((long)nb * (ag + 1) / nag);  // terms of this CTA
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm_tab + (ahi - alo) * nm1);
  const int c = threadIdx.x % TC, j = threadIdx.x / TC;
  const Lay L{reinterpret_cast<float2*>(smraw), c};
  const int cc = blockIdx.x * TC + c;
  const int k1 = blockIdx.y;
  const int n1 = wrapn(k1, N);
  const int warp = threadIdx.x >> 5;
  if (warp == 0) tmem_alloc(tslot, CF::NCOLS);
  for (int i = threadIdx.x; i < (ahi - alo) * nm1; i += blockDim.x) sm_tab[i] = phitab[(long)(alpha0 + alo) * nm1 + i];
  const float2* pb = phi + ((long)b * N * N + k1) * NH;  // + k0 * N * NH + k2
  if (blockIdx.x == 0) {
    for (int k0 = threadIdx.x; k0 < N; k0 += blockDim.x) {
      const int n0 = wrapn(k0, N);
      sm_nyq[k0] = pb[(long)k0 * N * NH + H];
      sm_cn[k0] = lut[n0 * n0 + n1 * n1 + H * H];
    }
  }
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  const uint32_t tbase = *tslot + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(64 * (warp >> 2));
  {
    float u[16];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int k0 = j + (8 * h + i) * P;
        const float2 v = pb[(long)k0 * N * NH + cc];
        u[2 * i] = v.x;
        u[2 * i + 1] = v.y;
      }
      tmem_st16(tbase + 16 * h, u);
    }
#pragma unroll
    for (int r = 0; r < E; ++r) {
      const int n0 = wrapn(j + r * P, N);
      u[r] = __int_as_float((int)lut[n0 * n0 + n1 * n1 + cc * cc]);
    }
    tmem_st16(tbase + 32, u);
    if constexpr (N <= 256) tw8_tm_store<N>(tbase + 48, j, tw);  // 8 last-stage twiddles in columns 48-63
    tmem_wait_st();
  }
  const long fstride = (long)N * N * H;  // one field
  const float fj = (float)j;
  for (int a = alo; a < ahi; ++a) {
    const float* tab = sm_tab + (a - alo) * nm1;
#pragma unroll 1
    for (int D = 0; D < 2; ++D) {
      float2 v[E];
      {
        // the filter values of this term, looked up from the cells (keeping them in tensor memory for the second
        // field was measured slower)
        float fl[16], u[16];
        tmem_ld16(tbase + 32, fl);
#pragma unroll
        for (int r = 0; r < E; ++r) fl[r] = tab[__float_as_int(fl[r])];
        // the 8 inputs of half h.  DER: times i n0^D(k0), k0 = j + r P (k0 < N/2 exactly when r < E/2; zero on the
        // Nyquist index r = E/2, j = 0), folded into the filter value.  NYQ: the CTA holds packed column 0, whose
        // thread c = 0 adds i V(k2 = N/2) with its own cell.  Both are compile-time, so the other CTAs' loops carry
        // no per-value branches.
        auto fill = [&](auto der, auto nyq, int h) {
          constexpr bool DER = decltype(der)::value, NYQ = decltype(nyq)::value;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int r = 8 * h + i;
            const float nd = r < E / 2 ? fj + (float)(r * P) : ((r == E / 2 && j == 0) ? 0.f : fj + (float)(r * P - N));
            float2 x;
            if (NYQ && cc == 0) {
              const float f = fl[r];
              x = make_float2(f * u[2 * i], f * u[2 * i + 1]);
              const int k0 = j + r * P;
              const float fn = tab[sm_cn[k0]];
              const float2 yn = sm_nyq[k0];
              x = make_float2(x.x - fn * yn.y, x.y + fn * yn.x);
              if constexpr (DER) x = make_float2(-nd * x.y, nd * x.x);
            } else if constexpr (DER) {
              const float g = fl[r] * nd;
              x = make_float2(-g * u[2 * i + 1], g * u[2 * i]);
            } else {
              const float f = fl[r];
              x = make_float2(f * u[2 * i], f * u[2 * i + 1]);
            }
            v[r] = x;
          }
        };
        const std::true_type yes{};
        const std::false_type no{};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          tmem_ld16(tbase + 16 * h, u);
          if (blockIdx.x == 0) {
            if (D) fill(yes, yes, h);
            else fill(no, yes, h);
          } else {
            if (D) fill(yes, no, h);
            else fill(no, no, h);
          }
        }
      }
      if constexpr (N <= 256) fft_pencil_tw8_tm<N, Lay, SyncBlock>(v, j, L, tw, tbase + 48, SyncBlock());
      else fft_pencil<float, N, E, +1, Lay, SyncBlock>(v, j, L, tw, SyncBlock());
      float2* dst = (D ? Tb : Ta) + ((long)b * nb + a) * fstride + t_index<float, N>(k1, cc);
#pragma unroll
      for (int r = 0; r < E; ++r) dst[(long)(j + r * P) * N * H] = v[r];
    }
  }
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  if (warp == 0) tmem_dealloc(*tslot, CF::NCOLS);
}

// ---------------------------------------------------------------- second and last inverse pass in one kernel
// P23 (FP32, N = 64): from Ta, Tb (the first pass's output for all terms) straight to the product, without storing the
// three fields per term that k_p2 hands to the last pass.  A CTA owns one plane a0, 64 x 64 points, whose six product
// components stay in tensor memory for the whole sum over its group of term pairs.
//   Z_A = (i n2^D - n1^D) Ta^a  -> g2^a + i g1^a      Z_0 = Tb^a + i Tb^{a+1}  -> g0^a + i g0^{a+1}
// over the full range of k2 (the half spectrum is mirrored as it is read), so a term pair costs three complex 2-D
// transforms.
//   - Planes [k1][c] (16 KB) arrive by cp.async.bulk in a ring of NSLOT; their columns are stored as c ^ 8 (k1 mod 2), so
//     that the two rows of a half warp fall into different halves of the banks.
//   - Axis 1: a warp takes 8 columns of k2, thread (c, j) 16 of the 64 points (radix 16 then 4); its exchange uses the
//     memory that holds the rows the warp owns afterwards, so only warp barriers are needed.
//   - Rows: the transformed columns go to the row buffer (two block barriers a transform, the only ones), a warp owns
//     8 rows, and the exchange of the row transform (radix 16 then 4) is in place.
// Bounded waits, error flag and the drain before exit as in k_p3.
// What bounds it: the shared-memory path (ncu: 283 wavefronts a warp and transform, 61 % of the path's cycles while
// active) with 16 warps a SM, issue 50 %; DRAM 17 %.  Four groups of term pairs: 256 CTAs for one realisation, two a SM.
// 50 terms of both kernels of one realisation take 161 us (k_p2 and k_p3 before 432), of eight 976 us (2044).  Both kernels
// in one launch with two groups each took 146 and 915 us, but T of both, 4 fields a term, is more than the plan's other
// forms need (+38 % device memory).  The same split at N = 128 (two residue classes of a1 per plane) was slower than the
// two passes there (715 against 690 us then, 520 now): its shared-memory traffic grows while HBM already carries them.
template <int N>
struct P23Cfg {
  static_assert(N == 64, "one plane per CTA, two CTAs per SM");
  static constexpr int H = N / 2, M = 64, E = 16;
  static constexpr int THREADS = M * N / E, WARPS = THREADS / 32;  // 256, 8
  static constexpr int P = N / E;             // threads per row: 4
  static constexpr int RPW = M / WARPS;       // rows per warp: 8
  static constexpr int NSLOT = 3;
  static constexpr int TILE = N * H;          // complex values of one plane
  static constexpr uint32_t NCOLS = 128 * (WARPS / 4);  // per warp: 96 accumulators, 32 for row twiddles
  static constexpr int CTAS = 2;
  // Row buffer: element p of a row at p + 2 (p / 16) (16-byte pairs of the radix-16 outputs), rows PITCH apart, the rows
  // of a warp in bit-reversed order.  PITCH mod 16 = 16 / RPW, so the RPW rows x (16 / RPW) threads of a half warp
  // read 16 different 8-byte banks, and the two rows of a half warp's column store lie 8 banks apart.
  static constexpr int PITCH = 82;
  static constexpr size_t SMEM = (size_t)NSLOT * TILE * 8 + (size_t)M * PITCH * 8 + (size_t)N * 8 + 64;
  static __host__ __device__ constexpr int slot_of(int row) {  // place of row a1 in the row buffer (its own inverse)
    return (row & ~7) | ((row & 1) << 2) | (row & 2) | ((row >> 2) & 1);
  }
};

template <int N> struct P23RowLay {
  static constexpr bool SINGLE = true;
  static constexpr bool VEC = true;
  float2* base;
  __device__ __forceinline__ float2* buf(int) const { return base; }
  __device__ __forceinline__ int idx(int p) const { return p + 2 * (p >> 4); }
};

template <int N>
__global__ void __launch_bounds__(P23Cfg<N>::THREADS, P23Cfg<N>::CTAS) k_p23(
    const float2* __restrict__ Ta, const float2* __restrict__ Tb, const float* __restrict__ sigma, int n_alpha,
    float2* __restrict__ F, long fgstride, int n_c, const float2* __restrict__ tw, int* __restrict__ err,
    long long wait_limit) {
  using CF = P23Cfg<N>;
  using RL = P23RowLay<N>;
  constexpr int E = 16, H = CF::H, P = CF::P, RPW = CF::RPW, NSLOT = CF::NSLOT, PITCH = CF::PITCH;
  constexpr int RLAST = N / 16, NB = 16 / RLAST;  // radix of the rows' last stage, butterflies per thread
  extern __shared__ __align__(128) unsigned char smraw[];
  float2* ring = reinterpret_cast<float2*>(smraw);
  float2* rows = ring + NSLOT * CF::TILE;       // [64][PITCH]
  float2* twN = rows + CF::M * PITCH;           // e^{+2 pi i k / N}
  uint64_t* bars = reinterpret_cast<uint64_t*>(twN + N);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + NSLOT);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int a0 = blockIdx.x;
  const int b = blockIdx.y;
  const int allpairs = (n_alpha + 1) / 2;
  const int pr0 = allpairs * (int)blockIdx.z / (int)gridDim.z;
  const int pr1 = allpairs * ((int)blockIdx.z + 1) / (int)gridDim.z;
  const int nterms = min(2 * pr1, n_alpha) - 2 * pr0;  // terms of this group
  const int ntiles = 2 * nterms;
  F += (long)blockIdx.z * fgstride;
  const long fstride = (long)N * N * H;
  const long poff = ((long)b * n_alpha + 2 * pr0) * fstride + (long)a0 * CF::TILE;
  if (warp == 0) tmem_alloc(tslot, CF::NCOLS);
  if (threadIdx.x == 0) {
    for (int s = 0; s < NSLOT; ++s) mbar_init(bars + s, 1);
    mbar_init_fence();
  }
  for (int i = threadIdx.x; i < N; i += CF::THREADS) twN[i] = conjg<float>(__ldg(tw + i));
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  // Planes of this group in the order they are used: Tb^a, Tb^{a+1}, Ta^a, Ta^{a+1} of each pair.
  auto issue = [&](int q) {  // thread 0
    const int lp = q >> 2, left = nterms - 2 * lp;  // terms from this pair on
    const int e = q & 3;
    const bool two = left >= 2;
    const int term = 2 * lp + (two ? (e & 1) : 0);
    const bool isb = two ? e < 2 : e < 1;
    const int s = q % NSLOT;
    fence_proxy_async();
    mbar_expect_tx(bars + s, CF::TILE * 8);
    bulk_g2s(ring + s * CF::TILE, (isb ? Tb : Ta) + poff + (long)term * fstride, CF::TILE * 8, bars + s);
  };
  int issued = min(NSLOT, ntiles);  // planes whose copies thread 0 has issued
  if (threadIdx.x == 0)
    for (int q = 0; q < issued; ++q) issue(q);
  const uint32_t tbase = *tslot + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(128 * (warp >> 2));
  auto tcol = [&](int c) { return tbase + (uint32_t)(16 * c); };
  // axis 1: column c2 of the full spectrum, points j + 4 r;  rows: place 8 warp + rr, points jj + P r
  const int c8 = lane & 7, j = lane >> 3, jo = j & 1;
  const int c2 = 8 * warp + c8;
  const int cm = c2 == H ? 0 : (c2 > H ? N - c2 : c2);  // stored column
  const float fn2 = c2 < H ? (float)c2 : (c2 == H ? 0.f : (float)(c2 - N));
  const float fj = (float)j;
  const int jj = lane / RPW, rr = lane % RPW;
  const RL L{rows + (warp * RPW + rr) * PITCH};
  const int arow = CF::slot_of(warp * RPW + rr);  // a1 of this row
  // plane offsets of (k1 = j, stored column) and, mirrored, of (N - j, column); k1 steps of 4 are constants
  const int od = j * H + (cm ^ (jo << 3)), om = (N - j) * H + (cm ^ (jo << 3));
  const int om0 = j == 0 ? cm : om;  // mirrored k1 = 0
  // axis-1 exchange in the warp's own rows: point p of column c at 8 (p ^ (p / 16 mod 2)) + c, so that two threads of a
  // pencil (16 or 1 points apart) fall into different halves of the banks
  float2* const xb = rows + warp * (RPW * PITCH) + c8;
  float2* const xw0 = xb + 8 * (16 * j + jo);
  float2* const xw1 = xb + 8 * (16 * j + 1 - jo);
  const float2* const xr0 = xb + 8 * j;
  const float2* const xr1 = xb + 8 * (j ^ 1);
  // column stores: row a1 = j + 4 m
  float2* const zc0 = rows + CF::slot_of(j) * PITCH + c2 + 2 * (c2 >> 4);
  {
    float z0[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) z0[i] = 0.f;
#pragma unroll
    for (int c = 0; c < 6; ++c) tmem_st16(tcol(c), z0);
    // last-stage row twiddles: W_N^{r k}, k = (jj + t P) mod 16
    float w[2][16];
#pragma unroll
    for (int i = 0; i < 16; ++i) w[0][i] = w[1][i] = 0.f;
#pragma unroll
    for (int t = 0; t < NB; ++t)
#pragma unroll
      for (int r = 1; r < RLAST; ++r) {
        const int q = t * (RLAST - 1) + r - 1;
        const float2 x = twN[r * ((jj + t * P) & 15)];
        w[q >> 3][2 * (q & 7)] = x.x;
        w[q >> 3][2 * (q & 7) + 1] = x.y;
      }
    tmem_st16(tcol(6), w[0]);
    tmem_st16(tcol(7), w[1]);
    tmem_wait_st();
  }
  // Stored value behind the full spectrum at (k1 = j + 4 r, c2); MIR: from (-k1, -c2), to be conjugated by the caller;
  // SPEC: the warp holds c2 = 0 or c2 = N/2, both unpacked from column 0 (X(k1, 0) + i X(k1, N/2)).
  auto spec = [&](auto mir, auto special, const float2* t, int r) -> float2 {
    constexpr bool MIR = decltype(mir)::value, SPEC = decltype(special)::value;
    float2 x = MIR ? t[r == 0 ? om0 : om - 4 * r * H] : t[od + 4 * r * H];
    if (SPEC && cm == 0) {  // one lane column
      const int k1 = j + 4 * r, ko = MIR ? k1 : (N - k1) & (N - 1);
      const float2 o = t[ko * H + (jo << 3)];
      // X(k1, 0) = (Y + conj Y-) / 2; X(k1, N/2) = -i (Y - conj Y-) / 2, here conjugated for the mirrored caller
      x = MIR ? make_float2(0.5f * (o.y + x.y), 0.5f * (o.x - x.x)) : make_float2(0.5f * (x.x + o.x), 0.5f * (x.y - o.y));
    }
    return x;
  };
  // the 16 axis-1 inputs of a transform: Z_0 (FIRST) from two planes or Z_A from one
  auto load = [&](auto mir, auto special, auto first, float2 (&v)[E], const float2* t0, const float2* t1) {
    constexpr bool MIR = decltype(mir)::value, FIRST = decltype(first)::value;
#pragma unroll
    for (int r = 0; r < E; ++r) {
      const float2 x = spec(mir, special, t0, r);
      if constexpr (FIRST) {
        const float2 y = t1 ? spec(mir, special, t1, r) : make_float2(0.f, 0.f);
        v[r] = MIR ? make_float2(x.x + y.y, y.x - x.y) : make_float2(x.x - y.y, x.y + y.x);
      } else {
        const float n = r < 8 ? fj + (float)(4 * r) : ((r == 8 && j == 0) ? 0.f : fj + (float)(4 * r - 64));
        const float2 d = __fmul2_rn(x, make_float2(n, n));
        v[r] = MIR ? make_float2(fmaf(fn2, x.y, -d.x), fmaf(fn2, x.x, d.y))
                   : make_float2(fmaf(-fn2, x.y, -d.x), fmaf(fn2, x.x, -d.y));
      }
    }
  };
  auto load_any = [&](auto first, float2 (&v)[E], const float2* t0, const float2* t1) {
    const std::true_type yes{};
    const std::false_type no{};
    if (warp == 0) load(no, yes, first, v, t0, t1);
    else if (warp < H / 8) load(no, no, first, v, t0, t1);
    else if (warp == H / 8) load(yes, yes, first, v, t0, t1);
    else load(yes, no, first, v, t0, t1);
  };
  bool ok = true;
  int q = 0;  // planes used so far
  for (int lp = 0; 2 * lp < nterms; ++lp) {
    const bool two = nterms - 2 * lp >= 2;
    float2 zB[E];
    const float* sg = sigma + 2 * (pr0 + lp);
#pragma unroll 1
    for (int ph = 0; ph < (two ? 3 : 2); ++ph) {
      float2 v[E];
      const int used = (ph == 0 && two) ? 2 : 1;
      for (int u = 0; u < used; ++u)
        if (ok) ok = mbar_wait(bars + (q + u) % NSLOT, (uint32_t)(((q + u) / NSLOT) & 1), err, kWaitFused, wait_limit);
      const float2* t0 = ring + (q % NSLOT) * CF::TILE;
      if (ph == 0) load_any(std::true_type{}, v, t0, two ? ring + ((q + 1) % NSLOT) * CF::TILE : nullptr);
      else load_any(std::false_type{}, v, t0, nullptr);
      // ---- axis 1, 64 points: radix 16, exchange, radix 4
      dftR<float, +1, E>(v);
      __syncwarp();  // the warp's rows of the transform before have been read
#pragma unroll
      for (int r = 0; r < E; ++r) (r & 1 ? xw1 : xw0)[16 * (r >> 1)] = v[r];
      __syncwarp();
      {
        float w[32];  // the row transform's roots: the same length, and jj = j
        tmem_ld32(tcol(6), w);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          float2 a[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) a[r] = (r & 1 ? xr1 : xr0)[8 * (4 * t + 16 * r)];
#pragma unroll
          for (int r = 1; r < 4; ++r) {
            const int i = 3 * t + r - 1;
            a[r] = mul<float>(a[r], make_float2(w[2 * i], w[2 * i + 1]));
          }
          dftR<float, +1, 4>(a);
#pragma unroll
          for (int r = 0; r < 4; ++r) v[t + 4 * r] = a[r];
        }
      }
      __syncthreads();  // every exchange and every plane read is over
      if (threadIdx.x == 0 && ok) {
        for (int u = 0; u < used; ++u)
          if (q + u + NSLOT < ntiles) {
            issue(q + u + NSLOT);
            issued = q + u + NSLOT + 1;
          }
      }
      q += used;
#pragma unroll
      for (int m = 0; m < E; ++m)  // row a1 = j + 4 m, column c2
        zc0[(CF::slot_of(4 * m)) * PITCH] = v[m];
      __syncthreads();
      // ---- rows: radix 16, exchange in place, radix 4
#pragma unroll
      for (int r = 0; r < E; ++r) v[r] = L.base[jj + L.idx(P * r)];
      dftR<float, +1, E>(v);
      __syncwarp();
#pragma unroll
      for (int m = 0; m < E / 2; ++m)
        *reinterpret_cast<float4*>(L.base + 18 * jj + 2 * m) =
            make_float4(v[2 * m].x, v[2 * m].y, v[2 * m + 1].x, v[2 * m + 1].y);
      __syncwarp();
      {
        float w[32];
        tmem_ld32(tcol(6), w);
#pragma unroll
        for (int t = 0; t < NB; ++t) {
          float2 a[RLAST];
#pragma unroll
          for (int r = 0; r < RLAST; ++r) a[r] = L.base[jj + t * P + 18 * r];
#pragma unroll
          for (int r = 1; r < RLAST; ++r) {
            const int i = t * (RLAST - 1) + r - 1;
            a[r] = mul<float>(a[r], make_float2(w[2 * i], w[2 * i + 1]));
          }
          dftR<float, +1, RLAST>(a);
#pragma unroll
          for (int r = 0; r < RLAST; ++r) v[t + r * NB] = a[r];
        }
      }
      if (ph == 0) {
#pragma unroll
        for (int r = 0; r < E; ++r) zB[r] = v[r];
        continue;
      }
      // ---- the term's products: v = (g2, g1), g0 = Re or Im of zB.  Columns: s00, s12 (16 each), (s22, s11) and
      // (s02, s01) interleaved (32 each).
      const float sa = __ldg(sg + ph - 1);
      if (ph == 2) {
#pragma unroll
        for (int r = 0; r < E; ++r) zB[r].x = zB[r].y;
      }
      {
        float u[32];
        tmem_ld32(tcol(0), u);
#pragma unroll
        for (int r = 0; r < E; ++r) {
          u[r] = fmaf(sa * zB[r].x, zB[r].x, u[r]);
          u[16 + r] = fmaf(sa * v[r].y, v[r].x, u[16 + r]);
        }
        tmem_st32(tcol(0), u);
      }
      {
        float u[32];
        tmem_ld32(tcol(2), u);
#pragma unroll
        for (int r = 0; r < E; ++r) {
          const float2 c = __ffma2_rn(__fmul2_rn(v[r], make_float2(sa, sa)), v[r], make_float2(u[2 * r], u[2 * r + 1]));
          u[2 * r] = c.x;
          u[2 * r + 1] = c.y;
        }
        tmem_st32(tcol(2), u);
        tmem_ld32(tcol(4), u);
#pragma unroll
        for (int r = 0; r < E; ++r) {
          const float t0s = sa * zB[r].x;
          const float2 d = __ffma2_rn(make_float2(t0s, t0s), v[r], make_float2(u[2 * r], u[2 * r + 1]));
          u[2 * r] = d.x;
          u[2 * r + 1] = d.y;
        }
        tmem_st32(tcol(4), u);
      }
      tmem_wait_st();
    }
  }
  if (threadIdx.x == 0) {  // the last copy issued into each slot has landed before the CTA may exit
    for (int s = 0; s < NSLOT && s < issued; ++s) {
      const int last = s + ((issued - 1 - s) / NSLOT) * NSLOT;
      mbar_wait(bars + s, (uint32_t)((last / NSLOT) & 1), err, kWaitFused);
    }
  }
  // ---- forward R2C of the six real rows along axis 2, two per complex transform: (s00, s11), (s22, s01), (s02, s12)
  __syncwarp();
  const long row = (long)a0 * N + arow;
  const int ncp = n_c + 1;
#pragma unroll 1
  for (int h3 = 0; h3 < 3; ++h3) {
    float2 z[E];
    {
      float u[16], w[16];
      if (h3 == 0) {
        tmem_ld16(tcol(0), u);
#pragma unroll
        for (int r = 0; r < E; ++r) z[r].x = u[r];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          tmem_ld16(tcol(2) + 16 * h, w);
#pragma unroll
          for (int i = 0; i < 8; ++i) z[8 * h + i].y = w[2 * i + 1];
        }
      } else if (h3 == 1) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          tmem_ld16(tcol(2) + 16 * h, u);
          tmem_ld16(tcol(4) + 16 * h, w);
#pragma unroll
          for (int i = 0; i < 8; ++i) z[8 * h + i] = make_float2(u[2 * i], w[2 * i + 1]);
        }
      } else {
        tmem_ld16(tcol(1), u);
#pragma unroll
        for (int r = 0; r < E; ++r) z[r].y = u[r];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          tmem_ld16(tcol(4) + 16 * h, w);
#pragma unroll
          for (int i = 0; i < 8; ++i) z[8 * h + i].x = w[2 * i];
        }
      }
    }
    fft_pencil<float, N, E, -1, RL, SyncWarp>(z, jj, L, tw, SyncWarp());
#pragma unroll
    for (int r = 0; r < E; ++r) L.base[L.idx(jj + r * P)] = z[r];
    __syncwarp();
    // stored component order of F: (00, 11, 22, 01, 02, 12) = 0..5
    float2* f1 = F + (((long)b * 6 + 2 * h3) * N * N + row) * ncp;
    float2* f2 = f1 + (long)N * N * ncp;
    for (int k = jj; k <= n_c; k += P) {
      const float2 zk = L.base[L.idx(k)];
      const float2 zm = conjg<float>(L.base[L.idx((N - k) & (N - 1))]);
      f1[k] = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y + zm.y));
      f2[k] = make_float2(0.5f * (zk.y - zm.y), -0.5f * (zk.x - zm.x));
    }
    __syncwarp();
  }
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  if (warp == 0) tmem_dealloc(*tslot, CF::NCOLS);
}

// F2: forward DFT along axis 1 of F[b][comp][a0][a1][k2] (k2 = 0..n_c), keeping n1 in [n1lo, n1lo + nk1).  F is the
// sum, in order, of `parts` partial fields fgstride elements apart (one per term group of the pass before).
template <typename T, int N>
__global__ void __launch_bounds__(256) k_f2(const cx<T>* __restrict__ F, int parts, long fgstride,
                                            cx<T>* __restrict__ F2, int n_c, int n1lo, int nk1,
                                            const cx<T>* __restrict__ tw) {
  using SH = Shape<T, N>;
  constexpr int E = SH::ES, P = SH::PS, TC = SH::TC;
  // one exchange buffer (a CTA runs one transform): half the shared memory of two, so more CTAs share an SM
  using Lay = ColLayout<T, N, TC, E, true>;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int c = threadIdx.x % TC, j = threadIdx.x / TC;
  const Lay L{reinterpret_cast<cx<T>*>(smraw), c};
  const int ncp = n_c + 1;
  const int cc = blockIdx.x * TC + c;
  const bool valid = cc < ncp;
  const int a0 = blockIdx.y;
  const long bc = blockIdx.z;  // b * 6 + comp
  const cx<T>* in = F + (bc * N + a0) * (long)N * ncp + cc;
  cx<T> v[E];
#pragma unroll
  for (int r = 0; r < E; ++r) v[r] = valid ? in[(long)(j + r * P) * ncp] : mk<T>((T)0, (T)0);
  for (int g = 1; g < parts; ++g) {
    in += fgstride;
#pragma unroll
    for (int r = 0; r < E; ++r)
      if (valid) v[r] = add<T>(v[r], in[(long)(j + r * P) * ncp]);
  }
  fft_pencil<T, N, E, -1, Lay, SyncBlock, false>(v, j, L, tw, SyncBlock());
  if (valid) {
    cx<T>* out = F2 + (bc * N + a0) * (long)nk1 * ncp + cc;
#pragma unroll
    for (int r = 0; r < E; ++r) {
      const int idx = wrapn(j + r * P, N) - n1lo;
      if (idx >= 0 && idx < nk1) out[(long)idx * ncp] = v[r];
    }
  }
}

// The two TT amplitudes e^+_ij(k_hat) S_ij and e^x_ij(k_hat) S_ij (Sec. sec_sigw basis: u = k x e0 / |k x e0|,
// e1 in place of e0 when k is parallel to e0, v = k x u; e^+ = (uu - vv)/sqrt2, e^x = (uv + vu)/sqrt2).
// S = (00, 11, 22, 01, 02, 12).  With the integer vector n, m2 = n1^2 + n2^2 and U = (0, n2, -n1), V = (-m2, n0 n1, n0 n2):
// u = U / sqrt(m2), v = V / (|n| sqrt(m2)), so one root and one division serve all (FP64; six divisions and two roots made
// this the larger part of a jackknife's last forward pass).
__device__ __forceinline__ void tt_amp(int n0, int n1, int n2, const double2* S, double2& ap, double2& ax) {
  const double2 s00 = S[0], s11 = S[1], s22 = S[2], s01 = S[3], s02 = S[4], s12 = S[5];
  const double h = 0.70710678118654752440, q = 1.41421356237309504880;
  const int m2 = n1 * n1 + n2 * n2;
  if (m2 == 0) {  // k along e0: u = (0, 0, sign n0), v = (0, -1, 0)
    const double sg = n0 < 0 ? q : -q;
    ap = make_double2((s22.x - s11.x) * h, (s22.y - s11.y) * h);
    ax = make_double2(sg * s12.x, sg * s12.y);
    return;
  }
  const double a0 = n0, a1 = n1, a2 = n2, m = m2, nn2 = (double)(n0 * n0 + m2);
  const double inv = 1.0 / (nn2 * m);  // 1 / (|n|^2 m2)
  const double iu = nn2 * inv, iw = sqrt(nn2) * inv;
  auto part = [&](double p00, double p11, double p22, double p01, double p02, double p12, double& plus, double& cross) {
    const double uu = a2 * a2 * p11 + a1 * a1 * p22 - 2.0 * a1 * a2 * p12;
    const double x1 = a1 * p01 + a2 * p02;                                   // (0, n1, n2) . S . e0
    const double x2 = a1 * a1 * p11 + a2 * a2 * p22 + 2.0 * a1 * a2 * p12;   // (0, n1, n2) . S . (0, n1, n2)
    const double vv = m * m * p00 - 2.0 * m * a0 * x1 + a0 * a0 * x2;
    const double uv = -m * (a2 * p01 - a1 * p02) + a0 * (a1 * a2 * (p11 - p22) + (a2 * a2 - a1 * a1) * p12);
    plus = (uu * iu - vv * inv) * h;
    cross = uv * iw * q;
  };
  part(s00.x, s11.x, s22.x, s01.x, s02.x, s12.x, ap.x, ax.x);
  part(s00.y, s11.y, s22.y, s01.y, s02.y, s12.y, ap.y, ax.y);
}
// Sum over the two polarisations of |e^l_ij(k_hat) S_ij|^2, written with the TT projector instead of the basis:
// sum_l e^l_ij e^l_lm = (P_il P_jm + P_im P_jl - P_ij P_lm) / 2 with P = I - n n^T / |n|^2, which annihilates the
// identity, so S may first lose its trace (S' = S - tr(S) I / 3; that also removes most of the cancellation when S
// is near-isotropic).  For symmetric S':
//   |S'|^2 - 2 |S' n|^2 / |n|^2 + |n.S'.n|^2 / (2 |n|^4),
// rational in the integer mode (one division, no square root) and the same for n and -n.
// R is the arithmetic type (FP64 for the FP64 path).
template <typename R>
__device__ __forceinline__ R tt_power(int n0, int n1, int n2, const cx<R>* S) {
  const R m0 = (R)n0, m1 = (R)n1, m2 = (R)n2;
  const R inv = (R)1 / (m0 * m0 + m1 * m1 + m2 * m2);
  const R third = (R)1 / (R)3;
  const R tx = (S[0].x + S[1].x + S[2].x) * third, ty = (S[0].y + S[1].y + S[2].y) * third;
  const cx<R> s00 = mk<R>(S[0].x - tx, S[0].y - ty), s11 = mk<R>(S[1].x - tx, S[1].y - ty),
              s22 = mk<R>(S[2].x - tx, S[2].y - ty), s01 = S[3], s02 = S[4], s12 = S[5];
  const cx<R> a0 = mk<R>(s00.x * m0 + s01.x * m1 + s02.x * m2, s00.y * m0 + s01.y * m1 + s02.y * m2);
  const cx<R> a1 = mk<R>(s01.x * m0 + s11.x * m1 + s12.x * m2, s01.y * m0 + s11.y * m1 + s12.y * m2);
  const cx<R> a2 = mk<R>(s02.x * m0 + s12.x * m1 + s22.x * m2, s02.y * m0 + s12.y * m1 + s22.y * m2);
  const R qx = m0 * a0.x + m1 * a1.x + m2 * a2.x, qy = m0 * a0.y + m1 * a1.y + m2 * a2.y;
  const R ss = s00.x * s00.x + s00.y * s00.y + s11.x * s11.x + s11.y * s11.y + s22.x * s22.x + s22.y * s22.y +
               (R)2 * (s01.x * s01.x + s01.y * s01.y + s02.x * s02.x + s02.y * s02.y + s12.x * s12.x +
                       s12.y * s12.y);
  const R aa = a0.x * a0.x + a0.y * a0.y + a1.x * a1.x + a1.y * a1.y + a2.x * a2.x + a2.y * a2.y;
  return ss - (R)2 * aa * inv + (R)0.5 * (qx * qx + qy * qy) * inv * inv;
}
// The same power from FP32 components, evaluated in FP32 (the FP32 path's S carries FP32 rounding already; the
// shell sums stay FP64, and their relative error is of order eps_32 |S|^2 / power, ~1e-6).  S is first scaled by an
// exact power of two that brings its largest component near 1, so neither the squares nor the |n|^2 factors leave
// the FP32 range, and the factor is put back in FP64.
__device__ __forceinline__ double tt_power_f32(int n0, int n1, int n2, const float2* S) {
  uint32_t mb = 0;
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    mb = max(mb, __float_as_uint(S[q].x) & 0x7fffffffu);
    mb = max(mb, __float_as_uint(S[q].y) & 0x7fffffffu);
  }
  if (mb == 0) return 0.0;
  const int e = min(max((int)(mb >> 23) - 127, -126), 126);  // exponent of the largest component
  const float sc = __uint_as_float((uint32_t)(127 - e) << 23);  // 2^-e
  float2 T[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) T[q] = make_float2(S[q].x * sc, S[q].y * sc);
  const double back = __longlong_as_double((long long)(1023 + 2 * e) << 52);  // 2^(2e)
  return (double)tt_power<float>(n0, n1, n2, T) * back;
}

// F3: forward DFT along axis 0 of the six components for a tile of columns (n1 fixed, n2 = k2),
// TT projection on the modes of shell n_c and the FP64 sum, one partial per CTA.
// Half-spectrum weight: a stored mode with 0 < k2 < H also stands for its partner wrap(-n), whose
// direction is -n_hat except on Nyquist indices; the partner is projected with its own direction.
// With Xj (jackknife), the amplitudes of the stored shell modes are also written to the standard half spectra
// Xj[b][0] = e^+ : S and Xj[b][1] = -i e^x : S (both Hermitian in this basis away from the Nyquist shell),
// [b][f][k0][k1][k2], k2 = 0..N/2; every other entry is left as it is (zero).
// blockIdx.z = m * batch + b: the fields of kernel m follow those of the one before (F2 and Xj), and its partial sums are
// mstride further.
template <typename T, int N>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 2 : 1) k_f3(const cx<T>* __restrict__ F2, int n_c, int n1lo, int nk1,
                                            double* __restrict__ partial, long pbstride, long mstride,
                                            int batch, const cx<T>* __restrict__ tw, cx<T>* __restrict__ Xj) {
  using SH = Shape<T, N>;
  constexpr int E = SH::E3, P = SH::P3, TC = SH::TC3, H = N / 2;
  using Lay = ColLayout<T, N, TC, E>;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ double red[32];
  const int c = threadIdx.x % TC, j = threadIdx.x / TC;
  const Lay L{reinterpret_cast<cx<T>*>(smraw), c};
  const int ncp = n_c + 1;
  const int k1i = blockIdx.y;
  const int n1 = n1lo + k1i;
  const int b = blockIdx.z;  // m * batch + realisation
  partial += (long)(b % batch) * pbstride + (long)(b / batch) * mstride;
  const long blk = (long)blockIdx.y * gridDim.x + blockIdx.x;
  const int cc0 = blockIdx.x * TC;
  const int rmax = n_c * n_c + n_c;  // |n|^2 < (n_c + 1/2)^2
  const int rmin = n_c * n_c - n_c + 1;  // |n|^2 >= (n_c - 1/2)^2
  if (!(cc0 < ncp && n1 * n1 + cc0 * cc0 <= rmax)) {  // no column of this tile reaches the shell
    if (threadIdx.x == 0) partial[blk] = 0.0;
    return;
  }
  const int cc = cc0 + c;
  const bool valid = cc < ncp && n1 * n1 + cc * cc <= rmax;
  // all six components are loaded before the first transform, so their latencies overlap (a barrier inside a
  // transform would otherwise hold back the loads of the next component)
  cx<T> X[6][E];
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const cx<T>* in = F2 + (((long)b * 6 + q) * N * nk1 + k1i) * (long)ncp + (valid ? cc : 0);
#pragma unroll
    for (int r = 0; r < E; ++r) X[q][r] = valid ? in[(long)(j + r * P) * nk1 * ncp] : mk<T>((T)0, (T)0);
  }
#pragma unroll
  for (int q = 0; q < 6; ++q) fft_pencil<T, N, E, -1, Lay, SyncBlock>(X[q], j, L, tw, SyncBlock());
  double acc = 0.0;
  if (valid) {
    const int n2 = cc;
#pragma unroll
    for (int r = 0; r < E; ++r) {
      const int n0 = wrapn(j + r * P, N);
      const int msq = n0 * n0 + n1 * n1 + n2 * n2;
      if (msq >= rmin && msq <= rmax) {
        cx<T> St[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) St[q] = X[q][r];
        auto power = [&](int a0, int a1, int a2) -> double {
          if constexpr (sizeof(T) == 4) return tt_power_f32(a0, a1, a2, St);
          else return tt_power<T>(a0, a1, a2, St);
        };
        const double pw = power(n0, n1, n2);
        acc += pw;
        if (Xj) {
          double2 S[6];
#pragma unroll
          for (int q = 0; q < 6; ++q) S[q] = make_double2((double)X[q][r].x, (double)X[q][r].y);
          double2 ap, ax;
          tt_amp(n0, n1, n2, S, ap, ax);
          constexpr long NNH = (long)N * N * (H + 1);
          const long o = ((long)b * 2 * N + (j + r * P)) * N * (H + 1) + (long)((n1 + N) % N) * (H + 1) + n2;
          Xj[o] = mk<T>((T)ap.x, (T)ap.y);
          Xj[o + NNH] = mk<T>((T)ax.y, (T)-ax.x);
        }
        if (n2 > 0 && n2 < H) {  // the partner -n has the same projector unless n0 or n1 is a Nyquist index
          if (n0 == H || n1 == H) {
            const int p0 = (n0 == H) ? H : -n0, p1 = (n1 == H) ? H : -n1;
            acc += power(p0, p1, -n2);
          } else {
            acc += pw;
          }
        }
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x + 31) / 32; ++w) t += red[w];
    partial[blk] = t;
  }
}

// Jackknife sub-volume energies: for field f (blockIdx.y) of R[f][x0][x1][x2] and sub-volume `sub` of the M^3
// blocks of s = N/M cells per side, CTA (sub, t) sums R^2 over the plane x0 = a s + t of that block in FP64:
// out[(f * M^3 + sub) * s + t].
template <typename T>
__global__ void __launch_bounds__(256) k_subvol(const T* __restrict__ R, int N, int M, double* __restrict__ out) {
  __shared__ double red[8];
  const int s = N / M;
  const int t = blockIdx.x % s, sub = blockIdx.x / s;
  const int a = sub / (M * M), bb = (sub / M) % M, c = sub % M;
  const long f = blockIdx.y;
  const T* plane = R + (f * N + (long)a * s + t) * N * N;
  double acc = 0.0;
  for (int e = threadIdx.x; e < s * s; e += blockDim.x) {
    const int x1 = bb * s + e / s, x2 = c * s + e % s;
    const double v = (double)plane[(long)x1 * N + x2];
    acc += v * v;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tot = 0.0;
    for (int w = 0; w < (int)(blockDim.x + 31) / 32; ++w) tot += red[w];
    out[(f * M * M * M + sub) * s + t] = tot;
  }
}

#ifdef SIGW_COMMON_KERNELS
// Synthesis amplitude sqrt(P_zeta(k) dx^3) per integer |n|^2 (k = k_f |n|), P_zeta = 2 pi^2 Delta^2 / k^3 with the
// log-normal Delta^2 of Eq. eq_lognormal: amp[b][msq], msq = 0..msq_max (zero at 0).  Evaluated in FP64; on the host it
// took longer than the rest of a call's host work (4 realisations at 256^3: 197 k logarithms and exponentials, 3.6 ms).
template <typename T>
__global__ void k_amp(const PzArgs* __restrict__ pz, T* __restrict__ amp, long msq1, double L, int N) {
  const long msq = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (msq >= msq1) return;
  const int b = blockIdx.y;
  double v = 0.0;
  if (msq > 0) {
    const double pi = 3.14159265358979323846;
    const double dx = L / N, sg = pz[b].sigma;
    const double k = 2.0 * pi / L * sqrt((double)msq);
    const double lk = log(k / pz[b].kstar);
    const double d2 = pz[b].A / sqrt(2.0 * pi * sg * sg) * exp(-lk * lk / (2.0 * sg * sg));
    v = sqrt(2.0 * pi * pi * d2 / (k * k * k) * dx * dx * dx);
  }
  amp[b * msq1 + msq] = (T)v;
}

// Deterministic second-stage reduction and the Omega constants:
//   P_X = C^2 sum / (V N_k), C = 4 dx^3 / (n_c^2 V^2), Omega = k_c^3 / (48 pi^2) (P_A + P_B).
// One CTA per (realisation, shell), two warps per kernel: 64 threads add strided partials, then a
// fixed tree.  (One thread per pair walked up to 33 k partials: 0.52 ms at 256^3, 1.04 ms at 512^3.)
__global__ void __launch_bounds__(128) k_fin(const double* __restrict__ partial, long pbstride, int maxblk, int n_shells,
                                             const __grid_constant__ ShellList shells,
                                             const double* __restrict__ Nk, int N, double L, int tc3, double* __restrict__ out) {
  __shared__ double red[4];
  const int b = blockIdx.x / n_shells, s = blockIdx.x % n_shells;
  const int n_c = shells.n_c[s];
  const int H = N / 2;
  const int n1lo = max(-n_c, -H + 1), n1hi = min(n_c, H);
  const int nk1 = n1hi - n1lo + 1;
  const int nblk = ((n_c + 1 + tc3 - 1) / tc3) * nk1;
  const int m = threadIdx.x >> 6;
  const double* p = partial + (long)b * pbstride + ((long)s * 2 + m) * maxblk;
  double t = 0.0;
#pragma unroll 4
  for (int k = threadIdx.x & 63; k < nblk; k += 64) t += p[k];
  for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x) return;
  const double pi = 3.14159265358979323846;
  const double V = L * L * L, dx = L / N;
  const double C = 4.0 * dx * dx * dx / ((double)n_c * n_c * V * V);
  const double nk = Nk[n_c - 1];
  const double PA = C * C * (red[0] + red[1]) / (V * nk), PB = C * C * (red[2] + red[3]) / (V * nk);
  const double kc = n_c * 2.0 * pi / L;
  double* o = out + (long)blockIdx.x * 4;
  o[0] = PA;
  o[1] = PB;
  o[2] = nk;
  o[3] = kc * kc * kc / (48.0 * pi * pi) * (PA + PB);
}

#endif

}  // namespace sigw
