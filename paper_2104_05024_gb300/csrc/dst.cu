// Box solver of the corrected 5/7-point system by sine transforms
// (Sections 5.2-5.3: the correction leaves the symmetric definite matrix
// unchanged, so an FFT-based fast Poisson/Helmholtz solver applies).
//
//   v = (2/N)^d S( mu^{-1} o S r ),   S_{kp} = sin(pi k p / N),  k, p = 1..N-1,
//   mu_p = sum_a mu1[p_a] - lambda,  mu1[p] = -(4/h^2) sin^2(pi p / (2N)).
//
// Work arrays are padded to N^d with index 0 of every axis holding the zero
// Dirichlet value, so every line of the DST-I of length N-1 is a length-N row
// starting at an aligned address.  Each 1-D DST-I of length N-1 runs as: sine
// pre-fold into a real sequence of length N, complex FFT of length N/2, split
// into the real DFT, and a prefix sum for the odd outputs: float64 lines in
// 64-bit block fixed point (dst_fix.cuh), float32 lines in registers
// (dst_reg.cuh), lines shorter than 32 by a Stockham FFT in shared memory.  A
// block owns a tile of W independent lines laid out [transform index][line] so that every butterfly
// stage is vectorised across the lines (consecutive threads touch consecutive
// words).  Passes:
//   x forward  : assembles r = alpha*src + corrections (irregular nodes) while
//                loading, transforms along x;
//   y forward  : strided rows, coalesced W-wide segments;
//   z solve    : elimination per (x, y) mode, or forward DST, spectral divide,
//                inverse DST in one pass;
//   y forward  : (the DST-I is its own inverse up to the folded scale);
//   x inverse  : transforms along x and writes the padded grid and/or a user
//                layout output  beta*v + gamma*aux.
// In 2-D the middle pass is the y solve.
#include <cuda_runtime.h>

#include <cudaTypedefs.h>

#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>

#include "dst_fix.cuh"
#include "dst_reg.cuh"
#include "ffloat.cuh"
#include "internal.cuh"

namespace kfbi {
namespace {

// Compiled twice, with KFBI_DST_BITS = 32 and 64 (the float32 and the float64
// kernels, in parallel): everything below is templates but for the entry
// points at the end, which are split by type.
#if KFBI_DST_BITS != 32 && KFBI_DST_BITS != 64
#error "KFBI_DST_BITS must be 32 or 64"
#endif

constexpr int NT = 256;

// float64 <-> T for float T on the bit patterns (a float64 conversion
// instruction costs as much as a float64 add here); identities for double
template <typename T>
__device__ __forceinline__ T to_T(double x) {
  if constexpr (sizeof(T) == 4)
    return ffl::narrow(x);
  else
    return x;
}
template <typename T>
__device__ __forceinline__ double to_double(T v) {
  if constexpr (sizeof(T) == 4)
    return ffl::widen(v);
  else
    return v;
}

// Tile geometry: N transform rows by W independent lines, row stride RS
// (W + 1 pads against bank conflicts of transposed loads; W for dense TMA
// tiles), G threads per line in the scan.
template <typename T_, int N_, int W_, int RS_>
struct Tile {
  using T = T_;
  static constexpr int N = N_, W = W_, RS = RS_;
  static constexpr int L = N / 2;
  static constexpr int G = NT / W;
  // fixed-point DST of float64 lines, register DST of float32 lines; shorter
  // lines take the Stockham path in shared memory
  static constexpr bool FIX = sizeof(T) == 8 && N >= 32;
  static constexpr bool REG = sizeof(T) == 4 && N >= 32 && N <= 512;
  // tables and scratch: those of the fixed-point path, or scan totals,
  // twiddles e^{i pi j/N} (2N complex) and sines (register path)
  static constexpr size_t mem_elems = FIX ? fixdst::table_words<N>() : (size_t)G * W + 4 * N + N;
  static constexpr size_t smem_elems = (size_t)N * RS + mem_elems;
  // resident blocks per SM the registers are budgeted for (shared memory
  // allows no more for long lines)
  static constexpr int BLOCKS = FIX ? (N <= 256 ? 2 : 1) : REG ? (N <= 256 ? 4 : 2) : 1;
};

template <typename T, int N>
struct WSel {
  static constexpr int W = N < 32 ? N : 32;
};

template <typename T, int N>
struct Cfg : Tile<T, N, WSel<T, N>::W, WSel<T, N>::W + 1> {};

__host__ __device__ constexpr int pick_radix(int L) {
  return (L % 8 == 0) ? 8 : (L % 4 == 0) ? 4 : (L % 2 == 0) ? 2 : (L % 3 == 0) ? 3 : 0;
}

// ---------------------------------------------------------------- butterflies
template <typename T, int R>
struct Dft;

template <typename T>
struct Dft<T, 2> {
  static __device__ __forceinline__ void run(T* xr, T* xi) {
    T ar = xr[0] + xr[1], ai = xi[0] + xi[1];
    xr[1] = xr[0] - xr[1];
    xi[1] = xi[0] - xi[1];
    xr[0] = ar;
    xi[0] = ai;
  }
};

// b_p = sum_q a_q e^{+2 pi i p q / 4}
template <typename T>
struct Dft<T, 4> {
  static __device__ __forceinline__ void run(T* xr, T* xi) {
    T t0r = xr[0] + xr[2], t0i = xi[0] + xi[2];
    T t1r = xr[0] - xr[2], t1i = xi[0] - xi[2];
    T t2r = xr[1] + xr[3], t2i = xi[1] + xi[3];
    T t3r = xr[1] - xr[3], t3i = xi[1] - xi[3];
    xr[0] = t0r + t2r;
    xi[0] = t0i + t2i;
    xr[2] = t0r - t2r;
    xi[2] = t0i - t2i;
    // b1 = t1 + i t3, b3 = t1 - i t3
    xr[1] = t1r - t3i;
    xi[1] = t1i + t3r;
    xr[3] = t1r + t3i;
    xi[3] = t1i - t3r;
  }
};

template <typename T>
struct Dft<T, 8> {
  static __device__ __forceinline__ void run(T* xr, T* xi) {
    T er[4] = {xr[0], xr[2], xr[4], xr[6]}, ei[4] = {xi[0], xi[2], xi[4], xi[6]};
    T orr[4] = {xr[1], xr[3], xr[5], xr[7]}, oi[4] = {xi[1], xi[3], xi[5], xi[7]};
    Dft<T, 4>::run(er, ei);
    Dft<T, 4>::run(orr, oi);
    const T c = (T)0.70710678118654752440;
    // w8^p O_p with w8 = e^{+i pi/4}
    T w1r = c * (orr[1] - oi[1]), w1i = c * (orr[1] + oi[1]);
    T w2r = -oi[2], w2i = orr[2];
    T w3r = -c * (orr[3] + oi[3]), w3i = c * (orr[3] - oi[3]);
    xr[0] = er[0] + orr[0];
    xi[0] = ei[0] + oi[0];
    xr[4] = er[0] - orr[0];
    xi[4] = ei[0] - oi[0];
    xr[1] = er[1] + w1r;
    xi[1] = ei[1] + w1i;
    xr[5] = er[1] - w1r;
    xi[5] = ei[1] - w1i;
    xr[2] = er[2] + w2r;
    xi[2] = ei[2] + w2i;
    xr[6] = er[2] - w2r;
    xi[6] = ei[2] - w2i;
    xr[3] = er[3] + w3r;
    xi[3] = ei[3] + w3i;
    xr[7] = er[3] - w3r;
    xi[7] = ei[3] - w3i;
  }
};

template <typename T>
struct Dft<T, 3> {
  static __device__ __forceinline__ void run(T* xr, T* xi) {
    const T s3 = (T)0.86602540378443864676;
    T tr = xr[1] + xr[2], ti = xi[1] + xi[2];
    T ur = xr[1] - xr[2], ui = xi[1] - xi[2];
    T mr = xr[0] - (T)0.5 * tr, mi = xi[0] - (T)0.5 * ti;
    xr[0] = xr[0] + tr;
    xi[0] = xi[0] + ti;
    // b1 = m + i s3 u, b2 = m - i s3 u
    xr[1] = mr - s3 * ui;
    xi[1] = mi + s3 * ur;
    xr[2] = mr + s3 * ui;
    xi[2] = mi - s3 * ur;
  }
};

// One in-place Stockham stage of radix R on the complex sequence stored in
// rows (2m, 2m+1) of every column.  All reads precede all writes.  Ls is a
// compile-time constant so every index division is a shift or a constant.
template <typename C, int R, int Ls>
__device__ __forceinline__ void fft_stage(typename C::T* s, const typename C::T* tw) {
  using T = typename C::T;
  constexpr int L = C::L, W = C::W, RS = C::RS;
  constexpr int NB = (L / R) * W;
  constexpr int PER = NB > 0 ? (NB + NT - 1) / NT : 1;  // stages never taken for small L still compile
  T xr[PER][R], xi[PER][R];
#pragma unroll
  for (int b = 0; b < PER; ++b) {
    const int idx = threadIdx.x + b * NT;
    if (idx < NB) {
      const int c = idx % W, j = idx / W, k = j % Ls;
      const int tstep = (L / (R * Ls)) * k;
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const int m = j + q * (L / R);
        T ar = s[(2 * m) * RS + c], ai = s[(2 * m + 1) * RS + c];
        if (q > 0) {
          const int e = 4 * ((tstep * q) % L);
          const T wr = tw[2 * e], wi = tw[2 * e + 1];
          const T t = ar * wr - ai * wi;
          ai = ar * wi + ai * wr;
          ar = t;
        }
        xr[b][q] = ar;
        xi[b][q] = ai;
      }
      Dft<T, R>::run(xr[b], xi[b]);
    }
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < PER; ++b) {
    const int idx = threadIdx.x + b * NT;
    if (idx < NB) {
      const int c = idx % W, j = idx / W, k = j % Ls;
      const int base = (j - k) * R + k;
#pragma unroll
      for (int p = 0; p < R; ++p) {
        const int m = base + p * Ls;
        s[(2 * m) * RS + c] = xr[b][p];
        s[(2 * m + 1) * RS + c] = xi[b][p];
      }
    }
  }
  __syncthreads();
}

// the stage sequence of a length-Lrem transform, unrolled at compile time
template <typename C, int Ls, int Lrem>
struct Stages {
  static __device__ __forceinline__ void run(typename C::T* s, const typename C::T* tw) {
    constexpr int R = pick_radix(Lrem);
    fft_stage<C, R, Ls>(s, tw);
    Stages<C, Ls * R, Lrem / R>::run(s, tw);
  }
};
template <typename C, int Ls>
struct Stages<C, Ls, 1> {
  static __device__ __forceinline__ void run(typename C::T*, const typename C::T*) {}
};

// DST-I of every column of the tile s[N][RS] (rows 1..N-1 in, rows 1..N-1
// out, row 0 holds 0).  tw = e^{i pi j / N}, j = 0..2N-1 (interleaved re, im);
// tot = scan scratch [G][W].
template <typename C>
__device__ void dst1_tile(typename C::T* s, const typename C::T* tw, typename C::T* tot) {
  using T = typename C::T;
  constexpr int N = C::N, L = C::L, W = C::W, RS = C::RS, G = C::G;
  // sine pre-fold: y_j = sin(j pi/N)(x_j + x_{N-j}) + (x_j - x_{N-j})/2
  for (int idx = threadIdx.x; idx < (N / 2 + 1) * W; idx += NT) {
    const int c = idx % W, j = idx / W;
    if (j == 0) {
      s[c] = (T)0;
    } else if (j == N / 2) {
      s[j * RS + c] *= (T)2;
    } else {
      const T a = s[j * RS + c], b = s[(N - j) * RS + c];
      const T sj = tw[2 * j + 1];
      const T t1 = sj * (a + b), t2 = (T)0.5 * (a - b);
      s[j * RS + c] = t1 + t2;
      s[(N - j) * RS + c] = t1 - t2;
    }
  }
  __syncthreads();
  // complex FFT of length L = N/2 on z_m = y_{2m} + i y_{2m+1}
  Stages<C, 1, L>::run(s, tw);
  // real-DFT split: Y_k = (A + conj B)/2 - i w_k (A - conj B)/2, A = Z_k,
  // B = Z_{L-k}, w_k = e^{2 pi i k / N}; store I_k in row 2k, R_k in row 2k+1
  for (int idx = threadIdx.x; idx < (L / 2 + 1) * W; idx += NT) {
    const int c = idx % W, k = idx / W;
    if (k == 0) {
      const T a = s[c], b = s[RS + c];
      s[c] = (T)0;
      s[RS + c] = (T)0.5 * (a + b);  // F_1 = R_0 / 2
    } else {
      const int kk = L - k;
      const T Ar = s[(2 * k) * RS + c], Ai = s[(2 * k + 1) * RS + c];
      const T Br = s[(2 * kk) * RS + c], Bi = s[(2 * kk + 1) * RS + c];
      {
        const T wr = tw[2 * (2 * k)], wi = tw[2 * (2 * k) + 1];
        const T Sr = Ar + Br, Si = Ai - Bi, Dr = Ar - Br, Di = Ai + Bi;
        const T Yr = (T)0.5 * (Sr + wr * Di + wi * Dr);
        const T Yi = (T)0.5 * (Si - wr * Dr + wi * Di);
        s[(2 * k) * RS + c] = Yi;
        s[(2 * k + 1) * RS + c] = Yr;
      }
      if (kk != k) {
        const T wr = tw[2 * (2 * kk)], wi = tw[2 * (2 * kk) + 1];
        const T Sr = Br + Ar, Si = Bi - Ai, Dr = Br - Ar, Di = Bi + Ai;
        const T Yr = (T)0.5 * (Sr + wr * Di + wi * Dr);
        const T Yi = (T)0.5 * (Si - wr * Dr + wi * Di);
        s[(2 * kk) * RS + c] = Yi;
        s[(2 * kk + 1) * RS + c] = Yr;
      }
    }
  }
  __syncthreads();
  // odd outputs: F_{2k+1} = F_{2k-1} + R_k (column-wise inclusive scan)
  {
    constexpr int SEG = (L + G - 1) / G;
    const int c = threadIdx.x % W, g = threadIdx.x / W;
    const int k0 = g * SEG;
    const int k1 = (k0 + SEG < L) ? k0 + SEG : L;
    T acc = (T)0;
    for (int k = k0; k < k1; ++k) {
      acc += s[(2 * k + 1) * RS + c];
      s[(2 * k + 1) * RS + c] = acc;
    }
    tot[g * W + c] = acc;
    __syncthreads();
    T off = (T)0;
    for (int g2 = 0; g2 < g; ++g2) off += tot[g2 * W + c];
    for (int k = k0; k < k1; ++k) s[(2 * k + 1) * RS + c] += off;
    __syncthreads();
  }
}

template <typename T, int N>
__device__ __forceinline__ void load_twiddles(T* tw_s, const T* tw_g) {
  for (int i = threadIdx.x; i < 4 * N; i += NT) tw_s[i] = tw_g[i];
}

// Tile loads as asynchronous element copies (cp.async, 4 or 8 bytes): every
// copy of the tile is in flight at once instead of a few loads per thread,
// which is what keeps HBM busy when the grid does not fit in L2.
template <typename T>
__device__ __forceinline__ void copy_async(T* dst_smem, const T* src) {
  static_assert(sizeof(T) == 4 || sizeof(T) == 8, "element copies of 4 or 8 bytes");
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst_smem));
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(sizeof(T)) : "memory");
}
__device__ __forceinline__ void copy_async16(void* dst_smem, const void* src) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst_smem));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// sines sin(pi j / N) for the register path's pre-fold (imaginary parts of tw)
template <typename C>
__device__ __forceinline__ void load_sines(typename C::T* sinv, const typename C::T* tw_g) {
  if constexpr (C::REG)
    for (int i = threadIdx.x; i < C::N; i += NT) sinv[i] = tw_g[2 * i + 1];
}

// a tile's tables to shared memory mem[C::mem_elems] (before the first barrier)
template <typename C>
__device__ __forceinline__ void load_tables(typename C::T* mem, const typename C::T* tw_g) {
  if constexpr (C::FIX) {
    fixdst::load_tables<C::N>(reinterpret_cast<fixdst::ll*>(mem), tw_g);
  } else {
    typename C::T* tw = mem + C::G * C::W;
    load_twiddles<typename C::T, C::N>(tw, tw_g);
    load_sines<C>(tw + 4 * C::N, tw_g);
  }
}

struct NoMap {
  template <typename T>
  __device__ __forceinline__ T operator()(int, T v) const {
    return v;
  }
};

// the DST-I of every column of the tile, rows 1..N-1; map: applied to the
// outputs (register path only)
template <typename C, class Map = NoMap>
__device__ __forceinline__ void dst_tile(typename C::T* s, typename C::T* mem, const Map& map = Map()) {
  if constexpr (C::FIX) {
    fixdst::dst1_tile_fix<fixdst::Geo<C::N, C::RS>>(s, reinterpret_cast<fixdst::ll*>(mem));
  } else if constexpr (C::REG) {
    const typename C::T* tw = mem + C::G * C::W;
    regdst::dst1_tile_reg<regdst::Geo<C::N, C::RS>>(s, tw + 4 * C::N, reinterpret_cast<const regdst::cf2*>(tw), mem,
                                                    map);
  } else {
    dst1_tile<C>(s, mem + C::G * C::W, mem);
  }
}

// spectral divide v * scale / (mu1[j] + mu1[p] + mu1[q] - lambda) applied to
// the forward transform's outputs as they are written (register path)
struct DivPost {
  const float* mu;  // mu1 in shared memory
  float base;       // mu1[p] + mu1[q] - lambda
  float scale;
  bool zero;        // boundary column p = 0
  bool on = true;   // false: identity (the inverse transform of the same body)
  __device__ __forceinline__ float operator()(int j, float v) const {
    if (!on) return v;
    return zero ? 0.0f : v * __fdividef(scale, mu[j] + base);
  }
};

// how many of a lane's per values are loaded together: a divisor of per, 8 at
// most
__host__ __device__ constexpr int batch_of(int per) {
  int c = per < 8 ? per : 8;
  while (per % c != 0) --c;
  return c;
}

// The W x-lines y0 .. y0 + W - 1 of plane z of a field (interior nodes, rows
// of N - 1 values) to the tile s[x][line], mapped by f, with zeros at x = 0
// and on line y = 0.  A warp takes whole lines and issues a line's loads
// together (rows start at odd addresses, so each is a coalesced run of single
// values): with one load in flight per thread at a time a float64 source cost
// the 512^3 float32 pass 0.98 ms, four times the pass without a source.
template <typename C, int DIM, typename S, typename F>
__device__ __forceinline__ void fill_lines(typename C::T* s, const S* __restrict__ src, int y0, int z, const F& f) {
  constexpr int N = C::N, W = C::W, RS = C::RS, n1 = N - 1;
  if constexpr (N >= 32) {
    constexpr int PER = N / 32, CH = batch_of(PER);  // values per lane and line, loads issued together
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int c = threadIdx.x >> 5; c < W; c += NT / 32) {
      const int y = y0 + c;
      const S* row = src + ((DIM == 3 ? (size_t)(z - 1) * n1 : 0) + (y - 1)) * n1 - 1;
#pragma unroll
      for (int i0 = 0; i0 < PER; i0 += CH) {
        static_assert(PER % CH == 0, "whole batches");
        S v[CH];
#pragma unroll
        for (int i = 0; i < CH; ++i) {
          const int x = lane + 32 * (i0 + i);
          v[i] = x > 0 && y > 0 ? __ldg(&row[x]) : (S)0;
        }
#pragma unroll
        for (int i = 0; i < CH; ++i) s[(lane + 32 * (i0 + i)) * RS + c] = f(v[i]);
      }
    }
  } else {
    for (int idx = threadIdx.x; idx < N * W; idx += NT) {
      const int x = idx % N, c = idx / N, y = y0 + c;
      S v = (S)0;
      if (x > 0 && y > 0) v = src[((DIM == 3 ? (size_t)(z - 1) * n1 : 0) + (y - 1)) * n1 + (x - 1)];
      s[x * RS + c] = f(v);
    }
  }
}

// The corrections of the tile's lines y0 .. y0 + W - 1 of plane z (0 in 2-D),
// summed values (corr) or, in 2-D, CSR rows on the density vector (rows):
// each line's irregular nodes (distinct x, so distinct words) are shared out
// over the NT / W threads of its column.  In 2-D rows save the gather's own
// launch (4 us of 45); in 3-D the rows' dependent loads cost the x pass more
// than the gather kernel takes (A psi at 256^3 150 -> 156 us).
template <typename C, int DIM>
__device__ __forceinline__ void add_corrections(typename C::T* s, const double* __restrict__ corr, const CorrRows& rows,
                                                const int32_t* __restrict__ irr, const int32_t* __restrict__ line_start,
                                                int y0, int z) {
  using T = typename C::T;
  constexpr int W = C::W, RS = C::RS, n1 = C::N - 1, G = NT / W;
  const int c = threadIdx.x % W, g = threadIdx.x / W, y = y0 + c;
  if ((corr == nullptr && (DIM == 3 || rows.x == nullptr)) || y <= 0) return;
  const int line = DIM == 3 ? (z - 1) * n1 + (y - 1) : (y - 1);
  const int i0 = line_start[line], i1 = line_start[line + 1];
  for (int i = i0 + g; i < i1; i += G) {
    const int x = irr[i] % n1 + 1;
    double v = 0.0;
    if (DIM == 2 && rows.x != nullptr) {
      const int k1 = rows.ptr[i + 1];
#pragma unroll 4
      for (int k = rows.ptr[i]; k < k1; ++k) v += rows.w[k] * rows.x[rows.pid[k]];
    } else {
      v = corr[i];
    }
    s[x * RS + c] += (T)v;
  }
}

// ------------------------------------------------------------- x forward
// Tile: W consecutive lines y0..y0+W-1 of plane z; assembles
// r = alpha*src + corrections on the fly.
template <typename T, int N, int DIM>
__global__ void __launch_bounds__(NT, Cfg<T, N>::BLOCKS) k_xfwd(T* __restrict__ a, const double* __restrict__ src, double alpha,
                                             const float* __restrict__ src32,
                                             const double* __restrict__ corr, CorrRows rows,
                                             const int32_t* __restrict__ irr,
                                             const int32_t* __restrict__ line_start, const T* __restrict__ tw_g,
                                             const int* __restrict__ skip, int yoff, int zoff) {
  using C = Cfg<T, N>;
  constexpr int W = C::W, RS = C::RS, n1 = N - 1;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* s = reinterpret_cast<T*>(smem_raw);
  T* mem = s + N * RS;
  load_tables<C>(mem, tw_g);
  pdl_wait();
  if (skip != nullptr && *skip != 0) return;
  const int y0 = blockIdx.x * W + yoff;
  const int z = DIM == 3 ? blockIdx.y + zoff : 0;
  // the branch on src stays outside the loops: inside, the compiler
  // evaluates the (float64) scaling for every element, taken or not
  if (src != nullptr) {
    const T a_t = (T)alpha;
    fill_lines<C, DIM>(s, src, y0, z, [&](double v) { return a_t * to_T<T>(v); });
  } else if (src32 != nullptr) {
    fill_lines<C, DIM>(s, src32, y0, z, [&](float v) { return (T)v; });
  } else {
    for (int idx = threadIdx.x; idx < N * W; idx += NT) s[(idx % N) * RS + idx / N] = (T)0;
  }
  __syncthreads();
  add_corrections<C, DIM>(s, corr, rows, irr, line_start, y0, z);
  __syncthreads();
  dst_tile<C>(s, mem);
  pdl_launch_next();
  const size_t plane = (size_t)z * N * N;
  for (int idx = threadIdx.x; idx < N * W; idx += NT) {
    const int x = idx % N, c = idx / N;
    a[plane + (size_t)(y0 + c) * N + x] = s[x * RS + c];
  }
}

// The tile's lines y0 .. y0 + W - 1 of plane z to the work grid (keep) and/or
// to a field.
template <typename C, int DIM>
__device__ __forceinline__ void put_lines(const typename C::T* s, typename C::T* __restrict__ a, bool keep,
                                          double* __restrict__ out, const double* __restrict__ aux, double beta,
                                          double gamma, const float* __restrict__ aux32, int y0, int z) {
  using T = typename C::T;
  constexpr int N = C::N, W = C::W, RS = C::RS, n1 = N - 1;
  const size_t plane = (size_t)z * N * N;
  if (out == nullptr) {
    if (keep)
      for (int idx = threadIdx.x; idx < N * W; idx += NT) {
        const int x = idx % N, c = idx / N;
        a[plane + (size_t)(y0 + c) * N + x] = s[x * RS + c];
      }
    return;
  }
  // out = beta v + gamma aux with beta applied in T (one float64 operation
  // per element without aux, two with), or out = beta v + aux32 with aux32 a
  // padded float grid of the same layout as a (one float64 addition); a
  // line's loads of aux are issued together
  const T b_t = (T)beta;
  constexpr int LW = N < 32 ? N : 32;             // lanes along x
  constexpr int PER = N / LW, CH = batch_of(PER);
  const int lane = threadIdx.x % LW;
#pragma unroll 1
  for (int c = threadIdx.x / LW; c < W; c += NT / LW) {
    const int y = y0 + c;
    const size_t pidx = plane + (size_t)y * N + lane;
    const size_t o = ((DIM == 3 ? (size_t)(z - 1) * n1 : 0) + (y - 1)) * n1 + lane - 1;
#pragma unroll
    for (int i0 = 0; i0 < PER; i0 += CH) {
      double w[CH];
      if (aux32 != nullptr) {
#pragma unroll
        for (int i = 0; i < CH; ++i) w[i] = ffl::widen(aux32[pidx + LW * (i0 + i)]);
      } else if (aux != nullptr) {
#pragma unroll
        for (int i = 0; i < CH; ++i) w[i] = y > 0 && lane + i0 + i > 0 ? aux[o + LW * (i0 + i)] : 0.0;
      }
#pragma unroll
      for (int i = 0; i < CH; ++i) {
        const T v = s[(lane + LW * (i0 + i)) * RS + c];
        if (keep) a[pidx + LW * (i0 + i)] = v;
        if (y > 0 && lane + i0 + i > 0) {
          const double bv = to_double(b_t * v);
          out[o + LW * (i0 + i)] = aux32 != nullptr ? bv + w[i] : aux != nullptr ? fma(gamma, w[i], bv) : bv;
        }
      }
    }
  }
}

// ------------------------------------------------------------- x inverse
template <typename T, int N, int DIM>
__global__ void __launch_bounds__(NT, Cfg<T, N>::BLOCKS) k_xinv(T* __restrict__ a, bool keep, double* __restrict__ out,
                                             const double* __restrict__ aux, double beta, double gamma,
                                             const T* __restrict__ tw_g, const int* __restrict__ skip,
                                             const float* __restrict__ aux32, int yoff, int zoff) {
  using C = Cfg<T, N>;
  constexpr int W = C::W, RS = C::RS;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* s = reinterpret_cast<T*>(smem_raw);
  T* mem = s + N * RS;
  load_tables<C>(mem, tw_g);
  pdl_wait();
  if (skip != nullptr && *skip != 0) return;
  const int y0 = blockIdx.x * W + yoff;
  const int z = DIM == 3 ? blockIdx.y + zoff : 0;
  const size_t plane = (size_t)z * N * N;
  for (int idx = threadIdx.x; idx < N * W; idx += NT) {
    const int x = idx % N, c = idx / N;
    copy_async(&s[x * RS + c], &a[plane + (size_t)(y0 + c) * N + x]);
  }
  copy_async_wait();
  __syncthreads();
  dst_tile<C>(s, mem);
  pdl_launch_next();
  put_lines<C, DIM>(s, a, keep, out, aux, beta, gamma, aux32, y0, z);
}

// ------------------------------------------------ asynchronous bulk copies
constexpr int TMA_W = 32;
// a poll of an incomplete mbarrier takes about 4 us on GB300, so 2^18 polls give up
// after about a second (a tile load completes in microseconds)
constexpr long TMA_WAIT_CAP = 1L << 18;

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void tma_load3(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
          smem_addr(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_addr(bar))
      : "memory");
}
__device__ __forceinline__ void tma_store3(const CUtensorMap* map, const void* src, int x, int y, int z) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(x), "r"(y), "r"(z), "r"(smem_addr(src))
               : "memory");
}
__device__ __forceinline__ void tma_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void tma_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tma_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// bulk copies of contiguous bytes (multiples of 16, both addresses aligned
// to 16): completion on an mbarrier, or in the thread's bulk group
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}
__device__ __forceinline__ void bulk_store(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_addr(src)), "r"(bytes)
               : "memory");
}
// bounded wait of a whole phase; false when it gave up
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  for (long it = 0; it < TMA_WAIT_CAP; ++it)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

// --------------------------------------------------- strided (y / z) passes
// Tile rows = transform index k (stride row_stride), columns x0..x0+W-1 of
// plane q = blockIdx.y + qoff; rows outside `in` are zero and not read, rows
// outside `out` are not written.  SOLVE = forward DST, spectral multiply,
// inverse DST.  A row of a tile is 256 (float64) or 128 (float32) contiguous
// bytes (N >= 32).  Float64 rows move by one bulk copy of one thread each way:
// element copies with their addresses were 8 of 146 instructions per point.
// Float32 rows move by 16-byte asynchronous copies and vector stores (bulk
// copies of 128 bytes were slower: 393 against 286 us for the 512^3 y pass
// with element copies).
template <typename T, int N>
struct StridedCfg : Tile<T, N, WSel<T, N>::W, N >= 32 ? 32 : WSel<T, N>::W + 1> {};

template <typename T, int N, bool SOLVE, int DIM>
__global__ void __launch_bounds__(NT, StridedCfg<T, N>::BLOCKS) k_strided(
    T* __restrict__ a, size_t row_stride, size_t plane_stride, int qoff, const T* __restrict__ mu1, T lambda, T scale,
    const T* __restrict__ tw_g, const int* __restrict__ skip, const T* __restrict__ rinv, int reps, Span in, Span out,
    int* __restrict__ err) {
  using C = StridedCfg<T, N>;
  constexpr int W = C::W, RS = C::RS;
  constexpr bool BULK = N >= 32 && sizeof(T) == 8, VEC = N >= 32 && sizeof(T) == 4;
  constexpr uint32_t row_bytes = W * sizeof(T);
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar;
  T* s = reinterpret_cast<T*>(smem_raw);
  T* mem = s + N * RS;
  if (BULK && threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_fence_init();
    mbar_expect_tx(&bar, (uint32_t)(in.hi - in.lo) * row_bytes);
  }
  load_tables<C>(mem, tw_g);
  pdl_wait();
  if (skip != nullptr && *skip != 0) return;
  const int x0 = blockIdx.x * W;
  const int q = blockIdx.y + qoff;
  T* base = a + (size_t)q * plane_stride + x0;
  if constexpr (BULK) {
    __syncthreads();
    for (int k = in.lo + threadIdx.x; k < in.hi; k += NT)
      bulk_load(s + k * RS, base + (size_t)k * row_stride, row_bytes, &bar);
    if (SOLVE && C::FIX && rinv != nullptr)
      // the tile's mode factors on their way to L2 (read after the forward
      // transform)
      for (int k = threadIdx.x; k < 2 * N; k += NT)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(rinv + ((size_t)q * N + k / 2) * N + x0 + 16 * (k & 1)));
    for (int i = threadIdx.x; i < in.lo * W; i += NT) s[i] = (T)0;
    for (int i = in.hi * W + threadIdx.x; i < N * W; i += NT) s[i] = (T)0;
    if (!mbar_wait(&bar, 0u)) {
      // recorded by every thread that gives up (the others may go on without
      // it); the copies of this block finish before its shared memory goes
      if (err != nullptr) atomicOr(err, DEVERR_TIMEOUT);
      mbar_wait(&bar, 0u);
      return;
    }
  } else if constexpr (VEC) {
    const int c = 4 * (threadIdx.x & 7), k0 = in.lo + (threadIdx.x >> 3);
    const T* src = base + (size_t)k0 * row_stride + c;
#pragma unroll 4
    for (int k = k0; k < in.hi; k += NT / 8, src += NT / 8 * row_stride) copy_async16(s + k * RS + c, src);
    for (int i = threadIdx.x; i < in.lo * W; i += NT) s[i] = (T)0;
    for (int i = in.hi * W + threadIdx.x; i < N * W; i += NT) s[i] = (T)0;
    copy_async_wait();
  } else {
    constexpr int DR = NT / W;
    const int c = threadIdx.x % W;
    for (int k = threadIdx.x / W; k < N; k += DR)
      s[k * RS + c] = k >= in.lo && k < in.hi ? base[(size_t)k * row_stride + c] : (T)0;
  }
  __syncthreads();
  const T muq = DIM == 3 ? mu1[q] : (T)0;
  if constexpr (C::REG) {
    if constexpr (SOLVE) {
      // forward DST with the spectral divide applied to its outputs, then the
      // inverse DST by the same (single inlined) body; mu1 is read from
      // global memory (L1-resident, N values)
      const int p = x0 + (int)(threadIdx.x & 31);
      DivPost post{mu1, mu1[p] + muq - lambda, scale, p == 0, true};
#pragma unroll 1
      for (int rep = 0; rep < reps; ++rep) {
        dst_tile<C>(s, mem, post);
        post.on = false;
      }
    } else {
      dst_tile<C>(s, mem);
    }
  } else if constexpr (SOLVE) {
#pragma unroll 1
    for (int rep = 0; rep < reps; ++rep) {
      if (rep == 1) {
        // the mode factors scale / mu_p from the table built for this lambda
        // (same expression, so the same value), else divided here; a batch
        // of table values is loaded together
        constexpr int DR = NT / W, PER = (N + DR - 1) / DR, CH = batch_of(PER);
        const int c = threadIdx.x % W, k0 = threadIdx.x / W, p = x0 + c;
        const T* rq = rinv != nullptr ? rinv + (size_t)q * N * N + p : nullptr;
        const T base_mu = mu1[p] + muq - lambda;
#pragma unroll 1
        for (int i0 = 0; i0 < PER; i0 += CH) {
          T f[CH];
#pragma unroll
          for (int i = 0; i < CH; ++i) {
            const int k = k0 + DR * (i0 + i);
            if (k >= N) continue;
            if (rq != nullptr)
              f[i] = rq[(size_t)k * N];
            else
              f[i] = k > 0 && p > 0 ? scale / (mu1[k] + base_mu) : (T)0;
          }
#pragma unroll
          for (int i = 0; i < CH; ++i) {
            const int k = k0 + DR * (i0 + i);
            if (k < N) s[k * RS + c] *= f[i];
          }
        }
        __syncthreads();
      }
      dst_tile<C>(s, mem);
    }
  } else {
    dst_tile<C>(s, mem);
  }
  pdl_launch_next();
  if constexpr (BULK) {
    fence_async_shared();
    __syncthreads();
    for (int k = out.lo + threadIdx.x; k < out.hi; k += NT)
      bulk_store(base + (size_t)k * row_stride, s + k * RS, row_bytes);
    tma_commit();
    tma_wait_all();
  } else if constexpr (VEC) {
    const int c = 4 * (threadIdx.x & 7), k0 = out.lo + (threadIdx.x >> 3);
    T* dst = base + (size_t)k0 * row_stride + c;
#pragma unroll 4
    for (int k = k0; k < out.hi; k += NT / 8, dst += NT / 8 * row_stride)
      *reinterpret_cast<float4*>(dst) = *reinterpret_cast<const float4*>(s + k * RS + c);
  } else {
    constexpr int DR = NT / W;
    const int c = threadIdx.x % W;
    for (int k = out.lo + threadIdx.x / W; k < out.hi; k += DR) base[(size_t)k * row_stride + c] = s[k * RS + c];
  }
}

// ------------------------------------------- TMA-fed strided passes (float32)
// Persistent blocks walk over [N x 32] tiles of the padded float grid.  One
// thread issues a TMA tensor load of the next tile into the other shared
// buffer (completion counted on an mbarrier) while all threads transform the
// current tile; the finished tile goes back by a TMA tensor store.  Every
// wait is bounded: on timeout the block records DEVERR_TIMEOUT and returns.
// Three resident blocks per SM (shared memory allows three at N = 256), so 80
// registers.  At 256 rows the plain pass over whole rows just fits them, as
// long as it runs its single transform inside the runtime-bounded loop (the
// compile-time bound of one lets the compiler schedule it into spills); the
// other forms spill: 32 bytes a thread over ranges, 48 with the solve, 36 with
// both.
constexpr int TMA_BLOCKS = 3;

template <int N>
using TmaTile = Tile<float, N, TMA_W, TMA_W>;

// two tiles, scan totals, twiddles, sines, mu1, two mbarriers
template <int N>
constexpr size_t tma_smem_bytes() {
  return (2 * (size_t)N * TMA_W + (size_t)TmaTile<N>::G * TMA_W + 6 * (size_t)N) * sizeof(float) + 2 * sizeof(uint64_t);
}

// mode 0: tiles [y][x-chunk] of the planes z = q; mode 1: tiles [z][x-chunk]
// of the rows y = q, q in `planes`.  map_in / map_out: boxes of the rows `in`
// that are read (the others are zero) and `out` that are written; PART =
// false: all N of both (known at compile time: the runtime spans cost the
// 256-row kernels register spills, 24.5 -> 26.4 us a pass).
template <int N, bool SOLVE, bool PART>
__global__ void __launch_bounds__(NT, TMA_BLOCKS) k_strided_tma(const __grid_constant__ CUtensorMap map_in,
                                                    const __grid_constant__ CUtensorMap map_out, int mode,
                                                    Span planes_p, Span in_p, Span out_p,
                                                    const float* __restrict__ mu1, float lambda, float scale,
                                                    const float* __restrict__ tw_g, int* __restrict__ err,
                                                    int reps, const int* __restrict__ skip) {
  using C = TmaTile<N>;
  constexpr int W = TMA_W, NX = N / TMA_W;
  const Span planes = PART ? planes_p : Span{1, N}, in = PART ? in_p : Span{0, N}, out = PART ? out_p : Span{0, N};
  const int ntiles = NX * (planes.hi - planes.lo);
  const uint32_t bytes = (uint32_t)((in.hi - in.lo) * W * sizeof(float));
  extern __shared__ __align__(128) unsigned char smem_tma[];
  float* buf0 = reinterpret_cast<float*>(smem_tma);
  float* buf1 = buf0 + N * W;
  float* tot = buf1 + N * W;
  float* tw = tot + C::G * W;
  float* sinv = tw + 4 * N;
  float* mus = sinv + N;
  uint64_t* bar = reinterpret_cast<uint64_t*>(mus + N);
  for (int i = threadIdx.x; i < 4 * N; i += NT) tw[i] = tw_g[i];
  for (int i = threadIdx.x; i < N; i += NT) {
    sinv[i] = tw_g[2 * i + 1];
    mus[i] = mu1[i];
  }
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_fence_init();
  }
  pdl_wait();
  // an iteration enqueued ahead of the convergence test: nothing to do (the
  // flag is tested before any copy is issued)
  if (skip != nullptr && *skip != 0) return;
  pdl_launch_next();
  __syncthreads();
  auto coords = [&](int t, int row, int& x, int& y, int& z) {
    const int q = t / NX + planes.lo;
    x = (t % NX) * W;
    y = mode == 0 ? row : q;
    z = mode == 0 ? q : row;
  };
  int t = blockIdx.x;
  if (t < ntiles && threadIdx.x == 0) {
    int x, y, z;
    coords(t, in.lo, x, y, z);
    mbar_expect_tx(&bar[0], bytes);
    tma_load3(buf0 + in.lo * W, &map_in, &bar[0], x, y, z);
  }
  for (int i = 0; t < ntiles; t += gridDim.x, ++i) {
    const int b = i & 1;
    float* s = b ? buf1 : buf0;
    float* s_next = b ? buf0 : buf1;
    const int tn = t + gridDim.x;
    if (threadIdx.x == 0 && tn < ntiles) {
      tma_wait_read_all();  // the store of the previous tile has left s_next
      int x, y, z;
      coords(tn, in.lo, x, y, z);
      mbar_expect_tx(&bar[b ^ 1], bytes);
      tma_load3(s_next + in.lo * W, &map_in, &bar[b ^ 1], x, y, z);
    }
    bool ok = false;
    for (long it = 0; it < TMA_WAIT_CAP; ++it)
      if (mbar_try_wait(&bar[b], (uint32_t)((i >> 1) & 1))) {
        ok = true;
        break;
      }
    if (!ok) {
      atomicOr(err, DEVERR_TIMEOUT);  // by every thread that gives up
      if (threadIdx.x == 0) {
        // the copies this block issued finish before its shared memory goes:
        // stores by their bulk group, the pending load by its barrier
        tma_wait_all();
        if (tn < ntiles)
          for (long it = 0; it < TMA_WAIT_CAP; ++it)
            if (mbar_try_wait(&bar[b ^ 1], (uint32_t)(((i + 1) >> 1) & 1))) break;
      }
      return;
    }
    {
      // forward DST with the spectral divide applied to its outputs, then the
      // inverse DST by the same (single inlined) body
      if (PART && in.hi - in.lo < N) {
        // the buffer's other rows hold the tile before last's results
        const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        float4* s4 = reinterpret_cast<float4*>(s);
        for (int i4 = threadIdx.x; i4 < in.lo * (W / 4); i4 += NT) s4[i4] = zero;
        for (int i4 = in.hi * (W / 4) + threadIdx.x; i4 < N * (W / 4); i4 += NT) s4[i4] = zero;
        __syncthreads();
      }
      const int q = t / NX + planes.lo, p = (t % NX) * W + (int)(threadIdx.x & 31);
      DivPost post{mus, mus[p] + mus[q] - lambda, scale, p == 0, SOLVE};
#pragma unroll 1
      for (int rep = 0; rep < (SOLVE ? 2 : reps); ++rep) {
        regdst::dst1_tile_reg<regdst::Geo<N, W>>(s, sinv, reinterpret_cast<const regdst::cf2*>(tw), tot, post);
        post.on = false;
      }
    }
    fence_async_shared();
    __syncthreads();
    if (threadIdx.x == 0) {
      int x, y, z;
      coords(t, out.lo, x, y, z);
      tma_store3(&map_out, s + out.lo * W, x, y, z);
      tma_commit();
    }
  }
  if (threadIdx.x == 0) tma_wait_all();
}

// ------------------------------------- z solve by elimination (3-D, N >= 32)
// After the x and y transforms every (p, q) mode leaves one symmetric Toeplitz
// tridiagonal system along z,
//   (2 + eps) v_k - v_{k-1} - v_{k+1} = R_k = -h^2 (2/N)^2 r_k,
//   eps = -h^2 (mu1[p] + mu1[q] - lambda) > 0,
// which elimination solves in about 5 operations per value, against two
// transforms of 20 to 25 each and a division.  Eliminating from both ends to
// the middle halves the serial chain and shares its pivots (they depend on
// the distance from the end only); a tile of TW columns is two threads per
// column.  The pivots d_k = 1 + s_k are kept as s_k = eps + s_{k-1} /
// d_{k-1}, all terms positive, so that eps (as small as 1e-4) is never
// rounded against 2; the middle row's pivot is eps + 2 s / d.  float32 forms
// 1 / d as it goes; float64, whose divisions would be the whole cost, reads
// it from a table built per lambda (N/2 values per mode, row 0 the inverse of
// the middle pivot).
// Measured at 256^3: float32 59 -> 40 us, float64 292 -> 192 us a pass (512^3
// float32 515 -> 451 us): bound by the chain and the tile's load latency at
// 8 warps per SM (48 KB of rows and pivots per 32 columns).
template <typename T, int N>
struct ZTri {
  static constexpr int TW = sizeof(T) == 8 && N >= 384 ? 16 : 32;  // columns (64 KB of float64 at most)
  static constexpr int NTH = 2 * TW, M = N / 2;
  static constexpr bool INLINE_G = sizeof(T) == 4;
  static constexpr size_t smem = ((size_t)N * TW + (INLINE_G ? (size_t)M * TW : 0) + NTH) * sizeof(T);
};

template <typename T, int N>
__global__ void __launch_bounds__(ZTri<T, N>::NTH) k_ztri(T* __restrict__ a, const T* __restrict__ mu1, T lambda, T h2,
                                                          T rs, const T* __restrict__ tab, const int* __restrict__ skip,
                                                          Span in, Span out) {
  using Z = ZTri<T, N>;
  constexpr int TW = Z::TW, NTH = Z::NTH, M = Z::M, CH = 8;
  constexpr int CPR = TW * (int)sizeof(T) / 16, RPS = NTH / CPR, EPC = 16 / (int)sizeof(T);  // 16-byte pieces of a row
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* s = reinterpret_cast<T*>(smem_raw);
  T* gs = s + N * TW;                                  // 1 / d_j (float32)
  T* mid = gs + (Z::INLINE_G ? M * TW : 0);
  pdl_wait();
  if (skip != nullptr && *skip != 0) return;
  const int x0 = blockIdx.x * TW, q = blockIdx.y + 1;
  constexpr size_t rstride = (size_t)N * N;
  T* base = a + (size_t)q * N + x0;
  const int piece = EPC * (threadIdx.x % CPR), r0 = threadIdx.x / CPR;
#pragma unroll 4
  for (int k = in.lo + r0; k < in.hi; k += RPS) copy_async16(s + k * TW + piece, base + k * rstride + piece);
  for (int i = threadIdx.x; i < in.lo * TW; i += NTH) s[i] = (T)0;
  for (int i = in.hi * TW + threadIdx.x; i < N * TW; i += NTH) s[i] = (T)0;
  const int half = threadIdx.x / TW, c = threadIdx.x % TW, p = x0 + c;
  const T eps = -h2 * (mu1[p] + mu1[q] - lambda);
  const T* tq = tab + (Z::INLINE_G ? 0 : (size_t)q * M * N + p);
  copy_async_wait();
  __syncthreads();
  // rows j = 1 .. M - 1 from this half's end
  T* sr = s + (half ? N * TW : 0) + c;
  const int rstep = half ? -TW : TW;
  auto pivot = [&](T sv) -> T {
    const float d = 1.0f + (float)sv, r = __fdividef(1.0f, d);
    return (T)fmaf(r, fmaf(-d, r, 1.0f), r);
  };
  T y = (T)0, g = (T)0, sv = (T)0;
  // rows (and table pivots) in batches of CH; with the table the next batch
  // is loaded before this one's chain (223 -> 192 us at 256^3; float32, whose
  // batches come from shared memory, ran slower with it: 40 -> 47 us)
  constexpr bool AHEAD = !Z::INLINE_G;
  T r[CH], gg[CH];
  auto fetch = [&](int j0) {
#pragma unroll
    for (int u = 0; u < CH; ++u) {
      const bool on = j0 + u < M;
      r[u] = on ? sr[(j0 + u) * rstep] : (T)0;
      if constexpr (!Z::INLINE_G) gg[u] = on ? tq[(size_t)(j0 + u) * N] : (T)0;
    }
  };
  if (AHEAD) fetch(1);
#pragma unroll 1
  for (int j0 = 1; j0 < M; j0 += CH) {
    if (!AHEAD) fetch(j0);
    T rc[CH], gc[CH];
#pragma unroll
    for (int u = 0; u < CH; ++u) {
      rc[u] = r[u];
      gc[u] = gg[u];
    }
    if (AHEAD) fetch(j0 + CH);
#pragma unroll
    for (int u = 0; u < CH; ++u) {
      const int j = j0 + u;
      if (j < M) {
        y = fma(g, y, rs * rc[u]);
        if constexpr (Z::INLINE_G) {
          sv = j == 1 ? 1.0f + eps : sv * g + eps;
          g = pivot(sv);
          if (half == 0) gs[j * TW + c] = g;
        } else {
          g = gc[u];
        }
        sr[j * rstep] = y;
      }
    }
  }
  mid[threadIdx.x] = y * g;
  const T rm = rs * s[M * TW + c];
  __syncthreads();
  const T num = rm + mid[c] + mid[TW + c];
  T v;
  if constexpr (Z::INLINE_G)
    v = num / (eps + 2.0f * sv * g);
  else
    v = num * tq[0];
  if (half == 0) s[M * TW + c] = v;
  auto fetch_back = [&](int j0) {
#pragma unroll
    for (int u = 0; u < CH; ++u) {
      const int j = j0 - u;
      r[u] = j > 0 ? sr[j * rstep] : (T)0;
      if constexpr (Z::INLINE_G)
        gg[u] = j > 0 ? gs[j * TW + c] : (T)0;
      else
        gg[u] = j > 0 ? tq[(size_t)j * N] : (T)0;
    }
  };
  if (AHEAD) fetch_back(M - 1);
#pragma unroll 1
  for (int j0 = M - 1; j0 > 0; j0 -= CH) {
    if (!AHEAD) fetch_back(j0);
    T rc[CH], gc[CH];
#pragma unroll
    for (int u = 0; u < CH; ++u) {
      rc[u] = r[u];
      gc[u] = gg[u];
    }
    if (AHEAD) fetch_back(j0 - CH);
#pragma unroll
    for (int u = 0; u < CH; ++u)
      if (j0 - u > 0) {
        v = (rc[u] + v) * gc[u];
        sr[(j0 - u) * rstep] = v;
      }
  }
  __syncthreads();
  pdl_launch_next();
#pragma unroll 4
  for (int k = out.lo + r0; k < out.hi; k += RPS)
    *reinterpret_cast<float4*>(base + k * rstride + piece) = *reinterpret_cast<const float4*>(s + k * TW + piece);
}

// 1 / (1 + s) with the rounding of 1 + s taken back: the pivots of
// neighbouring rows are nearly equal, so a shared error of theirs adds up over
// the rows that a mode remembers (z stage error at 48 rows 5.5e-16 ->
// 4.5e-16).  Two Newton steps from the float reciprocal, the second on the
// pair d + e = 1 + s (a table of 256^3 / 2 values in 0.13 ms, 0.27 ms by a
// division and a correction after it, 0.12 ms by the division alone).
__device__ __forceinline__ double ztab_pivot(double s) {
  const double d = 1.0 + s;
  if (__double2hiint(d) >= 0x46300000) return 1.0 / d;  // from 2^100 on: the float range ends
  const double e = s - (d - 1.0);
  double g = ffl::widen(1.0f / ffl::narrow(d));
  g = fma(g, fma(-g, d, 1.0), g);
  return fma(g, fma(-g, e, fma(-g, d, 1.0)), g);
}
// 1 / d_j of every (q, p) mode at row j of its table, the inverse of the
// middle pivot at row 0
__global__ void k_ztab(const double* __restrict__ mu1, double lambda, double h2, int N, double* __restrict__ tab) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x, q = blockIdx.y, M = N / 2;
  if (p >= N) return;
  const double eps = -h2 * (mu1[p] + mu1[q] - lambda);
  double* t = tab + (size_t)q * M * N + p;
  double s = 1.0 + eps, g = ztab_pivot(s);
  t[N] = g;
  int j = 2;
  for (; j < M; ++j) {
    const double next = fma(s, g, eps);
    if (next == s) break;  // the pivots have converged: most modes, within a few rows
    s = next;
    g = ztab_pivot(s);
    t[(size_t)j * N] = g;
  }
  for (; j < M; ++j) t[(size_t)j * N] = g;
  t[0] = 1.0 / fma(2.0 * s, g, eps);
}

// ------------------------------- fused x and y passes (thread-block clusters)
// One z-plane of the padded float32 grid is transformed along x and then y
// by a cluster of N / 32 blocks (N <= 256) that exchange the plane through
// distributed shared memory, so the plane crosses global memory once per
// direction instead of twice.  Block r of the cluster owns the 32 y-lines
// y = 32 r + c (tile A: rows x, columns c) for the x transform and the 32
// x-modes kx = 32 r + c (tile B: rows y, columns c) for the y transform.
// Between the two, block r reads from every block q the 32 x 32 piece
// A_q[32 r .. 32 r + 31][0 .. 31] (rows of 32 consecutive words in the
// owner's shared memory) and writes it transposed into B rows 32 q ..
// 32 q + 31; the row stride 33 keeps both sides free of bank conflicts.  A
// cluster barrier after the first transform makes every A complete before it
// is read; a second one after the exchange keeps each block's shared memory
// alive until its peers have read it.
namespace cg = cooperative_groups;

template <int N>
constexpr size_t xy_smem_bytes() {
  using C = Cfg<float, N>;
  return (2 * (size_t)N * C::RS + C::mem_elems) * sizeof(float);
}

// dst[(32 q + lane) RS + j] = src_q[(y0 + j) RS + lane] for every block q of
// the cluster and j < 32: the transposed 32 x 32 pieces.  Warp w moves rows
// j = w + 8 i; the distributed-shared-memory loads of four blocks are issued
// together (16 in flight per thread) before their stores.
template <typename T, int N>
__device__ __forceinline__ void xy_exchange(const cg::cluster_group& cluster, T* src, T* dst, int y0) {
  using C = Cfg<T, N>;
  constexpr int W = C::W, RS = C::RS, CL = N / W, R = W / (NT / 32), QB = CL < 4 ? CL : 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll 1
  for (int q0 = 0; q0 < CL; q0 += QB) {
    T v[QB][R];
#pragma unroll
    for (int k = 0; k < QB; ++k) {
      const T* ps = cluster.map_shared_rank(src, q0 + k);
#pragma unroll
      for (int i = 0; i < R; ++i) v[k][i] = ps[(y0 + warp + (NT / 32) * i) * RS + lane];
    }
#pragma unroll
    for (int k = 0; k < QB; ++k)
#pragma unroll
      for (int i = 0; i < R; ++i) dst[((q0 + k) * W + lane) * RS + warp + (NT / 32) * i] = v[k][i];
  }
}

// forward: r = alpha src + corrections (as k_xfwd), x DST, exchange, y DST
template <int N>
__global__ void __launch_bounds__(NT) k_xy_fwd(float* __restrict__ a, const double* __restrict__ src, double alpha,
                                               const float* __restrict__ src32, const double* __restrict__ corr,
                                               const int32_t* __restrict__ irr, const int32_t* __restrict__ line_start,
                                               const float* __restrict__ tw_g, const int* __restrict__ skip) {
  using C = Cfg<float, N>;
  constexpr int W = C::W, RS = C::RS, n1 = N - 1, CL = N / W;
  static_assert(W == 32 && N % W == 0 && CL <= 8, "one cluster of at most 8 blocks per plane");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float* sA = reinterpret_cast<float*>(smem_raw);
  float* sB = sA + N * RS;
  float* mem = sB + N * RS;
  cg::cluster_group cluster = cg::this_cluster();
  // the flag is set before this launch by the stream's previous kernels, so
  // every block of a cluster sees the same value
  const bool skipped = skip != nullptr && *skip != 0;
  load_tables<C>(mem, tw_g);
  if (skipped) return;
  const int r = (int)cluster.block_rank();
  const int y0 = r * W;
  const int z = blockIdx.y + 1;
  if (src != nullptr) {
    const float a_t = (float)alpha;
    for (int idx = threadIdx.x; idx < N * W; idx += NT) {
      const int x = idx % N, c = idx / N, y = y0 + c;
      float v = 0.0f;
      if (x > 0 && y > 0) v = a_t * ffl::narrow(src[((size_t)(z - 1) * n1 + (y - 1)) * n1 + (x - 1)]);
      sA[x * RS + c] = v;
    }
  } else if (src32 != nullptr) {
    for (int idx = threadIdx.x; idx < N * W; idx += NT) {
      const int x = idx % N, c = idx / N, y = y0 + c;
      float v = 0.0f;
      if (x > 0 && y > 0) v = src32[((size_t)(z - 1) * n1 + (y - 1)) * n1 + (x - 1)];
      sA[x * RS + c] = v;
    }
  } else {
    for (int idx = threadIdx.x; idx < N * W; idx += NT) sA[(idx % N) * RS + idx / N] = 0.0f;
  }
  __syncthreads();
  add_corrections<C, 3>(sA, corr, CorrRows{}, irr, line_start, y0, z);
  __syncthreads();
  dst_tile<C>(sA, mem);
  cluster.sync();
  xy_exchange<float, N>(cluster, sA, sB, y0);
  cluster.sync();
  dst_tile<C>(sB, mem);
  const size_t plane = (size_t)z * N * N;
  for (int idx = threadIdx.x; idx < N * W; idx += NT) {
    const int c = idx % W, y = idx / W;
    a[plane + (size_t)y * N + y0 + c] = sB[y * RS + c];
  }
}

// inverse: y DST, exchange, x DST, output as k_xinv
template <int N>
__global__ void __launch_bounds__(NT) k_xy_inv(float* __restrict__ a, bool keep, double* __restrict__ out,
                                               const double* __restrict__ aux, double beta, double gamma,
                                               const float* __restrict__ tw_g, const int* __restrict__ skip,
                                               const float* __restrict__ aux32) {
  using C = Cfg<float, N>;
  constexpr int W = C::W, RS = C::RS, n1 = N - 1, CL = N / W;
  static_assert(W == 32 && N % W == 0 && CL <= 8, "one cluster of at most 8 blocks per plane");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float* sA = reinterpret_cast<float*>(smem_raw);
  float* sB = sA + N * RS;
  float* mem = sB + N * RS;
  cg::cluster_group cluster = cg::this_cluster();
  const bool skipped = skip != nullptr && *skip != 0;
  load_tables<C>(mem, tw_g);
  if (skipped) return;
  const int r = (int)cluster.block_rank();
  const int y0 = r * W;
  const int z = blockIdx.y + 1;
  const size_t plane = (size_t)z * N * N;
  for (int idx = threadIdx.x; idx < N * W; idx += NT) {
    const int c = idx % W, y = idx / W;
    copy_async(&sB[y * RS + c], &a[plane + (size_t)y * N + y0 + c]);
  }
  copy_async_wait();
  __syncthreads();
  dst_tile<C>(sB, mem);
  cluster.sync();
  xy_exchange<float, N>(cluster, sB, sA, y0);
  cluster.sync();
  dst_tile<C>(sA, mem);
  if (out == nullptr) {
    if (keep)
      for (int idx = threadIdx.x; idx < N * W; idx += NT) {
        const int x = idx % N, c = idx / N;
        a[plane + (size_t)(y0 + c) * N + x] = sA[x * RS + c];
      }
    return;
  }
  const float b_t = (float)beta;
  for (int idx = threadIdx.x; idx < N * W; idx += NT) {
    const int x = idx % N, c = idx / N, y = y0 + c;
    const float v = sA[x * RS + c];
    const size_t pidx = plane + (size_t)y * N + x;
    if (keep) a[pidx] = v;
    if (x > 0 && y > 0) {
      const size_t o = ((size_t)(z - 1) * n1 + (y - 1)) * n1 + (x - 1);
      const double bv = ffl::widen(b_t * v);
      if (aux32 != nullptr)
        out[o] = bv + ffl::widen(aux32[pidx]);
      else
        out[o] = aux != nullptr ? fma(gamma, aux[o], bv) : bv;
    }
  }
}

// The whole 2-D solve in one launch: a cluster of N / 32 blocks (N <= 256),
// block r with the x lines y = 32 r .. 32 r + 31 (tile A: rows x) and then the
// x modes 32 r .. 32 r + 31 (tile B: rows y): x DST, exchange, y DST, spectral
// multiply, y DST, exchange, x DST, output.  A plane of this size is a few
// blocks' work, so its time is latency: as three launches (x forward, y
// solve, x inverse) with the grid through memory between them a float64
// 128^2 solve took 37 us of kernel time.  The four transforms run one inlined
// body; the values are those of the three passes.
template <typename T, int N>
__global__ void __launch_bounds__(NT, 1) k_solve2d(T* __restrict__ a, const double* __restrict__ src, double alpha,
                                                   const float* __restrict__ src32, const double* __restrict__ corr,
                                                   CorrRows rows, const int32_t* __restrict__ irr,
                                                   const int32_t* __restrict__ line_start, const T* __restrict__ tw_g,
                                                   const T* __restrict__ mu1, T lambda, T scale,
                                                   const T* __restrict__ rinv, bool keep, double* __restrict__ out,
                                                   const double* __restrict__ aux, double beta, double gamma,
                                                   const float* __restrict__ aux32, const int* __restrict__ skip,
                                                   int reps) {
  using C = Cfg<T, N>;
  constexpr int W = C::W, RS = C::RS;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* sA = reinterpret_cast<T*>(smem_raw);
  T* sB = sA + N * RS;
  T* mem = sB + N * RS;
  cg::cluster_group cluster = cg::this_cluster();
  load_tables<C>(mem, tw_g);
  pdl_wait();
  // set by earlier kernels of the stream: the same for every block
  if (skip != nullptr && *skip != 0) return;
  pdl_launch_next();
  const int y0 = (int)cluster.block_rank() * W;
  if (src != nullptr) {
    const T a_t = (T)alpha;
    fill_lines<C, 2>(sA, src, y0, 0, [&](double v) { return a_t * to_T<T>(v); });
  } else if (src32 != nullptr) {
    fill_lines<C, 2>(sA, src32, y0, 0, [&](float v) { return (T)v; });
  } else {
    for (int idx = threadIdx.x; idx < N * W; idx += NT) sA[(idx % N) * RS + idx / N] = (T)0;
  }
  __syncthreads();
  add_corrections<C, 2>(sA, corr, rows, irr, line_start, y0, 0);
  __syncthreads();
#pragma unroll 1
  for (int rep = 0; rep < reps; ++rep) {
    dst_tile<C>(rep == 0 || rep == 3 ? sA : sB, mem);
    if (rep == 0 || rep == 2) {
      // every tile complete, the pieces exchanged, every piece read
      cluster.sync();
      xy_exchange<T, N>(cluster, rep == 0 ? sA : sB, rep == 0 ? sB : sA, y0);
      cluster.sync();
    } else if (rep == 1) {
      const int c = threadIdx.x % W, p = y0 + c;
      const T base = mu1[p] - lambda;
#pragma unroll 4
      for (int k = threadIdx.x / W; k < N; k += NT / W) {
        T f;
        if constexpr (sizeof(T) == 4)
          f = p == 0 ? 0.0f : __fdividef(scale, mu1[k] + base);
        else
          f = rinv != nullptr ? rinv[(size_t)k * N + p]
                              : (k > 0 && p > 0 ? scale / (mu1[k] + mu1[p] + (T)0 - lambda) : (T)0);
        sB[k * RS + c] *= f;
      }
      __syncthreads();
    }
  }
  put_lines<C, 2>(sA, a, keep, out, aux, beta, gamma, aux32, y0, 0);
}

template <typename K, typename... Args>
cudaError_t launch_cluster(K kernel, int cl, dim3 grid, size_t smem, cudaStream_t st, bool pdl, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(NT, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cl;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// opt each kernel into its dynamic shared-memory size once per process
template <typename K>
int prep(K kernel, size_t smem) {
  static const void* done[256];
  static int ndone = 0;
  const void* key = (const void*)kernel;
  for (int i = 0; i < ndone; ++i)
    if (done[i] == key) return KFBI_OK;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) {
    set_error("cudaFuncSetAttribute failed: %s", cudaGetErrorString(e));
    return KFBI_ERR_CUDA;
  }
  if (ndone < 256) done[ndone++] = key;
  return KFBI_OK;
}

// a transform pass, chained to its predecessor by programmatic dependent
// launch; not for handles whose tables the stream has just written (the
// allocation-free box solve: no mode-factor table either)
template <typename K, typename... Args>
cudaError_t launch_pass(kfbi_handle* h, K kernel, dim3 grid, size_t smem, Args... args) {
  if (h->owner) return launch_pdl(kernel, grid, dim3(NT), smem, h->stream, args...);
  kernel<<<grid, NT, smem, h->stream>>>(args...);
  return cudaGetLastError();
}

// what a strided pass covers: its planes, the rows it reads (the others are
// zero) and the rows it writes
struct PassSpan {
  Span planes, in, out;
};
template <int N>
PassSpan whole() {
  return PassSpan{Span{1, N}, Span{0, N}, Span{0, N}};
}

// one strided 3-D pass (mode 0: along y, mode 1: along z); float32 grids of
// 32 <= N <= 256 go through the TMA-fed persistent kernel
template <typename T, int N>
int launch_strided3(kfbi_handle* h, int mode, bool solve, T* work, const T* mu1, T lam, T scale, const T* tw,
                    const T* rinv, const PassSpan& ps) {
  using C = Cfg<T, N>;
  int rc;
  if constexpr (sizeof(T) == 4 && N >= TMA_W && N <= 256) {
    const bool second = (const void*)work == (const void*)h->w.grid32b;
    if (h->tma) {
      constexpr size_t smem = tma_smem_bytes<N>();
      const CUtensorMap& min = h->tmap[second][ps.in.hi - ps.in.lo < N][mode];
      const CUtensorMap& mout = h->tmap[second][ps.out.hi - ps.out.lo < N][mode];
      const int tiles = (N / TMA_W) * (ps.planes.hi - ps.planes.lo);
      const int nb = TMA_BLOCKS * h->sms;
      const int grid = tiles < nb ? tiles : nb;
      const bool part = ps.planes.hi - ps.planes.lo < N - 1 || ps.in.hi - ps.in.lo < N || ps.out.hi - ps.out.lo < N;
      auto go = [&](auto kernel, int reps) -> int {
        if (int e = prep(kernel, smem)) return e;
        return launch_pdl(kernel, dim3(grid), dim3(NT), smem, h->stream, min, mout, mode, ps.planes, ps.in, ps.out, mu1,
                          lam, scale, tw, h->w.err, reps, (const int*)h->skip) == cudaSuccess
                   ? KFBI_OK
                   : launch_failed("TMA strided pass");
      };
      if (solve) return part ? go(k_strided_tma<N, true, true>, 2) : go(k_strided_tma<N, true, false>, 2);
      return part ? go(k_strided_tma<N, false, true>, 1) : go(k_strided_tma<N, false, false>, 1);
    }
  }
  const size_t smem = C::smem_elems * sizeof(T);
  const size_t NN = (size_t)N * N;
  const dim3 grid(N / C::W, ps.planes.hi - ps.planes.lo);
  const size_t rstride = mode == 0 ? (size_t)N : NN, pstride = mode == 0 ? NN : (size_t)N;
  cudaError_t e;
  if (solve) {
    if ((rc = prep(k_strided<T, N, true, 3>, smem))) return rc;
    e = launch_pass(h, k_strided<T, N, true, 3>, grid, smem, work, rstride, pstride, ps.planes.lo, mu1, lam, scale, tw,
                    (const int*)h->skip, rinv, 2, ps.in, ps.out, h->w.err);
  } else {
    if ((rc = prep(k_strided<T, N, false, 3>, smem))) return rc;
    e = launch_pass(h, k_strided<T, N, false, 3>, grid, smem, work, rstride, pstride, ps.planes.lo, mu1, lam, scale, tw,
                    (const int*)h->skip, (const T*)nullptr, 1, ps.in, ps.out, h->w.err);
  }
  return e == cudaSuccess ? KFBI_OK : launch_failed("strided pass");
}

// The passes of a 3-D solve and what each covers.  With corrections alone as
// the right-hand side (no source field) the grid is zero outside the ranges
// near_y, near_z of the irregular nodes: x lines outside them and planes
// outside near_z are not transformed, and the y and z passes take those rows
// as zero.  With only the interface limit reading the solution (near_only)
// the z pass writes near_z alone, the y pass its planes and the rows near_y,
// the x pass those lines.  The values computed are the same bit for bit.
struct SolveSpans {
  PassSpan yf, z, yi;
  Span xf_y, xf_z, xi_y, xi_z;  // lines and planes of the x passes
};
inline bool near_source(const kfbi_handle* h, const SolveArgs& sa) {
  return sa.src == nullptr && sa.src32 == nullptr && sa.corr != nullptr && h->near_y.hi > 0;
}
inline bool near_result(const kfbi_handle* h, const SolveArgs& sa) {
  return sa.near_only && sa.out_user == nullptr && h->near_y.hi > 0;
}
template <int N>
SolveSpans solve_spans(const kfbi_handle* h, bool in, bool out) {
  const Span all{0, N}, planes{1, N};
  const Span iy = in ? h->near_y : all, iz = in ? h->near_z : all;
  const Span oy = out ? h->near_y : all, oz = out ? h->near_z : all;
  auto from1 = [](Span s) { return Span{s.lo < 1 ? 1 : s.lo, s.hi}; };
  SolveSpans s;
  s.xf_y = iy;
  s.xf_z = from1(iz);
  s.yf = PassSpan{from1(iz), iy, all};
  s.z = PassSpan{planes, iz, oz};
  s.yi = PassSpan{from1(oz), all, oy};
  s.xi_y = oy;
  s.xi_z = from1(oz);
  return s;
}

// Whether the z systems of this lambda are solved by elimination.  Its error
// grows with the number of rows 1 / sqrt(eps) over which the slowest mode (p
// = q = 1) remembers its roundings; the line is drawn at 48 rows for both
// types.  z stage alone against 80 bits (2-norm, dense, smooth, sparse and
// single-mode right-hand sides):
//  - float32: below the two transforms' (4e-7 at 256 rows and 5e-7 at 512 for
//    lambda = 60, where the transforms leave 9e-7 and 1.7e-6; 3e-6 at 110
//    rows);
//  - float64: 2.7e-16 to 3.1e-16 at 256 lines and 16 rows (lambda = 60),
//    3.7e-16 to 4.8e-16 at 48 rows; at 512 lines and 32 rows 3.6e-16 to
//    4.2e-16.  That is a quarter of what two transforms in float64
//    arithmetic leave (0.9e-15 to 1.6e-15 and 1.7e-15 to 3.3e-15), and 1.0 to
//    2.4 times what the two fixed-point transforms leave (1.9e-16 to 3.0e-16
//    and 2.6e-16 to 3.2e-16), for two thirds of their time.  Up to 128 lines,
//    where no lambda >= 0 reaches more than 29 rows, it stays below two thirds
//    of the former.
// The time-step problems (lambda = 40, 60, ...) are well inside; Poisson and
// nearly Poisson problems on fine grids keep the transforms.
template <int N>
bool z_by_elimination(const kfbi_handle* h, double lambda) {
  if (N < 32 || h->grid.dim != 3) return false;
  const double s = std::sin(3.14159265358979323846 / (2.0 * N));
  const double eps = h->grid.h * h->grid.h * lambda + 8.0 * s * s;  // -h^2 (2 mu1[1] - lambda)
  return eps * (48.0 * 48.0) >= 1.0;
}

// storage of a table, nullptr where it cannot be had
inline double* table_alloc(kfbi_handle* h, int64_t n) {
  double* p = nullptr;
  if (dalloc(h, &p, (size_t)n) == KFBI_OK) return p;
  cudaGetLastError();
  return nullptr;
}

// the float64 pivot table for this lambda (N^3 / 2 values, built once per
// lambda), nullptr where the handle has none
inline const double* z_table(kfbi_handle* h, double lambda, int N) {
  if (!h->owner) return nullptr;
  return h->ztab.get(
      lambda, [&] { return table_alloc(h, (int64_t)N * N * (N / 2)); },
      [&](double* p) {
        k_ztab<<<dim3((N + 127) / 128, N), 128, 0, h->stream>>>(h->t.mu, lambda, h->grid.h * h->grid.h, N, p);
        KFBI_COUNT(1);
      });
}

// the z pass of a 3-D solve: elimination where z_by_elimination allows it,
// else forward transform, spectral divide, inverse transform
template <typename T, int N>
const T* mode_factors(kfbi_handle* h, double lambda, double scale);
template <typename T, int N>
int launch_zsolve(kfbi_handle* h, double lambda, T* work, const T* mu1, T scale, const T* tw, const PassSpan& ps) {
  if constexpr (N >= 32) {
    using Z = ZTri<T, N>;
    bool tri = z_by_elimination<N>(h, lambda);
    const T* tab = nullptr;
    if constexpr (sizeof(T) == 8) {
      if (tri) tab = z_table(h, lambda, N);
      tri = tri && tab != nullptr;
    }
    if (tri) {
      int rc;
      if ((rc = prep(k_ztri<T, N>, Z::smem))) return rc;
      const double h2 = h->grid.h * h->grid.h;
      const T rs = (T)(-h2 * (2.0 / N) * (2.0 / N));
      if (launch_pdl(k_ztri<T, N>, dim3(N / Z::TW, N - 1), dim3(Z::NTH), Z::smem, h->stream, work, mu1, (T)lambda,
                     (T)h2, rs, tab, (const int*)h->skip, ps.in, ps.out) != cudaSuccess)
        return launch_failed("z elimination pass");
      return KFBI_OK;
    }
  }
  return launch_strided3<T, N>(h, 1, true, work, mu1, (T)lambda, scale, tw,
                               mode_factors<T, N>(h, lambda, (double)scale), ps);
}

// scale / mu_p over the mode grid (q, k, p) of the float64 middle pass,
// mu_p = (mu1[k] + mu1[p]) + mu1[q] (3-D) - lambda, in the pass's own order;
// n modes per axis, mode 0 absent (sine modes) or present (cosine modes)
__global__ void k_rinv(const double* __restrict__ mu1, double lambda, double scale, int n, int dim, bool mode0,
                       double* __restrict__ out, int64_t total) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int p = (int)(i % n), k = (int)((i / n) % n), q = (int)(i / ((int64_t)n * n));
    const double muq = dim == 3 ? mu1[q] : 0.0;
    const bool on = mode0 || (k > 0 && p > 0 && (dim == 2 || q > 0));
    out[i] = on ? scale / (mu1[k] + mu1[p] + muq - lambda) : 0.0;
  }
}

// the float64 solve's mode factors for this lambda: built once per lambda
// in a table of N^dim values that the handle owns (none for float32, nor for
// handles that must not allocate)
template <typename T, int N>
const T* mode_factors(kfbi_handle* h, double lambda, double scale) {
  if constexpr (sizeof(T) != 8) {
    return nullptr;
  } else {
    if (!h->owner) return nullptr;
    const bool cosine = h->grid.bc == KFBI_BOX_NEUMANN;
    const int n = cosine ? N + 1 : N;
    const int64_t total = h->grid.dim == 3 ? (int64_t)n * n * n : (int64_t)n * n;
    return h->rinv.get(
        lambda, [&] { return table_alloc(h, total); },
        [&](double* p) {
          const int nb = (int)std::min<int64_t>((total + 255) / 256, 152 * 16);
          k_rinv<<<nb, 256, 0, h->stream>>>(h->t.mu, lambda, scale, n, h->grid.dim, cosine, p, total);
          KFBI_COUNT(1);
        });
  }
}

template <typename T, int N>
int run_solve(kfbi_handle* h, const SolveArgs& sa, T* work, const T* mu1, const T* tw) {
  using C = Cfg<T, N>;
  constexpr int W = C::W;
  const size_t smem = C::smem_elems * sizeof(T);
  const int dim = h->grid.dim;
  cudaStream_t st = h->stream;
  const Tables& t = h->t;
  const T lam = (T)sa.lambda;
  const T scale = (T)(dim == 3 ? (2.0 / N) * (2.0 / N) * (2.0 / N) : (2.0 / N) * (2.0 / N));
  int rc;
  if (dim == 3) {
    dim3 grid(N / W, N - 1);
    if constexpr (sizeof(T) == 4 && N >= 32 && N <= 256) {
      // fused x-y passes: three passes per solve (xy forward, z solve, xy inverse)
      if (h->xy_fused) {
        constexpr size_t sxy = xy_smem_bytes<N>();
        if ((rc = prep(k_xy_fwd<N>, sxy))) return rc;
        if ((rc = prep(k_xy_inv<N>, sxy))) return rc;
        cudaError_t e = launch_cluster(k_xy_fwd<N>, N / 32, grid, sxy, st, false, work, sa.src, sa.alpha, sa.src32, sa.corr,
                                       (const int32_t*)t.irr, (const int32_t*)t.line_start, tw, h->skip);
        if (e == cudaSuccess) {
          if ((rc = launch_zsolve<T, N>(h, sa.lambda, work, mu1, scale, tw, whole<N>()))) return rc;
          e = launch_cluster(k_xy_inv<N>, N / 32, grid, sxy, st, false, work, sa.keep || sa.out_user == nullptr,
                             sa.out_user, sa.aux, sa.beta, sa.gamma, tw, h->skip, sa.aux32);
          if (e != cudaSuccess) {
            set_error("cluster launch of the fused x-y inverse pass failed: %s", cudaGetErrorString(e));
            return KFBI_ERR_CUDA;
          }
          KFBI_CHECK_LAUNCH_N(3);
          return KFBI_OK;
        }
        // no cluster of this size fits: the five-pass path from now on
        cudaGetLastError();
        h->xy_fused = false;
      }
    }
    if ((rc = prep(k_xfwd<T, N, 3>, smem))) return rc;
    if ((rc = prep(k_xinv<T, N, 3>, smem))) return rc;
    // the five passes chained by programmatic dependent launch
    const SolveSpans sp = solve_spans<N>(h, near_source(h, sa), near_result(h, sa));
    const dim3 gf((sp.xf_y.hi - sp.xf_y.lo) / W, sp.xf_z.hi - sp.xf_z.lo);
    const dim3 gi((sp.xi_y.hi - sp.xi_y.lo) / W, sp.xi_z.hi - sp.xi_z.lo);
    if (launch_pass(h, k_xfwd<T, N, 3>, gf, smem, work, sa.src, sa.alpha, sa.src32, sa.corr, sa.rows, (const int32_t*)t.irr,
                    (const int32_t*)t.line_start, tw, (const int*)h->skip, sp.xf_y.lo, sp.xf_z.lo) != cudaSuccess)
      return launch_failed("x forward pass");
    if ((rc = launch_strided3<T, N>(h, 0, false, work, mu1, lam, scale, tw, nullptr, sp.yf))) return rc;
    if ((rc = launch_zsolve<T, N>(h, sa.lambda, work, mu1, scale, tw, sp.z))) return rc;
    if ((rc = launch_strided3<T, N>(h, 0, false, work, mu1, lam, scale, tw, nullptr, sp.yi))) return rc;
    if (launch_pass(h, k_xinv<T, N, 3>, gi, smem, work, sa.keep || sa.out_user == nullptr, sa.out_user,
                    (const double*)sa.aux, sa.beta, sa.gamma, tw, (const int*)h->skip, sa.aux32, sp.xi_y.lo,
                    sp.xi_z.lo) != cudaSuccess)
      return launch_failed("x inverse pass");
  } else {
    dim3 grid(N / W, 1);
    const T* rinv = mode_factors<T, N>(h, sa.lambda, (double)scale);
    if constexpr (N >= 32 && N <= 256) {
      constexpr size_t s2 = (2 * (size_t)N * C::RS + C::mem_elems) * sizeof(T);
      if ((rc = prep(k_solve2d<T, N>, s2))) return rc;
      if (launch_cluster(k_solve2d<T, N>, N / 32, dim3(N / 32), s2, st, h->owner, work, sa.src, sa.alpha, sa.src32,
                         sa.corr, sa.rows, (const int32_t*)t.irr, (const int32_t*)t.line_start, tw, mu1, lam, scale,
                         rinv, sa.keep || sa.out_user == nullptr, sa.out_user, sa.aux, sa.beta, sa.gamma, sa.aux32,
                         (const int*)h->skip, 4) == cudaSuccess) {
        KFBI_CHECK_LAUNCH();
        return KFBI_OK;
      }
      cudaGetLastError();  // no cluster of this size fits: three passes
    }
    if ((rc = prep(k_xfwd<T, N, 2>, smem))) return rc;
    if ((rc = prep(k_strided<T, N, true, 2>, smem))) return rc;
    if ((rc = prep(k_xinv<T, N, 2>, smem))) return rc;
    if (launch_pass(h, k_xfwd<T, N, 2>, grid, smem, work, sa.src, sa.alpha, sa.src32, sa.corr, sa.rows, (const int32_t*)t.irr,
                    (const int32_t*)t.line_start, tw, (const int*)h->skip, 0, 0) != cudaSuccess)
      return launch_failed("x forward pass");
    if (launch_pass(h, k_strided<T, N, true, 2>, grid, smem, work, (size_t)N, (size_t)0, 0, mu1, lam, scale, tw,
                    (const int*)h->skip, rinv, 2, Span{0, N}, Span{0, N}, h->w.err) != cudaSuccess)
      return launch_failed("y solve pass");
    if (launch_pass(h, k_xinv<T, N, 2>, grid, smem, work, sa.keep || sa.out_user == nullptr, sa.out_user,
                    (const double*)sa.aux, sa.beta, sa.gamma, tw, (const int*)h->skip, sa.aux32, 0, 0) != cudaSuccess)
      return launch_failed("x inverse pass");
  }
  KFBI_CHECK_LAUNCH_N(dim == 3 ? 5 : 3);
  return KFBI_OK;
}

// one pass of the solver on the padded work grid (timing of single kernels)
template <typename T, int N>
int run_pass(kfbi_handle* h, int pass, double lambda, T* work, const T* mu1, const T* tw) {
  using C = Cfg<T, N>;
  constexpr int W = C::W;
  const size_t smem = C::smem_elems * sizeof(T);
  const int dim = h->grid.dim;
  cudaStream_t st = h->stream;
  const Tables& t = h->t;
  const T lam = (T)lambda;
  const T scale = (T)(dim == 3 ? (2.0 / N) * (2.0 / N) * (2.0 / N) : (2.0 / N) * (2.0 / N));
  const size_t NN = (size_t)N * N;
  dim3 grid(N / W, dim == 3 ? N - 1 : 1);
  int rc;
  if (dim == 3) {
    if (pass == 0) {
      if ((rc = prep(k_xfwd<T, N, 3>, smem))) return rc;
      k_xfwd<T, N, 3><<<grid, NT, smem, st>>>(work, nullptr, 1.0, nullptr, nullptr, CorrRows{}, t.irr, t.line_start, tw, nullptr, 0,
                                               1);
    } else if (pass == 1) {
      if ((rc = launch_strided3<T, N>(h, 0, false, work, mu1, lam, scale, tw, nullptr, whole<N>()))) return rc;
    } else if (pass == 2) {
      if ((rc = launch_zsolve<T, N>(h, lambda, work, mu1, scale, tw, whole<N>()))) return rc;
    } else if (pass == 3) {
      if ((rc = prep(k_xinv<T, N, 3>, smem))) return rc;
      k_xinv<T, N, 3><<<grid, NT, smem, st>>>(work, true, nullptr, nullptr, 1.0, 0.0, tw, nullptr, nullptr, 0, 1);
    } else {
      // 4 / 5: the fused x-y forward / inverse pass
      if constexpr (sizeof(T) == 4 && N >= 32 && N <= 256) {
        if (h->xy_fused) {
          constexpr size_t sxy = xy_smem_bytes<N>();
          cudaError_t e;
          if (pass == 4) {
            if ((rc = prep(k_xy_fwd<N>, sxy))) return rc;
            e = launch_cluster(k_xy_fwd<N>, N / 32, grid, sxy, st, false, work, (const double*)nullptr, 1.0,
                               (const float*)nullptr, (const double*)nullptr, (const int32_t*)t.irr,
                               (const int32_t*)t.line_start, tw, (const int*)nullptr);
          } else {
            if ((rc = prep(k_xy_inv<N>, sxy))) return rc;
            e = launch_cluster(k_xy_inv<N>, N / 32, grid, sxy, st, false, work, true, (double*)nullptr,
                               (const double*)nullptr, 1.0, 0.0, tw, (const int*)nullptr, (const float*)nullptr);
          }
          if (e != cudaSuccess) {
            set_error("cluster launch failed: %s", cudaGetErrorString(e));
            return KFBI_ERR_CUDA;
          }
          KFBI_CHECK_LAUNCH();
          return KFBI_OK;
        }
      }
      set_error("no fused x-y pass for this grid and precision");
      return KFBI_ERR_ARG;
    }
    (void)NN;
  } else {
    if (pass == 0) {
      if ((rc = prep(k_xfwd<T, N, 2>, smem))) return rc;
      k_xfwd<T, N, 2><<<grid, NT, smem, st>>>(work, nullptr, 1.0, nullptr, nullptr, CorrRows{}, t.irr, t.line_start, tw, nullptr, 0,
                                               0);
    } else if (pass == 1 || pass == 2) {
      const T* rinv = mode_factors<T, N>(h, lambda, (double)scale);
      if ((rc = prep(k_strided<T, N, true, 2>, smem))) return rc;
      k_strided<T, N, true, 2><<<grid, NT, smem, st>>>(work, N, 0, 0, mu1, lam, scale, tw, nullptr, rinv, 2, Span{0, N},
                                                       Span{0, N}, h->w.err);
    } else {
      if ((rc = prep(k_xinv<T, N, 2>, smem))) return rc;
      k_xinv<T, N, 2><<<grid, NT, smem, st>>>(work, true, nullptr, nullptr, 1.0, 0.0, tw, nullptr, nullptr, 0, 0);
    }
  }
  KFBI_CHECK_LAUNCH();
  return KFBI_OK;
}

// ------------------------------------------ coupled anisotropic solve pass
// Middle pass of the coupled box solve (3-D: along z, 2-D: along y) on the
// two padded work grids a (intracellular) and b (extracellular): forward
// DST of both tiles, the per-mode 2 x 2 solve of Eq. pde1 with diagonal
// conductivities (Section 5.2, Eq. FDE),
//   [A_i - kappa, kappa; kappa, A_e - kappa] (v_i, v_e) = (r_i, r_e),
//   A_c = sum_a d_c,a mu1(p_a),
// scaled by (2/N)^d, then the inverse DST of both tiles.  The solve takes
// its three factors per mode (v_i = f0 r_i + f1 r_e, v_e = f1 r_i + f2 r_e)
// from a table built once per kappa in float64 (k_cpl_factors).
//
// Two tiles per block where they fit in shared memory.  They do not for
// float64 lines of 512 (284 672 bytes): there one tile takes the fields in
// turn, and field a's modes wait in its work grid (every element read back by
// the thread that wrote it, from L2); the values are the same.
constexpr size_t SMEM_MAX = 232448;  // shared memory a block can have
template <typename T, int N>
struct CoupledTiles {
  using C = Cfg<T, N>;
  static constexpr size_t one = (size_t)N * C::RS, max_elems = SMEM_MAX / sizeof(T);
  static constexpr bool TWO = 2 * one + C::mem_elems <= max_elems;
  static constexpr size_t smem = ((TWO ? 2 : 1) * one + C::mem_elems) * sizeof(T);
  static_assert(smem <= SMEM_MAX, "tiles of the coupled pass");
};

template <typename T, int N, int DIM>
__global__ void __launch_bounds__(NT, N <= 128 ? 2 : 1) k_strided_coupled(T* __restrict__ a, T* __restrict__ b, size_t row_stride,
                                                        size_t plane_stride, int qoff, const T* __restrict__ cf,
                                                        size_t cf_stride, const T* __restrict__ tw_g,
                                                        const int* __restrict__ skip, Span in, Span out) {
  using C = Cfg<T, N>;
  constexpr int W = C::W, RS = C::RS;
  constexpr bool TWO = CoupledTiles<T, N>::TWO;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* sa = reinterpret_cast<T*>(smem_raw);
  T* sb = TWO ? sa + N * RS : sa;
  T* mem = sb + N * RS;
  load_tables<C>(mem, tw_g);
  pdl_wait();
  if (skip != nullptr && *skip != 0) return;
  const int x0 = blockIdx.x * W;
  const int q = blockIdx.y + qoff;
  T* ba = a + (size_t)q * plane_stride + x0;
  T* bb = b + (size_t)q * plane_stride + x0;
  // table row of this plane: modes (q, k, p), p fastest
  const T* f0 = cf + (size_t)q * N * N + x0;
  if constexpr (TWO) {
    for (int idx = threadIdx.x; idx < N * W; idx += NT) {
      const int c = idx % W, k = idx / W;
      if (k >= in.lo && k < in.hi) {
        copy_async(&sa[k * RS + c], &ba[(size_t)k * row_stride + c]);
        copy_async(&sb[k * RS + c], &bb[(size_t)k * row_stride + c]);
      } else {
        sa[k * RS + c] = (T)0;
        sb[k * RS + c] = (T)0;
      }
    }
    copy_async_wait();
    __syncthreads();
#pragma unroll 1
    for (int f = 0; f < 2; ++f) dst_tile<C>(f == 0 ? sa : sb, mem);
    for (int idx = threadIdx.x; idx < N * W; idx += NT) {
      const int c = idx % W, k = idx / W;
      const size_t o = (size_t)k * N + c;
      const T g0 = f0[o], g1 = f0[o + cf_stride], g2 = f0[o + 2 * cf_stride];
      const T ri = sa[k * RS + c], re = sb[k * RS + c];
      sa[k * RS + c] = g0 * ri + g1 * re;
      sb[k * RS + c] = g1 * ri + g2 * re;
    }
    __syncthreads();
#pragma unroll 1
    for (int f = 0; f < 2; ++f) dst_tile<C>(f == 0 ? sa : sb, mem);
    for (int idx = threadIdx.x + out.lo * W; idx < out.hi * W; idx += NT) {
      const int c = idx % W, k = idx / W;
      ba[(size_t)k * row_stride + c] = sa[k * RS + c];
      bb[(size_t)k * row_stride + c] = sb[k * RS + c];
    }
  } else {
    // steps: a forward, b forward and the 2 x 2 solve, b inverse, a inverse
    // (one inlined transform); between two steps each thread passes on the
    // elements idx = threadIdx.x + i NT of the grids and the tile alone
#pragma unroll 1
    for (int step = 0; step < 4; ++step) {
      if (step != 2) {
        const T* src = step == 1 ? bb : ba;
        for (int idx = threadIdx.x; idx < N * W; idx += NT) {
          const int c = idx % W, k = idx / W;
          sa[k * RS + c] = step == 3 || (k >= in.lo && k < in.hi) ? src[(size_t)k * row_stride + c] : (T)0;
        }
      }
      __syncthreads();
      dst_tile<C>(sa, mem);
      for (int idx = threadIdx.x; idx < N * W; idx += NT) {
        const int c = idx % W, k = idx / W;
        T* ga = &ba[(size_t)k * row_stride + c];
        T* s = &sa[k * RS + c];
        if (step == 0) {
          *ga = *s;
        } else if (step == 1) {
          const size_t o = (size_t)k * N + c;
          const T g0 = f0[o], g1 = f0[o + cf_stride], g2 = f0[o + 2 * cf_stride];
          const T ri = *ga, re = *s;
          *ga = g0 * ri + g1 * re;
          *s = g1 * ri + g2 * re;
        } else if (k >= out.lo && k < out.hi) {
          (step == 2 ? bb : ba)[(size_t)k * row_stride + c] = *s;
        }
      }
      __syncthreads();
    }
  }
}

// factors of the per-mode 2 x 2 solve over the mode grid (q, k, p) of the
// middle pass (3-D: y = q, z = k; 2-D: y = k, q = 0), x = p:
//   [A_i - kappa, kappa; kappa, A_e - kappa]^{-1} scale
//     = (scale / det) [A_e - kappa, -kappa; -kappa, A_i - kappa],
//   A_c = sum_a d_c,a mu1(p_a), det = (A_i - kappa)(A_e - kappa) - kappa^2,
// computed in float64 and stored as T (0 for the absent sine modes)
template <typename T>
__global__ void k_cpl_factors(const double* __restrict__ mu1, Coupling cp, int N, int dim, T* __restrict__ cf,
                              int64_t total) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int p = (int)(i % N), k = (int)((i / N) % N), q = (int)(i / ((int64_t)N * N));
    double g0 = 0.0, g1 = 0.0, g2 = 0.0;
    if (k > 0 && p > 0 && (dim == 2 || q > 0)) {
      const double mx = mu1[p], my = dim == 3 ? mu1[q] : mu1[k], mz = dim == 3 ? mu1[k] : 0.0;
      const double ai = cp.di[0] * mx + cp.di[1] * my + cp.di[2] * mz - cp.kappa;
      const double ae = cp.de[0] * mx + cp.de[1] * my + cp.de[2] * mz - cp.kappa;
      const double sc = cp.scale / (ai * ae - cp.kappa * cp.kappa);
      g0 = ae * sc;
      g1 = -cp.kappa * sc;
      g2 = ai * sc;
    }
    cf[i] = (T)g0;
    cf[i + total] = (T)g1;
    cf[i + 2 * total] = (T)g2;
  }
}

// the handle's factor table of element type T for this kappa (built when
// kappa changes)
template <typename T>
const T* coupled_factors(kfbi_handle* h, const Coupling& cp, int N, int64_t total) {
  T** tab;
  double* kap;
  if constexpr (sizeof(T) == 8) {
    tab = &h->cpl64;
    kap = &h->cpl64_kappa;
  } else {
    tab = &h->cpl32;
    kap = &h->cpl32_kappa;
  }
  if (*tab == nullptr) {
    if (dalloc(h, tab, (size_t)(3 * total)) != KFBI_OK) return nullptr;
    *kap = std::nan("");
  }
  if (!(*kap == cp.kappa)) {
    const int nb = (int)std::min<int64_t>((total + 255) / 256, 152 * 16);
    k_cpl_factors<T><<<nb, 256, 0, h->stream>>>(h->t.mu, cp, N, h->grid.dim, *tab, total);
    KFBI_COUNT(1);
    *kap = cp.kappa;
  }
  return *tab;
}

// the coupled box solve on two padded grids of element type T: x forward
// (sources and corrections), y, the coupled z solve, y, x inverse (outputs).
// The y passes of both fields use the plain strided kernel (the tensor maps
// describe only the handle's first float grid).
template <typename T, int N>
int run_solve_coupled(kfbi_handle* h, const SolveArgs& si, const SolveArgs& se, const Coupling& cp0, T* wa, T* wb,
                      const T* mu1T, const T* tw) {
  using C = Cfg<T, N>;
  constexpr int W = C::W;
  const size_t smem = C::smem_elems * sizeof(T);
  constexpr size_t smem2 = CoupledTiles<T, N>::smem;
  const int dim = h->grid.dim;
  cudaStream_t st = h->stream;
  const Tables& t = h->t;
  Coupling cp = cp0;
  cp.scale = dim == 3 ? (2.0 / N) * (2.0 / N) * (2.0 / N) : (2.0 / N) * (2.0 / N);
  int rc;
  const dim3 grid(N / W, dim == 3 ? N - 1 : 1);
  const int64_t total = dim == 3 ? (int64_t)N * N * N : (int64_t)N * N;
  const T* cf = coupled_factors<T>(h, cp, N, total);
  if (cf == nullptr) {
    set_error("allocation of the coupled solve's factor table failed");
    return KFBI_ERR_OOM;
  }
  if (dim == 3) {
    if ((rc = prep(k_xfwd<T, N, 3>, smem))) return rc;
    if ((rc = prep(k_strided_coupled<T, N, 3>, smem2))) return rc;
    if ((rc = prep(k_xinv<T, N, 3>, smem))) return rc;
    const SolveSpans sp = solve_spans<N>(h, near_source(h, si) && near_source(h, se),
                                         near_result(h, si) && near_result(h, se));
    const SolveArgs* sas[2] = {&si, &se};
    T* grids[2] = {wa, wb};
    const size_t NN = (size_t)N * N;
    for (int f = 0; f < 2; ++f) {
      const SolveArgs& sa = *sas[f];
      const dim3 gf((sp.xf_y.hi - sp.xf_y.lo) / W, sp.xf_z.hi - sp.xf_z.lo);
      if (launch_pass(h, k_xfwd<T, N, 3>, gf, smem, grids[f], sa.src, sa.alpha, sa.src32, sa.corr, sa.rows,
                      (const int32_t*)t.irr, (const int32_t*)t.line_start, tw, (const int*)h->skip, sp.xf_y.lo,
                      sp.xf_z.lo) != cudaSuccess)
        return launch_failed("x forward pass");
      if ((rc = launch_strided3<T, N>(h, 0, false, grids[f], mu1T, (T)0, (T)1, tw, nullptr, sp.yf))) return rc;
    }
    if (launch_pass(h, k_strided_coupled<T, N, 3>, grid, smem2, wa, wb, NN, (size_t)N, 1, cf, (size_t)total, tw,
                    (const int*)h->skip, sp.z.in, sp.z.out) != cudaSuccess)
      return launch_failed("coupled z pass");
    for (int f = 0; f < 2; ++f) {
      const SolveArgs& sa = *sas[f];
      const dim3 gi((sp.xi_y.hi - sp.xi_y.lo) / W, sp.xi_z.hi - sp.xi_z.lo);
      if ((rc = launch_strided3<T, N>(h, 0, false, grids[f], mu1T, (T)0, (T)1, tw, nullptr, sp.yi))) return rc;
      if (launch_pass(h, k_xinv<T, N, 3>, gi, smem, grids[f], sa.keep || sa.out_user == nullptr, sa.out_user,
                      (const double*)sa.aux, sa.beta, sa.gamma, tw, (const int*)h->skip, (const float*)nullptr,
                      sp.xi_y.lo, sp.xi_z.lo) != cudaSuccess)
        return launch_failed("x inverse pass");
    }
  } else {
    if ((rc = prep(k_xfwd<T, N, 2>, smem))) return rc;
    if ((rc = prep(k_strided_coupled<T, N, 2>, smem2))) return rc;
    if ((rc = prep(k_xinv<T, N, 2>, smem))) return rc;
    k_xfwd<T, N, 2><<<grid, NT, smem, st>>>(wa, si.src, si.alpha, si.src32, si.corr, si.rows, t.irr, t.line_start, tw, h->skip,
                                             0, 0);
    k_xfwd<T, N, 2><<<grid, NT, smem, st>>>(wb, se.src, se.alpha, se.src32, se.corr, se.rows, t.irr, t.line_start, tw, h->skip,
                                             0, 0);
    k_strided_coupled<T, N, 2><<<grid, NT, smem2, st>>>(wa, wb, N, 0, 0, cf, (size_t)total, tw, h->skip, Span{0, N},
                                                        Span{0, N});
    k_xinv<T, N, 2><<<grid, NT, smem, st>>>(wa, si.keep || si.out_user == nullptr, si.out_user, si.aux, si.beta,
                                             si.gamma, tw, h->skip, nullptr, 0, 0);
    k_xinv<T, N, 2><<<grid, NT, smem, st>>>(wb, se.keep || se.out_user == nullptr, se.out_user, se.aux, se.beta,
                                             se.gamma, tw, h->skip, nullptr, 0, 0);
  }
  KFBI_CHECK_LAUNCH_N(dim == 3 ? 9 : 5);
  return KFBI_OK;
}

template <typename T>
int dispatch(kfbi_handle* h, const SolveArgs& sa, T* work, const T* mu1, const T* tw) {
  switch (h->grid.N) {
    case 8: return run_solve<T, 8>(h, sa, work, mu1, tw);
    case 16: return run_solve<T, 16>(h, sa, work, mu1, tw);
    case 32: return run_solve<T, 32>(h, sa, work, mu1, tw);
    case 64: return run_solve<T, 64>(h, sa, work, mu1, tw);
    case 128: return run_solve<T, 128>(h, sa, work, mu1, tw);
    case 256: return run_solve<T, 256>(h, sa, work, mu1, tw);
    case 384: return run_solve<T, 384>(h, sa, work, mu1, tw);
    case 512: return run_solve<T, 512>(h, sa, work, mu1, tw);
    default:
      set_error("unsupported grid size N=%d", h->grid.N);
      return KFBI_ERR_ARG;
  }
}

template <typename T>
int dispatch_pass(kfbi_handle* h, int pass, double lambda, T* work, const T* mu1, const T* tw) {
  switch (h->grid.N) {
    case 8: return run_pass<T, 8>(h, pass, lambda, work, mu1, tw);
    case 16: return run_pass<T, 16>(h, pass, lambda, work, mu1, tw);
    case 32: return run_pass<T, 32>(h, pass, lambda, work, mu1, tw);
    case 64: return run_pass<T, 64>(h, pass, lambda, work, mu1, tw);
    case 128: return run_pass<T, 128>(h, pass, lambda, work, mu1, tw);
    case 256: return run_pass<T, 256>(h, pass, lambda, work, mu1, tw);
    case 384: return run_pass<T, 384>(h, pass, lambda, work, mu1, tw);
    case 512: return run_pass<T, 512>(h, pass, lambda, work, mu1, tw);
    default:
      set_error("unsupported grid size N=%d", h->grid.N);
      return KFBI_ERR_ARG;
  }
}

// ------------------------------------------------------ Neumann box (DCT-I)
// The box Green's function of Section 4 with zero normal derivative on the
// box boundary: all (N+1)^d nodes are unknowns, the boundary rows use the
// mirrored ghost value, and the cosine modes diagonalise the operator,
//   v = (2/N)^d C( mu^{-1} o C r ),  C_{kp} = c_k cos(pi k p / N),
//   c_0 = c_N = 1/2, c_k = 1 otherwise, k, p = 0..N,
// with the same mu_p as the sine solve (p = 0..N).  Work and user grids share
// the layout (N+1)^d, x fastest.  A tile holds N+1 transform rows by W lines.

// (float64 lines take the shared-memory FFT, whose long tiles stay at 16 lines)
template <typename T, int N>
struct NCfg : Tile<T, N, (sizeof(T) == 8 && N >= 384 ? 16 : WSel<T, N>::W),
                   (sizeof(T) == 8 && N >= 384 ? 16 : WSel<T, N>::W) + 1> {};

template <typename C>
constexpr size_t dct_smem_elems() {
  // tile, scan totals, twiddles, X_1 per column, sines (register path)
  return (size_t)(C::N + 1) * C::RS + (size_t)C::G * C::W + 4 * (size_t)C::N + C::W + C::N;
}

// DCT-I X_p = sum_k c_k x_k cos(pi k p / N) of every column of the tile
// s[N+1][RS] in place.  The same length-N/2 complex FFT as the sine
// transform, after the cosine pre-fold
//   y_0 = (x_0 + x_N)/2,  y_j = (x_j + x_{N-j})/2 - sin(pi j/N)(x_j - x_{N-j}),
// gives Y_k = sum_j y_j e^{2 pi i j k / N} with X_{2k} = Re Y_k and
// X_{2k+1} = X_{2k-1} + Im Y_k (from 2 sin a sin b = cos(a-b) - cos(a+b)),
// started by X_1 = sum_k c_k x_k cos(pi k / N), summed directly.
// x1 = scratch [W].
template <typename C>
__device__ void dct1_tile(typename C::T* s, const typename C::T* tw, typename C::T* tot, typename C::T* x1) {
  using T = typename C::T;
  constexpr int N = C::N, L = C::L, W = C::W, RS = C::RS, G = C::G;
  {
    constexpr int SEG = (N + 1 + G - 1) / G;
    const int c = threadIdx.x % W, g = threadIdx.x / W;
    const int j0 = g * SEG;
    const int j1 = (j0 + SEG < N + 1) ? j0 + SEG : N + 1;
    T acc = (T)0;
    for (int j = j0; j < j1; ++j) {
      T cw = tw[2 * j];
      if (j == 0 || j == N) cw *= (T)0.5;
      acc += cw * s[j * RS + c];
    }
    tot[g * W + c] = acc;
    __syncthreads();
    if (g == 0) {
      T sum = (T)0;
      for (int g2 = 0; g2 < G; ++g2) sum += tot[g2 * W + c];
      x1[c] = sum;
    }
    __syncthreads();
  }
  for (int idx = threadIdx.x; idx < (N / 2 + 1) * W; idx += NT) {
    const int c = idx % W, j = idx / W;
    if (j == 0) {
      s[c] = (T)0.5 * (s[c] + s[N * RS + c]);
    } else if (j < N / 2) {
      const T a = s[j * RS + c], b = s[(N - j) * RS + c];
      const T m = (T)0.5 * (a + b), d = tw[2 * j + 1] * (a - b);
      s[j * RS + c] = m - d;
      s[(N - j) * RS + c] = m + d;
    }
  }
  __syncthreads();
  Stages<C, 1, L>::run(s, tw);
  // split into the real DFT: X_0, X_N from Z_0; X_{2k} in row 2k and the
  // increments Im Y_k in row 2k+1
  for (int idx = threadIdx.x; idx < (L / 2 + 1) * W; idx += NT) {
    const int c = idx % W, k = idx / W;
    if (k == 0) {
      const T a = s[c], b = s[RS + c];
      s[c] = a + b;
      s[N * RS + c] = a - b;
      s[RS + c] = (T)0;
    } else {
      const int kk = L - k;
      const T Ar = s[(2 * k) * RS + c], Ai = s[(2 * k + 1) * RS + c];
      const T Br = s[(2 * kk) * RS + c], Bi = s[(2 * kk + 1) * RS + c];
      {
        const T wr = tw[2 * (2 * k)], wi = tw[2 * (2 * k) + 1];
        const T Sr = Ar + Br, Si = Ai - Bi, Dr = Ar - Br, Di = Ai + Bi;
        s[(2 * k) * RS + c] = (T)0.5 * (Sr + wr * Di + wi * Dr);
        s[(2 * k + 1) * RS + c] = (T)0.5 * (Si - wr * Dr + wi * Di);
      }
      if (kk != k) {
        const T wr = tw[2 * (2 * kk)], wi = tw[2 * (2 * kk) + 1];
        const T Sr = Br + Ar, Si = Bi - Ai, Dr = Br - Ar, Di = Bi + Ai;
        s[(2 * kk) * RS + c] = (T)0.5 * (Sr + wr * Di + wi * Dr);
        s[(2 * kk + 1) * RS + c] = (T)0.5 * (Si - wr * Dr + wi * Di);
      }
    }
  }
  __syncthreads();
  // odd outputs: column-wise inclusive scan of the increments, plus X_1
  {
    constexpr int SEG = (L + G - 1) / G;
    const int c = threadIdx.x % W, g = threadIdx.x / W;
    const int k0 = g * SEG;
    const int k1 = (k0 + SEG < L) ? k0 + SEG : L;
    T acc = (T)0;
    for (int k = k0; k < k1; ++k) {
      acc += s[(2 * k + 1) * RS + c];
      s[(2 * k + 1) * RS + c] = acc;
    }
    tot[g * W + c] = acc;
    __syncthreads();
    T off = x1[c];
    for (int g2 = 0; g2 < g; ++g2) off += tot[g2 * W + c];
    for (int k = k0; k < k1; ++k) s[(2 * k + 1) * RS + c] += off;
    __syncthreads();
  }
}

// the cosine transform of every column of the tile, rows 0..N: the
// register-resident path for float32 tiles of 32 <= N <= 512 lines, the
// shared-memory FFT otherwise
template <typename C>
__device__ __forceinline__ void dct_tile(typename C::T* s, const typename C::T* tw, const typename C::T* sinv,
                                         typename C::T* tot, typename C::T* x1) {
  if constexpr (C::REG) {
    regdst::dct1_tile_reg<regdst::Geo<C::N, C::RS>>(s, sinv, reinterpret_cast<const regdst::cf2*>(tw), tot, x1);
  } else {
    dct1_tile<C>(s, tw, tot, x1);
  }
}

// Whether the Neumann box's x passes take a line's values together (on; plain:
// but not on the way out where nothing is loaded there).  Not in float64,
// whose passes are bound by the transform (box solve 5.48 instead of 5.43 ms
// at 256^3, 821 instead of 804 us at 128^3), nor for lines so short that a
// warp has too few values to batch (float32 solve at 64^3 38.9 instead of 36.9
// us with the results batched too).
template <typename T, int N>
struct NBatch {
  static constexpr bool on = sizeof(T) == 4 && N >= 64, plain = N < 128;
};

// The W x-lines y0 .. y0 + W - 1 (zero beyond y = N) of a plane of the
// Neumann layout to the tile s[x][line], mapped by f; a line's loads are
// issued together (as in fill_lines; N >= 32).
template <typename C, typename S, typename F>
__device__ __forceinline__ void fill_lines_n(typename C::T* s, const S* __restrict__ src, int y0, const F& f) {
  constexpr int N = C::N, W = C::W, RS = C::RS, P = N + 1;
  constexpr int LW = N < 32 ? N : 32, PER = N / LW, CH = batch_of(PER);
  const int lane = threadIdx.x % LW;
#pragma unroll 1
  for (int c = threadIdx.x / LW; c < W; c += NT / LW) {
    const bool on = y0 + c <= N;
    const S* row = src + (size_t)(y0 + c) * P;
    const S last = on && lane == 0 ? __ldg(&row[N]) : (S)0;
#pragma unroll
    for (int i0 = 0; i0 < PER; i0 += CH) {
      S v[CH];
#pragma unroll
      for (int i = 0; i < CH; ++i) v[i] = on ? __ldg(&row[lane + LW * (i0 + i)]) : (S)0;
#pragma unroll
      for (int i = 0; i < CH; ++i) s[(lane + LW * (i0 + i)) * RS + c] = f(v[i]);
    }
    if (lane == 0) s[N * RS + c] = f(last);
  }
}

// x forward on the Neumann layout: W lines y0..y0+W-1 (y <= N) of plane z,
// r = alpha*src + corrections assembled while loading.  The irregular nodes
// (all interior) are listed per interior x-line in the interior numbering.
template <typename T, int N, int DIM>
__global__ void __launch_bounds__(NT) k_nxfwd(T* __restrict__ a, const double* __restrict__ src, double alpha,
                                              const float* __restrict__ src32,
                                              const double* __restrict__ corr, const int32_t* __restrict__ irr,
                                              const int32_t* __restrict__ line_start, const T* __restrict__ tw_g,
                                              const int* __restrict__ skip) {
  using C = NCfg<T, N>;
  constexpr int W = C::W, RS = C::RS, P = N + 1, n1 = N - 1;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* s = reinterpret_cast<T*>(smem_raw);
  T* tot = s + P * RS;
  T* tw = tot + C::G * W;
  T* x1 = tw + 4 * N;
  T* sinv = x1 + W;
  const bool skipped = skip != nullptr && *skip != 0;
  load_twiddles<T, N>(tw, tw_g);
  load_sines<C>(sinv, tw_g);
  if (skipped) return;
  const int y0 = blockIdx.x * W;
  const int z = DIM == 3 ? blockIdx.y : 0;
  const size_t plane = (size_t)z * P * P;
  if constexpr (!NBatch<T, N>::on) {
    for (int idx = threadIdx.x; idx < P * W; idx += NT) {
      const int x = idx % P, c = idx / P, y = y0 + c;
      T v = (T)0;
      if (y <= N) {
        if (src != nullptr) v = (T)alpha * to_T<T>(src[plane + (size_t)y * P + x]);
        else if (src32 != nullptr) v = (T)src32[plane + (size_t)y * P + x];
      }
      s[x * RS + c] = v;
    }
  } else if (src != nullptr) {
    const T a_t = (T)alpha;
    fill_lines_n<C>(s, src + plane, y0, [&](double v) { return a_t * to_T<T>(v); });
  } else if (src32 != nullptr) {
    fill_lines_n<C>(s, src32 + plane, y0, [&](float v) { return (T)v; });
  } else {
    for (int idx = threadIdx.x; idx < P * W; idx += NT) s[(idx % P) * RS + idx / P] = (T)0;
  }
  __syncthreads();
  if (corr != nullptr) {
    constexpr int G = NT / W;
    const int c = threadIdx.x % W, g = threadIdx.x / W, y = y0 + c;
    if (y >= 1 && y <= n1 && (DIM == 2 || (z >= 1 && z <= n1))) {
      const int line = DIM == 3 ? (z - 1) * n1 + (y - 1) : (y - 1);
      const int i0 = line_start[line], i1 = line_start[line + 1];
      for (int i = i0 + g; i < i1; i += G) {
        const int x = irr[i] % n1 + 1;
        s[x * RS + c] += (T)corr[i];
      }
    }
  }
  __syncthreads();
  dct_tile<C>(s, tw, sinv, tot, x1);
  for (int idx = threadIdx.x; idx < P * W; idx += NT) {
    const int x = idx % P, c = idx / P, y = y0 + c;
    if (y <= N) a[plane + (size_t)y * P + x] = s[x * RS + c];
  }
}

// x inverse on the Neumann layout: the work grid keeps v (keep) and/or
// out = beta v + gamma aux
template <typename T, int N, int DIM>
__global__ void __launch_bounds__(NT) k_nxinv(T* __restrict__ a, bool keep, double* __restrict__ out,
                                              const double* __restrict__ aux, double beta, double gamma,
                                              const T* __restrict__ tw_g, const int* __restrict__ skip,
                                              const float* __restrict__ aux32) {
  using C = NCfg<T, N>;
  constexpr int W = C::W, RS = C::RS, P = N + 1;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* s = reinterpret_cast<T*>(smem_raw);
  T* tot = s + P * RS;
  T* tw = tot + C::G * W;
  T* x1 = tw + 4 * N;
  T* sinv = x1 + W;
  if (skip != nullptr && *skip != 0) return;
  load_twiddles<T, N>(tw, tw_g);
  load_sines<C>(sinv, tw_g);
  const int y0 = blockIdx.x * W;
  const int z = DIM == 3 ? blockIdx.y : 0;
  const size_t plane = (size_t)z * P * P;
  for (int idx = threadIdx.x; idx < P * W; idx += NT) {
    const int x = idx % P, c = idx / P, y = y0 + c;
    if (y <= N) copy_async(&s[x * RS + c], &a[plane + (size_t)y * P + x]);
    else s[x * RS + c] = (T)0;
  }
  copy_async_wait();
  __syncthreads();
  dct_tile<C>(s, tw, sinv, tot, x1);
  const bool batch = NBatch<T, N>::on && (!NBatch<T, N>::plain || aux32 != nullptr || aux != nullptr);
  if (!NBatch<T, N>::on || !batch) {
    for (int idx = threadIdx.x; idx < P * W; idx += NT) {
      const int x = idx % P, c = idx / P, y = y0 + c;
      if (y > N) continue;
      const size_t o = plane + (size_t)y * P + x;
      const T v = s[x * RS + c];
      if (keep) a[o] = v;
      if (out != nullptr) {
        const double bv = to_double((T)beta * v);
        if (sizeof(T) == 4 && aux32 != nullptr)
          out[o] = bv + ffl::widen(aux32[o]);
        else
          out[o] = aux != nullptr ? fma(gamma, aux[o], bv) : bv;
      }
    }
  } else if constexpr (NBatch<T, N>::on) {
    constexpr int PER = N / 32, CH = batch_of(PER);
    const int lane = threadIdx.x & 31;
    const T b_t = (T)beta;
    auto put = [&](size_t o, T v, double w) {
      if (keep) a[o] = v;
      if (out != nullptr) {
        const double bv = to_double(b_t * v);
        out[o] = aux32 != nullptr ? bv + w : aux != nullptr ? fma(gamma, w, bv) : bv;
      }
    };
    auto other = [&](size_t o) { return aux32 != nullptr ? ffl::widen(aux32[o]) : aux != nullptr ? aux[o] : 0.0; };
#pragma unroll 1
    for (int c = threadIdx.x / 32; c < W; c += NT / 32) {
      if (y0 + c > N) continue;
      const size_t o = plane + (size_t)(y0 + c) * P + lane;
#pragma unroll
      for (int i0 = 0; i0 < PER; i0 += CH) {
        double w[CH];
#pragma unroll
        for (int i = 0; i < CH; ++i) w[i] = other(o + 32 * (i0 + i));
#pragma unroll
        for (int i = 0; i < CH; ++i) put(o + 32 * (i0 + i), s[(lane + 32 * (i0 + i)) * RS + c], w[i]);
      }
      if (lane == 0) put(o + N, s[N * RS + c], other(o + N));
    }
  }
}

// strided (y / z) pass on the Neumann layout: rows k = 0..N at row_stride,
// columns x0..x0+W-1 (x <= N) of plane q.  SOLVE: forward DCT, multiply by
// scale / (mu1[k] + mu1[p] + mu1[q] - lambda), inverse DCT.
template <typename T, int N, bool SOLVE, int DIM>
__global__ void __launch_bounds__(NT) k_nstrided(T* __restrict__ a, size_t row_stride, size_t plane_stride,
                                                 const T* __restrict__ mu1, T lambda, T scale,
                                                 const T* __restrict__ tw_g, const int* __restrict__ skip,
                                                 const T* __restrict__ rinv = nullptr) {
  using C = NCfg<T, N>;
  constexpr int W = C::W, RS = C::RS, P = N + 1;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* s = reinterpret_cast<T*>(smem_raw);
  T* tot = s + P * RS;
  T* tw = tot + C::G * W;
  T* x1 = tw + 4 * N;
  T* sinv = x1 + W;
  const bool skipped = skip != nullptr && *skip != 0;
  load_twiddles<T, N>(tw, tw_g);
  load_sines<C>(sinv, tw_g);
  if (skipped) return;
  const int x0 = blockIdx.x * W;
  const int q = blockIdx.y;
  T* base = a + (size_t)q * plane_stride + x0;
  for (int idx = threadIdx.x; idx < P * W; idx += NT) {
    const int c = idx % W, k = idx / W;
    if (x0 + c <= N) copy_async(&s[k * RS + c], &base[(size_t)k * row_stride + c]);
    else s[k * RS + c] = (T)0;
  }
  copy_async_wait();
  __syncthreads();
  dct_tile<C>(s, tw, sinv, tot, x1);
  if (SOLVE) {
    const T muq = DIM == 3 ? mu1[q] : (T)0;
    const T* rq = rinv != nullptr ? rinv + (size_t)q * P * P : nullptr;
    for (int idx = threadIdx.x; idx < P * W; idx += NT) {
      const int c = idx % W, k = idx / W, p = x0 + c;
      if (p <= N)
        s[k * RS + c] *= rq != nullptr ? rq[(size_t)k * P + p] : scale / (mu1[k] + mu1[p] + muq - lambda);
    }
    __syncthreads();
    dct_tile<C>(s, tw, sinv, tot, x1);
  }
  for (int idx = threadIdx.x; idx < P * W; idx += NT) {
    const int c = idx % W, k = idx / W;
    if (x0 + c <= N) base[(size_t)k * row_stride + c] = s[k * RS + c];
  }
}

template <typename T, int N>
int run_solve_neumann(kfbi_handle* h, const SolveArgs& sa, T* work, const T* mu1, const T* tw) {
  using C = NCfg<T, N>;
  constexpr int W = C::W, P = N + 1;
  const size_t smem = dct_smem_elems<C>() * sizeof(T);
  const int dim = h->grid.dim;
  cudaStream_t st = h->stream;
  const Tables& t = h->t;
  const T scale = (T)(dim == 3 ? (2.0 / N) * (2.0 / N) * (2.0 / N) : (2.0 / N) * (2.0 / N));
  const T lam = (T)sa.lambda;
  const dim3 grid((P + W - 1) / W, dim == 3 ? P : 1);
  const size_t PP = (size_t)P * P;
  const T* rinv = mode_factors<T, N>(h, sa.lambda, (double)scale);
  int rc;
  if (dim == 3) {
    if ((rc = prep(k_nxfwd<T, N, 3>, smem))) return rc;
    if ((rc = prep(k_nstrided<T, N, false, 3>, smem))) return rc;
    if ((rc = prep(k_nstrided<T, N, true, 3>, smem))) return rc;
    if ((rc = prep(k_nxinv<T, N, 3>, smem))) return rc;
    k_nxfwd<T, N, 3><<<grid, NT, smem, st>>>(work, sa.src, sa.alpha, sa.src32, sa.corr, t.irr, t.line_start, tw,
                                                h->skip);
    k_nstrided<T, N, false, 3><<<grid, NT, smem, st>>>(work, P, PP, mu1, lam, scale, tw, h->skip);
    k_nstrided<T, N, true, 3><<<grid, NT, smem, st>>>(work, PP, P, mu1, lam, scale, tw, h->skip, rinv);
    k_nstrided<T, N, false, 3><<<grid, NT, smem, st>>>(work, P, PP, mu1, lam, scale, tw, h->skip);
    k_nxinv<T, N, 3><<<grid, NT, smem, st>>>(work, sa.keep || sa.out_user == nullptr, sa.out_user, sa.aux, sa.beta,
                                              sa.gamma, tw, h->skip, sa.aux32);
    KFBI_CHECK_LAUNCH_N(5);
  } else {
    if ((rc = prep(k_nxfwd<T, N, 2>, smem))) return rc;
    if ((rc = prep(k_nstrided<T, N, true, 2>, smem))) return rc;
    if ((rc = prep(k_nxinv<T, N, 2>, smem))) return rc;
    k_nxfwd<T, N, 2><<<grid, NT, smem, st>>>(work, sa.src, sa.alpha, sa.src32, sa.corr, t.irr, t.line_start, tw,
                                                h->skip);
    k_nstrided<T, N, true, 2><<<grid, NT, smem, st>>>(work, P, 0, mu1, lam, scale, tw, h->skip, rinv);
    k_nxinv<T, N, 2><<<grid, NT, smem, st>>>(work, sa.keep || sa.out_user == nullptr, sa.out_user, sa.aux, sa.beta,
                                              sa.gamma, tw, h->skip, sa.aux32);
    KFBI_CHECK_LAUNCH_N(3);
  }
  return KFBI_OK;
}

template <typename T>
int box_solve_neumann(kfbi_handle* h, const SolveArgs& sa, T* work, const T* mu1, const T* tw) {
  if (!(sa.lambda > 0.0)) {
    set_error("the Neumann box needs lambda > 0 (no Green's function of the Poisson operator exists)");
    return KFBI_ERR_ARG;
  }
  switch (h->grid.N) {
    case 8: return run_solve_neumann<T, 8>(h, sa, work, mu1, tw);
    case 16: return run_solve_neumann<T, 16>(h, sa, work, mu1, tw);
    case 32: return run_solve_neumann<T, 32>(h, sa, work, mu1, tw);
    case 64: return run_solve_neumann<T, 64>(h, sa, work, mu1, tw);
    case 128: return run_solve_neumann<T, 128>(h, sa, work, mu1, tw);
    case 256: return run_solve_neumann<T, 256>(h, sa, work, mu1, tw);
    case 384: return run_solve_neumann<T, 384>(h, sa, work, mu1, tw);
    case 512: return run_solve_neumann<T, 512>(h, sa, work, mu1, tw);
    default:
      set_error("unsupported grid size N=%d", h->grid.N);
      return KFBI_ERR_ARG;
  }
}

}  // namespace

#if KFBI_DST_BITS == 32
// TMA descriptors of the padded float32 grid for the strided passes (3-D,
// 32 <= N <= 256): boxes of 32 x-values by N rows along y or along z.
int make_tma_maps(kfbi_handle* h) {
  h->tma = false;
  {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && sms > 0)
      h->sms = sms;
    cudaGetLastError();
  }
  const int N = h->grid.N;
  if (h->grid.dim != 3 || N < TMA_W || N > 256) return KFBI_OK;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess || fn == nullptr) {
    cudaGetLastError();
    return KFBI_OK;  // no tensor maps: the strided passes keep their plain loads
  }
  auto encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  const cuuint64_t dims[3] = {(cuuint64_t)N, (cuuint64_t)N, (cuuint64_t)N};
  const cuuint64_t strides[2] = {(cuuint64_t)N * sizeof(float), (cuuint64_t)N * N * sizeof(float)};
  const cuuint32_t estr[3] = {1, 1, 1};
  for (int second = 0; second < 2; ++second)
    for (int near = 0; near < 2; ++near)
      for (int axis = 0; axis < 2; ++axis) {
        const Span r = near == 0 ? Span{0, N} : axis == 0 ? h->near_y : h->near_z;
        const cuuint32_t rows = (cuuint32_t)(r.hi - r.lo);
        const cuuint32_t box[3] = {(cuuint32_t)TMA_W, axis == 0 ? rows : 1, axis == 0 ? 1 : rows};
        const CUresult e = encode(&h->tmap[second][near][axis], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3,
                                  second ? h->w.grid32b : h->w.grid32, dims, strides, box, estr,
                                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (e != CUDA_SUCCESS) {
          set_error("cuTensorMapEncodeTiled failed (%d)", (int)e);
          return KFBI_ERR_CUDA;
        }
      }
  h->tma = true;
  // fused x-y passes need cluster launches (a cluster of N/32 blocks per
  // plane).  They pay off only for small planes: measured per float32 solve
  // (CUDA events, back-to-back) 18.8 against 24.4 us at 64^3, 48.4 against
  // 47.7 us at 128^3 and 211 against 172 us at 256^3, where the separate
  // passes are bound by the transforms' instruction issue with the grid in
  // L2, and the fused blocks add two cluster barriers and the exchange.
  int dev = 0, cl = 0;
  cudaGetDevice(&dev);
  if (N <= 64 && cudaDeviceGetAttribute(&cl, cudaDevAttrClusterLaunch, dev) == cudaSuccess && cl) h->xy_fused = true;
  cudaGetLastError();
  return KFBI_OK;
}

int transform_pass32(kfbi_handle* h, int pass, double lambda) {
  return dispatch_pass<float>(h, pass, lambda, h->w.grid32, h->t.mu32, h->t.tw32);
}

int dst_supported(int N) {
  return N == 8 || N == 16 || N == 32 || N == 64 || N == 128 || N == 256 || N == 384 || N == 512;
}

int box_solve32(kfbi_handle* h, const SolveArgs& a, float* work) {
  if (h->grid.bc == KFBI_BOX_NEUMANN) return box_solve_neumann<float>(h, a, work, h->t.mu32, h->t.tw32);
  return dispatch<float>(h, a, work, h->t.mu32, h->t.tw32);
}
#else
int transform_pass64(kfbi_handle* h, int pass, double lambda) {
  return dispatch_pass<double>(h, pass, lambda, h->w.grid64, h->t.mu, h->t.tw64);
}

int box_solve64(kfbi_handle* h, const SolveArgs& a, double* work) {
  if (h->grid.bc == KFBI_BOX_NEUMANN) return box_solve_neumann<double>(h, a, work, h->t.mu, h->t.tw64);
  return dispatch<double>(h, a, work, h->t.mu, h->t.tw64);
}
#endif

namespace {
template <typename T>
int dispatch_coupled(kfbi_handle* h, const SolveArgs& si, const SolveArgs& se, const Coupling& cp, T* wa, T* wb,
                     const T* mu1T, const T* tw) {
  switch (h->grid.N) {
    case 16: return run_solve_coupled<T, 16>(h, si, se, cp, wa, wb, mu1T, tw);
    case 32: return run_solve_coupled<T, 32>(h, si, se, cp, wa, wb, mu1T, tw);
    case 64: return run_solve_coupled<T, 64>(h, si, se, cp, wa, wb, mu1T, tw);
    case 128: return run_solve_coupled<T, 128>(h, si, se, cp, wa, wb, mu1T, tw);
    case 256: return run_solve_coupled<T, 256>(h, si, se, cp, wa, wb, mu1T, tw);
    case 384: return run_solve_coupled<T, 384>(h, si, se, cp, wa, wb, mu1T, tw);
    case 512: return run_solve_coupled<T, 512>(h, si, se, cp, wa, wb, mu1T, tw);
    default:
      set_error("unsupported grid size N=%d for the coupled solve", h->grid.N);
      return KFBI_ERR_ARG;
  }
}
}  // namespace

#if KFBI_DST_BITS == 64
int box_solve_coupled64(kfbi_handle* h, const SolveArgs& si, const SolveArgs& se, const Coupling& cp, double* wa,
                        double* wb) {
  return dispatch_coupled<double>(h, si, se, cp, wa, wb, h->t.mu, h->t.tw64);
}
#else
int box_solve_coupled32(kfbi_handle* h, const SolveArgs& si, const SolveArgs& se, const Coupling& cp, float* wa,
                        float* wb) {
  return dispatch_coupled<float>(h, si, se, cp, wa, wb, h->t.mu32, h->t.tw32);
}

namespace {
// an mbarrier that nothing ever completes, polled with the transform
// kernels' bounded wait: the poll cap must end the wait and raise the flag
__global__ void k_selftest_wait(long cap, int* err) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_fence_init();
  }
  __syncthreads();
  bool ok = false;
  for (long it = 0; it < cap; ++it)
    if (mbar_try_wait(&bar, 0u)) {
      ok = true;
      break;
    }
  if (!ok && threadIdx.x == 0) atomicOr(err, DEVERR_TIMEOUT);
}
}  // namespace
#endif  // KFBI_DST_BITS

}  // namespace kfbi

#if KFBI_DST_BITS == 32
extern "C" int kfbi_selftest_bounded_wait(int polls, int* timed_out, double* ms) {
  using namespace kfbi;
  if (polls < 1 || polls > (1 << 20) || !timed_out) {
    set_error("polls must be in 1 .. 2^20");
    return KFBI_ERR_ARG;
  }
  int* err = nullptr;
  KFBI_CUDA(cudaMalloc(&err, sizeof(int)));
  cudaEvent_t a, b;
  cudaEventCreate(&a);
  cudaEventCreate(&b);
  cudaMemset(err, 0, sizeof(int));
  cudaEventRecord(a);
  k_selftest_wait<<<1, 32>>>((long)polls, err);
  cudaEventRecord(b);
  const cudaError_t e = cudaEventSynchronize(b);
  int herr = 0;
  if (e == cudaSuccess) cudaMemcpy(&herr, err, sizeof(int), cudaMemcpyDeviceToHost);
  float t = 0.0f;
  cudaEventElapsedTime(&t, a, b);
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  cudaFree(err);
  if (e != cudaSuccess) {
    set_error("self-test launch failed: %s", cudaGetErrorString(e));
    return KFBI_ERR_CUDA;
  }
  *timed_out = (herr & DEVERR_TIMEOUT) ? 1 : 0;
  if (ms) *ms = t;
  KFBI_COUNT(1);
  return KFBI_OK;
}
#endif  // KFBI_DST_BITS
