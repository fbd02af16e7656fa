// DST-I of the W = 32 columns of a float64 tile in 64-bit block fixed point,
// 256 threads (8 warps) per tile (Sections 5.2-5.3: the box solve is a sine
// transform along each axis).
//
// GB300 issues 2 float64 instructions per SM per clock and 64 or more integer
// ones, and a transform is additions and products with constants of size at
// most 1: both are exact or nearly exact on integers.  Each column (one
// transform line) is scaled by a power of two, transformed on 64-bit
// integers, and scaled back:
//  - an addition is exact (two 32-bit instructions);
//  - a product with a table value w, held as round(w 2^62) or round(w 2^63),
//    takes three 32 x 32 -> 64 bit products and is rounded to the nearest
//    unit;
//  - values enter by shifts of their bits and leave by two float64
//    operations.
//
// Scale.  Let |x| <= m in a column of integers and A = sum |x|.  The folded
// values are |y| <= 2 m max(sin, 1/2); a component of a sum over the P complex
// values of the FFT's first level stays below min(1.83 P m, 2 A) (the largest
// over all levels' angles), any later one below min(1.44 N m, 2 A) (sum |y_j|
// <= sum over pairs of 4 m max(sin, 1/2), or 2 (|x_j| + |x_{N-j}|)).  The
// column's largest value gets as many bits as keep these below 2^61: `early`
// bits up to the first level's twiddles, whose products are shifted down to
// `late` bits.  A costs three integer instructions per value and pays in lines
// with few large values (corrections along x, decaying spectra): without it
// those lost two to three bits.
//
// Rounding.  The running sum of the odd outputs collects what the values
// before it share: a mean of a quarter unit in the first level's results cost
// lines of a background and a few larger values a factor of up to four.  So
// values enter the pre-fold at 60 bits (below 2^-60 of the largest cut off)
// and are rounded once, after it; products round to the nearest unit at their
// final scale; and integers that a shift alone brings there, where half units
// are common, round half to even (the first level's, see phase A1, up and
// down in turn).
// Error (2-norm, against 80-bit arithmetic, over that of the same transform in
// float64 with exact tables): 0.1 to 0.6 over smooth, dense, sparse, widely
// scaled and single-mode lines.  Its worst lines are a low background with
// few values far above it, whose unit is that of the largest: at most 0.6 up
// to 256 lines, 0.9 at 512 and 1.2 at 384.
//
// Measured (GB300, CUDA events): a 256^3 float64 box solve took 4.16 ms with
// float64 butterflies (26 float64 instructions per point and transform, at
// 1/32 of the integer rate) and takes 0.76 ms; its error against dense
// float64 products went from 5.3e-15 to 1.9e-15 (2-norm, smooth field).
//
// The decomposition is that of dst_reg.cuh (two-level FFT m = a + 8q, k = k1
// + P k2, one exchange, split pairs in registers, segmented scan); here the
// pre-fold works on pairs (j, N - j) held by one thread, so that each value
// is converted once, and the scan's additions are exact.
//
// The phases are plain functions of (a, c) and per-thread state, run on the
// host too, one simulated thread at a time, to check index arithmetic and
// error.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifndef KFBI_HD
#ifdef __CUDACC__
#define KFBI_HD __host__ __device__ __forceinline__
#else
#define KFBI_HD inline
#endif
#endif

namespace kfbi {
namespace fixdst {

typedef long long ll;

// ------------------------------------------------------------ bit access
KFBI_HD ll bits_of(double x) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(x);
#else
  ll r;
  memcpy(&r, &x, 8);
  return r;
#endif
}
KFBI_HD double double_of(ll b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double r;
  memcpy(&r, &b, 8);
  return r;
#endif
}
KFBI_HD int32_t hi_of(ll a) { return (int32_t)(a >> 32); }
KFBI_HD int32_t lo_of(ll a) { return (int32_t)(uint32_t)(uint64_t)a; }
KFBI_HD ll make_ll(int32_t hi, uint32_t lo) { return (ll)(((uint64_t)(uint32_t)hi << 32) | lo); }

// ------------------------------------------------------------ fixed constants
// a table value as two signed words: w 2^S = h 2^32 + l, |l| <= 2^31
struct fx {
  int32_t h, l;
};
// a complex twiddle at S = 62 (|w| <= 1, so |h| <= 2^30)
struct alignas(16) cfx {
  fx r, i;
};

KFBI_HD constexpr fx fx_of(ll v) {
  const uint32_t lo = (uint32_t)(uint64_t)v;
  // l = -2^31 is avoided, so that -l is representable
  ll w = lo == 0x80000000u ? v + 1 : v;
  const int32_t l = (int32_t)(uint32_t)(uint64_t)w;
  return fx{(int32_t)((w - (ll)l) >> 32), l};
}

// round-to-nearest of w 2^S on the bits of w (|w| <= 1, S = 62 or 63)
KFBI_HD ll scaled_int(double w, int S) {
  const ll b = bits_of(w);
  const int e = (int)((b >> 52) & 0x7ff);
  ll m = (b & 0x000fffffffffffffLL) | (e ? 0x0010000000000000LL : 0);
  const int sh = e - 1075 + S;  // |w| = m 2^(e - 1075)
  if (sh >= 0)
    m <<= sh;
  else if (sh > -60)
    m = ((m >> (-sh - 1)) + 1) >> 1;
  else
    m = 0;
  return b < 0 ? -m : m;
}
KFBI_HD fx fx_table(double w, int S) {
  ll v = scaled_int(w, S);
  if ((uint32_t)(uint64_t)v == 0x80000000u) v += 1;
  const int32_t l = lo_of(v);
  return fx{(int32_t)((v - (ll)l) >> 32), l};
}

// ------------------------------------------------------------ products
// a = h 2^32 + l with signed l
KFBI_HD void halves(ll a, int32_t& h, int32_t& l) {
  l = lo_of(a);
  h = hi_of(a) + (int32_t)((uint32_t)l >> 31);
}

// round(a w) for w at S = 63, |w| < 1, |a| < 2^62 - 2^32
KFBI_HD ll mul63(ll a, fx w) {
  int32_t h, l;
  halves(a, h, l);
  const ll t = (ll)h * w.l + ((ll)l * w.h + (1LL << 30));
  return (ll)(2 * h) * w.h + (t >> 31);
}

// (xr + i xi) w for w at S = 62, |w| <= 1, |xr|, |xi| < 2^61 - 2^32; with
// half = 2^(29 + sh) the caller's shift of the result by sh rounds to the
// nearest (half = 2^29: rounded here)
KFBI_HD void cmul62(ll& xr, ll& xi, const cfx& w, ll half = 1LL << 29) {
  int32_t rh, rl, ih, il;
  halves(xr, rh, rl);
  halves(xi, ih, il);
  const int32_t nh = -w.i.h, nl = -w.i.l;
  const ll t = (ll)rh * w.r.l + ((ll)rl * w.r.h + ((ll)ih * nl + ((ll)il * nh + half)));
  const ll u = (ll)rh * w.i.l + ((ll)rl * w.i.h + ((ll)ih * w.r.l + ((ll)il * w.r.h + half)));
  const int32_t r4 = 4 * rh, i4 = 4 * ih;
  xr = (ll)r4 * w.r.h + ((ll)i4 * nh + (t >> 30));
  xi = (ll)r4 * w.i.h + ((ll)i4 * w.r.h + (u >> 30));
}

// a / 2 rounded half to even (floor would leave a bias that the sums collect)
KFBI_HD ll half_even(ll a) { return (a + (ll)((lo_of(a) >> 1) & 1)) >> 1; }
// a / 2^sh rounded half to even (sh >= 0)
KFBI_HD ll shift_even(ll a, int sh) {
  const ll r = (1LL << sh) >> 1;
  return (a + r - (ll)((int32_t)(sh > 0) & ~lo_of(a >> sh) & 1)) >> sh;
}

// sqrt(1/2) and sqrt(3)/2 at S = 63, cos(pi/8), sin(pi/8) at S = 62
#define KFBI_FX_R2 fx_of(0x5A827999FCEF3242LL)
#define KFBI_FX_S3 fx_of(0x6ED9EBA16132A9CFLL)
#define KFBI_FX_C8 fx_of(0x3B20D79E651A8C51LL)
#define KFBI_FX_S8 fx_of(0x187DE2A6AEA962D2LL)

// ------------------------------------------------------------ butterflies
// b_p = sum_q a_q e^{+2 pi i p q / R}, in place
template <int R>
struct Dft;

template <>
struct Dft<1> {
  static KFBI_HD void run(ll*, ll*) {}
};

template <>
struct Dft<2> {
  static KFBI_HD void run(ll* xr, ll* xi) {
    const ll ar = xr[0] + xr[1], ai = xi[0] + xi[1];
    xr[1] = xr[0] - xr[1];
    xi[1] = xi[0] - xi[1];
    xr[0] = ar;
    xi[0] = ai;
  }
};

template <>
struct Dft<3> {
  static KFBI_HD void run(ll* xr, ll* xi) {
    const ll tr = xr[1] + xr[2], ti = xi[1] + xi[2];
    const ll ur = mul63(xr[1] - xr[2], KFBI_FX_S3), ui = mul63(xi[1] - xi[2], KFBI_FX_S3);
    const ll mr = xr[0] - half_even(tr), mi = xi[0] - half_even(ti);
    xr[0] += tr;
    xi[0] += ti;
    xr[1] = mr - ui;  // m + i s3 u
    xi[1] = mi + ur;
    xr[2] = mr + ui;  // m - i s3 u
    xi[2] = mi - ur;
  }
};

template <>
struct Dft<4> {
  static KFBI_HD void run(ll* xr, ll* xi) {
    const ll t0r = xr[0] + xr[2], t0i = xi[0] + xi[2];
    const ll t1r = xr[0] - xr[2], t1i = xi[0] - xi[2];
    const ll t2r = xr[1] + xr[3], t2i = xi[1] + xi[3];
    const ll t3r = xr[1] - xr[3], t3i = xi[1] - xi[3];
    xr[0] = t0r + t2r;
    xi[0] = t0i + t2i;
    xr[2] = t0r - t2r;
    xi[2] = t0i - t2i;
    xr[1] = t1r - t3i;  // t1 + i t3
    xi[1] = t1i + t3r;
    xr[3] = t1r + t3i;  // t1 - i t3
    xi[3] = t1i - t3r;
  }
};

// (xr + i xi) e^{i pi / 4}
KFBI_HD void rot1(ll& xr, ll& xi) {
  const ll r = mul63(xr - xi, KFBI_FX_R2), i = mul63(xr + xi, KFBI_FX_R2);
  xr = r;
  xi = i;
}
// (xr + i xi) e^{3 i pi / 4}
KFBI_HD void rot3(ll& xr, ll& xi) {
  const ll r = -mul63(xr + xi, KFBI_FX_R2), i = mul63(xr - xi, KFBI_FX_R2);
  xr = r;
  xi = i;
}

template <>
struct Dft<8> {
  static KFBI_HD void run(ll* xr, ll* xi) {
    ll er[4] = {xr[0], xr[2], xr[4], xr[6]}, ei[4] = {xi[0], xi[2], xi[4], xi[6]};
    ll qr[4] = {xr[1], xr[3], xr[5], xr[7]}, qi[4] = {xi[1], xi[3], xi[5], xi[7]};
    Dft<4>::run(er, ei);
    Dft<4>::run(qr, qi);
    rot1(qr[1], qi[1]);
    rot3(qr[3], qi[3]);
    xr[0] = er[0] + qr[0];
    xi[0] = ei[0] + qi[0];
    xr[4] = er[0] - qr[0];
    xi[4] = ei[0] - qi[0];
    xr[1] = er[1] + qr[1];
    xi[1] = ei[1] + qi[1];
    xr[5] = er[1] - qr[1];
    xi[5] = ei[1] - qi[1];
    xr[2] = er[2] - qi[2];  // + i O_2
    xi[2] = ei[2] + qr[2];
    xr[6] = er[2] + qi[2];
    xi[6] = ei[2] - qr[2];
    xr[3] = er[3] + qr[3];
    xi[3] = ei[3] + qi[3];
    xr[7] = er[3] - qr[3];
    xi[7] = ei[3] - qi[3];
  }
};

// 16 = 4 x 4: q = 4 q1 + q2, p = p1 + 4 p2; radix 4 over q1, twiddle
// e^{2 pi i p1 q2 / 16}, radix 4 over q2; the outputs end in order
template <>
struct Dft<16> {
  static KFBI_HD void run(ll* xr, ll* xi) {
    const cfx w1 = {KFBI_FX_C8, KFBI_FX_S8};                                  // e = 1
    const cfx w3 = {KFBI_FX_S8, KFBI_FX_C8};                                  // e = 3
    const cfx w9 = {{-KFBI_FX_C8.h, -KFBI_FX_C8.l}, {-KFBI_FX_S8.h, -KFBI_FX_S8.l}};  // e = 9
    ll ar[4][4], ai[4][4];  // [q2][p1]
#pragma unroll
    for (int q2 = 0; q2 < 4; ++q2) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        ar[q2][u] = xr[q2 + 4 * u];
        ai[q2][u] = xi[q2 + 4 * u];
      }
      Dft<4>::run(ar[q2], ai[q2]);
    }
    cmul62(ar[1][1], ai[1][1], w1);
    rot1(ar[1][2], ai[1][2]);
    cmul62(ar[1][3], ai[1][3], w3);
    rot1(ar[2][1], ai[2][1]);
    {  // e = 4: times i
      const ll t = ar[2][2];
      ar[2][2] = -ai[2][2];
      ai[2][2] = t;
    }
    rot3(ar[2][3], ai[2][3]);
    cmul62(ar[3][1], ai[3][1], w3);
    rot3(ar[3][2], ai[3][2]);
    cmul62(ar[3][3], ai[3][3], w9);
#pragma unroll
    for (int p1 = 0; p1 < 4; ++p1) {
      ll tr[4] = {ar[0][p1], ar[1][p1], ar[2][p1], ar[3][p1]};
      ll ti[4] = {ai[0][p1], ai[1][p1], ai[2][p1], ai[3][p1]};
      Dft<4>::run(tr, ti);
#pragma unroll
      for (int p2 = 0; p2 < 4; ++p2) {
        xr[p1 + 4 * p2] = tr[p2];
        xi[p1 + 4 * p2] = ti[p2];
      }
    }
  }
};

// P = R1 R2 with twiddles e^{2 pi i e / P} = sp[e N/P] (its second half by
// sign) from the shared table sp[k] = e^{2 pi i k / N}, k < N/2
template <int R1, int R2>
struct DftT {
  static KFBI_HD void run(ll* xr, ll* xi, const cfx* sp, int step) {
    constexpr int P = R1 * R2;
#pragma unroll
    for (int q2 = 0; q2 < R2; ++q2) {
      ll tr[R1], ti[R1];
#pragma unroll
      for (int q1 = 0; q1 < R1; ++q1) {
        tr[q1] = xr[q2 + R2 * q1];
        ti[q1] = xi[q2 + R2 * q1];
      }
      Dft<R1>::run(tr, ti);
#pragma unroll
      for (int p1 = 0; p1 < R1; ++p1) {
        const int e = (p1 * q2) % P;
        if (e != 0) cmul62(tr[p1], ti[p1], sp[(e % (P / 2)) * step]);
        xr[q2 + R2 * p1] = e < P / 2 ? tr[p1] : -tr[p1];
        xi[q2 + R2 * p1] = e < P / 2 ? ti[p1] : -ti[p1];
      }
    }
    ll outr[P], outi[P];
#pragma unroll
    for (int p1 = 0; p1 < R1; ++p1) {
      Dft<R2>::run(xr + R2 * p1, xi + R2 * p1);
#pragma unroll
      for (int p2 = 0; p2 < R2; ++p2) {
        outr[p1 + R1 * p2] = xr[R2 * p1 + p2];
        outi[p1 + R1 * p2] = xi[R2 * p1 + p2];
      }
    }
#pragma unroll
    for (int i = 0; i < P; ++i) {
      xr[i] = outr[i];
      xi[i] = outi[i];
    }
  }
};

template <int P, int N>
KFBI_HD void dft_first(ll* xr, ll* xi, const cfx* sp) {
  if constexpr (P == 24) {
    DftT<3, 8>::run(xr, xi, sp, N / P);
  } else if constexpr (P == 32) {
    DftT<4, 8>::run(xr, xi, sp, N / P);
  } else {
    Dft<P>::run(xr, xi);
  }
}

// ------------------------------------------------------------ column scale
// Scale of a column from the exponent field emax of its largest value and
// asum >= 2^20 A / 2^(emax - 1023): late bits 2^late with |x| < 2^(emax -
// 1022).  Exponents below 64 count as 64 (values below 2^-959 then have fewer
// bits).  A column that holds an infinity or NaN is transformed to NaN
// throughout, as in float64.
constexpr double HUGE_STEP = 0x1p512;
constexpr int FOLD_BITS = 60;  // the sum of two values stays below 2^62 - 2^32
struct Scale {
  int in;          // shift of a 63-bit significand of the largest exponent, plus its exponent field
  int fold;        // shift of twice a folded value from FOLD_BITS to early bits
  int sh;          // early - late
  double out, oc;  // 2^(-k-1) (the integers are twice the outputs) and (2^84 + 2^63 + 2^52) 2^(-k-1)
  bool huge;       // both are smaller by HUGE_STEP (oc would overflow): the outputs need it back
};
KFBI_HD int bit_length(uint32_t v) {
#ifdef __CUDA_ARCH__
  return 32 - __clz((int)v);
#else
  return v ? 32 - __builtin_clz(v) : 0;
#endif
}
constexpr int EARLY_MORE = 4;
template <int N>
KFBI_HD constexpr int late_bits() {
  // 1.44 N 2^late < 2^61 and 1.83 (N / 16) 2^(late + EARLY_MORE) < 2^61
  return N <= 32 ? 55 : N <= 64 ? 54 : N <= 128 ? 53 : N <= 256 ? 52 : 51;
}
template <int N>
KFBI_HD Scale scale_of(int emax, uint32_t asum) {
  Scale s;
  const int e = emax < 64 ? 64 : emax;
  // 2 A 2^(b - (emax - 1022)) < 2^(bit_length - 20 + b) = 2^60
  const int b1 = 80 - bit_length(asum);
  const int late = b1 > late_bits<N>() ? b1 : late_bits<N>();
  // twice that is enough for sums that no difference doubles
  const int early = b1 + 1 > late_bits<N>() + EARLY_MORE ? b1 + 1 : late_bits<N>() + EARLY_MORE;
  s.in = e + 63 - FOLD_BITS;
  s.fold = FOLD_BITS + 1 - early;
  s.sh = early - late;
  s.huge = e > 1900;
  const int eo = e - late - (s.huge ? 512 : 0);  // biased exponent of 2^(-k-1)
  s.out = double_of(emax == 0x7ff ? 0x7ff8000000000000LL : (ll)eo << 52);
  s.oc = s.out * double_of(0x4530000080100000LL);  // 2^84 + 2^63 + 2^52
  return s;
}
// x as an integer of FOLD_BITS bits, on its bits: the significand shifted by
// the distance to the largest exponent (truncated: 53 bits lose theirs from
// 2^-7 of the largest value on, below any later unit; zeros and subnormal
// values come out as 0, their distance being 64 or more)
KFBI_HD ll to_fix(double x, const Scale& s) {
  const ll b = bits_of(x);
  const int32_t h = hi_of(b);
  int d = s.in - ((h >> 20) & 0x7ff);
  d = d > 63 ? 63 : d;
  const uint64_t m = (uint64_t)make_ll((h & 0x000fffff) | 0x00100000, (uint32_t)lo_of(b)) << 10;
  const ll n = (ll)(m >> d);
  const ll sg = (ll)(h >> 31);
  return (n ^ sg) - sg;
}
// n 2^(-k-1), rounded once: 2^84 + 2^63 + (high word) 2^32 and 2^52 + (low word)
// have their words in place, so both are formed on the bits
KFBI_HD double from_fix(ll n, const Scale& s) {
  const double h = double_of(make_ll(0x45300000, (uint32_t)hi_of(n) ^ 0x80000000u));
  const double l = double_of(make_ll(0x43300000, (uint32_t)lo_of(n)));
  // (nested differently, the sum would not be exact before its last addition)
  const double t = fma(h, s.out, -s.oc);
  return fma(l, s.out, t);
}

// ------------------------------------------------------------ tile phases
// N rows (transform index), W = 32 columns, row stride RS; 8 warps, P points
// per thread in the first level
template <int N_, int RS_>
struct Geo {
  static constexpr int N = N_, RS = RS_, W = 32, T = 8;
  static constexpr int L = N / 2;
  static constexpr int P = L / T;
  static constexpr int NG = P / 2 > 0 ? P / 2 : 1;
  static constexpr int GPT = (NG + T - 1) / T;
  static_assert(N >= 32 && L % T == 0, "tile too short for the fixed-point DST");
};

template <class G>
struct State {
  double xa[G::P], xb[G::P];       // rows j = a + 8 i and N - j (phase 0)
  ll zr[G::P], zi[G::P];           // first level
  ll Ar[G::GPT][8], Ai[G::GPT][8];
  ll Br[G::GPT][8], Bi[G::GPT][8];
  ll v[G::P];                      // scan segment
  int emax;
  Scale sc;
};

// phase 0: the thread's row pairs of column c to registers, its largest
// exponent field to mx[a][c].  Thread 0 of the column holds row N/2 (its own
// mirror image) in place of the pair of row 0.
template <class G>
KFBI_HD void phase_0(State<G>& st, const double* s, int* mx, int a, int c) {
  constexpr int N = G::N, RS = G::RS, T = G::T, P = G::P, W = G::W;
  uint32_t m = 0;
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const int j = a + T * i;
    const int ja = j == 0 ? N / 2 : j, jb = j == 0 ? N / 2 : N - j;
    st.xa[i] = s[ja * RS + c];
    st.xb[i] = s[jb * RS + c];
  }
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const uint32_t ha = (uint32_t)hi_of(bits_of(st.xa[i])) & 0x7fffffffu;
    const uint32_t hb = (uint32_t)hi_of(bits_of(st.xb[i])) & 0x7fffffffu;
    m = ha > m ? ha : m;
    m = hb > m ? hb : m;
  }
  mx[a * W + c] = (int)(m >> 20);
}

// phase S: the thread's share of A, in units of 2^-20 of the largest power
// of two (rounded up), to sm[a][c]
template <class G>
KFBI_HD void phase_s(State<G>& st, const int* mx, uint32_t* sm, int a, int c) {
  constexpr int T = G::T, P = G::P, W = G::W;
  int e = 0;
#pragma unroll
  for (int b = 0; b < T; ++b) e = mx[b * W + c] > e ? mx[b * W + c] : e;
  st.emax = e;
  uint32_t sum = 2 * P;
#pragma unroll
  for (int i = 0; i < P; ++i) {
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const uint32_t h = (uint32_t)hi_of(bits_of(side ? st.xb[i] : st.xa[i]));
      int d = e - (int)((h >> 20) & 0x7ff);
      d = d > 31 ? 31 : d;
      sum += ((h & 0x000fffffu) | 0x00100000u) >> d;
    }
  }
  sm[a * W + c] = sum;
}

// phase 1: column scale, conversion, sine pre-fold of the pairs
//   y_j = sin(pi j / N)(x_j + x_{N-j}) + (x_j - x_{N-j}) / 2,  y_0 = 0,
// twice y_j at FOLD_BITS bits shifted down to early bits
template <class G>
KFBI_HD void phase_1(State<G>& st, ll* s, const uint32_t* sm, const fx* sinv, int a, int c) {
  constexpr int N = G::N, RS = G::RS, T = G::T, P = G::P, W = G::W;
  uint32_t asum = 0;
#pragma unroll
  for (int b = 0; b < T; ++b) asum += sm[b * W + c];
  st.sc = scale_of<N>(st.emax, asum);
  const int fold = st.sc.fold;
  const ll r = 1LL << (fold - 1);
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const int j = a + T * i;
    const ll na = to_fix(st.xa[i], st.sc), nb = to_fix(st.xb[i], st.sc);
    if (i == 0 && a == 0) {
      s[c] = 0;
      s[(N / 2) * RS + c] = (4 * na + r) >> fold;
    } else {
      const ll t = 2 * mul63(na + nb, sinv[j]) + r, d = na - nb;
      s[j * RS + c] = (t + d) >> fold;
      s[(N - j) * RS + c] = (t - d) >> fold;
    }
  }
}

// phase A1: first-level DFT over q and twiddle w_L^{a k1} (lv[a][k1])
template <class G>
KFBI_HD void phase_a1(State<G>& st, const ll* s, const cfx* sp, const cfx* lv, int a, int c) {
  constexpr int N = G::N, RS = G::RS, T = G::T, P = G::P;
#pragma unroll
  for (int q = 0; q < P; ++q) {
    const int j = 2 * (a + T * q);
    st.zr[q] = s[j * RS + c];
    st.zi[q] = s[(j + 1) * RS + c];
  }
  dft_first<P, N>(st.zr, st.zi, sp);
  const int sh = st.sc.sh;
  st.zr[0] = shift_even(st.zr[0], sh);
  st.zi[0] = shift_even(st.zi[0], sh);
  // for a = 0 all twiddles are 1 and half units are common: they round up
  // for even k1 and down for odd k1, which the running sum over k cancels
  const ll half = 1LL << (29 + sh);
#pragma unroll
  for (int k1 = 1; k1 < P; ++k1) {
    cmul62(st.zr[k1], st.zi[k1], lv[a * P + k1], half - (k1 & 1));
    st.zr[k1] >>= sh;
    st.zi[k1] >>= sh;
  }
}

struct alignas(16) c2 {
  ll x, y;
};

// phase A2: to the exchange buffer (after a barrier)
template <class G>
KFBI_HD void phase_a2(const State<G>& st, c2* ex, int a, int c) {
  constexpr int T = G::T, P = G::P, W = G::W;
#pragma unroll
  for (int k1 = 0; k1 < P; ++k1) ex[(k1 * T + a) * W + c] = c2{st.zr[k1], st.zi[k1]};
}

template <class G>
KFBI_HD void group_k1(int g, int& kA, int& kB) {
  kA = g == 0 ? 0 : g;
  kB = g == 0 ? G::P / 2 : G::P - g;
}

// phase C: radix-8 DFTs over a for the thread's k1 groups
template <class G>
KFBI_HD void phase_c(State<G>& st, const c2* ex, int a, int c) {
  constexpr int T = G::T, W = G::W;
#pragma unroll
  for (int gi = 0; gi < G::GPT; ++gi) {
    const int g = a + T * gi;
    if (g >= G::NG) continue;
    int kA, kB;
    group_k1<G>(g, kA, kB);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const c2 pa = ex[(kA * T + u) * W + c];
      st.Ar[gi][u] = pa.x;
      st.Ai[gi][u] = pa.y;
      const c2 pb = ex[(kB * T + u) * W + c];
      st.Br[gi][u] = pb.x;
      st.Bi[gi][u] = pb.y;
    }
    Dft<8>::run(st.Ar[gi], st.Ai[gi]);
    Dft<8>::run(st.Br[gi], st.Bi[gi]);
  }
}

// Both split values of the pair Z_k = A, Z_{L-k} = B (w = e^{2 pi i k / N};
// the partner's w_{L-k} = -conj(w), so one complex product serves both),
// doubled: 2 I_k to row 2k (even output), 2 R_k to row 2k + 1 (scan input).
// |D| <= 2 sum |y_odd| and |S| <= 2 sum |y_even| stay below the full sum's
// bound, since a pair (j, N - j) has one parity.
template <class G>
KFBI_HD void split_store(ll* s, const cfx* sp, const Scale& sc, int k, ll Ar, ll Ai, ll Br, ll Bi, int c,
                         bool both) {
  constexpr int RS = G::RS, L = G::L;
  double* sd = reinterpret_cast<double*>(s);
  const ll Sr = Ar + Br, Si = Ai - Bi;
  ll pr = Ar - Br, pi = Ai + Bi;
  // w (D_r + i D_i) = (wr Dr - wi Di) + i (wr Di + wi Dr)
  cmul62(pr, pi, sp[k]);
  sd[(2 * k) * RS + c] = from_fix(Si - pr, sc);
  s[(2 * k + 1) * RS + c] = Sr + pi;
  if (both) {
    const int kk = L - k;
    sd[(2 * kk) * RS + c] = from_fix(-(Si + pr), sc);
    s[(2 * kk + 1) * RS + c] = Sr - pi;
  }
}

// phase D: real-DFT split of the owned pairs (after a barrier)
template <class G>
KFBI_HD void phase_d(const State<G>& st, ll* s, const cfx* sp, int a, int c) {
  constexpr int T = G::T, P = G::P, RS = G::RS;
#pragma unroll
  for (int gi = 0; gi < G::GPT; ++gi) {
    const int g = a + T * gi;
    if (g >= G::NG) continue;
    int kA, kB;
    group_k1<G>(g, kA, kB);
    if (g == 0) {
      s[c] = 0;
      s[RS + c] = st.Ar[gi][0] + st.Ai[gi][0];  // 2 F_1 = R_0
#pragma unroll
      for (int k2 = 1; k2 <= 4; ++k2)
        split_store<G>(s, sp, st.sc, P * k2, st.Ar[gi][k2], st.Ai[gi][k2], st.Ar[gi][8 - k2], st.Ai[gi][8 - k2], c,
                       k2 < 4);
      // k1 = P/2: k = P/2 + P k2 pairs with P/2 + P (7 - k2)
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2)
        split_store<G>(s, sp, st.sc, kB + P * k2, st.Br[gi][k2], st.Bi[gi][k2], st.Br[gi][7 - k2], st.Bi[gi][7 - k2],
                       c, true);
    } else {
#pragma unroll
      for (int k2 = 0; k2 < 8; ++k2)
        split_store<G>(s, sp, st.sc, kA + P * k2, st.Ar[gi][k2], st.Ai[gi][k2], st.Br[gi][7 - k2], st.Bi[gi][7 - k2],
                       c, true);
    }
  }
}

// phase E1: inclusive sums of the warp's segment of R_k (rows 2k + 1)
template <class G>
KFBI_HD void phase_e1(State<G>& st, const ll* s, ll* tot, int a, int c) {
  constexpr int P = G::P, RS = G::RS, W = G::W;
  ll acc = 0;
#pragma unroll
  for (int i = 0; i < P; ++i) {
    acc += s[(2 * (a * P + i) + 1) * RS + c];
    st.v[i] = acc;
  }
  tot[a * W + c] = acc;
}

// phase E2: the preceding segments' totals added, odd outputs written
template <class G>
KFBI_HD void phase_e2(const State<G>& st, ll* s, const ll* tot, int a, int c) {
  constexpr int P = G::P, RS = G::RS, W = G::W;
  double* sd = reinterpret_cast<double*>(s);
  ll off = 0;
  for (int b = 0; b < a; ++b) off += tot[b * W + c];
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const int j = 2 * (a * P + i) + 1;
    sd[j * RS + c] = from_fix(st.v[i] + off, st.sc);
  }
}

// phase F (columns with huge values only): the outputs' missing factor
template <class G>
KFBI_HD void phase_f(const State<G>& st, double* s, int a, int c) {
  if (st.sc.huge)
    for (int j = a; j < G::N; j += G::T) s[j * G::RS + c] *= HUGE_STEP;
}

// words of shared memory (8 bytes each) besides the tile: split twiddles and
// level twiddles (N/2 entries of 2 words each), sines (N/2), exponent maxima
// and column sums (128 each), scan totals (256)
template <int N>
constexpr size_t table_words() {
  return 2 * (size_t)N + N / 2 + 128 + 128 + 256;
}

// entry i < N/2 of the three tables from the float64 table tw[j] = e^{i pi j / N}
template <int N>
KFBI_HD void table_entry(int i, const double* tw, cfx* sp, cfx* lv, fx* sinv) {
  constexpr int P = N / 16;
  sp[i] = cfx{fx_table(tw[4 * i], 62), fx_table(tw[4 * i + 1], 62)};
  const int j = 4 * (i / P) * (i % P);  // lv[a][k1], i = a P + k1: e^{2 pi i a k1 / L}
  lv[i] = cfx{fx_table(tw[2 * j], 62), fx_table(tw[2 * j + 1], 62)};
  sinv[i] = fx_table(tw[2 * i + 1], 63);
}

#ifdef __CUDACC__
template <int N>
__device__ __forceinline__ void load_tables(ll* mem, const double* tw_g) {
  cfx* sp = reinterpret_cast<cfx*>(mem);
  for (int i = threadIdx.x; i < N / 2; i += 256)
    table_entry<N>(i, tw_g, sp, sp + N / 2, reinterpret_cast<fx*>(mem + 2 * N));
}

// The whole transform of the tile s[N][RS] (rows 1..N-1 in and out; row 0
// becomes 0) by 256 threads; mem: the tables and scratch.  Ends with a
// barrier.
template <class G>
__device__ __forceinline__ void dst1_tile_fix(double* sd, ll* mem) {
  constexpr int N = G::N;
  const int a = threadIdx.x >> 5, c = threadIdx.x & 31;
  ll* s = reinterpret_cast<ll*>(sd);
  const cfx* sp = reinterpret_cast<const cfx*>(mem);
  const fx* sinv = reinterpret_cast<const fx*>(mem + 2 * N);
  int* mx = reinterpret_cast<int*>(mem + 2 * N + N / 2);
  uint32_t* sm = reinterpret_cast<uint32_t*>(mem + 2 * N + N / 2 + 128);
  ll* tot = mem + 2 * N + N / 2 + 256;
  State<G> st;
  c2* ex = reinterpret_cast<c2*>(s);
  phase_0<G>(st, sd, mx, a, c);
  __syncthreads();
  phase_s<G>(st, mx, sm, a, c);
  __syncthreads();
  phase_1<G>(st, s, sm, sinv, a, c);
  __syncthreads();
  phase_a1<G>(st, s, sp, sp + N / 2, a, c);
  __syncthreads();
  phase_a2<G>(st, ex, a, c);
  __syncthreads();
  phase_c<G>(st, ex, a, c);
  __syncthreads();
  phase_d<G>(st, s, sp, a, c);
  __syncthreads();
  phase_e1<G>(st, s, tot, a, c);
  __syncthreads();
  phase_e2<G>(st, s, tot, a, c);
  if (__syncthreads_or(st.sc.huge)) {
    phase_f<G>(st, sd, a, c);
    __syncthreads();
  }
}
#endif

}  // namespace fixdst
}  // namespace kfbi
