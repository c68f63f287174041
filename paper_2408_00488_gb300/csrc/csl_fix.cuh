// FP64-accurate sine transform of one line in 64-bit block fixed point.
//
// GB300 issues FP64 at 2 lanes per SM and clock (measured 1.6 to 2, one
// dependent operation every 67 clocks) but 64-bit integer sums at about 41 and
// 32 x 32 -> 64 bit products at 60, so an FFT in FP64 arithmetic is bound by
// that one pipe.  Here the line is scaled by one power of two, held as 64-bit
// integers, and transformed with integer butterflies.  Sums are exact; a
// product is rounded once.
//
// The algorithm is that of csl_fft.cuh (one length-N complex FFT per line,
// y_j = h_j (z_j + z_{N-j}) + (z_j - z_{N-j})/4, the C / S split and the
// prefix sum), as a Stockham FFT with radices R0 .. R3.
//
// Scales.  E = largest exponent of the line, so |re|, |im| < 2^(E-1022).  A
// value is held in units of 2^(E-1022-S1+t); t = 0 at the start and grows by
// the shifts to the right.  The magnitude of a complex value stays below
// 2^62.5, so nothing overflows for any input.  The rounding of the early passes
// is amplified by the later ones, and the prefix sum adds up the errors of N/2
// modes, so a coarse unit there shows where the line's norm is little more than
// its largest entry (a point source over a small background).
//   N <= 1024  S1 is the finest unit at which pass 1 cannot overflow; the later
//     passes shift while the twiddle is applied, only as far as needed: every
//     value of pass p is bounded by both sqrt(2) max|z| R0..Rp and by the line's
//     sum of |re| + |im| (the bound of every partial DFT sum, and of the result:
//     sum_j |y_j| <= sum_j |z_j| because max(s_j, 1/2) <= 1).
//   N >= 2048, staged (FixStaged)  these bounds are too coarse: with S1 of pass 1
//     a spike over a background of 10^-3 at N = 4096 had 14 times the error of
//     FP64 butterflies.  Here every pass starts with the line's largest value, as
//     measured after the pass before, just below 2^60, which leaves headroom for
//     two radix-2 stages, and a radix of 8 or 16 drops one or two bits after the
//     second one, unless the line's sum bounds the rest.
// The split and the prefix sum only add, modulo 2^64, and their results fit.
//
// Measured on a GB300, FP64 form, per iteration of MINRES, FP64 arithmetic and
// this (with the lanes of fix_lanes and the tables in the L1): n = 1023 in 2D, x
// pass with the Lanczos step 124.6 and 33.4 us, MID pass 252.5 and 69.1, inverse
// x pass 119.0 and 27.9, whole iteration 524 and 168; n = 63, 71 and 35 us;
// n = 127 in 3D 1067 and 360; n = 4095 9297 and 2680.  Error of one
// line against 64-bit mantissas or more, over that of FP64 butterflies with the
// same split and scan, root mean square over 96 lines of a kind (random, constant,
// alternating, one to eight spikes anywhere or at N/2 and N/4 over random and
// constant backgrounds of 10^-8 to 0.1, the modes of such lines;
// tests/fixed_point_host.cu): at most 0.2 for N <= 256, 0.3 at 512, 0.5 at 1024, 0.4
// at 2048, 0.7 at 4096 and 8192; random and constant lines 0.1 to 0.2.  A single
// line can come out either way.  What bounds the time is latency: at n = 1023 14
// warps per SM (the registers allow 16) keep the ALU 33 to 37% busy and issue in 38
// to 41% of the cycles.
//
// A line with an infinity or NaN returns NaN everywhere (the FP64 butterflies
// spread it over the line too); a zero line returns zeros.
#pragma once
#include "csl_common.cuh"

#include <climits>

namespace csl {

typedef longlong2 fx2;  // (re, im)
typedef int4 fxw;       // twiddle: signed 32-bit digits re_hi, re_lo, im_hi, im_lo (value hi 2^32 + lo)

// fractional bits of the twiddle tables: products are taken back by
// kFxTw + sh <= 64 bits, i.e. one 32-bit funnel shift by kFxTw - 32 + sh <= 32
constexpr int kFxTw = 61;
constexpr int kFxMaxShift = 3;
constexpr int kFxMaxLeft = 20;

// ---- constants -----------------------------------------------------------------
__host__ __device__ constexpr unsigned long long fx_mulhi(unsigned long long a, unsigned long long b) {
  const unsigned long long al = a & 0xffffffffull, ah = a >> 32, bl = b & 0xffffffffull, bh = b >> 32;
  const unsigned long long t = al * bl, u = ah * bl + (t >> 32), v = al * bh + (u & 0xffffffffull);
  return ah * bh + (u >> 32) + (v >> 32);
}

struct FxRoot {
  long long c, s;  // cos, sin with 62 fractional bits
};

// cos and sin of 2 pi num / den (den a power of two, 0 <= num < den) to within
// a few units of 2^-62: reduction to [0, pi/4] by exact symmetries, then the
// Taylor series by Horner's rule in fixed point (the first term left out is
// (pi/4)^20 / 20! < 2^-67).
__host__ __device__ constexpr FxRoot fx_root(int num, int den) {
  long long n = num, d = den;
  int ld = 0;
  while (d < 8) {
    n *= 2;
    d *= 2;
  }
  while ((1ll << ld) < d) ++ld;
  const int quad = (int)(n / (d / 4));
  long long r = n - quad * (d / 4);
  const bool swap = r > d / 8;
  if (swap) r = d / 4 - r;
  const unsigned long long pi61 = 0x6487ED5110B4611Aull;  // pi 2^61
  const unsigned long long one = 1ull << 62;
  const unsigned long long th = fx_mulhi(pi61, (unsigned long long)r << (66 - ld));  // 2 pi r / d, 62 fractional bits
  const unsigned long long u = fx_mulhi(th << 1, th << 1);
  unsigned long long vc = one, vs = one;
#pragma unroll
  for (int k = 18; k >= 2; k -= 2) {
    vc = one - fx_mulhi(u << 1, vc << 1) / (unsigned long long)(k * (k - 1));
    vs = one - fx_mulhi(u << 1, vs << 1) / (unsigned long long)(k * (k + 1));
  }
  vs = fx_mulhi(th << 1, vs << 1);
  long long c = (long long)(swap ? vs : vc), s = (long long)(swap ? vc : vs);
  // quadrant: multiply by i^quad
  for (int i = 0; i < quad; ++i) {
    const long long t = c;
    c = -s;
    s = t;
  }
  return {c, s};
}

// a value as two signed 32-bit digits (hi 2^32 + lo); lo = INT_MIN, which has
// no negative, is moved by one unit
struct FxDigits {
  int h, l;
};
__host__ __device__ constexpr FxDigits fx_digits(long long v) {
  int l = (int)(unsigned)(unsigned long long)v;
  if (l == INT_MIN) {
    v += 1;
    l += 1;
  }
  return {(int)((v - l) >> 32), l};
}
// drop the last 62 - bits fractional bits, rounded
__host__ __device__ constexpr long long fx_quant(long long v, int bits) {
  return bits == 62 ? v : (v + (1ll << (61 - bits))) >> (62 - bits);
}
// exp(-2 pi i num/den) as a table entry
__host__ __device__ inline fxw fx_twiddle(long num, long den) {
  const FxRoot r = fx_root((int)(num % den), (int)den);
  const FxDigits c = fx_digits(fx_quant(r.c, kFxTw)), s = fx_digits(fx_quant(-r.s, kFxTw));
  fxw w;
  w.x = c.h;
  w.y = c.l;
  w.z = s.h;
  w.w = s.l;
  return w;
}
// sin(pi j / N) / 2, j <= N/2, as a table entry with 62 fractional bits
__host__ __device__ inline int2 fx_half_sine(int j, int N) {
  const FxDigits s = fx_digits(fx_root(j, 2 * N).s >> 1);
  int2 r;
  r.x = s.h;
  r.y = s.l;
  return r;
}

// ---- arithmetic ----------------------------------------------------------------
__host__ __device__ __forceinline__ int fx_lo(long long v) { return (int)(unsigned)(unsigned long long)v; }
// high signed digit: v = fx_hi(v) 2^32 + fx_lo(v)
__host__ __device__ __forceinline__ int fx_hi(long long v) {
  return (int)(v >> 32) + (int)((unsigned)(unsigned long long)v >> 31);
}
__host__ __device__ __forceinline__ long long fx_wide(int a, int b) { return (long long)a * (long long)b; }

// (acc 2^32 + low word of mid) >> s, s <= 32
__host__ __device__ __forceinline__ long long fx_take(long long acc, long long mid, unsigned s) {
#ifdef __CUDA_ARCH__
  const unsigned m = (unsigned)mid, al = (unsigned)acc, ah = (unsigned)(acc >> 32);
  const unsigned lo = __funnelshift_rc(m, al, s), hi = __funnelshift_rc(al, ah, s);
  return (long long)(((unsigned long long)hi << 32) | lo);
#else
  const unsigned m = (unsigned)mid;
  if (s == 32) return acc;
  return (long long)(((unsigned long long)acc << (32 - s)) | (m >> s));
#endif
}

// v * w for real v and a constant of F fractional bits (digits h, l), rounded.
// LOW: with the product of the two low digits, at most 2^(62-F) units.  The half
// sines of long lines take it: the error of a spike over 10^-3 is 0.7 times that
// without at N = 8192, 0.8 at 1024.  At 512, where it is a third of FP64's anyway, it
// cost the 3D P^-1 2%; for the diagonal roots (F = 63) it made no difference.
template <int F, bool LOW = false>
__host__ __device__ __forceinline__ long long fx_rmul(long long v, int h, int l) {
  const int vh = fx_hi(v), vl = fx_lo(v);
  long long mid = (1ll << (F - 33)) + fx_wide(vh, l) + fx_wide(vl, h);
  if (LOW) mid += fx_wide(vl, l) >> 32;
  return fx_take(fx_wide(vh, h) + (mid >> 32), mid, F - 32);
}

// w * v / 2^(32 + s), rounded; rnd = 2^(s-1).  LOW: with the products of the low
// digits, up to 2^(31-s) units.  The tables' twiddles change from lane to lane and
// go without; the constants inside a radix 16 would repeat the same error over all
// of a pass, which the prefix sum adds up (the modes of a spike at N/2, N = 8192:
// 1.5 times the error of FP64 butterflies without, 0.5 with).
template <bool LOW = false>
__host__ __device__ __forceinline__ fx2 fx_cmul(const fxw& w, fx2 v, unsigned s, long long rnd) {
  const int xh = fx_hi(v.x), xl = fx_lo(v.x), yh = fx_hi(v.y), yl = fx_lo(v.y);
  const int nh = -w.z, nl = -w.w;
  long long mr = rnd, mi = rnd;
  if constexpr (LOW) {
    mr += (fx_wide(xl, w.y) + fx_wide(yl, nl)) >> 32;
    mi += (fx_wide(xl, w.w) + fx_wide(yl, w.y)) >> 32;
  }
  mr += fx_wide(xh, w.y) + fx_wide(xl, w.x) + fx_wide(yh, nl) + fx_wide(yl, nh);
  mi += fx_wide(xh, w.w) + fx_wide(xl, w.z) + fx_wide(yh, w.y) + fx_wide(yl, w.x);
  fx2 r;
  r.x = fx_take((mr >> 32) + fx_wide(xh, w.x) + fx_wide(yh, nh), mr, s);
  r.y = fx_take((mi >> 32) + fx_wide(xh, w.z) + fx_wide(yh, w.x), mi, s);
  return r;
}

// v / 2^sh, ties to even: a few bits are dropped, so ties are frequent, and
// the prefix sum would add up the bias of rounding them one way
__host__ __device__ __forceinline__ long long fx_shift(long long v, unsigned sh) {
  const long long half = (1ll << sh) >> 1;
  return (v + (sh ? half - 1 + ((v >> sh) & 1) : 0)) >> sh;
}

// v / 2^sh for either sign of sh; a shift to the left must fit
__host__ __device__ __forceinline__ long long fx_rescale(long long v, int sh) {
  return sh >= 0 ? fx_shift(v, (unsigned)sh) : (long long)((unsigned long long)v << -sh);
}

__host__ __device__ __forceinline__ fx2 fx_add(fx2 a, fx2 b) {
  a.x += b.x;
  a.y += b.y;
  return a;
}
__host__ __device__ __forceinline__ fx2 fx_sub(fx2 a, fx2 b) {
  a.x -= b.x;
  a.y -= b.y;
  return a;
}

// v * exp(-2 pi i K / R), the trivial and the diagonal roots without the
// general product
template <int K, int R>
__host__ __device__ __forceinline__ fx2 fx_rotate(fx2 v) {
  constexpr FxRoot root = fx_root(K, R);
  fx2 r;
  if constexpr (K == 0) {
    r = v;
  } else if constexpr (4 * K == R) {  // -i
    r.x = v.y;
    r.y = -v.x;
  } else if constexpr (8 * K == R || 8 * K == 3 * R) {  // (+-1 - i) / sqrt 2
    constexpr long long c63 = fx_root(1, 8).c << 1;
    constexpr FxDigits c = fx_digits(c63);
    const long long a = fx_rmul<63>(v.x + v.y, c.h, c.l), b = fx_rmul<63>(v.y - v.x, c.h, c.l);
    if constexpr (8 * K == R) {
      r.x = a;
      r.y = b;
    } else {
      r.x = b;
      r.y = -a;
    }
  } else {
    constexpr FxDigits c = fx_digits(root.c), s = fx_digits(-root.s);
    fxw w;
    w.x = c.h;
    w.y = c.l;
    w.z = s.h;
    w.w = s.l;
    r = fx_cmul<true>(w, v, 30, 1ll << 29);
  }
  return r;
}

// Butterflies of the radix-2 stage with half-length S, index K.  HEAD: there is
// headroom for two stages; before the third, `drop` bits of every value go.
template <int S, int K, int R, bool HEAD>
struct FxStage {
  static __host__ __device__ __forceinline__ void run(fx2 (&x)[R], unsigned drop) {
    if constexpr (HEAD && S == 4 && K == 0) {
      if (drop) {
#pragma unroll
        for (int i = 0; i < R; ++i) {
          x[i].x = fx_shift(x[i].x, drop);
          x[i].y = fx_shift(x[i].y, drop);
        }
      }
    }
#pragma unroll
    for (int b = 0; b < R; b += 2 * S) {
      const fx2 u = x[b + K], t = fx_rotate<K, 2 * S>(x[b + K + S]);
      x[b + K] = fx_add(u, t);
      x[b + K + S] = fx_sub(u, t);
    }
    if constexpr (K + 1 < S)
      FxStage<S, K + 1, R, HEAD>::run(x, drop);
    else if constexpr (2 * S < R)
      FxStage<2 * S, 0, R, HEAD>::run(x, drop);
  }
};

// in-register forward DFT of length R, natural order in and out
template <int R, bool HEAD = false>
__host__ __device__ __forceinline__ void fx_dft(fx2 (&x)[R], unsigned drop = 0) {
#pragma unroll
  for (int i = 0; i < R; ++i) {
    int j = 0;
#pragma unroll
    for (int b = 1; b < R; b <<= 1) j = (j << 1) | ((i & b) ? 1 : 0);
    if (j > i) {
      const fx2 t = x[i];
      x[i] = x[j];
      x[j] = t;
    }
  }
  FxStage<1, 0, R, HEAD>::run(x, drop);
}

// ---- conversions -----------------------------------------------------------------
__host__ __device__ __forceinline__ unsigned fx_dhi(double v) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2hiint(v);
#else
  unsigned long long b;
  __builtin_memcpy(&b, &v, 8);
  return (unsigned)(b >> 32);
#endif
}
__host__ __device__ __forceinline__ unsigned fx_dlo(double v) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2loint(v);
#else
  unsigned long long b;
  __builtin_memcpy(&b, &v, 8);
  return (unsigned)b;
#endif
}

// v as an integer multiple of 2^(E - 1022 - S1), truncated; E >= 1 is at least
// v's exponent field.  mag: |result| >> 32.
template <int S1>
__host__ __device__ __forceinline__ long long fx_from_double(double v, int E, unsigned& mag) {
  const unsigned hi = fx_dhi(v), lo = fx_dlo(v);
  const int e = (int)((hi >> 20) & 0x7ffu);
  const unsigned mh = (hi & 0xfffffu) | (e > 0 ? 0x100000u : 0u);  // subnormals have no leading one
  int d = E - (e > 0 ? e : 1);
  d = d > 63 ? 63 : d;
  unsigned long long m = (((unsigned long long)mh << 32) | lo) << (S1 - 53);
  m >>= d;
  mag = (unsigned)(m >> 32);
  return (hi >> 31) ? -(long long)m : (long long)m;
}

// d * 2^q for the few q at which the result could leave the normal range
static __device__ __noinline__ double fx_scale_far(double d, int q) { return scalbn(d, q); }

// v * 2^q.  The hardware conversion rounds to nearest (one FP64-pipe
// operation); the exponent is added with integer instructions.  The far case
// (zero lines, and lines near the ends of the range) stays a call: inlined, its
// products would be issued on the FP64 pipe for every value and discarded.
__device__ __forceinline__ double fx_to_double(long long v, int q) {
  const double d = __ll2double_rn(v);
  if (q < -1000 || q > 900) return fx_scale_far(d, q);
  const int hi = __double2hiint(d);
  return __hiloint2double(v == 0 ? hi : hi + (q << 20), __double2loint(d));
}

// ---- shapes ----------------------------------------------------------------------
// Lanes per line and radices.  One lane's values are a long serial chain on few
// warps, so a line takes as many lanes as leave each 4 to 8 values (16 at most):
// n = 63, 16 lanes instead of 8, iteration 48.8 -> 34.6 us; n = 127, 32 instead
// of 8, 77.8 -> 30.9; n = 31, 8 instead of 4, 48 -> 34.5.  N = 128 and 256 have
// two variants: with many lines, as in 3D, fewer lanes and passes win (n = 127
// in 3D 357 us with 16 lanes, 370 with 32, 384 with 8).  N = 512 and 1024: 64
// lanes (variant 1, and 0, which has no kernels of its own) or 128 (variant 2).
// A large first radix costs bits of S1, which shows with a spike over a small
// background: with 16 instead of 8 at N = 1024 a spike at N/2 over 10^-3 had 1.1
// times the error of FP64 butterflies (now 0.5), with 8 instead of 4 at 8192 a
// spike anywhere over it 0.9 times (0.6).
__host__ __device__ constexpr int fix_lanes(int N, int variant) {
  return N <= 8 ? 1 : N == 16 ? 4 : N == 32 ? 8 : N == 64 ? 16 : N == 128 ? (variant ? 32 : 16)
         : N == 256 ? (variant ? 64 : 32) : N <= 1024 ? (variant == 2 ? 128 : 64) : N <= 4096 ? 256 : 512;
}
template <int N, int TPL> struct FixShape;
template <> struct FixShape<16, 4> { enum { NP = 2, R0 = 4, R1 = 4, R2 = 1, R3 = 1 }; };
template <> struct FixShape<32, 8> { enum { NP = 3, R0 = 4, R1 = 4, R2 = 2, R3 = 1 }; };
template <> struct FixShape<64, 16> { enum { NP = 3, R0 = 4, R1 = 4, R2 = 4, R3 = 1 }; };
template <> struct FixShape<128, 16> { enum { NP = 3, R0 = 8, R1 = 4, R2 = 4, R3 = 1 }; };
template <> struct FixShape<128, 32> { enum { NP = 3, R0 = 8, R1 = 4, R2 = 4, R3 = 1 }; };
template <> struct FixShape<256, 32> { enum { NP = 3, R0 = 8, R1 = 8, R2 = 4, R3 = 1 }; };
template <> struct FixShape<256, 64> { enum { NP = 4, R0 = 4, R1 = 4, R2 = 4, R3 = 4 }; };
template <> struct FixShape<512, 64> { enum { NP = 3, R0 = 8, R1 = 8, R2 = 8, R3 = 1 }; };
template <> struct FixShape<512, 128> { enum { NP = 4, R0 = 8, R1 = 4, R2 = 4, R3 = 4 }; };
template <> struct FixShape<1024, 64> { enum { NP = 3, R0 = 8, R1 = 8, R2 = 16, R3 = 1 }; };
template <> struct FixShape<1024, 128> { enum { NP = 4, R0 = 8, R1 = 8, R2 = 4, R3 = 4 }; };
template <> struct FixShape<2048, 256> { enum { NP = 4, R0 = 8, R1 = 8, R2 = 8, R3 = 4 }; };
template <> struct FixShape<4096, 256> { enum { NP = 3, R0 = 16, R1 = 16, R2 = 16, R3 = 1 }; };
template <> struct FixShape<8192, 512> { enum { NP = 4, R0 = 4, R1 = 8, R2 = 16, R3 = 16 }; };

__host__ __device__ constexpr int fx_log2(int v) {
  int l = 0;
  while ((1 << l) < v) ++l;
  return l;
}

// the scale plan of a line of up to 1024 points: S1 and the shifts
template <int R0, int R1, int R2, int R3>
struct FixScale {
  enum { W0 = fx_log2(R0), W1 = fx_log2(R1), W2 = fx_log2(R2), W3 = fx_log2(R3), S1 = 62 - W0 };
  // right shift, in all, of the values that enter pass p = 1 .. NP-1 (and are
  // twiddled there); 2^lb bounds the line's sum of |re| + |im| at the scale of
  // S1.  A pass shifts by at most kFxMaxShift, so a pass before the last takes
  // more than its own bound asks for where the later ones could not.  A last
  // radix of 16 can need one bit more: it drops that one after two stages.
  template <int NP>
  static __host__ __device__ __forceinline__ int shift_at(int p, int lb) {
    int all = S1 + W0 + W1 + W2 + W3, own = S1 + W0 + W1 + (p >= 2 ? W2 : 0) + (p >= 3 ? W3 : 0);
    all = (all < lb ? all : lb) - 62;
    own = (own < lb ? own : lb) - 62;
    const int rest = all - kFxMaxShift * (NP - 1 - p) - (p < NP - 1 && W2 > 3);
    own = own > rest ? own : rest;
    return own > 0 ? own : 0;
  }
  // every shift and drop is within its limit
  static constexpr bool kFits = W1 <= 3 && W2 <= (R3 > 1 ? 3 : 4) && W3 <= 3;
};

// The scale plan of a staged line.  |re|, |im| < 2^60 at the start of a pass, so
// |z| < 2^60.5, 2^62.5 after two radix-2 stages, and below 2^62.5 again after all
// four of a radix 16 that drops two bits in between.  The line's sum bounds every
// value by 2^(lb-t), so from t = need on, where that is 2^62, nothing has to be
// shifted any more; and t must end there, for the results' sake.
template <int R0, int R1, int R2, int R3>
struct FixStaged {
  enum { S1 = 60, NEED = fx_log2(R0) + fx_log2(R1) + fx_log2(R2) + fx_log2(R3) + S1 - 62 };
  // a component of the results is at most N 2^S1 2^-t: NEED is always enough
  static __host__ __device__ __forceinline__ int need(int lb) {
    const int n = lb - 62 < (int)NEED ? lb - 62 : (int)NEED;
    return n > 0 ? n : 0;
  }
  // bits that radix r drops at most
  static __host__ __device__ constexpr int head(int r) { return r >= 8 ? fx_log2(r) - 2 : 0; }
  static __host__ __device__ __forceinline__ int drop(int r, int need, int t) {
    const int d = need - t;
    return d < 0 ? 0 : d < head(r) ? d : head(r);
  }
  // shift at the start of pass p = 1 .. NP-1, by -kFxMaxLeft to kFxMaxShift bits;
  // top: OR of the high words of the values' magnitudes.  The last line: what the
  // passes after this one's start could not make up for.
  template <int NP>
  static __host__ __device__ __forceinline__ int entry(int p, int need, int t, unsigned top) {
#ifdef __CUDA_ARCH__
    int sh = 64 - __clz((int)top) - 60;
#else
    int sh = (top ? 64 - __builtin_clz(top) : 32) - 60;
#endif
    sh = sh < need - t ? sh : need - t;
    sh = sh > -kFxMaxLeft ? sh : -kFxMaxLeft;
    const int later = kFxMaxShift * (NP - 1 - p) + head(R3) + (p <= 2 ? head(R2) : 0) + (p <= 1 ? head(R1) : 0);
    const int least = need - t - later;
    return sh > least ? sh : least;
  }
  // the passes together can always reach `need`
  static constexpr bool kFits =
      kFxMaxShift * ((R1 > 1) + (R2 > 1) + (R3 > 1)) + head(R0) + head(R1) + head(R2) + head(R3) >= (int)NEED;
};
// high word of |v| (of -v - 1 below zero)
__host__ __device__ __forceinline__ unsigned fx_top(long long v) {
  const int h = (int)(v >> 32);
  return (unsigned)(h ^ (h >> 31));
}
__host__ __device__ constexpr bool fix_staged(int N) { return N >= 2048; }

// entries of the pass tables [q][k] = w_{Ls r}^{q k}, passes 2 .. NP
template <typename S>
__host__ __device__ constexpr int fix_tp_entries() {
  return (int)S::R0 * S::R1 + (S::NP > 2 ? (int)S::R0 * S::R1 * S::R2 : 0) +
         (S::NP > 3 ? (int)S::R0 * S::R1 * S::R2 * S::R3 : 0);
}

// padded position of line element i: one slot per 8, so that lanes 8 elements
// apart (the first pass's stores, the chunks of the scan) hit distinct banks
__host__ __device__ constexpr int fpad(int i) { return i + (i >> 3); }
// fpad(base + q step), the step's part folded into a constant where it is a multiple of 8
template <int STEP>
__host__ __device__ __forceinline__ int fpad_step(int base, int q) {
  return STEP % 8 == 0 ? fpad(base) + q * (STEP + STEP / 8) : fpad(base + q * STEP);
}

// ---- one line in shared memory ------------------------------------------------------
__device__ __forceinline__ void fx_line_sync(int tpl) {
  if (tpl <= 32) {
    __syncwarp();
  } else if (tpl >= 256) {
    __syncthreads();
  } else {  // the lanes of one line only; barrier 0 is the CTA's
    asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)(threadIdx.x / tpl)), "r"(tpl) : "memory");
  }
}

// identity epilogue of FixLine::run
struct FixNoPost {
  __device__ __forceinline__ void start() {}
  __device__ __forceinline__ double2 operator()(int, double2 v) { return v; }
};

template <int N, int TPL>
struct FixLine {
  typedef FixShape<N, TPL> S;
  typedef FixScale<S::R0, S::R1, S::R2, S::R3> SC;
  typedef FixStaged<S::R0, S::R1, S::R2, S::R3> ST;
  static constexpr bool kStaged = fix_staged(N), kLow = N >= 1024;
  static_assert(kStaged ? (bool)ST::kFits : (bool)SC::kFits, "shifts");
  enum { NL = N / TPL, H = N / 2, CH = H / TPL, NW = TPL / 32, S1 = kStaged ? (int)ST::S1 : (int)SC::S1,
         // bits dropped from the magnitudes' high words so that their sum over
         // the line fits in 32 bits
         G = (S1 - 32) + fx_log2(2 * N) - 31 > 0 ? (S1 - 32) + fx_log2(2 * N) - 31 : 0 };
  // largest value over the line's lanes; slot: NW words of scratch
  static __device__ __forceinline__ unsigned line_max(unsigned v, unsigned* slot, int t) {
    if constexpr (TPL >= 32) {
      v = __reduce_max_sync(0xffffffffu, v);
    } else {
#pragma unroll
      for (int d = 1; d < TPL; d <<= 1) {
        const unsigned o = __shfl_xor_sync(0xffffffffu, v, d, TPL);
        v = v > o ? v : o;
      }
    }
    if constexpr (TPL > 32) {
      if ((t & 31) == 0) slot[t >> 5] = v;
      fx_line_sync(TPL);
#pragma unroll
      for (int w = 0; w < NW; ++w) v = v > slot[w] ? v : slot[w];
    } else {
      __syncwarp();
    }
    return v;
  }

  // OR over the line's warps of what a pass left in their slots
  static __device__ __forceinline__ unsigned line_or(const unsigned* slot) {
    unsigned v = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) v |= slot[w];
    return v;
  }

  // one pass; sh, drop: see FixScale and FixStaged.  TOP: leaves the OR of fx_top
  // over the results in slot, one word a warp.
  template <int R, int LSP, bool FIRST, bool TOP = false>
  static __device__ __forceinline__ void pass(fx2* a, int t, const fxw* tp, int sh, unsigned drop = 0,
                                              unsigned* slot = nullptr) {
    constexpr int GR = N / R, PER = (GR + TPL - 1) / TPL;
    const bool active = GR >= TPL || t < GR;  // a radix above N / TPL leaves lanes idle in its pass
    fx2 x[PER][R];
    const unsigned s = (unsigned)(kFxTw - 32 + sh);
    const long long rnd = 1ll << (s - 1);
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      if (!active) break;
      const int l = t + TPL * i, k = l & (LSP - 1);
#pragma unroll
      for (int q = 0; q < R; ++q) {
        fx2 v = a[fpad_step<GR>(l, q)];
        if constexpr (!FIRST) {
          if (q > 0) {
            // exact roots (k = 0) leave ties: rounded up and down in turn
            v = fx_cmul(tp[q * LSP + k], v, s, rnd - (q & 1));
          } else {
            v.x = kStaged ? fx_rescale(v.x, sh) : fx_shift(v.x, sh);
            v.y = kStaged ? fx_rescale(v.y, sh) : fx_shift(v.y, sh);
          }
        }
        x[i][q] = v;
      }
      fx_dft<R, kStaged || (!FIRST && R == 16)>(x[i], drop);
    }
    if constexpr (TOP) {
      static_assert(GR >= TPL && TPL >= 32, "every lane of the warp has values");
      unsigned top = 0;
#pragma unroll
      for (int i = 0; i < PER; ++i) {
#pragma unroll
        for (int q = 0; q < R; ++q) top |= fx_top(x[i][q].x) | fx_top(x[i][q].y);
      }
      top = __reduce_or_sync(0xffffffffu, top);
      if ((t & 31) == 0) slot[t >> 5] = top;
    }
    fx_line_sync(TPL);
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      if (!active) break;
      const int l = t + TPL * i, j = l / LSP, k = l & (LSP - 1);
#pragma unroll
      for (int q = 0; q < R; ++q)
        a[LSP == 1 && R % 8 == 0 ? fpad(j * R) + fpad(q) : fpad_step<LSP>(j * LSP * R + k, q)] = x[i][q];
    }
    fx_line_sync(TPL);
  }

  // lb: 2^lb bounds the line's sum of |re| + |im|; sum: its G-bit part, of the
  // lane's line (up to 32 lanes) or of each warp, in slot
  static __device__ __forceinline__ int sum_bits(const unsigned* slot, unsigned sum) {
    if constexpr (TPL > 32) {
      sum = 0;
#pragma unroll
      for (int w = 0; w < NW; ++w) sum += slot[w];
    }
    return 32 + G + 32 - __clz(sum + 2 * N);
  }

  // Unnormalised DST-I of the line (doubles at fpad(1) .. fpad(N-1)) in place.
  // scr: 2 max(NW, 4) 16-byte slots of the line.  post(m, value) is applied to
  // every result before it is stored (post.start() earlier, for its loads).
  // Every lane of the line must call it, and the line's input must be visible
  // to them.
  template <typename POST>
  static __device__ __forceinline__ void run(double2* line, int t, const int2* hs, const fxw* tp, void* scr,
                                             POST& post) {
    fx2* a = (fx2*)line;
    fx2* s_scan = (fx2*)scr;
    unsigned* s_max = (unsigned*)((char*)scr + 16 * NW);
    unsigned* s_sum = s_max + NW;
    int E;
    bool nonfinite;
    {  // ---- scale, pre-twiddle: the lane's pairs (m, N - m), m = 1 + t + TPL i
      double2 za[NL / 2], zb[NL / 2];
      unsigned mx = 0;
#pragma unroll
      for (int i = 0; i < NL / 2; ++i) {
        za[i] = line[fpad_step<TPL>(1 + t, i)];
        zb[i] = line[fpad_step<TPL>(N - 1 - t, -i)];
        const unsigned h0 = fx_dhi(za[i].x) & 0x7fffffffu, h1 = fx_dhi(za[i].y) & 0x7fffffffu;
        const unsigned h2 = fx_dhi(zb[i].x) & 0x7fffffffu, h3 = fx_dhi(zb[i].y) & 0x7fffffffu;
        mx = max(mx, max(max(h0, h1), max(h2, h3)));
      }
      mx = line_max(mx, s_max, t);
      E = (int)(mx >> 20);
      nonfinite = E == 0x7ff;
      E = E > 1 ? E : 1;
      unsigned sum = 0;
#pragma unroll
      for (int i = 0; i < NL / 2; ++i) {
        unsigned g0, g1, g2, g3;
        const fx2 u = {fx_from_double<S1>(za[i].x, E, g0), fx_from_double<S1>(za[i].y, E, g1)};
        const fx2 v = {fx_from_double<S1>(zb[i].x, E, g2), fx_from_double<S1>(zb[i].y, E, g3)};
        sum += ((g0 >> G) + (g1 >> G)) + ((g2 >> G) + (g3 >> G));
        const int2 h = hs[1 + t + TPL * i];
        const fx2 p = fx_add(u, v), d = fx_sub(u, v);
        const fx2 A = {fx_rmul<62, kLow>(p.x, h.x, h.y), fx_rmul<62, kLow>(p.y, h.x, h.y)};
        // the quarter, ties rounded up and down in turn
        const fx2 B = {(d.x + 1 + (i & 1)) >> 2, (d.y + 1 + (i & 1)) >> 2};
        a[fpad_step<TPL>(1 + t, i)] = fx_add(A, B);
        a[fpad_step<TPL>(N - 1 - t, -i)] = fx_sub(A, B);  // m = N/2: its own partner, B = 0
      }
      if (t == 0) a[0] = {0, 0};
      if constexpr (TPL >= 32) {
        sum = __reduce_add_sync(0xffffffffu, sum);
        if constexpr (TPL > 32) {
          if ((t & 31) == 0) s_sum[t >> 5] = sum;
        }
      } else {
#pragma unroll
        for (int d = 1; d < TPL; d <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d, TPL);
      }
      fx_line_sync(TPL);
      if constexpr (kStaged) {
        const int lb = sum_bits(s_sum, sum);
        const int need = ST::need(lb);
        int d = ST::drop(S::R0, need, 0), all = d, sh;
        pass<S::R0, 1, true, true>(a, t, tp, 0, d, s_max);
        sh = ST::template entry<S::NP>(1, need, all, line_or(s_max));
        d = ST::drop(S::R1, need, all + sh);
        all += sh + d;
        pass<S::R1, S::R0, false, true>(a, t, tp, sh, d, s_max);
        tp += S::R0 * S::R1;
        sh = ST::template entry<S::NP>(2, need, all, line_or(s_max));
        d = ST::drop(S::R2, need, all + sh);
        all += sh + d;
        pass<S::R2, S::R0 * S::R1, false, (S::NP > 3)>(a, t, tp, sh, d, s_max);
        if constexpr (S::NP > 3) {
          tp += S::R0 * S::R1 * S::R2;
          sh = ST::template entry<S::NP>(3, need, all, line_or(s_max));
          d = ST::drop(S::R3, need, all + sh);
          all += sh + d;
          pass<S::R3, S::R0 * S::R1 * S::R2, false>(a, t, tp, sh, d);
        }
        E += all;
      } else {
        pass<S::R0, 1, true>(a, t, tp, 0);
        const int lb = sum_bits(s_sum, sum);
        int t1 = 0, tn = SC::template shift_at<S::NP>(1, lb);
        pass<S::R1, S::R0, false>(a, t, tp, tn);
        if constexpr (S::NP > 2) {
          t1 = tn;
          tn = SC::template shift_at<S::NP>(2, lb);
          const int d = S::R2 == 16 && tn - t1 > kFxMaxShift ? 1 : 0;
          pass<S::R2, S::R0 * S::R1, false>(a, t, tp + S::R0 * S::R1, tn - t1 - d, d);
        }
        if constexpr (S::NP > 3) {
          t1 = tn;
          tn = SC::template shift_at<S::NP>(3, lb);
          pass<S::R3, S::R0 * S::R1 * S::R2, false>(a, t, tp + S::R0 * S::R1 + S::R0 * S::R1 * S::R2, tn - t1);
        }
        E += tn;
      }
    }
    post.start();
    // ---- split into C_k and S_k and prefix sum of C: the lane's chunk k = CH t + i
    const int q = E - 1022 - S1;  // results are multiples of 2^q
    fx2 cc[CH], ss[CH];
    fx2 tot = {0, 0};
#pragma unroll
    for (int i = 0; i < CH; ++i) {
      const int k = CH * t + i;
      const fx2 Yk = a[fpad(k)];
      fx2 Ym = {0, 0};
      if (i > 0 || t > 0) Ym = a[fpad(N - k)];
      tot = fx_add(tot, fx_add(Yk, Ym));
      cc[i] = tot;
      ss[i].x = Ym.y - Yk.y;
      ss[i].y = Yk.x - Ym.x;
    }
    fx2 inc = tot;
    const int lw = t & 31;
    constexpr int SW = TPL < 32 ? TPL : 32;
#pragma unroll
    for (int d = 1; d < SW; d <<= 1) {
      const long long ux = __shfl_up_sync(0xffffffffu, inc.x, d, SW), uy = __shfl_up_sync(0xffffffffu, inc.y, d, SW);
      if ((lw & (SW - 1)) >= d) {
        inc.x += ux;
        inc.y += uy;
      }
    }
    if constexpr (TPL > 32) {
      if (lw == 31) s_scan[t >> 5] = inc;
    }
    fx_line_sync(TPL);  // also: every read of Y precedes the stores below
    if constexpr (TPL > 32) {
      for (int w = 0; w < (t >> 5); ++w) inc = fx_add(inc, s_scan[w]);
    }
    const fx2 before = fx_sub(inc, tot);
    const double bad = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll
    for (int i = 0; i < CH; ++i) {
      const int k = CH * t + i;
      const fx2 o = fx_add(before, cc[i]);
      double2 vo = make_double2(fx_to_double(o.x, q), fx_to_double(o.y, q));
      double2 ve = make_double2(fx_to_double(ss[i].x, q), fx_to_double(ss[i].y, q));
      if (nonfinite) vo = ve = make_double2(bad, bad);
      if (i > 0 || t > 0) line[fpad(2 * k)] = post(2 * k, ve);
      line[fpad(2 * k + 1)] = post(2 * k + 1, vo);
    }
    fx_line_sync(TPL);
  }
};

// lines of 4 or 8 points: the whole line in one lane's registers
template <int N>
struct FixLine<N, 1> {
  enum { S1 = 62 - fx_log2(N) };
  template <typename POST>
  static __device__ __forceinline__ void run(double2* line, int, const int2* hs, const fxw*, void*, POST& post) {
    unsigned mx = 0;
#pragma unroll
    for (int j = 1; j < N; ++j) {
      const double2 z = line[fpad(j)];
      mx = max(mx, max(fx_dhi(z.x) & 0x7fffffffu, fx_dhi(z.y) & 0x7fffffffu));
    }
    int E = (int)(mx >> 20);
    const bool nonfinite = E == 0x7ff;
    E = E > 1 ? E : 1;
    fx2 x[N];
    x[0] = {0, 0};
#pragma unroll
    for (int j = 1; j <= N / 2; ++j) {
      unsigned g;
      const double2 za = line[fpad(j)], zb = line[fpad(N - j)];
      const fx2 u = {fx_from_double<S1>(za.x, E, g), fx_from_double<S1>(za.y, E, g)};
      const fx2 v = {fx_from_double<S1>(zb.x, E, g), fx_from_double<S1>(zb.y, E, g)};
      if (j == N / 2) {
        x[j] = u;
      } else {
        const int2 h = hs[j];
        const fx2 p = fx_add(u, v), d = fx_sub(u, v);
        const fx2 A = {fx_rmul<62>(p.x, h.x, h.y), fx_rmul<62>(p.y, h.x, h.y)};
        const fx2 B = {(d.x + 1 + (j & 1)) >> 2, (d.y + 1 + (j & 1)) >> 2};
        x[j] = fx_add(A, B);
        x[N - j] = fx_sub(A, B);
      }
    }
    fx_dft<N>(x);
    post.start();
    const int q = E - 1022 - S1;
    const double bad = __longlong_as_double(0x7ff8000000000000ll);
    fx2 sum = x[0];
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
      if (k > 0) {
        const fx2 Yk = x[k], Ym = x[N - k];
        sum = fx_add(sum, fx_add(Yk, Ym));
        double2 ve = make_double2(fx_to_double(Ym.y - Yk.y, q), fx_to_double(Yk.x - Ym.x, q));
        if (nonfinite) ve = make_double2(bad, bad);
        line[fpad(2 * k)] = post(2 * k, ve);
      }
      double2 vo = make_double2(fx_to_double(sum.x, q), fx_to_double(sum.y, q));
      if (nonfinite) vo = make_double2(bad, bad);
      line[fpad(2 * k + 1)] = post(2 * k + 1, vo);
    }
  }
};

// line stride in 16-byte slots: odd for short lines (one line per lane, or
// tiles of 8 and more columns), 2 mod 8 for long ones (tiles of 4 columns), so
// that column-wise tile copies spread over the banks
template <int N>
__host__ __device__ constexpr int fix_line_stride() {
  return N <= 256 ? fpad(N) | 1 : ((fpad(N) + 7) / 8) * 8 + 2;
}

// Pass table of the radices r[0 .. np-1], host or device: entry e of pass p is
// w_{Ls r_p}^{q k}, e = q Ls + k.
struct FixRadices {
  int np, r[4];
};
__host__ __device__ inline fxw fix_table_entry(const FixRadices& f, int e) {
  int ls = f.r[0];
  for (int p = 1; p < f.np; ++p) {
    const int n = ls * f.r[p];
    if (e < n) return fx_twiddle((long)(e / ls) * (e % ls), n);
    e -= n;
    ls = n;
  }
  return fxw{0, 0, 0, 0};
}
template <int N, int TPL>
__host__ __device__ constexpr FixRadices fix_radices() {
  typedef FixShape<N, TPL> S;
  return {S::NP, {S::R0, S::R1, S::R2, S::R3}};
}

}  // namespace csl
