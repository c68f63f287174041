// Host program of test_fixed_point_accuracy.py: the sine transform of one line
// with the fixed-point form's own functions (csl_fix.cuh), in the order in which
// FixLine::run applies them, and in FP64 butterflies (the same split of the
// modes and prefix sum, in chunks per lane as on the GPU), both against a long
// double FFT.  Prints, per length, lanes and kind of line,
//   N lanes kind rms_fixed rms_fp64 bad
// with the root mean square of the errors relative to the result's norm, and the
// number of values or shifts outside the documented limits.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <utility>
#include <vector>

#include "csl_fix.cuh"

using namespace csl;
typedef long double ld;
struct Cd { double x, y; };
struct Cl { ld x, y; };

static const ld kPi = 3.14159265358979323846264338327950288L;
static int g_bad = 0;

// exact transform: FFT of the odd extension (no amplification, 64 bits or more)
static std::vector<Cl> exact(const std::vector<Cd>& z) {
  const int N = (int)z.size(), M = 2 * N;
  std::vector<Cl> a(M, Cl{0, 0}), w(N);
  for (int i = 0; i < N; ++i) w[i] = {cosl(kPi * i / N), -sinl(kPi * i / N)};
  for (int j = 1; j < N; ++j) {
    a[j] = {z[j].x, z[j].y};
    a[M - j] = {-(ld)z[j].x, -(ld)z[j].y};
  }
  for (int i = 0, j = 0; i < M; ++i) {
    if (i < j) std::swap(a[i], a[j]);
    int m = M >> 1;
    while (m >= 1 && (j & m)) j ^= m, m >>= 1;
    j |= m;
  }
  for (int s = 1; s < M; s <<= 1)
    for (int b = 0; b < M; b += 2 * s)
      for (int k = 0; k < s; ++k) {
        const Cl ww = w[k * (N / s)], v = a[b + k + s], u = a[b + k];
        const Cl t = {ww.x * v.x - ww.y * v.y, ww.x * v.y + ww.y * v.x};
        a[b + k] = {u.x + t.x, u.y + t.y};
        a[b + k + s] = {u.x - t.x, u.y - t.y};
      }
  std::vector<Cl> o(N, Cl{0, 0});
  for (int k = 1; k < N; ++k) o[k] = {-a[k].y / 2, a[k].x / 2};
  return o;
}

// ---- FP64 butterflies
template <int R>
static void dft64(Cd* x, int N, const std::vector<Cd>& tw) {
  for (int i = 0; i < R; ++i) {
    int j = 0;
    for (int b = 1; b < R; b <<= 1) j = (j << 1) | ((i & b) ? 1 : 0);
    if (j > i) std::swap(x[i], x[j]);
  }
  for (int s = 1; s < R; s <<= 1)
    for (int k = 0; k < s; ++k) {
      const Cd w = tw[k * (N / (2 * s))];
      for (int b = 0; b < R; b += 2 * s) {
        const Cd u = x[b + k], v = x[b + k + s];
        const Cd t = k == 0 ? v : 2 * k == s ? Cd{v.y, -v.x}
                                             : Cd{fma(w.x, v.x, -w.y * v.y), fma(w.x, v.y, w.y * v.x)};
        x[b + k] = {u.x + t.x, u.y + t.y};
        x[b + k + s] = {u.x - t.x, u.y - t.y};
      }
    }
}
template <int R>
static void pass64(std::vector<Cd>& a, int Ls, const std::vector<Cd>& tw) {
  const int N = (int)a.size(), G = N / R;
  std::vector<Cd> o(N);
  for (int l = 0; l < G; ++l) {
    const int k = l % Ls, j = l / Ls;
    Cd x[R];
    for (int q = 0; q < R; ++q) {
      x[q] = a[l + q * G];
      if (q && Ls > 1) {
        const Cd v = x[q], w = tw[(long)q * k % (Ls * R) * (N / (Ls * R))];
        x[q] = {fma(w.x, v.x, -w.y * v.y), fma(w.x, v.y, w.y * v.x)};
      }
    }
    dft64<R>(x, N, tw);
    for (int s = 0; s < R; ++s) o[j * Ls * R + k + s * Ls] = x[s];
  }
  a = o;
}
static std::vector<Cd> fp64(const std::vector<Cd>& z, int lanes, const std::vector<int>& radices) {
  const int N = (int)z.size(), H = N / 2, CH = H / lanes, SW = lanes < 32 ? lanes : 32;
  std::vector<Cd> y(N), tw(N), out(N);
  for (int m = 0; m < N; ++m) tw[m] = {(double)cosl(2 * kPi * m / N), -(double)sinl(2 * kPi * m / N)};
  y[0] = {0, 0};
  for (int j = 1; j < N; ++j) {
    const Cd a = z[j], b = z[N - j];
    const double h = 0.5 * sin(M_PI * (j < N - j ? j : N - j) / N);
    y[j] = {fma(h, a.x + b.x, (a.x - b.x) * 0.25), fma(h, a.y + b.y, (a.y - b.y) * 0.25)};
  }
  int Ls = 1;
  for (int r : radices) {
    if (r == 4) pass64<4>(y, Ls, tw);
    if (r == 8) pass64<8>(y, Ls, tw);
    if (r == 16) pass64<16>(y, Ls, tw);
    Ls *= r;
  }
  auto C = [&](int k) { return k ? Cd{y[k].x + y[N - k].x, y[k].y + y[N - k].y} : y[0]; };
  std::vector<Cd> sum(lanes), inc(lanes);
  for (int t = 0; t < lanes; ++t) {
    Cd s = {0, 0};
    for (int i = 0; i < CH; ++i) s = {s.x + C(t * CH + i).x, s.y + C(t * CH + i).y};
    sum[t] = inc[t] = s;
  }
  for (int d = 1; d < SW; d <<= 1) {
    const std::vector<Cd> o = inc;
    for (int t = 0; t < lanes; ++t)
      if (t % SW >= d) inc[t] = {inc[t].x + o[t - d].x, inc[t].y + o[t - d].y};
  }
  const std::vector<Cd> tot = inc;
  for (int t = 0; t < lanes; ++t) {
    for (int u = 0; u < t / 32; ++u) inc[t] = {inc[t].x + tot[32 * u + 31].x, inc[t].y + tot[32 * u + 31].y};
    Cd r = {inc[t].x - sum[t].x, inc[t].y - sum[t].y};
    for (int i = 0; i < CH; ++i) {
      const int k = t * CH + i;
      r = {r.x + C(k).x, r.y + C(k).y};
      out[2 * k + 1] = r;
      if (k) out[2 * k] = {y[N - k].y - y[k].y, y[k].x - y[N - k].x};
    }
  }
  return out;
}

// ---- fixed point
template <int R, bool HEAD>
static unsigned pass(std::vector<fx2>& a, int Ls, int sh, int drop) {
  const int N = (int)a.size(), G = N / R;
  std::vector<fx2> o(N);
  for (int l = 0; l < G; ++l) {
    const int k = l % Ls, j = l / Ls;
    fx2 x[R];
    for (int q = 0; q < R; ++q) {
      fx2 v = a[l + q * G];
      if (Ls > 1) {
        const unsigned s = (unsigned)(kFxTw - 32 + sh);
        if (q > 0) {
          v = fx_cmul(fx_twiddle((long)q * k, (long)Ls * R), v, s, (1ll << (s - 1)) - (q & 1));
        } else {
          v.x = fx_rescale(v.x, sh);
          v.y = fx_rescale(v.y, sh);
        }
      }
      x[q] = v;
    }
    fx_dft<R, HEAD>(x, (unsigned)drop);
    for (int s = 0; s < R; ++s) o[j * Ls * R + k + s * Ls] = x[s];
  }
  a = o;
  unsigned top = 0;
  for (const fx2& v : a) {
    top |= fx_top(v.x) | fx_top(v.y);
    g_bad += sqrtl((ld)v.x * v.x + (ld)v.y * v.y) > 0x1p62L * 1.4143L;  // 2^62.5 and the roundings
  }
  return top;
}
template <bool STAGED>
static unsigned pass_r(int r, std::vector<fx2>& a, int Ls, int sh, int drop) {
  g_bad += sh > kFxMaxShift || sh < (STAGED ? -kFxMaxLeft : 0);
  return r == 2   ? pass<2, STAGED>(a, Ls, sh, drop)
         : r == 4 ? pass<4, STAGED>(a, Ls, sh, drop)
         : r == 8 ? pass<8, STAGED>(a, Ls, sh, drop)
                  : pass<16, true>(a, Ls, sh, drop);
}
template <int N, int LANES>
static std::vector<Cd> fixed(const std::vector<Cd>& z) {
  typedef FixShape<N, LANES> S;
  typedef FixScale<S::R0, S::R1, S::R2, S::R3> SC;
  typedef FixStaged<S::R0, S::R1, S::R2, S::R3> ST;
  constexpr bool STAGED = fix_staged(N);
  constexpr int S1 = STAGED ? (int)ST::S1 : (int)SC::S1;
  constexpr int G = (int)FixLine<N, LANES>::G;
  const int R[4] = {S::R0, S::R1, S::R2, S::R3};
  unsigned mx = 0, sum = 0;
  for (int j = 1; j < N; ++j)
    for (double v : {z[j].x, z[j].y}) mx = std::max(mx, fx_dhi(v) & 0x7fffffffu);
  const int E = std::max(1, (int)(mx >> 20));
  std::vector<fx2> a(N), y(N);
  for (int j = 1; j < N; ++j) {
    unsigned m;
    a[j].x = fx_from_double<S1>(z[j].x, E, m);
    sum += m >> G;
    a[j].y = fx_from_double<S1>(z[j].y, E, m);
    sum += m >> G;
  }
  const int lb = 32 + G + 32 - __builtin_clz(sum + 2 * N);
  y[0] = {0, 0};
  for (int j = 1; j <= N / 2; ++j) {
    const int2 h = fx_half_sine(j, N);
    const fx2 p = fx_add(a[j], a[N - j]), d = fx_sub(a[j], a[N - j]);
    constexpr bool LOW = FixLine<N, LANES>::kLow;
    const fx2 A = {fx_rmul<62, LOW>(p.x, h.x, h.y), fx_rmul<62, LOW>(p.y, h.x, h.y)};
    const int up = ((j - 1) / LANES) & 1;
    const fx2 B = {(d.x + 1 + up) >> 2, (d.y + 1 + up) >> 2};
    y[j] = fx_add(A, B);
    if (j < N - j) y[N - j] = fx_sub(A, B);
  }
  int t = 0, Ls = S::R0;
  if (STAGED) {
    const int need = ST::need(lb);
    int d = ST::drop(R[0], need, 0);
    unsigned top = pass_r<true>(R[0], y, 1, 0, d);
    t = d;
    for (int p = 1; p < S::NP; ++p, Ls *= R[p - 1]) {
      const int sh = ST::template entry<S::NP>(p, need, t, top);
      d = ST::drop(R[p], need, t + sh);
      top = pass_r<true>(R[p], y, Ls, sh, d);
      t += sh + d;
    }
    g_bad += t < need;
  } else {
    pass_r<false>(R[0], y, 1, 0, 0);
    for (int p = 1; p < S::NP; ++p, Ls *= R[p - 1]) {
      const int all = SC::template shift_at<S::NP>(p, lb);
      const int d = R[p] == 16 && all - t > kFxMaxShift ? 1 : 0;
      pass_r<false>(R[p], y, Ls, all - t - d, d);
      t = all;
    }
  }
  const int q = E - 1022 - S1 + t;
  auto cv = [&](fx2 v) { return Cd{ldexp((double)v.x, q), ldexp((double)v.y, q)}; };
  std::vector<Cd> out(N);
  fx2 run = y[0];
  out[1] = cv(run);
  for (int k = 1; k < N / 2; ++k) {
    const fx2 Yk = y[k], Ym = y[N - k];
    run = fx_add(run, fx_add(Yk, Ym));
    out[2 * k + 1] = cv(run);
    out[2 * k] = cv(fx2{Ym.y - Yk.y, Yk.x - Ym.x});
  }
  return out;
}

// ---- lines: `spikes` entries of about 1 (at N/2 and N/4 with `mid`) over a
// constant or random background; modes: the transform of such a line, as the
// inverse transforms get it
struct Kind {
  const char* name;
  int spikes;
  bool mid, random;
  double background;
  bool modes = false;
};
static const Kind kKinds[] = {
    {"random", 0, false, true, 1.0},       {"constant", 0, false, false, 1.0},    {"alternating", -1, false, false, 1.0},
    {"spike", 1, false, false, 0.0},       {"spike_r1e-8", 1, false, true, 1e-8}, {"spike_c1e-3", 1, false, false, 1e-3},
    {"spike_r1e-3", 1, false, true, 1e-3}, {"spike_c1e-2", 1, false, false, 1e-2}, {"spike_r1e-2", 1, false, true, 1e-2},
    {"spike_c0.1", 1, false, false, 0.1},  {"spike_r0.1", 1, false, true, 0.1},   {"mid_c1e-3", 1, true, false, 1e-3},
    {"modes_spike", 1, false, false, 1e-3, true}, {"modes_mid", 1, true, false, 1e-3, true},
    {"mid_r1e-3", 1, true, true, 1e-3},    {"two_mid_r1e-3", 2, true, true, 1e-3}, {"eight_r1e-2", 8, false, true, 1e-2},
};
static std::vector<Cd> line(const Kind& k, int N, std::mt19937_64& g) {
  auto ud = [&] { return (double)(long long)(g() >> 11) * 0x1p-52 - 1.0; };
  const double c0 = 1 + 0.5 * ud(), c1 = 1 + 0.5 * ud();
  std::vector<Cd> z(N, Cd{0, 0});
  for (int j = 1; j < N; ++j) {
    const double a = ud(), b = ud(), s = k.spikes < 0 && (j & 1) ? -1.0 : 1.0;
    z[j] = k.random ? Cd{k.background * a, k.background * b} : Cd{s * k.background * c0, s * k.background * c1};
  }
  for (int i = 0; i < k.spikes; ++i) {
    const int p = k.mid ? N / (i ? 4 : 2) : 1 + (int)(g() % (unsigned)(N - 1));
    z[p].x += ud() > 0 ? c0 : -c0;
    z[p].y += ud() > 0 ? c1 : -c1;
  }
  if (k.modes) {
    const std::vector<Cl> o = exact(z);
    for (int j = 0; j < N; ++j) z[j] = {(double)o[j].x, (double)o[j].y};
  }
  return z;
}

template <int N, int LANES>
static void test(int lanes64, const std::vector<int>& radices64) {
  const int reps = N >= 2048 ? 12 : 24;
  for (const Kind& k : kKinds) {
    std::mt19937_64 g(1000 * N + (&k - kKinds));
    double ef = 0, ed = 0;
    g_bad = 0;
    for (int r = 0; r < reps; ++r) {
      const std::vector<Cd> z = line(k, N, g);
      const std::vector<Cl> o = exact(z);
      const std::vector<Cd> f = fixed<N, LANES>(z), d = fp64(z, lanes64, radices64);
      ld sf = 0, sd = 0, n = 0;
      for (int m = 1; m < N; ++m) {
        sf += (f[m].x - o[m].x) * (f[m].x - o[m].x) + (f[m].y - o[m].y) * (f[m].y - o[m].y);
        sd += (d[m].x - o[m].x) * (d[m].x - o[m].x) + (d[m].y - o[m].y) * (d[m].y - o[m].y);
        n += o[m].x * o[m].x + o[m].y * o[m].y;
      }
      ef += (double)(sf / n);
      ed += (double)(sd / n);
    }
    printf("%d %d %s %.4e %.4e %d\n", N, LANES, k.name, sqrt(ef / reps), sqrt(ed / reps), g_bad);
  }
}

int main(int argc, char** argv) {
  const int only = argc > 1 ? atoi(argv[1]) : 0;
  // lanes and radices of the FP64 butterflies this form replaced
  if (!only || only == 64) test<64, 16>(8, {8, 8});
  if (!only || only == 128) test<128, 16>(8, {16, 8});
  if (!only || only == 256) test<256, 32>(16, {16, 16}), test<256, 64>(16, {16, 16});
  if (!only || only == 512) test<512, 64>(64, {8, 8, 8}), test<512, 128>(128, {8, 8, 8});
  if (!only || only == 1024) test<1024, 64>(64, {8, 8, 16}), test<1024, 128>(128, {8, 8, 16});
  if (!only || only == 2048) test<2048, 256>(256, {8, 16, 16});
  if (!only || only == 4096) test<4096, 256>(256, {16, 16, 16});
  if (!only || only == 8192) test<8192, 512>(512, {8, 8, 8, 16});
  return 0;
}
