// The line transforms against the definition of the DFT in long double:
//   codelets     every radix, both signs, FP64 and FP32, and every length that the
//                two-step passes split, forward from half a line and back to it
//   double_word  the error of the double-word arithmetic in the same transforms and in a
//                convolution, next to that of AccurateDWPlusDW and DWTimesDW3 (Joldes,
//                Muller and Popescu), a normalisation after every operation
#include "device_on_host.h"

#include <complex>
#include <cstdio>
#include <cstring>
#include <vector>

#include "vie_two.cuh"

namespace vie {
// The scalar double-word operations are those algorithms; here a complex type built from them.
struct published : df {
  using df::df;
};
struct cpublished {
  df x, y;
};
template <> struct CT<published> {
  typedef cpublished V;
  static V make(df a, df b) { return {a, b}; }
};
inline cpublished operator+(cpublished a, cpublished b) { return {a.x + b.x, a.y + b.y}; }
inline cpublished operator-(cpublished a, cpublished b) { return {a.x - b.x, a.y - b.y}; }
inline cpublished operator*(published s, cpublished a) { return {s * a.x, s * a.y}; }
inline cpublished cmul(cpublished a, cpublished b) { return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
inline cpublished cmulc(cpublished a, cpublished b) { return {a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y}; }
}  // namespace vie

using namespace vie;
typedef std::complex<long double> cl;
typedef std::vector<cl> Line;
static const long double kPi = 3.14159265358979323846264338327950288L;

static Line dft(const Line& x, int sign) {
  const int M = (int)x.size();
  Line w(M), y(M);
  for (int j = 0; j < M; ++j) w[j] = cl(cosl(2 * kPi * j / M), sign * sinl(2 * kPi * j / M));
  for (int k = 0; k < M; ++k)
    for (int j = 0; j < M; ++j) y[k] += x[j] * w[(long long)j * k % M];
  return y;
}
static double off(const Line& a, const Line& b) {
  long double e = 0, n = 0;
  for (size_t i = 0; i < b.size(); ++i) {
    e += std::norm(a[i] - b[i]);
    n += std::norm(b[i]);
  }
  return (double)sqrtl(e / n);
}
static unsigned long long g_seed = 1;
static double uniform() {
  g_seed = g_seed * 6364136223846793005ull + 1442695040888963407ull;
  return (double)(g_seed >> 11) / 9007199254740992.0;
}
static double gauss() {
  double s = 0;
  for (int i = 0; i < 12; ++i) s += uniform();
  return s - 6;
}

template <typename T> typename CT<T>::V put(cl v) { return CT<T>::make((T)(double)v.real(), (T)(double)v.imag()); }
template <> float2 put<float>(cl v) { return make_float2((float)v.real(), (float)v.imag()); }
template <> cdf put<df>(cl v) { return CT<df>::make(df((double)v.real()), df((double)v.imag())); }
static cl get(double2 v) { return cl(v.x, v.y); }
static cl get(float2 v) { return cl(v.x, v.y); }
static cl get(cpublished v) { return cl((long double)v.x.hi + v.x.lo, (long double)v.y.hi + v.y.lo); }
static cl get(cdf v) { return cl((long double)v.h.x + v.l.x, (long double)v.h.y + v.l.y); }

template <typename T> std::vector<typename CT<T>::V> twiddles(int M) {
  std::vector<typename CT<T>::V> tw;
  for (int j = 0; j < M; ++j) tw.push_back(put<T>(cl(cosl(2 * kPi * j / M), -sinl(2 * kPi * j / M))));
  return tw;
}
// Half a line to its spectrum, and a spectrum to half a line, as the two-step passes do it.
template <typename T> std::vector<typename CT<T>::V> forward(const TwoPlan& p, const Line& x) {
  typedef typename CT<T>::V V;
  const std::vector<V> tw = twiddles<T>(p.M);
  std::vector<V> s(p.R1 * p.PF), X(p.M);
  const int n = (int)x.size();
  for (int i = 0; i < p.R2; ++i)
    two_fwd1<0, T>(p, i, s.data(), tw.data(), [&](int j) { return j < n ? put<T>(x[j]) : put<T>(cl(0)); });
  for (int k = 0; k < p.R1; ++k) two_fwd2<0, T>(p, k, s.data(), [&](int k2, V v) { X[k + p.R1 * k2] = v; });
  return X;
}
template <typename T> Line inverse(const TwoPlan& p, const std::vector<typename CT<T>::V>& X, int n) {
  typedef typename CT<T>::V V;
  const std::vector<V> tw = twiddles<T>(p.M);
  std::vector<V> s(p.R1 * p.PF);
  Line x(n);
  for (int k = 0; k < p.R1; ++k) two_invA<0, T>(p, k, s.data(), tw.data(), [&](int k2) { return X[k + p.R1 * k2]; });
  for (int i = 0; i < p.R2; ++i)
    two_invB<0, T>(p, i, s.data(), [&](int n1, V v) {
      if (p.R2 * n1 + i < n) x[p.R2 * n1 + i] = get(v);
    });
  return x;
}

static int g_bad = 0;
static void check(const char* what, int len, double err, double bound) {
  if (err <= bound) return;
  printf("%s %d: %.3e above %.3e\n", what, len, err, bound);
  ++g_bad;
}

// A codelet of up to 32 points is at most eight operations deep: 8 u of the norm, twice that for its constants.
template <int R, int S, typename T> void codelet(double u) {
  Line x(R), y(R);
  typename CT<T>::V v[R];
  for (int i = 0; i < R; ++i) {
    v[i] = put<T>(cl(gauss(), gauss()));
    x[i] = get(v[i]);
  }
  Dft<R, S, T>::run(v);
  for (int i = 0; i < R; ++i) y[i] = get(v[i]);
  check(S > 0 ? "codelet +" : "codelet -", R, off(y, dft(x, S)), 16 * u);
}
template <int... R> void codelets() {
  (codelet<R, 1, double>(0x1p-53), ...);
  (codelet<R, -1, double>(0x1p-53), ...);
  (codelet<R, 1, float>(0x1p-24), ...);
  (codelet<R, -1, float>(0x1p-24), ...);
}
static int run_codelets() {
  codelets<2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 14, 15, 16, 18, 20, 21, 22, 24, 32>();
  int lengths = 0;
  for (int M = 16; M <= 576; M += 2) {
    TwoPlan p;
    if (!make_two_plan(M, &p)) continue;
    ++lengths;
    Line x(M / 2), X(M);
    for (cl& v : x) v = cl(gauss(), gauss());
    Line pad = x;
    pad.resize(M);
    std::vector<double2> F = forward<double>(p, x);
    Line f(M);
    for (int k = 0; k < M; ++k) f[k] = get(F[k]);
    check("two steps forward", M, off(f, dft(pad, -1)), 32 * 0x1p-53);
    for (int k = 0; k < M; ++k) F[k] = put<double>(X[k] = cl((double)gauss(), (double)gauss()));
    Line y = dft(X, 1);
    y.resize(M / 2);
    check("two steps back", M, off(inverse<double>(p, F, M / 2), y), 32 * 0x1p-53);
  }
  printf("%d lengths\n", lengths);
  return g_bad != 0 || lengths < 50;
}

// Root mean square over the lines of the relative errors of a transform and of a convolution.
struct Errors {
  double transform, convolution;
};
template <typename T> Errors errors(const TwoPlan& p, int lines) {
  g_seed = 17;
  double et = 0, ec = 0;
  const int M = p.M, n = M / 2;
  for (int r = 0; r < lines; ++r) {
    Line x(n), K(M), Y(M);
    for (int j = 0; j < n; ++j) {  // every other line smooth, as a medium's densities are
      const double t = 2 * (j + 0.5) / n - 1, g = exp(-t * t / 0.1);
      x[j] = get(put<df>((r & 1) ? cl(gauss(), gauss()) : cl(cos(9 * t + r) * g, sin(9 * t + r) * g)));
    }
    Line pad = x;
    pad.resize(M);
    const Line X = dft(pad, -1);
    for (int k = 0; k < M; ++k) {
      const int m = k <= n ? k : k - M;
      K[k] = get(put<df>(cl(gauss(), gauss()) / (1 + 0.01L * m * m) / (long double)M));
      Y[k] = K[k] * X[k];
    }
    Line y = dft(Y, 1);
    y.resize(n);
    auto F = forward<T>(p, x);
    Line f(M);
    for (int k = 0; k < M; ++k) {
      f[k] = get(F[k]);
      F[k] = cmul(put<T>(K[k]), F[k]);
    }
    et += pow(off(f, X), 2);
    ec += pow(off(inverse<T>(p, F, n), y), 2);
  }
  return {sqrt(et / lines), sqrt(ec / lines)};
}
static int run_double_word() {
  for (int M : {48, 64, 96, 128, 140, 192, 256, 300, 384, 440}) {
    TwoPlan p;
    if (!make_two_plan(M, &p)) return 2;
    const Errors now = errors<df>(p, 100), ref = errors<published>(p, 100);
    printf("%d: transform %.3e (published %.3e), convolution %.3e (%.3e)\n", M, now.transform, ref.transform,
           now.convolution, ref.convolution);
    check("double-word transform", M, now.transform, ref.transform);
    check("double-word convolution", M, now.convolution, ref.convolution);
  }
  return g_bad != 0;
}

int main(int argc, char** argv) {
  return argc > 1 && !strcmp(argv[1], "double_word") ? run_double_word() : run_codelets();
}
