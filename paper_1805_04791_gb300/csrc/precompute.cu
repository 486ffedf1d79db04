// Set-up kernels of a problem, on the device, to FP64 accuracy (FP64 arithmetic,
// except the kernel-transform line FFTs, which run in double-word arithmetic on
// the FP32 pipes unless VIE_SETUP_FP64=1):
//  * H_eps = (eps + I)^-1 (eps - I) per node (Eq. (rhodef), Lemma 1), stored as
//    the 6 entries of the symmetric tensor in FP64 and FP32;
//  * the transform of the truncated Green's function (Sec. 5, steps a-b),
//    tabulated once per distinct integer |m|^2 of the oversampled frequency grid;
//  * the discrete kernels of every Fourier symbol (1, i k_a, -k_a k_b) with the
//    grid Nyquist cutoff (Sec. 5, step c), brought to the (2n)^3 convolution
//    grid, on octants throughout (the kernels are even or odd in each axis).
#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <cmath>
#include <functional>
#include <vector>

#include "vie_internal.h"

namespace vie {

// ---------------------------------------------------------------- twiddles
template <typename V>
__global__ void k_twiddle(V* tw, int M) {
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= M) return;
  double s, c;
  sincospi(2.0 * (double)j / (double)M, &s, &c);
  tw[j].x = c;
  tw[j].y = -s;
}

// exp(-2 pi i num / den) for 0 <= num < den: the quarter turns are taken out
// in integer arithmetic, the rest is an angle in [0, pi/2).
static void exp_m2pi(long long num, long long den, double* c, double* s) {
  const long long q = (4 * num) / den, rem = 4 * num - q * den;
  const double t = M_PI * (double)rem / (2.0 * (double)den);
  const double c0 = std::cos(t), s0 = std::sin(t);
  double cc, ss;  // cos, sin of the full angle
  switch (q & 3) {
    case 0: cc = c0; ss = s0; break;
    case 1: cc = -s0; ss = c0; break;
    case 2: cc = -c0; ss = -s0; break;
    default: cc = s0; ss = -c0; break;
  }
  *c = cc;
  *s = -ss;
}

// Line table of a plan (line_table_len entries, layout of line_fft): the Q
// twiddles exp(-2 pi i j / Q) on the device; for a Bluestein plan then the
// chirps c-_j = exp(-pi i j^2 / M) and c+_j = conj(c-_j) with j^2 reduced mod
// 2M, and H-_k = (1/Q) sum_{|j|<M} c+_j exp(-2 pi i j k / Q)
//             = (1/Q) (1 + 2 sum_{0<j<M} c+_j cos(2 pi j k / Q)),
// all in FP64 on the host.
vie_status make_line_table(const FftPlan& pl, double2** t64, float2** t32, cudaStream_t st) {
  const int M = pl.M, Q = pl.Q, len = line_table_len(pl);
  VIE_CK(dalloc((void**)t64, sizeof(double2) * len, st));
  VIE_CK(dalloc((void**)t32, sizeof(float2) * len, st));
  k_twiddle<double2><<<(Q + 127) / 128, 128, 0, st>>>(*t64, Q);
  k_twiddle<float2><<<(Q + 127) / 128, 128, 0, st>>>(*t32, Q);
  VIE_CK(cudaGetLastError());
  if (Q == M) return VIE_OK;
  std::vector<double2> h(len - Q);
  std::vector<float2> h32(len - Q);
  for (int j = 0; j < M; ++j) {
    double c, sn;
    exp_m2pi(((long long)j * j) % (2LL * M), 2LL * M, &c, &sn);
    h[j] = make_double2(c, sn);
    h[M + j] = make_double2(c, -sn);
  }
  std::vector<double> cq(Q);
  for (int t = 0; t < Q; ++t) {
    double c, sn;
    exp_m2pi(t, Q, &c, &sn);
    cq[t] = c;
  }
  for (int k = 0; k < Q; ++k) {
    double re = 0.0, im = 0.0;
    int jk = 0;  // j k mod Q
    for (int j = 1; j < M; ++j) {
      jk += k;
      if (jk >= Q) jk -= Q;
      re += h[M + j].x * cq[jk];
      im += h[M + j].y * cq[jk];
    }
    h[2 * M + k] = make_double2((1.0 + 2.0 * re) / Q, 2.0 * im / Q);
  }
  for (size_t i = 0; i < h.size(); ++i) h32[i] = make_float2((float)h[i].x, (float)h[i].y);
  VIE_CK(cudaMemcpyAsync(*t64 + Q, h.data(), sizeof(double2) * h.size(), cudaMemcpyHostToDevice, st));
  VIE_CK(cudaMemcpyAsync(*t32 + Q, h32.data(), sizeof(float2) * h32.size(), cudaMemcpyHostToDevice, st));
  VIE_CK(cudaStreamSynchronize(st));  // the host vectors go out of scope
  return VIE_OK;
}

// ------------------------------------------------------------ medium tensor
// H = (A)^-1 (eps - I) = I - 2 A^-1 with A = eps + I, via the adjugate.
__global__ void k_medium(const double2* __restrict__ eps, double2* __restrict__ H64, float2* __restrict__ H32,
                         long long N, int realonly, int* flag) {
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < N; p += (long long)gridDim.x * blockDim.x) {
    double2 a[3][3];
    double mag = 0.0;
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) {
        double2 v = eps[(i * 3 + j) * N + p];
        if (realonly) v.y = 0.0;
        a[i][j] = v;
        mag = fmax(mag, fabs(v.x) + fabs(v.y));
      }
    const double tol = 1e-12 * (1.0 + mag);
    for (int i = 0; i < 3; ++i)
      for (int j = i + 1; j < 3; ++j)
        if (fabs(a[i][j].x - a[j][i].x) + fabs(a[i][j].y - a[j][i].y) > tol) atomicOr(flag, 1);
    for (int i = 0; i < 3; ++i) a[i][i].x += 1.0;
    double2 adj[3][3];
    adj[0][0] = cmul(a[1][1], a[2][2]) - cmul(a[1][2], a[2][1]);
    adj[0][1] = cmul(a[0][2], a[2][1]) - cmul(a[0][1], a[2][2]);
    adj[0][2] = cmul(a[0][1], a[1][2]) - cmul(a[0][2], a[1][1]);
    adj[1][0] = cmul(a[1][2], a[2][0]) - cmul(a[1][0], a[2][2]);
    adj[1][1] = cmul(a[0][0], a[2][2]) - cmul(a[0][2], a[2][0]);
    adj[1][2] = cmul(a[0][2], a[1][0]) - cmul(a[0][0], a[1][2]);
    adj[2][0] = cmul(a[1][0], a[2][1]) - cmul(a[1][1], a[2][0]);
    adj[2][1] = cmul(a[0][1], a[2][0]) - cmul(a[0][0], a[2][1]);
    adj[2][2] = cmul(a[0][0], a[1][1]) - cmul(a[0][1], a[1][0]);
    double2 det = cmul(a[0][0], adj[0][0]) + cmul(a[0][1], adj[1][0]) + cmul(a[0][2], adj[2][0]);
    const double dd = det.x * det.x + det.y * det.y;
    if (!(dd > 0.0) || !isfinite(dd)) {
      atomicOr(flag, 2);
      continue;
    }
    // 1/det = conj(det)/|det|^2
    const double2 inv = make_double2(det.x / dd, -det.y / dd);
    const int ii[6] = {0, 1, 2, 0, 0, 1};
    const int jj[6] = {0, 1, 2, 1, 2, 2};
    for (int e = 0; e < 6; ++e) {
      double2 q = cmul(adj[ii[e]][jj[e]], inv);
      double2 h = make_double2(-2.0 * q.x, -2.0 * q.y);
      if (ii[e] == jj[e]) h.x += 1.0;
      H64[e * N + p] = h;
      H32[e * N + p] = make_float2((float)h.x, (float)h.y);
    }
  }
}

vie_status build_medium(vie_problem* P, const void* eps, const void* mu, cudaStream_t st) {
  const long long N = (long long)P->n * P->n * P->n;
  VIE_CK(dalloc((void**)&P->He64, sizeof(double2) * 6 * N, st));
  VIE_CK(dalloc((void**)&P->He32, sizeof(float2) * 6 * N, st));
  VIE_CK(cudaMemsetAsync(P->dflag, 0, sizeof(int), st));
  const int blocks = (int)std::min<long long>((N + 255) / 256, 152LL * 16);
  k_medium<<<blocks, 256, 0, st>>>((const double2*)eps, P->He64, P->He32, N, P->kind == VIE_LAPLACE, P->dflag);
  VIE_CK(cudaGetLastError());
  if (P->has_mu) {
    VIE_CK(dalloc((void**)&P->Hm64, sizeof(double2) * 6 * N, st));
    VIE_CK(dalloc((void**)&P->Hm32, sizeof(float2) * 6 * N, st));
    k_medium<<<blocks, 256, 0, st>>>((const double2*)mu, P->Hm64, P->Hm32, N, 0, P->dflag);
    VIE_CK(cudaGetLastError());
  }
  int flag = 0;
  VIE_CK(cudaMemcpyAsync(&flag, P->dflag, sizeof(int), cudaMemcpyDeviceToHost, st));
  VIE_CK(cudaStreamSynchronize(st));
  if (flag & 1) {
    set_error("eps/mu must be symmetric at every node");
    return VIE_EINVAL;
  }
  if (flag & 2) {
    set_error("eps + I (or mu + I) is singular or non-finite at some node");
    return VIE_EINVAL;
  }
  return VIE_OK;
}

// ------------------------------------------------ truncated kernel transform
// G^_L(kappa) = (1/kappa) int_0^L sin(kappa r) e^{i w r} dr (Sec. 5, steps a-b),
// evaluated as [E(w + kappa) - E(w - kappa)] / (2 i kappa) with
// E(a) = int_0^L e^{i a r} dr = L e^{i a L/2} sinc(a L/2): no cancellation at
// kappa = w.  kappa = 0: int_0^L r e^{i w r} dr, closed form for wL >= 1/2,
// power series sum_q (i w L)^q L^2 / (q! (q + 2)) below.  On the grids used
// here every other kappa has kappa L >= 2 pi sqrt(3)/3, far from the
// cancellation of the E difference at small kappa L.
__device__ double2 dev_E(double a, double L) {
  const double t = 0.5 * a * L;
  const double sc = (t == 0.0) ? 1.0 : sin(t) / t;
  double s, c;
  sincos(t, &s, &c);
  return make_double2(L * c * sc, L * s * sc);
}

__device__ double2 dev_ghat(double kappa, double w, double L) {
  if (kappa == 0.0) {
    const double wl = w * L;
    if (fabs(wl) < 0.5) {
      double2 acc = make_double2(0.0, 0.0);
      double2 term = make_double2(1.0, 0.0);  // (i w L)^q / q!
      for (int q = 0; q < 40; ++q) {
        const double f = L * L / (double)(q + 2);
        acc = acc + f * term;
        term = cmul(term, make_double2(0.0, wl / (double)(q + 1)));
      }
      return acc;
    }
    double s, c;
    sincos(wl, &s, &c);
    return make_double2((c + s * wl - 1.0) / (w * w), (s - c * wl) / (w * w));
  }
  const double2 d = dev_E(w + kappa, L) - dev_E(w - kappa, L);
  return make_double2(d.y / (2.0 * kappa), -d.x / (2.0 * kappa));
}

__global__ void k_ghat_table(double2* tab, int jmax, double dk, double w, double L) {
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j > jmax) return;
  tab[j] = dev_ghat(dk * sqrt((double)j), w, L);
}

// The discrete kernels.  On the (sn)^3 frequency grid F(m) = S~(k_m) G^(|k_m|)
// depends on m only through |m_x|, |m_y|, |m_z| and one sign per axis (a factor
// k_a is odd in m_a, everything else is even), and "inverse DFT over sn, keep the
// offsets |d| < n, place them at d mod M, DFT over M" acts on each axis by
// itself, keeping that parity.  So a symbol's octant (nk + 1)^3 comes from the
// octant m >= 0 of F by one line operator per axis, x, y, z in turn, each in a
// single pass that reads sn/2 + 1 entries of a line and writes nk + 1: 4.75 n^2
// lines of sn and M points, against 27 n^2 and 12 n^2 for the whole cubes, and
// 10 n^3 against 210 n^3 values moved.  All symbols follow from four of them by
// exchanging axes (G^ is radial): 1, -k_z^2, -k_x k_y and i k_z, z being the
// axis that is not like the other two.
// Measured, 192^3 reduced Maxwell problem: 302 ms for seven symbols on whole cubes
// (279 ms of cube transforms, 21 ms to fill them); three bases here take 10.8 ms
// (29.5 with a normalisation after every double-word operation; the pairing in k_axis
// saved a sixth here and a quarter at Helmholtz 64^3, now 0.37 ms).
enum Base { BASE_1 = 0, BASE_ZZ, BASE_XY, BASE_DZ, BASE_COUNT };

static int base_of(int sym) {
  switch (sym) {
    case SYM_1: return BASE_1;
    case SYM_XX: case SYM_YY: case SYM_ZZ: return BASE_ZZ;
    case SYM_XY: case SYM_XZ: case SYM_YZ: return BASE_XY;
    default: return BASE_DZ;
  }
}
// Axis of the symbol that takes the place of its base's z (2 z, 1 y, 0 x).
static int axis_of(int sym) {
  switch (sym) {
    case SYM_XX: case SYM_YZ: case SYM_DX: return 0;
    case SYM_YY: case SYM_XZ: case SYM_DY: return 1;
    default: return 2;
  }
}

struct AxisPass {
  int axis;        // 0 x, 1 y, 2 z
  int base;        // Base
  int pair;        // a second base, odd in this axis, in the same transforms (-1: none)
  int n, nk, sn;
  int odd;         // the base is odd in this axis
  int nl;          // lines per tile
  int LS;          // pitch of a tile line
  double dk;       // frequency spacing 2 pi / (3 D)
  double scale;    // factor of the stored values (1, or 1/(sn)^3 in the last pass)
  FftPlan ps, pm;  // line plans of lengths sn and M = 2 nk
};

// F of base `b` at m >= 0 (all axes).  Even sn: m_a = sn/2 is the Nyquist entry,
// where an odd factor k_a is replaced by 0 (the mean of its values at -pi/h and
// +pi/h) and an even factor k_a^2 is kept.  Odd sn has no Nyquist entry.
__device__ __forceinline__ double2 base_sample(const double2* __restrict__ tab, int b, int mx, int my, int mz, int sn,
                                               double dk) {
  const double2 G = tab[mx * mx + my * my + mz * mz];
  auto kodd = [&](int m) { return 2 * m == sn ? 0.0 : dk * m; };
  if (b == BASE_1) return G;
  if (b == BASE_ZZ) return (-(dk * mz) * (dk * mz)) * G;
  if (b == BASE_XY) return (-kodd(mx) * kodd(my)) * G;
  const double oz = kodd(mz);
  return make_double2(-oz * G.y, oz * G.x);
}

// A base that is even in the axis and one that is odd go through one transform of
// their sum: the even part of the result is the first's, the odd part the second's
// (-k_z^2 and -k_x k_y, of the same magnitude, in the x and y passes).
//
// One line operator over `nl` lines per CTA (blockDim.y = nl, blockDim.x threads
// a line).  Layouts: x pass  tab -> out [mz][my][kx], y pass [mz][my][kx] ->
// [mz][ky][kx], z pass [mz][ky][kx] -> [kz][ky][kx]; 0 <= m <= sn/2, 0 <= k <= nk.
// The lines of a y or z tile are neighbours in kx, so a tile reads and writes
// runs of nl 16-byte values.
template <typename T>
__global__ void k_axis(const double2* __restrict__ in, double2* __restrict__ out, const double2* __restrict__ in2,
                       double2* __restrict__ out2, AxisPass q, const typename CT<T>::V* __restrict__ tws,
                       const typename CT<T>::V* __restrict__ twm) {
  typedef typename CT<T>::V V;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nl = q.nl, LS = q.LS, sn = q.sn, n = q.n, M = q.pm.M, Q = q.ps.Q, O = q.nk + 1, S = sn / 2 + 1;
  V* ts = (V*)smraw;
  V* tm = ts + Q;
  V* b0 = tm + M;
  V* b1 = b0 + nl * LS;
  const int tid = flat_tid(), nt = flat_nthreads();
  for (int j = tid; j < Q; j += nt) ts[j] = tws[j];
  for (int j = tid; j < M; j += nt) tm[j] = twm[j];
  // lines of this tile: x pass rows r0 + l < S^2; y, z passes kx = r0 + l < O of slab blockIdx.y
  const int r0 = blockIdx.x * nl, slab = blockIdx.y;
  const long long lines = q.axis == 0 ? (long long)S * S : O;
  // stride between entries of a line, and the first entry of line r, on the input and output side
  const long long istep = q.axis == 1 ? O : (long long)O * O;
  const long long ibase = q.axis == 1 ? (long long)slab * S * O : (long long)slab * O;
  const long long ostep = q.axis == 0 ? 1 : istep;
  const long long obase = q.axis == 1 ? (long long)slab * O * O : (long long)slab * O;
  for (int idx = tid; idx < nl * S; idx += nt) {
    int l, m;
    if (q.axis == 0) { l = idx / S; m = idx - l * S; } else { m = idx / nl; l = idx - m * nl; }
    const long long r = r0 + l;
    double2 v = make_double2(0.0, 0.0), v2 = v;
    if (r < lines) {
      if (q.axis == 0) {
        const int mz = (int)(r / S), my = (int)(r - (long long)mz * S);
        v = base_sample(in, q.base, m, my, mz, sn, q.dk);
        if (q.pair >= 0) v2 = base_sample(in, q.pair, m, my, mz, sn, q.dk);
      } else {
        v = in[ibase + m * istep + r];
        if (q.pair >= 0) v2 = in2[ibase + m * istep + r];
      }
    }
    V a = to_v<T>(v), am = q.odd ? vneg(a) : a;  // at m and at -m
    if (q.pair >= 0) {
      const V c = to_v<T>(v2);
      am = a - c;
      a = a + c;
    }
    b0[l * LS + m] = a;
    if (m > 0 && 2 * m != sn) b0[l * LS + sn - m] = am;
  }
  __syncthreads();
  V* r = line_fft<+1, T>(b0, b1, q.ps, ts, tws + Q, nl, LS);
  V* e = (r == b0) ? b1 : b0;
  // offsets d in [-(n-1), n-1] at index d mod M, zeros between
  for (int idx = tid; idx < nl * M; idx += nt) {
    const int l = idx / M, j = idx - l * M;
    e[l * LS + j] = j < n ? r[l * LS + j] : (j > M - n ? r[l * LS + j - M + sn] : CT<T>::make(0, 0));
  }
  __syncthreads();
  V* w = line_fft<-1, T>(e, r, q.pm, tm, twm + M, nl, LS);
  for (int idx = tid; idx < nl * O; idx += nt) {
    int l, k;
    if (q.axis == 0) { l = idx / O; k = idx - l * O; } else { k = idx / nl; l = idx - k * nl; }
    const long long row = r0 + l;
    if (row >= lines) continue;
    const long long at = q.axis == 0 ? row * O + k : obase + k * ostep + row;
    const V v = w[l * LS + k];
    if (q.pair < 0) {
      out[at] = q.scale * from_v<T>(v);
    } else {
      const V vm = w[l * LS + (k == 0 ? 0 : M - k)];
      out[at] = 0.5 * q.scale * from_v<T>(v + vm);
      out2[at] = 0.5 * q.scale * from_v<T>(v - vm);
    }
  }
}

// Octants of the bases in `mask`: the three line operators of each.  A1 holds
// [2][S][S][O], A2 [2][S][O][O], oct [BASE_COUNT][O][O][O].
template <typename T>
static vie_status base_octants(vie_problem* P, unsigned mask, const double2* tab, double2* A1, double2* A2, double2* oct,
                               const FftPlan& ps, const typename CT<T>::V* tws, const typename CT<T>::V* twm,
                               cudaStream_t st) {
  typedef typename CT<T>::V V;
  AxisPass q;
  q.n = P->n;
  q.nk = P->nk;
  q.sn = 3 * P->n;
  q.dk = 2.0 * M_PI / (3.0 * P->D);
  q.ps = ps;
  q.pm = P->planM;
  q.LS = std::max(ps.Q, P->planM.M) + 1;
  const int S = q.sn / 2 + 1, O = q.nk + 1;
  // lines per tile: up to eight (128-byte runs in the y and z passes), with the
  // tile within 110 KB, so that two CTAs share an SM, where that leaves two lines
  auto smem_of = [&](int nl) { return sizeof(V) * (ps.Q + P->planM.M + 2 * (size_t)nl * q.LS); };
  q.nl = 8;
  while (q.nl > 2 && smem_of(q.nl) > 110 * 1024) q.nl >>= 1;
  while (q.nl > 1 && smem_of(q.nl) > (size_t)smem_optin_bytes()) q.nl >>= 1;
  const size_t smem = smem_of(q.nl);
  if (smem > (size_t)smem_optin_bytes()) {
    set_error("set-up transform line too long for shared memory");
    return VIE_EINVAL;
  }
  VIE_CK(allow_smem(k_axis<T>));
  // threads a line: a power of two near Q / 8, at most 256 a block
  int tx = 8;
  while (tx * 8 < ps.Q && 2 * tx * q.nl <= 256) tx <<= 1;
  const dim3 blk(tx, q.nl);
  auto pass = [&](int axis, int base, int pair, const double2* src, double2* dst, const double2* src2,
                  double2* dst2) -> vie_status {
    q.axis = axis;
    q.base = base;
    q.pair = pair;
    q.odd = (base == BASE_XY && axis != 2) || (base == BASE_DZ && axis == 2);
    q.scale = axis == 2 ? 1.0 / ((double)q.sn * q.sn * q.sn) : 1.0;
    const dim3 grid = axis == 0 ? dim3((unsigned)(((long long)S * S + q.nl - 1) / q.nl))
                                : dim3((O + q.nl - 1) / q.nl, axis == 1 ? S : O);
    k_axis<T><<<grid, blk, smem, st>>>(src, dst, src2, dst2, q, tws, twm);
    VIE_CK(cudaGetLastError());
    return VIE_OK;
  };
  const long long n1 = (long long)S * S * O, n2 = (long long)S * O * O, O3 = (long long)O * O * O;
  const unsigned both = (1u << BASE_ZZ) | (1u << BASE_XY);
  const bool paired = (mask & both) == both;
  for (int b = 0; b < BASE_COUNT; ++b) {
    if (!(mask & (1u << b)) || (paired && b == BASE_XY)) continue;
    const bool two = paired && b == BASE_ZZ;
    const int pair = two ? BASE_XY : -1;
    vie_status s = pass(0, b, pair, tab, A1, nullptr, A1 + n1);
    if (s == VIE_OK) s = pass(1, b, pair, A1, A2, A1 + n1, A2 + n2);
    if (s == VIE_OK) s = pass(2, b, -1, A2, oct + b * O3, nullptr, nullptr);
    if (s == VIE_OK && two) s = pass(2, BASE_XY, -1, A2 + n2, oct + BASE_XY * O3, nullptr, nullptr);
    if (s != VIE_OK) return s;
  }
  return VIE_OK;
}

// Combine base octants into the kernel arrays of one pass.
//   coef layout per output array a: up to 2 terms (base octant, the axis that
//   takes its z, complex factor); base < 0: no term.
struct CombineDesc {
  int narr;
  int base[9][2];
  int axis[9][2];
  double2 fac[9][2];
  void set(int a, int t, int sym, double2 f) {
    base[a][t] = base_of(sym);
    axis[a][t] = axis_of(sym);
    fac[a][t] = f;
  }
};

// The bases are symmetric under exchange of their x and y, so a symbol whose
// odd-one-out axis is z or y reads base[oz][oy][ox] or base[oy][oz][ox], both
// contiguous in ox, and one whose axis is x reads base[ox][oz][oy], which a
// 32 x 32 tile in shared memory turns round.  grid = (ox tiles, oy tiles, oz).
__global__ void __launch_bounds__(256) k_combine(const double2* __restrict__ bases, double2* __restrict__ out64,
                                                 float2* __restrict__ out32, int O, CombineDesc cd,
                                                 double diag_add_scale, int diag_mask) {
  __shared__ double2 tile[32][33];
  const long long O3 = (long long)O * O * O;
  const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 32, oz = blockIdx.z;
  for (int a = 0; a < cd.narr; ++a) {
    double2 v[4];
    for (int i = 0; i < 4; ++i) v[i] = make_double2(0.0, 0.0);
    for (int t = 0; t < 2; ++t) {
      const int bs = cd.base[a][t], ax = cd.axis[a][t];
      if (bs < 0) continue;  // uniform over the grid
      const double2* src = bases + bs * O3;
      if (ax == 0) {
        __syncthreads();
        for (int i = 0; i < 4; ++i) {
          const int ox = x0 + threadIdx.y + 8 * i, oy = y0 + threadIdx.x;
          if (ox < O && oy < O) tile[threadIdx.y + 8 * i][threadIdx.x] = src[((long long)ox * O + oz) * O + oy];
        }
        __syncthreads();
      }
      for (int i = 0; i < 4; ++i) {
        const int ox = x0 + threadIdx.x, oy = y0 + threadIdx.y + 8 * i;
        if (ox >= O || oy >= O) continue;
        const double2 s = ax == 0 ? tile[threadIdx.x][threadIdx.y + 8 * i]
                                  : src[ax == 1 ? ((long long)oy * O + oz) * O + ox : ((long long)oz * O + oy) * O + ox];
        v[i] = v[i] + cmul(cd.fac[a][t], s);
      }
    }
    for (int i = 0; i < 4; ++i) {
      const int ox = x0 + threadIdx.x, oy = y0 + threadIdx.y + 8 * i;
      if (ox >= O || oy >= O) continue;
      if (diag_mask & (1 << a)) v[i].x += diag_add_scale;
      const long long idx = a * O3 + ((long long)oz * O + oy) * O + ox;
      out64[idx] = v[i];
      out32[idx] = make_float2((float)v[i].x, (float)v[i].y);
    }
  }
}

static vie_status combine(vie_problem* P, KernelSet& K, int mode, const CombineDesc& cd, double diag_add,
                          int diag_mask, cudaStream_t st) {
  const long long O = P->nk + 1, O3 = O * O * O;
  double2* oct64 = nullptr;
  float2* oct32 = nullptr;
  cudaError_t e = dalloc((void**)&oct64, sizeof(double2) * cd.narr * O3, st);
  if (e == cudaSuccess) e = dalloc((void**)&oct32, sizeof(float2) * cd.narr * O3, st);
  if (e == cudaSuccess) {
    const unsigned tiles = (unsigned)((O + 31) / 32);
    k_combine<<<dim3(tiles, tiles, (unsigned)O), dim3(32, 8), 0, st>>>(P->base_oct, oct64, oct32, (int)O, cd, diag_add,
                                                                       diag_mask);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) {  // the set stays as it was: its arrays say whether it is built
    dfree(oct64, st);
    dfree(oct32, st);
    return cuda_fail(e, "kernel set");
  }
  K.mode = mode;
  K.narr = cd.narr;
  K.oct64 = oct64;
  K.oct32 = oct32;
  return VIE_OK;
}

static vie_status to_df(const double2* src, cdf** dst, long long count, cudaStream_t st);

// Compute the base octants that the symbols in `syms` (bit = Sym) need and that
// are not there yet.
static vie_status compute_symbols(vie_problem* P, unsigned syms, cudaStream_t st) {
  unsigned mask = 0;
  for (int s = 0; s < SYM_COUNT; ++s)
    if (syms & (1u << s)) mask |= 1u << base_of(s);
  mask &= ~P->base_mask;
  if (!mask) return VIE_OK;
  const int n = P->n, sn = 3 * n;
  const double dk = 2.0 * M_PI / (3.0 * P->D);
  const int jmax = 3 * (sn / 2) * (sn / 2);
  const double w = P->kind == VIE_LAPLACE ? 0.0 : P->omega;
  FftPlan plsn;
  if (!make_line_plan(sn, &plsn)) {
    set_error("bad oversampled grid size");
    return VIE_EINVAL;
  }
  double2 *tab = nullptr, *A1 = nullptr, *A2 = nullptr, *tw_sn = nullptr;
  float2* tw_sn32 = nullptr;
  cdf *tw_sndf = nullptr, *tw_2ndf = nullptr;
  struct Guard {  // the scratch goes back on every way out
    std::function<void()> f;
    ~Guard() { f(); }
  } guard{[&] {
    void* all[] = {A1, A2, tab, tw_sn, tw_sn32, tw_sndf, tw_2ndf};
    for (void* q : all) dfree(q, st);
  }};
  const long long O = P->nk + 1, S = sn / 2 + 1, O3 = O * O * O;
  if (!P->base_oct) VIE_CK(dalloc((void**)&P->base_oct, sizeof(double2) * BASE_COUNT * O3, st));
  VIE_CK(dalloc((void**)&tab, sizeof(double2) * (jmax + 1), st));
  k_ghat_table<<<(jmax + 256) / 256, 256, 0, st>>>(tab, jmax, dk, w, P->L);
  VIE_CK(cudaGetLastError());
  VIE_CK(dalloc((void**)&A1, sizeof(double2) * 2 * S * S * O, st));
  VIE_CK(dalloc((void**)&A2, sizeof(double2) * 2 * S * O * O, st));
  vie_status s = make_line_table(plsn, &tw_sn, &tw_sn32, st);
  if (s != VIE_OK) return s;
  // the transforms run in double-word arithmetic (FP64 accuracy on the FP32
  // pipes); VIE_SETUP_FP64=1 keeps them in native FP64
  const char* e64 = getenv("VIE_SETUP_FP64");
  const bool dw = !(e64 && e64[0] == '1');
  if (dw) {
    s = to_df(tw_sn, &tw_sndf, line_table_len(plsn), st);
    if (s == VIE_OK) s = to_df(P->tw64, &tw_2ndf, line_table_len(P->planM), st);
    if (s != VIE_OK) return s;
  }
  s = dw ? base_octants<df>(P, mask, tab, A1, A2, P->base_oct, plsn, tw_sndf, tw_2ndf, st)
         : base_octants<double>(P, mask, tab, A1, A2, P->base_oct, plsn, tw_sn, P->tw64, st);
  if (s != VIE_OK) return s;
  P->base_mask |= mask;
  return VIE_OK;
}

static const unsigned kQmask = (1u << SYM_XX) | (1u << SYM_YY) | (1u << SYM_ZZ) | (1u << SYM_XY) | (1u << SYM_XZ) |
                               (1u << SYM_YZ);
static const unsigned kDmask = (1u << SYM_DX) | (1u << SYM_DY) | (1u << SYM_DZ);

// Kernel sets: `which` 0 = operator apply, 1 = scattered field.
static vie_status combine_sets(vie_problem* P, int which, cudaStream_t st);

// ------------------------------------------------ operator norm bound
__device__ __forceinline__ double dnorm2c(double2 a) { return a.x * a.x + a.y * a.y; }

// max over points of the Frobenius norm of a symmetric 3x3 tensor field stored
// as 6 arrays (xx yy zz xy xz yz) of stride S, with 3 more arrays (a curl
// symbol p: the 6x6 Maxwell kernel [[Q, p x], [-p x, Q]]) when np == 3, into
// *out as the bit pattern of a non-negative double (ordered like the double).
__global__ void k_fro_max(const double2* __restrict__ a, long long S, int np, unsigned long long* out) {
  double mx = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < S; i += (long long)gridDim.x * blockDim.x) {
    double f = 0.0;
    for (int e = 0; e < 6; ++e) f += (e < 3 ? 1.0 : 2.0) * dnorm2c(a[e * S + i]);
    if (np == 3) {
      double p = 0.0;
      for (int e = 6; e < 9; ++e) p += dnorm2c(a[e * S + i]);
      f = 2.0 * f + 4.0 * p;
    }
    mx = fmax(mx, f);
  }
  for (int off = 16; off > 0; off >>= 1) mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, off));
  if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(sqrt(mx)));
}

// Upper bound of ||A||_2 = ||I + H conv||_2 <= 1 + max ||H||_F max_k ||K^(k)||_F with
// the kernel's eigenvalues M^3 K_stored (the 1/M^3 of the inverse DFT is folded
// into the stored octants).  Used to bound the error of an FP32 apply.
static vie_status op_norm_bound(vie_problem* P, cudaStream_t st) {
  unsigned long long* d = nullptr;
  VIE_CK(dalloc((void**)&d, 3 * sizeof(unsigned long long), st));
  VIE_CK(cudaMemsetAsync(d, 0, 3 * sizeof(unsigned long long), st));
  const long long O = P->nk + 1, O3 = O * O * O, N = (long long)P->n * P->n * P->n;
  const int np = P->kapply.mode == KM_MAXWELL6 ? 3 : 0;
  k_fro_max<<<152 * 4, 256, 0, st>>>(P->kapply.oct64, O3, np, d);
  k_fro_max<<<152 * 4, 256, 0, st>>>(P->He64, N, 0, d + 1);
  if (P->Hm64) k_fro_max<<<152 * 4, 256, 0, st>>>(P->Hm64, N, 0, d + 2);
  VIE_CK(cudaGetLastError());
  unsigned long long h[3];
  VIE_CK(cudaMemcpyAsync(h, d, sizeof(h), cudaMemcpyDeviceToHost, st));
  VIE_CK(cudaStreamSynchronize(st));
  dfree(d, st);
  double v[3];
  for (int i = 0; i < 3; ++i) memcpy(&v[i], &h[i], sizeof(double));
  const double M = 2.0 * P->nk;
  P->opnorm = 1.0 + std::max(v[1], v[2]) * v[0] * M * M * M;
  return VIE_OK;
}

vie_status build_kernels(vie_problem* P, cudaStream_t st) {
  // the operator needs -k_a k_b (and, for Maxwell, 1; with mu also the curl
  // symbols i k_a); the symbols only the scattered field needs are built on
  // its first use
  unsigned mask = kQmask;
  if (P->kind == VIE_MAXWELL) mask |= (1u << SYM_1) | (P->has_mu ? kDmask : 0u);
  vie_status s = compute_symbols(P, mask, st);
  if (s != VIE_OK) return s;
  s = combine_sets(P, 0, st);
  if (s != VIE_OK) return s;
  return op_norm_bound(P, st);
}

vie_status build_eval_kernels(vie_problem* P, cudaStream_t st) {
  if (P->keval.oct64) return VIE_OK;
  const unsigned mask = P->kind == VIE_MAXWELL ? (kQmask | kDmask | (1u << SYM_1)) : kDmask;
  vie_status s = compute_symbols(P, mask, st);
  if (s != VIE_OK) return s;
  return combine_sets(P, 1, st);
}

static vie_status combine_sets(vie_problem* P, int which, cudaStream_t st) {
  const int M = 2 * P->nk;
  const long long M3 = (long long)M * M * M;
  const double w = P->kind == VIE_LAPLACE ? 0.0 : P->omega;
  vie_status s = VIE_OK;
  // Fold constants: apply kernels give u with y = x + H u; the 1/(2n)^3 of the
  // inverse DFT is folded in too.
  const double nrm = 1.0 / (double)M3;
  const int Q[6] = {SYM_XX, SYM_YY, SYM_ZZ, SYM_XY, SYM_XZ, SYM_YZ};
  const int Dd[3] = {SYM_DX, SYM_DY, SYM_DZ};
  CombineDesc ca{}, ce{};
  for (int a = 0; a < 9; ++a)
    for (int t = 0; t < 2; ++t) {
      ca.base[a][t] = -1;
      ce.base[a][t] = -1;
      ca.fac[a][t] = make_double2(0, 0);
      ce.fac[a][t] = make_double2(0, 0);
    }
  const double w2 = w * w;
  if (P->kind == VIE_LAPLACE || P->kind == VIE_HELMHOLTZ) {
    // Laplace  (Eq. (eq:intLap)):  u = -2 T_0 x  (y = x + H_eps u)
    // Helmholtz (Eq. (eq:intH), H_{eps^-1} = -H_eps): u = +2 T_w x
    const double sg = P->kind == VIE_LAPLACE ? -2.0 : 2.0;
    ca.narr = 6;
    for (int a = 0; a < 6; ++a) {
      ca.set(a, 0, Q[a], make_double2(sg * nrm, 0));
    }
    if (which == 0) {
      s = combine(P, P->kapply, KM_SYM3, ca, sg * 0.5 * nrm, 0x7, st);
      if (s != VIE_OK) return s;
    }
    // phi_sc = div V J
    ce.narr = 3;
    for (int a = 0; a < 3; ++a) {
      ce.set(a, 0, Dd[a], make_double2(nrm, 0));
    }
    if (which == 1) {
      s = combine(P, P->keval, KM_DIV, ce, 0.0, 0, st);
      if (s != VIE_OK) return s;
    }
  } else {
    // Maxwell (Eq. (eq:intM)): u_J = Q' J + P' x M, u_M = Q' M - P' x J with
    // Q' = -2 (K + I/2 + w^2 V), P'_a = -2 i w K_{i k_a}.
    ca.narr = P->has_mu ? 9 : 6;
    for (int a = 0; a < 6; ++a) {
      ca.set(a, 0, Q[a], make_double2(-2.0 * nrm, 0));
      if (a < 3) {
        ca.set(a, 1, SYM_1, make_double2(-2.0 * w2 * nrm, 0));
      }
    }
    for (int a = 0; a < 3; ++a) {
      ca.set(6 + a, 0, Dd[a], make_double2(0, -2.0 * w * nrm));
    }
    if (which == 0) {
      s = combine(P, P->kapply, P->has_mu ? KM_MAXWELL6 : KM_SYM3, ca, -nrm, 0x7, st);
      if (s != VIE_OK) return s;
    }
    // E_sc = Q'' J + P'' x M, H_sc = Q'' M - P'' x J; Q'' = K + w^2 V, P''_a = i w K_{i k_a}
    ce.narr = 9;
    for (int a = 0; a < 6; ++a) {
      ce.set(a, 0, Q[a], make_double2(nrm, 0));
      if (a < 3) {
        ce.set(a, 1, SYM_1, make_double2(w2 * nrm, 0));
      }
    }
    for (int a = 0; a < 3; ++a) {
      ce.set(6 + a, 0, Dd[a], make_double2(0, w * nrm));
    }
    if (which == 1) {
      s = combine(P, P->keval, P->has_mu ? KM_MAXWELL6 : KM_EMRED, ce, 0.0, 0, st);
      if (s != VIE_OK) return s;
    }
  }
  VIE_CK(cudaStreamSynchronize(st));
  return VIE_OK;
}

// ------------------------------------------------------------ double-word copies
// v -> (hi, lo) with hi = fl32(v), lo = fl32(v - hi): the double-word value
// equals v to about 2^-48 relative.
__global__ void k_to_df(const double2* __restrict__ src, cdf* __restrict__ dst, long long count) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x) {
    const double2 v = src[i];
    dst[i] = CT<df>::make(df(v.x), df(v.y));
  }
}

static vie_status to_df(const double2* src, cdf** dst, long long count, cudaStream_t st) {
  VIE_CK(dalloc((void**)dst, sizeof(cdf) * (size_t)count, st));
  const long long blocks = std::min<long long>((count + 255) / 256, 4096);
  k_to_df<<<(unsigned)blocks, 256, 0, st>>>(src, *dst, count);
  VIE_CK(cudaGetLastError());
  return VIE_OK;
}

vie_status build_df(vie_problem* P, cudaStream_t st) {
  if (P->kapply.octdf) return VIE_OK;
  const long long N = (long long)P->n * P->n * P->n;
  const long long O3 = (long long)(P->nk + 1) * (P->nk + 1) * (P->nk + 1);
  vie_status s = VIE_OK;
  if (!P->twdf) s = to_df(P->tw64, &P->twdf, line_table_len(P->planM), st);
  if (s == VIE_OK && !P->Hedf) s = to_df(P->He64, &P->Hedf, 6 * N, st);
  if (s == VIE_OK && P->Hm64 && !P->Hmdf) s = to_df(P->Hm64, &P->Hmdf, 6 * N, st);
  if (s == VIE_OK) s = to_df(P->kapply.oct64, &P->kapply.octdf, (long long)P->kapply.narr * O3, st);
  return s;
}

}  // namespace vie
