// Five passes of the operator apply on two-step line transforms of any length
// M = R1 R2 with R1, R2 codelet radices (4 <= R2 <= R1 <= 24): the general kernels
// of every grid without register-resident ones of its own, in all three
// arithmetics (the shared-memory Stockham passes of apply.cu remain for the
// lengths without such a split).
//
//   forward  X[k1 + R1 k2] = sum_n2 W_R2^{n2 k2} W_M^{n2 k1} sum_n1 W_R1^{n1 k1} x[R2 n1 + n2]
//   inverse  the mirror image, R2 points first
//
// as in vie_fft2.cuh, but with R1 and R2 chosen at run time: each step switches
// once to the codelet of its radix.  A value crosses shared memory once per
// transform (written by step 1 as it comes from global memory, read by step 2 on
// its way back), where the Stockham passes move it there and back once per stage
// and once more at either end: 2 crossings instead of 10 at M = 300 = 4 3 5 5.
// The z pass keeps its spectra in place (every task owns the row or column it
// reads), so one line buffer serves the forward transform, the kernel mixing and
// the inverse.
//
// Measured against the Stockham passes (whole apply): FP32 reduced Maxwell 70^3
// 271 -> 136 us, 150^3 2.57 -> 1.01 ms, 220^3 8.46 -> 3.15 ms; FP64 Helmholtz 70^3
// 2.54 -> 1.91 ms; double-word 64^3 0.54 -> 0.44, 96^3 1.44 -> 1.10 ms (the same
// arithmetic on both sides; 0.46 and 1.17 ms with today's).  FP32 at 150^3: the x and y
// passes move their bytes at 3.8 to 4.5 TB/s; the z pass (0.57 ms) issues 55 % of the
// cycles at 24 warps an SM, waiting in equal parts for its barriers, its loads and FP32
// latencies.  FP64 passes keep the FP64 pipe 81 - 84 % busy (70^3), the double-word z
// pass the FP32 pipe 63 % (96^3).
#pragma once

#include <type_traits>

#include "vie_fft2.cuh"
#include "vie_internal.h"

namespace vie {

struct TwoPlan {
  int M, R1, R2;
  int PF;  // row pitch of a line in shared memory: odd, so that rows fall on different banks
};

// Radices with a codelet in the run-time switches.
constexpr bool two_radix(int r) { return r >= 4 && r <= 24 && r != 13 && r != 17 && r != 19 && r != 23; }

// The most balanced split with R1 >= R2.
constexpr bool make_two_plan(int M, TwoPlan* p) {
  for (int r2 = 24; r2 >= 4; --r2) {
    if (r2 * r2 > M || M % r2 || !two_radix(r2) || !two_radix(M / r2) || (M / r2 > 16 && r2 < 9)) continue;
    p->M = M;
    p->R1 = M / r2;
    p->R2 = r2;
    p->PF = r2 | 1;
    return true;
  }
  return false;
}

constexpr bool has_two_plan(int M) {
  TwoPlan p{};
  return make_two_plan(M, &p);
}

// Whether the z pass has a two-step kernel for M: all but the double-word one
// above radix 16, which exists on half lines only.
inline bool two_z_fits(const TwoPlan& p, bool dw) {
  TwoPlan h;
  return !dw || p.R1 <= 16 || (make_two_plan(p.M / 2, &h) && h.R1 <= 16);
}

// Line pitch for tiles whose lanes run over `nl` lines first: the lanes of one
// 128-byte access fall on distinct banks when the pitch is odd (16 lines of 8
// bytes, 8 of 16) or 2 modulo the lanes of an access (half as many lines, two rows).
inline int two_pitch(const TwoPlan& p, int nl, size_t esz) {
  const int lanes = 128 / (int)esz, len = p.R1 * p.PF;
  return nl >= lanes ? (len | 1) : (len + lanes - 3) / lanes * lanes + 2;
}

// f(integral_constant<R>) for a run-time radix of class RM: 16 (both radices at most
// 16), 24 (R1 above 16; R2 is then at least 9 for every length split here), or 0
// (any).  Step FIRST is the one of R1.
template <int RM, bool FIRST, typename F>
__device__ __forceinline__ void radix_switch(int R, F&& f) {
#define VIE_RADIX(r) case r: f(std::integral_constant<int, r>{}); return;
  if constexpr (RM != 24) {
    switch (R) {
      VIE_RADIX(4) VIE_RADIX(5) VIE_RADIX(6) VIE_RADIX(7) VIE_RADIX(8)
      default: break;
    }
  }
  if constexpr (RM != 24 || !FIRST) {
    switch (R) {
      VIE_RADIX(9) VIE_RADIX(10) VIE_RADIX(11) VIE_RADIX(12) VIE_RADIX(14) VIE_RADIX(15) VIE_RADIX(16)
      default: break;
    }
  }
  if constexpr (RM != 16) {
    switch (R) {
      VIE_RADIX(18) VIE_RADIX(20) VIE_RADIX(21) VIE_RADIX(22) VIE_RADIX(24)
      default: break;
    }
  }
#undef VIE_RADIX
}

// Zero-padded lines: dft_half_in and dft_half_out beat the whole codelet for the
// power-of-two radices (the others have no twiddles to save).
template <int R> constexpr bool kHalf = (R == 8 || R == 16);

template <int R, typename T>
__device__ __forceinline__ void two_dft_in(typename CT<T>::V* u) {
  if constexpr (kHalf<R>) dft_half_in<R, -1, T>(u);
  else Dft<R, -1, T>::run(u);
}
template <int R, typename T>
__device__ __forceinline__ void two_dft_out(typename CT<T>::V* u) {
  if constexpr (kHalf<R>) dft_half_out<R, +1, T>(u);
  else Dft<R, +1, T>::run(u);
}

// Step 1 forward of one task (line s, n2): u[n1] = ld(R2 n1 + n2), zero from n1 = R1/2 on.
template <int RM, typename T, typename LD>
__device__ __forceinline__ void two_fwd1(const TwoPlan& p, int n2, typename CT<T>::V* s,
                                         const typename CT<T>::V* tw, LD&& ld) {
  typedef typename CT<T>::V V;
  radix_switch<RM, true>(p.R1, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    V u[R];
#pragma unroll
    for (int i = 0; i < R; ++i) u[i] = i < (R + 1) / 2 ? ld(p.R2 * i + n2) : CT<T>::make(0, 0);
    two_dft_in<R, T>(u);
    s[n2] = u[0];
#pragma unroll
    for (int i = 1; i < R; ++i) s[i * p.PF + n2] = cmul(u[i], tw[n2 * i]);
  });
}
// Step 2 forward of one task (line s, k1): st(k2, X[k1 + R1 k2]).
template <int RM, typename T, typename ST>
__device__ __forceinline__ void two_fwd2(const TwoPlan& p, int k1, const typename CT<T>::V* s, ST&& st) {
  typedef typename CT<T>::V V;
  radix_switch<RM, false>(p.R2, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    V u[R];
#pragma unroll
    for (int i = 0; i < R; ++i) u[i] = s[k1 * p.PF + i];
    Dft<R, -1, T>::run(u);
#pragma unroll
    for (int i = 0; i < R; ++i) st(i, u[i]);
  });
}
// Step A inverse of one task (line s, k1): u[k2] = ld(k2).
template <int RM, typename T, typename LD>
__device__ __forceinline__ void two_invA(const TwoPlan& p, int k1, typename CT<T>::V* s,
                                         const typename CT<T>::V* tw, LD&& ld) {
  typedef typename CT<T>::V V;
  radix_switch<RM, false>(p.R2, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    V u[R];
#pragma unroll
    for (int i = 0; i < R; ++i) u[i] = ld(i);
    Dft<R, +1, T>::run(u);
    s[k1 * p.PF] = u[0];
#pragma unroll
    for (int i = 1; i < R; ++i) s[k1 * p.PF + i] = cmulc(u[i], tw[k1 * i]);
  });
}
// Step B inverse of one task (line s, n2): st(n1, x[R2 n1 + n2]) for n1 < (R1 + 1)/2, the
// outputs that can lie below M/2.
template <int RM, typename T, typename ST>
__device__ __forceinline__ void two_invB(const TwoPlan& p, int n2, const typename CT<T>::V* s, ST&& st) {
  typedef typename CT<T>::V V;
  radix_switch<RM, true>(p.R1, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    V u[R];
#pragma unroll
    for (int i = 0; i < R; ++i) u[i] = s[i * p.PF + n2];
    two_dft_out<R, T>(u);
#pragma unroll
    for (int i = 0; i < (R + 1) / 2; ++i) st(i, u[i]);
  });
}

template <typename V>
__device__ __forceinline__ void two_twiddles(V* tw, const V* __restrict__ twg, int M) {
  const int nt = blockDim.x * blockDim.y * blockDim.z;
  for (int j = (threadIdx.z * blockDim.y + threadIdx.y) * blockDim.x + threadIdx.x; j < M; j += nt) tw[j] = twg[j];
}

// P1, x-lines: block (R1, rows), lanes along the line.
template <typename T, int RM>
__global__ void __launch_bounds__(256) k2_p1(const typename IOT<T>::E* __restrict__ x, typename CT<T>::V* __restrict__ A,
                                             int n, TwoPlan p, int LS, int C,
                                             const typename CT<T>::V* __restrict__ twg) {
  after_previous();
  typedef typename CT<T>::V V;
  extern __shared__ __align__(16) unsigned char smraw[];
  V* tw = (V*)smraw;
  V* sm = tw + p.M;
  two_twiddles(tw, twg, p.M);
  const int rows = n * n, r0 = blockIdx.x * blockDim.y;
  const int c = blockIdx.y, b = blockIdx.z, nc = gridDim.y;
  __syncthreads();
  {  // step 1: (row, n2) packed densely into the warps
    const int t = threadIdx.y * blockDim.x + threadIdx.x, l = t / p.R2, n2 = t - l * p.R2;
    const bool ok = r0 + l < rows;
    const typename IOT<T>::E* src = x + (((long long)b * nc + c) * rows + r0 + l) * n;
    if (l < blockDim.y)
      two_fwd1<RM, T>(p, n2, sm + l * LS, tw,
                      [&](int j) { return ok && j < n ? to_v<T>(src[j]) : CT<T>::make(0, 0); });
  }
  __syncthreads();
  const int i = threadIdx.x, row = r0 + threadIdx.y;
  V* dst = A + (((long long)b * C + c) * rows + row) * p.M + i;
  if (row < rows) two_fwd2<RM, T>(p, i, sm + threadIdx.y * LS, [&](int k2, V v) { dst[p.R1 * k2] = v; });
}

// P2 (S < 0) and P4 (S > 0), y-lines: block (nl, R1), lanes along kx.
template <typename T, int RM, int S>
__global__ void __launch_bounds__(sizeof(typename CT<T>::V) == 8 ? 384 : 192, 2)
k2_py(const typename CT<T>::V* __restrict__ in, typename CT<T>::V* __restrict__ out, int n, TwoPlan p, int LS, int C,
      int ncomp, const typename CT<T>::V* __restrict__ twg) {
  after_previous();
  typedef typename CT<T>::V V;
  extern __shared__ __align__(16) unsigned char smraw[];
  V* tw = (V*)smraw;
  V* s = tw + p.M + threadIdx.x * LS;
  two_twiddles(tw, twg, p.M);
  const int M = p.M, kx = blockIdx.x * blockDim.x + threadIdx.x, z = blockIdx.y, i = threadIdx.y;
  const bool ok = kx < M;
  const int b = blockIdx.z / ncomp, c = blockIdx.z - b * ncomp;
  const long long plane = ((long long)b * C + c) * n + z;
  const V* src = in + plane * (long long)(S < 0 ? n : M) * M + kx;
  V* dst = out + plane * (long long)(S < 0 ? M : n) * M + kx;
  __syncthreads();
  if (S < 0) {
    if (i < p.R2)
      two_fwd1<RM, T>(p, i, s, tw, [&](int j) { return ok && j < n ? src[(long long)j * M] : CT<T>::make(0, 0); });
    __syncthreads();
    if (ok) two_fwd2<RM, T>(p, i, s, [&](int k2, V v) { dst[(long long)(i + p.R1 * k2) * M] = v; });
  } else {
    two_invA<RM, T>(p, i, s, tw,
                    [&](int k2) { return ok ? src[(long long)(i + p.R1 * k2) * M] : CT<T>::make(0, 0); });
    __syncthreads();
    if (ok && i < p.R2)
      two_invB<RM, T>(p, i, s, [&](int n1, V v) {
        const int y = p.R2 * n1 + i;
        if (y < n) dst[(long long)y * M] = v;
      });
  }
}

// acc + a b, in FP32 and FP64 as four FMAs.
template <typename V>
__device__ __forceinline__ V cmac(V acc, V a, V b) { return acc + cmul(a, b); }
template <>
__device__ __forceinline__ double2 cmac(double2 acc, double2 a, double2 b) {
  return make_double2(fma(-a.y, b.y, fma(a.x, b.x, acc.x)), fma(a.y, b.x, fma(a.x, b.y, acc.y)));
}
template <>
__device__ __forceinline__ float2 cmac(float2 acc, float2 a, float2 b) {
  return make_float2(fmaf(-a.y, b.y, fmaf(a.x, b.x, acc.x)), fmaf(a.y, b.x, fmaf(a.x, b.y, acc.y)));
}

// Kernel mixing at one frequency: u (cin spectra) -> o (cout), q the kernel values.
template <typename V>
__device__ __forceinline__ void mix_point(int mode, const V* u, const V* q, V* o) {
  if (mode == KM_DIV) {
    o[0] = cmac(cmac(cmul(q[0], u[0]), q[1], u[1]), q[2], u[2]);
    return;
  }
  // symmetric 3x3: xx yy zz xy xz yz
  o[0] = cmac(cmac(cmul(q[0], u[0]), q[3], u[1]), q[4], u[2]);
  o[1] = cmac(cmac(cmul(q[3], u[0]), q[1], u[1]), q[5], u[2]);
  o[2] = cmac(cmac(cmul(q[4], u[0]), q[5], u[1]), q[2], u[2]);
  if (mode == KM_SYM3) return;
  const V m0 = vneg(q[6]), m1 = vneg(q[7]), m2 = vneg(q[8]);
  if (mode == KM_EMRED) {  // - P x J
    o[3] = cmac(cmul(q[8], u[1]), m1, u[2]);
    o[4] = cmac(cmul(q[6], u[2]), m2, u[0]);
    o[5] = cmac(cmul(q[7], u[0]), m0, u[1]);
  } else {  // Q J + P x M, Q M - P x J
    o[3] = cmac(cmac(cmac(cmac(cmul(q[0], u[3]), q[3], u[4]), q[4], u[5]), m1, u[2]), q[8], u[1]);
    o[4] = cmac(cmac(cmac(cmac(cmul(q[3], u[3]), q[1], u[4]), q[5], u[5]), m2, u[0]), q[6], u[2]);
    o[5] = cmac(cmac(cmac(cmac(cmul(q[4], u[3]), q[5], u[4]), q[2], u[5]), m0, u[1]), q[7], u[0]);
    o[0] = cmac(cmac(o[0], q[7], u[5]), m2, u[4]);
    o[1] = cmac(cmac(o[1], q[8], u[3]), m0, u[5]);
    o[2] = cmac(cmac(o[2], q[6], u[4]), m1, u[3]);
  }
}

// P3, z-pencils: block (nl, R1, TZ), lanes along kx, the TZ thread slices taking
// the components in turn; lines of component c and pencil l at (c nl + l) LS.
// The mixing takes kz and M - kz together (one read of the octant's values for
// both), and the CTAs of the rows ky and M - ky, which read the same octant
// values, are neighbours in launch order so that those come from L2.
// MODE -1: a kernel for both operator sets, told apart at run time (the
// double-word codelets are long to compile; FP32 and FP64 have one per set).
template <typename T, int RM, int MODE> struct TwoP3 {
  static constexpr int NL = sizeof(typename CT<T>::V) == 8 ? 8 : 4;
  // thread slices: three (of one or two components each), one a component in
  // double-word arithmetic: the warps they bring hide the latencies
  static constexpr int TZ = MODE < 0 ? 6 : 3;
  static constexpr int N = NL * RM * TZ;
  static constexpr int MINB = RM > 16 || MODE < 0 ? 1 : 2;
};
template <typename T, int RM, int MODE>
__global__ void __launch_bounds__(TwoP3<T, RM, MODE>::N, TwoP3<T, RM, MODE>::MINB)
k2_p3(typename CT<T>::V* __restrict__ B, int n, TwoPlan p, int LS, int C, int mode_rt,
      const typename CT<T>::V* __restrict__ K, const typename CT<T>::V* __restrict__ twg) {
  after_previous();
  typedef typename CT<T>::V V;
  const int mode = MODE < 0 ? mode_rt : MODE;
  const int CI = mode == KM_MAXWELL6 ? 6 : 3, CO = mode == KM_SYM3 ? 3 : (mode == KM_DIV ? 1 : 6);
  const int NARR = mode == KM_SYM3 ? 6 : (mode == KM_DIV ? 3 : 9);
  extern __shared__ __align__(16) unsigned char smraw[];
  const int M = p.M, R1 = p.R1, R2 = p.R2, nk = M / 2, nl = blockDim.x;
  V* tw = (V*)smraw;
  V* sm = tw + M + threadIdx.x * LS;
  const int cs_sm = nl * LS;  // shared-memory stride of a component
  const int nt = (M + nl - 1) / nl, g = blockIdx.x >> 1, kyp = g / nt;
  if ((blockIdx.x & 1) && (kyp == 0 || kyp == nk)) return;  // rows that mirror onto themselves
  const int ky = (blockIdx.x & 1) ? M - kyp : kyp, kx = (g - kyp * nt) * nl + threadIdx.x;
  const bool ok = kx < M;
  two_twiddles(tw, twg, M);
  const int i = threadIdx.y, cz = threadIdx.z, TZ = blockDim.z;
  const long long zs = (long long)M * M, cs = (long long)n * zs;
  V* base = B + (long long)blockIdx.y * C * cs + (long long)ky * M + kx;
  __syncthreads();
  if (i < R2)
    for (int c = cz; c < CI; c += TZ)
      two_fwd1<RM, T>(p, i, sm + c * cs_sm, tw,
                      [&](int z) { return ok && z < n ? base[c * cs + z * zs] : CT<T>::make(0, 0); });
  __syncthreads();
  for (int c = cz; c < CI; c += TZ) {
    V* row = sm + c * cs_sm + i * p.PF;
    two_fwd2<RM, T>(p, i, sm + c * cs_sm, [&](int k2, V v) { row[k2] = v; });
  }
  __syncthreads();
  {
    const int O = nk + 1;
    const long long O3 = (long long)O * O * O;
    const bool fy = ky > nk, fx = kx > nk;
    const V* kp = K + (long long)(fy ? M - ky : ky) * O + (ok ? (fx ? M - kx : kx) : 0);
    V q[9], qn[9];  // kernel values of this step, and of the next one on their way
    auto fetch = [&](int k2) {
      const long long kz = i + R1 * k2;
      if (kz > nk) return;
#pragma unroll
      for (int a = 0; a < 9; ++a)
        if (a < NARR) qn[a] = kp[a * O3 + kz * O * O];
    };
    fetch(cz);
    for (int k2 = cz; i + R1 * k2 <= nk; k2 += TZ) {
      const int kz = i + R1 * k2;
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        if (a >= NARR) break;
        const int par = sym_parity(mode == KM_DIV ? 6 + a : a);
        q[a] = (((par & 2) && fy) != ((par & 1) && fx)) ? vneg(qn[a]) : qn[a];
      }
      fetch(k2 + TZ);
      auto point = [&](int pos) {
        V u[6], o[6];
#pragma unroll
        for (int c = 0; c < 6; ++c)
          if (c < CI) u[c] = sm[c * cs_sm + pos];
        mix_point(mode, u, q, o);
#pragma unroll
        for (int c = 0; c < 6; ++c)
          if (c < CO) sm[c * cs_sm + pos] = o[c];
      };
      point(i * p.PF + k2);
      if (kz > 0 && 2 * kz != M) {  // M - kz, where the arrays odd in z change sign
#pragma unroll
        for (int a = 0; a < 9; ++a)
          if (a < NARR && (sym_parity(mode == KM_DIV ? 6 + a : a) & 4)) q[a] = vneg(q[a]);
        point(i == 0 ? R2 - k2 : (R1 - i) * p.PF + R2 - 1 - k2);
      }
    }
  }
  __syncthreads();
  for (int c = cz; c < CO; c += TZ) {
    V* row = sm + c * cs_sm + i * p.PF;
    two_invA<RM, T>(p, i, sm + c * cs_sm, tw, [&](int k2) { return row[k2]; });
  }
  __syncthreads();
  if (ok && i < R2)
    for (int c = cz; c < CO; c += TZ)
      two_invB<RM, T>(p, i, sm + c * cs_sm, [&](int n1, V v) {
        const int z = R2 * n1 + i;
        if (z < n) base[c * cs + z * zs] = v;
      });
}

// P3 on half lines, for M = 2 nk with nk = R1 R2 and radices up to 16 where M
// itself would need larger ones.  Only z < n <= nk of a pencil is nonzero, so with
// w = exp(-2 pi i / M) its spectrum splits by the parity r of the frequency,
//   X[2k + r] = sum_{z < nk} (x[z] w^{r z}) W_nk^{z k},
// two transforms of length nk without a zero in them (a radix-20 step of the
// direct split works on ten zeros), the inverse is the sum of the two inverses
// with the odd one twisted back, and the partner M - kz of a frequency is in the
// same half.  Block (nl, R1, TZ) and lines as in k2_p3; the halves of component c
// and pencil l at ((2 c + r) nl + l) LS; p is the split of nk, twg the table of M.
template <typename T, int MODE>
__global__ void __launch_bounds__(TwoP3<T, 16, MODE>::N, TwoP3<T, 16, MODE>::MINB)
k2_p3h(typename CT<T>::V* __restrict__ B, int n, TwoPlan p, int LS, int C, int mode_rt,
       const typename CT<T>::V* __restrict__ K, const typename CT<T>::V* __restrict__ twg) {
  after_previous();
  typedef typename CT<T>::V V;
  const int mode = MODE < 0 ? mode_rt : MODE;
  const int CI = mode == KM_MAXWELL6 ? 6 : 3, CO = mode == KM_SYM3 ? 3 : (mode == KM_DIV ? 1 : 6);
  const int NARR = mode == KM_SYM3 ? 6 : (mode == KM_DIV ? 3 : 9);
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nk = p.M, M = 2 * nk, R1 = p.R1, R2 = p.R2, nl = blockDim.x;
  V* tw = (V*)smraw;
  V* sm = tw + M + threadIdx.x * LS;
  const int hs = nl * LS;  // shared-memory stride of a half
  const int nt = (M + nl - 1) / nl, g = blockIdx.x >> 1, kyp = g / nt;
  if ((blockIdx.x & 1) && (kyp == 0 || kyp == nk)) return;  // rows that mirror onto themselves
  const int ky = (blockIdx.x & 1) ? M - kyp : kyp, kx = (g - kyp * nt) * nl + threadIdx.x;
  const bool ok = kx < M;
  two_twiddles(tw, twg, M);
  const int i = threadIdx.y, cz = threadIdx.z, TZ = blockDim.z;
  const long long zs = (long long)M * M, cs = (long long)n * zs;
  V* base = B + (long long)blockIdx.y * C * cs + (long long)ky * M + kx;
  __syncthreads();
  if (i < R2)
    radix_switch<16, true>(R1, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for (int c = cz; c < CI; c += TZ) {
        V* s = sm + 2 * c * hs + i;
#pragma unroll 1
        for (int r = 0; r < 2; ++r, s += hs) {  // the second reading of the inputs comes from L1
          V u[R];
#pragma unroll
          for (int k = 0; k < R; ++k) {
            const int z = R2 * k + i;
            u[k] = ok && z < n ? base[c * cs + z * zs] : CT<T>::make(0, 0);
          }
          if (r) {
#pragma unroll
            for (int k = 0; k < R; ++k) u[k] = cmul(u[k], tw[R2 * k + i]);
          }
          Dft<R, -1, T>::run(u);
          s[0] = u[0];
#pragma unroll
          for (int k = 1; k < R; ++k) s[k * p.PF] = cmul(u[k], tw[2 * i * k]);
        }
      }
    });
  __syncthreads();
  for (int h = 2 * cz; h < 2 * CI; h += (h & 1) ? 2 * TZ - 1 : 1) {
    V* row = sm + h * hs + i * p.PF;
    two_fwd2<16, T>(p, i, sm + h * hs, [&](int k2, V v) { row[k2] = v; });
  }
  __syncthreads();
  {
    const int O = nk + 1;
    const long long O3 = (long long)O * O * O;
    const bool fy = ky > nk, fx = kx > nk;
    const V* kp = K + (long long)(fy ? M - ky : ky) * O + (ok ? (fx ? M - kx : kx) : 0);
    V q[9], qn[9];  // kernel values of this step, and of the next one on their way
    // frequency of step t: half t & 1, column t >> 1
    auto freq = [&](int t) { return 2 * (i + R1 * (t >> 1)) + (t & 1); };
    auto fetch = [&](int t) {
      const long long kz = freq(t);
      if (kz > nk) return;
#pragma unroll
      for (int a = 0; a < 9; ++a)
        if (a < NARR) qn[a] = kp[a * O3 + kz * O * O];
    };
    fetch(cz);
    for (int t = cz; freq(t) <= nk; t += TZ) {
      const int r = t & 1, k2 = t >> 1, kz = freq(t);
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        if (a >= NARR) break;
        const int par = sym_parity(mode == KM_DIV ? 6 + a : a);
        q[a] = (((par & 2) && fy) != ((par & 1) && fx)) ? vneg(qn[a]) : qn[a];
      }
      fetch(t + TZ);
      auto point = [&](int pos) {
        V u[6], o[6];
#pragma unroll
        for (int c = 0; c < 6; ++c)
          if (c < CI) u[c] = sm[(2 * c + r) * hs + pos];
        mix_point(mode, u, q, o);
#pragma unroll
        for (int c = 0; c < 6; ++c)
          if (c < CO) sm[(2 * c + r) * hs + pos] = o[c];
      };
      point(i * p.PF + k2);
      if (kz > 0 && kz < nk) {  // M - kz, where the arrays odd in z change sign
#pragma unroll
        for (int a = 0; a < 9; ++a)
          if (a < NARR && (sym_parity(mode == KM_DIV ? 6 + a : a) & 4)) q[a] = vneg(q[a]);
        point(r ? (R1 - 1 - i) * p.PF + R2 - 1 - k2 : (i == 0 ? R2 - k2 : (R1 - i) * p.PF + R2 - 1 - k2));
      }
    }
  }
  __syncthreads();
  for (int h = 2 * cz; h < 2 * CO; h += (h & 1) ? 2 * TZ - 1 : 1) {
    V* row = sm + h * hs + i * p.PF;
    radix_switch<16, false>(R2, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      V u[R];
#pragma unroll
      for (int k = 0; k < R; ++k) u[k] = row[k];
      Dft<R, +1, T>::run(u);
      row[0] = u[0];
#pragma unroll
      for (int k = 1; k < R; ++k) row[k] = cmulc(u[k], tw[2 * i * k]);
    });
  }
  __syncthreads();
  if (ok && i < R2)
    radix_switch<16, true>(R1, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for (int c = cz; c < CO; c += TZ) {
        V* s = sm + 2 * c * hs + i;
        V u[R];
#pragma unroll
        for (int k = 0; k < R; ++k) u[k] = s[hs + k * p.PF];
        Dft<R, +1, T>::run(u);
        // the twisted odd half waits in the column it came from
#pragma unroll
        for (int k = 0; k < R; ++k) s[hs + k * p.PF] = cmulc(u[k], tw[R2 * k + i]);
#pragma unroll
        for (int k = 0; k < R; ++k) u[k] = s[k * p.PF];
        Dft<R, +1, T>::run(u);
#pragma unroll
        for (int k = 0; k < R; ++k) {
          const int z = R2 * k + i;
          if (z < n) base[c * cs + z * zs] = u[k] + s[hs + k * p.PF];
        }
      }
    });
}

// P5, x-lines of all components: block (R1, rows, TZ); the inverse leaves x[R2 n1 +
// n2] at row n1, column n2 of its line (each step-B task owns its column), then
// the epilogue of f_p5 runs node by node.
template <typename T, int RM>
__global__ void __launch_bounds__(256, sizeof(typename CT<T>::V) == 8 ? 2 : 1) k2_p5(const typename CT<T>::V* __restrict__ A,
                                             const typename IOT<T>::E* __restrict__ xin,
                                             typename IOT<T>::E* __restrict__ y, int n, TwoPlan p, int LS, int C, int cout,
                                             const typename CT<T>::V* __restrict__ He,
                                             const typename CT<T>::V* __restrict__ Hm, int with_identity,
                                             const typename CT<T>::V* __restrict__ twg) {
  after_previous();
  typedef typename CT<T>::V V;
  typedef typename IOT<T>::E E;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int M = p.M, nr = blockDim.y, i = threadIdx.x, cz = threadIdx.z, TZ = blockDim.z;
  V* tw = (V*)smraw;
  V* sm = tw + M + threadIdx.y * LS;  // component c of this row at sm + c nr LS
  two_twiddles(tw, twg, M);
  const int rows = n * n, row = blockIdx.x * nr + threadIdx.y, b = blockIdx.y;
  const bool ok = row < rows;
  const long long N = (long long)rows * n, cs = (long long)rows * M;
  const V* src = A + (long long)b * C * cs + (long long)row * M;
  __syncthreads();
  for (int c = cz; c < cout; c += TZ)
    two_invA<RM, T>(p, i, sm + c * nr * LS, tw,
                    [&](int k2) { return ok ? src[c * cs + i + p.R1 * k2] : CT<T>::make(0, 0); });
  __syncthreads();
  {  // step B: (row, n2) packed densely into the warps
    const int t = threadIdx.y * blockDim.x + i, l = t / p.R2, n2 = t - l * p.R2;
    if (l < nr)
      for (int c = cz; c < cout; c += TZ) {
        V* s = tw + M + (c * nr + l) * LS;
        two_invB<RM, T>(p, n2, s, [&](int n1, V v) { s[n1 * p.PF + n2] = v; });
      }
  }
  __syncthreads();
  if (!ok) return;
  for (int xx = i + p.R1 * cz; xx < n; xx += p.R1 * TZ) {
    const int q = xx / p.R2, pos = q * p.PF + xx - q * p.R2;
    const long long pt = (long long)row * n + xx;
    if (!with_identity) {
      for (int c = 0; c < cout; ++c) y[((long long)b * cout + c) * N + pt] = from_v<T>(sm[c * nr * LS + pos]);
      continue;
    }
    for (int blk = 0; blk < cout / 3; ++blk) {
      const V* H = blk == 0 ? He : Hm;
      const V hxx = H[pt], hyy = H[N + pt], hzz = H[2 * N + pt];
      const V hxy = H[3 * N + pt], hxz = H[4 * N + pt], hyz = H[5 * N + pt];
      const E* xi = xin + ((long long)b * cout + 3 * blk) * N + pt;
      E* yo = y + ((long long)b * cout + 3 * blk) * N + pt;
      const V a0 = sm[(3 * blk) * nr * LS + pos], a1 = sm[(3 * blk + 1) * nr * LS + pos],
              a2 = sm[(3 * blk + 2) * nr * LS + pos];
      if (with_identity == 1) {
        yo[0] = add_id<T>(xi[0], cmul(hxx, a0), cmul(hxy, a1), cmul(hxz, a2));
        yo[N] = add_id<T>(xi[N], cmul(hxy, a0), cmul(hyy, a1), cmul(hyz, a2));
        yo[2 * N] = add_id<T>(xi[2 * N], cmul(hxz, a0), cmul(hyz, a1), cmul(hzz, a2));
      } else {  // 2: H u alone
        yo[0] = from_v<T>(cmul(hxx, a0) + cmul(hxy, a1) + cmul(hxz, a2));
        yo[N] = from_v<T>(cmul(hxy, a0) + cmul(hyy, a1) + cmul(hyz, a2));
        yo[2 * N] = from_v<T>(cmul(hxz, a0) + cmul(hyz, a1) + cmul(hzz, a2));
      }
    }
  }
}

// Arguments of a pass; every pointer as in apply.cu.
struct TwoArgs {
  int n, mode, C, cin, cout, nrhs, with_identity;
  const void *x, *He, *Hm, *K, *tw;
  void *y, *A, *B;
};

template <typename V>
inline size_t two_smem(const TwoPlan& p, size_t lines, int LS) { return sizeof(V) * (p.M + lines * LS); }

// P1, P2 and P4 on plan p.
template <typename T, int RM>
vie_status two_line_pass(int pass, const TwoPlan& p, const TwoArgs& a, cudaStream_t st) {
  typedef typename CT<T>::V V;
  const int n = a.n, M = p.M;
  const V* tw = (const V*)a.tw;
  if (pass == 1) {
    const int rows = std::max(1, 256 / p.R1), LS = (p.R1 * p.PF) | 1;
    VIE_CK(allow_smem(k2_p1<T, RM>));
    VIE_CK(launch_after<kOverlap<T>>(k2_p1<T, RM>, dim3((n * n + rows - 1) / rows, a.cin, a.nrhs), dim3(p.R1, rows), two_smem<V>(p,
                        rows, LS), st, (const typename IOT<T>::E*)a.x, (V*)a.A, n, p, LS, a.C, tw));
  } else {
    const int nl = sizeof(V) == 8 ? 16 : 8, LS = two_pitch(p, nl, sizeof(V)), nc = pass == 2 ? a.cin : a.cout;
    const dim3 grid((M + nl - 1) / nl, n, a.nrhs * nc), blk(nl, p.R1);
    if (pass == 2) {
      VIE_CK(allow_smem(k2_py<T, RM, -1>));
      VIE_CK(launch_after<kOverlap<T>>(k2_py<T, RM, -1>, grid, blk, two_smem<V>(p, nl, LS), st, (const V*)a.A, (V*)a.B, n, p, LS,
                          a.C, nc, tw));
    } else {
      VIE_CK(allow_smem(k2_py<T, RM, 1>));
      VIE_CK(launch_after<kOverlap<T>>(k2_py<T, RM, 1>, grid, blk, two_smem<V>(p, nl, LS), st, (const V*)a.B, (V*)a.A, n, p, LS,
                          a.C, nc, tw));
    }
  }
  VIE_CK(cudaGetLastError());
  return VIE_OK;
}

template <typename T, int RM>
vie_status two_z_pass(const TwoPlan& p, const TwoArgs& a, cudaStream_t st) {
  typedef typename CT<T>::V V;
  TwoPlan h = p;
  bool half = RM > 16 && make_two_plan(p.M / 2, &h) && h.R1 <= 16;
  auto smem_of = [&](int nl) {
    return sizeof(V) * (p.M + (size_t)a.C * (half ? 2 : 1) * nl * two_pitch(h, nl, sizeof(V)));
  };
  // FP32 with six lines a pencil: half lines only while two CTAs share an SM (100^3
  // with mu 299 us against 383, 150^3 1640 against 1080)
  if (half && sizeof(V) == 8 && a.C == 6 && smem_of(TwoP3<T, RM, KM_SYM3>::NL) > 112 * 1024) half = false;
  if (!half) h = p;
  if (std::is_same<T, df>::value && RM > 16 && !half) return VIE_EINVAL;  // see two_z_fits
  int nl = TwoP3<T, RM, KM_SYM3>::NL;
  const int tz = std::is_same<T, df>::value ? a.C : 3;
  while (nl > 1 && smem_of(nl) > (size_t)smem_optin_bytes()) nl >>= 1;
  const int LS = two_pitch(h, nl, sizeof(V));
  const dim3 grid(2 * ((p.M + nl - 1) / nl) * (p.M / 2 + 1), a.nrhs), blk(nl, h.R1, tz);
  auto go = [&](auto kern) -> vie_status {
    VIE_CK(allow_smem(kern));
    VIE_CK(launch_after<kOverlap<T>>(kern, grid, blk, smem_of(nl), st, (V*)a.B, a.n, h, LS, a.C, a.mode, (const V*)a.K,
                        (const V*)a.tw));
    return VIE_OK;
  };
  if constexpr (std::is_same<T, df>::value) {  // the operator's kernel sets only
    if constexpr (RM > 16) return go(k2_p3h<T, -1>);
    else return go(k2_p3<T, RM, -1>);
  } else {
    constexpr bool f64 = std::is_same<T, double>::value;  // the scattered field's sets are FP64 only
    if constexpr (RM > 16) {
      if (half && a.mode == KM_SYM3) return go(k2_p3h<T, KM_SYM3>);
      if (half && a.mode == KM_MAXWELL6) return go(k2_p3h<T, KM_MAXWELL6>);
      if constexpr (f64) {
        if (half && a.mode == KM_DIV) return go(k2_p3h<T, KM_DIV>);
        if (half) return go(k2_p3h<T, KM_EMRED>);
      }
    }
    if (a.mode == KM_SYM3) return go(k2_p3<T, RM, KM_SYM3>);
    if (a.mode == KM_MAXWELL6) return go(k2_p3<T, RM, KM_MAXWELL6>);
    if constexpr (f64) return a.mode == KM_DIV ? go(k2_p3<T, RM, KM_DIV>) : go(k2_p3<T, RM, KM_EMRED>);
    return VIE_EINVAL;
  }
}

template <typename T, int RM>
vie_status two_last_pass(const TwoPlan& p, const TwoArgs& a, cudaStream_t st) {
  typedef typename CT<T>::V V;
  typedef typename IOT<T>::E E;
  const int tz = std::min(3, a.cout), LS = (p.R1 * p.PF) | 1;
  int rows = std::max(1, 256 / (p.R1 * tz));
  while (rows > 1 && two_smem<V>(p, (size_t)a.cout * rows, LS) > 100 * 1024) --rows;
  VIE_CK(allow_smem(k2_p5<T, RM>));
  VIE_CK(launch_after<kOverlap<T>>(k2_p5<T, RM>, dim3((a.n * a.n + rows - 1) / rows, a.nrhs), dim3(p.R1, rows, tz), two_smem<V>(p,
                      (size_t)a.cout * rows, LS), st, (const V*)a.A, (const E*)a.x, (E*)a.y, a.n, p, LS, a.C, a.cout,
                      (const V*)a.He, (const V*)a.Hm, a.with_identity, (const V*)a.tw));
  return VIE_OK;
}

// Pass `pass` (1..5): one translation unit per arithmetic and radix class, and
// one per kernel for the double-word codelets (apply_two_*.cu).
#define VIE_TWO_UNITS(X) X(f32_16) X(f32_24) X(f64_16) X(f64_24) X(df_16) X(df_24)
#define VIE_TWO_DECL(U) vie_status two_pass_##U(int pass, const TwoPlan& p, const TwoArgs& a, cudaStream_t st);
VIE_TWO_UNITS(VIE_TWO_DECL)
vie_status two_z_df_16(const TwoPlan& p, const TwoArgs& a, cudaStream_t st);
vie_status two_z_df_24(const TwoPlan& p, const TwoArgs& a, cudaStream_t st);

template <typename T, int RM>
vie_status two_pass(int pass, const TwoPlan& p, const TwoArgs& a, cudaStream_t st) {
  if (pass == 3) return two_z_pass<T, RM>(p, a, st);
  if (pass == 5) return two_last_pass<T, RM>(p, a, st);
  return two_line_pass<T, RM>(pass, p, a, st);
}

}  // namespace vie
