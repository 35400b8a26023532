// Device building blocks shared by the 2D and 3D kernels of the sPTT channel
// step: complex arithmetic in double and single precision, mixed-radix
// Stockham FFTs in shared memory (single precision here; FP64-accurate in
// 64-bit block fixed point, ptt_fx.cuh), SBDF coefficients, warp-cooperative
// Chebyshev recurrences and quasi-tridiagonal tau sweeps, the Chebyshev
// column transforms (Gauss and Gauss-Lobatto grids) and the Fourier row
// transforms.  Included by each kernel translation unit (internal linkage).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "ptt_div.h"
#include "ptt_fx.cuh"
#include "ptt_internal.h"

namespace ptt {
namespace {

// Block coordinates of one launch, explicit so that a kernel body can also
// run as one block of a launch over several shape groups (MultiMap).
struct Blk {
  int x, y, z;
};
__device__ __forceinline__ Blk this_blk() { return Blk{(int)blockIdx.x, (int)blockIdx.y, (int)blockIdx.z}; }

// One launch over the shape groups of a context: group q contributes
// gx[q] * gy[q] * gz[q] blocks, numbered from start[q] in x-fastest order,
// so that each group's blocks see the coordinates of its own launch.
constexpr int kMaxGroupsMulti = 64;
struct MultiMap {
  int ng;
  int gid[kMaxGroupsMulti];      // index of entry q among the context's groups
  int gx[kMaxGroupsMulti], gy[kMaxGroupsMulti], gz[kMaxGroupsMulti];
  unsigned start[kMaxGroupsMulti + 1];
};
// The group of this block (its index among the context's groups) and the
// block's coordinates within that group's launch.
__device__ __forceinline__ int multi_locate(const MultiMap& mm, Blk& bk) {
  const unsigned v = blockIdx.x;
  int lo = 0, hi = mm.ng - 1;   // the entry q with start[q] <= v < start[q + 1]
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (mm.start[mid] <= v) lo = mid; else hi = mid - 1;
  }
  const unsigned l = v - mm.start[lo];
  const unsigned gx = (unsigned)mm.gx[lo], gy = (unsigned)mm.gy[lo];
  bk.x = (int)(l % gx);
  bk.y = (int)((l / gx) % gy);
  bk.z = (int)(l / (gx * gy));
  return mm.gid[lo];
}

// ------------------------------------------------------------ complex math
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cscl(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 mul_i(double2 a) { return make_double2(-a.y, a.x); }
__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double2 cfma(double s, double2 a, double2 c) {  // s*a + c
  return make_double2(fma(s, a.x, c.x), fma(s, a.y, c.y));
}
__device__ __forceinline__ double2 czero() { return make_double2(0.0, 0.0); }

// single precision twins (mixed-precision transforms)
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cscl(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 mul_i(float2 a) { return make_float2(-a.y, a.x); }
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 cfma(float s, float2 a, float2 c) {
  return make_float2(fmaf(s, a.x, c.x), fmaf(s, a.y, c.y));
}

// compute types of the transforms: float2 (mixed groups), fxc (FP64-accurate,
// 64-bit block fixed point between FP64 arrays)
template <typename C2> struct RealOf;
template <> struct RealOf<double2> { using T = double; };
template <> struct RealOf<float2> { using T = float; };
template <typename C2> __device__ __forceinline__ C2 zero2();
template <> __device__ __forceinline__ double2 zero2<double2>() { return make_double2(0.0, 0.0); }
template <> __device__ __forceinline__ float2 zero2<float2>() { return make_float2(0.f, 0.f); }
template <typename D> __device__ __forceinline__ D cvt2(double2 v);
template <typename D> __device__ __forceinline__ D cvt2(float2 v);
template <> __device__ __forceinline__ double2 cvt2<double2>(double2 v) { return v; }
template <> __device__ __forceinline__ float2 cvt2<float2>(double2 v) { return make_float2((float)v.x, (float)v.y); }
template <> __device__ __forceinline__ double2 cvt2<double2>(float2 v) { return make_double2(v.x, v.y); }
template <> __device__ __forceinline__ float2 cvt2<float2>(float2 v) { return v; }

// FP64 <-> FP32 by integer operations (no FP64 pipe work).  Truncated:
// values below the FP32 normal range give zero, beyond it infinity, NaN
// stays NaN.
__device__ __forceinline__ float f32_from_f64_trunc(double d) {
  const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
  const uint32_t sign = hi & 0x80000000u;
  const int ef = (int)((hi >> 20) & 0x7FF) - 1023 + 127;
  if (ef >= 255) {
    const bool nan = (hi & 0x7FF00000u) == 0x7FF00000u && ((hi & 0xFFFFFu) | lo) != 0u;
    return __uint_as_float(sign | 0x7F800000u | (nan ? 0x400000u : 0u));
  }
  if (ef <= 0) return __uint_as_float(sign);
  return __uint_as_float(sign | ((uint32_t)ef << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29));
}
// exact for normal values; zero and subnormals give a signed zero,
// infinities stay, NaN is NaN
__device__ __forceinline__ double f64_from_f32(float v) {
  const uint32_t b = __float_as_uint(v);
  const uint32_t sign = b & 0x80000000u, e = (b >> 23) & 0xFFu, m = b & 0x7FFFFFu;
  if (e == 0u) return __hiloint2double((int)sign, 0);
  if (e == 255u) return __hiloint2double((int)(sign | 0x7FF00000u | (m ? 0x80000u : 0u)), 0);
  return __hiloint2double((int)(sign | ((e + 896u) << 20) | (m >> 3)), (int)((m & 7u) << 29));
}

// ------------------------------------------- mean / fluctuation products
// The mixed form's products split every field on the padded grid into its
// mean over the periodic directions, a(y), and the fluctuation a'.  The
// products' mean part (a b with both means) is the same at every point of a
// row and is formed once per row in FP64; at each point only the
// fluctuation part a b' + a' b + a' b' is formed, in FP32 with the means
// rounded to FP32 as multipliers.  The FP32 rounding then scales with the
// fluctuations, not with the O(10^4) stretch components of the base state.
// mfl carries (mean as FP32 multiplier, fluctuation) through the same
// product code as the plain types; only its fluctuation part is used.
struct mfl {
  float m, f;
  mfl() = default;
  __host__ __device__ constexpr mfl(float m_, float f_) : m(m_), f(f_) {}
  __host__ __device__ constexpr mfl(int v) : m((float)v), f(0.f) {}        // a constant
  __host__ __device__ explicit constexpr mfl(double v) : m((float)v), f(0.f) {}
};
__device__ __forceinline__ mfl operator+(mfl a, mfl b) { return mfl(a.m + b.m, a.f + b.f); }
__device__ __forceinline__ mfl operator-(mfl a, mfl b) { return mfl(a.m - b.m, a.f - b.f); }
__device__ __forceinline__ mfl operator-(mfl a) { return mfl(-a.m, -a.f); }
__device__ __forceinline__ mfl operator*(mfl a, mfl b) {
  return mfl(a.m * b.m, fmaf(a.m, b.f, fmaf(a.f, b.m, a.f * b.f)));
}
__device__ __forceinline__ mfl& operator+=(mfl& a, mfl b) { a = a + b; return a; }

// ------------------------------------------------------------ radix DFTs
// DIR = -1: exp(-2 pi i jk/R) (forward); DIR = +1: exp(+2 pi i jk/R).
template <int DIR, int R> struct Bfly;

template <int DIR> struct Bfly<DIR, 2> {
  template <typename C2>
  static __device__ __forceinline__ void run(C2* v) {
    C2 t = v[0];
    v[0] = cadd(t, v[1]);
    v[1] = csub(t, v[1]);
  }
};

template <int DIR> struct Bfly<DIR, 4> {
  template <typename C2>
  static __device__ __forceinline__ void run(C2* v) {
    C2 s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]);
    C2 s13 = cadd(v[1], v[3]), d13 = mul_i(csub(v[1], v[3]));
    v[0] = cadd(s02, s13);
    v[2] = csub(s02, s13);
    if (DIR < 0) { v[1] = csub(d02, d13); v[3] = cadd(d02, d13); }
    else         { v[1] = cadd(d02, d13); v[3] = csub(d02, d13); }
  }
};

template <int DIR> struct Bfly<DIR, 3> {
  template <typename C2>
  static __device__ __forceinline__ void run(C2* v) {
    using T = typename RealOf<C2>::T;
    const T s = (T)(DIR * 0.86602540378443864676);  // sin(2 pi / 3), signed
    C2 t1 = cadd(v[1], v[2]);
    C2 it2 = mul_i(csub(v[1], v[2]));
    C2 m = cfma((T)-0.5, t1, v[0]);
    v[0] = cadd(v[0], t1);
    v[1] = cfma(s, it2, m);
    v[2] = cfma(-s, it2, m);
  }
};

template <int DIR> struct Bfly<DIR, 5> {
  template <typename C2>
  static __device__ __forceinline__ void run(C2* v) {
    using T = typename RealOf<C2>::T;
    const T c1 = (T)0.30901699437494742410;   // cos(2 pi / 5)
    const T c2 = (T)-0.80901699437494742410;  // cos(4 pi / 5)
    const T s1 = (T)(DIR * 0.95105651629515357212);  // sin(2 pi / 5), signed
    const T s2 = (T)(DIR * 0.58778525229247312917);  // sin(4 pi / 5), signed
    C2 t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
    C2 t3 = mul_i(csub(v[1], v[4])), t4 = mul_i(csub(v[2], v[3]));
    C2 b1 = cfma(c1, t1, cfma(c2, t2, v[0]));
    C2 b2 = cfma(c2, t1, cfma(c1, t2, v[0]));
    C2 e1 = cfma(s1, t3, cscl(t4, s2));
    C2 e2 = cfma(s2, t3, cscl(t4, -s1));
    v[0] = cadd(v[0], cadd(t1, t2));
    v[1] = cadd(b1, e1);
    v[4] = csub(b1, e1);
    v[2] = cadd(b2, e2);
    v[3] = csub(b2, e2);
  }
};

// Radix 8: with w = exp(DIR 2 pi i / 8),
// a_r = v_r + v_{r+4}, b_r = (v_r - v_{r+4}) w^r (r < 4), the even outputs
// are the 4-point DFT of a and the odd ones that of b:
//   y_{2k} = sum_r a_r w^{2rk},  y_{2k+1} = sum_r b_r w^{2rk}.
template <int DIR> struct Bfly<DIR, 8> {
  template <typename C2>
  static __device__ __forceinline__ void run(C2* v) {
    using T = typename RealOf<C2>::T;
    const T h = (T)0.70710678118654752440;   // cos(pi/4)
    C2 a[4], b[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      a[r] = cadd(v[r], v[r + 4]);
      b[r] = csub(v[r], v[r + 4]);
    }
    // w = (1 + DIR i)/sqrt 2, w^2 = DIR i, w^3 = (-1 + DIR i)/sqrt 2
    {
      const C2 ib1 = mul_i(b[1]), ib3 = mul_i(b[3]);
      if (DIR > 0) {
        b[1] = cscl(cadd(b[1], ib1), h);
        b[2] = mul_i(b[2]);
        b[3] = cscl(csub(ib3, b[3]), h);
      } else {
        b[1] = cscl(csub(b[1], ib1), h);
        C2 t;
        t.x = b[2].y;
        t.y = -b[2].x;
        b[2] = t;
        const C2 s3 = cadd(b[3], ib3);
        t.x = -s3.x;
        t.y = -s3.y;
        b[3] = cscl(t, h);
      }
    }
    Bfly<DIR, 4>::run(a);
    Bfly<DIR, 4>::run(b);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[2 * k] = a[k];
      v[2 * k + 1] = b[k];
    }
  }
};

// Constants of pass s of a plan, read from the plan (host-computed): the
// passes divide nothing at run time.
struct PassC {
  int nb, st, Ns;
  FastDiv dnb, dns;
};
__device__ __forceinline__ PassC pass_c(const FftPlan& pl, int s) {
  PassC c;
  c.nb = pl.pnb[s];
  c.st = pl.pst[s];
  c.Ns = pl.pns[s];
  c.dnb = FastDiv{pl.pmb[s], pl.pmb[s] == 0u};
  c.dns = FastDiv{pl.pms[s], pl.pms[s] == 0u};
  return c;
}

// One Stockham pass of radix R over nl lines (line l at offset l*ls).
template <int DIR, int R, typename C2>
__device__ __forceinline__ void fft_pass(const C2* __restrict__ src, C2* __restrict__ dst,
                                         int nl, int ls, const PassC& c,
                                         const C2* __restrict__ tw) {
  const int nb = c.nb, st = c.st, Ns = c.Ns;
  const int total = nl * nb;
  const FastDiv dnb = c.dnb, dns = c.dns;
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    const int l = (int)fdiv((unsigned)t, dnb);
    const int j = t - l * nb;
    const C2* s = src + l * ls;
    C2* d = dst + l * ls;
    const int jq = (int)fdiv((unsigned)j, dns);
    const int jm = j - jq * Ns;
    C2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = s[j + r * nb];
    if (Ns > 1) {
#pragma unroll
      for (int r = 1; r < R; ++r) {
        C2 w = __ldg(&tw[jm * r * st]);
        if (DIR > 0) w.y = -w.y;
        v[r] = cmul(v[r], w);
      }
    }
    Bfly<DIR, R>::run(v);
    const int o = jq * Ns * R + jm;
#pragma unroll
    for (int r = 0; r < R; ++r) d[o + r * Ns] = v[r];
  }
}

__device__ __forceinline__ double flip_sign(double v, bool c) {
  return __hiloint2double(__double2hiint(v) ^ (c ? (int)0x80000000 : 0), __double2loint(v));
}

// First pass of radix 3 (no twiddles) for lines that are zero in their
// middle third [n/3, 2n/3) -- the inverse transforms of spectra padded to
// n >= 3K points for K kept modes: with v1 = 0 the butterfly is
// y0 = v0 + v2, y1,2 = v0 - v2/2 -+ DIR sin(2 pi/3) i v2 (8 operations).
template <int DIR, typename C2>
__device__ __forceinline__ void fft_pass_r3_zmid(const C2* __restrict__ src, C2* __restrict__ dst,
                                                 int nl, int ls, const PassC& c) {
  using T = typename RealOf<C2>::T;
  const int nb = c.nb;
  const int total = nl * nb;
  const FastDiv dnb = c.dnb;
  const T sn = (T)(DIR * 0.86602540378443864676);  // sin(2 pi / 3), signed
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    const int l = (int)fdiv((unsigned)t, dnb);
    const int j = t - l * nb;
    const C2 v0 = src[l * ls + j], v2 = src[l * ls + j + 2 * nb];
    C2 m, y1, y2;
    m.x = fma((T)-0.5, v2.x, v0.x);
    m.y = fma((T)-0.5, v2.y, v0.y);
    y1.x = fma(sn, v2.y, m.x);
    y1.y = fma(-sn, v2.x, m.y);
    y2.x = fma(-sn, v2.y, m.x);
    y2.y = fma(sn, v2.x, m.y);
    C2* d = dst + l * ls + 3 * j;
    d[0] = cadd(v0, v2);
    d[1] = y1;
    d[2] = y2;
  }
}

// Unnormalised FP32 DFT of nl lines of length pl.n held in `a`, using `b` as
// the ping-pong buffer.  Returns the buffer holding the result.  Must be
// called by the whole block after a __syncthreads(); ends with one.
// zero_mid: the lines are zero in their middle third and the plan starts
// with radix 3.  Radices 2 to 5 and 8 (the padded lengths are 5-smooth).
template <int DIR>
__device__ float2* fft_lines(float2* a, float2* b, int nl, int ls, const FftPlan& pl, bool zero_mid = false) {
  float2* src = a;
  float2* dst = b;
  const float2* tw = pl.twf;
  for (int s = 0; s < pl.nst; ++s) {
    const int R = pl.radix[s];
    const PassC c = pass_c(pl, s);
    if (s == 0 && zero_mid && R == 3) {
      fft_pass_r3_zmid<DIR>(src, dst, nl, ls, c);
    } else {
      switch (R) {
        case 2: fft_pass<DIR, 2>(src, dst, nl, ls, c, tw); break;
        case 3: fft_pass<DIR, 3>(src, dst, nl, ls, c, tw); break;
        case 4: fft_pass<DIR, 4>(src, dst, nl, ls, c, tw); break;
        case 5: fft_pass<DIR, 5>(src, dst, nl, ls, c, tw); break;
        default: fft_pass<DIR, 8>(src, dst, nl, ls, c, tw); break;
      }
    }
    __syncthreads();
    float2* t = src; src = dst; dst = t;
  }
  return src;
}

// SBDF coefficients, orders 1..4: a_0..a_4 and b_0..b_3 (Sec. 2: 4th-order
// semi-implicit BDF; lower orders start the history).
__constant__ double c_sa[4][5] = {{1.0, -1.0, 0.0, 0.0, 0.0},
                                  {1.5, -2.0, 0.5, 0.0, 0.0},
                                  {11.0 / 6.0, -3.0, 1.5, -1.0 / 3.0, 0.0},
                                  {25.0 / 12.0, -4.0, 3.0, -4.0 / 3.0, 0.25}};
__constant__ double c_sb[4][4] = {{1.0, 0.0, 0.0, 0.0},
                                  {2.0, -1.0, 0.0, 0.0},
                                  {3.0, -3.0, 1.0, 0.0},
                                  {4.0, -6.0, 4.0, -1.0}};
__constant__ float c_sbf[4][4] = {{1.f, 0.f, 0.f, 0.f},   // the same (exact in FP32)
                                  {2.f, -1.f, 0.f, 0.f},
                                  {3.f, -3.f, 1.f, 0.f},
                                  {4.f, -6.f, 4.f, -1.f}};

// 2D mixed groups keep the explicit-term history and its SBDF sum in FP32
// for every mode but the mean (the explicit terms carry FP32 accuracy there):
// each member's FP32 history sits in the first half of its own block of the
// FP64 history array, the mean mode's FP64 history in the second half (so
// checkpoints copy the same byte ranges).  FP64 <-> FP32 by integer
// operations.
__device__ __forceinline__ float2 f2_trunc(double2 v) {
  return make_float2(f32_from_f64_trunc(v.x), f32_from_f64_trunc(v.y));
}
__device__ __forceinline__ double2 d2_exact(float2 v) {
  return make_double2(f64_from_f32(v.x), f64_from_f32(v.y));
}

// ------------------------------------------- warp-cooperative recurrences
// FP64 runs at a few lanes per clock per SM on this part, so a warp FP64
// instruction costs the same pipe time whether 1 or 32 lanes are active.
// The Chebyshev recurrences and the tau sweeps are therefore written as
// warp scans: each lane takes a contiguous chunk, composes it sequentially,
// and the chunks are combined with shuffles.
constexpr unsigned kFull = 0xffffffffu;
// tau solves: above this top elimination factor the top coefficient of a
// parity is taken from its wall row (see warp_qt_solve)
constexpr double kTopFromWall = 1e3;
constexpr int kMaxChunk = 8;  // tau sweeps: up to 8 rows per lane (ny <= 513)

__device__ __forceinline__ double2 shfl_down2(double2 v, int o) {
  return make_double2(__shfl_down_sync(kFull, v.x, o), __shfl_down_sync(kFull, v.y, o));
}
__device__ __forceinline__ float2 shfl_down2(float2 v, int o) {
  return make_float2(__shfl_down_sync(kFull, v.x, o), __shfl_down_sync(kFull, v.y, o));
}
__device__ __forceinline__ double2 shfl_up2(double2 v, int o) {
  return make_double2(__shfl_up_sync(kFull, v.x, o), __shfl_up_sync(kFull, v.y, o));
}
__device__ __forceinline__ double2 warp_allsum2(double2 v) {
  for (int o = 16; o > 0; o >>= 1) {
    v.x += __shfl_xor_sync(kFull, v.x, o);
    v.y += __shfl_xor_sync(kFull, v.y, o);
  }
  return v;
}

// 0 <= k < 2^23 as a double, without the FP64 pipe and without branches.
__device__ __forceinline__ double lane_i2d(int k) {
  const unsigned b = __float_as_uint(__uint_as_float(0x4B000000u | (unsigned)k) - 8388608.f);
  return __hiloint2double((int)((b >> 3) + (k ? 0x38000000u : 0u)), (int)(b << 29));
}
template <typename T> __device__ __forceinline__ T int_as(int k);
template <> __device__ __forceinline__ double int_as<double>(int k) { return lane_i2d(k); }
template <> __device__ __forceinline__ float int_as<float>(int k) { return (float)k; }
// Mean over y of T_n (n even), 2/(1 - n^2): four times the tau rows' table
// w2_n = 1/(2 (n^2 - 1)) with its sign turned (w holds w1, w2, w3 from n = 2).
__device__ __forceinline__ double cheb_mean_weight(const double* w, int N, int n) {
  return n == 0 ? 2.0 : -4.0 * w[N + n];
}

// Chebyshev derivative by one warp: out_n = (2/c_n) sum_{p > n, p + n odd} p a_p
// (c_0 = 2), as two same-parity suffix sums T(k) = sum_{p >= k, p = k mod 2} p a_p
// with out_{k-1} = (2/c_{k-1}) T(k).  `out` must not alias `a`.
template <typename C2>
__device__ void warp_cheb_deriv_par(const C2* a, C2* out, int N, int par) {
  using T = typename RealOf<C2>::T;
  const int lane = threadIdx.x & 31;
  const int L = (N - par + 1) / 2;
  const int c = (L + 31) / 32;
  const int i0 = min(lane * c, L), i1 = min(i0 + c, L);
  // partial sums carried doubled (2 k a_k): b_{k-1} = acc + ex for k >= 2
  // and (acc + ex)/2 for k = 1, with no scaling in the sweeps
  C2 acc = zero2<C2>();
  for (int i = i1 - 1; i >= i0; --i) {
    const int k = par + 2 * i;
    acc = cfma(int_as<T>(2 * k), a[k], acc);
    if (k >= 1) out[k - 1] = acc;
  }
  C2 inc = acc;
  for (int o = 1; o < 32; o <<= 1) {
    const C2 v = shfl_down2(inc, o);
    if (lane + o < 32) inc = cadd(inc, v);
  }
  C2 ex = shfl_down2(inc, 1);
  if (lane == 31) ex = zero2<C2>();
  for (int i = i0; i < i1; ++i) {
    const int k = par + 2 * i;
    if (k >= 2) out[k - 1] = cadd(ex, out[k - 1]);
    else if (k == 1) out[0] = cscl(cadd(ex, out[0]), (T)0.5);
  }
  // out_{N-1} (parity of N - 1) has no term
  if (lane == 0 && ((N - 1 - par) & 1)) out[N - 1] = zero2<C2>();
  __syncwarp();
}

template <typename C2>
__device__ void warp_cheb_deriv(const C2* a, C2* out, int N) {
  warp_cheb_deriv_par(a, out, N, 0);
  warp_cheb_deriv_par(a, out, N, 1);
}

// -x for complex values by sign-bit flips (integer operations, no FP64 work)
__device__ __forceinline__ double2 cneg_bits(double2 v) {
  return make_double2(flip_sign(v.x, true), flip_sign(v.y, true));
}

// Warp-cooperative quasi-tridiagonal tau solve (system stated at k_spec): the backward
// elimination P_i = alpha_i + beta_i P_{i+1} and the forward substitution
// a_i = P_i + Q_i a_{i-1} are affine recurrences, evaluated as warp scans of
// affine maps; the boundary sums are warp reductions.  `out` may alias R.
// CH >= the rows per lane, ceil((L - 1)/32) (register arrays of that size).
// WALL: the wall row has a right-hand side (bcfac sum R), else it is 0.
template <int CH, bool WALL>
__device__ void warp_qt_solve(int N, int p, double alpha, const double2* R, double2* out,
                              const double* Q, const double* inv, const double* F, double G,
                              const double* w1, const double* w2, const double* w3,
                              double bcfac, double rsign) {
  const int lane = threadIdx.x & 31;
  const int L = (N - p + 1) / 2;  // unknowns a_{p+2i}, i < L; rows i = 1..L-1
  const int nr = L - 1;
  const int c = (nr + 31) / 32;
  const int i0 = min(1 + lane * c, L), i1 = min(i0 + c, L);
  double2 al[CH];
  double be[CH];
  double2 rs = czero();
#pragma unroll
  for (int t = 0; t < CH; ++t) {
    const int i = i0 + t;
    if (t < c && i < i1) {
      const int n = p + 2 * i;
      const double2 Rm2 = R[n - 2];
      const double2 R0 = R[n];
      const double w1n = w1[n], iv = inv[n];   // w1 counts twice at n = 2
      double2 r = cscl(Rm2, -__hiloint2double(__double2hiint(w1n) + (n == 2 ? 0x100000 : 0), __double2loint(w1n)));
      if (n <= N - 3) r = cfma(w2[n], R0, r);
      double un = 0.0;
      if (n <= N - 5) {
        const double w3n = w3[n];
        r = cfma(-w3n, R[n + 2], r);
        un = alpha * w3n;
      }
      al[t] = cscl(r, iv);
      be[t] = un * iv;
      if (WALL) rs = cadd(rs, R0);
    } else {
      al[t] = czero();
      be[t] = 1.0;
    }
  }
  if (WALL && lane == 0) rs = cadd(rs, R[p]);
  __syncwarp();
  // backward: chunk map P_{i0} = A + B P_{i1}
  double2 A = czero();
  double B = 1.0;
#pragma unroll
  for (int t = CH - 1; t >= 0; --t) {
    if (t < c && i0 + t < i1) {
      A = cfma(be[t], A, al[t]);
      B *= be[t];
    }
  }
  double2 SA = A;
  double SB = B;
  for (int o = 1; o < 32; o <<= 1) {
    const double2 hA = shfl_down2(SA, o);
    const double hB = __shfl_down_sync(kFull, SB, o);
    if (lane + o < 32) {
      SA = cfma(SB, hA, SA);
      SB *= hB;
    }
  }
  double2 Pin = shfl_down2(SA, 1);
  if (lane == 31) Pin = czero();
  double2 U = czero();
  double2 P = Pin;
#pragma unroll
  for (int t = CH - 1; t >= 0; --t) {
    const int i = i0 + t;
    if (t < c && i < i1) {
      const int n = p + 2 * i;
      P = cfma(be[t], P, al[t]);
      out[n] = P;
      U = cfma(F[n], P, U);
    }
  }
  const double2 a0 = cscl(warp_allsum2(WALL ? make_double2(fma(bcfac, rs.x, -U.x), fma(bcfac, rs.y, -U.y))
                                            : cneg_bits(U)), G);
  // forward: chunk map a_{i1-1} = C + D a_{i0-1}
  double2 Cc = czero();
  double Dd = 1.0;
  double2 Pv[CH];
  double Qv[CH];
#pragma unroll
  for (int t = 0; t < CH; ++t) {
    const int i = i0 + t;
    if (t < c && i < i1) {
      const int n = p + 2 * i;
      Pv[t] = out[n];
      Qv[t] = Q[n];
      Cc = cfma(Qv[t], Cc, Pv[t]);
      Dd *= Qv[t];
    }
  }
  double2 IC = Cc;
  double ID = Dd;
  for (int o = 1; o < 32; o <<= 1) {
    const double2 hC = shfl_up2(IC, o);
    const double hD = __shfl_up_sync(kFull, ID, o);
    if (lane >= o) {
      IC = cfma(ID, hC, IC);
      ID *= hD;
    }
  }
  double2 EC = shfl_up2(IC, 1);
  double ED = __shfl_up_sync(kFull, ID, 1);
  if (lane == 0) { EC = czero(); ED = 1.0; }
  double2 av = cfma(ED, a0, EC);
  const int nl = p + 2 * (L - 1);
  const bool top = L > 1 && fabs(Q[nl]) > kTopFromWall;
  double2 part = (lane == 0) ? a0 : czero();  // sum of a_{p+2i}, i < L-1, where top
  __syncwarp();
#pragma unroll
  for (int t = 0; t < CH; ++t) {
    const int i = i0 + t;
    if (t < c && i < i1) {
      av = cfma(Qv[t], av, Pv[t]);
      out[p + 2 * i] = av;
      if (top && i < L - 1) part = cadd(part, av);
    }
  }
  if (lane == 0) out[p] = a0;
  __syncwarp();
  // Top coefficient from the wall row when the top elimination factor is
  // large: with a small diagonal (diffusivity kappa) the forward
  // substitution forms a_top = P + Q a_{top-2} with |Q| ~ alpha/(4 n^2 kappa)
  // and amplifies the rounding of a_{top-2}; the wall row of the same system
  // gives a_top = g - sum of the others with rounding of the sum only.
  if (top) {
    if (WALL) part = make_double2(fma(-bcfac, rs.x, part.x), fma(-bcfac, rs.y, part.y));
    part = warp_allsum2(part);
    if (lane == 0) out[nl] = cneg_bits(part);
    __syncwarp();
  }
  // the solve above is of (alpha - beta D^2) a = R; the system's right-hand
  // side is rsign R, so a flips sign with it
  if (rsign < 0.0) {
    for (int i = lane; i < L; i += 32) out[p + 2 * i] = cneg_bits(out[p + 2 * i]);
    __syncwarp();
  }
}

// Lane-sequential forms for the per-mode spectral stage: one lane owns one
// (Fourier mode, Chebyshev parity) pair and walks its ~N/2 coefficients in
// order, so a warp advances 32 independent recurrences with every lane busy.
// Columns are indexed by n (stride 1).  Bound by the FP64 pipe (64 cycles per
// warp instruction, as long as its latency: one warp keeps a sub-partition's
// pipe full), so whatever can be formed on the way through a recurrence is
// (the loads of the next row are issued before the current row's arithmetic),
// and what needs no FP64 instruction has none.

// x / 2 where z holds, by integer instructions.
__device__ __forceinline__ double lane_half(double x, bool z) {
  const int h = __double2hiint(x);
  const bool scale = z && (((unsigned)h >> 20) & 0x7FFu) - 2u < 2045u;   // normal, result normal
  return __hiloint2double(scale ? h - 0x100000 : h, __double2loint(x));
}
__device__ __forceinline__ double2 lane_half2(double2 v, bool z) {
  return make_double2(lane_half(v.x, z), lane_half(v.y, z));
}

// Explicit momentum term of one component, outputs n = p mod 2:
//   out_n = nr_n + gam ((D cy)_n + i (kx cx_n + kz cz_n)),
// (D cy)_n = sum over k = n + 1, n + 3, ... of 2 k cy_k, halved at n = 0.
__device__ __forceinline__ void lane_div_h(int N, int p, const double2* __restrict__ cy,
                                           const double2* __restrict__ cx, const double2* __restrict__ cz,
                                           const double2* __restrict__ nr, double gam, double gkx, double gkz,
                                           double2* __restrict__ out) {
  const int nl = ((N - 1 - p) & ~1) + p;
  double2 acc = czero();
#pragma unroll 4
  for (int n = nl; n >= p; n -= 2) {
    const int k = min(n + 1, N - 1);   // n = N - 1 has no term: times 0
    acc = cfma(n + 1 < N ? lane_i2d(2 * k) : 0.0, cy[k], acc);
    const double2 a = cx[n], c = cz[n], d = lane_half2(acc, n == 0);
    double2 h = cfma(gam, d, nr[n]);
    h.x = fma(-gkz, c.y, fma(-gkx, a.y, h.x));
    h.y = fma(gkz, c.x, fma(gkx, a.x, h.y));
    out[n] = h;
  }
}

// q_n = (D^2 v)_n - k2 v_n for n = p mod 2 (the inner derivative's entries of
// the other parity stay in a register).
__device__ __forceinline__ void lane_lap(int N, int p, const double2* __restrict__ v, double k2,
                                         double2* __restrict__ out) {
  const int nl = ((N - 1 - p) & ~1) + p;
  double2 a1 = czero(), a2 = czero(), vp = czero();   // vp = v_{n+2}
#pragma unroll 4
  for (int n = nl; n >= p; n -= 2) {
    a1 = cfma(lane_i2d(2 * (n + 2)), vp, a1);   // (D v)_{n+1}
    a2 = cfma(lane_i2d(2 * (n + 1)), a1, a2);
    vp = v[n];
    out[n] = cfma(-k2, vp, lane_half2(a2, n == 0));
  }
}

// One row of the histories of an evolved column: the current values x, nn and
// the older slots (E: values, Nn: explicit terms).
struct LaneHist {
  const double2 *E0, *E1, *E2;
  ptrdiff_t dn;    // from a slot of E to that of N
  double ca[4];    // -sa_{j+1}/dt
  int o;           // order - 1
};
struct LaneRow { double2 e[3], m[3]; };
template <bool FULL>
__device__ __forceinline__ LaneRow lane_hist_row(const LaneHist& h, int n) {
  LaneRow r;
  if (FULL || h.o >= 1) { r.e[0] = h.E0[n]; r.m[0] = h.E0[n + h.dn]; }
  if (FULL || h.o >= 2) { r.e[1] = h.E1[n]; r.m[1] = h.E1[n + h.dn]; }
  if (FULL) { r.e[2] = h.E2[n]; r.m[2] = h.E2[n + h.dn]; }
  return r;
}
// R = sb_0 nn + sum_j (-sa_{j+1}/dt) x^{n-j} + sum_{j>=1} sb_j N^{n-j}; FULL:
// order 4, else orders 1 to 3 of the first steps.
template <bool FULL>
__device__ __forceinline__ double2 lane_sbdf(const LaneHist& h, const LaneRow& r, double2 x, double2 nn) {
  const double* cb = c_sb[FULL ? 3 : h.o];
  double2 acc = cfma(cb[0], nn, cscl(x, h.ca[0]));
  if (FULL || h.o >= 1) acc = cfma(cb[1], r.m[0], cfma(h.ca[1], r.e[0], acc));
  if (FULL || h.o >= 2) acc = cfma(cb[2], r.m[1], cfma(h.ca[2], r.e[1], acc));
  if (FULL) acc = cfma(cb[3], r.m[2], cfma(h.ca[3], r.e[2], acc));
  return acc;
}

// Quasi-tridiagonal tau solve of one parity (system stated at k_spec), in two
// passes.  lane_qt_back: the backward elimination
//   P_n = inv_n (w2_n R_n - w1_n R_{n-2} - w3_n (R_{n+2} - alpha P_{n+2}))
// (w1 twice its table at n = 2; no w2 term on the last row, no w3 term on the
// last two) and the boundary sum U = sum F_n P_n, with rs = sum R_n where SUM;
// R comes from ld(n) (a row's loads) and ev(row, n), called once for every n
// in descending order.  lane_qt_fwd: a_p = (bcfac rs - U) G, then
// a_n = P_n + Q_n a_{n-2}, in place or into out.  Q, inv, F: the
// right-hand-side-independent elimination factors of this (alpha, mode,
// parity), precomputed on the host.
template <bool SUM, typename Ld, typename Ev>
__device__ __forceinline__ double2 lane_qt_back(int N, int p, double alpha, Ld ld, Ev ev, double2* __restrict__ P,
                                                const double* __restrict__ inv, const double* __restrict__ F,
                                                const double* __restrict__ w, double2& rs) {
  const int nl = ((N - 1 - p) & ~1) + p;
  auto row = ld(nl);
  double iv1 = inv[nl], f1 = F[nl];
  double2 R0 = ev(row, nl), Rp = czero(), Pp = czero(), U = czero();
  row = ld(max(nl - 2, p));
  rs = SUM ? R0 : czero();
#pragma unroll 1
  for (int n = nl; n >= p + 2; n -= 2) {
    const double iv = iv1, f = f1;
    const double w1t = w[n], w2t = w[N + n], w3t = w[2 * N + n];
    const double2 Rm = ev(row, n - 2);
    row = ld(max(n - 4, p));   // in flight during the elimination's own arithmetic
    iv1 = inv[n - 2];
    f1 = F[n - 2];
    const double w1 = __hiloint2double(__double2hiint(w1t) + (n == 2 ? 0x100000 : 0), __double2loint(w1t));
    const double w2 = (n <= N - 3) ? w2t : 0.0, w3 = (n <= N - 5) ? w3t : 0.0;
    const double2 S = cfma(-alpha, Pp, Rp);
    const double2 r = cfma(-w3, S, cfma(w2, R0, cscl(Rm, -w1)));
    const double2 Pn = cscl(r, iv);
    P[n] = Pn;
    U = cfma(f, Pn, U);
    if (SUM) rs = cadd(rs, Rm);
    Pp = Pn;
    Rp = R0;
    R0 = Rm;
  }
  return U;
}
// use(n, a_n) is called once for every n, in ascending order.
template <typename Use>
__device__ __forceinline__ void lane_qt_fwd(int N, int p, double2 a, double2 wall, const double2* P, double2* out,
                                            const double* __restrict__ Q, Use use) {
  constexpr int kU = 4;
  const int nl = ((N - 1 - p) & ~1) + p;
  out[p] = a;
  use(p, a);
  if (nl == p) return;
  for (int n0 = p + 2; n0 < nl; n0 += 2 * kU) {
    double2 v[kU];
    double q[kU];
#pragma unroll
    for (int t = 0; t < kU; ++t) {
      const int n = min(n0 + 2 * t, nl);
      v[t] = P[n];
      q[t] = Q[n];
    }
#pragma unroll
    for (int t = 0; t < kU; ++t) {
      const int n = n0 + 2 * t;
      if (n < nl) {
        a = cfma(q[t], a, v[t]);
        out[n] = a;
        use(n, a);
      }
    }
  }
  const double ql = Q[nl];
  a = cfma(ql, a, P[nl]);
  if (fabs(ql) > kTopFromWall) {   // top coefficient from the wall row
    double2 part = czero();
    for (int n = p; n < nl; n += 2) part = cadd(part, out[n]);
    a = csub(wall, part);
  }
  out[nl] = a;
  use(nl, a);
}

// ---------------------------------------------- per-mode spectral stage
// ------------------------------------------------------ Chebyshev columns
// Column transforms along y for a batch of members and fields.  Coefficient
// side: column m, row n at m*cm + n*cn; value side: column m, row j at
// m*vm + j*vj (within one field of one member).  Input and output may be in
// double or single precision independently of the compute type.
constexpr int kYFields = 17;   // columns per launch (blockIdx.y): the 3D inverse pass
struct YJob {
  const void* src;
  void* dst;
  long long src_mstride, dst_mstride;  // per member (elements)
  long long src_fstride, dst_fstride;  // per field (elements)
  int src_field[kYFields];
  int src_field2[kYFields];  // inverse only: >= 0 adds this field to src_field
  int src_field3[kYFields];  // inverse only: >= 0 adds a third field
  int dst_field[kYFields];
  int deriv[kYFields];       // inverse only: transform d/dy of the field
  long long cm, cn;   // coefficient-side strides
  long long vm, vj;   // value-side strides
  int K;              // columns
  int N, M;           // Chebyshev modes, grid intervals / points
  int inverse;        // 1: coefficients -> values; 0: values -> coefficients (N rows)
  int gauss;          // 0: M+1 Gauss-Lobatto points (DCT-I, FFT length 2M);
                      // 1: M Gauss points (DCT-II/III, FFT length M, M even)
  int src_f32, dst_f32;  // element types of src / dst (0: complex double, 1: complex float)
  const float2* tw4f;    // gauss, FP32: quarter-period table of this direction, k < M:
                         // forward (s_k/2) exp(-i pi k/(2M)) (s_0 = 1/M, s_k = 2/M),
                         // inverse (1/2) exp(+i pi k/(2M))
  const int4* tw4x;      // gauss, fixed point (GroupDev::tw4Px, tw4Pix): forward
                         // with the factor 2^fexp times the normalisation of the
                         // whole forward transform, inverse exp(+i pi k/(2M))
  int fexp;
  int C;              // columns per block
  const int* status;  // skip members with status != 0 (may be null)
  FftPlan pl;
};

// Element formats of transform inputs and outputs (YJob / ZJob src_f32,
// dst_f32): 0 complex double, 1 complex float.
__device__ __forceinline__ float2 ld2(const void* p, long long i, int f32) {
  return f32 ? static_cast<const float2*>(p)[i] : cvt2<float2>(static_cast<const double2*>(p)[i]);
}
__device__ __forceinline__ void st2(void* p, long long i, int f32, float2 v) {
  if (f32) static_cast<float2*>(p)[i] = v;
  else static_cast<double2*>(p)[i] = cvt2<double2>(v);
}

// Values at the M Gauss points y_j = cos(pi (2j+1)/(2M)) from coefficients
// (DCT-III) and back (DCT-II), each as one complex FFT of length M: the
// output (input) order is permuted v_n = f_{2n}, v_{M-1-n} = f_{2n+1}, and a
// quarter-period twiddle exp(-+ i pi k/(2M)) maps between the two (Makhoul's
// construction; the real and imaginary parts of a column ride in one FFT).
// FP32 form.
__device__ void ycols_gauss(const YJob& J, const void* src, const void* src2, const void* src3,
                            void* dst, float2* A, float2* B, int c0, int nc, int f) {
  const int C = J.C, N = J.N, Mg = J.M;
  const int tid = threadIdx.x, nt = blockDim.x;
  if (J.inverse) {
    for (int i = tid; i < Mg * C; i += nt) {
      const int c = (int)fdiv((unsigned)i, fast_div((unsigned)Mg)), n = i - c * Mg;
      float2 v = zero2<float2>();
      if (c < nc && n < N) {
        const long long o = (c0 + c) * J.cm + n * J.cn;
        v = ld2(src, o, J.src_f32);
        if (src2) v = cadd(v, ld2(src2, o, J.src_f32));
        if (src3) v = cadd(v, ld2(src3, o, J.src_f32));
      }
      A[i] = v;
    }
    __syncthreads();
    if (J.deriv[f]) {
      for (int c = tid >> 5; c < C; c += (nt >> 5)) warp_cheb_deriv(A + c * Mg, B + c * Mg, N);
      __syncthreads();
      for (int i = tid; i < N * C; i += nt) {
        const int c = (int)fdiv((unsigned)i, fast_div((unsigned)N)), n = i - c * N;
        A[c * Mg + n] = B[c * Mg + n];
      }
      __syncthreads();
    }
    // V_0 = a_0, V_k = (1/2) exp(+i pi k/(2M)) (a_k - i a_{M-k}), the factor
    // taken from the inverse table
    for (int i = tid; i < Mg * C; i += nt) {
      const int c = (int)fdiv((unsigned)i, fast_div((unsigned)Mg)), k = i - c * Mg;
      const float2 ak = A[i];
      float2 V;
      if (k == 0) {
        V = ak;
      } else {
        const float2 amk = A[c * Mg + Mg - k];
        float2 z;
        z.x = ak.x + amk.y;
        z.y = ak.y - amk.x;
        V = cmul(__ldg(&J.tw4f[k]), z);
      }
      B[i] = V;
    }
    __syncthreads();
    float2* res = fft_lines<+1>(B, A, C, Mg, J.pl);
    for (int i = tid; i < Mg * C; i += nt) {
      const int j = (int)fdiv((unsigned)i, fast_div((unsigned)C)), c = i - j * C;
      if (c < nc) {
        const int pos = (j & 1) ? (Mg - 1 - (j >> 1)) : (j >> 1);
        st2(dst, j * J.vj + (c0 + c) * J.vm, J.dst_f32, res[c * Mg + pos]);
      }
    }
  } else {
    for (int i = tid; i < Mg * C; i += nt) {
      const int j = (int)fdiv((unsigned)i, fast_div((unsigned)C)), c = i - j * C;
      const int pos = (j & 1) ? (Mg - 1 - (j >> 1)) : (j >> 1);
      A[c * Mg + pos] = (c < nc) ? ld2(src, j * J.vj + (c0 + c) * J.vm, J.src_f32) : zero2<float2>();
    }
    __syncthreads();
    float2* res = fft_lines<-1>(A, B, C, Mg, J.pl);
    // with s = V_k + conj V_{M-k}, d = V_k - conj V_{M-k} (the transforms of
    // the real and imaginary parts, times 2 and 2i) and the forward table
    // F_k = (s_k/2) exp(-i pi k/(2M)):  a_k = (Re(F_k s), Re(F_k (-i d)))
    for (int i = tid; i < N * C; i += nt) {
      const int c = (int)fdiv((unsigned)i, fast_div((unsigned)N)), k = i - c * N;
      if (c < nc) {
        const float2 Vk = res[c * Mg + k];
        const float2 Rm = res[c * Mg + (k == 0 ? 0 : Mg - k)];
        const float sx = Vk.x + Rm.x, sy = Vk.y - Rm.y;
        const float dx = Vk.x - Rm.x, dy = Vk.y + Rm.y;
        const float2 w = __ldg(&J.tw4f[k]);
        float2 o;
        o.x = w.x * sx - w.y * sy;
        o.y = w.x * dy + w.y * dx;
        st2(dst, (c0 + c) * J.cm + k * J.cn, J.dst_f32, o);
      }
    }
  }
}

// The same in fixed point, FP64 in and out: a warp per column outside the
// FFT.  Bd: room for the derivative of the block's columns (only for fields
// with deriv).
constexpr int kFxCols = 16;   // columns per block, at most
__device__ void ycols_gauss_fx(const YJob& J, const double2* src, const double2* src2, const double2* src3,
                               double2* dst, fxc* A, double2* Bd, FxS* fs, int c0, int nc, int f) {
  const int C = J.C, N = J.N, Mg = J.M;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, nw = nt >> 5;
  const FastDiv dC = fast_div((unsigned)C);
  const FastDiv dN = fast_div((unsigned)N);
  if (J.inverse) {
    for (int i = tid; i < nc * N; i += nt) {
      const int c = (int)fdiv((unsigned)i, dN), n = i - c * N;
      const long long o = (c0 + c) * J.cm + n * J.cn;
      double2 v = src[o];
      if (src2) v = cadd(v, src2[o]);
      if (src3) v = cadd(v, src3[o]);
      reinterpret_cast<double2*>(A)[c * Mg + n] = v;
    }
    __syncthreads();
    const bool dy = J.deriv[f] != 0;
    for (int c = tid >> 5; c < nc; c += nw) {
      const double2* raw = reinterpret_cast<const double2*>(A + c * Mg);
      if (dy) {
        double2* D = Bd + c * N;
        warp_cheb_deriv(raw, D, N);
        raw = D;
      }
      unsigned m = 0u;
      for (int n = lane; n < N; n += 32) m = max(m, fx_mag2(raw[n]));
      const FxS s = fx_warp_scale(m, N, [raw](int n) { return raw[n]; }, 1);
      if (lane == 0) fs[c] = s;
    }
    __syncthreads();
    // twice the V_k: V_0 = 2 a_0, V_k = exp(+i pi k/(2M)) (a_k - i a_{M-k}), the
    // pair k, M - k by one thread (in place when raw is the column itself); by the
    // whole block, as a block of one column (the mean's) has one warp at work above
    const int np = Mg / 2 + 1;
    const FastDiv dP = fast_div((unsigned)np);
    for (int i = tid; i < nc * np; i += nt) {
      const int c = (int)fdiv((unsigned)i, dP), k = i - c * np, km = Mg - k;
      fxc* V = A + c * Mg;
      const fxc* rx = dy ? reinterpret_cast<const fxc*>(Bd + c * N) : V;
      const int base = fs[c].base;
      const fxc a = (k < N) ? fx_from2(fx_raw(rx[k]), base) : fx_zero();
      if (k == 0) {
        V[0] = cadd(a, a);
      } else {
        const fxc b = (km < N) ? fx_from2(fx_raw(rx[km]), base) : fx_zero();
        V[k] = fx_cmul<false>(mk_fxc(a.x + b.y, a.y - b.x), __ldg(&J.tw4x[k]));
        if (km != k) V[km] = fx_cmul<false>(mk_fxc(b.x + a.y, b.y - a.x), __ldg(&J.tw4x[km]));
      }
    }
    __syncthreads();
    fx_lines<+1, false>(A, nc, Mg, &J.pl, false);
    for (int i = tid; i < Mg * C; i += nt) {
      const int j = (int)fdiv((unsigned)i, dC), c = i - j * C;
      if (c < nc) {
        const int pos = (j & 1) ? (Mg - 1 - (j >> 1)) : (j >> 1);
        dst[j * J.vj + (c0 + c) * J.vm] = fx_to2(A[c * Mg + pos], fs[c], 1);
      }
    }
  } else {
    double2* R = reinterpret_cast<double2*>(A);
    for (int i = tid; i < Mg * C; i += nt) {
      const int j = (int)fdiv((unsigned)i, dC), c = i - j * C;
      const int pos = (j & 1) ? (Mg - 1 - (j >> 1)) : (j >> 1);
      if (c < nc) R[c * Mg + pos] = src[j * J.vj + (c0 + c) * J.vm];
    }
    __syncthreads();
    for (int c = tid >> 5; c < nc; c += nw) {
      const double2* raw = R + c * Mg;
      unsigned m = 0u;
      for (int n = lane; n < Mg; n += 32) m = max(m, fx_mag2(raw[n]));
      const FxS s = fx_warp_scale(m, Mg, [raw](int n) { return raw[n]; }, 0);
      if (lane == 0) fs[c] = s;
    }
    __syncthreads();
    const FastDiv dM = fast_div((unsigned)Mg);
    for (int i = tid; i < nc * Mg; i += nt)
      A[i] = fx_from2(fx_raw(A[i]), fs[fdiv((unsigned)i, dM)].base);
    __syncthreads();
    fx_lines<-1, false>(A, nc, Mg, &J.pl, false);
    for (int i = tid; i < nc * N; i += nt) {
      const int c = (int)fdiv((unsigned)i, dN), k = i - c * N;
      const fxc* V = A + c * Mg;
      const fxc Vk = V[k], Rm = V[k == 0 ? 0 : Mg - k];
      const int4 w = __ldg(&J.tw4x[k]);
      dst[(c0 + c) * J.cm + k * J.cn] =
          make_double2(fx_to(fx_dot(Vk.x + Rm.x, Vk.y - Rm.y, w), fs[c], J.fexp),
                       fx_to(fx_dot(Vk.y + Rm.y, Rm.x - Vk.x, w), fs[c], J.fexp));
    }
  }
}

// Gauss-Lobatto path (fixed point, FP64 in and out): DCT-I by the even
// extension.
__device__ void ycols_lobatto(const YJob& J, const double2* src, const double2* src2, const double2* src3,
                              double2* dst, fxc* A, fxc* a0s, FxS* fs, int c0, int nc) {
  const int C = J.C, N = J.N, M = J.M, P = 2 * J.M;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, nw = nt >> 5;
  const FastDiv dC = fast_div((unsigned)C);
  if (!J.inverse) {
    double2* R = reinterpret_cast<double2*>(A);
    for (int i = tid; i < (M + 1) * C; i += nt) {
      const int j = (int)fdiv((unsigned)i, dC), c = i - j * C;
      if (c < nc) R[c * P + j] = src[j * J.vj + (c0 + c) * J.vm];
    }
    __syncthreads();
  }
  const int cnt = J.inverse ? N : M + 1;
  for (int c = tid >> 5; c < nc; c += nw) {
    double2* R = reinterpret_cast<double2*>(A + c * P);
    unsigned m = 0u;
    for (int n = lane; n < cnt; n += 32) {
      double2 v;
      if (J.inverse) {
        const long long o = (c0 + c) * J.cm + n * J.cn;
        v = src[o];
        if (src2) v = cadd(v, src2[o]);
        if (src3) v = cadd(v, src3[o]);
        R[n] = v;
      } else {
        v = R[n];
      }
      m = max(m, fx_mag2(v));
    }
    const FxS s = fx_warp_scale(m, cnt, [R](int n) { return R[n]; }, 1);
    if (lane == 0) fs[c] = s;
    __syncwarp();
    // even extension: A[n] = a_n (n <= M, zero for n >= N), A[P - n] = a_n
    fxc* V = A + c * P;
    for (int n = lane; n <= M; n += 32) {
      const fxc a = (n < cnt) ? fx_from2(fx_raw(V[n]), s.base) : fx_zero();
      V[n] = a;
      if (n > 0 && n < M) V[P - n] = a;
      if (n == 0) a0s[c] = a;
      if (n == M) a0s[C + c] = a;
    }
  }
  __syncthreads();
  fx_lines<-1, true>(A, nc, P, &J.pl, false);
  if (J.inverse) {   // f_j = (F_j + a_0 + (-1)^j a_M) / 2
    for (int i = tid; i < (M + 1) * C; i += nt) {
      const int j = (int)fdiv((unsigned)i, dC), c = i - j * C;
      if (c < nc) {
        fxc v = cadd(A[c * P + j], a0s[c]);
        v = (j & 1) ? csub(v, a0s[C + c]) : cadd(v, a0s[C + c]);
        dst[j * J.vj + (c0 + c) * J.vm] = fx_to2(v, fs[c], 1);
      }
    }
  } else {
    const double inv = 1.0 / M;
    for (int c = tid >> 5; c < nc; c += nw)
      for (int n = lane; n < N; n += 32) {
        const double s = (n == 0 || n == M) ? 0.5 * inv : inv;
        dst[(c0 + c) * J.cm + n * J.cn] = cscl(fx_to2(A[c * P + n], fs[c]), s);
      }
  }
}

// FP32 columns (CT = float2, Gauss grid only) or fixed point (CT = fxc).
// BIG: the Gauss-Lobatto (unpadded) path, whose FFT length 2 (ny - 1) may
// hold radices 7, 11, 13; the Gauss (padded) path runs without it.
template <typename CT, bool BIG = false>
__device__ __forceinline__ void ycols_block(const YJob& J, Blk bk) {
  const int b = bk.z;
  if (J.status && J.status[b]) return;
  const int f = bk.y;
  // FFT length per column: M on the Gauss grid, 2M (even extension) on the
  // Gauss-Lobatto grid (shared memory: smem_ycols, smem_ycols_fx)
  const int C = J.C, K = J.K, P = J.gauss ? J.M : 2 * J.M;
  const int c0 = bk.x * C;
  const int nc = min(C, K - c0);
  extern __shared__ __align__(16) unsigned char smraw[];
  CT* A = reinterpret_cast<CT*>(smraw);
  CT* B = A + (size_t)C * P;
  const size_t es = J.src_f32 ? sizeof(float2) : sizeof(double2);
  const size_t ed = J.dst_f32 ? sizeof(float2) : sizeof(double2);
  const void* src = static_cast<const char*>(J.src) + (b * J.src_mstride + J.src_field[f] * J.src_fstride) * es;
  void* dst = static_cast<char*>(J.dst) + (b * J.dst_mstride + J.dst_field[f] * J.dst_fstride) * ed;
  const void* src2 = (J.inverse && J.src_field2[f] >= 0)
      ? static_cast<const char*>(J.src) + (b * J.src_mstride + J.src_field2[f] * J.src_fstride) * es
      : nullptr;
  const void* src3 = (J.inverse && J.src_field3[f] >= 0)
      ? static_cast<const char*>(J.src) + (b * J.src_mstride + J.src_field3[f] * J.src_fstride) * es
      : nullptr;
  if constexpr (std::is_same<CT, fxc>::value) {
    __shared__ FxS fs[kFxCols];
    const double2 *s1 = static_cast<const double2*>(src), *s2 = static_cast<const double2*>(src2),
                  *s3 = static_cast<const double2*>(src3);
    if constexpr (BIG) ycols_lobatto(J, s1, s2, s3, static_cast<double2*>(dst), A, B, fs, c0, nc);
    else ycols_gauss_fx(J, s1, s2, s3, static_cast<double2*>(dst), A, reinterpret_cast<double2*>(B), fs, c0, nc, f);
  } else {
    ycols_gauss(J, src, src2, src3, dst, A, B, c0, nc, f);
  }
}

template <typename CT, bool BIG = false>
__global__ void __launch_bounds__(256, BIG ? 3 : 4) k_ycols(const __grid_constant__ YJob J) {
  ycols_block<CT, BIG>(J, this_blk());
}

// The same over the shape groups of a context (job q of jobs for group q).
template <typename CT, bool BIG = false>
__global__ void __launch_bounds__(256, BIG ? 3 : 4) k_ycols_multi(const YJob* __restrict__ jobs, MultiMap mm) {
  Blk bk;
  const int q = multi_locate(mm, bk);
  ycols_block<CT, BIG>(jobs[q], bk);
}

// ---------------------------------------------------------- Fourier rows
// Row transforms along x: complex modes m < K <-> real values at n points,
// two real fields packed in one complex line.
struct XJob {
  const double2* srcC;  // c2r: complex rows
  const double* srcR;   // r2c: real rows
  double2* dstC;
  double* dstR;
  long long src_mstride, dst_mstride, src_fstride, dst_fstride;
  int src_rstep, dst_rstep;  // row index multipliers (elements per row = K or n)
  int nf;                    // fields (packed in pairs, (nf + 1) / 2 lines)
  int K, n;
  int c2r;
  // c2r with nf = 1: pair_rows lines per block, line p of all synthesises rows
  // 2p and 2p + 1 (< nrows) as its real and imaginary parts (xrows_pairs)
  int pair_rows, nrows;
  // 3D physical values of a caller: real row y zy_nz + z lies at z zy_ny + y
  // (zy_nz = 0: rows in order)
  int zy_nz, zy_ny;
  const int* status;
  FftPlan pl;
};
__device__ __forceinline__ int xrow_real(const XJob& J, int row) {
  if (J.zy_nz == 0) return row;
  const int y = row / J.zy_nz;
  return (row - y * J.zy_nz) * J.zy_ny + y;
}

// Fixed-point lines of real fields, shared by the x transforms: two fields
// per line of n points, field q of the block on scale fs[q] (line q >> 1).

// One field of a line from its Fourier modes, by a warp: raw modes get(k),
// k < K, waiting at h[k] (the even field) or h[n - k], h[K] for k = 0 (the odd
// one).  Converted by fx_xpack once both fields are there.
__device__ __forceinline__ int fx_xslot(int odd, int k, int K, int n) {
  return odd ? (k == 0 ? K : n - k) : k;
}
// The packed line F + iG of Hermitian pairs, in place, by a warp.
__device__ __forceinline__ void fx_xpack(fxc* h, int n, int K, int bF, int bG) {
  for (int k = threadIdx.x & 31; k < K; k += 32) {
    const int g = fx_xslot(1, k, K, n);
    const fxc F = fx_from2(fx_raw(h[k]), bF), G = fx_from2(fx_raw(h[g]), bG);
    h[k] = mk_fxc(F.x - G.y, F.y + G.x);
    h[g] = (k == 0) ? fx_zero() : mk_fxc(F.x + G.y, G.x - F.y);
  }
}
// Scales and packing of a line whose raw modes (of both fields) wait in h; mF,
// mG: the lane's largest fx_mag of each.
__device__ __forceinline__ void fx_xline(fxc* h, int n, int K, unsigned mF, unsigned mG, FxS& sF, FxS& sG) {
  const FxS a = fx_warp_scale(mF, K, [h](int k) { return fx_raw(h[k]); }, 2);
  const FxS b = fx_warp_scale(mG, K, [=](int k) { return fx_raw(h[fx_xslot(1, k, K, n)]); }, 2);
  if ((threadIdx.x & 31) == 0) { sF = a; sG = b; }
  __syncwarp();
  fx_xpack(h, n, K, a.base, b.base);
}
// A line of raw values of two real fields (re, im), n points, by a warp: less
// their first values (returned, for k = 0), each on its own scale.  A row that
// hardly varies is then held to the size of its variation.
__device__ __forceinline__ double2 fx_fields(fxc* h, int n, FxS& sF, FxS& sG) {
  const int lane = threadIdx.x & 31;
  const double2 ref = fx_raw(h[0]);
  __syncwarp();
  unsigned m0 = 0u, m1 = 0u;
  for (int i = lane; i < n; i += 32) {
    const double2 v = csub(fx_raw(h[i]), ref);
    h[i] = fx_bits(v.x, v.y);
    m0 = max(m0, fx_mag(v.x));
    m1 = max(m1, fx_mag(v.y));
  }
  const int e0 = (int)(__reduce_max_sync(0xffffffffu, m0) >> 20), e1 = (int)(__reduce_max_sync(0xffffffffu, m1) >> 20);
  unsigned q0 = 0u, q1 = 0u;
  for (int i = lane; i < n; i += 32) {
    const double2 v = fx_raw(h[i]);
    q0 += fx_units(v.x, e0);
    q1 += fx_units(v.y, e1);
  }
  const FxS a = fx_scale(e0, __reduce_add_sync(0xffffffffu, q0), 1);
  const FxS b = fx_scale(e1, __reduce_add_sync(0xffffffffu, q1), 1);
  if (lane == 0) { sF = a; sG = b; }
  for (int i = lane; i < n; i += 32) {
    const double2 v = fx_raw(h[i]);
    h[i] = mk_fxc(fx_from(v.x, a.base), fx_from(v.y, b.base));
  }
  return ref;
}
// Mode k of the two fields of a transformed line, unnormalised: F = (h_k +
// conj h_{-k})/2, G = (h_k - conj h_{-k})/(2i), plus n times the first values
// on k = 0.
__device__ __forceinline__ double2 fx_mode_f(const fxc* h, int n, int k, const FxS& f, double ref) {
  const fxc hk = h[k], hm = h[k == 0 ? 0 : n - k];
  double2 F = fx_to2(mk_fxc(hk.x + hm.x, hk.y - hm.y), f, 1);
  if (k == 0) F.x = fma((double)n, ref, F.x);
  return F;
}
__device__ __forceinline__ double2 fx_mode_g(const fxc* h, int n, int k, const FxS& f, double ref) {
  const fxc hk = h[k], hm = h[k == 0 ? 0 : n - k];
  double2 G = fx_to2(mk_fxc(hk.y + hm.y, hm.x - hk.x), f, 1);
  if (k == 0) G.x = fma((double)n, ref, G.x);
  return G;
}

// Lines per block of the paired rows: a warp each, within 48 KB.
inline int xrows_pairs(int n, int nrows) {
  int l = 48 * 1024 / (n * 16);
  if (l > 8) l = 8;
  while (l > 1 && (long long)l * 304 > (nrows + 1) / 2) l >>= 1;   // at least two blocks per SM
  return l < 1 ? 1 : l;
}
inline unsigned xrows_pair_blocks(int lines, int nrows) { return (unsigned)(((nrows + 1) / 2 + lines - 1) / lines); }

__device__ __forceinline__ void xrows_block(const XJob& J, Blk bk) {
  const int b = bk.y;
  if (J.status && J.status[b]) return;
  const int row = bk.x;
  const bool pr = J.pair_rows != 0;
  const int K = J.K, n = J.n, nf = J.nf;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ FxS fs[16];
  __shared__ double2 ref[8];
  fxc* A = reinterpret_cast<fxc*>(smraw);
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, nw = nt >> 5;
  const FastDiv dn = fast_div((unsigned)n);
  if (J.c2r) {
    // real field q of the block: a field of the row, or (paired rows) the row
    // r0 + q of the one field
    const int r0 = pr ? 2 * J.pair_rows * row : row;
    const int nq = pr ? min(2 * J.pair_rows, J.nrows - r0) : nf, nl = (nq + 1) / 2;
    const long long sfs = pr ? (long long)J.src_rstep * K : J.src_fstride;
    const long long dfs = pr ? (long long)J.dst_rstep * n : J.dst_fstride;
    const double2* src = J.srcC + b * J.src_mstride + (long long)r0 * J.src_rstep * K;
    for (int l = tid >> 5; l < nl; l += nw) {
      fxc* h = A + l * n;
      unsigned mF = 0u, mG = 0u;
#pragma unroll 2
      for (int k = lane; k < K; k += 32) {
        double2 F = src[(2 * l) * sfs + k];
        double2 G = (2 * l + 1 < nq) ? src[(2 * l + 1) * sfs + k] : czero();
        if (k == 0) { F.y = 0.0; G.y = 0.0; }
        h[k] = fx_bits(F.x, F.y);
        h[fx_xslot(1, k, K, n)] = fx_bits(G.x, G.y);
        mF = max(mF, fx_mag2(F));
        mG = max(mG, fx_mag2(G));
      }
      __syncwarp();
      fx_xline(h, n, K, mF, mG, fs[2 * l], fs[2 * l + 1]);
    }
    __syncthreads();
    fx_lines<+1, true>(A, nl, n, &J.pl, false);
    double* dst = J.dstR + b * J.dst_mstride + (long long)xrow_real(J, r0) * J.dst_rstep * n;
    for (int i = tid; i < nl * n; i += nt) {
      const int l = (int)fdiv((unsigned)i, dn), x = i - l * n;
      const fxc h = A[i];
      dst[(2 * l) * dfs + x] = fx_to(h.x, fs[2 * l]);
      if (2 * l + 1 < nq) dst[(2 * l + 1) * dfs + x] = fx_to(h.y, fs[2 * l + 1]);
    }
  } else {
    const int nl = (nf + 1) / 2;
    const double* src = J.srcR + b * J.src_mstride + (long long)xrow_real(J, row) * J.src_rstep * n;
    for (int l = tid >> 5; l < nl; l += nw) {
      fxc* h = A + l * n;
      for (int x = lane; x < n; x += 32)
        h[x] = fx_bits(src[(2 * l) * J.src_fstride + x], (2 * l + 1 < nf) ? src[(2 * l + 1) * J.src_fstride + x] : 0.0);
      __syncwarp();
      const double2 r = fx_fields(h, n, fs[2 * l], fs[2 * l + 1]);
      if (lane == 0) ref[l] = r;
    }
    __syncthreads();
    fx_lines<-1, true>(A, nl, n, &J.pl, false);
    double2* dst = J.dstC + b * J.dst_mstride + (long long)row * J.dst_rstep * K;
    const double inv = 1.0 / n;
    for (int l = tid >> 5; l < nl; l += nw)
      for (int k = lane; k < K; k += 32) {
        dst[(2 * l) * J.dst_fstride + k] = cscl(fx_mode_f(A + l * n, n, k, fs[2 * l], ref[l].x), inv);
        if (2 * l + 1 < nf)
          dst[(2 * l + 1) * J.dst_fstride + k] = cscl(fx_mode_g(A + l * n, n, k, fs[2 * l + 1], ref[l].y), inv);
      }
  }
}


constexpr int kFxThreads = 256;   // threads per block of the 2D fixed-point x pass, at most

__global__ void __launch_bounds__(256, 3) k_xrows(const __grid_constant__ XJob J) { xrows_block(J, this_blk()); }

__global__ void __launch_bounds__(256, 3) k_xrows_multi(const XJob* __restrict__ jobs, MultiMap mm) {
  Blk bk;
  const int q = multi_locate(mm, bk);
  xrows_block(jobs[q], bk);
}


// ------------------------------------------------------------ reductions
// The diagnostics compare, bound and count doubles through order-preserving
// integer keys: FP64 compares, min/max and additions run at the FP64 rate
// (about 1/64 of the FP32 rate here), integer ones at the ALU rate.
// key(x) < key(y) exactly when x < y, for x, y not NaN, except -0 < +0.
__device__ __forceinline__ long long dkey(double x) {
  const long long b = __double_as_longlong(x);
  return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double dkey_val(long long k) {   // inverse of dkey
  return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffLL));
}
__device__ __forceinline__ bool isnan_bits(double x) {
  return (__double_as_longlong(x) & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL;
}

// Extrema of Tr c as keys (min, max) and |Tr c| as bits (a non-negative
// double orders as its bit pattern); NaN values are left out, as fmin and
// fmax leave them out.  Empty: min LLONG_MAX, max LLONG_MIN, amax 0.
struct KeyExt {
  long long mn, mx, ma;
};
__device__ __forceinline__ KeyExt keyext_empty() {
  return KeyExt{0x7fffffffffffffffLL, (long long)0x8000000000000000ULL, 0LL};
}
__device__ __forceinline__ void keyext_add(KeyExt& e, double t) {
  if (isnan_bits(t)) return;
  const long long k = dkey(t);
  e.mn = min(e.mn, k);
  e.mx = max(e.mx, k);
  e.ma = max(e.ma, __double_as_longlong(t) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ void keyext_merge(KeyExt& e, const KeyExt& o) {
  e.mn = min(e.mn, o.mn);
  e.mx = max(e.mx, o.mx);
  e.ma = max(e.ma, o.ma);
}
__device__ __forceinline__ KeyExt keyext_shfl_down(const KeyExt& e, int o) {
  return KeyExt{__shfl_down_sync(0xffffffffu, e.mn, o), __shfl_down_sync(0xffffffffu, e.mx, o),
                __shfl_down_sync(0xffffffffu, e.ma, o)};
}

// The counts of t < 3, t < 0, |t - 3| <= tau and |t| <= tau on keys.  For
// tau <= 1.5, t - 3 is exact wherever |t - 3| <= tau can hold (Sterbenz's
// lemma), so the band is the closed interval [RU(3 - tau), RD(3 + tau)] of
// doubles; |t| <= tau is [-tau, tau] exactly.  A larger tau (a field far
// past any physical value) takes the FP64 test.  NaN counts nowhere, as in
// the FP64 comparisons.
struct TrBands {
  long long k3, lo3, hi3, lo0, hi0;
  double tau;
  bool exact;
};
__device__ __forceinline__ TrBands tr_bands(double tau) {
  TrBands B;
  B.tau = tau;
  B.exact = (tau <= 1.5);
  B.k3 = dkey(3.0);
  B.lo3 = dkey(__dsub_ru(3.0, tau));
  B.hi3 = dkey(__dadd_rd(3.0, tau));
  B.lo0 = dkey(-tau);
  B.hi0 = dkey(tau);
  return B;
}
struct TrCounts {
  int c3, c0, b3, b0;
};
__device__ __forceinline__ void tr_count(TrCounts& c, double t, const TrBands& B) {
  if (isnan_bits(t)) return;
  const long long k = dkey(t);
  c.c3 += (k < B.k3);
  c.c0 += (k < -1LL);   // below key(-0.0) = -1: negative and nonzero
  if (B.exact) {
    c.b3 += (k >= B.lo3 && k <= B.hi3);
    c.b0 += (k >= B.lo0 && k <= B.hi0);
  } else {
    c.b3 += (fabs(t - 3.0) <= B.tau);
    c.b0 += (fabs(t) <= B.tau);
  }
}

// Block reductions of the diagnostics in one barrier: warps reduce into shared
// memory (sums of FP64 in lane order, then warps in index order: a fixed order;
// counts and extrema on integers), one thread adds the warps.
constexpr int kRedWarps = 8;   // 256 threads
__device__ __forceinline__ double warp_sum_down(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ KeyExt warp_keyext(KeyExt e) {
  for (int o = 16; o > 0; o >>= 1) keyext_merge(e, keyext_shfl_down(e, o));
  return e;
}
// Tile results: energy, mean of Tr c (MEAN), extrema, counts (NC of them).
template <int NC, bool MEAN>
struct TileRed {
  double e[kRedWarps], mt[kRedWarps];
  long long mn[kRedWarps], mx[kRedWarps], ma[kRedWarps];
  int cnt[kRedWarps][NC];
  __device__ __forceinline__ void warp(double te, double tm, KeyExt x, const int (&c)[NC]) {
    const int w = threadIdx.x >> 5;
    te = warp_sum_down(te);
    if (MEAN) tm = warp_sum_down(tm);
    x = warp_keyext(x);
    int n[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) n[k] = __reduce_add_sync(0xffffffffu, c[k]);
    if ((threadIdx.x & 31) == 0) {
      e[w] = te; mt[w] = tm;
      mn[w] = x.mn; mx[w] = x.mx; ma[w] = x.ma;
#pragma unroll
      for (int k = 0; k < NC; ++k) cnt[w][k] = n[k];
    }
  }
  // after the barrier, any thread
  __device__ __forceinline__ double energy() const { return sum(e); }
  __device__ __forceinline__ double mean() const { return sum(mt); }
  __device__ __forceinline__ long long count(int k) const {
    long long t = 0;
    for (int w = 0; w < kRedWarps; ++w) t += cnt[w][k];
    return t;
  }
  __device__ __forceinline__ KeyExt ext() const {
    KeyExt x = keyext_empty();
    for (int w = 0; w < kRedWarps; ++w) keyext_merge(x, KeyExt{mn[w], mx[w], ma[w]});
    return x;
  }
  static __device__ __forceinline__ double sum(const double* v) {
    double t = v[0];
    for (int w = 1; w < kRedWarps; ++w) t += v[w];
    return t;
  }
};
// Counts of a block: out[k], k < 4, after a barrier (by threads k).
__device__ __forceinline__ void counts_warp(const TrCounts& c, int (*sh)[4]) {
  const int n0 = __reduce_add_sync(0xffffffffu, c.c3), n1 = __reduce_add_sync(0xffffffffu, c.c0);
  const int n2 = __reduce_add_sync(0xffffffffu, c.b3), n3 = __reduce_add_sync(0xffffffffu, c.b0);
  if ((threadIdx.x & 31) == 0) {
    int* o = sh[threadIdx.x >> 5];
    o[0] = n0; o[1] = n1; o[2] = n2; o[3] = n3;
  }
}
__device__ __forceinline__ long long counts_total(const int (*sh)[4], int k) {
  long long t = 0;
  for (int w = 0; w < kRedWarps; ++w) t += sh[w][k];
  return t;
}

// Sums of 32 per-thread values over the block, one total per value: a
// reduce-scatter across the lanes (at each of five levels a lane keeps half
// of its values and adds its partner's copies of them: 31 additions per
// lane, against 5 per value for a tree per value), then across the warps in
// index order.  v is consumed; on return red[k], k < 32, holds the total of
// v[k] (a fixed order: deterministic).  red: 32 * (blockDim.x / 32) doubles
// of shared memory.  Only the first nw warps hold values.
__device__ void block_sum_scatter(double (&v)[32], double* red, int nw) {
  const int l = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (w < nw)
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) {
    const bool up = (l & s) != 0;
#pragma unroll
    for (int i = 0; i < s; ++i) {
      const double send = up ? v[i] : v[i + s];
      const double keep = up ? v[i + s] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
    }
  }
  // lane l holds its warp's total of value l (index bits kept level by level)
  if (w < nw) red[w * 32 + l] = v[0];
  __syncthreads();
  if (threadIdx.x < 32) {
    double t = red[threadIdx.x];
    for (int i = 1; i < nw; ++i) t += red[i * 32 + threadIdx.x];
    red[threadIdx.x] = t;
  }
  __syncthreads();
}

// Max of the non-negative doubles stored as bits in pp[t * kPart + slot]
// over the ntile tiles of one member, on their bit patterns; every thread of
// the block receives it.
__device__ double block_tiles_amax(const double* pp, int ntile, int slot) {
  __shared__ long long smk[32];
  const long long* q = reinterpret_cast<const long long*>(pp);
  long long m = 0;
  for (int t = threadIdx.x; t < ntile; t += blockDim.x) m = max(m, q[(size_t)t * kPart + slot]);
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_down_sync(0xffffffffu, m, o));
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  __syncthreads();
  if (l == 0) smk[w] = m;
  __syncthreads();
  for (int i = 0; i < nw; ++i) m = max(m, smk[i]);
  __syncthreads();
  return __longlong_as_double(m);
}

// Histogram slot of x for the range [lo, hi) (PTT_HIST_BINS uniform bins,
// slot 0 below lo, slot PTT_HIST_BINS + 1 at or above hi or not finite);
// -1 when the quantity is switched off (lo >= hi).
__device__ __forceinline__ int hist_slot(double x, double lo, double hi) {
  if (!(lo < hi)) return -1;
  if (!isfinite(x) || x >= hi) return PTT_HIST_BINS + 1;
  if (x < lo) return 0;
  const int k = (int)floor((x - lo) * ((double)PTT_HIST_BINS / (hi - lo)));
  return 1 + min(k, PTT_HIST_BINS - 1);
}

inline unsigned cdiv(long long a, long long b) { return (unsigned)((a + b - 1) / b); }

}  // namespace
}  // namespace ptt
