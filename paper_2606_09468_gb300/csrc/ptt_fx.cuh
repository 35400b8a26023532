// FP64-accurate Fourier transforms in 64-bit block fixed point.
//
// One FP64 instruction holds this part's FP64 pipe of an SM sub-partition for
// 64 cycles per warp (measured: DADD, DMUL and DFMA loops); an integer
// addition takes 1, a 32 x 32 -> 64-bit product (mul.wide.s32) 4 cycles.  An
// FFT is additions and products with constants of modulus at most 1, so its
// values have a known common scale, and 64-bit integers on that scale carry
// more digits than FP64 does: a twiddled radix-8 butterfly takes about 550
// cycles per warp here against about 4200 on the FP64 pipe (66 FP64
// instructions).  3D 128 x 97 x 64, FP64, launch-shape defaults: the fused x
// pass 3.40 -> 0.94 ms, inverse y and z 1.56 -> 0.71 ms, forward 0.70 -> 0.27
// ms; the 27-run 2D sweep 3.85 -> 1.88 ms per step.
//
// A line of complex values x_k is taken to integers v_k = x_k 2^B with
//   sum_k (|re x_k| + |im x_k|) 2^B < 2^60,
// the largest such power of two up to a factor 2 (the sum is formed on the
// top 20 mantissa bits).  Every intermediate and result of the transform is
// a sum of the inputs with coefficients of modulus at most 1, so it stays
// below 2^60 and needs no further scaling; the butterflies' own partial sums
// stay below 2^61.  Additions are exact; a product with a twiddle or a
// butterfly constant (62 fractional bits) drops only the product of the low
// halves and the final shift, an error of about one unit.  A unit is 2^-60 of
// the line's sum of moduli: with N inputs of like size about 2^-60 N of one,
// with one input dominating 2^-60 of it, against FP64's 2^-53 sqrt(N) and
// 2^-53.
//
// A field (or complex line) with a NaN or an infinity gives NaN everywhere
// (an FFT in floating point spreads them over the whole line, too).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "ptt_internal.h"

namespace ptt {
namespace {

struct __align__(16) fxc { long long x, y; };   // re, im on a line's scale

__device__ __forceinline__ fxc mk_fxc(long long x, long long y) { fxc r; r.x = x; r.y = y; return r; }
__device__ __forceinline__ fxc cadd(fxc a, fxc b) { return mk_fxc(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ fxc csub(fxc a, fxc b) { return mk_fxc(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ fxc mul_i(fxc a) { return mk_fxc(-a.y, a.x); }
__device__ __forceinline__ fxc fx_zero() { return mk_fxc(0, 0); }
// The raw doubles of a line wait in its buffer as bit patterns.  Between two
// barriers a buffer is read and written as one type (the compiler may reorder
// accesses of different types).
__device__ __forceinline__ double2 fx_raw(fxc v) {
  return make_double2(__longlong_as_double(v.x), __longlong_as_double(v.y));
}
__device__ __forceinline__ fxc fx_bits(double x, double y) {
  return mk_fxc(__double_as_longlong(x), __double_as_longlong(y));
}

// mul.wide and mad.wide as single instructions: half the time of what the
// compiler makes of the same sums in C (56 against 108 cycles per warp for a
// complex product)
__device__ __forceinline__ long long fx_mw(int a, int b) {
  long long r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
}
// v = h 2^32 + l with l signed
__device__ __forceinline__ int fx_lo(long long v) { return (int)v; }
__device__ __forceinline__ int fx_hi(long long v) { return (int)(v >> 32) - ((int)v >> 31); }

__device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
// a w (CONJ: a conj w), w = (c, s) in 62 fractional bits, each split into a
// high and a signed low half: (c_h, c_l, s_h, s_l).  |a| < 2^61.
template <bool CONJ>
__device__ __forceinline__ fxc fx_cmul(fxc a, int4 w) {
  const int rl = fx_lo(a.x), rh = fx_hi(a.x), il = fx_lo(a.y), ih = fx_hi(a.y);
  const int sh = CONJ ? -w.z : w.z, sl = CONJ ? -w.w : w.w, nh = -sh, nl = -sl;
  const long long m = fx_mad(ih, nl, fx_mad(il, nh, fx_mad(rh, w.y, fx_mw(rl, w.x))));
  const long long n = fx_mad(ih, w.y, fx_mad(il, w.x, fx_mad(rh, sl, fx_mw(rl, sh))));
  const int r4 = rh << 2, i4 = ih << 2;
  return mk_fxc(fx_mad(i4, nh, fx_mad(r4, w.x, m >> 30)), fx_mad(i4, w.x, fx_mad(r4, sh, n >> 30)));
}
// a c - b s
__device__ __forceinline__ long long fx_dot(long long a, long long b, int4 w) {
  const int al = fx_lo(a), ah = fx_hi(a), bl = fx_lo(b), bh = fx_hi(b);
  const long long m = (fx_mw(al, w.x) + fx_mw(ah, w.y)) - (fx_mw(bl, w.z) + fx_mw(bh, w.w));
  return (m >> 30) + (fx_mw(ah << 2, w.x) - fx_mw(bh << 2, w.z));
}
// v K 2^-62 for a compile-time constant, |K| < 2^63
template <long long K>
__device__ __forceinline__ long long fx_kmul(long long v) {
  constexpr int kl = (int)(K & 0xffffffffLL);
  constexpr int kh = (int)((K - (long long)kl) >> 32);
  const int l = fx_lo(v), h = fx_hi(v);
  return ((fx_mw(l, kh) + fx_mw(h, kl)) >> 30) + fx_mw(h << 2, kh);
}
template <long long K>
__device__ __forceinline__ fxc fx_kmul2(fxc a) { return mk_fxc(fx_kmul<K>(a.x), fx_kmul<K>(a.y)); }

// ------------------------------------------------------------ butterflies
// DIR = -1: exp(-2 pi i jk/R); DIR = +1: the conjugate.  Constants in 62
// fractional bits.
constexpr long long kFxSin60 = 3993837246235628775LL;      // sin(2 pi/3)
constexpr long long kFxRt8 = 3260954456333195553LL;        // 1/sqrt 2
constexpr long long kFxRt5 = 2578010857022246787LL;        // sqrt(5)/4
constexpr long long kFxS1 = 4385974038932618941LL;         // sin(2 pi/5)
constexpr long long kFxS1mS2 = 1675293009097605857LL;      // sin(2 pi/5) - sin(4 pi/5)
constexpr long long kFxS1pS2 = 7096655068767632024LL;      // sin(2 pi/5) + sin(4 pi/5)

template <int DIR> __device__ __forceinline__ fxc fx_iadd(fxc a, fxc b) {   // a + DIR i b
  return DIR > 0 ? mk_fxc(a.x - b.y, a.y + b.x) : mk_fxc(a.x + b.y, a.y - b.x);
}

template <int DIR, int R> struct FxBfly;
template <int DIR> struct FxBfly<DIR, 2> {
  static __device__ __forceinline__ void run(fxc* v) {
    const fxc t = v[0];
    v[0] = cadd(t, v[1]);
    v[1] = csub(t, v[1]);
  }
};
template <int DIR> struct FxBfly<DIR, 3> {
  static __device__ __forceinline__ void run(fxc* v) {
    const fxc t = cadd(v[1], v[2]), d = fx_kmul2<kFxSin60>(csub(v[1], v[2]));
    const fxc m = mk_fxc(v[0].x - (t.x >> 1), v[0].y - (t.y >> 1));
    v[0] = cadd(v[0], t);
    v[1] = fx_iadd<DIR>(m, d);
    v[2] = fx_iadd<-DIR>(m, d);
  }
};
template <int DIR> struct FxBfly<DIR, 4> {
  static __device__ __forceinline__ void run(fxc* v) {
    const fxc s = cadd(v[0], v[2]), d = csub(v[0], v[2]);
    const fxc t = cadd(v[1], v[3]), e = csub(v[1], v[3]);
    v[0] = cadd(s, t);
    v[2] = csub(s, t);
    v[1] = fx_iadd<DIR>(d, e);
    v[3] = fx_iadd<-DIR>(d, e);
  }
};
// Radix 5 with t1 = v1 + v4, t2 = v2 + v3, d1 = v1 - v4, d2 = v2 - v3:
// cos(2 pi/5), cos(4 pi/5) = (-1 +- sqrt 5)/4, so
//   b1,2 = v0 - (t1 + t2)/4 +- (sqrt 5/4)(t1 - t2),
// and with k = S1 (d1 + d2): S1 d1 + S2 d2 = k - (S1 - S2) d2,
// S2 d1 - S1 d2 = (S1 + S2) d1 - k (8 real products instead of 16).
template <int DIR> struct FxBfly<DIR, 5> {
  static __device__ __forceinline__ void run(fxc* v) {
    const fxc t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
    const fxc d1 = csub(v[1], v[4]), d2 = csub(v[2], v[3]);
    const fxc a = cadd(t1, t2);
    const fxc q = fx_kmul2<kFxRt5>(csub(t1, t2));
    const fxc m = mk_fxc(v[0].x - (a.x >> 2), v[0].y - (a.y >> 2));
    const fxc b1 = cadd(m, q), b2 = csub(m, q);
    const fxc k = fx_kmul2<kFxS1>(cadd(d1, d2));
    const fxc e1 = csub(k, fx_kmul2<kFxS1mS2>(d2));
    const fxc e2 = csub(fx_kmul2<kFxS1pS2>(d1), k);
    v[0] = cadd(v[0], a);
    v[1] = fx_iadd<DIR>(b1, e1);
    v[4] = fx_iadd<-DIR>(b1, e1);
    v[2] = fx_iadd<DIR>(b2, e2);
    v[3] = fx_iadd<-DIR>(b2, e2);
  }
};
// Radix 6 without twiddles (Good's prime-factor mapping): input
// (3 n1 + 2 n2) mod 6, output by the Chinese remainder theorem.
template <int DIR> struct FxBfly<DIR, 6> {
  static __device__ __forceinline__ void run(fxc* v) {
    fxc a[3], b[3];
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      const fxc p = v[(2 * n) % 6], q = v[(3 + 2 * n) % 6];
      a[n] = cadd(p, q);
      b[n] = csub(p, q);
    }
    FxBfly<DIR, 3>::run(a);
    FxBfly<DIR, 3>::run(b);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      v[(4 * k) % 6] = a[k];
      v[(3 + 4 * k) % 6] = b[k];
    }
  }
};
template <int DIR> struct FxBfly<DIR, 8> {
  static __device__ __forceinline__ void run(fxc* v) {
    fxc a[4], b[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      a[r] = cadd(v[r], v[r + 4]);
      b[r] = csub(v[r], v[r + 4]);
    }
    // times w, w^2, w^3, w = (1 + DIR i)/sqrt 2
    b[1] = fx_kmul2<kFxRt8>(fx_iadd<DIR>(b[1], b[1]));
    b[2] = DIR > 0 ? mk_fxc(-b[2].y, b[2].x) : mk_fxc(b[2].y, -b[2].x);
    b[3] = fx_kmul2<kFxRt8>(DIR > 0 ? mk_fxc(-b[3].x - b[3].y, b[3].x - b[3].y)
                                    : mk_fxc(b[3].y - b[3].x, -b[3].x - b[3].y));
    FxBfly<DIR, 4>::run(a);
    FxBfly<DIR, 4>::run(b);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[2 * k] = a[k];
      v[2 * k + 1] = b[k];
    }
  }
};
// Odd primes 7, 11, 13 (unpadded lengths): y_j, y_{R-j} = b_j +- i DIR e_j with
// b_j = v_0 + sum_k cos(2 pi jk/R) t_k, e_j = sum_k sin(2 pi jk/R) d_k.
template <int R, int M> struct FxOdd;   // cos, sin of 2 pi M/R
#define PTT_FX_ODD(R, M, CV, SV) \
  template <> struct FxOdd<R, M> { static constexpr long long c = CV##LL, s = SV##LL; }
PTT_FX_ODD(7, 1, 2875339201863983833, 3605561316464170519);
PTT_FX_ODD(7, 2, -1026196679933739317, 4496061421583520199);
PTT_FX_ODD(7, 3, -4154985531143938469, 2000935573311439104);
PTT_FX_ODD(11, 1, 3879597155310203735, 2493265698851133051);
PTT_FX_ODD(11, 2, 1915763607305631188, 4194937154890639038);
PTT_FX_ODD(11, 3, -656311349879663986, 4564745704261934814);
PTT_FX_ODD(11, 4, -3020012090752568663, 3485279745481982533);
PTT_FX_ODD(11, 5, -4424880331197296226, 1299262093321420667);
PTT_FX_ODD(13, 1, 4083445173437190589, 2143157354953472948);
PTT_FX_ODD(13, 2, 2619736250061566421, 3795343187733095619);
PTT_FX_ODD(13, 3, 555877323041125914, 4578061635046789725);
PTT_FX_ODD(13, 4, -1635326399640084757, 4312001333394836946);
PTT_FX_ODD(13, 5, -3451896551983290448, 3058113491511478315);
PTT_FX_ODD(13, 6, -4477678804130201671, 1103648702985592706);
#undef PTT_FX_ODD
template <int R, int J, int K> struct FxOddAcc {   // adds the terms k = K .. 1 of row J
  static __device__ __forceinline__ void run(const fxc* t, const fxc* d, fxc& b, fxc& e) {
    constexpr int H = (R - 1) / 2, mm = (J * K) % R, mi = (mm <= H) ? mm : R - mm;
    FxOddAcc<R, J, K - 1>::run(t, d, b, e);
    b = cadd(b, fx_kmul2<FxOdd<R, mi>::c>(t[K - 1]));
    const fxc p = fx_kmul2<FxOdd<R, mi>::s>(d[K - 1]);
    e = (mm <= H) ? cadd(e, p) : csub(e, p);
  }
};
template <int R, int J> struct FxOddAcc<R, J, 0> {
  static __device__ __forceinline__ void run(const fxc*, const fxc*, fxc&, fxc&) {}
};
template <int DIR, int R, int J> struct FxOddRows {
  static __device__ __forceinline__ void run(const fxc* t, const fxc* d, fxc v0, fxc* y) {
    FxOddRows<DIR, R, J - 1>::run(t, d, v0, y);
    fxc b = v0, e = fx_zero();
    FxOddAcc<R, J, (R - 1) / 2>::run(t, d, b, e);
    y[J] = fx_iadd<DIR>(b, e);
    y[R - J] = fx_iadd<-DIR>(b, e);
  }
};
template <int DIR, int R> struct FxOddRows<DIR, R, 0> {
  static __device__ __forceinline__ void run(const fxc*, const fxc*, fxc, fxc*) {}
};
template <int DIR, int R> struct FxBflyOdd {
  static __device__ __forceinline__ void run(fxc* v) {
    constexpr int H = (R - 1) / 2;
    fxc t[H], d[H], y[R];
    y[0] = v[0];
#pragma unroll
    for (int k = 1; k <= H; ++k) {
      t[k - 1] = cadd(v[k], v[R - k]);
      d[k - 1] = csub(v[k], v[R - k]);
      y[0] = cadd(y[0], t[k - 1]);
    }
    FxOddRows<DIR, R, H>::run(t, d, v[0], y);
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = y[r];
  }
};
template <int DIR> struct FxBfly<DIR, 7> : FxBflyOdd<DIR, 7> {};
template <int DIR> struct FxBfly<DIR, 11> : FxBflyOdd<DIR, 11> {};
template <int DIR> struct FxBfly<DIR, 13> : FxBflyOdd<DIR, 13> {};

// ------------------------------------------------------------ passes
// One Stockham pass of radix R over nl lines (line l at offset l * ls), in
// place: the lines go in groups whose butterflies sit in registers, one per
// thread (fx_mb(R) of radix 2 and 3); the block waits between a group's loads
// and its stores.  One buffer instead of two: the 3D x pass at 192 points takes
// 55 KB a block, so several blocks share an SM and one block's barriers and
// FP64 products run under another's butterflies.  (More butterflies per
// thread would save barriers, but ptxas spills them.)  The twiddles of a pass
// are stored [r - 1][jm], consecutive lanes reading consecutive entries.
// Needs n / R <= fx_mb(R) blockDim.x (fx_min_threads).
struct FxPassC {
  int nb, Ns;
  unsigned mb, ms;   // multiply-high reciprocals (0: divisor 1)
};
__device__ __forceinline__ unsigned fx_div(unsigned x, unsigned m) { return m == 0u ? x : __umulhi(x, m); }

// Shared-memory accesses by 32-bit address.
__device__ __forceinline__ fxc fx_lds(unsigned a) {
  fxc v;
  asm volatile("ld.shared.v2.s64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void fx_sts(unsigned a, fxc v) {
  asm volatile("st.shared.v2.s64 [%0], {%1, %2};" ::"r"(a), "l"(v.x), "l"(v.y) : "memory");
}

// ZM: the line is zero in its middle third (first pass, radix 3 or 6).
template <int DIR, int R, bool ZM>
__device__ __forceinline__ void fx_pass(unsigned a, int nl, int ls, const FxPassC c, const int4* __restrict__ tw) {
  constexpr int MB = fx_mb(R);
  const int nb = c.nb, Ns = c.Ns, tid = threadIdx.x, nt = blockDim.x;
  const int per = max(1, (int)fx_div((unsigned)(nt * MB), c.mb));
  for (int l0 = 0; l0 < nl; l0 += per) {
    const int total = min(per, nl - l0) * nb;
    const unsigned base = a + (unsigned)(l0 * ls) * 16u;
    fxc v[MB][R];
#pragma unroll
    for (int q = 0; q < MB; ++q) {
      // threads past the end load the last butterfly: a register array that is
      // set on one side of a branch only stays live in every pass (and spills)
      const int t = min(tid + q * nt, total - 1);
      const int l = (int)fx_div((unsigned)t, c.mb), j = t - l * nb;
      const unsigned s = base + (unsigned)(l * ls + j) * 16u;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const bool z = ZM && 3 * r >= R && 3 * r < 2 * R;
        v[q][r] = z ? fx_zero() : fx_lds(s + (unsigned)(r * nb) * 16u);
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < MB; ++q) {
      const int t = tid + q * nt;
      if (t < total) {
        const int l = (int)fx_div((unsigned)t, c.mb), j = t - l * nb;
        const int jq = (int)fx_div((unsigned)j, c.ms), jm = j - jq * Ns;
        if (Ns > 1) {
#pragma unroll
          for (int r = 1; r < R; ++r) v[q][r] = fx_cmul<(DIR > 0)>(v[q][r], __ldg(&tw[(r - 1) * Ns + jm]));
        }
        FxBfly<DIR, R>::run(v[q]);
        const unsigned d = base + (unsigned)(l * ls + jq * Ns * R + jm) * 16u;
#pragma unroll
        for (int r = 0; r < R; ++r) fx_sts(d + (unsigned)(r * Ns) * 16u, v[q][r]);
      }
    }
  }
  __syncthreads();
}

// Unnormalised DFT of nl lines of length pl.n in place, at A (shared memory,
// line l at l * ls).  zero_mid: the lines are zero in their middle third
// [n/3, 2n/3).  BIG: the plan may hold radices 7, 11, 13 (unpadded lengths; the
// padded ones are 5-smooth).  Called by the whole block after a
// __syncthreads(); ends with one.
template <int DIR, bool BIG>
__device__ __forceinline__ void fx_lines(fxc* A, int nl, int ls, const FftPlan* plan, bool zero_mid) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(A);
  const FftPlan& pl = *plan;
  for (int s = 0; s < pl.nst; ++s) {
    const int R = pl.radix[s];
    const FxPassC c{pl.pnb[s], pl.pns[s], pl.pmb[s], pl.pms[s]};
    const int4* tw = pl.twx + pl.xoff[s];
    const bool zm = zero_mid && s == 0;
    switch (R) {
      case 2: fx_pass<DIR, 2, false>(a, nl, ls, c, tw); break;
      case 3:
        if (DIR > 0 && zm) fx_pass<DIR, 3, true>(a, nl, ls, c, tw);
        else fx_pass<DIR, 3, false>(a, nl, ls, c, tw);
        break;
      case 4: fx_pass<DIR, 4, false>(a, nl, ls, c, tw); break;
      case 5: fx_pass<DIR, 5, false>(a, nl, ls, c, tw); break;
      case 6:
        if (DIR > 0 && zm) fx_pass<DIR, 6, true>(a, nl, ls, c, tw);
        else fx_pass<DIR, 6, false>(a, nl, ls, c, tw);
        break;
      case 8: fx_pass<DIR, 8, false>(a, nl, ls, c, tw); break;
      default:
        if constexpr (BIG) {
          if (R == 7) fx_pass<DIR, 7, false>(a, nl, ls, c, tw);
          else if (R == 11) fx_pass<DIR, 11, false>(a, nl, ls, c, tw);
          else if (R == 13) fx_pass<DIR, 13, false>(a, nl, ls, c, tw);
        }
        break;
    }
  }
}

// ------------------------------------------------------------ scales
// One scale per complex line, or, in lines that pack two real fields, one
// per field: the transform is linear and keeps the two apart, so each is
// held to its own size however much larger the other is (c_xx ~ 3e4 rides
// with dv/dx ~ 1e-3).  A warp takes a whole line: its maximum, then the sum
// of moduli, are warp reductions over integers (their order does not matter),
// and the line is converted with no wait for the rest of the block.
struct __align__(16) FxS {
  int C;             // v = x 2^(1084 - C)
  unsigned am, om;   // masks of the results' words: a zero line, a bad line (NaN)
  int base;          // right shift of a value with exponent field e: base - e
};
__device__ __forceinline__ unsigned d_hi(double d) { return (unsigned)__double2hiint(d); }
__device__ __forceinline__ unsigned d_lo(double d) { return (unsigned)__double2loint(d); }
// |x| as an ordered integer (the high word)
__device__ __forceinline__ unsigned fx_mag(double x) { return d_hi(x) & 0x7FFFFFFFu; }
__device__ __forceinline__ unsigned fx_mag2(double2 v) { return max(fx_mag(v.x), fx_mag(v.y)); }
// Upper bound of |x| in units of 2^(emax - 1042).
__device__ __forceinline__ unsigned fx_units(double x, int emax) {
  const unsigned h = d_hi(x);
  const int e = (int)((h >> 20) & 0x7FFu);
  const unsigned m = (h & 0xFFFFFu) | 0x100000u;
  return (e == 0) ? 0u : (m >> min(emax - e + 1, 31)) + 1u;
}
// The scale of a line with largest exponent field emax and sum of moduli
// below sum 2^(emax - 1042), whose transform inputs may exceed that sum by
// 2^extra: |x| < 2^(nbits + emax - 1042) in sum, so v = x 2^B with
// B = 1102 - extra - nbits - emax stays below 2^(60 - extra) in sum; a 53-bit
// mantissa shifted left by 8 then goes right by (emax - e) + nbits + extra - 19
// >= 1.  A line of zeros (or of values below 2^-927, where fx_to's exponents end)
// gives exact zeros: its part of a packed line holds the other field's rounding.
// One with a NaN or an infinity, or whose results could pass the largest double
// (a sum of moduli of 2^1018 or more), gives NaN.
constexpr int kFxMaxC = 2044;     // results below 2^62 units: exponent fields up to C + 2
constexpr int kFxMinExp = 96;     // fx_to: C - 60 - k >= emax + 2 - 60 - 28 > 0
__device__ __forceinline__ FxS fx_scale(int emax, unsigned sum, int extra) {
  FxS s;
  const int nbits = 32 - __clz((int)sum), C = emax + nbits + extra - 18;
  const bool zero = emax < kFxMinExp, bad = emax == 2047 || C > kFxMaxC;
  s.C = (zero || bad) ? 1084 : C;
  s.am = (zero || bad) ? 0u : 0xFFFFFFFFu;
  s.om = bad ? 0x7FF80000u : 0u;
  s.base = (zero || bad) ? 4096 : C - 1;
  return s;
}
// The scale of a line of cnt values get(i); m: the lane's largest fx_mag of
// the values i = lane, lane + 32, ...  Called by a whole warp.
template <typename Get>
__device__ __forceinline__ FxS fx_warp_scale(unsigned m, int cnt, Get get, int extra) {
  const int emax = (int)(__reduce_max_sync(0xffffffffu, m) >> 20);
  unsigned q = 0u;
  for (int i = threadIdx.x & 31; i < cnt; i += 32) {
    const double2 v = get(i);
    q += fx_units(v.x, emax) + fx_units(v.y, emax);
  }
  return fx_scale(emax, __reduce_add_sync(0xffffffffu, q), extra);
}

// x on a line's scale (FxS::base), rounded to nearest (half a unit
// of input error spreads over the line like the sqrt of its length, the
// largest part of the transforms' error).
__device__ __forceinline__ long long fx_from(double x, int base) {
  const unsigned h = d_hi(x), l = d_lo(x);
  const int e = (int)((h >> 20) & 0x7FFu);
  const unsigned mh = (h & 0xFFFFFu) | 0x100000u;
  const unsigned long long M = ((unsigned long long)__funnelshift_l(l, mh, 8) << 32) | (l << 8);
  unsigned long long v;   // twice the magnitude; shifts beyond 63 give 0
  asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(M), "r"(base - 1 - e));
  const long long s = (long long)((int)h >> 31);
  return (((long long)v ^ s) + 1) >> 1;   // for s = -1: floor(-v/2)
}
__device__ __forceinline__ fxc fx_from2(double2 v, int base) { return mk_fxc(fx_from(v.x, base), fx_from(v.y, base)); }

// A complex line of n raw values onto its scale, in place, by a warp.
__device__ __forceinline__ void fx_line(fxc* h, int n, FxS& sc) {
  const int lane = threadIdx.x & 31;
  unsigned m = 0u;
  for (int i = lane; i < n; i += 32) m = max(m, fx_mag2(fx_raw(h[i])));
  const FxS s = fx_warp_scale(m, n, [h](int i) { return fx_raw(h[i]); }, 0);
  if (lane == 0) sc = s;
  for (int i = lane; i < n; i += 32) h[i] = fx_from2(fx_raw(h[i]), s.base);
}

// v 2^(C - 1084 - k) as a double, rounded to nearest by about 26 integer
// instructions (a conversion and a scaling would hold the FP64 pipe for 128
// cycles).  The magnitude is the ones' complement of a negative v, one unit
// short; its top bit's position comes from the leading word rounded down to
// FP32 (the low word, two bits down, when the high one is zero).  Below four
// units (t = 0) the result is zero, so sh <= 30 wherever it counts and the
// exponent, C - k - 60 at least, is positive for k <= 28 (fexpP, at most
// log2 of 800 768 768).  (Its two instructions take no time that shows: 3D
// 128 x 97 x 64 23.43 and 23.33 ms for ten steps, the 2D sweep 35.91 and 35.82.)
__device__ __forceinline__ double fx_to(long long v, const FxS& f, int k = 0) {
  const int s = (int)(v >> 63);
  const unsigned hi = (unsigned)((int)(v >> 32) ^ s), lo = (unsigned)((int)v ^ s);
  const bool big = hi != 0u;
  const unsigned t = big ? hi : lo >> 2, l = big ? lo : lo << 30;
  const unsigned am = t ? f.am : 0u;
  const int sh = 157 - (int)(__float_as_uint(__uint2float_rz(t)) >> 23);   // top bit to bit 62
  const unsigned long long N =
      (((unsigned long long)__funnelshift_l(l, t, sh) << 32) | (l << (sh & 31))) + 0x200u;
  const unsigned H = (unsigned)(N >> 32), L = (unsigned)N;
  const unsigned hw = (H >> 10) + ((unsigned)(f.C - k - (big ? 0 : 30) - sh) << 20);
  return __hiloint2double((int)(((hw | ((unsigned)s & 0x80000000u)) & am) | f.om),
                          (int)(__funnelshift_r(L, H, 10) & am));
}
__device__ __forceinline__ double2 fx_to2(fxc v, const FxS& f, int k = 0) {
  return make_double2(fx_to(v.x, f, k), fx_to(v.y, f, k));
}

}  // namespace
}  // namespace ptt
