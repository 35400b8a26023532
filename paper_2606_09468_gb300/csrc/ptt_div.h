// Unsigned division by a runtime divisor through a multiply-high, for the device
// and (the same arithmetic) for host code without CUDA.
#pragma once

#if defined(__CUDACC__)
#define PTT_DIV __host__ __device__ __forceinline__
#else
#define PTT_DIV inline
#endif

namespace ptt {

// The method of Granlund and Montgomery, "Division by invariant integers using
// multiplication", PLDI 1994, in its round-up form: with
// m = floor((2^32 - 1)/d) + 1 = ceil(2^32/d), (x m) >> 32 exceeds x/d by
// x (m d - 2^32)/(d 2^32), less than x/2^32.  So fdiv is floor(x/d) exactly
// wherever x d < 2^32 (the excess is then below 1/d): every index within a
// block's lines, a 2D energy grid or the rows of a z pass (x < 2^21, d < 2^11).
// For any x the excess is below one and the quotient at most one too high, which
// fdiv_any takes back.  d = 1 is passed through.
struct FastDiv {
  unsigned m;
  bool one;
};
PTT_DIV FastDiv fast_div(unsigned d) {
  FastDiv f;
  f.one = (d == 1u);
  f.m = f.one ? 0u : 0xFFFFFFFFu / d + 1u;
  return f;
}
PTT_DIV unsigned fdiv(unsigned x, FastDiv f) {
#if defined(__CUDA_ARCH__)
  return f.one ? x : __umulhi(x, f.m);
#else
  return f.one ? x : (unsigned)(((unsigned long long)x * f.m) >> 32);
#endif
}
// floor(x/d) for any x (d the divisor of f).
PTT_DIV unsigned fdiv_any(unsigned x, FastDiv f, unsigned d) {
  const unsigned q = fdiv(x, f);
  return q * d > x ? q - 1u : q;   // q d <= x + d - 1: no wrap while x + d < 2^32
}

}  // namespace ptt
