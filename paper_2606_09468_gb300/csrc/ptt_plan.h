// Factorisations of the transform lengths (host code, no CUDA): which radices
// an FFT of length n runs through, and the check that they make one.
#pragma once
#include <algorithm>
#include <vector>

#if defined(__CUDACC__)
#define PTT_HOST_DEVICE __host__ __device__
#else
#define PTT_HOST_DEVICE
#endif

namespace ptt {

constexpr int kMaxStages = 8;   // passes of a plan (n <= 1080: at most 7)

// Threads of the kernels that run fixed-point passes (the fused x passes may
// have up to twice as many): a pass holds all butterflies of a line at once.
constexpr int kFxPassThreads = 256;
// Butterflies of radix R held by a thread in a fixed-point pass.  Two of
// radix 2 or 3 take no more registers than one of radix 8; with them a radix-3
// pass covers lines of up to 1536 points.  (With one of radix 3, 810, 882, 972
// and 990, lengths of ny = 401 to 496, have no factorisation.)  No other plan
// changes, and neither do the times: 20 FP64 steps of 350 x 155 (Mx = 540 =
// 3 5 6 6) 3.175 -> 3.178 ms, of the 27-run 2D sweep 35.94 -> 35.90 ms, ten of
// 3D 128 x 97 x 64 23.45 -> 23.44 ms.
PTT_HOST_DEVICE constexpr int fx_mb(int R) { return R <= 3 ? 2 : 1; }

struct HostPlan {
  int n = 0;
  std::vector<int> radix;
};

// FP32 plans (mixed groups: the padded lengths and the energy grid), radices
// 2 to 5 and 8 (few passes: each is a shared-memory round trip, and the
// transforms are bound by instruction issue).  three_first: the padded x and z
// lengths (3K or more for K kept modes), whose inverse lines are zero in the
// middle third [n/3, 2n/3): a first pass of radix 3 has one zero input; used
// where n has no factor 5.
inline HostPlan make_plan(int n, bool three_first = false) {
  HostPlan p;
  p.n = n;
  int r = n;
  if (three_first && n % 3 == 0 && n % 5 != 0) { p.radix.push_back(3); r /= 3; }
  // radix 5 first: the first pass takes no twiddles
  for (int f : {5, 8, 4, 2, 3})
    while (r % f == 0) { p.radix.push_back(f); r /= f; }
  return p;
}

// Fixed-point plans: the factorisation of least estimated time per point, from
// the cycles per warp of a butterfly (additions 2, products with a constant
// 17, twiddles 55 per complex value) and about 35 per point and pass for the
// shared-memory round trip and the indexes.  Primes 7, 11 and 13 (unpadded
// lengths) take one pass each.  The first pass is an odd radix where there is
// one: its stores are a radix apart, and even strides collide in the
// shared-memory banks; three_first as above (radix 3 or 6).
inline HostPlan make_plan_fx(int n, bool three_first = false) {
  HostPlan p;
  p.n = n;
  int r = n;
  std::vector<int> odd;
  for (int f : {13, 11, 7})
    while (r % f == 0) { odd.push_back(f); r /= f; }
  const int rad[6] = {8, 6, 5, 4, 3, 2};
  const double cost[6] = {103, 107, 121, 84, 94, 66};
  std::vector<int> best, cur;
  double bc = 1e30;
  auto search = [&](auto&& self, int m, int from, double c) -> void {
    if (c >= bc) return;
    if (m == 1) { bc = c; best = cur; return; }
    for (int i = from; i < 6; ++i)
      if (m % rad[i] == 0 && n / rad[i] <= kFxPassThreads * fx_mb(rad[i])) {
        cur.push_back(rad[i]);
        self(self, m / rad[i], i, c + cost[i]);
        cur.pop_back();
      }
  };
  search(search, r, 0, 0.0);
  auto lead = [&](int f) {
    auto it = std::find(best.begin(), best.end(), f);
    if (it == best.end()) return false;
    best.erase(it);
    p.radix.push_back(f);
    return true;
  };
  if (three_first) { if (!lead(3)) lead(6); }
  else if (odd.empty() && !lead(5)) lead(3);
  p.radix.insert(p.radix.end(), odd.begin(), odd.end());
  // then by size: the later passes' stores are contiguous
  for (int f : {5, 3, 6, 4, 2, 8})
    for (int b : best)
      if (b == f) p.radix.push_back(f);
  return p;
}

// Whether a plan is one: its radices multiply to n and are few enough, and (fx)
// every pass's butterflies fit the threads that run them.
inline bool plan_ok(const HostPlan& p, bool fx) {
  long long m = 1;
  for (int R : p.radix) {
    m *= R;
    if (fx && p.n / R > kFxPassThreads * fx_mb(R)) return false;
  }
  return m == p.n && p.radix.size() <= (size_t)kMaxStages;
}

}  // namespace ptt
