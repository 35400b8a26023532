// Device code of the 3D pseudo-spectral sPTT channel step (sm_103a).
//
// Nine fields u, v, w, c_xx, c_xy, c_xz, c_yy, c_yz, c_zz; spectral arrays
// [member][field][mode][n] with mode = mx * nz + mz (mx < nx/2, mz in FFT
// order, the Nyquist slot nz/2 kept zero).  One step (Sec. 2):
//   k_ycols  (inverse)  17 columns per mode on the padded Gauss y grid
//                       (9 fields and 8 y-derivatives; d/dy of v follows from
//                       continuity)
//   k_zcols  (inverse)  per (y row, mx) line: 26 z syntheses of length Mz
//                       (the 17 fields and 9 z-derivatives)
//   k_xfused3           per (y, z) row: 35 physical fields (9 more
//                       x-derivatives), the products of Eqs. 1-2, 9 forward
//                       x transforms
//   k_zcols  (forward), k_ycols (forward): back to truncated spectral terms
//   k_spec3             per mode: explicit linear terms, SBDF sums, tau solves
//                       (six c, phi-v with the influence correction, eta; U and
//                       W on the mean mode), u and w from continuity and eta
//   k_tick              step counters
// followed by the Sec. 3 diagnostics over the nx x ny x nz grid and the
// (x, z) mid-plane.
#include <cstdio>

#include "ptt_device.cuh"

namespace ptt {
namespace {

// ------------------------------------------------------------ z lines
// Inverse: src [field][j][mx*nz + mz] (modes) -> dst [field][j][z][mx] (values
// at Mz points, optional d/dz).  Forward: src [field][j][z][mx] (values) ->
// dst [field][j][mx*nz + mz] (modes, truncated, Nyquist slot zero).
struct ZJob {
  const void* src;
  void* dst;
  long long src_mstride, dst_mstride;  // per member (elements)
  long long src_fstride, dst_fstride;  // per field (elements)
  int src_field[32];
  int dst_field[32];
  int dz[32];         // inverse: transform d/dz of the field
  int K, nz, Mz;      // x modes, z modes, z points
  double inv;         // forward: 1 / Mz (host-computed), and its FP32 rounding
  float invf;
  int inverse;
  int C;              // mx lines per block
  int rows;           // y rows per field
  const int* status;
  const MemberPrm* prm;
  FftPlan pl;         // length Mz
  FastDiv dC, dnz, dMz, drows;   // of C, nz, Mz, rows (z_set_lines)
  // mixed groups' step passes (mean/fluctuation split, see k_xfused3):
  // mean = 1, inverse: the kx = 0 line leaves its kz = 0 (mean) mode out;
  // mean = 2, forward: the kx = 0 line's mean mode is added in FP64 to
  // zm[member][dst field][row] and left zero in dst
  int mean;
  double2* zm;
};

// Fixed-point z lines between FP64 arrays.  BIG: unpadded z length nz
// (radices 7, 11, 13 possible); the padded length Mz of the step runs
// without it.  Forward: times J.inv (1 in the step, whose y table holds the
// normalisation).
template <bool BIG>
__global__ void __launch_bounds__(256, BIG ? 3 : 5) k_zcols_fx(const __grid_constant__ ZJob J) {
  const int b = blockIdx.z;
  if (J.status && J.status[b]) return;
  const int f = blockIdx.y / J.rows;
  const int j = blockIdx.y - f * J.rows;
  const int C = J.C, K = J.K, nz = J.nz, Mz = J.Mz;
  const int m0 = blockIdx.x * C;
  const int nc = min(C, K - m0);
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ FxS fs[64];
  fxc* A = reinterpret_cast<fxc*>(smraw);
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, nw = nt >> 5;
  const int hz = nz / 2;
  const FastDiv dC = fast_div((unsigned)C);
  if (J.inverse) {
    const double2* src = static_cast<const double2*>(J.src) + b * J.src_mstride +
                         J.src_field[f] * J.src_fstride + (long long)j * K * nz;
    double2* dst = static_cast<double2*>(J.dst) + b * J.dst_mstride + J.dst_field[f] * J.dst_fstride +
                   (long long)j * Mz * K;
    const double kfac = J.prm[b].kz1;
    const int dz = J.dz[f], gap = Mz - nz;
    for (int c = tid >> 5; c < nc; c += nw) {   // a warp per line
      fxc* h = A + c * Mz;
      const double2* s = src + (long long)(m0 + c) * nz;
      unsigned m = 0u;
#pragma unroll 2
      for (int q = lane; q < nz; q += 32) {   // modes 0 .. hz-1, the slot hz (zero), the negative ones
        double2 v = czero();
        if (q != hz) {
          v = s[q];
          if (dz) v = cscl(mul_i(v), kfac * (q < hz ? q : q - nz));
        }
        h[q <= hz ? q : q + gap] = fx_bits(v.x, v.y);
        m = max(m, fx_mag2(v));
      }
      for (int q = hz + 1 + lane; q <= hz + gap; q += 32) h[q] = fx_zero();
      __syncwarp();
      auto at = [=](int q) { return q <= hz ? q : q + gap; };
      const FxS sc = fx_warp_scale(m, nz, [=](int q) { return fx_raw(h[at(q)]); }, 0);
      if (lane == 0) fs[c] = sc;
      __syncwarp();
      for (int q = lane; q < nz; q += 32) h[at(q)] = fx_from2(fx_raw(h[at(q)]), sc.base);
    }
    __syncthreads();
    // padded synthesis (Mz >= 3 nz/2): the slots nz/2 .. Mz - nz/2 are zero
    fx_lines<+1, BIG>(A, nc, Mz, &J.pl, J.pl.radix[0] % 3 == 0 && Mz >= 3 * hz);
    for (int i = tid; i < Mz * C; i += nt) {
      const int z = (int)fdiv((unsigned)i, dC), c = i - z * C;
      if (c < nc) dst[(long long)z * K + m0 + c] = fx_to2(A[c * Mz + z], fs[c]);
    }
  } else {
    const double2* src = static_cast<const double2*>(J.src) + b * J.src_mstride +
                         J.src_field[f] * J.src_fstride + (long long)j * Mz * K;
    double2* dst = static_cast<double2*>(J.dst) + b * J.dst_mstride + J.dst_field[f] * J.dst_fstride +
                   (long long)j * K * nz;
    double2* R = reinterpret_cast<double2*>(smraw);
    for (int i = tid; i < Mz * C; i += nt) {
      const int z = (int)fdiv((unsigned)i, dC), c = i - z * C;
      if (c < nc) {
        // the kx = 0 line (the x means) less its first value: it may hardly vary
        double2 v = src[(long long)z * K + m0 + c];
        if (m0 + c == 0) v = csub(v, src[0]);
        R[c * Mz + z] = v;
      }
    }
    __syncthreads();
    for (int c = tid >> 5; c < nc; c += nw) fx_line(A + c * Mz, Mz, fs[c]);
    __syncthreads();
    fx_lines<-1, BIG>(A, nc, Mz, &J.pl, false);
    for (int c = tid >> 5; c < nc; c += nw)
      for (int q = lane; q < nz; q += 32) {
        double2 v = czero();
        if (q != hz) {
          v = fx_to2(A[c * Mz + (q < hz ? q : q - nz + Mz)], fs[c]);
          if (q == 0 && m0 + c == 0) v = cfma((double)Mz, src[0], v);
          if (J.inv != 1.0) v = cscl(v, J.inv);
        }
        dst[(long long)(m0 + c) * nz + q] = v;
      }
  }
}

// FP32 z lines (mixed groups' step).  Bound by instruction issue: three points
// a thread or six, so what a block sets up counts.  The index divisors come
// from the host and one loop fills the padded lines (before: a division per
// loop and thread, a fill and a barrier of its own); 128 x 97 x 64, ten steps:
// 12.99 -> 12.81 ms.
__global__ void __launch_bounds__(256) k_zcols(ZJob J) {
  using CT = float2;
  const int b = blockIdx.z;
  if (J.status && J.status[b]) return;
  const int f = (int)fdiv(blockIdx.y, J.drows);
  const int j = blockIdx.y - f * J.rows;
  const int C = J.C, K = J.K, nz = J.nz, Mz = J.Mz;
  const int m0 = blockIdx.x * C;
  const int nc = min(C, K - m0);
  extern __shared__ __align__(16) unsigned char smraw[];
  CT* A = reinterpret_cast<CT*>(smraw);
  CT* B = A + (size_t)C * Mz;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int hz = nz / 2;
  if (J.inverse) {
    const CT* src = static_cast<const CT*>(J.src) + b * J.src_mstride + J.src_field[f] * J.src_fstride +
                    (long long)j * K * nz;
    CT* dst = static_cast<CT*>(J.dst) + b * J.dst_mstride + J.dst_field[f] * J.dst_fstride +
              (long long)j * Mz * K;
    const float kfac = J.prm[b].kz1f;
    const int dz = J.dz[f];
    const bool skip0 = (J.mean == 1 && m0 == 0);
    for (int i = tid; i < C * Mz; i += nt) {
      // slot q of line c: mode q, or q - Mz from the end; the padded middle is zero
      const int c = (int)fdiv((unsigned)i, J.dMz), q = i - c * Mz;
      const int s = (q < hz) ? q : q - Mz;
      CT v = zero2<CT>();
      if (c < nc && s > -hz && s < hz && !(skip0 && i == 0)) {
        v = src[(m0 + c) * nz + (s < 0 ? s + nz : s)];
        if (dz) v = cscl(mul_i(v), kfac * (float)s);
      }
      A[i] = v;
    }
    __syncthreads();
    // padded synthesis (Mz >= 3 nz/2): the slots nz/2 .. Mz - nz/2 are zero
    CT* res = fft_lines<+1>(A, B, C, Mz, J.pl, J.pl.radix[0] == 3 && Mz >= 3 * hz);
    for (int i = tid; i < Mz * C; i += nt) {
      const int z = (int)fdiv((unsigned)i, J.dC), c = i - z * C;
      if (c < nc) dst[z * K + m0 + c] = res[c * Mz + z];
    }
  } else {
    const CT* src = static_cast<const CT*>(J.src) + b * J.src_mstride + J.src_field[f] * J.src_fstride +
                    (long long)j * Mz * K;
    CT* dst = static_cast<CT*>(J.dst) + b * J.dst_mstride + J.dst_field[f] * J.dst_fstride +
              (long long)j * K * nz;
    for (int i = tid; i < Mz * C; i += nt) {
      const int z = (int)fdiv((unsigned)i, J.dC), c = i - z * C;
      A[c * Mz + z] = (c < nc) ? src[z * K + m0 + c] : zero2<CT>();
    }
    __syncthreads();
    CT* res = fft_lines<-1>(A, B, C, Mz, J.pl);
    const float inv = J.invf;
    for (int i = tid; i < C * nz; i += nt) {
      const int c = (int)fdiv((unsigned)i, J.dnz), mz = i - c * nz;
      if (c < nc) {
        CT v = zero2<CT>();
        if (mz != hz) {
          const int s = (mz < hz) ? mz : mz - nz;
          v = cscl(res[c * Mz + (s >= 0 ? s : s + Mz)], inv);
        }
        if (J.mean == 2 && m0 + c == 0 && mz == 0) {
          J.zm[((size_t)b * 9 + J.dst_field[f]) * J.rows + j].x += (double)v.x;
          v = zero2<CT>();
        }
        dst[(m0 + c) * nz + mz] = v;
      }
    }
  }
}

// ------------------------------------------------ fused x pass + products
// Z3 fields (26): 0 u, 1 v, 2 w, 3 cxx, 4 cxy, 5 cxz, 6 cyy, 7 cyz, 8 czz,
// 9 uy, 10 wy, 11-16 c_y (xx, xy, xz, yy, yz, zz), 17 uz, 18 vz, 19 wz,
// 20-25 c_z.  Physical fields (35): the 26 plus x-derivatives of fields 0-8
// (26 ux, 27 vx, 28 wx, 29-34 c_x), packed in pairs into 18 complex lines.
// W3 outputs (9): N_cxx, N_cxy, N_cxz, N_cyy, N_cyz, N_czz, N_u, N_v, N_w.
// The products of Eqs. 1-2 at one point from the 35 physical fields q (Z3
// order, then the x-derivatives of fields 0-8 at 26-34; q[35] unused) to
// N_cxx, N_cxy, N_cxz, N_cyy, N_cyz, N_czz, N_u, N_v, N_w.
template <typename T>
__device__ __forceinline__ void products3d(const T (&q)[36], T eps, T iwi, T (&out)[9]) {
  const T u = q[0], v = q[1], w = q[2];
  const T C[3][3] = {{q[3], q[4], q[5]}, {q[4], q[6], q[7]}, {q[5], q[7], q[8]}};
  const T ux = q[26], vx = q[27], wx = q[28];
  const T uy = q[9], wy = q[10];
  const T uz = q[17], vz = q[18], wz = q[19];
  // L_ij = d u_i / d x_j, L_yy = -ux - wz (Eq. 3)
  const T L[3][3] = {{ux, uy, uz}, {vx, -ux - wz, vz}, {wx, wy, wz}};
  const T rw = ((T)1 + eps * (q[3] + q[6] + q[8] - (T)3)) * iwi;
  // components in storage order xx, xy, xz, yy, yz, zz; gradients in q
  const int ci[6] = {0, 0, 0, 1, 1, 2}, cj2[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const int i = ci[c], jj = cj2[c];
    const T adv = u * q[29 + c] + v * q[11 + c] + w * q[20 + c];
    T st = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) st += L[i][k] * C[k][jj] + C[i][k] * L[jj][k];
    const T dlt = (i == jj) ? (T)1 : (T)0;
    out[c] = -adv + st - (C[i][jj] - dlt) * rw;
  }
  // Eq. 2 advection: -(u . grad) u_i = -sum_k u_k L_ik
  const T uu[3] = {u, v, w};
#pragma unroll
  for (int i = 0; i < 3; ++i) out[6 + i] = -(uu[0] * L[i][0] + uu[1] * L[i][1] + uu[2] * L[i][2]);
}

// The same in FP64 with the fewest FP64 instructions (67 against about 100;
// each holds the pipe for 64 cycles): every output one chain of fused
// multiply-adds, the "+ rw" of -(c - 1) rw and the constants of the relaxation
// factor folded into its start, factors 2 as exponent increments on the
// integer pipe.  e1 = eps/Wi, e0 = (1 - 3 eps)/Wi.
__device__ __forceinline__ double twice3(double x) {   // 2 x by the exponent
  const int h = __double2hiint(x);
  const bool n = (h & 0x7FF00000) != 0 && (h & 0x7FF00000) < 0x7FE00000;
  return n ? __hiloint2double(h + 0x100000, __double2loint(x)) : x + x;
}
// get(i): field i, read where it is used (the velocity, its gradient and c stay
// in registers, the gradients of c do not).
template <typename Get>
__device__ __forceinline__ void products3d_fp64(Get get, double e1, double e0, double (&out)[9]) {
  const double u = get(0), v = get(1), w = get(2);
  const double c3 = get(3), c4 = get(4), c5 = get(5), c6 = get(6), c7 = get(7), c8 = get(8);
  const double C[3][3] = {{c3, c4, c5}, {c4, c6, c7}, {c5, c7, c8}};
  const double ux = get(26), wz = get(19);
  const double L[3][3] = {{ux, get(9), get(17)}, {get(27), -ux - wz, get(18)}, {get(28), get(10), wz}};
  const double rw = fma(e1, c3 + c6 + c8, e0);
  const int ci[6] = {0, 0, 0, 1, 1, 2}, cj[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const int i = ci[c], j = cj[c];
    const double gx = get(29 + c), gy = get(11 + c), gz = get(20 + c);
    double t = (i == j) ? fma(-u, gx, rw) : -u * gx;
    t = fma(-w, gz, fma(-v, gy, t));
#pragma unroll
    for (int k = 0; k < 3; ++k)
      t = (i == j) ? fma(twice3(L[i][k]), C[k][j], t) : fma(C[i][k], L[j][k], fma(L[i][k], C[k][j], t));
    out[c] = fma(-C[i][j], rw, t);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) out[6 + i] = fma(-w, L[i][2], fma(-v, L[i][1], -u * L[i][0]));
}

// FP64-accurate form: fixed-point transforms (ptt_fx.cuh) between FP64 arrays,
// products in FP64; 18 lines of Mx in one shared-memory buffer.  W3 is left
// without its 1/Mx (the y table's normalisation holds it).  Bound by
// instruction issue and latency, next the FP64 pipe of the products: four
// blocks of 256 threads per SM take 0.94 ms at 128 x 97 x 64, three 1.08, two
// 1.26 (FP64 lines on the FP64 pipe: 3.40).  Beyond 256 threads (ptt_autotune,
// where one block fills the shared memory) one block per SM.
template <int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_xfused3_fx(const __grid_constant__ GroupDev g) {
  const int b = blockIdx.y;
  if (g.status[b]) return;
  const int row = blockIdx.x;  // j * Mz + z
  const int K = g.K, Mx = g.Mx;
  const long long plane = (long long)g.M * g.Mz * K;  // one field of one member
  const MemberPrm pr = g.prm[b];
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ FxS fs[36], fo[10];
  __shared__ double2 ref[5];
  fxc* A = reinterpret_cast<fxc*>(smraw);
  const double2* Z = g.Z3 + (size_t)b * 26 * plane + (size_t)row * K;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, nw = nt >> 5;
  // lines 0-12: the 26 loaded fields in pairs (2l, 2l+1); line 13 + r
  // (r < 5): their x-derivatives i k (fields 2r, 2r+1; line 17 field 8
  // alone).  A warp per line: its two fields' modes, then their scales and
  // the packed line; the padded middle is zero.
  for (int l = tid >> 5; l < 18; l += nw) {
    fxc* h = A + l * Mx;
    const int r = (l < 13) ? l : l - 13;
    const double2* zF = Z + (size_t)(2 * r) * plane;
    unsigned mF = 0u, mG = 0u;
#pragma unroll 2
    for (int k = lane; k < K; k += 32) {
      double2 F = zF[k], G = (l < 17) ? zF[plane + k] : czero();
      if (k == 0) { F.y = 0; G.y = 0; }
      if (l >= 13) {
        const double fk = pr.kx1 * k;
        F = cscl(mul_i(F), fk);
        G = cscl(mul_i(G), fk);
      }
      h[k] = fx_bits(F.x, F.y);
      h[fx_xslot(1, k, K, Mx)] = fx_bits(G.x, G.y);
      mF = max(mF, fx_mag2(F));
      mG = max(mG, fx_mag2(G));
    }
    for (int k = K + 1 + lane; k <= Mx - K; k += 32) h[k] = fx_zero();
    __syncwarp();
    fx_xline(h, Mx, K, mF, mG, fs[2 * l], fs[2 * l + 1]);
  }
  __syncthreads();
  fx_lines<+1, false>(A, 18, Mx, &g.plMx, g.plMx.radix[0] % 3 == 0);
  const double e1 = pr.eps * pr.inv_wi, e0 = (1.0 - 3.0 * pr.eps) * pr.inv_wi;
  for (int x = tid; x < Mx; x += nt) {   // a column x is read and rewritten by one thread
    double out[9];
    products3d_fp64(
        [&](int i) {
          const fxc h = A[(i >> 1) * Mx + x];
          return fx_to((i & 1) ? h.y : h.x, fs[i]);
        },
        e1, e0, out);
#pragma unroll
    for (int l = 0; l < 5; ++l) A[l * Mx + x] = fx_bits(out[2 * l], (2 * l + 1 < 9) ? out[2 * l + 1] : 0.0);
  }
  __syncthreads();
  for (int l = tid >> 5; l < 5; l += nw) {
    const double2 r = fx_fields(A + l * Mx, Mx, fo[2 * l], fo[2 * l + 1]);
    if (lane == 0) ref[l] = r;
  }
  __syncthreads();
  fx_lines<-1, false>(A, 5, Mx, &g.plMx, false);
  double2* W = g.W3 + (size_t)b * 9 * plane + (size_t)row * K;
  const FastDiv dK = fast_div((unsigned)K);
  for (int i = tid; i < 5 * K; i += nt) {
    const int l = (int)fdiv((unsigned)i, dK), k = i - l * K;
    W[(size_t)(2 * l) * plane + k] = fx_mode_f(A + l * Mx, Mx, k, fo[2 * l], ref[l].x);
    if (2 * l + 1 < 9) W[(size_t)(2 * l + 1) * plane + k] = fx_mode_g(A + l * Mx, Mx, k, fo[2 * l + 1], ref[l].y);
  }
}

// Mixed form: FP32 transforms; mean/fluctuation split of the products (see
// xfused_block in the 2D kernels): the z pass left the mean mode out of the
// lines, the means of the 17 y-pass fields at this row's y come from g.Ym (the
// z- and x-derivatives have zero mean), the mean products go to g.Zm (written
// by the rows at z = 0; the forward z pass adds the fluctuations' mean).
__global__ void __launch_bounds__(512) k_xfused3(GroupDev g) {
  using C2 = float2;
  const int b = blockIdx.y;
  if (g.status[b]) return;
  const int row = blockIdx.x;  // j * Mz + z
  const int K = g.K, Mx = g.Mx;
  const long long plane = (long long)g.M * g.Mz * K;  // one field of one member
  const MemberPrm pr = g.prm[b];
  extern __shared__ __align__(16) unsigned char smraw[];
  C2* A = reinterpret_cast<C2*>(smraw);
  C2* B = A + 18 * Mx;
  const C2* Z = g.Z3f + (size_t)b * 26 * plane + (size_t)row * K;
  const float kfac = pr.kx1f;
  const int tid = threadIdx.x, nt = blockDim.x;
  __shared__ float s_mq[17];
  {
    const int jy = row / g.Mz;
    const double2* ym = g.Ym + (size_t)b * 17 * g.M + jy;
    if (tid < 17) s_mq[tid] = (float)ym[(size_t)tid * g.M].x;
    if (tid == 32 && row - jy * g.Mz == 0) {
      double q[36], o[9];
      for (int i = 0; i < 36; ++i) q[i] = (i < 17) ? ym[(size_t)i * g.M].x : 0.0;
      products3d<double>(q, pr.eps, pr.inv_wi, o);
      double2* zm = g.Zm + (size_t)b * 9 * g.M + jy;
      for (int i = 0; i < 9; ++i) zm[(size_t)i * g.M] = make_double2(o[i], 0.0);
    }
  }
  // the padded middle K <= k <= Mx - K of every line is zero
  {
    const int nmid = Mx - 2 * K + 1;
    for (int i = tid; i < 18 * nmid; i += nt) {
      const int l = (int)fdiv((unsigned)i, fast_div((unsigned)nmid)), k = K + (i - l * nmid);
      A[l * Mx + k] = zero2<C2>();
    }
  }
  // the lines and items of the fixed-point form
  {
    constexpr int kB = 4;   // items in flight per thread
    const int nitem = 13 * K;
    const FastDiv dK = fast_div((unsigned)K);
    for (int i0 = tid; i0 < nitem; i0 += kB * nt) {
      C2 F[kB], G[kB];
#pragma unroll
      for (int u = 0; u < kB; ++u) {
        const int it = i0 + u * nt;
        F[u] = G[u] = zero2<C2>();
        if (it < nitem) {
          const int l = (int)fdiv((unsigned)it, dK), kk = it - l * K;
          F[u] = Z[(size_t)(2 * l) * plane + kk];
          G[u] = Z[(size_t)(2 * l + 1) * plane + kk];
        }
      }
#pragma unroll
      for (int u = 0; u < kB; ++u) {
        const int it = i0 + u * nt;
        if (it >= nitem) continue;
        const int l = (int)fdiv((unsigned)it, dK), kk = it - l * K;
        C2 f = F[u], gg = G[u];
        if (kk == 0) { f.y = 0; gg.y = 0; }
        A[l * Mx + kk] = cadd(f, mul_i(gg));
        if (kk > 0) A[l * Mx + Mx - kk] = cadd(cconj(f), mul_i(cconj(gg)));
        if (l < 5) {
          const float fk = kfac * (float)kk;
          C2 df = cscl(mul_i(F[u]), fk), dg = cscl(mul_i(G[u]), fk);
          if (l == 4) dg = zero2<C2>();
          if (kk == 0) { df.y = 0; dg.y = 0; }
          const int ld = 13 + l;
          A[ld * Mx + kk] = cadd(df, mul_i(dg));
          if (kk > 0) A[ld * Mx + Mx - kk] = cadd(cconj(df), mul_i(cconj(dg)));
        }
      }
    }
  }
  __syncthreads();
  C2* res = fft_lines<+1>(A, B, 18, Mx, g.plMx, g.plMx.radix[0] == 3);
  C2* oth = (res == A) ? B : A;
  for (int x = tid; x < Mx; x += nt) {
    mfl q[36], om[9];
#pragma unroll
    for (int l = 0; l < 18; ++l) {
      const C2 h = res[l * Mx + x];
      q[2 * l] = mfl(2 * l < 17 ? s_mq[2 * l] : 0.f, h.x);
      q[2 * l + 1] = mfl(2 * l + 1 < 17 ? s_mq[2 * l + 1] : 0.f, h.y);
    }
    products3d<mfl>(q, mfl(pr.epsf, 0.f), mfl(pr.inv_wif, 0.f), om);
#pragma unroll
    for (int l = 0; l < 5; ++l) oth[l * Mx + x] = make_float2(om[2 * l].f, (2 * l + 1 < 9) ? om[2 * l + 1].f : 0.f);
  }
  __syncthreads();
  C2* r2 = fft_lines<-1>(oth, res, 5, Mx, g.plMx);
  C2* W = g.W3f + (size_t)b * 9 * plane + (size_t)row * K;
  const float inv = g.invMxf;
  for (int i = tid; i < 5 * K; i += nt) {
    const int l = (int)fdiv((unsigned)i, fast_div((unsigned)K)), k = i - l * K;
    const C2 hk = r2[l * Mx + k];
    const C2 hm = cconj(r2[l * Mx + (k == 0 ? 0 : Mx - k)]);
    const C2 F = cscl(cadd(hk, hm), 0.5f * inv);
    const C2 d = csub(hk, hm);
    W[(size_t)(2 * l) * plane + k] = F;
    if (2 * l + 1 < 9) W[(size_t)(2 * l + 1) * plane + k] = make_float2(0.5f * inv * d.y, -0.5f * inv * d.x);
  }
}

// ---------------------------------------------- per-mode spectral stage
// Explicit terms (Eq. 2): H_i = N_u,i + gam (div c)_i (+ 2/Re on the mean
// mode, x); forcings of the evolved velocity quantities (k != 0):
// q1 = -D(i kx H_x + i kz H_z) - k^2 H_y (phi = (D^2 - k^2) v),
// q2 = i kz H_x - i kx H_z (eta = i kz u - i kx w); mean mode: H_x, H_z.
// Evolved (8): c (6), q1 state, q2 state.  Solves per mode: six c (wall rows
// of Eq. 1 at kappa = 0), phi -> v -> influence correction (k != 0) or U,
// eta (k != 0) or W; then u = i (kx Dv - kz eta)/k^2, w = i (kz Dv + kx eta)/k^2.
//
// A block takes 16 modes; lane l of every warp owns mode l/2 of the block and
// Chebyshev parity l%2, and each of the eight warps runs one chain:
//   V    q1 = (D^2 - k^2) v; then, in one descending pass, its forcing from H,
//        the history and the SBDF sum and the phi elimination; the v system;
//        the influence correction with D v
//   Q2   q2, its forcing, SBDF sum and system (eta, W)
//   C0-5 a conformation component's SBDF sum and system; three of them first
//        form a component of H
// About 300 FP64 instructions per coefficient pair and 64 cycles each make
// the FP64 pipe the bound (0.2 ms at 128 x 97 x 64 were every SM equally
// loaded); 256 blocks on 152 SMs put 2/1.7 of that on the busiest, and the
// chains are paired per sub-partition (a warp's index mod 4) as evenly as
// they go: V + C5, Q2 + C0, C1 + C2, C3 + C4.  Blocks turn the pairs by one
// partition each, so that two of an SM do not load the same one.
// Measured at 128 x 97 x 64: 0.61 -> 0.40 ms (one pass per recurrence, a
// barrier between any two, 390 FP64 instructions); rows loaded one ahead while
// the elimination's arithmetic runs (both rows at once spill at the 128
// registers that two blocks per SM leave).
// Per-mode scratch columns live in SS (workspace; L2-resident while the block
// runs):
enum {
  S3_HX = 0, S3_HY, S3_HZ,   // explicit momentum terms H
  S3_P,                      // 6: the c components' eliminations
  S3_PHI = S3_P + 6,         // phi
  S3_ETA, S3_DVN,            // eta, D of the new v
  kScr3
};
constexpr int kModesPerBlock = 16;

// Named barriers: `n` threads of the block in all, those that only signal
// (after their writes) and those that wait.
__device__ __forceinline__ void bar_signal(int id, int n) {
  __threadfence_block();
  __syncwarp();
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_wait(int id, int n) {
  __threadfence_block();
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// The lane's mode and its tables.
struct Mode3 {
  int N, p, md, o;
  bool mean;
  double kx, kz, k2;
  size_t NK, col;
};

__device__ __forceinline__ LaneHist hist3(const GroupDev& g, const Mode3& m, int b, int slot, int q, double idt) {
  LaneHist h;
  h.o = m.o;
  for (int j = 0; j < 4; ++j) h.ca[j] = -c_sa[m.o][j + 1] * idt;
  auto at = [&](double2* base, int j) {
    return base + ((((size_t)((slot - j) & 3)) * g.nb + b) * 8 + q) * m.NK + m.col;
  };
  h.E0 = at(g.Eh, 1); h.E1 = at(g.Eh, 2); h.E2 = at(g.Eh, 3);
  h.dn = g.Nh - g.Eh;
  return h;
}

// Elimination of a conformation component x with explicit term nn.
template <bool FULL>
__device__ __forceinline__ double2 chain3_c(const Mode3& m, const LaneHist& h, const double2* __restrict__ x,
                                            const double2* __restrict__ nn, double2* __restrict__ E,
                                            double2* __restrict__ Nn, double alpha, double2* __restrict__ P,
                                            const double* inv, const double* F, const double* w, bool solve,
                                            double2& rs) {
  struct Row { LaneRow h; double2 x, nn; };
  auto ld = [&](int n) {
    Row r;
    r.h = lane_hist_row<FULL>(h, n);
    r.x = x[n];
    r.nn = nn[n];
    return r;
  };
  auto ev = [&](const Row& r, int n) {
    E[n] = r.x;
    Nn[n] = r.nn;
    return lane_sbdf<FULL>(h, r.h, r.x, r.nn);
  };
  if (solve) return lane_qt_back<true>(m.N, m.p, alpha, ld, ev, P, inv, F, w, rs);
  // no diffusion: P = R / alpha
  const double ia = 1.0 / alpha;
#pragma unroll 2
  for (int n = m.p; n < m.N; n += 2) P[n] = cscl(ev(ld(n), n), ia);
  return czero();
}

// Elimination of q1 (phi, or U of the mean mode): forcing
// -D(i kx H_x + i kz H_z) - k^2 H_y (mean mode: H_x) on the way down.
template <bool FULL>
__device__ __forceinline__ double2 chain3_v(const Mode3& m, const LaneHist& h, const double2* __restrict__ Hx,
                                            const double2* __restrict__ Hy, const double2* __restrict__ Hz,
                                            const double2* __restrict__ E, double2* __restrict__ Nn, double alpha,
                                            double2* __restrict__ P, const double* inv, const double* F,
                                            const double* w) {
  struct Row { LaneRow h; double2 x, hx, hz, hy; };
  auto ld = [&](int n) {
    Row r;
    r.h = lane_hist_row<FULL>(h, n);
    r.x = E[n];
    const int k = m.mean ? n : min(n + 1, m.N - 1);
    r.hx = Hx[k];
    r.hz = Hz[k];
    r.hy = Hy[n];
    return r;
  };
  double2 acc = czero();
  auto ev = [&](const Row& r, int n) {
    const double2 s = cfma(m.kz, r.hz, cscl(r.hx, m.kx));
    acc = cfma(n + 1 < m.N ? lane_i2d(2 * (n + 1)) : 0.0, s, acc);
    const double2 d = lane_half2(acc, n == 0);
    double2 f = make_double2(fma(-m.k2, r.hy.x, d.y), fma(-m.k2, r.hy.y, -d.x));
    if (m.mean) f = r.hx;
    Nn[n] = f;
    return lane_sbdf<FULL>(h, r.h, r.x, f);
  };
  double2 rs;
  return lane_qt_back<false>(m.N, m.p, alpha, ld, ev, P, inv, F, w, rs);
}

// Elimination of q2 = i kz u - i kx w with forcing i kz H_x - i kx H_z (mean
// mode: w and H_z).
template <bool FULL>
__device__ __forceinline__ double2 chain3_q(const Mode3& m, const LaneHist& h, const double2* __restrict__ u,
                                            const double2* __restrict__ w_, const double2* __restrict__ Hx,
                                            const double2* __restrict__ Hz, double2* __restrict__ E,
                                            double2* __restrict__ Nn, double alpha, double2* __restrict__ P,
                                            const double* inv, const double* F, const double* w) {
  struct Row { LaneRow h; double2 u, w, hx, hz; };
  auto ld = [&](int n) {
    Row r;
    r.h = lane_hist_row<FULL>(h, n);
    r.u = u[n];
    r.w = w_[n];
    r.hx = Hx[n];
    r.hz = Hz[n];
    return r;
  };
  auto ev = [&](const Row& r, int n) {
    double2 x = mul_i(cfma(-m.kx, r.w, cscl(r.u, m.kz)));
    double2 f = mul_i(cfma(-m.kx, r.hz, cscl(r.hx, m.kz)));
    if (m.mean) { x = r.w; f = r.hz; }
    E[n] = x;
    Nn[n] = f;
    return lane_sbdf<FULL>(h, r.h, x, f);
  };
  double2 rs;
  return lane_qt_back<false>(m.N, m.p, alpha, ld, ev, P, inv, F, w, rs);
}

__global__ void __launch_bounds__(256, 2) k_spec3(const __grid_constant__ GroupDev g, int mode) {
  const int b = blockIdx.y;
  if (g.status[b]) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int p = lane & 1;
  const int KZ = g.KZ, N = g.N, nb = g.nb, nz = g.nz;
  const size_t NK = (size_t)N * KZ;
  const int md0 = blockIdx.x * kModesPerBlock + (lane >> 1);
  const bool inb = md0 < KZ;
  const int md = inb ? md0 : KZ - 1;
  const int mx = md / nz, mzi = md - mx * nz, hz = nz / 2;
  const bool nyq = (mzi == hz);
  const bool act = inb && !nyq;
  const MemberPrm pr = g.prm[b];
  const long long cnt = g.count[b];
  const int slot = (int)(cnt & 3);
  const int o = (cnt < 3) ? (int)cnt : 3;
  const int sz = (mzi < hz) ? mzi : mzi - nz;
  Mode3 m;
  m.N = N; m.p = p; m.md = md; m.o = o;
  m.mean = (mx == 0 && mzi == 0);
  m.kx = pr.kx1 * mx;
  m.kz = pr.kz1 * sz;
  m.k2 = m.kx * m.kx + m.kz * m.kz;
  m.NK = NK; m.col = (size_t)md * N;
  const bool mean = m.mean;
  const size_t col = m.col;
  double2* X = g.X + (size_t)b * 9 * NK + col;          // field f at X + f * NK
  const double2* NR = g.NR + (size_t)b * 9 * NK + col;
  double2* S = g.SS + (size_t)b * kScr3 * NK + col;     // scratch column a at S + a * NK
  auto SC = [&](int a) { return S + (size_t)a * NK; };

  // the dropped Nyquist slot stays zero
  if (warp == 0 && inb && nyq) {
    if (mode == 0) {
      for (int f = 0; f < 9; ++f)
        for (int n = p; n < N; n += 2) X[f * NK + n] = czero();
      double2* E = g.Eh + ((size_t)slot * nb + b) * 8 * NK + col;
      double2* Nn = g.Nh + ((size_t)slot * nb + b) * 8 * NK + col;
      for (int s2 = 0; s2 < 8; ++s2)
        for (int n = p; n < N; n += 2) { E[s2 * NK + n] = czero(); Nn[s2 * NK + n] = czero(); }
    } else {
      double2* R = g.Rb + (size_t)b * 4 * NK + col;
      for (int f = 0; f < 3; ++f)
        for (int n = p; n < N; n += 2) R[f * NK + n] = czero();
    }
  }
  __shared__ double s_ik2[32];   // 1/k^2 of the lanes, by V
  // the warp's chain: 0-5 a c component, 6 V, 7 Q2
  const int part = (warp - (int)blockIdx.x - (int)blockIdx.x / 152) & 3;   // 152 SMs: block i + 152 joins block i
  const int role = (warp < 4) ? (part == 0 ? 6 : part == 1 ? 7 : part == 2 ? 1 : 3)
                              : (part == 0 ? 5 : part == 1 ? 0 : part == 2 ? 2 : 4);
  // explicit momentum term t on component warp t + 1:
  // (div c)_i = i kx c_xi + D c_yi + i kz c_zi
  if (role >= 1 && role <= 3) {
    const int t = role - 1;
    const int cx = 3 + t;                               // c_xx, c_xy, c_xz
    const int cy = (t == 0) ? 4 : 5 + t;                // c_xy, c_yy, c_yz
    const int cz = (t == 0) ? 5 : 6 + t;                // c_xz, c_yz, c_zz
    double2* H = (mode == 1) ? g.Rb + ((size_t)b * 4 + t) * NK + col : SC(S3_HX + t);
    if (act) {
      lane_div_h(N, p, X + cy * NK, X + cx * NK, X + cz * NK, NR + (size_t)(6 + t) * NK, pr.gam, pr.gam * m.kx,
                 pr.gam * m.kz, H);
      if (mean && t == 0 && p == 0) H[0].x += pr.forcing;
    }
  }
  if (mode == 1) return;   // explicit right-hand side only: H in Rb
  const double* w = g.wrow;
  const double a0dt = g.prm[b].a0dt[o], idt = pr.idt;
  const double* qt = g.qt + ((size_t)b * 4 + o) * 3 * 3 * NK + col;
  auto T = [&](int sys, int k) { return qt + (size_t)(sys * 3 + k) * NK; };
  auto G = [&](int sys) { return g.qtG[((((size_t)b * 4 + o) * 3 + sys) * 2 + p) * KZ + md]; };
  auto cur = [&](double2* base, int q) { return base + (((size_t)slot * nb + b) * 8 + q) * NK + col; };
  if (role < 6) {
    if (role >= 1 && role <= 3) bar_signal(1, 160);   // H is there (the other end: V and Q2)
    const double alpha = fma(pr.kappa, m.k2, a0dt);
    const bool solve = pr.kappa != 0.0;
    double2 U = czero(), rs = czero();
    double2* P = SC(S3_P + role);
    double2* x = X + (size_t)(3 + role) * NK;
    if (act) {
      const LaneHist h = hist3(g, m, b, slot, role, idt);
      const double2* nn = NR + (size_t)role * NK;
      U = (o == 3) ? chain3_c<true>(m, h, x, nn, cur(g.Eh, role), cur(g.Nh, role), alpha, P, T(0, 1), T(0, 2), w,
                                    solve, rs)
                   : chain3_c<false>(m, h, x, nn, cur(g.Eh, role), cur(g.Nh, role), alpha, P, T(0, 1), T(0, 2), w,
                                     solve, rs);
    }
    bar_wait(2, 192);   // H has read the old c (the six component warps)
    if (act) {
      if (solve) {
        const double2 wall = cscl(rs, g.prm[b].dta0[o]);
        lane_qt_fwd(N, p, cscl(csub(wall, U), G(0)), wall, P, x, T(0, 0), [](int, double2) {});
      } else {
#pragma unroll 4
        for (int n = p; n < N; n += 2) x[n] = P[n];
      }
    }
  } else if (role == 6) {
    double2* E = cur(g.Eh, 6);
    double2* v = X + NK;
    if (act) {
      if (mean) {
#pragma unroll 4
        for (int n = p; n < N; n += 2) E[n] = X[n];
      } else {
        lane_lap(N, p, v, m.k2, E);
      }
    }
    s_ik2[lane] = mean ? 0.0 : 1.0 / m.k2;
    bar_wait(1, 160);
    if (act) {
      const LaneHist h = hist3(g, m, b, slot, 6, idt);
      double2* phi = SC(S3_PHI);
      const double alpha = mean ? a0dt : fma(pr.nu, m.k2, a0dt);
      const double2 U = (o == 3) ? chain3_v<true>(m, h, SC(S3_HX), SC(S3_HY), SC(S3_HZ), E, cur(g.Nh, 6), alpha, phi,
                                                  T(1, 1), T(1, 2), w)
                                 : chain3_v<false>(m, h, SC(S3_HX), SC(S3_HY), SC(S3_HZ), E, cur(g.Nh, 6), alpha, phi,
                                                   T(1, 1), T(1, 2), w);
      lane_qt_fwd(N, p, cscl(U, -G(1)), czero(), phi, mean ? X : phi, T(1, 0), [](int, double2) {});
      if (mean) {
        for (int n = p; n < N; n += 2) v[n] = czero();
      } else {
        // (D^2 - k^2) v = phi: the solve's right-hand side is -phi
        double2 rs, sacc = czero();
        const double2 U2 = lane_qt_back<false>(
            N, p, m.k2, [&](int n) { return phi[n]; },
            [&](double2 r, int) { return cneg_bits(r); }, v, T(2, 1), T(2, 2), w, rs);
        lane_qt_fwd(N, p, cscl(U2, -G(2)), czero(), v, v, T(2, 0),
                    [&](int n, double2 a) { sacc = cfma(lane_i2d(n * n), a, sacc); });
        // influence correction and D v, top down
        const double* __restrict__ vh = g.vh + ((size_t)b * 4 + o) * NK + col;
        double2* __restrict__ dv = SC(S3_DVN);
        double2* __restrict__ vr = v;
        const double2 coef = cscl(sacc, -g.vhS[(((size_t)b * 4 + o) * 2 + p) * KZ + md]);
        const int nl = ((N - 1 - p) & ~1) + p;
        double2 acc = czero();
        if (nl != N - 1) dv[N - 1] = czero();
#pragma unroll 4
        for (int n = nl; n >= p; n -= 2) {
          const double f = vh[n];
          const double2 a = vr[n];
          const double2 vn = make_double2(fma(coef.x, f, a.x), fma(coef.y, f, a.y));
          vr[n] = vn;
          acc = cfma(lane_i2d(2 * n), vn, acc);
          if (n > 0) dv[n - 1] = lane_half2(acc, n == 1);
        }
      }
    }
  } else {
    bar_wait(1, 160);
    if (act) {
      const LaneHist h = hist3(g, m, b, slot, 7, idt);
      double2* eta = SC(S3_ETA);
      const double alpha = mean ? a0dt : fma(pr.nu, m.k2, a0dt);
      const double2 U = (o == 3) ? chain3_q<true>(m, h, X, X + 2 * NK, SC(S3_HX), SC(S3_HZ), cur(g.Eh, 7),
                                                  cur(g.Nh, 7), alpha, eta, T(1, 1), T(1, 2), w)
                                 : chain3_q<false>(m, h, X, X + 2 * NK, SC(S3_HX), SC(S3_HZ), cur(g.Eh, 7),
                                                   cur(g.Nh, 7), alpha, eta, T(1, 1), T(1, 2), w);
      lane_qt_fwd(N, p, cscl(U, -G(1)), czero(), eta, mean ? X + 2 * NK : eta, T(1, 0), [](int, double2) {});
    }
  }
  __syncthreads();
  // u, w from D v and eta (k != 0), warp w on elements [w c8, (w + 1) c8) of
  // its lane's parity
  if (act && !mean) {
    const int Lp = (N - p + 1) / 2, c8 = (Lp + 7) / 8;
    const int e0 = min(Lp, warp * c8), e1 = min(Lp, e0 + c8);
    const double2* __restrict__ dv = SC(S3_DVN);
    const double2* __restrict__ et = SC(S3_ETA);
    double2* __restrict__ u = X;
    double2* __restrict__ wv = X + 2 * NK;
    const double ax = m.kx * s_ik2[lane], az = m.kz * s_ik2[lane];
#pragma unroll 4
    for (int i = e0; i < e1; ++i) {
      const int n = p + 2 * i;
      const double2 d = dv[n], e = et[n];
      u[n] = mul_i(cfma(-az, e, cscl(d, ax)));
      wv[n] = mul_i(cfma(ax, e, cscl(d, az)));
    }
  }
}

__global__ void k_tick3(GroupDev g) {
  const int b = threadIdx.x + blockIdx.x * blockDim.x;
  if (b < g.nb && !g.status[b]) g.count[b] += 1;
}

// ------------------------------------------------------------ diagnostics
// Tile slots: P_E a double; P_MIN, P_MAX keys (dkey) of Tr c; P_AMAX the
// bits of max |Tr c|; P_BAD and the counts 64-bit integers; P_MS the
// mid-plane power sums (doubles, in the first mid_tiles tiles only).
enum { P_E = 0, P_MIN, P_MAX, P_AMAX, P_BAD, P_C3, P_C0, P_B3, P_B0,
       P_MC3, P_MC0, P_MB3, P_MB0, P_MS = 16 /* 8 quantities x 4 powers */ };
constexpr int kMidLanes3 = 8, kMidModesPerBlock3 = 256 / kMidLanes3;   // k_diag_mid3
constexpr int kMidTilePts = 2048;   // mid-plane points per tile of k_diag_count3

__device__ __forceinline__ long long* islots3(double* pp) { return reinterpret_cast<long long*>(pp); }
__device__ __forceinline__ const long long* islots3(const double* pp) {
  return reinterpret_cast<const long long*>(pp);
}
__device__ __forceinline__ bool nonfinite3(double x) {
  return (__double_as_longlong(x) & 0x7ff0000000000000LL) == 0x7ff0000000000000LL;
}
// mid-plane points per tile (at least kMidTilePts, and all npl points within
// the ntile tiles) and the number of tiles that carry them
__device__ __forceinline__ int mid_per(int npl, int ntile) {
  return max(kMidTilePts, (npl + ntile - 1) / ntile);
}
__device__ __forceinline__ int mid_tiles(int npl, int ntile) {
  const int per = mid_per(npl, ntile);
  return (npl + per - 1) / per;
}

// Energy (Fejer in y, Parseval in x and z), extrema of Tr c on the unpadded
// grid, non-finite test; ntile blocks per member.
__global__ void __launch_bounds__(256) k_diag_part3(GroupDev g) {
  const int b = blockIdx.y, tile = blockIdx.x;
  if (g.status[b]) return;
  const int KZ = g.KZ, N = g.N, nx = g.nx, nz = g.nz, Je = g.Me;
  const size_t NK = (size_t)N * KZ;
  const double2* DY = g.DY + (size_t)b * 3 * Je * KZ;
  double e = 0.0;
  KeyExt ext = keyext_empty();
  int bad = 0;
  {
    // modes mx > 0 count twice (Parseval over +-kx)
    const unsigned tot = (unsigned)Je * KZ, per = (tot + g.ntile - 1) / g.ntile;
    const unsigned i0 = tile * per, i1 = min(tot, i0 + per);
    const FastDiv dKZ = fast_div((unsigned)KZ);
    double e0 = 0.0, e1 = 0.0;
#pragma unroll 2
    for (unsigned i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
      // i KZ passes 2^32 (192 x 129 x 96: 2.3e10), where fdiv's last modes of some
      // rows would land in the next row
      const unsigned j = fdiv_any(i, dKZ, (unsigned)KZ), md = i - j * KZ;
      const double2 a0 = DY[i], a1 = DY[(size_t)Je * KZ + i], a2 = DY[(size_t)2 * Je * KZ + i];
      const double q = fma(a0.x, a0.x, fma(a0.y, a0.y, fma(a1.x, a1.x, fma(a1.y, a1.y,
                           fma(a2.x, a2.x, a2.y * a2.y)))));
      if (md < (unsigned)nz) e0 = fma(g.ccw[j], q, e0);   // mx = 0
      else e1 = fma(g.ccw[j], q, e1);
    }
    e = fma(2.0, e1, e0);
  }
  {
    const double* tr = g.DV + (size_t)b * N * nz * nx;
    const long long tot = (long long)N * nz * nx, per = (tot + g.ntile - 1) / g.ntile;
    const long long i0 = tile * per, i1 = min(tot, i0 + per);
    for (long long i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
      const double t = tr[i];
      bad |= nonfinite3(t);
      keyext_add(ext, t);
    }
  }
  {
    const double* Xd = reinterpret_cast<const double*>(g.X + (size_t)b * 9 * NK);
    const long long tot = 18LL * NK, per = (tot + g.ntile - 1) / g.ntile;
    const long long i0 = tile * per, i1 = min(tot, i0 + per);
#pragma unroll 4
    for (long long i = i0 + threadIdx.x; i < i1; i += blockDim.x) bad |= nonfinite3(Xd[i]);
  }
  __shared__ TileRed<1, false> red;
  red.warp(e, 0.0, ext, {bad});
  __syncthreads();
  if (threadIdx.x == 0) {
    double* pp = g.part + ((size_t)b * g.ntile + tile) * kPart;
    ext = red.ext();
    pp[P_E] = red.energy();
    islots3(pp)[P_MIN] = ext.mn;
    islots3(pp)[P_MAX] = ext.mx;
    islots3(pp)[P_AMAX] = ext.ma;
    islots3(pp)[P_BAD] = red.count(0) ? 1 : 0;
  }
}

// Counts of Tr c < 3, < 0 and the tie bands over the volume (every tile)
// and, in the first mid_tiles tiles, over the (x, z) mid-plane values
// MV[b][8][nz][nx] the same counts and the power sums of the 8 mid-plane
// quantities (histograms too); ntile blocks per member.
__global__ void __launch_bounds__(256) k_diag_count3(GroupDev g) {
  const int b = blockIdx.y, tile = blockIdx.x;
  if (g.status[b]) return;
  const TrBands B = tr_bands(1e-9 * block_tiles_amax(g.part + (size_t)b * g.ntile * kPart, g.ntile, P_AMAX));
  TrCounts c{0, 0, 0, 0}, mc{0, 0, 0, 0};
  {
    const double* tr = g.DV + (size_t)b * g.N * g.nz * g.nx;
    const long long tot = (long long)g.N * g.nz * g.nx, per = (tot + g.ntile - 1) / g.ntile;
    const long long i0 = tile * per, i1 = min(tot, i0 + per);
    for (long long i = i0 + threadIdx.x; i < i1; i += blockDim.x) tr_count(c, tr[i], B);
  }
  __shared__ int sc[kRedWarps][4];
  counts_warp(c, sc);
  __syncthreads();
  double* pp = g.part + ((size_t)b * g.ntile + tile) * kPart;
  if (threadIdx.x < 4) islots3(pp)[P_C3 + threadIdx.x] = counts_total(sc, threadIdx.x);   // P_C3, P_C0, P_B3, P_B0
  const int npl = g.nz * g.nx;
  if (tile >= mid_tiles(npl, g.ntile)) return;   // block-uniform
  double sums[32];
#pragma unroll
  for (int k = 0; k < 32; ++k) sums[k] = 0.0;
  {
    const double* MV = g.MV + (size_t)b * 8 * npl;
    const int per = mid_per(npl, g.ntile);
    const int i0 = tile * per, i1 = min(npl, i0 + per);
    const double* hr = g.hrange + (size_t)b * 16;
    unsigned long long* gh = g.hist + (size_t)b * 8 * (PTT_HIST_BINS + 2);
    for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {   // mid-plane histograms
        const int sl = hist_slot(MV[(size_t)q * npl + i], hr[2 * q], hr[2 * q + 1]);
        if (sl >= 0) atomicAdd(&gh[q * (PTT_HIST_BINS + 2) + sl], 1ULL);
      }
      tr_count(mc, MV[i], B);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const double a = MV[(size_t)q * npl + i], a2 = a * a;
        sums[4 * q] += a; sums[4 * q + 1] += a2; sums[4 * q + 2] += a2 * a; sums[4 * q + 3] += a2 * a2;
      }
    }
  }
  __shared__ double red[8 * 32];
  __shared__ int smc[kRedWarps][4];
  counts_warp(mc, smc);
  block_sum_scatter(sums, red, kRedWarps);   // its barriers also complete the counts
  if (threadIdx.x < 32) pp[P_MS + threadIdx.x] = red[threadIdx.x];
  if (threadIdx.x < 4) islots3(pp)[P_MC3 + threadIdx.x] = counts_total(smc, threadIdx.x);   // P_MC3 ... P_MB0
}

// Mid-plane spectra at y = 0 per mode (kMidLanes3 lanes each): DM[b][q][mode]
// for q = Tr c, u', w', du/dx, du/dz, dw/dx, dw/dz, v (u', w' without the
// mean).
__device__ __forceinline__ double2 seg_sum2_3(double2 v) {
#pragma unroll
  for (int o = kMidLanes3 / 2; o > 0; o >>= 1) {
    v.x += __shfl_down_sync(0xffffffffu, v.x, o, kMidLanes3);
    v.y += __shfl_down_sync(0xffffffffu, v.y, o, kMidLanes3);
  }
  return v;
}
__global__ void __launch_bounds__(256) k_diag_mid3(GroupDev g) {
  const int b = blockIdx.y;
  if (g.status[b]) return;
  const int sub = threadIdx.x & (kMidLanes3 - 1);
  const int md = blockIdx.x * (blockDim.x / kMidLanes3) + (threadIdx.x / kMidLanes3);
  const int KZ = g.KZ, N = g.N, nz = g.nz;
  const bool on = md < KZ;   // every lane takes part in the shuffles
  const size_t NK = (size_t)N * KZ;
  const double2* X = g.X + (size_t)b * 9 * NK + (size_t)(on ? md : 0) * N;
  double2 tr = czero(), u = czero(), v = czero(), w = czero();
  if (on) {   // even n, one residue of n mod 4 per lane
    const double s = (sub & 1) ? -1.0 : 1.0;
    for (int n = 2 * sub; n < N; n += 2 * kMidLanes3) {
      tr = cfma(s, cadd(X[3 * NK + n], cadd(X[6 * NK + n], X[8 * NK + n])), tr);
      u = cfma(s, X[n], u);
      v = cfma(s, X[NK + n], v);
      w = cfma(s, X[2 * NK + n], w);
    }
  }
  tr = seg_sum2_3(tr);
  u = seg_sum2_3(u);
  v = seg_sum2_3(v);
  w = seg_sum2_3(w);
  if (on && sub == 0) {
    const MemberPrm pr = g.prm[b];
    const int mx = md / nz, mzi = md - mx * nz, hz = nz / 2;
    const int sz = (mzi < hz) ? mzi : mzi - nz;
    const double kx = pr.kx1 * mx;
    const double kz = (mzi == hz) ? 0.0 : pr.kz1 * sz;
    double2 q[8] = {tr, u, w, cscl(mul_i(u), kx), cscl(mul_i(u), kz), cscl(mul_i(w), kx),
                    cscl(mul_i(w), kz), v};
    if (md == 0) { q[1] = czero(); q[2] = czero(); }
    double2* D = g.DM + (size_t)b * 8 * KZ + md;
    for (int k = 0; k < 8; ++k) D[(size_t)k * KZ] = q[k];
  }
}

// Per member: reduce the tiles (each thread a fixed set of tiles, then
// fixed-order trees: deterministic; the energy and the mid-plane sums in
// FP64, extrema and counts on integers), <Tr c>, blow-up test, record.
__global__ void __launch_bounds__(256) k_diag_final3(GroupDev g) {
  const int b = blockIdx.x;
  if (g.status[b]) return;
  const int KZ = g.KZ, N = g.N;
  const size_t NK = (size_t)N * KZ;
  const MemberPrm pr = g.prm[b];
  const double* pp = g.part + (size_t)b * g.ntile * kPart;
  const double2* X = g.X + (size_t)b * 9 * NK;
  __shared__ TileRed<9, true> tr;
  const int nmt = mid_tiles(g.nz * g.nx, g.ntile);
  {
    double te = 0.0, mt = 0.0;
    KeyExt x = keyext_empty();
    int tc[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};   // volume and mid-plane counts, non-finite tiles
    for (int n = 2 * threadIdx.x; n < N; n += 2 * blockDim.x)
      mt += (X[3 * NK + n].x + X[6 * NK + n].x + X[8 * NK + n].x) * cheb_mean_weight(g.wrow, N, n);
    for (int t = threadIdx.x; t < g.ntile; t += blockDim.x) {
      const double* q = pp + (size_t)t * kPart;
      const long long* qi = islots3(q);
      te += q[P_E];
      keyext_merge(x, KeyExt{qi[P_MIN], qi[P_MAX], qi[P_AMAX]});
      tc[8] += (int)qi[P_BAD];
#pragma unroll
      for (int k = 0; k < 4; ++k) tc[k] += (int)qi[P_C3 + k];
    }
    for (int t = threadIdx.x; t < nmt; t += blockDim.x)
#pragma unroll
      for (int k = 0; k < 4; ++k) tc[4 + k] += (int)islots3(pp + (size_t)t * kPart)[P_MC3 + k];
    tr.warp(te, mt, x, tc);
  }
  __syncthreads();
  const long long step = g.count[b];
  ptt_diag& r = g.ring[(size_t)b * kRing + (size_t)(step % kRing)];
  // mid-plane sums: thread k < 32 adds slot k over the mid tiles in order, for
  // the record and its member's window
  if (threadIdx.x < 33) {
    const int k = threadIdx.x;
    double a = 0.0;
    if (k < 32) {
#pragma unroll 4
      for (int t = 0; t < nmt; ++t) a += pp[(size_t)t * kPart + P_MS + k];
      r.mid_sums[k >> 2][k & 3] = a;
    }
    window_add(g.macc + (size_t)b * kMacc, k, a);
  }
  if (threadIdx.x == blockDim.x - 1) {
    const double e = 0.25 * tr.energy();
    const KeyExt ext = tr.ext();
    const bool bad = (tr.count(8) != 0);
    const double qnan = __longlong_as_double(0x7ff8000000000000LL);
    r.step = step;
    r.t = step * pr.dt;
    r.energy = e;
    r.mean_trc = 0.5 * tr.mean();
    r.min_trc = bad ? qnan : dkey_val(ext.mn);
    const double mx = bad ? qnan : dkey_val(ext.mx);
    r.max_trc = mx;
    r.n_lt3 = tr.count(0); r.n_lt0 = tr.count(1);
    r.n_band3 = tr.count(2); r.n_band0 = tr.count(3);
    r.n_mid_lt3 = tr.count(4); r.n_mid_lt0 = tr.count(5);
    r.n_mid_band3 = tr.count(6); r.n_mid_band0 = tr.count(7);
    const bool blow = bad || !isfinite(e) || mx > pr.trc_max || sqrt(2.0 * e) > pr.u_max;
    r.status = blow ? PTT_BLOWUP : PTT_OK;
    r.reserved = 0;
    if (blow) g.status[b] = 1;
  }
}

__global__ void k_reset3(GroupDev g, int b) {
  if (threadIdx.x == 0) {
    g.count[b] = 0;
    g.status[b] = 0;
  }
}

YJob yjob3(const GroupDev& g, bool inverse, int M, int C, const FftPlan& pl, bool gauss) {
  YJob J{};
  J.gauss = gauss ? 1 : 0;
  J.tw4f = inverse ? g.tw4Pif : g.tw4Pf;   // the quarter-period tables of this direction
  J.tw4x = inverse ? g.tw4Pix : g.tw4Px;
  J.fexp = g.fexpP;
  J.K = g.KZ;
  J.N = g.N;
  J.M = M;
  J.inverse = inverse ? 1 : 0;
  J.C = C;
  J.pl = pl;
  J.status = g.status;
  J.cm = g.N;
  J.cn = 1;
  J.vm = 1;
  J.vj = g.KZ;
  for (int i = 0; i < kYFields; ++i) J.src_field2[i] = J.src_field3[i] = -1;
  return J;
}

static void z_set_lines(ZJob& Z, int C) {
  Z.C = C;
  Z.dC = fast_div((unsigned)C);
}

ZJob zjob(const GroupDev& g, bool inverse, int Mz, int rows, const FftPlan& pl) {
  ZJob Z{};
  Z.K = g.K;
  Z.nz = g.nz;
  Z.Mz = Mz;
  Z.inv = 1.0 / Mz;
  Z.invf = (float)Z.inv;
  Z.inverse = inverse ? 1 : 0;
  Z.rows = rows;
  Z.status = g.status;
  Z.prm = g.prm;
  Z.pl = pl;
  Z.dnz = fast_div((unsigned)Z.nz);
  Z.dMz = fast_div((unsigned)Mz);
  Z.drows = fast_div((unsigned)rows);
  z_set_lines(Z, 8);
  return Z;
}

size_t smem_zcols(int C, int Mz) { return (size_t)C * Mz * 16; }   // two FP32 buffers, or one of fxc

template <typename F>
cudaError_t optin3(F* fn, int optin_bytes) {
  cudaFuncAttributes a;
  cudaError_t e = cudaFuncGetAttributes(&a, fn);
  if (e) return e;
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              optin_bytes - (int)a.sharedSizeBytes);
}

}  // namespace

size_t smem_xfused3(int Mx, int f32) {
  (void)f32;                                   // two FP32 buffers take what one of fxc takes
  const size_t b = (size_t)18 * Mx * 16;
  return b <= kSmemMax - 2048 ? b : 0;
}
size_t spec3_scratch_columns() { return kScr3; }
size_t smem_zcols3(int C, int Mz) { return smem_zcols(C, Mz); }

cudaError_t set_kernel_attributes3(int optin_bytes) {
  cudaError_t e;
  if ((e = optin3(k_ycols<float2>, optin_bytes))) return e;
  if ((e = optin3(k_ycols<fxc>, optin_bytes))) return e;
  if ((e = optin3(k_ycols<fxc, true>, optin_bytes))) return e;
  if ((e = optin3(k_zcols, optin_bytes))) return e;
  if ((e = optin3(k_zcols_fx<false>, optin_bytes))) return e;
  if ((e = optin3(k_zcols_fx<true>, optin_bytes))) return e;
  if ((e = optin3(k_xfused3, optin_bytes))) return e;
  if ((e = optin3(k_xfused3_fx<256, 4>, optin_bytes))) return e;
  if ((e = optin3(k_xfused3_fx<512, 1>, optin_bytes))) return e;
  if ((e = optin3(k_xrows, optin_bytes))) return e;
  return cudaSuccess;
}

static void launch_spec3(const GroupDev& g, int mode, cudaStream_t st) {
  k_spec3<<<dim3(cdiv(g.KZ, kModesPerBlock), g.nb), 256, 0, st>>>(g, mode);
}

// Stage s of one 3D step for one group (same numbering as the 2D stages).
cudaError_t launch_stage3(const GroupDev& g, int stage, cudaStream_t st, int* nl) {
  const int M = g.M, K = g.K, KZ = g.KZ, Mz = g.Mz;
  const size_t NK = (size_t)g.N * KZ;
  const long long yplane = (long long)M * KZ;          // Y3 / V3 field size
  const long long zplane = (long long)M * Mz * K;      // Z3 / W3 field size
  const int f32 = g.f32;
  int n = 0;
  switch (stage) {
    case 0: {  // inverse y (17 fields) then inverse z (26 lines)
      YJob J = yjob3(g, true, M, g.Ccol, g.plP, true);
      J.src = g.X;
      J.dst = f32 ? (void*)g.Y3f : (void*)g.Y3;
      J.dst_f32 = f32;
      J.src_mstride = 9 * NK; J.dst_mstride = 17 * yplane;
      J.src_fstride = NK; J.dst_fstride = yplane;
      const int sf[17] = {0, 1, 2, 3, 4, 5, 6, 7, 8, 0, 2, 3, 4, 5, 6, 7, 8};
      const int dv[17] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 1, 1, 1, 1, 1, 1, 1, 1};
      for (int i = 0; i < 17; ++i) { J.src_field[i] = sf[i]; J.dst_field[i] = i; J.deriv[i] = dv[i]; }
      const dim3 grid(cdiv(KZ, g.Ccol), 17, g.nb);
      if (f32 && g.ymma) {
        cudaError_t e = launch_cheb_mma(g, true, st, g.nsm);
        if (e) return e;
      } else if (f32) {
        k_ycols<float2><<<grid, 256, smem_ycols(g.Ccol, M), st>>>(J);
      } else {
        k_ycols<fxc><<<grid, 256, smem_ycols_fx(g.Ccol, M, g.N), st>>>(J);
      }
      ++n;
      if (f32) {   // the mean column (kx = kz = 0) in fixed point, FP64 out
        YJob Jm = J;
        Jm.K = 1; Jm.C = 1; Jm.pl = g.plPn;
        Jm.dst = g.Ym; Jm.dst_f32 = 0;
        Jm.dst_mstride = 17LL * M; Jm.dst_fstride = M;
        Jm.vm = 1; Jm.vj = 1;
        k_ycols<fxc><<<dim3(1, 17, g.nb), 256, smem_ycols_fx(1, M, g.N), st>>>(Jm);
        ++n;
      }
      ZJob Z = zjob(g, true, Mz, M, g.plMz);
      z_set_lines(Z, g.zC);
      Z.src = J.dst;
      Z.dst = f32 ? (void*)g.Z3f : (void*)g.Z3;
      Z.mean = f32 ? 1 : 0;
      Z.src_mstride = 17 * yplane; Z.dst_mstride = 26 * zplane;
      Z.src_fstride = yplane; Z.dst_fstride = zplane;
      for (int i = 0; i < 26; ++i) {
        Z.src_field[i] = (i < 17) ? i : i - 17;
        Z.dst_field[i] = i;
        Z.dz[i] = (i >= 17) ? 1 : 0;
      }
      const dim3 zgrid(cdiv(K, Z.C), 26 * M, g.nb);
      if (f32) k_zcols<<<zgrid, 256, smem_zcols(Z.C, Mz), st>>>(Z);
      else k_zcols_fx<false><<<zgrid, 256, smem_zcols(Z.C, Mz), st>>>(Z);
      ++n;
      break;
    }
    case 1: {
      const dim3 grid(M * Mz, g.nb);
      const size_t sm = smem_xfused3(g.Mx, f32);
      if (f32) k_xfused3<<<grid, g.xthreads, sm, st>>>(g);
      else if (g.xthreads <= 256) k_xfused3_fx<256, 4><<<grid, g.xthreads, sm, st>>>(g);
      else k_xfused3_fx<512, 1><<<grid, g.xthreads, sm, st>>>(g);
      n = 1;
      break;
    }
    case 2: {  // forward z (9) then forward y (9)
      ZJob Z = zjob(g, false, Mz, M, g.plMz);
      z_set_lines(Z, g.zC);
      Z.src = f32 ? (const void*)g.W3f : (const void*)g.W3;
      Z.dst = f32 ? (void*)g.V3f : (void*)g.V3;
      Z.mean = f32 ? 2 : 0;
      Z.zm = g.Zm;
      Z.inv = 1.0;   // fixed point: the y table holds the normalisation
      Z.src_mstride = 9 * zplane; Z.dst_mstride = 9 * yplane;
      Z.src_fstride = zplane; Z.dst_fstride = yplane;
      for (int i = 0; i < 9; ++i) { Z.src_field[i] = i; Z.dst_field[i] = i; Z.dz[i] = 0; }
      const dim3 zgrid(cdiv(K, Z.C), 9 * M, g.nb);
      if (f32) k_zcols<<<zgrid, 256, smem_zcols(Z.C, Mz), st>>>(Z);
      else k_zcols_fx<false><<<zgrid, 256, smem_zcols(Z.C, Mz), st>>>(Z);
      YJob F = yjob3(g, false, M, g.Ccol, g.plP, true);
      F.src = Z.dst; F.src_f32 = f32;
      F.dst = g.NR;
      F.src_mstride = 9 * yplane; F.dst_mstride = 9 * NK;
      F.src_fstride = yplane; F.dst_fstride = NK;
      for (int i = 0; i < 9; ++i) { F.src_field[i] = i; F.dst_field[i] = i; F.deriv[i] = 0; }
      const dim3 grid(cdiv(KZ, g.Ccol), 9, g.nb);
      if (f32 && g.ymma) {
        cudaError_t e = launch_cheb_mma(g, false, st, g.nsm);
        if (e) return e;
      } else if (f32) {
        k_ycols<float2><<<grid, 256, smem_ycols(g.Ccol, M), st>>>(F);
      } else {
        k_ycols<fxc><<<grid, 256, smem_ycols_fx(g.Ccol, M, 0), st>>>(F);
      }
      n = 2;
      if (f32) {   // the mean column in fixed point, over the FP32 pass's zeros
        YJob Fm = F;
        Fm.K = 1; Fm.C = 1; Fm.pl = g.plPn;
        Fm.src = g.Zm; Fm.src_f32 = 0;
        Fm.src_mstride = 9LL * M; Fm.src_fstride = M;
        Fm.vm = 1; Fm.vj = 1;
        k_ycols<fxc><<<dim3(1, 9, g.nb), 256, smem_ycols_fx(1, M, 0), st>>>(Fm);
        ++n;
      }
      break;
    }
    case 3:
      launch_spec3(g, 0, st);
      k_tick3<<<cdiv(g.nb, 128), 128, 0, st>>>(g);
      n = 2;
      break;
    case 4: {  // diagnostics, in order on one stream
      const DiagStreams d{{st, st, st}, {nullptr, nullptr, nullptr}};
      return launch_diag_split3(g, d, nl);
    }
    default:
      return cudaErrorInvalidValue;
  }
  if (nl) *nl += n;
  return cudaGetLastError();
}

// Fork d.s[1], d.s[2] off d.s[0] (when distinct) before the parts, join after.
static cudaError_t diag_fork3(const DiagStreams& d) {
  if (d.s[1] == d.s[0]) return cudaSuccess;
  cudaError_t e = cudaEventRecord(d.ev[0], d.s[0]);
  if (!e) e = cudaStreamWaitEvent(d.s[1], d.ev[0], 0);
  if (!e) e = cudaStreamWaitEvent(d.s[2], d.ev[0], 0);
  return e;
}
static cudaError_t diag_join3(const DiagStreams& d) {
  if (d.s[1] == d.s[0]) return cudaSuccess;
  cudaError_t e = cudaEventRecord(d.ev[1], d.s[1]);
  if (!e) e = cudaEventRecord(d.ev[2], d.s[2]);
  if (!e) e = cudaStreamWaitEvent(d.s[0], d.ev[1], 0);
  if (!e) e = cudaStreamWaitEvent(d.s[0], d.ev[2], 0);
  return e;
}

// The diagnostics' y transforms (they write only DY, DT): u, v, w on the Me
// Gauss points; c_xx + c_yy + c_zz on the unpadded Gauss-Lobatto rows.
static void diag_energy_y3(const GroupDev& g, cudaStream_t st) {
  const int KZ = g.KZ;
  const size_t NK = (size_t)g.N * KZ;
  YJob J = yjob3(g, true, g.Me, g.CcolE, g.plPe, true);
  J.tw4f = g.tw4Ef;   // mixed groups transform in FP32 (the sums stay FP64)
  J.tw4x = g.tw4Ex;
  J.src = g.X; J.dst = g.DY;
  J.src_mstride = 9 * NK; J.dst_mstride = 3LL * g.Me * KZ;
  J.src_fstride = NK; J.dst_fstride = (long long)g.Me * KZ;
  for (int i = 0; i < 3; ++i) { J.src_field[i] = i; J.dst_field[i] = i; J.deriv[i] = 0; }
  const dim3 grid(cdiv(KZ, g.CcolE), 3, g.nb);
  if (g.f32) k_ycols<float2><<<grid, 256, smem_ycols(g.CcolE, g.Me), st>>>(J);
  else k_ycols<fxc><<<grid, 256, smem_ycols_fx(g.CcolE, g.Me, 0), st>>>(J);
}
static void diag_trc_y3(const GroupDev& g, cudaStream_t st) {
  const int KZ = g.KZ;
  const size_t NK = (size_t)g.N * KZ;
  YJob T = yjob3(g, true, g.N - 1, g.CcolU, g.plPu, false);
  T.src = g.X; T.dst = g.DT;
  T.src_mstride = 9 * NK; T.dst_mstride = (long long)NK;
  T.src_fstride = NK; T.dst_fstride = 0;
  T.src_field[0] = 3; T.src_field2[0] = 6; T.src_field3[0] = 8; T.dst_field[0] = 0; T.deriv[0] = 0;
  k_ycols<fxc, true><<<dim3(cdiv(KZ, g.CcolU), 1, g.nb), 256, smem_ycols_fx(g.CcolU, g.Pu, 0), st>>>(T);
}

cudaError_t launch_diag_transforms3(const GroupDev& g, cudaStream_t st) {
  diag_energy_y3(g, st);
  diag_trc_y3(g, st);
  return cudaGetLastError();
}

cudaError_t launch_diag_split3(const GroupDev& g, const DiagStreams& d, int* nl) {
  const int KZ = g.KZ, K = g.K;
  const size_t NK = (size_t)g.N * KZ;
  cudaError_t e = diag_fork3(d);
  if (e) return e;
  diag_energy_y3(g, d.s[1]);
  // mid-plane: per-mode sums, then z and x syntheses of the 8 quantities
  k_diag_mid3<<<dim3(cdiv(KZ, kMidModesPerBlock3), g.nb), 256, 0, d.s[2]>>>(g);
  ZJob Zm = zjob(g, true, g.nz, 1, g.plNz);
  Zm.src = g.DM; Zm.dst = g.DMZ;
  Zm.src_mstride = 8LL * KZ; Zm.dst_mstride = 8LL * g.nz * K;
  Zm.src_fstride = KZ; Zm.dst_fstride = (long long)g.nz * K;
  for (int i = 0; i < 8; ++i) { Zm.src_field[i] = i; Zm.dst_field[i] = i; Zm.dz[i] = 0; }
  k_zcols_fx<true><<<dim3(cdiv(K, Zm.C), 8, g.nb), 256, smem_zcols(Zm.C, g.nz), d.s[2]>>>(Zm);
  XJob Xm{};
  Xm.srcC = g.DMZ; Xm.dstR = g.MV;
  Xm.src_mstride = 8LL * g.nz * K; Xm.dst_mstride = 8LL * g.nz * g.nx;
  Xm.src_fstride = (long long)g.nz * K; Xm.dst_fstride = (long long)g.nz * g.nx;
  Xm.src_rstep = 1; Xm.dst_rstep = 1;
  Xm.nf = 8; Xm.K = K; Xm.n = g.nx; Xm.c2r = 1; Xm.status = g.status; Xm.pl = g.plNx;
  k_xrows<<<dim3(g.nz, g.nb), 256, smem_xrows(4, g.nx), d.s[2]>>>(Xm);
  // Tr c = c_xx + c_yy + c_zz on the unpadded grid: y (Gauss-Lobatto) -> z -> x
  diag_trc_y3(g, d.s[0]);
  ZJob Z = zjob(g, true, g.nz, g.N, g.plNz);
  Z.src = g.DT; Z.dst = g.DZ;
  Z.src_mstride = (long long)NK; Z.dst_mstride = (long long)g.N * g.nz * K;
  Z.src_fstride = 0; Z.dst_fstride = 0;
  Z.src_field[0] = 0; Z.dst_field[0] = 0; Z.dz[0] = 0;
  k_zcols_fx<true><<<dim3(cdiv(K, Z.C), g.N, g.nb), 256, smem_zcols(Z.C, g.nz), d.s[0]>>>(Z);
  XJob X{};
  X.srcC = g.DZ; X.dstR = g.DV;
  X.src_mstride = (long long)g.N * g.nz * K; X.dst_mstride = (long long)g.N * g.nz * g.nx;
  X.src_fstride = 0; X.dst_fstride = 0;
  X.src_rstep = 1; X.dst_rstep = 1;
  X.nf = 1; X.K = K; X.n = g.nx; X.c2r = 1; X.status = g.status; X.pl = g.plNx;
  X.nrows = g.N * g.nz; X.pair_rows = xrows_pairs(g.nx, X.nrows * g.nb);
  k_xrows<<<dim3(xrows_pair_blocks(X.pair_rows, X.nrows), g.nb), 256, smem_xrows(X.pair_rows, g.nx), d.s[0]>>>(X);
  if ((e = cudaGetLastError()) || (e = diag_join3(d))) return e;
  k_diag_part3<<<dim3(g.ntile, g.nb), 256, 0, d.s[0]>>>(g);
  k_diag_count3<<<dim3(g.ntile, g.nb), 256, 0, d.s[0]>>>(g);
  k_diag_final3<<<g.nb, 256, 0, d.s[0]>>>(g);
  if (nl) *nl += 10;
  return cudaGetLastError();
}

cudaError_t launch_step3(const GroupDev& g, cudaStream_t st, int* nl) {
  for (int s = 0; s < 4; ++s) {
    cudaError_t e = launch_stage3(g, s, st, nl);
    if (e) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_diag3(const GroupDev& g, cudaStream_t st, int* nl) { return launch_stage3(g, 4, st, nl); }

cudaError_t launch_explicit3(const GroupDev& g, cudaStream_t st) {
  for (int s = 0; s < 3; ++s) {
    cudaError_t e = launch_stage3(g, s, st, nullptr);
    if (e) return e;
  }
  launch_spec3(g, 1, st);
  return cudaGetLastError();
}

cudaError_t launch_reset_member3(const GroupDev& g, int b, cudaStream_t st) {
  k_reset3<<<1, 32, 0, st>>>(g, b);
  return cudaGetLastError();
}

// physical staging [9][ny][nz][nx] -> state of member b: x analysis per
// (y, z) row, z analysis per (y, mx), y analysis (DCT-I) per mode.
cudaError_t launch_phys_to_state3(const GroupDev& g, int b, bool abi, cudaStream_t st) {
  const int K = g.K, KZ = g.KZ, N = g.N, nz = g.nz, nx = g.nx;
  const size_t NK = (size_t)N * KZ;
  const long long rowsp = (long long)N * nz;
  XJob X{};
  X.srcR = g.stage; X.dstC = g.DZ;   // DZ reused as [9][N][nz][K]
  if (abi) { X.zy_nz = nz; X.zy_ny = N; }
  X.src_fstride = rowsp * nx; X.dst_fstride = rowsp * K;
  X.src_rstep = 1; X.dst_rstep = 1;
  X.nf = 9; X.K = K; X.n = nx; X.c2r = 0; X.status = nullptr; X.pl = g.plNx;
  k_xrows<<<dim3((unsigned)rowsp, 1), 256, smem_xrows(5, nx), st>>>(X);
  ZJob Z = zjob(g, false, nz, N, g.plNz);
  Z.status = nullptr;
  Z.src = g.DZ; Z.dst = g.stageS;     // stageS reused as [9][N][KZ]
  Z.src_fstride = rowsp * K; Z.dst_fstride = (long long)N * KZ;
  for (int i = 0; i < 9; ++i) { Z.src_field[i] = i; Z.dst_field[i] = i; Z.dz[i] = 0; }
  k_zcols_fx<true><<<dim3(cdiv(K, Z.C), 9 * N, 1), 256, smem_zcols(Z.C, nz), st>>>(Z);
  YJob J = yjob3(g, false, N - 1, g.CcolU, g.plPu, false);
  J.status = nullptr;
  J.src = g.stageS; J.dst = g.X + (size_t)b * 9 * NK;
  J.src_fstride = (long long)N * KZ; J.dst_fstride = NK;
  for (int i = 0; i < 9; ++i) { J.src_field[i] = i; J.dst_field[i] = i; J.deriv[i] = 0; }
  k_ycols<fxc, true><<<dim3(cdiv(KZ, g.CcolU), 9, 1), 256, smem_ycols_fx(g.CcolU, g.Pu, 0), st>>>(J);
  k_reset3<<<1, 32, 0, st>>>(g, b);
  return cudaGetLastError();
}

cudaError_t launch_state_to_phys3(const GroupDev& g, int b, cudaStream_t st) {
  const int K = g.K, KZ = g.KZ, N = g.N, nz = g.nz, nx = g.nx;
  const size_t NK = (size_t)N * KZ;
  const long long rowsp = (long long)N * nz;
  YJob J = yjob3(g, true, N - 1, g.CcolU, g.plPu, false);
  J.status = nullptr;
  J.src = g.X + (size_t)b * 9 * NK; J.dst = g.stageS;
  J.src_fstride = NK; J.dst_fstride = (long long)N * KZ;
  for (int i = 0; i < 9; ++i) { J.src_field[i] = i; J.dst_field[i] = i; J.deriv[i] = 0; }
  k_ycols<fxc, true><<<dim3(cdiv(KZ, g.CcolU), 9, 1), 256, smem_ycols_fx(g.CcolU, g.Pu, 0), st>>>(J);
  ZJob Z = zjob(g, true, nz, N, g.plNz);
  Z.status = nullptr;
  Z.src = g.stageS; Z.dst = g.DZ;
  Z.src_fstride = (long long)N * KZ; Z.dst_fstride = rowsp * K;
  for (int i = 0; i < 9; ++i) { Z.src_field[i] = i; Z.dst_field[i] = i; Z.dz[i] = 0; }
  k_zcols_fx<true><<<dim3(cdiv(K, Z.C), 9 * N, 1), 256, smem_zcols(Z.C, nz), st>>>(Z);
  XJob X{};
  X.srcC = g.DZ; X.dstR = g.stage;
  X.zy_nz = nz; X.zy_ny = N;
  X.src_fstride = rowsp * K; X.dst_fstride = rowsp * nx;
  X.src_rstep = 1; X.dst_rstep = 1;
  X.nf = 9; X.K = K; X.n = nx; X.c2r = 1; X.status = nullptr; X.pl = g.plNx;
  k_xrows<<<dim3((unsigned)rowsp, 1), 256, smem_xrows(5, nx), st>>>(X);
  return cudaGetLastError();
}

}  // namespace ptt
