// Two-stage register FFT building blocks for the common grid sides (N = R1 * R2,
// both factors at most 32).  A thread takes R1 elements of a line straight from
// global memory into registers and does the first decimation-in-frequency stage
// there; the only shared-memory round trip is the transpose to the second stage,
// whose outputs go back to global memory in the digit-reversed order that the
// general in-place passes also leave (so both kinds of pass share the tables).
#pragma once

#include "icm_internal.h"

namespace icm {
namespace {

// exp(-2 pi i j / 96), j = 0..95, correctly rounded: the twiddles of every small
// DFT below (orders 2, 3, 4, 6, 8, 12, 16, 24, 32 all divide 96).
__constant__ double2 c_w96d[96] = {
  {1.0, 0.0},
  {0.9978589232386035, -0.06540312923014306},
  {0.9914448613738104, -0.1305261922200516},
  {0.9807852804032304, -0.19509032201612828},
  {0.9659258262890683, -0.25881904510252074},
  {0.9469301294951057, -0.3214394653031616},
  {0.9238795325112867, -0.3826834323650898},
  {0.8968727415326883, -0.4422886902190013},
  {0.8660254037844386, -0.5},
  {0.8314696123025452, -0.5555702330196022},
  {0.7933533402912352, -0.6087614290087207},
  {0.7518398074789774, -0.6593458151000688},
  {0.7071067811865476, -0.7071067811865476},
  {0.6593458151000688, -0.7518398074789774},
  {0.6087614290087207, -0.7933533402912352},
  {0.5555702330196022, -0.8314696123025452},
  {0.5, -0.8660254037844386},
  {0.4422886902190013, -0.8968727415326883},
  {0.3826834323650898, -0.9238795325112867},
  {0.3214394653031616, -0.9469301294951057},
  {0.25881904510252074, -0.9659258262890683},
  {0.19509032201612828, -0.9807852804032304},
  {0.1305261922200516, -0.9914448613738104},
  {0.06540312923014306, -0.9978589232386035},
  {0.0, -1.0},
  {-0.06540312923014306, -0.9978589232386035},
  {-0.1305261922200516, -0.9914448613738104},
  {-0.19509032201612828, -0.9807852804032304},
  {-0.25881904510252074, -0.9659258262890683},
  {-0.3214394653031616, -0.9469301294951057},
  {-0.3826834323650898, -0.9238795325112867},
  {-0.4422886902190013, -0.8968727415326883},
  {-0.5, -0.8660254037844386},
  {-0.5555702330196022, -0.8314696123025452},
  {-0.6087614290087207, -0.7933533402912352},
  {-0.6593458151000688, -0.7518398074789774},
  {-0.7071067811865476, -0.7071067811865476},
  {-0.7518398074789774, -0.6593458151000688},
  {-0.7933533402912352, -0.6087614290087207},
  {-0.8314696123025452, -0.5555702330196022},
  {-0.8660254037844386, -0.5},
  {-0.8968727415326883, -0.4422886902190013},
  {-0.9238795325112867, -0.3826834323650898},
  {-0.9469301294951057, -0.3214394653031616},
  {-0.9659258262890683, -0.25881904510252074},
  {-0.9807852804032304, -0.19509032201612828},
  {-0.9914448613738104, -0.1305261922200516},
  {-0.9978589232386035, -0.06540312923014306},
  {-1.0, 0.0},
  {-0.9978589232386035, 0.06540312923014306},
  {-0.9914448613738104, 0.1305261922200516},
  {-0.9807852804032304, 0.19509032201612828},
  {-0.9659258262890683, 0.25881904510252074},
  {-0.9469301294951057, 0.3214394653031616},
  {-0.9238795325112867, 0.3826834323650898},
  {-0.8968727415326883, 0.4422886902190013},
  {-0.8660254037844386, 0.5},
  {-0.8314696123025452, 0.5555702330196022},
  {-0.7933533402912352, 0.6087614290087207},
  {-0.7518398074789774, 0.6593458151000688},
  {-0.7071067811865476, 0.7071067811865476},
  {-0.6593458151000688, 0.7518398074789774},
  {-0.6087614290087207, 0.7933533402912352},
  {-0.5555702330196022, 0.8314696123025452},
  {-0.5, 0.8660254037844386},
  {-0.4422886902190013, 0.8968727415326883},
  {-0.3826834323650898, 0.9238795325112867},
  {-0.3214394653031616, 0.9469301294951057},
  {-0.25881904510252074, 0.9659258262890683},
  {-0.19509032201612828, 0.9807852804032304},
  {-0.1305261922200516, 0.9914448613738104},
  {-0.06540312923014306, 0.9978589232386035},
  {0.0, 1.0},
  {0.06540312923014306, 0.9978589232386035},
  {0.1305261922200516, 0.9914448613738104},
  {0.19509032201612828, 0.9807852804032304},
  {0.25881904510252074, 0.9659258262890683},
  {0.3214394653031616, 0.9469301294951057},
  {0.3826834323650898, 0.9238795325112867},
  {0.4422886902190013, 0.8968727415326883},
  {0.5, 0.8660254037844386},
  {0.5555702330196022, 0.8314696123025452},
  {0.6087614290087207, 0.7933533402912352},
  {0.6593458151000688, 0.7518398074789774},
  {0.7071067811865476, 0.7071067811865476},
  {0.7518398074789774, 0.6593458151000688},
  {0.7933533402912352, 0.6087614290087207},
  {0.8314696123025452, 0.5555702330196022},
  {0.8660254037844386, 0.5},
  {0.8968727415326883, 0.4422886902190013},
  {0.9238795325112867, 0.3826834323650898},
  {0.9469301294951057, 0.3214394653031616},
  {0.9659258262890683, 0.25881904510252074},
  {0.9807852804032304, 0.19509032201612828},
  {0.9914448613738104, 0.1305261922200516},
  {0.9978589232386035, 0.06540312923014306}
};
__constant__ float2 c_w96f[96] = {
  {1.0f, 0.0f},
  {0.9978589232386035f, -0.06540312923014306f},
  {0.9914448613738104f, -0.1305261922200516f},
  {0.9807852804032304f, -0.19509032201612828f},
  {0.9659258262890683f, -0.25881904510252074f},
  {0.9469301294951057f, -0.3214394653031616f},
  {0.9238795325112867f, -0.3826834323650898f},
  {0.8968727415326883f, -0.4422886902190013f},
  {0.8660254037844386f, -0.5f},
  {0.8314696123025452f, -0.5555702330196022f},
  {0.7933533402912352f, -0.6087614290087207f},
  {0.7518398074789774f, -0.6593458151000688f},
  {0.7071067811865476f, -0.7071067811865476f},
  {0.6593458151000688f, -0.7518398074789774f},
  {0.6087614290087207f, -0.7933533402912352f},
  {0.5555702330196022f, -0.8314696123025452f},
  {0.5f, -0.8660254037844386f},
  {0.4422886902190013f, -0.8968727415326883f},
  {0.3826834323650898f, -0.9238795325112867f},
  {0.3214394653031616f, -0.9469301294951057f},
  {0.25881904510252074f, -0.9659258262890683f},
  {0.19509032201612828f, -0.9807852804032304f},
  {0.1305261922200516f, -0.9914448613738104f},
  {0.06540312923014306f, -0.9978589232386035f},
  {0.0f, -1.0f},
  {-0.06540312923014306f, -0.9978589232386035f},
  {-0.1305261922200516f, -0.9914448613738104f},
  {-0.19509032201612828f, -0.9807852804032304f},
  {-0.25881904510252074f, -0.9659258262890683f},
  {-0.3214394653031616f, -0.9469301294951057f},
  {-0.3826834323650898f, -0.9238795325112867f},
  {-0.4422886902190013f, -0.8968727415326883f},
  {-0.5f, -0.8660254037844386f},
  {-0.5555702330196022f, -0.8314696123025452f},
  {-0.6087614290087207f, -0.7933533402912352f},
  {-0.6593458151000688f, -0.7518398074789774f},
  {-0.7071067811865476f, -0.7071067811865476f},
  {-0.7518398074789774f, -0.6593458151000688f},
  {-0.7933533402912352f, -0.6087614290087207f},
  {-0.8314696123025452f, -0.5555702330196022f},
  {-0.8660254037844386f, -0.5f},
  {-0.8968727415326883f, -0.4422886902190013f},
  {-0.9238795325112867f, -0.3826834323650898f},
  {-0.9469301294951057f, -0.3214394653031616f},
  {-0.9659258262890683f, -0.25881904510252074f},
  {-0.9807852804032304f, -0.19509032201612828f},
  {-0.9914448613738104f, -0.1305261922200516f},
  {-0.9978589232386035f, -0.06540312923014306f},
  {-1.0f, 0.0f},
  {-0.9978589232386035f, 0.06540312923014306f},
  {-0.9914448613738104f, 0.1305261922200516f},
  {-0.9807852804032304f, 0.19509032201612828f},
  {-0.9659258262890683f, 0.25881904510252074f},
  {-0.9469301294951057f, 0.3214394653031616f},
  {-0.9238795325112867f, 0.3826834323650898f},
  {-0.8968727415326883f, 0.4422886902190013f},
  {-0.8660254037844386f, 0.5f},
  {-0.8314696123025452f, 0.5555702330196022f},
  {-0.7933533402912352f, 0.6087614290087207f},
  {-0.7518398074789774f, 0.6593458151000688f},
  {-0.7071067811865476f, 0.7071067811865476f},
  {-0.6593458151000688f, 0.7518398074789774f},
  {-0.6087614290087207f, 0.7933533402912352f},
  {-0.5555702330196022f, 0.8314696123025452f},
  {-0.5f, 0.8660254037844386f},
  {-0.4422886902190013f, 0.8968727415326883f},
  {-0.3826834323650898f, 0.9238795325112867f},
  {-0.3214394653031616f, 0.9469301294951057f},
  {-0.25881904510252074f, 0.9659258262890683f},
  {-0.19509032201612828f, 0.9807852804032304f},
  {-0.1305261922200516f, 0.9914448613738104f},
  {-0.06540312923014306f, 0.9978589232386035f},
  {0.0f, 1.0f},
  {0.06540312923014306f, 0.9978589232386035f},
  {0.1305261922200516f, 0.9914448613738104f},
  {0.19509032201612828f, 0.9807852804032304f},
  {0.25881904510252074f, 0.9659258262890683f},
  {0.3214394653031616f, 0.9469301294951057f},
  {0.3826834323650898f, 0.9238795325112867f},
  {0.4422886902190013f, 0.8968727415326883f},
  {0.5f, 0.8660254037844386f},
  {0.5555702330196022f, 0.8314696123025452f},
  {0.6087614290087207f, 0.7933533402912352f},
  {0.6593458151000688f, 0.7518398074789774f},
  {0.7071067811865476f, 0.7071067811865476f},
  {0.7518398074789774f, 0.6593458151000688f},
  {0.7933533402912352f, 0.6087614290087207f},
  {0.8314696123025452f, 0.5555702330196022f},
  {0.8660254037844386f, 0.5f},
  {0.8968727415326883f, 0.4422886902190013f},
  {0.9238795325112867f, 0.3826834323650898f},
  {0.9469301294951057f, 0.3214394653031616f},
  {0.9659258262890683f, 0.25881904510252074f},
  {0.9807852804032304f, 0.19509032201612828f},
  {0.9914448613738104f, 0.1305261922200516f},
  {0.9978589232386035f, 0.06540312923014306f}
};

template <typename R> __device__ __forceinline__ cplx_t<R> w96(int j);
template <> __device__ __forceinline__ float2 w96<float>(int j) { return c_w96f[j]; }
template <> __device__ __forceinline__ double2 w96<double>(int j) { return c_w96d[j]; }

// a exp(-2 pi i j / 96), j a constant after unrolling: quarter turns are swaps (as a product
// with a table entry they cost four operations), the rest are constant-bank operands.
template <typename R> __device__ __forceinline__ cplx_t<R> mulw96(cplx_t<R> a, int j) {
  if (j == 0) return a;
  if (j == 24) return cmul_mi(a);
  if (j == 48) return mk(-a.x, -a.y);
  if (j == 72) return cmul_pi(a);
  return cmul(a, w96<R>(j));
}

// Small forward DFTs in registers, natural order in and out.
template <typename R, int N> struct SDft;

// N = A*B: y_n1 = DFT_A(a[n1 + B n2]) W_N^(n1 k2); X[A k1 + k2] = DFT_B over n1 of y_n1[k2].
template <typename R, int A, int B>
struct SDftComp {
  __device__ __forceinline__ static void run(cplx_t<R>* a) {
    constexpr int N = A * B;
    cplx_t<R> t[N];
#pragma unroll
    for (int n1 = 0; n1 < B; ++n1) {
      cplx_t<R> y[A];
#pragma unroll
      for (int n2 = 0; n2 < A; ++n2) y[n2] = a[n1 + B * n2];
      SDft<R, A>::run(y);
#pragma unroll
      for (int k2 = 0; k2 < A; ++k2)
        t[n1 * A + k2] = mulw96<R>(y[k2], ((96 / N) * n1 * k2) % 96);
    }
#pragma unroll
    for (int k2 = 0; k2 < A; ++k2) {
      cplx_t<R> z[B];
#pragma unroll
      for (int n1 = 0; n1 < B; ++n1) z[n1] = t[n1 * A + k2];
      SDft<R, B>::run(z);
#pragma unroll
      for (int k1 = 0; k1 < B; ++k1) a[A * k1 + k2] = z[k1];
    }
  }
};
template <typename R> struct SDft<R, 1> {
  __device__ __forceinline__ static void run(cplx_t<R>*) {}
};
template <typename R> struct SDft<R, 2> {
  __device__ __forceinline__ static void run(cplx_t<R>* a) {
    const cplx_t<R> t = a[0];
    a[0] = cadd(t, a[1]);
    a[1] = csub(t, a[1]);
  }
};
// Differences that are used after a quarter turn are formed turned, -i (a - b), component by component, so
// that the additions they enter are whole complex ones.
template <typename C> __device__ __forceinline__ C csub_mi(C a, C b) { return mk(a.y - b.y, b.x - a.x); }
template <typename R> struct SDft<R, 3> {
  __device__ __forceinline__ static void run(cplx_t<R>* a) {
    const R s = R(0.86602540378443864676);
    const cplx_t<R> t1 = cadd(a[1], a[2]), e = csub_mi(a[1], a[2]);
    const cplx_t<R> t2 = cfmar<R>(R(-0.5), t1, a[0]);
    a[0] = cadd(a[0], t1);
    a[1] = cfmar<R>(s, e, t2);
    a[2] = cfmar<R>(-s, e, t2);
  }
};
template <typename R> struct SDft<R, 4> {
  __device__ __forceinline__ static void run(cplx_t<R>* a) {
    const cplx_t<R> s02 = cadd(a[0], a[2]), d02 = csub(a[0], a[2]), s13 = cadd(a[1], a[3]), e13 = csub_mi(a[1], a[3]);
    a[0] = cadd(s02, s13);
    a[2] = csub(s02, s13);
    a[1] = cadd(d02, e13);
    a[3] = csub(d02, e13);
  }
};
// 9 = 3 x 3 with W_9^(n1 k2), n1 k2 in {1, 2, 4} (cos and sin of 40, 80 and 160 degrees).
template <typename R> struct SDft<R, 9> {
  __device__ __forceinline__ static void run(cplx_t<R>* a) {
    const cplx_t<R> w1 = mk(R(0.76604444311897803520), R(-0.64278760968653932632));
    const cplx_t<R> w2 = mk(R(0.17364817766693034885), R(-0.98480775301220805937));
    const cplx_t<R> w4 = mk(R(-0.93969262078590838405), R(-0.34202014332566873304));
    cplx_t<R> y[3][3];
#pragma unroll
    for (int n1 = 0; n1 < 3; ++n1) {
#pragma unroll
      for (int n2 = 0; n2 < 3; ++n2) y[n1][n2] = a[n1 + 3 * n2];
      SDft<R, 3>::run(y[n1]);
    }
    y[1][1] = cmul(y[1][1], w1);
    y[1][2] = cmul(y[1][2], w2);
    y[2][1] = cmul(y[2][1], w2);
    y[2][2] = cmul(y[2][2], w4);
#pragma unroll
    for (int k2 = 0; k2 < 3; ++k2) {
      cplx_t<R> z[3] = {y[0][k2], y[1][k2], y[2][k2]};
      SDft<R, 3>::run(z);
#pragma unroll
      for (int k1 = 0; k1 < 3; ++k1) a[3 * k1 + k2] = z[k1];
    }
  }
};
template <typename R> struct SDft<R, 6> : SDftComp<R, 2, 3> {};
// DFT_4 of u_0, W_8 u_1, e_2 = -i u_2, W_8^3 u_3.  The factor sqrt(1/2) common to the two eighth turns rides
// on the last additions as a fused multiply-add: 20 operations where rotating first takes 24.  The FP64
// passes are bound by their operations; with this, inverses free of negations and the spectra kept doubled,
// x / y / z / y / x of the 128^3 solve take 148 / 146 / 424 / 145 / 164 us (165 / 153 / 451 / 153 / 180 before).
template <typename R>
__device__ __forceinline__ void eighth_column(cplx_t<R> u0, cplx_t<R> u1, cplx_t<R> e2, cplx_t<R> u3, cplx_t<R>& o0,
                                              cplx_t<R>& o1, cplx_t<R>& o2, cplx_t<R>& o3) {
  const R r = R(0.70710678118654752440);
  const cplx_t<R> s = cadd(u0, e2), d = csub(u0, e2);
  const R px = u1.x + u1.y, py = u1.y - u1.x, qx = u3.y - u3.x, qy = u3.x + u3.y;
  const cplx_t<R> p = mk(px + qx, py - qy), m = mk(py + qy, qx - px);
  o0 = cfmar<R>(r, p, s);
  o2 = cfmar<R>(-r, p, s);
  o1 = cfmar<R>(r, m, d);
  o3 = cfmar<R>(-r, m, d);
}
template <typename R> struct SDft<R, 8> {
  // 8 = 2 x 4: even outputs DFT_4 of the sums, odd ones the eighth-turn column of the differences
  __device__ __forceinline__ static void run(cplx_t<R>* a) {
    cplx_t<R> b[4], u[4];
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      b[n] = cadd(a[n], a[n + 4]);
      u[n] = n == 2 ? csub_mi(a[n], a[n + 4]) : csub(a[n], a[n + 4]);
    }
    SDft<R, 4>::run(b);
#pragma unroll
    for (int k = 0; k < 4; ++k) a[2 * k] = b[k];
    eighth_column<R>(u[0], u[1], u[2], u[3], a[1], a[3], a[5], a[7]);
  }
};
template <typename R> struct SDft<R, 16> {
  // 16 = 4 x 4: y_n1 = DFT_4(a[n1 + 4 n2]); X[4 k1 + k2] = DFT_4 over n1 of W_16^(n1 k2) y_n1[k2]
  __device__ __forceinline__ static void run(cplx_t<R>* a) {
    const R r = R(0.70710678118654752440);
    cplx_t<R> y[4][4];
#pragma unroll
    for (int n1 = 0; n1 < 4; ++n1) {
#pragma unroll
      for (int n2 = 0; n2 < 4; ++n2) y[n1][n2] = a[n1 + 4 * n2];
      SDft<R, 4>::run(y[n1]);
    }
    {
      cplx_t<R> z[4] = {y[0][0], y[1][0], y[2][0], y[3][0]};
      SDft<R, 4>::run(z);
#pragma unroll
      for (int k = 0; k < 4; ++k) a[4 * k] = z[k];
    }
    eighth_column<R>(y[0][2], y[1][2], cmul_mi(y[2][2]), y[3][2], a[2], a[6], a[10], a[14]);
#pragma unroll
    for (int k2 = 1; k2 <= 3; k2 += 2) {   // W^2 or W^6 on the third input: its sqrt(1/2) in the sums too
      const cplx_t<R> z1 = mulw96<R>(y[1][k2], 6 * k2), z3 = mulw96<R>(y[3][k2], (18 * k2) % 96);
      const cplx_t<R> u = y[2][k2], z0 = y[0][k2];
      const cplx_t<R> p = k2 == 1 ? mk(u.x + u.y, u.y - u.x) : mk(u.y - u.x, -u.x - u.y);
      const cplx_t<R> s = cfmar<R>(r, p, z0), d = cfmar<R>(-r, p, z0);
      const cplx_t<R> t = cadd(z1, z3), e = csub_mi(z1, z3);
      a[k2] = cadd(s, t);
      a[8 + k2] = csub(s, t);
      a[4 + k2] = cadd(d, e);
      a[12 + k2] = csub(d, e);
    }
  }
};
template <typename R> struct SDft<R, 12> : SDftComp<R, 4, 3> {};
template <typename R> struct SDft<R, 24> : SDftComp<R, 8, 3> {};
template <typename R> struct SDft<R, 32> : SDftComp<R, 4, 8> {};

// Inverse (unnormalised) small DFT: the forward one with its outputs in reverse order, which costs
// nothing.
template <typename R, int M>
__device__ __forceinline__ void sdft_inv(cplx_t<R>* a) {
  SDft<R, M>::run(a);
#pragma unroll
  for (int i = 1; 2 * i < M; ++i) {
    const cplx_t<R> t = a[i];
    a[i] = a[M - i];
    a[M - i] = t;
  }
}

// First-stage twiddles laid out as tw2[k2 * R2 + n1] = W_N^(n1 k2) (N entries), so
// that threads at consecutive n1 read consecutive words.
template <typename R, int R1, int R2>
__device__ __forceinline__ void load_stage_twiddles(cplx_t<R>* tw2, const cplx_t<R>* __restrict__ gtw, int tid,
                                                    int nthr) {
  for (int i = tid; i < R1 * R2; i += nthr) {
    const int k2 = i / R2, n1 = i - k2 * R2;
    tw2[i] = gtw[n1 * k2];
  }
}

// First DIF stage at line position n1: a[r] = x[n1 + R2 r] becomes
// y[n1 + R2 k2] = W_N^(n1 k2) DFT_R1(a)[k2], with tw = tw2 + n1 (stride R2); and its
// exact inverse.
template <typename R, int R1, int R2>
__device__ __forceinline__ void stage_a_fwd(cplx_t<R>* a, const cplx_t<R>* tw) {
  SDft<R, R1>::run(a);
#pragma unroll
  for (int k2 = 1; k2 < R1; ++k2) a[k2] = cmul(a[k2], tw[k2 * R2]);
}
template <typename R, int R1, int R2>
__device__ __forceinline__ void stage_a_inv(cplx_t<R>* a, const cplx_t<R>* tw) {
#pragma unroll
  for (int k2 = 1; k2 < R1; ++k2) a[k2] = cmul(a[k2], cconj(tw[k2 * R2]));
  sdft_inv<R, R1>(a);
}

}  // namespace
}  // namespace icm
