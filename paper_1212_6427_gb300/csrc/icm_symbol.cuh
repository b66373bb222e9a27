// The Helmholtz/projection symbol of the z passes (arXiv:1212.6427, Sec. III.D), applied to
// the three components of one wave vector in registers.
#pragma once

#include "icm_internal.h"

namespace icm {

template <typename R>
struct SymParams {
  R a, b;         // of a + b|d|^2 with d for unit spacing (unit_b)
  R inv_ntot;     // 1/(2 ncell): the forward passes leave twice the spectrum (they split two packed real
                  // rows without the factor 1/2)
  R mean_scale;   // the symbol's scale on the mean mode: 1/(2 a ncell), 0 when a = 0
  const cplx_t<R>* dx; const R* ddx;
  const cplx_t<R>* dy; const R* ddy;
  const cplx_t<R>* dz; const R* ddz;
  const double* k0sum;
  double k0mul;   // k0scale / ncell
};

namespace {
// P^ w / (a + b|d|^2) / ncell on one wave vector: (P^ w)_a = w_a - conj(d_a)(d . w)/|d|^2,
// identity on the mean mode, whose value is replaced by the FP64 bookkeeping if given
// (and which is zero when a = 0).
// One reciprocal r = 1/(|d|^2 (a + b|d|^2)) serves both divisions; |d|^2 = 0 only on the mean mode,
// whose scale is precomputed.  |d|^2 is between 4 sin^2(pi/512) = 1.5e-4 and 12, so the product is in range where
// a + b|d|^2 and its reciprocal are.
// 1/x, x normal and positive: the hardware reciprocal in FP32 (within one ulp); in FP64 the
// approximate reciprocal instruction and one step of third order, y (1 + e + e^2) with
// e = 1 - x y, three FP64 operations where a division takes about ten (FP64 operations bound
// the FP64 z pass).
template <typename R> __device__ __forceinline__ R recip(R x);
template <> __device__ __forceinline__ float recip<float>(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));   // within one ulp; x is never denormal here
  return r;
}
template <> __device__ __forceinline__ double recip<double>(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// The lines of a z tile: kZLines wave numbers k0.. of one row.  In FP64, where rows are one wave number
// longer than whole tiles (every nx = 16 m), the last wave number of kZLines rows makes a tile instead: one
// of its own per row would be seven eighths idle, a ninth of the blocks at nx = 128.  z pass of 128^3, last
// column alone / folded: FP64, bound by its operations, 424 / 375 us; FP32, bound by latency, which the
// scattered column makes longer, 21.7 / 23.4 us (and 310 / 325 us on 512 x 384 x 256).
constexpr int kZLines = 8;
template <typename R>
__host__ __device__ constexpr bool z_folds(int kx) { return sizeof(R) == 8 && kx % kZLines == 1 && kx > kZLines; }
template <typename R>
__host__ __device__ constexpr int z_tiles_x(int kx) { return z_folds<R>(kx) ? kx / kZLines : (kx + kZLines - 1) / kZLines; }
template <typename R>
__host__ __device__ constexpr int z_tiles(int kx, int ny) {
  return z_tiles_x<R>(kx) * ny + (z_folds<R>(kx) ? (ny + kZLines - 1) / kZLines : 0);
}
template <typename R>
struct ZTile {
  int k0, row0;     // wave number and row of line 0
  bool folded;      // lines are rows
  __device__ __forceinline__ ZTile(int t, int kx, int ny) {
    const int ntx = z_tiles_x<R>(kx), full = ntx * ny;
    folded = sizeof(R) == 8 && t >= full;
    row0 = folded ? (t - full) * kZLines : t / ntx;
    k0 = folded ? kx - 1 : (t - row0 * ntx) * kZLines;
  }
  __device__ __forceinline__ int k(int line) const { return folded ? k0 : k0 + line; }
  __device__ __forceinline__ int row(int line) const { return folded ? row0 + line : row0; }
  __device__ __forceinline__ bool live(int line, int kx, int ny) const { return k(line) < kx && row(line) < ny; }
  __device__ __forceinline__ size_t at(int line, int kxp) const { return (size_t)row(line) * kxp + k(line); }
};

// x > 0, in integer arithmetic for FP64 (and for what recip does not flush).
__device__ __forceinline__ bool positive(float x) { return x > 0.0f; }
__device__ __forceinline__ bool positive(double x) { return __double2hiint(x) >= 0x00100000; }

// Sums of products as chains of multiply-adds (FP64 z pass of 128^3: 376 us with products and sums apart, 353).
template <typename R>
__device__ __forceinline__ void apply_symbol(cplx_t<R>& c0, cplx_t<R>& c1, cplx_t<R>& c2, cplx_t<R> d0,
                                             cplx_t<R> d1, cplx_t<R> d2, R dd, const SymParams<R>& sp,
                                             bool mean_mode) {
  R scale = sp.mean_scale;   // a = 0 (the steady Stokes solve): the mean mode has no solution and is dropped
  if (!mean_mode) {          // |d|^2 = 0 only there: decided by index, comparisons are FP64 operations too
    const R den = sp.a + sp.b * dd;
    const R prod = dd * den;
    const R r = positive(prod) ? recip<R>(prod) : R(0);
    const cplx_t<R> div = cfma(d2, c2, cfma(d1, c1, cmul(d0, c0)));
    const R inv_dd = den * r;
    const cplx_t<R> q = cscaler<R>(div, inv_dd);
    c0 = cfms_conj(d0, q, c0);
    c1 = cfms_conj(d1, q, c1);
    c2 = cfms_conj(d2, q, c2);
    scale = sp.inv_ntot * (dd * r);
  }
  c0 = cscaler<R>(c0, scale);
  c1 = cscaler<R>(c1, scale);
  c2 = cscaler<R>(c2, scale);
  if (mean_mode && sp.k0sum != nullptr) {
    c0 = mk((R)(sp.k0sum[0] * sp.k0mul), R(0));
    c1 = mk((R)(sp.k0sum[1] * sp.k0mul), R(0));
    c2 = mk((R)(sp.k0sum[2] * sp.k0mul), R(0));
  }
}

}  // namespace
}  // namespace icm
