// Device-side building blocks shared by the ICM kernels (sm_103a).
//
// Complex helpers, the Philox4x32-10 generator (Salmon et al., SC'11), the
// Box-Muller transform, and the Peskin 3-/4-point kernel functions
// (arXiv:1212.6427, Sec. III.A.1, Eq. JS_invariance).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace icm {

template <typename R> struct Cplx;
template <> struct Cplx<float> { using T = float2; };
template <> struct Cplx<double> { using T = double2; };
template <typename R> using cplx_t = typename Cplx<R>::T;

__host__ __device__ inline float2 mk(float a, float b) { return make_float2(a, b); }
__host__ __device__ inline double2 mk(double a, double b) { return make_double2(a, b); }
template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return mk(a.x + b.x, a.y + b.y); }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { return mk(a.x - b.x, a.y - b.y); }
// z + r p, r real
template <typename R> __device__ __forceinline__ cplx_t<R> cfmar(R r, cplx_t<R> p, cplx_t<R> z) {
  return mk(fma(r, p.x, z.x), fma(r, p.y, z.y));
}
template <typename R> __device__ __forceinline__ cplx_t<R> cscaler(cplx_t<R> a, R s) { return mk(a.x * s, a.y * s); }
#if defined(__CUDA_ARCH__)
// FP32: both components in one instruction, with the same roundings (a - b as the exact product b (-1)
// added to a).  The FP32 passes have few warps and wait for what they issue: y inverse and x forward pass of
// 512 x 384 x 256 270 and 233 us component by component, 231 and 213 packed.
template <> __device__ __forceinline__ float2 cadd<float2>(float2 a, float2 b) { return __fadd2_rn(a, b); }
template <> __device__ __forceinline__ float2 csub<float2>(float2 a, float2 b) {
  return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a);
}
template <> __device__ __forceinline__ float2 cfmar<float>(float r, float2 p, float2 z) {
  return __ffma2_rn(make_float2(r, r), p, z);
}
template <> __device__ __forceinline__ float2 cscaler<float>(float2 a, float s) {
  return __fmul2_rn(a, make_float2(s, s));
}
#endif
template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
  return mk(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename C> __device__ __forceinline__ C cfma(C a, C b, C c) {   // c + a b
  return mk(fma(-a.y, b.y, fma(a.x, b.x, c.x)), fma(a.y, b.x, fma(a.x, b.y, c.y)));
}
template <typename C> __device__ __forceinline__ C cfms_conj(C a, C b, C c) {   // c - conj(a) b
  return mk(fma(-a.y, b.y, fma(-a.x, b.x, c.x)), fma(a.y, b.x, fma(-a.x, b.y, c.y)));
}
template <typename C> __device__ __forceinline__ C cconj(C a) { return mk(a.x, -a.y); }
// multiply by -i and +i
template <typename C> __device__ __forceinline__ C cmul_mi(C a) { return mk(a.y, -a.x); }
template <typename C> __device__ __forceinline__ C cmul_pi(C a) { return mk(-a.y, a.x); }

// Division of n < 2^31 by a fixed divisor (Granlund and Montgomery, 1994: the upper half of
// a 33-bit multiply, then a shift), for kernels that split flat indices by run-time sides.
struct FastDiv {
  uint32_t d = 1, mul = 1, sh = 0;
  FastDiv() = default;
  explicit FastDiv(uint32_t d_) : d(d_) {
    while ((1ull << sh) < d) ++sh;
    mul = (uint32_t)((((1ull << sh) - d) << 32) / d + 1);
  }
  __device__ __forceinline__ uint32_t div(uint32_t n) const { return (__umulhi(n, mul) + n) >> sh; }
};

// ---------------------------------------------------------------------------
// Philox4x32-10.  Round: words 0 and 2 are multiplied (full 64-bit products) by
// two constants; the high halves are xored with words 1, 3 and the key; the key
// is bumped by two Weyl constants between rounds.
// ---------------------------------------------------------------------------
struct u32x4 { uint32_t x, y, z, w; };

__host__ __device__ __forceinline__ u32x4 philox4x32_10(u32x4 c, uint32_t k0, uint32_t k1) {
  const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
  const uint32_t W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) { k0 += W0; k1 += W1; }
    // one widening 32 x 32 -> 64-bit multiply per word gives both halves
    const uint64_t p0 = (uint64_t)M0 * c.x, p1 = (uint64_t)M1 * c.z;
    const uint32_t hi0 = (uint32_t)(p0 >> 32), lo0 = (uint32_t)p0;
    const uint32_t hi1 = (uint32_t)(p1 >> 32), lo1 = (uint32_t)p1;
    c = u32x4{hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0};
  }
  return c;
}

// The ten round keys of one key (round r uses the key bumped r times), formed once so
// that a kernel drawing many numbers reads them as constants instead of bumping the
// key in every call.
struct PhiloxRoundKeys { uint32_t k0[10], k1[10]; };
inline PhiloxRoundKeys philox_round_keys(uint32_t k0, uint32_t k1) {
  PhiloxRoundKeys rk;
  for (int r = 0; r < 10; ++r) {
    rk.k0[r] = k0;
    rk.k1[r] = k1;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return rk;
}
__device__ __forceinline__ u32x4 philox4x32_10(u32x4 c, const PhiloxRoundKeys& rk) {
  const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint64_t p0 = (uint64_t)M0 * c.x, p1 = (uint64_t)M1 * c.z;
    const uint32_t hi0 = (uint32_t)(p0 >> 32), lo0 = (uint32_t)p0;
    const uint32_t hi1 = (uint32_t)(p1 >> 32), lo1 = (uint32_t)p1;
    c = u32x4{hi1 ^ c.y ^ rk.k0[r], lo1, hi0 ^ c.w ^ rk.k1[r], lo0};
  }
  return c;
}

// Box-Muller: two 32-bit words -> two unit normals (cos branch, sin branch).
// u = (x + 1/2) 2^-32 in (0, 1).  The FP64 form is in icm_grid.cu (its tables live there).
template <typename R> struct BoxMuller;
template <> struct BoxMuller<float> {
  __device__ __forceinline__ static void apply(uint32_t a, uint32_t b, float& z0, float& z1) {
    // u = (x + 1/2) 2^-32 with one rounding: exact for x < 2^23 (u < 2^-9, the tail
    // of the normal), relative error <= 2^-24 above
    const float u1 = fmaf(__uint2float_rn(a), 2.3283064365386963e-10f, 1.16415321826934814e-10f);
    const float u2 = fmaf(__uint2float_rn(b), 2.3283064365386963e-10f, 1.16415321826934814e-10f);
    // -2 ln u1 = -2 ln(2) log2(u1); the hardware log2 and reciprocal square root are
    // accurate to ~2^-22 relative, far inside the FP32 path's tolerance.  u1 may round
    // to 1, where the radius is 0: the floor keeps x * rsqrt(x) finite.
    // Neither argument is subnormal, so the .ftz forms give the same values without the
    // scaling around the others.
    float l, y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(u1));
    const float x = fmaxf(-1.38629436111989061f * l, 1e-30f);
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    const float rad = x * y;
    float s, c;
    __sincosf(6.28318530717958648f * u2, &s, &c);
    z0 = rad * c;
    z1 = rad * s;
  }
};

// The key as two words (the round keys formed in every call).
struct PhiloxKey { uint32_t k0, k1; };
__device__ __forceinline__ u32x4 philox4x32_10(u32x4 c, PhiloxKey k) { return philox4x32_10(c, k.k0, k.k1); }

// ---------------------------------------------------------------------------
// Peskin kernel functions of r in grid units.
// 3-point: (1 + sqrt(1 - 3 r^2))/3 for |r| <= 1/2, (5 - 3|r| - sqrt(1 - 3(1-|r|)^2))/6
//          for 1/2 <= |r| <= 3/2.  4-point: (3 - 2|r| + sqrt(1 + 4|r| - 4 r^2))/8 for
//          |r| <= 1, (5 - 2|r| - sqrt(-7 + 12|r| - 4 r^2))/8 for 1 <= |r| <= 2.
// ---------------------------------------------------------------------------
template <typename R> __device__ __forceinline__ R rsqrt0(R x) { return sqrt(x > R(0) ? x : R(0)); }

template <typename R, int K> struct Peskin;
template <typename R> struct Peskin<R, 3> {
  static constexpr int W = 3;
  __device__ __forceinline__ static R phi(R r) {
    r = fabs(r);
    if (r <= R(0.5)) return (R(1) + rsqrt0<R>(R(1) - R(3) * r * r)) / R(3);
    if (r <= R(1.5)) {
      const R t = R(1) - r;
      return (R(5) - R(3) * r - rsqrt0<R>(R(1) - R(3) * t * t)) / R(6);
    }
    return R(0);
  }
  // derivative: -r/sqrt(1-3r^2) inside, sign(r)(-3 - 3t/sqrt(1-3t^2))/6, t = 1-|r|, outside
  __device__ __forceinline__ static R dphi(R r) {
    const R a = fabs(r);
    if (a <= R(0.5)) return -r / sqrt(R(1) - R(3) * r * r);
    if (a <= R(1.5)) {
      const R t = R(1) - a;
      const R d = (R(-3) - R(3) * t / sqrt(R(1) - R(3) * t * t)) / R(6);   // d phi / d|r|
      return r < R(0) ? -d : d;
    }
    return R(0);
  }
  // first node of the support: round-half-up(s) - 1
  __device__ __forceinline__ static long long first(double s) { return (long long)floor(s + 0.5) - 1; }
  // the cell that fixes the support (its node 'first' + 1), as a double: round-half-up(s)
  __device__ __forceinline__ static double anchor(double s) { return floor(s + 0.5); }
};
template <typename R> struct Peskin<R, 4> {
  static constexpr int W = 4;
  __device__ __forceinline__ static R phi(R r) {
    r = fabs(r);
    if (r <= R(1)) return (R(3) - R(2) * r + rsqrt0<R>(R(1) + R(4) * r - R(4) * r * r)) / R(8);
    if (r <= R(2)) return (R(5) - R(2) * r - rsqrt0<R>(R(-7) + R(12) * r - R(4) * r * r)) / R(8);
    return R(0);
  }
  // derivative: sign(r)(-2 + (2-4|r|)/sqrt(1+4|r|-4r^2))/8 inside,
  // sign(r)(-2 - (6-4|r|)/sqrt(-7+12|r|-4r^2))/8 outside
  __device__ __forceinline__ static R dphi(R r) {
    const R a = fabs(r);
    R d;   // d phi / d|r|
    if (a <= R(1))
      d = (R(-2) + (R(2) - R(4) * a) / sqrt(R(1) + R(4) * a - R(4) * a * a)) / R(8);
    else if (a <= R(2))
      d = (R(-2) - (R(6) - R(4) * a) / sqrt(R(-7) + R(12) * a - R(4) * a * a)) / R(8);
    else
      return R(0);
    return r < R(0) ? -d : d;
  }
  __device__ __forceinline__ static long long first(double s) { return (long long)floor(s) - 1; }
  __device__ __forceinline__ static double anchor(double s) { return floor(s); }
};

// Status bits the device raises (read back by icm_sync).
enum : int { DEV_ERR_CFL = 1, DEV_ERR_NONFINITE = 2, DEV_ERR_TIMEOUT = 4, DEV_ERR_INDEX = 8 };

// Index checks of the checked build (compiled with -DICM_INDEX_CHECKS=1, the library
// libicm_checked.so): true when 0 <= i < n; otherwise the check raises DEV_ERR_INDEX in
// *err (if err is set) and returns false, and the caller skips the access.  It never
// traps.  In the ordinary build it is always true and compiles away.
#ifndef ICM_INDEX_CHECKS
#define ICM_INDEX_CHECKS 0
#endif
__device__ __forceinline__ bool index_ok(long long i, long long n, int* err) {
#if ICM_INDEX_CHECKS
  if (i >= 0 && i < n) return true;
  if (err != nullptr) atomicOr(err, DEV_ERR_INDEX);
  return false;
#else
  (void)i;
  (void)n;
  (void)err;
  return true;
#endif
}

}  // namespace icm
