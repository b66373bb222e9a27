// Blob-blob coupling matrices M = J(qi) (a - b L)^-1 P S(qj) (Sec. III.A.2) as sums over
// wave vectors, without a transform.
//
// In Fourier space J and S are multiplications by the transform of a stencil, which is a
// product of three 1-D sums of at most four terms, f(k) = sum_n phi_n exp(-2 pi i k n/N),
// and the solve is the symbol P^(k)/(a + b |d|^2).  By Parseval's identity
//   M_ab = (1/(h^3 N)) sum_k conj(J_a) (delta_ab - conj(d_a) d_b / |d|^2) S_b / (a + b|d|^2),
// so a pair of positions costs one pass over the half spectrum (17 operations per
// wave vector and pair, everything in registers) where solving for the three unit forces
// costs three round trips of the 3-D transform, memory passes and launches included.
//
// Bound by FP64 operations (an FP64 FMA issues at 1/64 of the FP32 rate on this chip), in
// both precisions: the sum is formed in FP64 for FP32 simulations too.  16 pairs on 32^3 in
// FP64, the whole call: 3.49 ms with the transforms (48 solves of eight launches), 0.087 ms
// with the sums.
#include <algorithm>

#include "icm_internal.h"
#include "icm_symbol.cuh"

namespace icm {
namespace {

// exp(-2 pi i k / n), k reduced to [0, n).
__device__ __forceinline__ double2 unit_root(int k, int n) {
  double s, c;
  sincospi(-2.0 * (double)k / (double)n, &s, &c);
  return make_double2(c, s);
}

// Table layout (double2 each): per position the x, y, z sums for the two stagger offsets,
// entry [off][k] of axis ax at axis_base(ax) + off * count(ax) + k; x holds nx/2 + 1 wave
// numbers.  The symbol table holds d_a by wave number and |d_a|^2 after it.
struct CoupleDims {
  int n[3];
  int count[3];
  __host__ __device__ int base(int ax) const { return ax == 0 ? 0 : 2 * (count[0] + (ax == 2 ? count[1] : 0)); }
  __host__ __device__ int per_position() const { return 2 * (count[0] + count[1] + count[2]); }
  __host__ __device__ int symbols() const { return count[0] + count[1] + count[2]; }
  __host__ __device__ int symbol_base(int ax) const { return ax == 0 ? 0 : count[0] + (ax == 2 ? count[1] : 0); }
};

// Blocks 0 .. 2 npair - 1: the stencil sums of one position, qi first (the roots of one axis at a time
// in shared memory).  Block 2 npair: the symbols.
__global__ void __launch_bounds__(128) k_couple_tables(CoupleDims d, double h, int kernel, int npair,
                                                       const double* __restrict__ qi, const double* __restrict__ qj,
                                                       double2* __restrict__ tab,
                                                       double2* __restrict__ sym, double* __restrict__ symdd) {
  __shared__ double2 roots[kMaxSide];
  const int p = blockIdx.x;
  if (p == 2 * npair) {
    for (int ax = 0; ax < 3; ++ax)
      for (int k = threadIdx.x; k < d.count[ax]; k += blockDim.x) {
        double s, c, sf;
        sincospi((double)k / (double)d.n[ax], &s, &c);
        sf = sinpi(2.0 * (double)k / (double)d.n[ax]);
        sym[d.symbol_base(ax) + k] = make_double2(-2.0 * s * s, sf);   // exp(i theta) - 1: unit spacing
        symdd[d.symbol_base(ax) + k] = 4.0 * s * s;
      }
    return;
  }
  const double* q = p < npair ? qi + 3 * p : qj + 3 * (p - npair);
  double2* out = tab + (size_t)p * d.per_position();
  for (int ax = 0; ax < 3; ++ax) {
    const int n = d.n[ax];
    __syncthreads();
    for (int k = threadIdx.x; k < n; k += blockDim.x) roots[k] = unit_root(k, n);
    __syncthreads();
    for (int off = 0; off < 2; ++off) {
      const double s = q[ax] / h - (off ? 0.5 : 0.0);
      const double anchor = kernel == 3 ? Peskin<double, 3>::anchor(s) : Peskin<double, 4>::anchor(s);
      const double frac = s - anchor;
      double w[4];
#pragma unroll
      for (int a = 0; a < 4; ++a)
        w[a] = a >= kernel ? 0.0
                           : (kernel == 3 ? Peskin<double, 3>::phi(frac + (1 - a)) : Peskin<double, 4>::phi(frac + (1 - a)));
      int first = (int)((long long)anchor - 1) % n;
      if (first < 0) first += n;
      for (int k = threadIdx.x; k < d.count[ax]; k += blockDim.x) {
        double2 f = make_double2(0.0, 0.0);
        int m = (int)(((long long)k * first) % n);   // k node mod n, advanced by k per node
        for (int a = 0; a < kernel; ++a) {
          f.x = fma(w[a], roots[m].x, f.x);
          f.y = fma(w[a], roots[m].y, f.y);
          m += k;
          if (m >= n) m -= n;
        }
        out[d.base(ax) + off * d.count[ax] + k] = f;
      }
    }
  }
}

// A thread takes one (ky, kz) column and one segment of kx.  With u = conj(J_x) S_x products of the x
// sums and c = 1/(|d|^2 (a + b|d|^2)), every entry of M is the real part of a y-z factor times one of five
// sums over kx, the same for every pair of components that shares their stagger offsets:
//   s0 = sum c u00,  s1 = sum c u11,  s2 = sum c |d_x|^2 u11,  s3 = sum c conj(d_x) u01,  s4 = sum c d_x u10,
// (u_ij: J of offset i, S of offset j), as the diagonal's 1/(a + b|d|^2) - c |d_a|^2 is c times the other
// two |d|^2.  So a wave vector costs ten multiply-adds and one reciprocal, 17 FP64 operations, where
// forming J, S and their nine products cost 96; the y-z factors are formed once per column and segment.
// Segments of at most 64 wave numbers spread one pair over the whole device; with 16, where the y-z factors
// weigh as much as the sums, one pair on 64^3 and 128^3 takes 85 and 135 us instead of 97 and 121, 64
// pairs 554 and 3476 instead of 400 and 2552.  One pair
// in an FP32 simulation, the whole call: 128^3 120 us, 256^3 409 us; with one sum per entry on at
// most 64 blocks 507 and 3431, with three FP32 solves 305 and 1388.
constexpr int kCoupleThreads = 128;
constexpr int kCoupleSegment = 64;      // wave numbers
constexpr int kCoupleBlocks = 1216;     // blocks per pair at most: eight per SM
struct CoupleShape {
  int nseg, seglen, colblocks;
  __host__ __device__ int blocks() const { return nseg * colblocks; }
};
CoupleShape couple_shape(const CoupleDims& d) {
  const int cols = d.count[1] * d.count[2];
  CoupleShape s;
  s.nseg = (d.count[0] + kCoupleSegment - 1) / kCoupleSegment;
  s.seglen = (d.count[0] + s.nseg - 1) / s.nseg;
  const int full = (cols + kCoupleThreads - 1) / kCoupleThreads;
  const int rounds = (full * s.nseg + kCoupleBlocks - 1) / kCoupleBlocks;   // columns per thread
  s.colblocks = (full + rounds - 1) / rounds;
  return s;
}

__device__ __forceinline__ double2 conj_mul(double2 a, double2 b) {   // conj(a) b
  return make_double2(fma(a.y, b.y, a.x * b.x), fma(a.x, b.y, -a.y * b.x));
}
__device__ __forceinline__ double re_mul(double2 a, double2 b) { return fma(a.x, b.x, -a.y * b.y); }

struct CoupleX {
  double2 u00, u11, u11dd, u01, u10;
  double dd, pad;
};

__global__ void __launch_bounds__(kCoupleThreads) k_couple_modes(CoupleDims d, CoupleShape sh, int npair, double a,
                                                                 double b, const double2* __restrict__ tab,
                                                                 const double2* __restrict__ sym,
                                                                 const double* __restrict__ symdd,
                                                                 double* __restrict__ partial) {
  __shared__ CoupleX xs[kCoupleSegment];
  __shared__ double red[kCoupleThreads / 32][9];
  const int pair = blockIdx.y, kx = d.count[0], tid = threadIdx.x;
  const int seg = blockIdx.x % sh.nseg, cb = blockIdx.x / sh.nseg;
  const int k0 = seg * sh.seglen, len = min(sh.seglen, kx - k0);
  const double2* ti = tab + (size_t)pair * d.per_position();
  const double2* tj = tab + (size_t)(npair + pair) * d.per_position();
  for (int i = tid; i < len; i += kCoupleThreads) {
    const int k = k0 + i;
    // every wave vector but those of kx = 0 and the Nyquist plane stands for its conjugate too
    const double w = k == 0 || 2 * k == d.n[0] ? 1.0 : 2.0, dd = symdd[k];
    const double2 i0 = make_double2(w * ti[k].x, w * ti[k].y), i1 = make_double2(w * ti[kx + k].x, w * ti[kx + k].y);
    const double2 j0 = tj[k], j1 = tj[kx + k], dx = sym[k];
    CoupleX x;
    x.u00 = conj_mul(i0, j0);
    x.u11 = conj_mul(i1, j1);
    x.u11dd = make_double2(dd * x.u11.x, dd * x.u11.y);
    x.u01 = conj_mul(cmul(dx, i0), j1);
    x.u10 = conj_mul(i1, cmul(dx, j0));
    x.dd = dd;
    xs[i] = x;
  }
  __syncthreads();
  double m[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) m[i] = 0.0;
  const int cols = d.count[1] * d.count[2], cy = d.count[1], cz = d.count[2];
  for (int c = cb * kCoupleThreads + tid; c < cols; c += sh.colblocks * kCoupleThreads) {
    const int kz = c / cy, ky = c - kz * cy;
    const double ddy = symdd[d.symbol_base(1) + ky], ddz = symdd[d.symbol_base(2) + kz], ddyz = ddy + ddz;
    double2 s0 = make_double2(0.0, 0.0), s1 = s0, s2 = s0, s3 = s0, s4 = s0;
#pragma unroll 4
    for (int k = 0; k < len; ++k) {
      const CoupleX& x = xs[k];
      const double dd = x.dd + ddyz, prod = dd * fma(b, dd, a);
      const double w = positive(prod) ? recip<double>(prod) : 0.0;
      s0 = cfmar<double>(w, x.u00, s0);
      s1 = cfmar<double>(w, x.u11, s1);
      s2 = cfmar<double>(w, x.u11dd, s2);
      s3 = cfmar<double>(w, x.u01, s3);
      s4 = cfmar<double>(w, x.u10, s4);
    }
    const double2* iy = ti + d.base(1) + ky;
    const double2* iz = ti + d.base(2) + kz;
    const double2* jy = tj + d.base(1) + ky;
    const double2* jz = tj + d.base(2) + kz;
    const double2 dy = sym[d.symbol_base(1) + ky], dz = sym[d.symbol_base(2) + kz];
    // y-z factors of the components x, y, z (a component's own axis has offset 0)
    const double2 Jx = cmul(iy[cy], iz[cz]), Jy = cmul(iy[0], iz[cz]), Jz = cmul(iy[cy], iz[0]);
    const double2 Sx = cmul(jy[cy], jz[cz]), Sy = cmul(jy[0], jz[cz]), Sz = cmul(jy[cy], jz[0]);
    const double2 xx = conj_mul(Jx, Sx), yy = conj_mul(Jy, Sy), zz = conj_mul(Jz, Sz);
    const double2 dJy = cmul(dy, Jy), dJz = cmul(dz, Jz), dSy = cmul(dy, Sy), dSz = cmul(dz, Sz);
    m[0] += ddyz * re_mul(xx, s0);
    m[1] -= re_mul(conj_mul(Jx, dSy), s3);
    m[2] -= re_mul(conj_mul(Jx, dSz), s3);
    m[3] -= re_mul(conj_mul(dJy, Sx), s4);
    m[4] += re_mul(yy, cfmar<double>(ddz, s1, s2));
    m[5] -= re_mul(conj_mul(dJy, dSz), s1);
    m[6] -= re_mul(conj_mul(dJz, Sx), s4);
    m[7] -= re_mul(conj_mul(dJz, dSy), s1);
    m[8] += re_mul(zz, cfmar<double>(ddy, s1, s2));
    // the mean mode (weight 0 above) is not projected, and dropped at a = 0
    if (c == 0 && k0 == 0 && a > 0.0) {
      m[0] += re_mul(xx, xs[0].u00) / a;
      m[4] += re_mul(yy, xs[0].u11) / a;
      m[8] += re_mul(zz, xs[0].u11) / a;
    }
  }
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    double x = m[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((tid & 31) == 0) red[tid >> 5][i] = x;
  }
  __syncthreads();
  if (tid < 9) {
    double x = 0.0;
    for (int w = 0; w < kCoupleThreads / 32; ++w) x += red[w][tid];
    partial[((size_t)pair * gridDim.x + blockIdx.x) * 9 + tid] = x;
  }
}

// One block per pair, one warp per entry.
__global__ void __launch_bounds__(9 * 32) k_couple_final(const double* __restrict__ partial, int nblk, double scale,
                                                         double* __restrict__ out) {
  const int e = threadIdx.x >> 5, lane = threadIdx.x & 31, pair = blockIdx.x;
  double x = 0.0;
  for (int b = lane; b < nblk; b += 32) x += partial[((size_t)pair * nblk + b) * 9 + e];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  if (lane == 0) out[9 * pair + e] = x * scale;
}

template <typename R>
__global__ void k_reciprocals(int n, const double* __restrict__ x, double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = (double)recip<R>((R)x[i]);
}

CoupleDims couple_dims(int nx, int ny, int nz) { return CoupleDims{{nx, ny, nz}, {nx / 2 + 1, ny, nz}}; }

}  // namespace

void symbol_reciprocals(int precision, int n, const double* x, double* out, cudaStream_t st) {
  const unsigned blocks = (unsigned)((n + 127) / 128);
  if (precision == 32)
    k_reciprocals<float><<<blocks, 128, 0, st>>>(n, x, out);
  else
    k_reciprocals<double><<<blocks, 128, 0, st>>>(n, x, out);
}

size_t couple_scratch_doubles(int nx, int ny, int nz, int npair) {
  const CoupleDims d = couple_dims(nx, ny, nz);
  return 2 * (size_t)(2 * npair) * d.per_position() + 3 * (size_t)d.symbols() + 9 * (size_t)npair * couple_shape(d).blocks();
}

void couple_pairs(int nx, int ny, int nz, double h, int kernel, int npair, const double* qi_dev, const double* qj_dev,
                  double a, double b, double* scratch, double* out_dev, cudaStream_t st) {
  const CoupleDims d = couple_dims(nx, ny, nz);
  const CoupleShape sh = couple_shape(d);
  const int nblk = sh.blocks();
  double2* tab = reinterpret_cast<double2*>(scratch);
  double2* sym = tab + (size_t)(2 * npair) * d.per_position();
  double* symdd = reinterpret_cast<double*>(sym + d.symbols());
  double* partial = symdd + d.symbols();
  k_couple_tables<<<2 * npair + 1, 128, 0, st>>>(d, h, kernel, npair, qi_dev, qj_dev, tab, sym, symdd);
  k_couple_modes<<<dim3(nblk, npair), kCoupleThreads, 0, st>>>(d, sh, npair, a, unit_b(b, h), tab, sym,
                                                                symdd, partial);
  const double scale = 1.0 / ((double)nx * ny * nz * h * h * h);
  k_couple_final<<<npair, 9 * 32, 0, st>>>(partial, nblk, scale, out_dev);
}

}  // namespace icm
