// Blob-blob coupling matrices M = J(qi) (a - b L)^-1 P S(qj) (Sec. III.A.2) as sums over
// wave vectors, without a transform.
//
// In Fourier space J and S are multiplications by the transform of a stencil, which is a
// product of three 1-D sums of at most four terms, f(k) = sum_n phi_n exp(-2 pi i k n/N),
// and the solve is the symbol P^(k)/(a + b |d|^2).  By Parseval's identity
//   M_ab = (1/(h^3 N)) sum_k conj(J_a) (delta_ab - conj(d_a) d_b / |d|^2) S_b / (a + b|d|^2),
// so a pair of positions costs one pass over the half spectrum (about 100 operations per
// wave vector and pair, everything in registers) where solving for the three unit forces
// costs three round trips of the 3-D transform, memory passes and launches included.
//
// Bound by FP64 operations (an FP64 FMA issues at 1/64 of the FP32 rate on this chip), in
// both precisions: the sum is formed in FP64 for FP32 simulations too.  16 pairs on 32^3 in
// FP64, the whole call: 3.49 ms with the transforms (48 solves of eight launches), 0.148 ms
// with the sums.
#include <algorithm>

#include "icm_internal.h"

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
        sym[d.symbol_base(ax) + k] = make_double2(-2.0 * s * s / h, sf / h);   // (exp(i theta) - 1)/h
        symdd[d.symbol_base(ax) + k] = 4.0 * s * s / (h * h);
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

// A thread takes one (ky, kz) column and sums over kx: the y-z products, the symbols and
// the nine sums stay in registers, and the x sums of the pair (the same for every thread
// at a time) are read as broadcasts from shared memory.  128 columns per block keep the
// FP64 pipe of an SM busy with one block; partial[pair][block][9] is summed by
// k_couple_final.
constexpr int kCoupleThreads = 128;
__global__ void __launch_bounds__(kCoupleThreads) k_couple_modes(CoupleDims d, int npair, double a, double b,
                                                                 const double2* __restrict__ tab,
                                                                 const double2* __restrict__ sym,
                                                                 const double* __restrict__ symdd,
                                                                 double* __restrict__ partial) {
  extern __shared__ __align__(16) double2 xs[];   // J off 0, J off 1, S off 0, S off 1, d_x, (|d_x|^2, weight)
  __shared__ double red[kCoupleThreads / 32][9];
  const int pair = blockIdx.y, kx = d.count[0], tid = threadIdx.x;
  const double2* ti = tab + (size_t)pair * d.per_position();
  const double2* tj = tab + (size_t)(npair + pair) * d.per_position();
  for (int k = tid; k < kx; k += kCoupleThreads) {
    xs[k] = ti[k];
    xs[kx + k] = ti[kx + k];
    xs[2 * kx + k] = tj[k];
    xs[3 * kx + k] = tj[kx + k];
    xs[4 * kx + k] = sym[k];
    // every wave vector but those of kx = 0 and the Nyquist plane stands for its conjugate too
    xs[5 * kx + k] = make_double2(symdd[k], k == 0 || 2 * k == d.n[0] ? 1.0 : 2.0);
  }
  __syncthreads();
  double m[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) m[i] = 0.0;
  const long long cols = (long long)d.count[1] * d.count[2];
  for (long long c = (long long)blockIdx.x * kCoupleThreads + tid; c < cols; c += (long long)gridDim.x * kCoupleThreads) {
    const int ky = (int)(c % d.count[1]), kz = (int)(c / d.count[1]);
    const double2* iy = ti + d.base(1) + ky;
    const double2* iz = ti + d.base(2) + kz;
    const double2* jy = tj + d.base(1) + ky;
    const double2* jz = tj + d.base(2) + kz;
    const double2 dy = sym[d.symbol_base(1) + ky], dz = sym[d.symbol_base(2) + kz];
    const double ddyz = symdd[d.symbol_base(1) + ky] + symdd[d.symbol_base(2) + kz];
    const int cy = d.count[1], cz = d.count[2];
    // y-z factors of the components x, y, z (a component's own axis has offset 0)
    const double2 Jx = cmul(iy[cy], iz[cz]), Jy = cmul(iy[0], iz[cz]), Jz = cmul(iy[cy], iz[0]);
    const double2 Sx = cmul(jy[cy], jz[cz]), Sy = cmul(jy[0], jz[cz]), Sz = cmul(jy[cy], jz[0]);
#pragma unroll 2
    for (int k = 0; k < kx; ++k) {
      const double2 dx = xs[4 * kx + k], wd = xs[5 * kx + k];
      const double2 i0 = xs[k], i1 = xs[kx + k], j0 = xs[2 * kx + k], j1 = xs[3 * kx + k];
      const double dd = wd.x + ddyz;
      const double den = a + b * dd;
      // c1 = 1/(a + b|d|^2), c2 = c1/|d|^2; the mean mode is not projected, and dropped at a = 0
      const double prod = dd * den;
      const double r = wd.y / (prod > 0.0 ? prod : 1.0);
      const double c1 = prod > 0.0 ? dd * r : (dd == 0.0 && a > 0.0 ? wd.y / a : 0.0);
      const double c2 = prod > 0.0 ? r : 0.0;
      const double2 J[3] = {cmul(i0, Jx), cmul(i1, Jy), cmul(i1, Jz)};
      const double2 S[3] = {cmul(j0, Sx), cmul(j1, Sy), cmul(j1, Sz)};
      const double2 dv[3] = {dx, dy, dz};
      double2 A[3], B[3];   // d_a J_a and c2 d_b S_b
#pragma unroll
      for (int t = 0; t < 3; ++t) {
        A[t] = cmul(dv[t], J[t]);
        B[t] = cmul(dv[t], S[t]);
        B[t] = make_double2(c2 * B[t].x, c2 * B[t].y);
        m[4 * t] = fma(c1, fma(J[t].x, S[t].x, J[t].y * S[t].y), m[4 * t]);   // Re conj(J) S
      }
#pragma unroll
      for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int s = 0; s < 3; ++s) m[3 * p + s] = fma(-A[p].x, B[s].x, fma(-A[p].y, B[s].y, m[3 * p + s]));
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

__global__ void k_couple_final(const double* __restrict__ partial, int nblk, int npair, double scale,
                               double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 9 * npair) return;
  const int pair = i / 9, e = i - 9 * pair;
  double x = 0.0;
  for (int b = 0; b < nblk; ++b) x += partial[((size_t)pair * nblk + b) * 9 + e];
  out[i] = x * scale;
}

CoupleDims couple_dims(int nx, int ny, int nz) { return CoupleDims{{nx, ny, nz}, {nx / 2 + 1, ny, nz}}; }

// Blocks per pair: one per 128 columns, at most 64 (the pairs fill the device; a grid of one
// pair still spreads over 64 SMs, which bounds the final sum's serial chain).
int couple_blocks(const CoupleDims& d) {
  const long long cols = (long long)d.count[1] * d.count[2];
  return (int)std::min<long long>((cols + kCoupleThreads - 1) / kCoupleThreads, 64);
}

}  // namespace

size_t couple_scratch_doubles(int nx, int ny, int nz, int npair) {
  const CoupleDims d = couple_dims(nx, ny, nz);
  return 2 * (size_t)(2 * npair) * d.per_position() + 3 * (size_t)d.symbols() + 9 * (size_t)npair * couple_blocks(d);
}

void couple_pairs(int nx, int ny, int nz, double h, int kernel, int npair, const double* qi_dev, const double* qj_dev,
                  double a, double b, double* scratch, double* out_dev, cudaStream_t st) {
  const CoupleDims d = couple_dims(nx, ny, nz);
  const int nblk = couple_blocks(d);
  double2* tab = reinterpret_cast<double2*>(scratch);
  double2* sym = tab + (size_t)(2 * npair) * d.per_position();
  double* symdd = reinterpret_cast<double*>(sym + d.symbols());
  double* partial = symdd + d.symbols();
  k_couple_tables<<<2 * npair + 1, 128, 0, st>>>(d, h, kernel, npair, qi_dev, qj_dev, tab, sym, symdd);
  k_couple_modes<<<dim3(nblk, npair), kCoupleThreads, 6 * (size_t)d.count[0] * sizeof(double2), st>>>(
      d, npair, a, b, tab, sym, symdd, partial);
  const double scale = 1.0 / ((double)nx * ny * nz * h * h * h);
  k_couple_final<<<(9 * npair + 127) / 128, 128, 0, st>>>(partial, nblk, npair, scale, out_dev);
}

}  // namespace icm
