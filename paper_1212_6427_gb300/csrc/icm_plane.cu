// The x and y transforms of whole z planes in one pass, any side 2^a 3^b.
//
// A block holds one z plane of one velocity component in shared memory: forward it loads
// the plane, adds the blobs' spread, transforms along x and y and writes the half spectrum;
// inverse it loads the half spectrum, transforms back, stores (or adds) the plane and gathers
// at the blobs.  The half spectrum between the x and the y transform never leaves the SM, which
// saves a write and a read of the spectrum, a launch and its ramp per direction against
// separate passes.
//
// Layout in shared memory, in place throughout: line l holds the real rows 2l and 2l + 1 as one
// complex row of nx; after the x transform, Hermitian symmetry splits line l in place into
// the two half spectra, wave number k of row 2l at slot k and of row 2l + 1 at slot nx - k
// (0 < k < nx/2).  The real columns k = 0 and nx/2 travel as one complex column of their own
// (col0), so a plane takes exactly nx/2 column transforms.  Lines are an odd number of
// complex values apart and x items run along lines, y items along columns: no stage has
// bank conflicts.  The x transform takes its input in digit-reversed order (a free permutation
// while the plane is loaded) and leaves natural order, the y transform the other way
// round, as the z pass expects.
//
// Transforms are chains of in-place register butterflies of radix 2 to 16 whose strides come
// from the axis plan at run time (divisions by multiplication), so one kernel serves every
// side; two factors do for most.
#include <algorithm>

#include "icm.h"
#include "icm_internal.h"
#include "icm_fft_reg.cuh"
#include "icm_rows.cuh"
#include "icm_symbol.cuh"



namespace icm {
namespace {

constexpr int kMaxFactors = 4;
constexpr int kPlaneList = 2048;   // blobs of a plane served at a time

struct StageAxis {
  int n, ns;
  int M[kMaxFactors], rad[kMaxFactors];   // stage s: blocks of M[s] (M[0] = n), radix rad[s]
  FastDiv dmr[kMaxFactors];               // division by M / rad
  const void* tw;
  const int* pof;                         // storage position of an index
};

struct PlaneArgs {
  StageAxis x, y;
  int nz, kx, kxp, nl, ls, ncol;
  FastDiv dnl, dncol;
  long long ncell;
};

// One in-place stage along a line or column: elements at p(r), r = 0 .. RAD - 1, with stage
// twiddles tw[r tstep].  DIT multiplies before the DFT, DIF after it; INV is the exact
// (unnormalised) inverse.
template <typename R, int RAD, bool DIT, bool INV>
__device__ __forceinline__ void butterfly(cplx_t<R> (&a)[RAD], const cplx_t<R>* __restrict__ tw, int tstep, bool twiddle) {
  const auto rotate = [&]() {
    if (twiddle) {
#pragma unroll
      for (int r = 1; r < RAD; ++r) {
        const cplx_t<R> w = tw[r * tstep];
        a[r] = cmul(a[r], INV ? cconj(w) : w);
      }
    }
  };
  if (DIT) rotate();
  if (INV)
    sdft_inv<R, RAD>(a);
  else
    SDft<R, RAD>::run(a);
  if (!DIT) rotate();
}

// Calls F<RAD>() for the run-time radix (uniform over the block).
#define ICM_RADIX_SWITCH(rad, CALL) \
  switch (rad) {                    \
    case 2: CALL(2); break;         \
    case 3: CALL(3); break;         \
    case 4: CALL(4); break;         \
    case 6: CALL(6); break;         \
    case 8: CALL(8); break;         \
    case 9: CALL(9); break;         \
    case 12: CALL(12); break;       \
    default: CALL(16); break;       \
  }

template <typename R, int RAD, bool INV, int NT>
__device__ __forceinline__ void x_stage(cplx_t<R>* __restrict__ buf, const PlaneArgs& A, int s,
                                        const cplx_t<R>* __restrict__ tw, int tid) {
  using C = cplx_t<R>;
  const int M = A.x.M[s], mr = M / RAD, tws = A.x.n / M;
  const int items = A.nl * (A.x.n / RAD);
  for (int it = tid; it < items; it += NT) {
    const int bf = A.dnl.div(it), line = it - bf * A.nl;
    const int blk = A.x.dmr[s].div(bf), n1 = bf - blk * mr;
    C* p = buf + line * A.ls + blk * M + n1;
    C a[RAD];
#pragma unroll
    for (int r = 0; r < RAD; ++r) a[r] = p[r * mr];
    butterfly<R, RAD, !INV, INV>(a, tw, n1 * tws, mr > 1);   // forward DIT, inverse DIF
#pragma unroll
    for (int r = 0; r < RAD; ++r) p[r * mr] = a[r];
  }
}

// Slot of element y of column c: column 0 in col0 (offset c0 from buf), others in the lines.
struct ColumnSlots {
  int a0, a1, step;   // elements y0 + mr r: r even from a0, r odd from a1, `step` per two
  __device__ __forceinline__ ColumnSlots(const PlaneArgs& A, int col, int y0, int mr) {
    const int y1 = y0 + mr;
    if (col == 0) {
      const int c0 = A.nl * A.ls;
      a0 = c0 + y0;
      a1 = c0 + y1;
      step = 2 * mr;
    } else {
      a0 = (y0 >> 1) * A.ls + ((y0 & 1) ? A.x.n - col : col);
      a1 = (y1 >> 1) * A.ls + ((y1 & 1) ? A.x.n - col : col);
      step = mr * A.ls;
    }
  }
  __device__ __forceinline__ int at(int r) const { return ((r & 1) ? a1 : a0) + (r >> 1) * step; }
};

// y stage s.  Forward (DIF) the last stage writes the spectrum (column 0 stays in shared memory);
// inverse (DIT) the last stage of the plan comes first and reads the spectrum.
template <typename R, int RAD, bool INV, bool GLOBAL, int NT>
__device__ __forceinline__ void y_stage(cplx_t<R>* __restrict__ buf, const PlaneArgs& A, int s,
                                        const cplx_t<R>* __restrict__ tw, cplx_t<R>* __restrict__ base, int tid) {
  using C = cplx_t<R>;
  const int M = A.y.M[s], mr = GLOBAL ? 1 : M / RAD, tws = A.y.n / M;
  const int items = A.ncol * (A.y.n / RAD);
  const bool nyq = (A.x.n & 1) == 0;
  for (int it = tid; it < items; it += NT) {
    const int bf = A.dncol.div(it), col = it - bf * A.ncol;
    const int blk = GLOBAL ? bf : (int)A.y.dmr[s].div(bf), n1 = GLOBAL ? 0 : bf - blk * mr;
    const ColumnSlots sl(A, col, blk * M + n1, mr);
    C* g = base + (size_t)(blk * RAD) * A.kxp + col;
    C a[RAD];
    if (GLOBAL && INV) {
#pragma unroll
      for (int r = 0; r < RAD; ++r) a[r] = g[(size_t)r * A.kxp];
      if (col == 0 && nyq) {   // the two real columns as one: F_0 + i F_nyquist
#pragma unroll
        for (int r = 0; r < RAD; ++r) {
          const C f = g[(size_t)r * A.kxp + A.x.n / 2];
          a[r] = mk(a[r].x - f.y, a[r].y + f.x);
        }
      }
    } else {
#pragma unroll
      for (int r = 0; r < RAD; ++r) a[r] = buf[sl.at(r)];
    }
    butterfly<R, RAD, INV, INV>(a, tw, n1 * tws, !GLOBAL && mr > 1);
    if (GLOBAL && !INV && col != 0) {
#pragma unroll
      for (int r = 0; r < RAD; ++r) g[(size_t)r * A.kxp] = a[r];
    } else {
#pragma unroll
      for (int r = 0; r < RAD; ++r) buf[sl.at(r)] = a[r];
    }
  }
}

// Loads (real rows to complex lines, digit-reversed along x) and stores (the reverse) take
// 16 bytes of a row per thread where rows are 16-byte aligned: two threads cover a 32-byte
// sector and the 16 threads of a half-warp lie on different lines, so the scattered
// shared accesses are free of conflicts.
template <typename R> struct Vec;
template <> struct Vec<float> {
  using T = float4;
  static constexpr int W = 4;
};
template <> struct Vec<double> {
  using T = double2;
  static constexpr int W = 2;
};
template <typename R, int NT, typename F>
__device__ __forceinline__ void for_each_vector(const PlaneArgs& A, int tid, F f) {
  constexpr int W = Vec<R>::W;
  const int groups = A.x.n / W, pairs = (groups + 1) / 2;
  for (int it = tid; it < 2 * pairs * A.nl; it += NT) {
    const int h = it >> 1, gp = A.dnl.div(h), line = h - gp * A.nl, xg = 2 * gp + (it & 1);
    if (xg < groups) f(line, xg * W);
  }
}
template <typename R, int NT, typename F>
__device__ __forceinline__ void for_each_scalar(const PlaneArgs& A, int tid, F f) {
  const int oct = (A.x.n + 7) / 8;
  for (int it = tid; it < 8 * oct * A.nl; it += NT) {
    const int h = it >> 3, go = A.dnl.div(h), line = h - go * A.nl, x = 8 * go + (it & 7);
    if (x < A.x.n) f(line, x);
  }
}

template <typename R>
struct PlaneSmem {
  cplx_t<R>* buf;   // lines, then col0
  cplx_t<R>* twx;
  cplx_t<R>* twy;
  int* pofx;
  uint16_t* list;
  __device__ __forceinline__ PlaneSmem(unsigned char* raw, const PlaneArgs& A) {
    buf = reinterpret_cast<cplx_t<R>*>(raw);
    twx = buf + A.nl * A.ls + A.y.n;
    twy = twx + A.x.n;
    pofx = reinterpret_cast<int*>(twy + A.y.n);
    list = reinterpret_cast<uint16_t*>(pofx + A.x.n);
  }
};
template <typename R> size_t plane_smem(const PlaneArgs& A, int nt, bool blobs) {
  const size_t n = (size_t)(A.nl * A.ls + A.x.n + 2 * A.y.n) * sizeof(cplx_t<R>) +
                   A.x.n * sizeof(int) +
                   (blobs ? kPlaneList * sizeof(uint16_t) : 0);
  return blobs ? std::max(n, 3 * (size_t)nt * sizeof(double)) : n;   // (the source sum's tree)
}

template <typename R, int NT>
__device__ __forceinline__ void load_plane_tables(const PlaneSmem<R>& S, const PlaneArgs& A, int tid) {
  const cplx_t<R>* gx = (const cplx_t<R>*)A.x.tw;
  const cplx_t<R>* gy = (const cplx_t<R>*)A.y.tw;
  for (int i = tid; i < A.x.n; i += NT) {
    S.twx[i] = gx[i];
    S.pofx[i] = A.x.pof[i];
  }
  for (int i = tid; i < A.y.n; i += NT) S.twy[i] = gy[i];
}

// Calls f(blob, c, r) with four lanes r = 0 .. 3 for every blob whose support along z covers plane z,
// c the plane's index in it (from -1 to K with EXT, where the Laplacian reaches one plane
// further).  The block scans the blobs' first nodes, a few coalesced bytes each, and compacts
// the hits, up to kPlaneList at a time: cheaper than building bins in three launches while the blobs
// are few (plane_blob_work in icm_api.cu draws the line).  Few enough hits are put in ascending order and served by one warp, so that
// what they add up to does not depend on the warps' timing.
constexpr int kOrdered = 16;
template <int NT, bool EXT, typename F>
__device__ __forceinline__ void for_each_blob_of_plane(const PlaneBlobs& pb, int z, int comp, uint16_t* list, int* count,
                                                       int tid, F f) {
  constexpr int PER = NT == 256 ? 4 : 2, SCAN = PER * NT;   // first nodes in flight per thread
  static_assert(SCAN <= kPlaneList, "one scan fits in the list");
  const int* zf = pb.zfirst + (comp == 2 ? 0 : pb.zstride);
  const int K = pb.p.kernel, nz = pb.p.nz, nb = (int)pb.s.nb;
  const auto plane_of = [&](int first) {   // planes from the first (with EXT the one before it) up to z, periodic
    const int c = z - first + (EXT ? 1 : 0);
    return c < 0 ? c + nz : (c >= nz ? c - nz : c);
  };
  for (int start = 0; start < nb;) {
    __syncthreads();   // the previous list has been used
    if (tid == 0) *count = 0;
    __syncthreads();
    int base = start, found = 0;
    do {
      int first[PER];
#pragma unroll
      for (int j = 0; j < PER; ++j) {
        const int b = base + j * NT + tid;
        first[j] = b < nb ? zf[b] : -1;
      }
#pragma unroll
      for (int j = 0; j < PER; ++j) {
        const bool hit = first[j] >= 0 && plane_of(first[j]) < (EXT ? K + 2 : K);
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        int at = 0;
        if ((tid & 31) == 0 && m) at = atomicAdd(count, __popc(m));
        at = __shfl_sync(0xffffffffu, at, 0);
        const int slot = at + __popc(m & ((1u << (tid & 31)) - 1u)), off = base + j * NT + tid - start;
        if (hit && index_ok(slot, kPlaneList, pb.p.err) && index_ok(off, 65536, pb.p.err) &&
            index_ok(first[j], nz, pb.p.err))
          list[slot] = (uint16_t)off;
      }
      base += SCAN;
      __syncthreads();
      found = *count;
      __syncthreads();
    } while (base < nb && found + SCAN <= kPlaneList && base + SCAN - start <= 65536);
    int threads = NT;
    if (found <= kOrdered) {
      threads = 32;
      if (tid < 32) {   // each entry to its rank
        const int mine = tid < found ? (int)list[tid] : 0;
        int rank = 0;
        for (int k = 0; k < found; ++k) rank += (int)list[k] < mine ? 1 : 0;
        __syncwarp();
        if (tid < found) list[rank] = (uint16_t)mine;
        __syncwarp();
      }
    }
    if (tid < threads)
      for (int t = tid >> 2; t < found; t += threads / 4) {
        if (!index_ok(t, kPlaneList, pb.p.err)) continue;   // (the same for the four lanes)
        const int b = start + list[t];
        if (!index_ok(b, nb, pb.p.err)) continue;
        f(b, plane_of(zf[b]) - (EXT ? 1 : 0), tid & 3);
      }
    start = base;
  }
}

// The x nodes of a stencil row: offsets (in reals) of a line's row 0 for K nodes from `first`.
template <int K>
__device__ __forceinline__ void row_offsets(int (&xo)[K], int first, int nx, const int* __restrict__ pofx) {
#pragma unroll
  for (int a = 0; a < K; ++a) xo[a] = 2 * pofx[wrap_add1(first, a, nx)];
}

// Lane r adds row r of the stencil's K x K nodes on this plane.
template <typename R, int K>
__device__ __forceinline__ void spread_lane(R* __restrict__ rows, const PlaneArgs& A, const int* __restrict__ pofx,
                                            const BlobStencil<R>& rec, int comp, int c, int r, R amp, int* err) {
  if (r >= K) return;
  const int4 f = *reinterpret_cast<const int4*>(rec.first[comp]);
  const int y = wrap_add1(f.y, r, A.y.n);
  R* row = rows + 2 * (y >> 1) * A.ls + (y & 1);
  int xo[K];
  row_offsets<K>(xo, f.x, A.x.n, pofx);
  const R w = rec.w[comp][1][r] * (rec.w[comp][2][c] * amp);
#pragma unroll
  for (int a = 0; a < K; ++a)
    if (index_ok(row - rows + xo[a], 2 * A.nl * A.ls, err)) atomicAdd(&row[xo[a]], rec.w[comp][0][a] * w);
}

__device__ __forceinline__ unsigned quad_mask() { return 0xFu << (threadIdx.x & 28); }
template <typename R> __device__ __forceinline__ R quad_sum(R x) {
  const unsigned m = quad_mask();
  x += __shfl_xor_sync(m, x, 1);
  return x + __shfl_xor_sync(m, x, 2);
}

// The part of (J field)_comp on this plane, c in [0, K): lane r takes row r; the sum is valid in every lane.
template <typename R, int K>
__device__ __forceinline__ R gather_lanes(const R* __restrict__ rows, const PlaneArgs& A, const int* __restrict__ pofx,
                                          const BlobStencil<R>& rec, int comp, int c, int r, int* err) {
  R t = R(0);
  if (r < K) {
    const int4 f = *reinterpret_cast<const int4*>(rec.first[comp]);
    const int y = wrap_add1(f.y, r, A.y.n);
    const R* row = rows + 2 * (y >> 1) * A.ls + (y & 1);
    int xo[K];
    row_offsets<K>(xo, f.x, A.x.n, pofx);
#pragma unroll
    for (int a = 0; a < K; ++a)
      if (index_ok(row - rows + xo[a], 2 * A.nl * A.ls, err)) t += rec.w[comp][0][a] * row[xo[a]];
    t *= rec.w[comp][1][r];
  }
  return quad_sum(t) * rec.w[comp][2][c];
}

// The part of (J L field)_comp on this plane without 1/h^2, c in [-1, K]: the gather with the
// discrete Laplacian of the weights; lane r takes rows r and r + 4 of K + 2.
template <typename R, int K>
__device__ __forceinline__ R gather_lap_lanes(const R* __restrict__ rows, const PlaneArgs& A,
                                              const int* __restrict__ pofx, const BlobStencil<R>& rec, int comp, int c,
                                              int r, int* err) {
  constexpr int E = K + 2;
  const int4 f = *reinterpret_cast<const int4*>(rec.first[comp]);
  // weight e - 1 of an axis (zero outside) and the second difference there
  const auto weight = [&](int ax, int e) { return e >= 1 && e <= K ? rec.w[comp][ax][e - 1] : R(0); };
  const auto second = [&](int ax, int e) { return weight(ax, e - 1) - R(2) * weight(ax, e) + weight(ax, e + 1); };
  const R wz = weight(2, c + 1), dz = second(2, c + 1);
  int xo[E];
  row_offsets<E>(xo, f.x == 0 ? A.x.n - 1 : f.x - 1, A.x.n, pofx);
  R wx[E], dx[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    wx[e] = weight(0, e);
    dx[e] = second(0, e);
  }
  R acc = R(0);
  for (int e = r; e < E; e += 4) {
    const int y = wrap_add1(f.y == 0 ? A.y.n - 1 : f.y - 1, e, A.y.n);
    const R* row = rows + 2 * (y >> 1) * A.ls + (y & 1);
    R t0 = R(0), t1 = R(0);
#pragma unroll
    for (int a = 0; a < E; ++a) {
      const R v = index_ok(row - rows + xo[a], 2 * A.nl * A.ls, err) ? row[xo[a]] : R(0);
      t0 += wx[a] * v;
      t1 += dx[a] * v;
    }
    acc += t1 * weight(1, e) * wz + t0 * (second(1, e) * wz + weight(1, e) * dz);
  }
  return quad_sum(acc);
}

// Component i = 3 b + a of dp = m_e (u - J v~ - du), the momentum change of step 4.
__device__ __forceinline__ double plane_dp(const PlaneBlobs& pb, int i, double jvt) {
  const BlobParams& p = pb.p;
  double du = p.slip == 1 ? 0.0 : 0.5 * (p.eta / p.rho) * p.dt * pb.s.g[i];
  if (p.slip == 2) du += pb.s.w1[i] - pb.s.w0[i];
  return pb.s.me[i / 3] * (pb.s.u[i] - jvt - du);
}

// Component i of what step 5 or 6 spreads: dp with weight m~_f/(rho (m~_f + m_e)), or less m_e J dv~.
__device__ __forceinline__ double plane_source(const PlaneBlobs& pb, int i) {
  const BlobParams& p = pb.p;
  const double me = pb.s.me[i / 3];
  const long long n3 = 3 * pb.s.nb;
  const double dp = plane_dp(pb, i, plane_sum(pb.jvt, n3, i, p.kernel));
  if (pb.source == PLANE_CDP) return p.mtf / (p.rho * (p.mtf + me)) * dp;
  return dp - me * plane_sum(pb.jdvt, n3, i, p.kernel);
}

// The grid sum of the source of step 6, for the momentum bookkeeping, and the values of J v~ and J dv~, whose parts
// make room for those of J dv in the inverse pass: NT elements per block.
template <int NT>
__device__ __forceinline__ void add_source_sum(const PlaneBlobs& pb, int block, int tid, double (*red)[NT]) {
  const int i = block * NT + tid, a = i % 3;
  double x = 0.0;
  if (i < 3 * (int)pb.s.nb) {
    const long long n3 = 3 * pb.s.nb;
    const double jvt = plane_sum(pb.jvt, n3, i, pb.p.kernel), jdvt = plane_sum(pb.jdvt, n3, i, pb.p.kernel);
    pb.s.jvt[i] = jvt;
    pb.s.cdp[i] = jdvt;
    x = plane_dp(pb, i, jvt) - pb.s.me[i / 3] * jdvt;
  }
  for (int c = 0; c < 3; ++c) red[c][tid] = c == a ? x : 0.0;
  __syncthreads();
  for (int w = NT / 2; w > 0; w >>= 1) {
    if (tid < w)
      for (int c = 0; c < 3; ++c) red[c][tid] += red[c][tid + w];
    __syncthreads();
  }
  if (tid < 3) atomicAdd(&pb.s.scal[SC_SUMSRC + tid], red[tid][0]);
}

template <typename R, int NT, bool BLOBS>
__global__ void __launch_bounds__(NT, sizeof(R) == 4 ? (NT == 256 ? 3 : 2) : 1)
    k_plane_fwd(const __grid_constant__ PlaneArgs A, const R* __restrict__ src, cplx_t<R>* __restrict__ spec,
                const __grid_constant__ PlaneBlobs pb, const RepFft* __restrict__ reps) {
  using C = cplx_t<R>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_count;
  const PlaneSmem<R> S(smem_raw, A);
  const int tid = threadIdx.x, z = blockIdx.x, comp = blockIdx.y % 3;
  if constexpr (BLOBS) {
    if (z >= A.nz) {   // the blocks past the planes (step 6, component 0 of the grid)
      if (comp == 0) add_source_sum<NT>(pb, z - A.nz, tid, reinterpret_cast<double (*)[NT]>(smem_raw));
      return;
    }
  }
  if (!BLOBS && reps != nullptr) {
    const RepFft& rp = reps[blockIdx.y / 3];
    src = reinterpret_cast<const R*>(rp.src);
    spec = reinterpret_cast<C*>(rp.spec);
  }
  const int nx = A.x.n, ny = A.y.n;
  if (!BLOBS || src != nullptr) {
    const R* p = src + comp * A.ncell + (size_t)z * nx * ny;
    if (nx % Vec<R>::W == 0) {
      for_each_vector<R, NT>(A, tid, [&](int line, int x) {
        using V = typename Vec<R>::T;
        const R* r0 = p + (size_t)(2 * line) * nx + x;
        const bool two = 2 * line + 1 < ny;
        const V a = *reinterpret_cast<const V*>(r0);
        V b{};
        if (two) b = *reinterpret_cast<const V*>(r0 + nx);
        C* o = S.buf + line * A.ls;
        const int* pof = A.x.pof + x;
        o[pof[0]] = mk(a.x, b.x);
        o[pof[1]] = mk(a.y, b.y);
        if constexpr (sizeof(R) == 4) {
          o[pof[2]] = mk(a.z, b.z);
          o[pof[3]] = mk(a.w, b.w);
        }
      });
    } else {
      for_each_scalar<R, NT>(A, tid, [&](int line, int x) {
        const R* r0 = p + (size_t)(2 * line) * nx + x;
        S.buf[line * A.ls + A.x.pof[x]] = mk(r0[0], 2 * line + 1 < ny ? r0[nx] : R(0));
      });
    }
  } else {
    for (int i = tid; i < A.nl * A.ls; i += NT) S.buf[i] = mk(R(0), R(0));
  }
  load_plane_tables<R, NT>(S, A, tid);
  if (BLOBS) {
    R* rows = reinterpret_cast<R*>(S.buf);
    const BlobStencil<R>* rec = reinterpret_cast<const BlobStencil<R>*>(pb.geo);
    const double inv_dvf = pb.p.inv_h * pb.p.inv_h * pb.p.inv_h;
    for_each_blob_of_plane<NT, false>(pb, z, comp, S.list, &s_count, tid, [&](int b, int c, int r) {
      const int i = 3 * b + comp;
      const R amp = (R)((pb.source == PLANE_VEC ? pb.vec[i] : plane_source(pb, i)) * inv_dvf);
      if (pb.p.kernel == 3)
        spread_lane<R, 3>(rows, A, S.pofx, rec[b], comp, c, r, amp, pb.p.err);
      else
        spread_lane<R, 4>(rows, A, S.pofx, rec[b], comp, c, r, amp, pb.p.err);
    });
  }
  __syncthreads();
  for (int s = A.x.ns - 1; s >= 0; --s) {
#define ICM_X(RAD) x_stage<R, RAD, false, NT>(S.buf, A, s, S.twx, tid)
    ICM_RADIX_SWITCH(A.x.rad[s], ICM_X)
#undef ICM_X
    __syncthreads();
  }
  C* col0 = S.buf + A.nl * A.ls;
  for (int it = tid; it < A.nl * A.ncol; it += NT) {
    const int k = A.dnl.div(it), l = it - k * A.nl;
    C* p = S.buf + l * A.ls;
    if (k == 0) {
      const C z0 = p[0], zh = nx % 2 == 0 ? p[nx / 2] : mk(R(0), R(0));
      col0[2 * l] = mk(z0.x, zh.x);
      if (2 * l + 1 < ny) col0[2 * l + 1] = mk(z0.y, zh.y);
    } else {
      const C zk = p[k], zm = p[nx - k];
      p[k] = mk(zk.x + zm.x, zk.y - zm.y);   // twice the spectrum (SymParams::inv_ntot)
      p[nx - k] = mk(zk.y + zm.y, zm.x - zk.x);
    }
  }
  __syncthreads();
  C* base = spec + ((size_t)(comp * A.nz + z) * ny) * A.kxp;
  for (int s = 0; s + 1 < A.y.ns; ++s) {
#define ICM_Y(RAD) y_stage<R, RAD, false, false, NT>(S.buf, A, s, S.twy, base, tid)
    ICM_RADIX_SWITCH(A.y.rad[s], ICM_Y)
#undef ICM_Y
    __syncthreads();
  }
  {
    const int s = A.y.ns - 1;
#define ICM_Y(RAD) y_stage<R, RAD, false, true, NT>(S.buf, A, s, S.twy, base, tid)
    ICM_RADIX_SWITCH(A.y.rad[s], ICM_Y)
#undef ICM_Y
  }
  __syncthreads();
  for (int f = tid; f < ny; f += NT) {   // the two real columns, by Hermitian symmetry along y
    const int p = A.y.pof[f], pm = A.y.pof[f == 0 ? 0 : ny - f];
    const C c = col0[p], d = col0[pm];
    base[(size_t)p * A.kxp] = mk(c.x + d.x, c.y - d.y);
    if (nx % 2 == 0) base[(size_t)p * A.kxp + nx / 2] = mk(c.y + d.y, d.x - c.x);
  }
}

// MODE and GATHER as in k_xinv2 (GATHER 0, 1 or 2).
template <typename R, int NT, int MODE, int GATHER>
__global__ void __launch_bounds__(NT, sizeof(R) == 4 ? (NT == 256 ? 3 : 2) : 1)
    k_plane_inv(const __grid_constant__ PlaneArgs A, const cplx_t<R>* __restrict__ spec, R* __restrict__ dst,
                R* __restrict__ dst2, const __grid_constant__ PlaneBlobs pb, const RepFft* __restrict__ reps) {
  using C = cplx_t<R>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_count;
  const PlaneSmem<R> S(smem_raw, A);
  const int tid = threadIdx.x, z = blockIdx.x, comp = blockIdx.y % 3;
  if (GATHER == 0 && reps != nullptr) {
    const RepFft& rp = reps[blockIdx.y / 3];
    spec = reinterpret_cast<const C*>(rp.spec);
    dst = reinterpret_cast<R*>(rp.dst);
    dst2 = reinterpret_cast<R*>(rp.dst2);
  }
  const int nx = A.x.n, ny = A.y.n;
  C* base = const_cast<C*>(spec) + ((size_t)(comp * A.nz + z) * ny) * A.kxp;
  load_plane_tables<R, NT>(S, A, tid);
  {
    const int s = A.y.ns - 1;
#define ICM_Y(RAD) y_stage<R, RAD, true, true, NT>(S.buf, A, s, S.twy, base, tid)
    ICM_RADIX_SWITCH(A.y.rad[s], ICM_Y)
#undef ICM_Y
  }
  __syncthreads();
  for (int s = A.y.ns - 2; s >= 0; --s) {
#define ICM_Y(RAD) y_stage<R, RAD, true, false, NT>(S.buf, A, s, S.twy, base, tid)
    ICM_RADIX_SWITCH(A.y.rad[s], ICM_Y)
#undef ICM_Y
    __syncthreads();
  }
  C* col0 = S.buf + A.nl * A.ls;
  for (int it = tid; it < A.nl * A.ncol; it += NT) {
    const int k = A.dnl.div(it), l = it - k * A.nl;
    C* p = S.buf + l * A.ls;
    const bool two = 2 * l + 1 < ny;
    if (k == 0) {
      const C c = col0[2 * l], d = two ? col0[2 * l + 1] : mk(R(0), R(0));
      p[0] = mk(c.x, d.x);
      if (nx % 2 == 0) p[nx / 2] = mk(c.y, d.y);
    } else {
      const C x1 = p[k], x2 = two ? p[nx - k] : mk(R(0), R(0));
      p[k] = mk(x1.x - x2.y, x1.y + x2.x);
      p[nx - k] = mk(x1.x + x2.y, x2.x - x1.y);
    }
  }
  __syncthreads();
  for (int s = 0; s < A.x.ns; ++s) {
#define ICM_X(RAD) x_stage<R, RAD, true, NT>(S.buf, A, s, S.twx, tid)
    ICM_RADIX_SWITCH(A.x.rad[s], ICM_X)
#undef ICM_X
    __syncthreads();
  }
  if (MODE != OUT_NONE) {
    const size_t off = comp * A.ncell + (size_t)z * nx * ny;
    if (nx % Vec<R>::W == 0) {
      for_each_vector<R, NT>(A, tid, [&](int line, int x) {
        using V = typename Vec<R>::T;
        const size_t o = off + (size_t)(2 * line) * nx + x;
        const bool two = 2 * line + 1 < ny;
        const C* q = S.buf + line * A.ls;
        V a, b;
        const int* pof = S.pofx + x;
        C c = q[pof[0]], d = q[pof[1]];
        a.x = c.x; b.x = c.y;
        a.y = d.x; b.y = d.y;
        if constexpr (sizeof(R) == 4) {
          c = q[pof[2]];
          d = q[pof[3]];
          a.z = c.x; b.z = c.y;
          a.w = d.x; b.w = d.y;
        }
        if (MODE == OUT_ADD_AND_STORE2) {
          *reinterpret_cast<V*>(dst2 + o) = a;
          if (two) *reinterpret_cast<V*>(dst2 + o + nx) = b;
        }
        if (MODE == OUT_ADD || MODE == OUT_ADD_AND_STORE2) {
          const V u = *reinterpret_cast<const V*>(dst + o);
          V w{};
          if (two) w = *reinterpret_cast<const V*>(dst + o + nx);
          a.x += u.x; a.y += u.y;
          b.x += w.x; b.y += w.y;
          if constexpr (sizeof(R) == 4) {
            a.z += u.z; a.w += u.w;
            b.z += w.z; b.w += w.w;
          }
        }
        *reinterpret_cast<V*>(dst + o) = a;
        if (two) *reinterpret_cast<V*>(dst + o + nx) = b;
      });
    } else {
      for_each_scalar<R, NT>(A, tid, [&](int line, int x) {
        const size_t o = off + (size_t)(2 * line) * nx + x;
        const C c = S.buf[line * A.ls + S.pofx[x]];
        const auto put = [&](size_t at, R val) {
          if (MODE == OUT_ADD_AND_STORE2) dst2[at] = val;
          dst[at] = MODE == OUT_STORE ? val : dst[at] + val;
        };
        put(o, c.x);
        if (2 * line + 1 < ny) put(o + nx, c.y);
      });
    }
  }
  if (GATHER) {
    const R* rows = reinterpret_cast<const R*>(S.buf);
    const BlobStencil<R>* rec = reinterpret_cast<const BlobStencil<R>*>(pb.geo);
    const long long n3 = 3 * pb.s.nb;
    for_each_blob_of_plane<NT, GATHER == 2>(pb, z, comp, S.list, &s_count, tid, [&](int b, int c, int r) {
      const long long i = 3 * (long long)b + comp;
      const bool three = pb.p.kernel == 3;
      if (c >= 0 && c < pb.p.kernel) {   // the same for the four lanes
        const R j = three ? gather_lanes<R, 3>(rows, A, S.pofx, rec[b], comp, c, r, pb.p.err)
                          : gather_lanes<R, 4>(rows, A, S.pofx, rec[b], comp, c, r, pb.p.err);
        if (r == 0 && index_ok(pb.part + c * n3 + i - pb.jvt, kPlaneParts * n3, pb.p.err)) pb.part[c * n3 + i] = (double)j;
      }
      if (GATHER == 2) {
        const R jl = three ? gather_lap_lanes<R, 3>(rows, A, S.pofx, rec[b], comp, c, r, pb.p.err)
                           : gather_lap_lanes<R, 4>(rows, A, S.pofx, rec[b], comp, c, r, pb.p.err);
        if (r == 0 && index_ok(pb.part_lap + (c + 1) * n3 + i - pb.jvt, kPlaneParts * n3, pb.p.err))
          pb.part_lap[(c + 1) * n3 + i] = (double)jl;
      }
    });
  }
}

// ---------------------------------------------------------------------------
// The z pass of sides without two-stage register kernels: a block transforms kZAny wave
// numbers of one y row for the three components, applies the symbol and transforms back.
// The first stage reads global memory into registers, the last one writes it, and the middle stage
// keeps the three components of its wave numbers in registers through the symbol.
// ---------------------------------------------------------------------------
constexpr int kZAny = kZLines;

template <typename R, int RAD, bool INV, bool GLOBAL, int NT>
__device__ __forceinline__ void z_stage(cplx_t<R>* __restrict__ buf, const StageAxis& Z, int s,
                                        const cplx_t<R>* __restrict__ tw, cplx_t<R>* __restrict__ base, size_t zs,
                                        size_t cs, bool live, int tid) {
  using C = cplx_t<R>;
  const int M = Z.M[s], mr = M / RAD, tws = Z.n / M, nbf = Z.n / RAD;
  for (int it = tid; it < 3 * nbf * kZAny; it += NT) {
    const int line = it % kZAny, rest = it / kZAny;
    const int comp = rest < nbf ? 0 : (rest < 2 * nbf ? 1 : 2), bf = rest - comp * nbf;
    const int blk = GLOBAL ? 0 : (int)Z.dmr[s].div(bf), n1 = GLOBAL ? bf : bf - blk * mr;
    C* p = buf + (comp * Z.n + blk * M + n1) * kZAny + line;
    C* g = base + comp * cs + n1 * zs;
    C a[RAD];
    if (GLOBAL && !INV) {
#pragma unroll
      for (int r = 0; r < RAD; ++r) a[r] = live ? g[(size_t)(r * mr) * zs] : mk(R(0), R(0));
    } else {
#pragma unroll
      for (int r = 0; r < RAD; ++r) a[r] = p[r * mr * kZAny];
    }
    butterfly<R, RAD, INV, INV>(a, tw, n1 * tws, true);
    if (GLOBAL && INV) {
      if (live) {
#pragma unroll
        for (int r = 0; r < RAD; ++r) g[(size_t)(r * mr) * zs] = a[r];
      }
    } else {
#pragma unroll
      for (int r = 0; r < RAD; ++r) p[r * mr * kZAny] = a[r];
    }
  }
}

// FP64: the last forward stage, the symbol and the first inverse stage one after the other, one
// butterfly or wave vector per thread: with three components held the symbols of a butterfly
// are a serial chain of FP64 operations (18.4 us against 12.2 per pass on 16^3).
template <typename R, int RAD, int NT>
__device__ __forceinline__ void z_symbol_apart(cplx_t<R>* __restrict__ buf, const StageAxis& Z, const SymParams<R>& sp,
                                               int k, int py, bool live, int tid) {
  using C = cplx_t<R>;
  const int cs = Z.n * kZAny, nbf = Z.n / RAD;
  const auto dft = [&](bool inv) {
    for (int it = tid; it < 3 * nbf * kZAny; it += NT) {
      C* p = buf + (it / kZAny) * (RAD * kZAny) + it % kZAny;   // blocks of RAD rows, component after component
      C b[RAD];
#pragma unroll
      for (int r = 0; r < RAD; ++r) b[r] = p[r * kZAny];
      if (inv)
        sdft_inv<R, RAD>(b);
      else
        SDft<R, RAD>::run(b);
#pragma unroll
      for (int r = 0; r < RAD; ++r) p[r * kZAny] = b[r];
    }
    __syncthreads();
  };
  dft(false);
  const C dyv = sp.dy[py];
  const R ddy = sp.ddy[py];
  for (int it = tid; it < cs; it += NT) {
    const int pz = it / kZAny;
    if (live)
      apply_symbol<R>(buf[it], buf[cs + it], buf[2 * cs + it], sp.dx[k], dyv, sp.dz[pz], sp.ddx[k] + ddy + sp.ddz[pz], sp,
                      k == 0 && py == 0 && pz == 0);
  }
  __syncthreads();
  dft(true);
}

template <typename R, int RAD, int NT>
__device__ __forceinline__ void z_symbol_stage(cplx_t<R>* __restrict__ buf, const StageAxis& Z, const SymParams<R>& sp,
                                               int k, int py, bool live, int tid) {
  using C = cplx_t<R>;
  const C dyv = sp.dy[py];
  const R ddy = sp.ddy[py];
  for (int it = tid; it < (Z.n / RAD) * kZAny; it += NT) {
    const int line = it % kZAny, blk = it / kZAny;
    if (!live) continue;
    C b[3][RAD];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
      for (int r = 0; r < RAD; ++r) b[c][r] = buf[(c * Z.n + blk * RAD + r) * kZAny + line];
      SDft<R, RAD>::run(b[c]);
    }
    const C d0 = sp.dx[k];
    const R dxy = sp.ddx[k] + ddy;
#pragma unroll
    for (int r = 0; r < RAD; ++r) {
      const int pz = blk * RAD + r;
      apply_symbol<R>(b[0][r], b[1][r], b[2][r], d0, dyv, sp.dz[pz], dxy + sp.ddz[pz], sp, k == 0 && py == 0 && pz == 0);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      sdft_inv<R, RAD>(b[c]);
#pragma unroll
      for (int r = 0; r < RAD; ++r) buf[(c * Z.n + blk * RAD + r) * kZAny + line] = b[c][r];
    }
  }
}

constexpr int kZAnyThreads = 128;
template <typename R>
__global__ void __launch_bounds__(kZAnyThreads, sizeof(R) == 4 ? 4 : 2)
    k_zsym_any(const __grid_constant__ StageAxis Z, cplx_t<R>* __restrict__ spec, int ny, int kx, int kxp,
               SymParams<R> sp) {
  using C = cplx_t<R>;
  constexpr int NT = kZAnyThreads;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw);
  C* tw = buf + 3 * Z.n * kZAny;
  const int tid = threadIdx.x;
  // NT is a multiple of kZAny: a thread keeps its line in every loop
  static_assert(NT % kZAny == 0, "fixed line per thread");
  const ZTile<R> zt(blockIdx.x, kx, ny);
  const bool live = zt.live(tid % kZAny, kx, ny);
  const int k = live ? zt.k(tid % kZAny) : 0, py = live ? zt.row(tid % kZAny) : 0;
  const size_t zs = (size_t)ny * kxp, cs = (size_t)Z.n * zs;
  C* base = spec + (size_t)py * kxp + k;
  for (int i = tid; i < Z.n; i += NT) tw[i] = ((const C*)Z.tw)[i];
  __syncthreads();
#define ICM_Z(RAD) z_stage<R, RAD, false, true, NT>(buf, Z, 0, tw, base, zs, cs, live, tid)
  ICM_RADIX_SWITCH(Z.rad[0], ICM_Z)
#undef ICM_Z
  __syncthreads();
  for (int s = 1; s + 1 < Z.ns; ++s) {
#define ICM_Z(RAD) z_stage<R, RAD, false, false, NT>(buf, Z, s, tw, base, zs, cs, live, tid)
    ICM_RADIX_SWITCH(Z.rad[s], ICM_Z)
#undef ICM_Z
    __syncthreads();
  }
#define ICM_Z(RAD)                                              \
  if constexpr (sizeof(R) == 4)                                 \
    z_symbol_stage<R, RAD, NT>(buf, Z, sp, k, py, live, tid); \
  else                                                          \
    z_symbol_apart<R, RAD, NT>(buf, Z, sp, k, py, live, tid)
  switch (Z.rad[Z.ns - 1]) {   // the last factor of a general side (general_factors)
    case 2: ICM_Z(2); break;
    case 3: ICM_Z(3); break;
    case 4: ICM_Z(4); break;
    case 6: ICM_Z(6); break;
    case 8: ICM_Z(8); break;
    case 9: ICM_Z(9); break;
    default: ICM_Z(12); break;
  }
#undef ICM_Z
  __syncthreads();
  for (int s = Z.ns - 2; s >= 1; --s) {
#define ICM_Z(RAD) z_stage<R, RAD, true, false, NT>(buf, Z, s, tw, base, zs, cs, live, tid)
    ICM_RADIX_SWITCH(Z.rad[s], ICM_Z)
#undef ICM_Z
    __syncthreads();
  }
#define ICM_Z(RAD) z_stage<R, RAD, true, true, NT>(buf, Z, 0, tw, base, zs, cs, live, tid)
  ICM_RADIX_SWITCH(Z.rad[0], ICM_Z)
#undef ICM_Z
}

static StageAxis stage_axis(const AxisPlan& P) {
  StageAxis a;
  a.n = P.n;
  a.ns = P.nstages;
  a.tw = P.tw;
  a.pof = P.pos_of_freq;
  int m = P.n;
  for (int s = 0; s < kMaxFactors; ++s) {
    a.M[s] = s < P.nstages ? m : 1;
    a.rad[s] = s < P.nstages ? P.radix[s] : 1;
    m /= a.rad[s];
    a.dmr[s] = FastDiv((uint32_t)std::max(1, a.M[s] / a.rad[s]));
  }
  return a;
}

template <typename R>
PlaneArgs plane_args(const FftCtx<R>& f) {
  PlaneArgs A;
  A.x = stage_axis(f.px);
  A.y = stage_axis(f.py);
  A.nz = f.nz;
  A.kx = f.kx;
  A.kxp = f.kxp;
  A.nl = (f.ny + 1) / 2;
  A.ls = f.nx | 1;
  A.ncol = 1 + (f.nx - 1) / 2;
  A.dnl = FastDiv((uint32_t)A.nl);
  A.dncol = FastDiv((uint32_t)A.ncol);
  A.ncell = f.ncell;
  return A;
}

// Threads of a plane block: 256, so that three blocks share an SM, or 512 where shared memory
// lets an SM hold fewer than three.
constexpr size_t kPlaneSmemOf3 = 74 * 1024;
template <typename R> bool plane_wide(const FftCtx<R>& f) {
  return (size_t)((f.ny + 1) / 2 * (f.nx | 1) + f.nx + 2 * f.ny) * sizeof(cplx_t<R>) > kPlaneSmemOf3;
}

}  // namespace

#if ICM_PLANE_PREC == 32
// Where the alternative is the general passes: whatever fits. Sides with register kernels along both:
// planes that two blocks per SM can hold, and in FP64, where a block keeps its SM's FP64 pipe busy by
// itself, only if the 3 nz planes fill whole waves of the SMs (to 0.8) or a part of one.
// Step of a simulation with n^3/1000 blobs, separate passes against planes (us): FP32 74 / 68 on
// 32^3, 113 / 92 on 64^3, 197 / 165 on 96^3, 302 / 270 on 128^3; x and y passes of an FP64 solve, launch
// gaps included: 78 / 59 on 48^3 (144 planes), 101 / 124 on 64^3 (192 planes, 1.3 waves), 344 / 301 on 96^3.
// 144 x 108 x 216 in FP32: 1180 / 530 per step.
bool plane_has_passes(int precision, int nx, int ny, int nz) {
  const size_t c = precision == 32 ? 8 : 16;
  const size_t need = ((size_t)((ny + 1) / 2) * (nx | 1) + nx + 2 * ny) * c + nx * 4 + kPlaneList * 2;
  int r1, r2;
  if ((fft_split(nx, r1, r2) && r1 > 16) || (fft_split(ny, r1, r2) && r1 > 16)) return false;   // no radix above 16 here
  if (!(fft_split(nx, r1, r2) && fft_split(ny, r1, r2))) return need <= (size_t)226 * 1024;
  if (need > (size_t)112 * 1024) return false;
  const int nsm = device_sms(), planes = 3 * nz, waves = (planes + nsm - 1) / nsm;
  return precision == 32 || waves == 1 || 10 * planes >= 8 * waves * nsm;
}

// A launch over many members keeps the device full whichever way, and then the separate passes' cheaper
// butterflies count.  In FP64 that is so from two members on: planes / separate, a step of the batch (us):
// 32^3, two members 299 / 248, 32 members 2226 / 1574; 48^3 583 / 570 and 7561 / 6693; 96^3 3427 / 3441
// and (16) 25729 / 25749.  In FP32 planes win up to one round of three blocks per SM, or two full ones,
// and from 96 x 96 on: 32^3, four members 99 / 103, 16 members 187 / 159; 48^3, three 127 / 155, six 185 /
// 203, 16 members 393 / 375; 64^3, two 140 / 141, 16 members 609 / 563; 96^3, 16 members 1643 / 1898;
// 128^3, two 540 / 497, eight 1749 / 1796.
bool plane_has_group_passes(int precision, int nx, int ny, int nz, int members) {
  if (!plane_has_passes(precision, nx, ny, nz)) return false;
  if (members == 1) return true;
  if (precision == 64) return false;
  const long long planes = 3LL * nz * members, round = 3LL * device_sms();
  return planes <= round || nx * ny >= 96 * 96 || (planes <= 2 * round && 10 * planes >= 18 * round);
}
#endif

template <typename R>
void plane_prepare() {
  const int big = 226 * 1024;
#define ICM_ATTR(K) cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
#define ICM_ATTRS(NT)                          \
  ICM_ATTR((k_plane_fwd<R, NT, false>))        \
  ICM_ATTR((k_plane_fwd<R, NT, true>))         \
  ICM_ATTR((k_plane_inv<R, NT, OUT_STORE, 0>)) \
  ICM_ATTR((k_plane_inv<R, NT, OUT_ADD_AND_STORE2, 0>)) \
  ICM_ATTR((k_plane_inv<R, NT, OUT_STORE, 1>)) \
  ICM_ATTR((k_plane_inv<R, NT, OUT_NONE, 1>))  \
  ICM_ATTR((k_plane_inv<R, NT, OUT_ADD, 2>))
  ICM_ATTRS(256)
  ICM_ATTRS(512)
  ICM_ATTR((k_zsym_any<R>))
#undef ICM_ATTRS
#undef ICM_ATTR
}

#if ICM_PLANE_PREC == 64
// Whether this context has the attributes of fft_prepare, whose last call is the one above for FP64.
bool plane_prepared() {
  cudaFuncAttributes a;
  if (cudaFuncGetAttributes(&a, k_zsym_any<double>) == cudaSuccess) return a.maxDynamicSharedSizeBytes == 226 * 1024;
  cudaGetLastError();
  return false;
}
#endif

template <typename R>
void plane_forward(const FftCtx<R>& f, const R* src, const PlaneBlobs* pb, const RepFft* reps, int G, cudaStream_t st) {
  const PlaneArgs A = plane_args(f);
  const bool wide = plane_wide(f);
  const int nt = wide ? 512 : 256;
  const int sums = pb && pb->source == PLANE_SRC ? (int)((3 * pb->s.nb + nt - 1) / nt) : 0;
  const dim3 grid(f.nz + sums, 3 * G);
  const PlaneBlobs none{};
  if (wide) {
    if (pb)
      k_plane_fwd<R, 512, true><<<grid, 512, plane_smem<R>(A, 512, true), st>>>(A, src, f.spec, *pb, nullptr);
    else
      k_plane_fwd<R, 512, false><<<grid, 512, plane_smem<R>(A, 512, false), st>>>(A, src, f.spec, none, reps);
  } else {
    if (pb)
      k_plane_fwd<R, 256, true><<<grid, 256, plane_smem<R>(A, 256, true), st>>>(A, src, f.spec, *pb, nullptr);
    else
      k_plane_fwd<R, 256, false><<<grid, 256, plane_smem<R>(A, 256, false), st>>>(A, src, f.spec, none, reps);
  }
}

template <typename R, int NT>
void plane_inverse_nt(const FftCtx<R>& f, R* dst, R* dst2, int mode, const PlaneBlobs* pb, const RepFft* reps, int G,
                      cudaStream_t st) {
  const PlaneArgs A = plane_args(f);
  const dim3 grid(f.nz, 3 * G);
  const size_t sm = plane_smem<R>(A, NT, pb != nullptr);
  const PlaneBlobs none{};
  if (pb) {
    if (mode == OUT_STORE)
      k_plane_inv<R, NT, OUT_STORE, 1><<<grid, NT, sm, st>>>(A, f.spec, dst, nullptr, *pb, nullptr);
    else if (mode == OUT_NONE)
      k_plane_inv<R, NT, OUT_NONE, 1><<<grid, NT, sm, st>>>(A, f.spec, dst, nullptr, *pb, nullptr);
    else
      k_plane_inv<R, NT, OUT_ADD, 2><<<grid, NT, sm, st>>>(A, f.spec, dst, nullptr, *pb, nullptr);
  } else if (mode == OUT_STORE) {
    k_plane_inv<R, NT, OUT_STORE, 0><<<grid, NT, sm, st>>>(A, f.spec, dst, dst2, none, reps);
  } else {
    k_plane_inv<R, NT, OUT_ADD_AND_STORE2, 0><<<grid, NT, sm, st>>>(A, f.spec, dst, dst2, none, reps);
  }
}
template <typename R>
void plane_inverse(const FftCtx<R>& f, R* dst, R* dst2, int mode, const PlaneBlobs* pb, const RepFft* reps, int G,
                   cudaStream_t st) {
  if (plane_wide(f))
    plane_inverse_nt<R, 512>(f, dst, dst2, mode, pb, reps, G, st);
  else
    plane_inverse_nt<R, 256>(f, dst, dst2, mode, pb, reps, G, st);
}

template <typename R>
void fft_z_any(const FftCtx<R>& f, const SymParams<R>& sp, cudaStream_t st) {
  const StageAxis Z = stage_axis(f.pz);
  const size_t sm = (size_t)(3 * f.nz * kZAny + f.nz) * sizeof(cplx_t<R>);
  k_zsym_any<R><<<z_tiles<R>(f.kx, f.ny), kZAnyThreads, sm, st>>>(Z, f.spec, f.ny, f.kx, f.kxp, sp);
}

// This file is compiled once per precision (-DICM_PLANE_PREC=32 or 64).
#define ICM_INST(R)                                                                                                \
  template void plane_prepare<R>();                                                                               \
  template void plane_forward<R>(const FftCtx<R>&, const R*, const PlaneBlobs*, const RepFft*, int, cudaStream_t); \
  template void plane_inverse<R>(const FftCtx<R>&, R*, R*, int, const PlaneBlobs*, const RepFft*, int, cudaStream_t); \
  template void fft_z_any<R>(const FftCtx<R>&, const SymParams<R>&, cudaStream_t);
#if ICM_PLANE_PREC == 32
ICM_INST(float)
#else
ICM_INST(double)
#endif
#undef ICM_INST

}  // namespace icm
