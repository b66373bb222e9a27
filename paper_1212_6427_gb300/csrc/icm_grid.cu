// Grid kernels of the ICM step (arXiv:1212.6427, Sec. III.B-C):
//   * the explicit right-hand side of Eq. provisional_step-1, one fused pass:
//       r = (rho/dt) v + (eta/2) L v + div Sigma^n - (3/2 A^n - 1/2 A^{n-1}),
//     with the stochastic stress Sigma^n = sqrt(kT eta/(dV_f dt)) (W + W^T) drawn
//     from Philox4x32-10 on the fly (never stored) and A = div(rho v v^T) in
//     centred conservative (skew-adjoint) form, Adams-Bashforth in time
//     (Eq. Adams_Bashforth).  A^n overwrites A^{n-1} in place.
//   * FP64 compensated sums of face fields (momentum bookkeeping, Sec. II).
#include <algorithm>
#include <atomic>
#include <cmath>

#include "icm_internal.h"

namespace icm {
namespace {

constexpr int TX = 32, TY = 16;     // cells per block in x and y (one thread each)
constexpr int HX = TX + 2, HY = TY + 2;
constexpr int NT = TX * TY;         // threads per block
constexpr int NHALO = 2 * HX + 2 * TY;   // ring of halo cells around the TX x TY tile

__device__ __forceinline__ int wrapi(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }
// Periodic index for any i (a tile can be several times wider than a short side).
__device__ __forceinline__ int wrapm(int i, int n) { return ((i % n) + n) % n; }

// ---------------------------------------------------------------------------
// FP64 Box-Muller.  FP64 operations are the scarce resource here (64 times slower than
// FP32), and log, sqrt and sincospi take about 97 of them per pair of normals.  With
// tables (Tang's table-driven method, ACM TOMS 16, 1990) and short Taylor polynomials the
// pair takes 28, at the same accuracy (-2 ln u within 3.2e-16 relative, sin and cos within
// 1.9e-16): 1024 intervals put the reduced arguments below 2^-10 and pi/1024, where
// degrees 6 (log), 5 (sin) and 4 (cos) are enough; gathers of 16 bytes from 33 KB of tables stay
// in L1.  u = m 2^-33 with m = 2 x + 1 keeps every reduction exact.
// ---------------------------------------------------------------------------
constexpr int kTab = 1024;
__device__ double2 g_log_tab[kTab];     // interval i of the mantissa: -2/c_i, 2 ln(1/c_i)
__device__ double2 g_circle_tab[kTab];  // cos, sin of 2 pi (i + 1/2)/1024
__device__ double g_ln2_tab[34];        // 2 k ln 2

// -2 ln((x + 1/2) 2^-32).  The mantissa is taken in [3/4, 3/2), so that u near 1 has exponent
// 0 and interval centre 1: the result keeps its relative accuracy there.
__device__ __forceinline__ double minus_two_log(uint32_t x) {
  const uint64_t m = 2ull * x + 1ull;
  const int lz = __clzll((long long)m);
  const uint64_t norm = m << lz;                 // leading one at bit 63
  const uint32_t hi = (uint32_t)(norm >> 32);
  const uint32_t half = (hi >> 30) & 1u;         // mantissa >= 3/2: halved
  const double2 t = __ldg(&g_log_tab[(hi >> 21) & (kTab - 1)]);
  const double k2 = __ldg(&g_ln2_tab[lz - 30 - (int)half]);
  const double f = __longlong_as_double((long long)(((norm >> 11) & 0xFFFFFFFFFFFFFull) |
                                                    ((uint64_t)(1023u - half) << 52)));
  const double s = fma(f, t.x, 2.0);             // -2 r, r = f/c - 1
  double p = fma(s, 1.0 / 192.0, 1.0 / 80.0);    // -2 ln(1 - s/2) = s + s^2/4 + s^3/12 + ...
  p = fma(s, p, 1.0 / 32.0);
  p = fma(s, p, 1.0 / 12.0);
  p = fma(s, p, 0.25);
  return (k2 + t.y) + fma(s * s, p, s);
}

// sqrt(x), x in [2e-10, 46]: the approximate reciprocal root instruction and one Householder
// step of third order, sqrt = g + g e (1/2 + 3/8 e) with g = x y, e = 1 - g y.
__device__ __forceinline__ double root_of(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double g = x * y, e = fma(-g, y, 1.0);
  return fma(g * e, fma(e, 0.375, 0.5), g);
}

template <typename R> struct NormalPair : BoxMuller<R> {};
template <> struct NormalPair<double> {
  __device__ __forceinline__ static void apply(uint32_t a, uint32_t b, double& z0, double& z1) {
    const double rad = root_of(minus_two_log(a));
    // 2 pi (b + 1/2) 2^-32 = centre of sector b >> 22 plus t, |t| < pi/1024
    const double2 cs = __ldg(&g_circle_tab[b >> 22]);
    const double d = __hiloint2double(0x43300000, (int)(2u * (b & 0x3FFFFFu) + 1u)) - 4503599631564800.0;   // 2^52 + 2^22
    const double t = d * 7.314590396335798e-10;
    const double t2 = t * t;
    const double st = fma(t * t2, fma(t2, 1.0 / 120.0, -1.0 / 6.0), t);
    const double cm = t2 * fma(t2, 1.0 / 24.0, -0.5);   // cos t - 1
    z0 = rad * fma(cs.x, cm, fma(-cs.y, st, cs.x));
    z1 = rad * fma(cs.y, cm, fma(cs.x, st, cs.y));
  }
};

// The 6 stress normals of one cell and step: (xx, yy, zz, xy, xz, yz).  Counters
// (cell, step, call, 0), key (seed_lo, seed_hi): call 0 of the cell gives xx, yy, zz,
// xy; call 1 serves two z planes: at the cell of plane 2m its words 0-1 give xz, yz of
// that cell, words 2-3 those of the cell above it (plane 2m + 1).  `odd`: the cell's
// plane is odd (its call 1 is the one at cell - plane).  KEYS: PhiloxKey or
// PhiloxRoundKeys.
template <typename R, typename KEYS>
__device__ __forceinline__ void cell_normals(uint32_t cell, uint32_t plane, bool odd, uint32_t step, const KEYS& key,
                                             R z[6]) {
  const u32x4 a = philox4x32_10(u32x4{cell, step, 0u, 0u}, key);
  const u32x4 b = philox4x32_10(u32x4{odd ? cell - plane : cell, step, 1u, 0u}, key);
  NormalPair<R>::apply(a.x, a.y, z[0], z[1]);
  NormalPair<R>::apply(a.z, a.w, z[2], z[3]);
  NormalPair<R>::apply(odd ? b.z : b.x, odd ? b.w : b.y, z[4], z[5]);
}

// Shared memory of the marching block.
//  * v: a ring of four velocity planes (three components, one-cell halo in x and y).
//    At plane k the block reads slots of planes k-1, k, k+1 and writes plane k+1's slot
//    before its barrier; that slot was last read by plane k-3, long finished.
//  * z: a ring of three planes of the stress normals that neighbours read (Z_xx, Z_yy,
//    Z_xy, Z_xz, Z_yz; Z_zz is only read by its own cell).  The normals of plane k+1
//    are written before plane k's barrier and read after plane k+1's; the slot was last
//    read at plane k-2.  Each thread keeps its own cell's normals in registers.
constexpr int kRing = 4, kZRing = 3;
template <typename R>
struct RhsSmem {
  R v[kRing][3][HY][HX];
  R z[kZRing][5][HY][HX];
};

// Halo cell h (0 <= h < NHALO) of the tile as (hx, hy) in the padded plane:
// bottom row, top row, left column, right column.
__device__ __forceinline__ void halo_cell(int h, int& hx, int& hy) {
  if (h < HX) {
    hx = h;
    hy = 0;
  } else if (h < 2 * HX) {
    hx = h - HX;
    hy = HY - 1;
  } else if (h < 2 * HX + TY) {
    hx = 0;
    hy = 1 + (h - 2 * HX);
  } else {
    hx = HX - 1;
    hy = 1 + (h - 2 * HX - TY);
  }
}

// The stress normals the tile's neighbours read from its halo cells, 144 per plane:
// Z_yy of the bottom row and Z_xx of the left column (the first Box-Muller pair of
// Philox call 0), Z_xy of the top row and of the right column (the second pair of call
// 0), Z_yz of the top row and Z_xz of the right column (the first pair of call 1).  Task
// tau = 32 warp + lane of warps 0-4 draws one of them: one Philox call and one
// Box-Muller pair per lane, the counter word, word pair and branch chosen per lane, so no
// warp diverges and none does more than one call.  The corners are read by no one.
struct HaloTask {
  int hx, hy;       // position in the padded plane
  int dst;          // z ring array: 0 xx, 1 yy, 2 xy, 3 xz, 4 yz
  uint32_t call;    // Philox counter word 2
  bool hi;          // Box-Muller on words (z, w) rather than (x, y)
  bool second;      // the sine branch rather than the cosine one
};
constexpr int kHaloTasks = 3 * TX + 3 * TY;   // 144
static_assert(kHaloTasks <= NT, "one halo task per thread at most");

__device__ __forceinline__ bool halo_task(int tau, HaloTask& t) {
  if (tau < TX) {                       // bottom row: Z_yy
    t = HaloTask{1 + tau, 0, 1, 0u, false, true};
  } else if (tau < TX + TY) {           // left column: Z_xx
    t = HaloTask{0, 1 + (tau - TX), 0, 0u, false, false};
  } else if (tau < 2 * TX + TY) {       // top row: Z_xy
    t = HaloTask{1 + (tau - TX - TY), HY - 1, 2, 0u, true, true};
  } else if (tau < 3 * TX + TY) {       // top row: Z_yz
    t = HaloTask{1 + (tau - 2 * TX - TY), HY - 1, 4, 1u, false, true};
  } else if (tau < 3 * TX + 2 * TY) {   // right column: Z_xy
    t = HaloTask{HX - 1, 1 + (tau - 3 * TX - TY), 2, 0u, true, true};
  } else if (tau < kHaloTasks) {        // right column: Z_xz
    t = HaloTask{HX - 1, 1 + (tau - 3 * TX - 2 * TY), 3, 1u, false, false};
  } else {
    return false;
  }
  return true;
}

// Philox of the RHS: with RK the round keys of the kernel parameters (read as
// constants), otherwise the key bumped in every call (parameters copied from memory).
template <bool RK>
__device__ __forceinline__ u32x4 rhs_philox(u32x4 c, const GridParams& g) {
  if constexpr (RK)
    return philox4x32_10(c, g.rk);
  else
    return philox4x32_10(c, g.key0, g.key1);
}

// Halo task t at flat cell index `cell` (plane `odd` or even) into slot `slot` of the z
// ring.  Its call-1 normals (Z_xz, Z_yz) on an odd plane are words 2-3 of the call at
// the cell one plane down (`plane` cells per plane).
template <typename R, bool RK>
__device__ __forceinline__ void gen_halo(RhsSmem<R>& sm, int slot, const HaloTask& t, uint32_t cell, uint32_t plane,
                                         bool odd, const GridParams& g, uint32_t step) {
  const bool up = t.call == 1u && odd;
  const u32x4 r = rhs_philox<RK>(u32x4{up ? cell - plane : cell, step, t.call, 0u}, g);
  const bool hi = t.hi || up;
  R c, sn;
  BoxMuller<R>::apply(hi ? r.z : r.x, hi ? r.w : r.y, c, sn);
  sm.z[slot][t.dst][t.hy][t.hx] = t.second ? sn : c;
}

// The own cell's normals of plane p (flat index `cell`) into z[] (registers) and the
// five that neighbours read into slot `slot` of the z ring.  The call-1 words of an
// even plane also hold the next plane's (Z_xz, Z_yz): kept in `next` (valid set) for
// the odd plane that follows in the march; an odd plane without them draws that call
// again at the cell below.
template <typename R, bool RK>
__device__ __forceinline__ void gen_own(RhsSmem<R>& sm, int slot, R (&z)[6], uint32_t cell, int p, uint32_t plane,
                                        const GridParams& g, uint32_t step, int lx, int ly, uint32_t (&next)[2],
                                        bool& valid) {
  const u32x4 a = rhs_philox<RK>(u32x4{cell, step, 0u, 0u}, g);
  BoxMuller<R>::apply(a.x, a.y, z[0], z[1]);
  BoxMuller<R>::apply(a.z, a.w, z[2], z[3]);
  uint32_t w0, w1;
  if ((p & 1) == 0) {
    const u32x4 b = rhs_philox<RK>(u32x4{cell, step, 1u, 0u}, g);
    w0 = b.x;
    w1 = b.y;
    next[0] = b.z;
    next[1] = b.w;
    valid = true;
  } else if (valid) {
    w0 = next[0];
    w1 = next[1];
    valid = false;
  } else {
    const u32x4 b = rhs_philox<RK>(u32x4{cell - plane, step, 1u, 0u}, g);
    w0 = b.z;
    w1 = b.w;
  }
  BoxMuller<R>::apply(w0, w1, z[4], z[5]);
  sm.z[slot][0][ly][lx] = z[0];
  sm.z[slot][1][ly][lx] = z[1];
  sm.z[slot][2][ly][lx] = z[3];
  sm.z[slot][3][ly][lx] = z[4];
  sm.z[slot][4][ly][lx] = z[5];
}

// The velocities around a cell that its right-hand side takes: component c at the cell and its six
// neighbours, and x_xpym = v_x at (+x, -y) and so on.
template <typename R>
struct RhsStencil {
  R c[3], xp[3], xm[3], yp[3], ym[3], zp[3], zm[3];
  R x_xpym, x_xpzm, y_ypxm, y_ypzm, z_zpxm, z_zpym;
};

// Divergence of the momentum flux.  Products ut_a ut_b at the edges, ut_a = (v_a[e] + v_a[e-e_b])/2 and
// ut_b = (v_b[e] + v_b[e-e_a])/2, and squared cell-centre averages, each without its factor 1/4 (in aq);
// the difference of two squares as difference times sum, and every product inside a
// multiply-add: 44 operations per cell where the plain sums take 57 (right-hand side of 128^3 with noise, both
// launches: FP64 702 -> 685 us; FP32 45.7 -> 43.6, with the two planes per turn of the march's loop).
template <typename R>
__device__ __forceinline__ void advection(const RhsStencil<R>& q, R aq, R (&a)[3]) {
  const R axy = q.c[0] + q.ym[0], bxy = q.c[1] + q.xm[1], axz = q.c[0] + q.zm[0], bxz = q.c[2] + q.xm[2];
  const R exy = axy * bxy, eyz = (q.c[1] + q.zm[1]) * (q.c[2] + q.ym[2]);
  const R sx = fma(axz, bxz, exy), sy = exy + eyz, sz = fma(axz, bxz, eyz);
  const R tx = fma(R(2), q.c[0], q.xp[0] + q.xm[0]), dx = q.xp[0] - q.xm[0];
  const R ty = fma(R(2), q.c[1], q.yp[1] + q.ym[1]), dy = q.yp[1] - q.ym[1];
  const R tz = fma(R(2), q.c[2], q.zp[2] + q.zm[2]), dz = q.zp[2] - q.zm[2];
  a[0] = aq * fma(dx, tx, fma(q.yp[0] + q.c[0], q.yp[1] + q.y_ypxm, fma(q.zp[0] + q.c[0], q.zp[2] + q.z_zpxm, -sx)));
  a[1] = aq * fma(dy, ty, fma(q.xp[0] + q.x_xpym, q.xp[1] + q.c[1], fma(q.zp[1] + q.c[1], q.zp[2] + q.z_zpym, -sy)));
  a[2] = aq * fma(dz, tz, fma(q.xp[0] + q.x_xpzm, q.xp[2] + q.c[2], fma(q.yp[1] + q.y_ypzm, q.yp[2] + q.c[2], -sz)));
}

// Advection and right-hand side of cell o: zd, ze are the differences of the diagonal and the off-diagonal
// stress normals, ao the advection of the step before (unless this is the first).
template <typename R, bool NOISE>
__device__ __forceinline__ void rhs_out(const GridParams& g, const RhsStencil<R>& q, const R (&a)[3], const R (&zd)[3],
                                        const R (&ze)[3], R (&ao)[3], bool hist, R* __restrict__ adv,
                                        R* __restrict__ rhs, uint32_t o) {
  const uint32_t nc = (uint32_t)g.ncell;
  const R ce = rhs_c<R>(g).ce, cc = rhs_c<R>(g).cc, sd = rhs_c<R>(g).sd, so = rhs_c<R>(g).so;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (!hist) ao[c] = a[c];
    const R nb = (q.xp[c] + q.xm[c]) + (q.yp[c] + q.ym[c]) + (q.zp[c] + q.zm[c]);
    R s = fma(R(-1.5), a[c], R(0.5) * ao[c]);
    if (NOISE) s = fma(sd, zd[c], fma(so, ze[c], s));
    adv[o + c * nc] = a[c];
    rhs[o + c * nc] = fma(cc, q.c[c], fma(ce, nb, s));
  }
}

// Marching block of TX x TY cells.  A block takes a contiguous range of planes: with
// g.kz > 0 the kz planes of one tile (grid = tiles x ceil(nz / kz)); with g.kz == 0 the
// blocks are persistent (about two per SM) in groups of one block per tile of a tile
// row, and the groups split all tile-row planes evenly.  A range is marched tile by
// tile; each run starts with a prologue of two planes.  Per
// plane: the global loads of the plane after next are issued first, the stress normals
// of the next plane are drawn while they are in flight, then the plane is computed from
// the thread's registers (its own column) and shared memory (its neighbours).
// One run of the marching block: planes k0 .. kend-1 of tile `tile` (tiles x-fastest).
template <typename R, bool NOISE, bool RK>
__device__ __forceinline__ void rhs_run(RhsSmem<R>& sm, const R* __restrict__ v, R* __restrict__ adv,
                                        R* __restrict__ rhs, const GridParams& g, uint32_t step, bool hist,
                                        long long tile, int k0, int kend, int tx, int ty) {
  const int tid = tx + TX * ty;
  const int ntx = (g.nx + TX - 1) / TX;
  // offsets in 32 bits: 3 ncell <= 3 x 512^3 < 2^32
  const uint32_t nc = (uint32_t)g.ncell;
  const uint32_t plane = (uint32_t)g.nx * (uint32_t)g.ny;
  const int lx = tx + 1, ly = ty + 1;
  {
    const int i0 = (int)(tile % ntx) * TX, j0 = (int)(tile / ntx) * TY;
    const int i = i0 + tx, j = j0 + ty;
    const bool active = i < g.nx && j < g.ny;
    // threads past a ragged edge hold the periodic images their neighbours read
    const uint32_t own = (uint32_t)wrapm(i, g.nx) + (uint32_t)g.nx * (uint32_t)wrapm(j, g.ny);
    // the halo cell whose velocities this thread loads, if any
    int hx = 0, hy = 0;
    const bool has_halo = tid < NHALO;
    uint32_t hoff = 0;
    if (has_halo) {
      halo_cell(tid, hx, hy);
      hoff = (uint32_t)wrapm(i0 - 1 + hx, g.nx) + (uint32_t)g.nx * (uint32_t)wrapm(j0 - 1 + hy, g.ny);
    }
    // the halo stress normal this thread draws, if any
    HaloTask ht{0, 0, 0, 0u, false, false};
    const bool hnoise = NOISE && halo_task(tid, ht);
    const uint32_t ncell = hnoise ? (uint32_t)(wrapm(i0 - 1 + ht.hx, g.nx) + g.nx * wrapm(j0 - 1 + ht.hy, g.ny)) : 0u;
    auto load = [&](R (&o)[3], R (&hv)[3], int k) {
      const uint32_t zo = plane * (uint32_t)wrapi(k, g.nz);
      const uint32_t a = zo + own;
#pragma unroll
      for (int c = 0; c < 3; ++c) o[c] = v[a + c * nc];
      if (has_halo) {
        const uint32_t b = zo + hoff;
#pragma unroll
        for (int c = 0; c < 3; ++c) hv[c] = v[b + c * nc];
      }
    };
    auto put = [&](int slot, const R (&o)[3], const R (&hv)[3]) {
#pragma unroll
      for (int c = 0; c < 3; ++c) sm.v[slot][c][ly][lx] = o[c];
      if (has_halo) {
#pragma unroll
        for (int c = 0; c < 3; ++c) sm.v[slot][c][hy][hx] = hv[c];
      }
    };
    // every thread is past the previous run's last plane before its slots are reused
    __syncthreads();
    R vp[3], vc[3], vn[3], vq[3], hq[3];   // own column: planes k-1, k, k+1, k+2; halo k+2
    R zc[6], zn[6], zzp = R(0);            // own normals: plane k, plane k+1, Z_zz of k-1
    load(vp, hq, k0 - 1);
    put(0, vp, hq);
    load(vc, hq, k0);
    put(1, vc, hq);
    load(vn, hq, k0 + 1);
    uint32_t next[2] = {0u, 0u};   // call-1 words of the plane after an even one
    bool nvalid = false;
    if (NOISE) {
      // plane k0-1: only the own cell's Z_zz is read (call 0); plane k0 into slot 1
      {
        const u32x4 a = rhs_philox<RK>(u32x4{own + plane * (uint32_t)wrapi(k0 - 1, g.nz), step, 0u, 0u}, g);
        R zxy;
        BoxMuller<R>::apply(a.z, a.w, zzp, zxy);
      }
      gen_own<R, RK>(sm, 1, zn, own + plane * (uint32_t)k0, k0, plane, g, step, lx, ly, next, nvalid);
      if (hnoise) gen_halo<R, RK>(sm, 1, ht, ncell + plane * (uint32_t)k0, plane, (k0 & 1) != 0, g, step);
    }
    int zs = 1, zsn = 2;   // slots of the normals of planes k, k+1
    // two planes per turn where normals are drawn: the registers that pass from plane to plane are renamed
    // instead of copied (256^3: 269 -> 259 us with noise; without, 171 -> 188)
#pragma unroll(NOISE ? 2 : 1)
    for (int k = k0; k < kend; ++k) {
      const int kk = k - k0;
      const int sp = kk % kRing, sc = (kk + 1) % kRing, sn = (kk + 2) % kRing;
      put(sn, vn, hq);                                         // plane k+1
      const uint32_t o = own + plane * (uint32_t)k;
      R ao[3] = {R(0), R(0), R(0)};
      if (active && hist) {
        ao[0] = adv[o];
        ao[1] = adv[o + nc];
        ao[2] = adv[o + 2 * nc];
      }
      if (k + 1 < kend) load(vq, hq, k + 2);                  // in flight during the noise
      if (NOISE) {
#pragma unroll
        for (int c = 0; c < 6; ++c) zc[c] = zn[c];
        const int p1 = wrapi(k + 1, g.nz);
        const uint32_t pk = plane * (uint32_t)p1;
        gen_own<R, RK>(sm, zsn, zn, own + pk, p1, plane, g, step, lx, ly, next, nvalid);
        if (hnoise) gen_halo<R, RK>(sm, zsn, ht, ncell + pk, plane, (p1 & 1) != 0, g, step);
      }
      __syncthreads();
      if (active) {
        const auto P = sm.v[sp];
        const auto C = sm.v[sc];
        const auto N = sm.v[sn];
        RhsStencil<R> q;
        q.c[0] = vc[0]; q.c[1] = vc[1]; q.c[2] = vc[2];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          q.xp[c] = C[c][ly][lx + 1]; q.xm[c] = C[c][ly][lx - 1];
          q.yp[c] = C[c][ly + 1][lx]; q.ym[c] = C[c][ly - 1][lx];
          q.zp[c] = vn[c]; q.zm[c] = vp[c];
        }
        q.x_xpym = C[0][ly - 1][lx + 1]; q.x_xpzm = P[0][ly][lx + 1];
        q.y_ypxm = C[1][ly + 1][lx - 1]; q.y_ypzm = P[1][ly + 1][lx];
        q.z_zpxm = N[2][ly][lx - 1]; q.z_zpym = N[2][ly - 1][lx];
        R zd[3], ze[3];
        if (NOISE) {
          const auto Z = sm.z[zs];   // plane k: [0] xx, [1] yy, [2] xy, [3] xz, [4] yz
          // divergence of the stress at the faces: Sigma_aa at cells, Sigma_ab on edges
          zd[0] = zc[0] - Z[0][ly][lx - 1]; ze[0] = (Z[2][ly + 1][lx] - zc[3]) + (zn[4] - zc[4]);
          zd[1] = zc[1] - Z[1][ly - 1][lx]; ze[1] = (Z[2][ly][lx + 1] - zc[3]) + (zn[5] - zc[5]);
          zd[2] = zc[2] - zzp; ze[2] = (Z[3][ly][lx + 1] - zc[4]) + (Z[4][ly + 1][lx] - zc[5]);
        }
        R a[3];
        advection<R>(q, rhs_c<R>(g).aq, a);
        rhs_out<R, NOISE>(g, q, a, zd, ze, ao, hist, adv, rhs, o);
      }
      if (NOISE) zzp = zc[2];
      zs = zsn;
      zsn = zsn == kZRing - 1 ? 0 : zsn + 1;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        vp[c] = vc[c];
        vc[c] = vn[c];
        vn[c] = vq[c];
      }
    }
  }
}

// A block takes a contiguous range [lo, hi) of planes: with g.kz > 0 the kz planes
// w = tile * nz + k of one tile (grid = tiles x ceil(nz / kz)); with g.kz == 0 the
// blocks are persistent (whole groups of one block per tile of a tile row, as many as
// the SMs hold at once) and a group's range is of tile-row planes u = row * nz + k, its
// block xt marching tile xt of each row.  A range is marched tile by tile.
template <typename R, bool NOISE>
__global__ void __launch_bounds__(NT, sizeof(R) == 4 ? 2 : 1) k_rhs(const R* __restrict__ v, R* __restrict__ adv,
                                                                      R* __restrict__ rhs, GridParams g,
                                                                      const long long* __restrict__ step_dev,
                                                                      const int* __restrict__ hist_dev) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  RhsSmem<R>& sm = *reinterpret_cast<RhsSmem<R>*>(smem_raw);
  const int ntx = (g.nx + TX - 1) / TX, nty = (g.ny + TY - 1) / TY;
  long long lo, hi;
  int xt = 0;
  if (g.kz > 0) {
    const long long tile = blockIdx.x + (long long)ntx * blockIdx.y;
    lo = tile * g.nz + (long long)blockIdx.z * g.kz;
    hi = min(lo + g.kz, (tile + 1) * g.nz);
  } else {
    // Persistent blocks in groups of ntx, one block per tile of a tile row: the groups
    // split the tile-row planes u = (tile row) nz + k evenly, and the blocks of a group
    // march the same planes side by side, so the halo columns a block reads are rows its
    // neighbours load at about the same time (found in L2, not fetched again).
    const int ngrp = gridDim.x / ntx, grp = blockIdx.x / ntx;
    xt = blockIdx.x - grp * ntx;
    const long long total = (long long)nty * g.nz;
    lo = total * grp / ngrp;
    hi = total * (grp + 1) / ngrp;
  }
  const uint32_t step = (uint32_t)(*step_dev);
  const bool hist = *hist_dev != 0;
  for (long long w = lo; w < hi;) {
    const long long q = w / g.nz;   // the tile (fixed marches) or the tile row (groups)
    const int k0 = (int)(w - q * g.nz);
    const int kend = (int)min((long long)g.nz, k0 + (hi - w));
    w += kend - k0;
    const long long tile = g.kz > 0 ? q : q * ntx + xt;
    rhs_run<R, NOISE, true>(sm, v, adv, rhs, g, step, hist, tile, k0, kend, threadIdx.x, threadIdx.y);
  }
}

// The right-hand side of every member of a batch: persistent blocks split the members'
// concatenated tile-planes evenly; a run never crosses from one member to the next.
template <typename R, bool NOISE>
__global__ void __launch_bounds__(NT, sizeof(R) == 4 ? 2 : 1) k_rhs_batch(const RhsMember<R>* __restrict__ mem,
                                                                            int nm, long long total) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  RhsSmem<R>& sm = *reinterpret_cast<RhsSmem<R>*>(smem_raw);
  const long long lo = total * blockIdx.x / gridDim.x, hi = total * (blockIdx.x + 1) / gridDim.x;
  int mi = 0;   // the member holding w: the last with w0 <= w
  {
    int a = 0, b = nm - 1;
    while (a < b) {
      const int c = (a + b + 1) / 2;
      if (mem[c].w0 <= lo) a = c; else b = c - 1;
    }
    mi = a;
  }
  for (long long w = lo; w < hi;) {
    while (mi + 1 < nm && mem[mi + 1].w0 <= w) ++mi;
    const RhsMember<R>& m = mem[mi];
    const GridParams g = m.g;
    const long long end = mi + 1 < nm ? min(hi, mem[mi + 1].w0) : hi;
    const long long lw = w - m.w0;
    const long long tile = lw / g.nz;
    const int k0 = (int)(lw - tile * g.nz);
    const int kend = (int)min((long long)g.nz, k0 + (end - w));
    w += kend - k0;
    rhs_run<R, NOISE, false>(sm, m.v, m.adv, m.rhs, g, (uint32_t)(*m.step_dev), *m.hist_dev != 0, tile, k0, kend,
                      threadIdx.x, threadIdx.y);
  }
}

// ---------------------------------------------------------------------------
// The right-hand side in two passes, the normals stored in between: one thread per pair of
// cells (planes 2m and 2m + 1 share a Philox call) draws them, one thread per cell takes the
// stencils through L1.  No thread waits for another, no normal is drawn twice and a
// grid of any size spreads over the whole device, where the marching block below needs its 512
// threads' worth of cells per plane and a prologue of two planes.  Used
//  * in FP64, always: the work is bound by the FP64 pipe, and the march draws 9% of its
//    normals twice, for halos;
//  * in FP32, on at most kFlatCells cells where the normals of all fit in the scratch (x sides up to 16, and
//    32) or there are none: elsewhere the march, in runs short enough for every SM (default_plan),
//    takes as long without storing anything.
// Measured with noise, both launches (us), march against stored normals: FP32 18.1 / 10.7 on 32^3, 13.9 /
// 15.3 on 64^3, 23.9 / 26.0 on 96^3, 25.7 / 19.4 on 81^3 (ragged tiles), 43.6 / 56.3 on 128^3, 259 / 386 on
// 256^3; FP64 449 / 24 on 32^3 (eight marching blocks) and 1422 / 700 on 128^3, where half of the
// gain is the cheaper normals above.
// ---------------------------------------------------------------------------
constexpr int kFlatThreads = 128;
constexpr long long kFlatCells = 1ll << 20;

// Normals of the pair `t` of cells: column t mod plane, planes 2 (t / plane) and the next.
template <typename R>
__device__ __forceinline__ void noise_pair(const GridParams& g, uint32_t t, uint32_t step, R* __restrict__ z) {
  const uint32_t plane = (uint32_t)g.nx * (uint32_t)g.ny, nc = (uint32_t)g.ncell;
  const uint32_t m = g.dny.div(g.dnx.div(t));
  const uint32_t c0 = t + m * plane, c1 = c0 + plane;   // t = column + m plane
  if (c0 >= nc) return;
  const PhiloxKey key{g.key0, g.key1};
  const u32x4 b = philox4x32_10(u32x4{c0, step, 1u, 0u}, key);
  const u32x4 a = philox4x32_10(u32x4{c0, step, 0u, 0u}, key);
  R p, q;
  const auto put = [&](uint32_t cell, int first, int second) {
    z[(size_t)first * nc + cell] = p;
    z[(size_t)second * nc + cell] = q;
  };
  NormalPair<R>::apply(a.x, a.y, p, q);
  put(c0, 0, 1);
  NormalPair<R>::apply(a.z, a.w, p, q);
  put(c0, 2, 3);
  NormalPair<R>::apply(b.x, b.y, p, q);
  put(c0, 4, 5);
  if (c1 >= nc) return;
  const u32x4 d = philox4x32_10(u32x4{c1, step, 0u, 0u}, key);
  NormalPair<R>::apply(d.x, d.y, p, q);
  put(c1, 0, 1);
  NormalPair<R>::apply(d.z, d.w, p, q);
  put(c1, 2, 3);
  NormalPair<R>::apply(b.z, b.w, p, q);
  put(c1, 4, 5);
}

// The normals live in the spectrum scratch, which no one needs before the first solve and which
// holds 3.2 to 6 reals per cell, so the right-hand side takes no memory of its own (a buffer for them was
// 40% more device memory in FP64).  Where the 6 of every cell do not fit, slab after slab of planes does: the
// normals of planes k0 - 1 .. k0 + n, then the right-hand sides of planes k0 .. k0 + n - 1.  All at once / in two
// slabs: 298 / 313 us on 96^3 in FP64, 685 / 707 on 128^3.
struct NormalSlabs {
  int n, count;   // planes per slab (all of them: no halo), slabs
  bool whole() const { return count == 1; }
};
NormalSlabs normal_slabs(long long plane, int nz, long long room) {
  const long long fit = room / (6 * plane);   // planes
  if (fit >= nz) return NormalSlabs{nz, 1};
  const int count = (int)((nz + fit - 3) / (fit - 2));
  return NormalSlabs{(nz + count - 1) / count, count};
}

// Normals of cell `t` of the slab of planes k0 - 1 .. k0 + n (periodic).  One cell per thread: two that share a Philox
// call are no faster on large grids (96^3 in FP64 315 us against 313) and slower where a thread's chain of
// operations is what takes the time (24^3 39.8 against 31.8).
template <typename R>
__device__ __forceinline__ void noise_slab_cell(const GridParams& g, uint32_t t, int k0, int n, uint32_t step,
                                                R* __restrict__ z) {
  const uint32_t plane = (uint32_t)g.nx * (uint32_t)g.ny, nc = plane * (uint32_t)(n + 2);
  if (t >= nc) return;
  const int slot = (int)g.dny.div(g.dnx.div(t));
  int k = k0 - 1 + slot;
  k = k < 0 ? k + g.nz : (k >= g.nz ? k - g.nz : k);
  const uint32_t cell = t - (uint32_t)slot * plane + (uint32_t)k * plane;
  R w[6];
  cell_normals<R>(cell, plane, (k & 1) != 0, step, PhiloxKey{g.key0, g.key1}, w);
#pragma unroll
  for (int c = 0; c < 6; ++c) z[(size_t)c * nc + t] = w[c];
}

// The right-hand side of one cell, the same sums as rhs_run's (its comments apply).  z holds the normals of all
// cells or, with slab, those of `slots` planes from plane k0 - 1 on.
template <typename R, bool NOISE>
__device__ __forceinline__ void rhs_cell(const GridParams& g, uint32_t o, bool hist, const R* __restrict__ v,
                                         R* __restrict__ adv, R* __restrict__ rhs, const R* __restrict__ z,
                                         bool slab = false, int k0 = 0, int slots = 0) {
  const uint32_t nc = (uint32_t)g.ncell, nx = g.nx, plane = nx * (uint32_t)g.ny;
  const uint32_t row = g.dnx.div(o), i = o - row * nx;
  const uint32_t k = g.dny.div(row), j = row - k * (uint32_t)g.ny;
  const uint32_t xp = i + 1 == nx ? o - (nx - 1) : o + 1, xm = i == 0 ? o + (nx - 1) : o - 1;
  const uint32_t sy = plane - nx, sz = nc - plane;
  const bool jl = j + 1 == (uint32_t)g.ny, jf = j == 0, kl = k + 1 == (uint32_t)g.nz, kf = k == 0;
  const auto up = [&](uint32_t c) { return jl ? c - sy : c + nx; };
  const auto down = [&](uint32_t c) { return jf ? c + sy : c - nx; };
  const auto above = [&](uint32_t c) { return kl ? c - sz : c + plane; };
  const auto below = [&](uint32_t c) { return kf ? c + sz : c - plane; };
  const uint32_t yp = up(o), ym = down(o), zp = above(o), zm = below(o);
  R ao[3] = {R(0), R(0), R(0)};
  if (hist) {
    ao[0] = adv[o];
    ao[1] = adv[o + nc];
    ao[2] = adv[o + 2 * nc];
  }
  const R *vx = v, *vy = v + nc, *vz = v + 2 * (size_t)nc;
  RhsStencil<R> q;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const R* u = v + c * (size_t)nc;
    q.c[c] = u[o];
    q.xp[c] = u[xp]; q.xm[c] = u[xm];
    q.yp[c] = u[yp]; q.ym[c] = u[ym];
    q.zp[c] = u[zp]; q.zm[c] = u[zm];
  }
  // every load before the first branch, so that all are in flight together
  const bool adv_on = g.advection != 0;
  q.x_xpym = adv_on ? vx[down(xp)] : R(0); q.x_xpzm = adv_on ? vx[below(xp)] : R(0);
  q.y_ypxm = adv_on ? vy[up(xm)] : R(0); q.y_ypzm = adv_on ? vy[below(yp)] : R(0);
  q.z_zpxm = adv_on ? vz[above(xm)] : R(0); q.z_zpym = adv_on ? vz[above(ym)] : R(0);
  R zd[3], ze[3];
  if (NOISE) {
    // the cell in z (o, or o - (k0 - 1) plane), and its neighbours there: a slab does not wrap along z
    const uint32_t zo = slab ? o + plane - (uint32_t)k0 * plane : o, zc = slab ? plane * (uint32_t)slots : nc;
    const uint32_t zd1 = slab ? zo - plane : zm, zu = slab ? zo + plane : zp;
    const uint32_t zxm = zo + (xm - o), zxp = zo + (xp - o), zym = zo + (ym - o), zyp = zo + (yp - o);
    const R *zxx = z, *zyy = z + zc, *zzz = z + 2 * (size_t)zc, *zxy = z + 3 * (size_t)zc, *zxz = z + 4 * (size_t)zc,
            *zyz = z + 5 * (size_t)zc;
    const R xy = zxy[zo], xz = zxz[zo], yz = zyz[zo];
    zd[0] = zxx[zo] - zxx[zxm]; ze[0] = (zxy[zyp] - xy) + (zxz[zu] - xz);
    zd[1] = zyy[zo] - zyy[zym]; ze[1] = (zxy[zxp] - xy) + (zyz[zu] - yz);
    zd[2] = zzz[zo] - zzz[zd1]; ze[2] = (zxz[zxp] - xz) + (zyz[zyp] - yz);
  }
  R a[3] = {R(0), R(0), R(0)};
  if (adv_on) advection<R>(q, rhs_c<R>(g).aq, a);
  rhs_out<R, NOISE>(g, q, a, zd, ze, ao, hist, adv, rhs, o);
}

template <typename R>
__global__ void __launch_bounds__(kFlatThreads / 2) k_noise(GridParams g, R* __restrict__ z,
                                                           const long long* __restrict__ step_dev) {
  noise_pair<R>(g, blockIdx.x * (kFlatThreads / 2) + threadIdx.x, (uint32_t)(*step_dev), z);
}

template <typename R, bool NOISE>
__global__ void __launch_bounds__(kFlatThreads) k_rhs_flat(GridParams g, const R* __restrict__ v, R* __restrict__ adv,
                                                         R* __restrict__ rhs, const R* __restrict__ z,
                                                         const int* __restrict__ hist_dev) {
  const uint32_t o = blockIdx.x * kFlatThreads + threadIdx.x;
  if (o < (uint32_t)g.ncell) rhs_cell<R, NOISE>(g, o, *hist_dev != 0, v, adv, rhs, z);
}

template <typename R>
__global__ void __launch_bounds__(kFlatThreads / 2) k_noise_slab(GridParams g, int k0, int n, R* __restrict__ z,
                                                                const long long* __restrict__ step_dev) {
  noise_slab_cell<R>(g, blockIdx.x * (kFlatThreads / 2) + threadIdx.x, k0, n, (uint32_t)(*step_dev), z);
}
template <typename R>
__global__ void __launch_bounds__(kFlatThreads) k_rhs_slab(GridParams g, int k0, int n,
                                                         const R* __restrict__ v, R* __restrict__ adv,
                                                         R* __restrict__ rhs, const R* __restrict__ z,
                                                         const int* __restrict__ hist_dev) {
  const uint32_t plane = (uint32_t)g.nx * (uint32_t)g.ny, t = blockIdx.x * kFlatThreads + threadIdx.x;
  if (t < plane * (uint32_t)n)
    rhs_cell<R, true>(g, t + (uint32_t)k0 * plane, *hist_dev != 0, v, adv, rhs, z, true, k0, n + 2);
}

// The same over every member of a batch: block u of a member (units of 128 cells or 64 pairs).
template <typename R>
__device__ __forceinline__ int member_of_unit(const RhsMember<R>* __restrict__ mem, int nm, long long w) {
  int a = 0, b = nm - 1;
  while (a < b) {
    const int c = (a + b + 1) / 2;
    if (mem[c].w0 <= w) a = c; else b = c - 1;
  }
  return a;
}
template <typename R>
__global__ void __launch_bounds__(kFlatThreads / 2) k_noise_batch(const RhsMember<R>* __restrict__ mem, int nm,
                                                                 long long total, const BlobMember* __restrict__ all,
                                                                 int n_all) {
  if (blockIdx.x >= total) {   // the blocks past the normals: the members' scalars
    const int e = (int)(blockIdx.x - total) * (kFlatThreads / 2) + threadIdx.x;
    if (e < 3 * n_all) scalars_before(all[e / 3].s.scal, all[e / 3].p.dt, e % 3);
    return;
  }
  const RhsMember<R>& m = mem[member_of_unit(mem, nm, blockIdx.x)];
  noise_pair<R>(m.g, (uint32_t)(blockIdx.x - m.w0) * (kFlatThreads / 2) + threadIdx.x, (uint32_t)(*m.step_dev),
                m.normals);
}
template <typename R, bool NOISE>
__global__ void __launch_bounds__(kFlatThreads) k_rhs_flat_batch(const RhsMember<R>* __restrict__ mem, int nm) {
  const RhsMember<R>& m = mem[member_of_unit(mem, nm, blockIdx.x)];
  const uint32_t o = (uint32_t)(blockIdx.x - m.w0) * kFlatThreads + threadIdx.x;
  if (o < (uint32_t)m.g.ncell) rhs_cell<R, NOISE>(m.g, o, *m.hist_dev != 0, m.v, m.adv, m.rhs, m.normals);
}

long long flat_units(long long plane, int nz) {
  const long long pairs = plane * ((nz + 1) / 2), cells = plane * nz;
  return std::max((cells + kFlatThreads - 1) / kFlatThreads, (2 * pairs + kFlatThreads - 1) / kFlatThreads);
}

template <typename R>
__global__ void k_normals(GridParams g, uint32_t step, R* __restrict__ out) {
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= g.ncell) return;
  R z[6];
  const uint32_t plane = (uint32_t)g.nx * (uint32_t)g.ny;
  cell_normals<R>((uint32_t)c, plane, ((uint32_t)c / plane) & 1u, step, PhiloxKey{g.key0, g.key1}, z);
#pragma unroll
  for (int a = 0; a < 6; ++a) out[a * g.ncell + c] = z[a];
}

template <typename R>
__global__ void k_normal_pairs(int n, const uint32_t* __restrict__ words, double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  R p, q;
  NormalPair<R>::apply(words[2 * i], words[2 * i + 1], p, q);
  out[2 * i] = (double)p;
  out[2 * i + 1] = (double)q;
}

__global__ void k_philox(long long n, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0, uint32_t k1,
                         uint32_t* __restrict__ out) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const u32x4 r = philox4x32_10(u32x4{c0 + (uint32_t)i, c1, c2, c3}, k0, k1);
  out[4 * i + 0] = r.x;
  out[4 * i + 1] = r.y;
  out[4 * i + 2] = r.z;
  out[4 * i + 3] = r.w;
}

// Kahan-compensated per-thread sums, FP64 tree within the block -> partial[comp][block].
template <typename R>
__global__ void k_sum_partial(const R* __restrict__ v, long long n, double* __restrict__ partial) {
  const int comp = blockIdx.y;
  const R* p = v + comp * n;
  double s = 0.0, c = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double y = (double)p[i] - c;
    const double t = s + y;
    c = (t - s) - y;
    s = t;
  }
  __shared__ double red[256];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[comp * gridDim.x + blockIdx.x] = red[0];
}

__global__ void k_sum_final(const double* __restrict__ partial, int np, double* __restrict__ out) {
  const int comp = blockIdx.x;
  double s = 0.0, c = 0.0;
  for (int i = threadIdx.x; i < np; i += blockDim.x) {
    const double y = partial[comp * np + i] - c;
    const double t = s + y;
    c = (t - s) - y;
    s = t;
  }
  __shared__ double red[256];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[comp] = red[0];
}

template <typename A, typename B>
__global__ void k_convert(const A* __restrict__ src, B* __restrict__ dst, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    dst[i] = (B)src[i];
}

__global__ void k_scal_before(double* scal, double dt) {
  const int a = threadIdx.x;
  if (a < 3) scalars_before(scal, dt, a);
}

__global__ void k_scal_after(double* scal, int inertial, long long* step_dev, int* hist_dev) {
  const int a = threadIdx.x;
  if (a < 3) scal[SC_PBAR + a] = scal[SC_K0 + a] + (inertial ? scal[SC_SUMSRC + a] : 0.0);
  if (a == 0) {
    *step_dev += 1;
    *hist_dev = 1;
  }
}

// Peak FMA rate: kFmaChains independent dependent chains x = x * a + b per thread,
// `iters` rounds; a = 1 - 2^-20 and b = 2^-30 keep every value normal and bounded.
// The sum of the chains is stored only if it equals a value it cannot take, so the
// work is not removed.
constexpr int kFmaChains = 8;
template <typename R>
__global__ void __launch_bounds__(256) k_fma_chain(R* __restrict__ out, int iters, R a, R b) {
  R x[kFmaChains];
#pragma unroll
  for (int c = 0; c < kFmaChains; ++c) x[c] = R(1) + R(threadIdx.x + c) * R(1e-3);
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int c = 0; c < kFmaChains; ++c) x[c] = fma(x[c], a, b);
  }
  R sum = R(0);
#pragma unroll
  for (int c = 0; c < kFmaChains; ++c) sum += x[c];
  if (out != nullptr && sum == R(-1)) out[blockIdx.x * blockDim.x + threadIdx.x] = sum;
}

template <typename R>
size_t rhs_smem() { return sizeof(RhsSmem<R>); }

}  // namespace

bool rhs_marches(int precision, int nx, int ny, int nz, bool noise) {
  if (precision == 64) return false;
  const bool whole = (nx / 2 + 1 + 15) / 16 * 16 >= nx;   // the row length of the spectrum
  return (long long)nx * ny * nz > kFlatCells || (noise && !whole);
}

template <typename R>
void explicit_rhs(const GridParams& g, const R* v, R* adv, R* rhs, R* normals, long long room, const long long* step_dev,
                  const int* hist_dev, cudaStream_t st) {
  if (!rhs_marches(8 * sizeof(R), g.nx, g.ny, g.nz, g.kT > 0.0)) {
    const long long plane = (long long)g.nx * g.ny;
    const auto blocks = [](long long threads, int nt) { return (unsigned)((threads + nt - 1) / nt); };
    if (!(g.kT > 0.0)) {
      k_rhs_flat<R, false><<<blocks(g.ncell, kFlatThreads), kFlatThreads, 0, st>>>(g, v, adv, rhs, normals, hist_dev);
      return;
    }
    const NormalSlabs ns = normal_slabs(plane, g.nz, room);
    if (ns.whole()) {
      k_noise<R><<<blocks(plane * ((g.nz + 1) / 2), kFlatThreads / 2), kFlatThreads / 2, 0, st>>>(g, normals, step_dev);
      k_rhs_flat<R, true><<<blocks(g.ncell, kFlatThreads), kFlatThreads, 0, st>>>(g, v, adv, rhs, normals, hist_dev);
      return;
    }
    if constexpr (sizeof(R) == 8) {   // (FP32: whole, see rhs_marches)
      for (int k0 = 0; k0 < g.nz; k0 += ns.n) {
        const int n = std::min(ns.n, g.nz - k0);
        k_noise_slab<R><<<blocks(plane * (n + 2), kFlatThreads / 2), kFlatThreads / 2, 0, st>>>(g, k0, n, normals, step_dev);
        k_rhs_slab<R><<<blocks(plane * n, kFlatThreads), kFlatThreads, 0, st>>>(g, k0, n, v, adv, rhs, normals, hist_dev);
      }
    }
    return;
  }
  if constexpr (sizeof(R) == 4) {
    const dim3 block(TX, TY);
    dim3 grid((g.nx + TX - 1) / TX, (g.ny + TY - 1) / TY, 1);
    if (g.kz > 0) {
      grid.z = (g.nz + g.kz - 1) / g.kz;
    } else {
      // persistent: as many blocks as the SMs hold at once, never more than tile-planes
      static int res = 0;
      if (res == 0) {
        int dev = 0, nsm = 0, per = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        if (g.kT > 0.0)
          cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_rhs<R, true>, NT, rhs_smem<R>());
        else
          cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_rhs<R, false>, NT, rhs_smem<R>());
        res = std::max(1, nsm) * std::max(1, per);
      }
      // whole groups of grid.x blocks (one per tile of a tile row), never more groups
      // than tile-row planes
      const long long rows = (long long)grid.y * g.nz;
      const long long ngrp = std::max<long long>(1, std::min<long long>(res / grid.x, rows));
      grid = dim3((unsigned)(ngrp * grid.x), 1, 1);
    }
    if (g.kT > 0.0)
      k_rhs<R, true><<<grid, block, rhs_smem<R>(), st>>>(v, adv, rhs, g, step_dev, hist_dev);
    else
      k_rhs<R, false><<<grid, block, rhs_smem<R>(), st>>>(v, adv, rhs, g, step_dev, hist_dev);
  }
}

long long rhs_batch_units(int precision, int nx, int ny, int nz) {
  if (precision == 64) return flat_units((long long)nx * ny, nz);
  return (long long)((nx + TX - 1) / TX) * ((ny + TY - 1) / TY) * nz;
}

template <typename R>
void batch_rhs(const RhsMember<R>* members, int nm, long long total, bool noise, cudaStream_t st) {
  if (nm <= 0 || total <= 0) return;
  if constexpr (sizeof(R) == 8) {
    if (noise) {
      k_rhs_flat_batch<R, true><<<(unsigned)total, kFlatThreads, 0, st>>>(members, nm);
    } else {
      k_rhs_flat_batch<R, false><<<(unsigned)total, kFlatThreads, 0, st>>>(members, nm);
    }
  } else {
    static int res = 0;
    if (res == 0) {
      int dev = 0, nsm = 0, per = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_rhs_batch<R, true>, NT, rhs_smem<R>());
      res = std::max(1, nsm) * std::max(1, per);
    }
    const dim3 grid((unsigned)std::min<long long>(res, total)), block(TX, TY);
    if (noise)
      k_rhs_batch<R, true><<<grid, block, rhs_smem<R>(), st>>>(members, nm, total);
    else
      k_rhs_batch<R, false><<<grid, block, rhs_smem<R>(), st>>>(members, nm, total);
  }
}

template <typename R>
void batch_noise(const RhsMember<R>* members, int nm, long long total, const BlobMember* all, int n_all,
                 cudaStream_t st) {
  if (nm <= 0 || total <= 0) {
    batch_scalars_before(all, n_all, st);
    return;
  }
  const int extra = (3 * n_all + kFlatThreads / 2 - 1) / (kFlatThreads / 2);
  k_noise_batch<R><<<(unsigned)(total + extra), kFlatThreads / 2, 0, st>>>(members, nm, total, all, n_all);
}
template void batch_noise<double>(const RhsMember<double>*, int, long long, const BlobMember*, int, cudaStream_t);

template <typename R>
void stress_normals(const GridParams& g, long long step, R* out, cudaStream_t st) {
  const int bs = 256;
  k_normals<R><<<(unsigned)((g.ncell + bs - 1) / bs), bs, 0, st>>>(g, (uint32_t)step, out);
}

void normal_pairs(int precision, int n, const uint32_t* words, double* out, cudaStream_t st) {
  const unsigned blocks = (unsigned)((n + 127) / 128);
  if (precision == 32)
    k_normal_pairs<float><<<blocks, 128, 0, st>>>(n, words, out);
  else
    k_normal_pairs<double><<<blocks, 128, 0, st>>>(n, words, out);
}

void philox_words(long long n, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0, uint32_t k1,
                  uint32_t* out, cudaStream_t st) {
  if (n <= 0) return;
  const int bs = 256;
  k_philox<<<(unsigned)((n + bs - 1) / bs), bs, 0, st>>>(n, c0, c1, c2, c3, k0, k1, out);
}

template <typename R>
void field_sums(const R* v, long long ncell, double* out_dev, double* partial_dev, int npartial, cudaStream_t st) {
  k_sum_partial<R><<<dim3(npartial, 3), 256, 0, st>>>(v, ncell, partial_dev);
  k_sum_final<<<3, 256, 0, st>>>(partial_dev, npartial, out_dev);
}

template <typename R>
void convert_to_double(const R* src, double* dst, long long n, cudaStream_t st) {
  k_convert<R, double><<<1024, 256, 0, st>>>(src, dst, n);
}
template <typename R>
void convert_from_double(const double* src, R* dst, long long n, cudaStream_t st) {
  k_convert<double, R><<<1024, 256, 0, st>>>(src, dst, n);
}

double fma_rate(int precision, int iters, int blocks_per_sm, cudaStream_t st, double* seconds) {
  int dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return -1.0;
  const int blocks = nsm * blocks_per_sm, threads = 256;
  void* out = nullptr;   // k_fma_chain stores nothing through a null pointer
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return -1.0;
  float ms = 0.0f;
  for (int rep = 0; rep < 2; ++rep) {   // the first launch warms up
    cudaEventRecord(e0, st);
    if (precision == 64)
      k_fma_chain<double><<<blocks, threads, 0, st>>>((double*)out, iters, 1.0 - 0x1p-20, 0x1p-30);
    else
      k_fma_chain<float><<<blocks, threads, 0, st>>>((float*)out, iters, 1.0f - 0x1p-20f, 0x1p-30f);
    cudaEventRecord(e1, st);
  }
  const cudaError_t e = cudaEventSynchronize(e1);
  if (e == cudaSuccess) cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (e != cudaSuccess || cudaGetLastError() != cudaSuccess || ms <= 0.0f) return -1.0;
  if (seconds) *seconds = ms * 1e-3;
  return 2.0 * kFmaChains * (double)iters * blocks * threads / (ms * 1e-3);
}

namespace {
std::atomic<bool> g_tables_ready[64];   // by device
int current_device() {
  int dev = 0;
  return cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 ? dev : -1;
}
// The Box-Muller tables, correctly rounded from long double.
struct NormalTables {
  double2 log_tab[kTab], circle[kTab];
  double ln2[34];
  NormalTables() {
    const long double pi = 3.141592653589793238462643383279502884L;
    for (int i = 0; i < kTab; ++i) {
      long double c = 1.0L + (i + 0.5L) / kTab;
      if (i >= kTab / 2) c *= 0.5L;
      const double inv = i == 0 || i == kTab - 1 ? 1.0 : (double)(1.0L / c);   // the intervals next to 1
      log_tab[i] = make_double2(-2.0 * inv, (double)(2.0L * logl((long double)inv)));
      circle[i] = make_double2((double)cosl(2.0L * pi * (i + 0.5L) / kTab), (double)sinl(2.0L * pi * (i + 0.5L) / kTab));
    }
    for (int k = 0; k < 34; ++k) ln2[k] = (double)(2.0L * k * logl(2.0L));
  }
};
}  // namespace

bool grid_prepare(cudaStream_t st, bool fresh) {
  cudaFuncSetAttribute(k_rhs<float, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rhs_smem<float>());
  cudaFuncSetAttribute(k_rhs<float, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rhs_smem<float>());
  cudaFuncSetAttribute(k_rhs_batch<float, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rhs_smem<float>());
  cudaFuncSetAttribute(k_rhs_batch<float, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rhs_smem<float>());
  const int dev = current_device();
  if (fresh && dev >= 0) g_tables_ready[dev].store(false);   // a context after a device reset has none
  if (dev >= 0 && g_tables_ready[dev].load()) return true;
  static const NormalTables tables;   // outlives the copies below
  return cudaMemcpyToSymbolAsync(g_log_tab, tables.log_tab, sizeof(tables.log_tab), 0, cudaMemcpyHostToDevice, st) ==
             cudaSuccess &&
         cudaMemcpyToSymbolAsync(g_circle_tab, tables.circle, sizeof(tables.circle), 0, cudaMemcpyHostToDevice, st) ==
             cudaSuccess &&
         cudaMemcpyToSymbolAsync(g_ln2_tab, tables.ln2, sizeof(tables.ln2), 0, cudaMemcpyHostToDevice, st) ==
             cudaSuccess;
}

void grid_ready() {
  const int dev = current_device();
  if (dev >= 0) g_tables_ready[dev].store(true);
}

void scalars_before_step(double* scal, double dt, double, double, cudaStream_t st) {
  k_scal_before<<<1, 32, 0, st>>>(scal, dt);
}
void scalars_after_step(double* scal, double, double, double, bool inertial, long long* step_dev, int* hist_dev,
                        cudaStream_t st) {
  k_scal_after<<<1, 32, 0, st>>>(scal, inertial ? 1 : 0, step_dev, hist_dev);
}

#define ICM_INST(R)                                                                                          \
  template void explicit_rhs<R>(const GridParams&, const R*, R*, R*, R*, long long, const long long*, const int*, cudaStream_t); \
  template void batch_rhs<R>(const RhsMember<R>*, int, long long, bool, cudaStream_t);                        \
  template void stress_normals<R>(const GridParams&, long long, R*, cudaStream_t);                           \
  template void field_sums<R>(const R*, long long, double*, double*, int, cudaStream_t);                      \
  template void convert_to_double<R>(const R*, double*, long long, cudaStream_t);                             \
  template void convert_from_double<R>(const double*, R*, long long, cudaStream_t);
ICM_INST(float)
ICM_INST(double)
#undef ICM_INST

}  // namespace icm
