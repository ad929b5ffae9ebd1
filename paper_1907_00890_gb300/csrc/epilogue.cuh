// Face epilogues and the interface-geometry pass:
//   * pressure correction u = u* - (dt/rho0) G p (§3.2, the step after Eq. lap_p);
//   * interface geometry per cell: s = mdot (1/rho2 - 1/rho1) |grad C| (Eq. ext_div right-hand side, the
//     source of Eq. lap_p) and n = -grad C / |grad C| (Eq. int_vel), computed once and kept in the plan;
//   * liquid-velocity extension u1e = u - G phi (Eq. jump_subtr) and interface velocity
//     uG = u1e - (mdot_f / rho1) n_f (Eq. int_vel), reading the stored n.
#pragma once

#include "stencil.cuh"

namespace vofp {

__host__ __device__ __forceinline__ size_t total_faces(const GridDev& g) {
  return (size_t)nface(g.nx, g.bcx) * g.ny * g.nz + (size_t)g.nx * nface(g.ny, g.bcy) * g.nz +
         (size_t)g.nx * g.ny * nface(g.nz, g.bcz);
}

// ---- the faces at the low corners of cells --------------------------------------------------------------------------
// A thread of a face kernel takes the x, y and z face at the corner (i, j, k) of cells (the last face of a bounded axis belongs
// to a corner past the last cell).  The cell fields the three share come from L1 after the first, and offsets are 32-bit (a
// plan has fewer than 2^31 cells).  Lanes run over the corners of a plane, row after row; while the blocks are fewer than
// eight an SM, a block takes the faces of one axis, so that a thread's chain is one face's loads and not three.
// (Tiles of 32 x 16 corners, a warp per row, leave lanes idle where a row is no multiple of 32 and make a warp wait for each
// row in turn: extension of 128^3 51.8 us on tiles, 39.1 flat; 20 x 20 x 160 12.0, 9.2; 33 x 33 x 300 30.0, 18.2; variable-density
// pass of 128^3 86, 74.)
constexpr int kCornerThreads = 128;
inline dim3 flat_grid(const GridDev& g) {
  const unsigned bx = (unsigned)((nface(g.nx, g.bcx) * nface(g.ny, g.bcy) + kCornerThreads - 1) / kCornerThreads);
  const unsigned nz = (unsigned)nface(g.nz, g.bcz);
  return dim3(bx, 1, (long)bx * nz < 1216 ? 3 * nz : nz);
}
// This thread's corner and plane (returned), and the axes it takes (a bit each).
__device__ __forceinline__ int flat_corner(const GridDev& g, int& i, int& j, int& axes) {
  const int nz = nface(g.nz, g.bcz), c = blockIdx.x * kCornerThreads + threadIdx.x, fx = nface(g.nx, g.bcx);
  j = c / fx;
  i = c - j * fx;
  axes = 7;
  if (gridDim.z == nz) return blockIdx.z;
  const int a = blockIdx.z / nz;
  axes = 1 << a;
  return blockIdx.z - a * nz;
}

// The velocity correction's other layout: a tile of 32 x kCornerRows corners of one plane, a warp per row, where its rows fill the
// warps; it moves the most bytes an operation, and a warp on one row moves them in fewer sectors (256 x 256 x 128 104 us on
// tiles, 116 flat; 250 x 150 x 128 65.4, 69.2).  Flat: tiles fewer than four an SM (20 x 20 x 160 8.7, 6.8) or a tenth of their
// lanes idle (130 x 130 x 128 41.0, 34.4; 33 x 33 x 300 16.1, 11.3; 200 x 200 x 60, 14% idle, 40.8, 38.4).
constexpr int kCornerRows = 16;
__host__ __device__ __forceinline__ int corner_tiles_x(const GridDev& g) { return (nface(g.nx, g.bcx) + 31) >> 5; }
__host__ __device__ __forceinline__ int corner_tiles_y(const GridDev& g) {
  return (nface(g.ny, g.bcy) + kCornerRows - 1) / kCornerRows;
}
inline dim3 corner_grid(const GridDev& g) {
  return dim3((unsigned)corner_tiles_x(g), (unsigned)corner_tiles_y(g), (unsigned)nface(g.nz, g.bcz));
}
inline bool corner_flat(const GridDev& g) {
  const long tiles = (long)corner_tiles_x(g) * corner_tiles_y(g);
  return tiles * nface(g.nz, g.bcz) < 608 || 10L * nface(g.nx, g.bcx) * nface(g.ny, g.bcy) < 9 * tiles * 32 * kCornerRows;
}

// Double a normal value by its exponent.
__device__ __forceinline__ double twice(double x) {
  return __hiloint2double(__double2hiint(x) + 0x100000, __double2loint(x));
}

// A face: its offset, the cells on both sides (the end cell twice on a bounded end) and what it is: 0 inside or across a
// periodic wrap, -1 an N face, 1 / 2 a low / high D face.
struct FaceRef {
  unsigned off, lo, hi;
  int e;
};
template <int AXIS>
__device__ __forceinline__ bool corner_face(const GridDev& g, int i, int j, int k, FaceRef& r) {
  const int fx = AXIS == 0 ? nface(g.nx, g.bcx) : g.nx;
  const int fy = AXIS == 1 ? nface(g.ny, g.bcy) : g.ny;
  const int fz = AXIS == 2 ? nface(g.nz, g.bcz) : g.nz;
  if (i >= fx || j >= fy || k >= fz) return false;
  const int n = AXIS == 0 ? g.nx : (AXIS == 1 ? g.ny : g.nz), bc = AXIS == 0 ? g.bcx : (AXIS == 1 ? g.bcy : g.bcz);
  const int f = AXIS == 0 ? i : (AXIS == 1 ? j : k);
  const unsigned st = AXIS == 0 ? 1u : (AXIS == 1 ? (unsigned)g.nx : (unsigned)g.nx * g.ny);
  r.off = ((unsigned)k * fy + j) * fx + i;
  r.hi = ((unsigned)k * g.ny + j) * g.nx + i;
  r.lo = r.hi - st;
  r.e = 0;
  if (f == 0) {
    r.lo = bc == VOFP_BC_P ? r.hi + (n - 1) * st : r.hi;
    r.e = bc == VOFP_BC_P ? 0 : (bc == VOFP_BC_NN || bc == VOFP_BC_ND ? -1 : 1);
  } else if (f == n) {
    r.hi = r.lo;
    r.e = bc == VOFP_BC_NN || bc == VOFP_BC_DN ? -1 : 2;
  }
  return VOFP_IN(r.off, (size_t)fx * fy * fz, CHK_FACE_STORE) && VOFP_IN(r.lo, ncells(g), CHK_FACE_LINE) &&
         VOFP_IN(r.hi, ncells(g), CHK_FACE_LINE);
}
// The difference of a cell field across the face (the ghost's sign at a D end; e >= 0).
__device__ __forceinline__ double face_diff(const double* __restrict__ q, const FaceRef& r) {
  double hi = __ldg(q + r.hi), lo = __ldg(q + r.lo);
  if (r.e == 2) hi = 0.0;
  if (r.e == 1) lo = 0.0;
  return one_path(hi) - one_path(lo);
}
// 1 / distance of those values: the centre distance, half the end cell's width at a D end.
template <int AXIS>
__device__ __forceinline__ double face_rdist(const GridDev& g, int k, int e) {
  const double h = AXIS == 0 ? g.rdx
                             : (AXIS == 1 ? g.rdy : __ldg(e <= 0 ? g.rhz + k : g.rdz + (e == 1 ? 0 : g.nz - 1)));
  return e > 0 ? twice(h) : h;
}

// u -= s G p on the faces at a corner; c = s / dx, s / dy, s / (distance across z face k):
// a subtraction and a multiply-add in FP64 on every face.  128^3: 33.2 us, 46.3 with a thread per face and selects around
// FP64 instructions; 320 x 320 x 640: 0.75 ms, 1.29 before.
template <int AXIS>
__device__ __forceinline__ void grad_face(const GridDev& g, const double* __restrict__ p, double* F, double c, int i,
                                          int j, int k) {
  FaceRef r;
  if (!corner_face<AXIS>(g, i, j, k, r) || r.e < 0) return;
  if (AXIS != 2 && r.e > 0) c = twice(c);
  F[r.off] = fma(-c, face_diff(p, r), F[r.off]);
}
__device__ __forceinline__ double grad_sz(const GridDev& g, double s, int k) {
  // (half the end cell's width at a D end)
  const bool dlo = k == 0 && (g.bcz == VOFP_BC_DD || g.bcz == VOFP_BC_DN);
  const bool dhi = k == g.nz && (g.bcz == VOFP_BC_DD || g.bcz == VOFP_BC_ND);
  return s * face_rdist<2>(g, k, dlo ? 1 : (dhi ? 2 : 0));
}
__device__ __forceinline__ void grad_tile(const GridDev& g, const double* __restrict__ p, double* u, double* v, double* w,
                                          double s, double sx, double sy, int tx, int ty, int k) {
  const int i = tx * 32 + (threadIdx.x & 31);
  const double sz = grad_sz(g, s, k);
  for (int q = threadIdx.x >> 5; q < kCornerRows; q += blockDim.x >> 5) {
    const int j = ty * kCornerRows + q;
    grad_face<0>(g, p, u, sx, i, j, k);
    grad_face<1>(g, p, v, sy, i, j, k);
    grad_face<2>(g, p, w, sz, i, j, k);
  }
}
template <bool FLAT>
static __global__ void __launch_bounds__(kCornerThreads) k_grad_update(GridDev g, const double* __restrict__ p, double* u,
                                                                       double* v, double* w, double s, double sx,
                                                                       double sy) {
  if (FLAT) {
    int i, j, axes;
    const int k = flat_corner(g, i, j, axes);
    if (axes & 1) grad_face<0>(g, p, u, sx, i, j, k);
    if (axes & 2) grad_face<1>(g, p, v, sy, i, j, k);
    if (axes & 4) grad_face<2>(g, p, w, grad_sz(g, s, k), i, j, k);
  } else {
    grad_tile(g, p, u, v, w, s, sx, sy, blockIdx.x, blockIdx.y, blockIdx.z);
  }
}

// Interface geometry per cell: s = coef * mdot * |grad C| and n = -grad C / |grad C| (clipped).  Away from the interface
// C is constant and both are zero: a cell whose differences vanish (an integer test; of all 27 values with Youngs' corner
// average) does no FP64 arithmetic, and n is stored only where it is not zero, marked by a bit per cell (`mask`, a word
// per 32 cells of a row).  The FP64 pipe bounds the cells that are left, memory the others: 128^3 droplet (22% of the cells
// with a gradient, 7% with a normal) 44.7 us, 71.7 before; FP32-pair plans 31.4 us, 43.4 before; Youngs' average on 96 x
// 80 x 72 82.5 us, 154 before.
__host__ __device__ __forceinline__ int mask_words(int nx) { return (nx + 31) >> 5; }
__device__ __forceinline__ bool any_bits(double a, double b, double c) {
  return ((__double_as_longlong(a) | __double_as_longlong(b) | __double_as_longlong(c)) << 1) != 0;
}

// Store n where it is not zero and the warp's mask word (lanes are 32 consecutive cells of a row, all active).  A cell
// whose mdot is not finite is marked too: the face means then read it, as they would without the mask.
__device__ __forceinline__ void store_normal(const GridDev& g, bool act, unsigned t, int i, int j, int k, double n0,
                                             double n1, double n2, bool mark, double* __restrict__ nx,
                                             double* __restrict__ ny, double* __restrict__ nz,
                                             unsigned* __restrict__ mask) {
  const bool bit = act && (mark || any_bits(n0, n1, n2));
  const unsigned w = __ballot_sync(0xffffffffu, bit);
  if ((threadIdx.x & 31) == 0 && j < g.ny) mask[((size_t)k * g.ny + j) * mask_words(g.nx) + (i >> 5)] = w;
  if (bit) {
    nx[t] = n0;
    ny[t] = n1;
    nz[t] = n2;
  }
}

// Launch shape: a warp per row of 32 cells, four rows a block, marching kGeoPlanes planes (C of three planes in registers); one
// plane while the blocks are fewer than four an SM, each plane's loads waiting for the last one's.
constexpr int kGeoPlanes = 4;
inline dim3 geometry_grid(const GridDev& g) {
  const unsigned bx = (unsigned)mask_words(g.nx), by = (unsigned)((g.ny + 3) / 4);
  const unsigned bz = (unsigned)((g.nz + kGeoPlanes - 1) / kGeoPlanes);
  return dim3(bx, by, (long)bx * by * bz < 608 ? (unsigned)g.nz : bz);
}
// FF: everything after the C differences in FP32 pairs (reduced-precision plans, central differences) -- scaling,
// |grad C|^2, the reciprocal square root (FP32 seed and one FP32-pair Newton step), s and n -- with integer-pipe
// conversions: 9 FP64 operations instead of some 25, the same to about 1e-14 relative.
template <int MODE, bool FF>
static __global__ void __launch_bounds__(128) k_geometry(GridDev g, const double* __restrict__ C,
                                                        const double* __restrict__ mdot, double coef,
                                                        double* __restrict__ s, double* __restrict__ nx,
                                                        double* __restrict__ ny, double* __restrict__ nz,
                                                        unsigned* __restrict__ mask) {
  const int i = blockIdx.x * 32 + (threadIdx.x & 31), j = blockIdx.y * 4 + (threadIdx.x >> 5);
  const int planes = gridDim.z == g.nz ? 1 : kGeoPlanes;
  const int k0 = blockIdx.z * planes, k1 = k0 + planes < g.nz ? k0 + planes : g.nz;
  const bool act = i < g.nx && j < g.ny;
  const unsigned plane = (unsigned)g.nx * g.ny;
  // in-plane offsets of the neighbours (clamped at bounded ends, wrapped at periodic ones), x fastest
  const int ii = act ? i : 0, jj = act ? j : 0;
  const int xs[3] = {cw(ii - 1, g.nx, g.bcx), ii, cw(ii + 1, g.nx, g.bcx)};
  const int ys[3] = {cw(jj - 1, g.ny, g.bcy) * g.nx, jj * g.nx, cw(jj + 1, g.ny, g.bcy) * g.nx};
  auto at = [&](int k, int a, int b) { return ldg_in(C + (size_t)k * plane, (size_t)(ys[b] + xs[a]), plane, CHK_CELL_LOAD); };
  constexpr int W = MODE == 1 ? 9 : 1;  // values of a plane kept: the 3 x 3 cells, or the middle one
  double m[W], c[W], p[W];
  auto load = [&](int k, double* v) {
#pragma unroll
    for (int q = 0; q < W; ++q) v[q] = MODE == 1 ? at(k, q % 3, q / 3) : at(k, 1, 1);
  };
  load(cw(k0 - 1, g.nz, g.bcz), m);
  load(k0, c);
  for (int k = k0; k < k1; ++k) {
    load(cw(k + 1, g.nz, g.bcz), p);
    double sv = 0.0, n0 = 0.0, n1 = 0.0, n2 = 0.0;
    bool fin = true;
    const unsigned t = (unsigned)k * plane + ys[1] + xs[1];
    if (act) {
      const double md = __ldg(mdot + t);
      fin = finite_bits(md);
      double xm, xp, ym, yp;
      bool flat;
      if (MODE == 1) {
        flat = finite_bits(c[4 % W]);
#pragma unroll
        for (int q = 0; q < W; ++q) flat = flat && same_bits(m[q], c[4 % W]) && same_bits(c[q], c[4 % W]) && same_bits(p[q], c[4 % W]);
      } else {
        xm = at(k, 0, 1), xp = at(k, 2, 1), ym = at(k, 1, 0), yp = at(k, 1, 2);
        flat = same_value(xp, xm) && same_value(yp, ym) && same_value(p[0], m[0]);
      }
      if (FF) {
        if (!flat) {
          const ff gx = ff_split(xp - xm) * ff_split(g.hrdx);
          const ff gy = ff_split(yp - ym) * ff_split(g.hrdy);
          const ff gz = ff_split(p[0] - m[0]) * ff_split(__ldg(g.rzc + k));
          const ff m2 = gx * gx + gy * gy + gz * gz;
          if (m2.hi > 0.0f) {
            const float y0 = rsqrtf(m2.hi);
            const ff y(y0, 0.0f);
            const ff r = y * (ff(1.5f, 0.0f) - ff(0.5f, 0.0f) * (m2 * y * y));  // one Newton step for 1/sqrt(m2)
            sv = wide_of(ff_split(md * coef) * (m2 * r));
            if (fmin(c[0], 1.0 - c[0]) >= 1e-8) {
              n0 = wide_of(-(gx * r));
              n1 = wide_of(-(gy * r));
              n2 = wide_of(-(gz * r));
            }
          }
        }
      } else if (!(flat && fin)) {
        double3 gc;
        if (MODE == 1) {
          gc = youngs_gradient(g, m, c, p, k);
        } else {
          gc = make_double3((xp - xm) * g.hrdx, (yp - ym) * g.hrdy, (p[0] - m[0]) * __ldg(g.rzc + k));
        }
        double3 n;
        sv = md * coef * normal_of(gc, c[4 % W], n);
        n0 = n.x, n1 = n.y, n2 = n.z;
      }
      if (VOFP_IN(t, ncells(g), CHK_CELL_STORE)) s[t] = sv;
    }
    if (nx) store_normal(g, act, t, i, j, k, n0, n1, n2, !fin, nx, ny, nz, mask);
#pragma unroll
    for (int q = 0; q < W; ++q) {
      m[q] = c[q];
      c[q] = p[q];
    }
  }
}

struct ExtArgs {
  GridDev g;
  const double* phi;
  const double* u;
  const double* v;
  const double* w;
  const double* mdot;
  const double* n[3];       // cell normals, stored where the mask has a bit
  const unsigned* mask;     // see k_geometry
  double quarter_inv_rho1;  // 1 / (4 rho1)
  double* ue;
  double* ve;
  double* we;
  double* ug;
  double* vg;
  double* wg;
};

// The cells on both sides of face f along AXIS (the end cell twice on a bounded end).
template <int AXIS>
__device__ __forceinline__ void face_cells(const GridDev& g, int f, int& lo, int& hi) {
  const int n = AXIS == 0 ? g.nx : (AXIS == 1 ? g.ny : g.nz), bc = AXIS == 0 ? g.bcx : (AXIS == 1 ? g.bcy : g.bcz);
  lo = f > 0 ? f - 1 : (bc == VOFP_BC_P ? n - 1 : 0);
  hi = f < n ? f : n - 1;
}
template <int AXIS>
__device__ __forceinline__ void extend_face(const ExtArgs& a, int i, int j, int k) {
  const GridDev& g = a.g;
  FaceRef r;
  if (!corner_face<AXIS>(g, i, j, k, r)) return;
  double ue = __ldg((AXIS == 0 ? a.u : (AXIS == 1 ? a.v : a.w)) + r.off);
  if (r.e >= 0) ue = fma(-face_rdist<AXIS>(g, k, r.e), face_diff(a.phi, r), ue);
  (AXIS == 0 ? a.ue : (AXIS == 1 ? a.ve : a.we))[r.off] = ue;
  if (!a.ug) return;
  // mask bits of the two cells
  int lo, hi;
  face_cells<AXIS>(g, AXIS == 0 ? i : (AXIS == 1 ? j : k), lo, hi);
  const int nw = mask_words(g.nx), il = AXIS == 0 ? lo : i, ih = AXIS == 0 ? hi : i;
  const unsigned rl = (unsigned)(AXIS == 2 ? lo : k) * g.ny + (AXIS == 1 ? lo : j);
  const unsigned rh = (unsigned)(AXIS == 2 ? hi : k) * g.ny + (AXIS == 1 ? hi : j);
  const unsigned wl = __ldg(a.mask + (size_t)rl * nw + (il >> 5)), wh = __ldg(a.mask + (size_t)rh * nw + (ih >> 5));
  const bool bl = (wl >> (il & 31)) & 1u, bh = (wh >> (ih & 31)) & 1u;
  double ug = ue;
  if (bl || bh) {
    // (mean mdot)(mean n) / rho1 = (sum mdot)(sum n) / (4 rho1)
    const double md = __ldg(a.mdot + r.lo) + __ldg(a.mdot + r.hi);
    const double nf = (bl ? __ldg(a.n[AXIS] + r.lo) : 0.0) + (bh ? __ldg(a.n[AXIS] + r.hi) : 0.0);
    ug = fma(-a.quarter_inv_rho1 * md, nf, ue);
  }
  (AXIS == 0 ? a.ug : (AXIS == 1 ? a.vg : a.wg))[r.off] = ug;
}
// 39.1 us at 128^3 (87.8 with a thread per face, six FP64 operations on each and n read everywhere): a face away from the
// interface takes a subtraction and a multiply-add; 126 us at 256 x 256 x 128, 334 before.
static __global__ void __launch_bounds__(kCornerThreads) k_extend_epi(ExtArgs a) {
  int i, j, axes;
  const int k = flat_corner(a.g, i, j, axes);
  if (axes & 1) extend_face<0>(a, i, j, k);
  if (axes & 2) extend_face<1>(a, i, j, k);
  if (axes & 4) extend_face<2>(a, i, j, k);
}

// Variable-density pressure splitting (§3.2, Eq. lap_p and the update after it): u* -= dt (1/rho_f - 1/rho0)
// G p_hat on every face, p_hat = (1 + r) p^n - r p^{n-1} (p^n alone when pm is NULL), rho_f = rho2 + (rho1 -
// rho2) C_f with C_f the mean of C over the face's two cells (its one cell at a bounded end); N faces carry no
// flux.  The constant-coefficient projection of the result with dt/rho0 completes the step.
struct VdArgs {
  GridDev g;
  const double* pn;
  const double* pm;
  double opr, r;        // 1 + dt/dt_prev, dt/dt_prev
  const double* C;
  double half_drho;     // (rho1 - rho2) / 2
  double rho2;
  double dt;
  double dt_over_rho0;
  double cc[2];         // dt (1/rho - 1/rho0) where C = 0, C = 1
  double* u;
  double* v;
  double* w;
};
// Inside a phase (C exactly 0, or 1, on both sides; an integer test) the coefficient is that phase's constant cc[0 / 1]; where
// it is zero -- rho0 is the lighter phase's density -- nothing is read but p and C (a pressure that is not finite is left to
// the arithmetic) and the velocity stays.  128^3 droplet: 74 us, 171 with some 14 FP64 operations on every face.
__device__ __forceinline__ bool ordinary(double a) { return (__double2hiint(a) & 0x7ff00000) < 0x7f000000; }
template <int AXIS>
__device__ __forceinline__ void vd_face(const VdArgs& a, int i, int j, int k) {
  const GridDev& g = a.g;
  FaceRef r;
  if (!corner_face<AXIS>(g, i, j, k, r) || r.e < 0) return;  // (N face: no flux)
  const double cl = __ldg(a.C + r.lo), ch = __ldg(a.C + r.hi);
  double ph = __ldg(a.pn + r.hi), pl = __ldg(a.pn + r.lo), mh = 0.0, ml = 0.0;
  if (a.pm) {
    mh = __ldg(a.pm + r.hi);
    ml = __ldg(a.pm + r.lo);
  }
  const bool gas = ((__double_as_longlong(cl) | __double_as_longlong(ch)) << 1) == 0;
  const bool pure = gas || (same_bits(cl, 1.0) && same_bits(ch, 1.0));
  const double cc = a.cc[gas ? 0 : 1];
  if (pure && (__double_as_longlong(cc) << 1) == 0 && ordinary(ph) && ordinary(pl) && ordinary(mh) && ordinary(ml)) return;
  if (r.e == 2) ph = mh = 0.0;  // (the ghost's sign at a D end, as face_diff)
  if (r.e == 1) pl = ml = 0.0;
  double d = one_path(ph) - one_path(pl);
  if (a.pm) d = fma(a.opr, d, -a.r * (one_path(mh) - one_path(ml)));  // the difference of p_hat
  const double h = face_rdist<AXIS>(g, k, r.e);  // 1 / distance between the values differenced
  double c = cc;
  if (!pure) {
    const double rho_f = fma(a.half_drho, cl + ch, a.rho2);
    c = fma(a.dt, recip_newton(rho_f), -a.dt_over_rho0);  // dt (1/rho_f - 1/rho0)
  }
  double* F = AXIS == 0 ? a.u : (AXIS == 1 ? a.v : a.w);
  F[r.off] = fma(-(h * one_path(c)), d, F[r.off]);
}
static __global__ void __launch_bounds__(kCornerThreads) k_vd_predict(VdArgs a) {
  int i, j, axes;
  const int k = flat_corner(a.g, i, j, axes);
  if (axes & 1) vd_face<0>(a, i, j, k);
  if (axes & 2) vd_face<1>(a, i, j, k);
  if (axes & 4) vd_face<2>(a, i, j, k);
}

}  // namespace vofp
