// MAC-grid stencils shared by the transform passes and the epilogues (device code).
//
// Face arrays: index i along the face's axis is the low face of cell i; a periodic axis stores n faces,
// a bounded axis n + 1.  Divergence (Eq. mass, discretised): sum over axes of (F_{i+1} - F_i) / w_i.
// Gradient on faces (correction after Eq. lap_p): (p_i - p_{i-1}) / h with h the centre distance; an N
// boundary face is left untouched, a D boundary face uses the ghost value -p (2 p_0 / w_0 low end,
// -2 p_{n-1} / w_{n-1} high end).  |grad C| and n (§3.2 regularised delta, §3.6 Eq. int_vel): central or
// Youngs corner-averaged differences with C copied into ghost cells at bounded ends and wrapped at periodic
// ends; n = -grad C / |grad C|, zero where min(C, 1 - C) < 1e-8 or |grad C| = 0.
// FP64 divisions are replaced by multiplications with reciprocal tables built once per plan (the FP64 pipe
// of the GB300 is narrow; a division costs about ten multiply-adds).
#pragma once

#include "vofp_internal.cuh"

namespace vofp {

struct GridDev {
  int nx, ny, nz;
  int bcx, bcy, bcz;
  double dx, dy;
  double rdx, rdy;    // 1/dx, 1/dy
  double rdx2, rdy2;  // 1/dx^2, 1/dy^2
  double hrdx, hrdy;  // 1/(2 dx), 1/(2 dy): central differences
  const double* dz;   // nz widths
  const double* hz;   // nz + 1 centre distances across z faces (ghost distances at the ends)
  const double* rdz;  // 1/dz
  const double* rhz;  // 1/hz
  const double* rzc;  // 1/(hz[k] + hz[k+1]): central difference in z
  const double* vol;  // cell volume per plane (dx dy dz_k)
  const double* czp;  // residual stencil: coefficient of p_{k+1}, rhz[k+1] / dz_k
  const double* czm;  //   of p_{k-1}, rhz[k] / dz_k
  const double* czc;  //   of p_k, -2 (1/dx^2 + 1/dy^2) - czp - czm
  const float* volf;  // cell volume per plane, FP32
  const ff* dzff;     // dz per plane, FP32 pair
};

__device__ __forceinline__ bool same_bits(double a, double b) {
  return __double_as_longlong(a) == __double_as_longlong(b);
}
__device__ __forceinline__ bool finite_bits(double a) { return (__double2hiint(a) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool same_value(double a, double b) { return same_bits(a, b) && finite_bits(a); }

// Keeps what follows in one copy: the compiler would split FP64 instructions over the cases of a select, and one that is
// predicated off still takes its turn on the FP64 pipe (the correction kernel issued 9.2 FP64 instructions a cell for
// the six it needs).
__device__ __forceinline__ double one_path(double x) {
  asm volatile("" : "+d"(x));
  return x;
}

__host__ __device__ __forceinline__ int nface(int n, int bc) { return n + (bc != VOFP_BC_P); }
__host__ __device__ __forceinline__ size_t ncells(const GridDev& g) { return (size_t)g.nx * g.ny * g.nz; }
// the u, v, w face arrays: nface cells along their own axis
__host__ __device__ __forceinline__ size_t nfaces(const GridDev& g, int axis) {
  return (size_t)(axis == 0 ? nface(g.nx, g.bcx) : g.nx) * (axis == 1 ? nface(g.ny, g.bcy) : g.ny) *
         (axis == 2 ? nface(g.nz, g.bcz) : g.nz);
}

// Neighbour index for a cell field: wrapped on a periodic axis, clamped (ghost copy) on a bounded one.
__device__ __forceinline__ int cw(int i, int n, int bc) {
  if (i < 0) return bc == VOFP_BC_P ? i + n : 0;
  if (i >= n) return bc == VOFP_BC_P ? i - n : n - 1;
  return i;
}

// Divergence of the face field (u, v, w) at cell (i, j, k) plus `addend`, the addend taken into the last
// multiply-add (three subtractions and three multiply-adds in FP64).
__device__ __forceinline__ double divergence_at(const GridDev& g, const double* __restrict__ u,
                                                const double* __restrict__ v, const double* __restrict__ w, int i,
                                                int j, int k, double addend = 0.0) {
  const int nxf = nface(g.nx, g.bcx), nyf = nface(g.ny, g.bcy);
  const size_t ub = ((size_t)k * g.ny + j) * nxf;
  const int ip = (g.bcx == VOFP_BC_P && i + 1 == g.nx) ? 0 : i + 1;
  const size_t nu = nfaces(g, 0), nv = nfaces(g, 1), nw = nfaces(g, 2);
  const double du = ldg_in(u, ub + ip, nu, CHK_FACE_LOAD) - ldg_in(u, ub + i, nu, CHK_FACE_LOAD);
  const size_t vb = (size_t)k * nyf * g.nx + i;
  const int jp = (g.bcy == VOFP_BC_P && j + 1 == g.ny) ? 0 : j + 1;
  const double dv = ldg_in(v, vb + (size_t)jp * g.nx, nv, CHK_FACE_LOAD) -
                    ldg_in(v, vb + (size_t)j * g.nx, nv, CHK_FACE_LOAD);
  const size_t plane = (size_t)g.ny * g.nx;
  const int kp = (g.bcz == VOFP_BC_P && k + 1 == g.nz) ? 0 : k + 1;
  const size_t wb = (size_t)j * g.nx + i;
  const double dw = ldg_in(w, wb + kp * plane, nw, CHK_FACE_LOAD) - ldg_in(w, wb + k * plane, nw, CHK_FACE_LOAD);
  return fma(du, g.rdx, fma(dv, g.rdy, fma(dw, __ldg(g.rdz + k), addend)));
}

__device__ __forceinline__ double cval(const GridDev& g, const double* __restrict__ C, int i, int j, int k) {
  i = cw(i, g.nx, g.bcx);
  j = cw(j, g.ny, g.bcy);
  k = cw(k, g.nz, g.bcz);
  return ldg_in(C, ((size_t)k * g.ny + j) * g.nx + i, ncells(g), CHK_CELL_LOAD);
}

// Youngs' corner average at the middle of the 3 x 3 cells (x fastest) m, c, p of planes k - 1, k, k + 1: differences first
// (C near 0 or 1 loses nothing in them), then the (1, 2, 1) / 4 filter of both transverse directions by the sums of the
// corner (weight 1), edge (2) and middle (4) differences; on a uniform axis the two one-sided differences add up to one
// over two cells.
__device__ __forceinline__ double3 youngs_gradient(const GridDev& g, const double* m, const double* c, const double* p,
                                                   int k) {
  const double x = fma(4.0, c[5] - c[3], fma(2.0, ((c[2] - c[0]) + (c[8] - c[6])) + ((m[5] - m[3]) + (p[5] - p[3])),
                                             ((m[2] - m[0]) + (m[8] - m[6])) + ((p[2] - p[0]) + (p[8] - p[6]))));
  const double y = fma(4.0, c[7] - c[1], fma(2.0, ((c[6] - c[0]) + (c[8] - c[2])) + ((m[7] - m[1]) + (p[7] - p[1])),
                                             ((m[6] - m[0]) + (m[8] - m[2])) + ((p[6] - p[0]) + (p[8] - p[2]))));
  auto z = [](const double* lo, const double* hi) {
    return fma(4.0, hi[4] - lo[4], fma(2.0, ((hi[1] - lo[1]) + (hi[7] - lo[7])) + ((hi[3] - lo[3]) + (hi[5] - lo[5])),
                                       ((hi[0] - lo[0]) + (hi[2] - lo[2])) + ((hi[6] - lo[6]) + (hi[8] - lo[8]))));
  };
  return make_double3(0.03125 * g.rdx * x, 0.03125 * g.rdy * y,
                      0.03125 * fma(z(m, c), __ldg(g.rhz + k), z(c, p) * __ldg(g.rhz + k + 1)));
}

// Cell-centred gradient of C: mode 0 central, mode 1 Youngs.
__device__ __forceinline__ double3 grad_c_at(const GridDev& g, const double* __restrict__ C, int i, int j, int k,
                                             int mode) {
  double3 r;
  if (mode == 0) {
    r.x = (cval(g, C, i + 1, j, k) - cval(g, C, i - 1, j, k)) * g.hrdx;
    r.y = (cval(g, C, i, j + 1, k) - cval(g, C, i, j - 1, k)) * g.hrdy;
    r.z = (cval(g, C, i, j, k + 1) - cval(g, C, i, j, k - 1)) * __ldg(g.rzc + k);
    return r;
  }
  double q[3][9];
  for (int b = -1; b <= 1; ++b)
    for (int a = 0; a < 9; ++a) q[b + 1][a] = cval(g, C, i + a % 3 - 1, j + a / 3 - 1, k + b);
  return youngs_gradient(g, q[0], q[1], q[2], k);
}

constexpr long long kClipHigh = 0x3feffffffaa19c47ll;  // the bits of the largest C with 1 - C >= 1e-8

// 1 / sqrt(x) for x > 0: an FP32 seed of x's mantissa (exponent halved in integers, relative error below 2^-21) and one
// third-order step, y (1 + e/2 + 3 e^2/8) with e = 1 - x y^2: error 5 e^3 / 16, five FP64 operations.
__device__ __forceinline__ double rsqrt_step(double x) {
  const int hi = __double2hiint(x), e = (hi >> 20) - 1023;
  if (e < -900 || e > 900) return rsqrt(x);  // (near the ends of the range, infinities and NaN)
  const int odd = e & 1;
  const unsigned m = __funnelshift_l((unsigned)__double2loint(x), (unsigned)hi, 3) & 0x7fffffu;
  double y = f64_of_bits(rsqrtf(__uint_as_float(m | ((unsigned)(127 + odd) << 23))));
  y = __hiloint2double(__double2hiint(y) - (((e - odd) / 2) << 20), __double2loint(y));
  const double r = fma(-(x * y), y, 1.0);
  return fma(y * r, fma(0.375, r, 0.5), y);
}

// |grad C| and the unit normal n = -grad C / |grad C| (zero where clipped) from a cell's gradient and its C.
__device__ __forceinline__ double normal_of(double3 gc, double c, double3& n) {
  const double m2 = fma(gc.x, gc.x, fma(gc.y, gc.y, gc.z * gc.z));
  n = make_double3(0.0, 0.0, 0.0);
  if (__double_as_longlong(m2) == 0) return 0.0;
  const double r = rsqrt_step(m2);
  // min(C, 1 - C) >= 1e-8 by the bits of C: 1 - C is exact there, and kClipHigh the last such C
  const long long b = __double_as_longlong(c);
  if (b >= __double_as_longlong(1e-8) && b <= kClipHigh) {
    n.x = -gc.x * r;
    n.y = -gc.y * r;
    n.z = -gc.z * r;
  }
  return m2 * r;
}

}  // namespace vofp
