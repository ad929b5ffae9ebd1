// Volume-of-fluid update with the interface velocity (§3.1): the directional split of Eq. fluxes, each
// one-dimensional step implicit in its own result, then the correction of Eq. final_corr_1 with the implicit
// volume deflation of Eq. final_corr_2:
//
//   C*   (1 - dt du/dx) = C^n  - (f_{i+1/2} - f_{i-1/2}) / dx        f = dt uG C_upwind(C^n)
//   C**  (1 - dt dv/dy) = C*   - (g_{j+1/2} - g_{j-1/2}) / dy        g = dt vG C_upwind(C*)
//   C*** (1 - dt dw/dz) = C**  - (h_{k+1/2} - h_{k-1/2}) / dz_k      h = dt wG C_upwind(C**)
//   C^{n+1} (1 - dt div uG) = C*** - dt (C* du/dx + C** dv/dy + C*** dw/dz)
//
// with du/dx = (uG_{i+1/2} - uG_{i-1/2}) / dx and so on.  The paper takes f, g, h from an MTHINC reconstruction
// it does not restate; these are first-order upwind fluxes (the cell the face velocity comes from; beyond a
// bounded end the boundary cell itself).  All steps run in one FP64 pass that marches through the planes (see
// k_vof_fused); the implicit steps divide through an FP32-seeded reciprocal with one Newton step (relative
// error about 1e-14; the pass is bound by its FP64 arithmetic) and pick upwind cells by an integer sign test.
#include <cmath>
#include <cstdint>

#include "solve_internal.h"
#include "stencil.cuh"

namespace vofp {

// ---- the fused update: one pass marching through the planes -------------------------------------------------
// A CTA owns a column of kVofTX x kVofTY cells and a run of kVofKC planes [k0, k1).  Marching from plane k0 - 1
// to k1 (wrapped on a periodic z axis, clamped on a bounded one -- the upwind rule takes the boundary plane
// itself beyond an end), it forms for each plane m C* (the x step, from C^n in global memory) on its rows plus
// one halo row on each side (recomputed: the y step needs its y neighbours), then C** (the y step, from C* in
// shared memory) into a ring of three planes, and once C** of m is there, the z step and the correction of Eq.
// final_corr_2 for plane m - 1, which needs C** of m - 2, m - 1 and m.  C^n, uG, vG, wG are read and C^{n+1}
// written once per cell (40 bytes) and C*, C** never leave shared memory; the price is the recomputed halo rows
// and planes (x step x (1 + 2/kVofTY)(1 + 2/kVofKC), y step x (1 + 2/kVofKC)).  Cells whose neighbours hold the same C -- the
// inside of each phase -- take no FP64 arithmetic: 128^3 droplet 108 us, 218 when every cell did on tiles of 32 x 16 x 16
// (FP64 pipe 77-84% busy).  Small tiles, for all their halo: the interface makes some tiles long and the others short
// (32 x 16 x 16 cells 166 us, 16 x 4 126, 8 x 16 131, 4 x 8 125); a C that varies in every cell takes 211 us (214 on the
// large tiles without the test), 472 at 250 x 150 x 128 (461).
constexpr int kVofTX = 32, kVofTY = 8, kVofKC = 4;

__device__ __forceinline__ int wrap_clamp(int j, int n, int bc) {
  if (j < 0) return bc == VOFP_BC_P ? j + n : 0;
  if (j >= n) return bc == VOFP_BC_P ? j - n : n - 1;
  return j;
}

// The implicit one-dimensional step of a cell from its value q, its neighbours' values across the low and
// high faces (qm, qp) and the two face velocities; sets dv_rw to the velocity difference over the width.  With dt
// factored out of the fluxes,
//   q_new = (q - dt/w (v_hi q_up(hi) - v_lo q_up(lo))) / (1 - dt/w (v_hi - v_lo)),
// q_up the cell the flow comes from (sign bit of the velocity: a zero velocity of either sign gives a zero flux whichever
// cell is taken), the quotient taken as a product with the Newton reciprocal of the denominator.
__device__ __forceinline__ double vof_step_local(double qm, double q, double qp, double vlo, double vhi, double rw,
                                                 double dt, double& dv_rw) {
  const double qlo = __double2hiint(vlo) >= 0 ? qm : q;  // upwind across the low face
  const double qhi = __double2hiint(vhi) >= 0 ? q : qp;  // upwind across the high face
  const double dtrw = dt * rw, dv = vhi - vlo;
  dv_rw = dv * rw;
  const double num = fma(-dtrw, fma(vhi, qhi, -vlo * qlo), q);
  return num * recip_newton1(fma(-dtrw, dv, 1.0));
}

// The same where C is the same in the three cells (velocities finite): the step returns it, without arithmetic.
__device__ __forceinline__ bool vof_flat(double qm, double q, double qp, double vlo, double vhi) {
  return same_bits(qm, q) && same_value(q, qp) && finite_bits(vlo) && finite_bits(vhi);
}

static __global__ void __launch_bounds__(kVofTX * kVofTY) k_vof_fused(GridDev g, const double* __restrict__ C,
                                                                     const double* __restrict__ uG,
                                                                     const double* __restrict__ vG,
                                                                     const double* __restrict__ wG, double dt,
                                                                     double* __restrict__ out) {
  __shared__ double cs[2][kVofTY + 2][kVofTX];  // C* of the last two planes, with the halo rows
  __shared__ double css[3][kVofTY][kVofTX];     // C** of the last three planes
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int i0 = blockIdx.x * kVofTX, j0 = blockIdx.y * kVofTY;
  const int k0 = blockIdx.z * kVofKC;
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  const int k1 = k0 + kVofKC < nz ? k0 + kVofKC : nz;
  const int i = i0 + tx, j = j0 + ty;
  const bool act = i < nx && j < ny;
  const size_t plane = (size_t)nx * ny;
  const int nyf = nface(ny, g.bcy);
  // local row r of cs <-> grid row j0 - 1 + r (wrapped or clamped at the ends); rows past ny are unused
  auto row_used = [&](int r) { return j0 - 1 + r <= ny && i < nx; };
  const int nxf = nface(nx, g.bcx);
  const int im = wrap_clamp(i - 1, nx, g.bcx), iq = wrap_clamp(i + 1, nx, g.bcx);
  const int ip = (g.bcx == VOFP_BC_P && i + 1 == nx) ? 0 : i + 1;  // the high x face
  const int jp = (g.bcy == VOFP_BC_P && j + 1 == ny) ? 0 : j + 1;  // the high y face
  auto x_cell = [&](int k, int row) {  // C* of cell (i, row, k)
    const size_t cb = ((size_t)k * ny + row) * nx, ub = ((size_t)k * ny + row) * nxf;
    if (!VOFP_IN(cb + nx - 1, plane * nz, CHK_VOF_LOAD) || !VOFP_IN(ub + nxf - 1, nfaces(g, 0), CHK_VOF_LOAD)) return 0.0;
    const double vlo = __ldg(uG + ub + i), vhi = __ldg(uG + ub + ip);
    const double qm = __ldg(C + cb + im), q = __ldg(C + cb + i), qp = __ldg(C + cb + iq);
    if (vof_flat(qm, q, qp, vlo, vhi)) return q;
    double du;
    return vof_step_local(qm, q, qp, vlo, vhi, g.rdx, dt, du);
  };
  auto x_step = [&](int k, double* dst) {  // C* of plane k: each thread its row, rows 0 / 1 the halo rows
    if (row_used(ty + 1)) dst[(ty + 1) * kVofTX + tx] = x_cell(k, wrap_clamp(j, ny, g.bcy));
    if (ty < 2) {
      const int r = ty == 0 ? 0 : kVofTY + 1;
      if (row_used(r)) dst[r * kVofTX + tx] = x_cell(k, wrap_clamp(j0 - 1 + r, ny, g.bcy));
    }
  };
  auto y_step = [&](int k, const double* src, double* dst) {  // C** of plane k from C* in shared memory
    if (!act) return;
    const size_t vb = (size_t)k * nyf * nx + i;
    const double vlo = ldg_in(vG, vb + (size_t)j * nx, nfaces(g, 1), CHK_VOF_LOAD);
    const double vhi = ldg_in(vG, vb + (size_t)jp * nx, nfaces(g, 1), CHK_VOF_LOAD);
    const double qm = src[ty * kVofTX + tx], q = src[(ty + 1) * kVofTX + tx], qp = src[(ty + 2) * kVofTX + tx];
    double v = q, dv;
    if (!vof_flat(qm, q, qp, vlo, vhi)) v = vof_step_local(qm, q, qp, vlo, vhi, g.rdy, dt, dv);
    dst[ty * kVofTX + tx] = v;
  };
  // z step and correction of plane k from C** of planes k - 1, k, k + 1 and C* of plane k
  auto finish = [&](int k, const double* qm, const double* q, const double* qp, const double* c1) {
    if (!act) return;
    const int o = ty * kVofTX + tx;
    const size_t fb = (size_t)j * nx + i;
    const int kp = (g.bcz == VOFP_BC_P && k + 1 == nz) ? 0 : k + 1;
    const double wlo = ldg_in(wG, fb + (size_t)k * plane, nfaces(g, 2), CHK_VOF_LOAD);
    const double whi = ldg_in(wG, fb + (size_t)kp * plane, nfaces(g, 2), CHK_VOF_LOAD);
    const double cs = c1[(ty + 1) * kVofTX + tx], css = q[o];
    double v = css;
    // (all three steps returned C: so does the correction, C (1 - dt div uG) / (1 - dt div uG))
    if (!(vof_flat(qm[o], css, qp[o], wlo, whi) && same_bits(cs, css))) {
      double dw;
      const double c3 = vof_step_local(qm[o], css, qp[o], wlo, whi, __ldg(g.rdz + k), dt, dw);
      const size_t ub = ((size_t)k * ny + j) * nxf;
      const double du =
          (ldg_in(uG, ub + ip, nfaces(g, 0), CHK_VOF_LOAD) - ldg_in(uG, ub + i, nfaces(g, 0), CHK_VOF_LOAD)) * g.rdx;
      const size_t vb = (size_t)k * nyf * nx + i;
      const double dv = (ldg_in(vG, vb + (size_t)jp * nx, nfaces(g, 1), CHK_VOF_LOAD) -
                         ldg_in(vG, vb + (size_t)j * nx, nfaces(g, 1), CHK_VOF_LOAD)) * g.rdy;
      const double F = fma(cs, du, fma(css, dv, c3 * dw));
      v = fma(-dt, F, c3) * recip_newton1(fma(-dt, du + dv + dw, 1.0));
    }
    if (VOFP_IN((size_t)k * plane + fb, plane * nz, CHK_CELL_STORE)) out[(size_t)k * plane + fb] = v;
  };
  for (int m = k0 - 1; m <= k1; ++m) {
    const int s = m - (k0 - 1);  // march step: ring slots s & 1 (C*) and s % 3 (C**)
    const int pm = wrap_clamp(m, nz, g.bcz);
    x_step(pm, &cs[s & 1][0][0]);
    __syncthreads();
    y_step(pm, &cs[s & 1][0][0], &css[s % 3][0][0]);
    __syncthreads();
    if (m >= k0 + 1)
      finish(m - 1, &css[(s + 1) % 3][0][0], &css[(s + 2) % 3][0][0], &css[s % 3][0][0], &cs[(s + 1) & 1][0][0]);
    __syncthreads();
  }
}

}  // namespace vofp

using namespace vofp;

extern "C" int vofp_vof_update(vofp_plan* pl, const double* C, const double* uG, const double* vG, const double* wG,
                               double dt, double* C_out, double* work, void* stream) {
  if (!pl || !C || !uG || !vG || !wG || !C_out || !work || !(dt > 0) || !std::isfinite(dt))
    return VOFP_ERR_INVALID_ARG;
  const GridDev g = grid_dev(pl);
  const size_t cells = (size_t)g.nx * g.ny * g.nz;
  // the workspace [work, work + 2 cells) must not overlap C or C_out (the passes read and write through
  // restrict pointers)
  auto overlaps = [](const double* a, size_t na, const double* b, size_t nb) {
    const uintptr_t a0 = (uintptr_t)a, a1 = a0 + na * sizeof(double);
    const uintptr_t b0 = (uintptr_t)b, b1 = b0 + nb * sizeof(double);
    return a0 < b1 && b0 < a1;
  };
  if (overlaps(work, 2 * cells, C, cells) || overlaps(work, 2 * cells, C_out, cells)) return VOFP_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  // the CTAs read C in their neighbours' columns while others already write theirs: an output over C goes to
  // the workspace first and is copied back
  const bool in_place = overlaps(C_out, cells, C, cells);
  double* dst = in_place ? work : C_out;
  const dim3 grid((unsigned)((g.nx + kVofTX - 1) / kVofTX), (unsigned)((g.ny + kVofTY - 1) / kVofTY),
                  (unsigned)((g.nz + kVofKC - 1) / kVofKC));
  VOFP_LAUNCH(KID_VOF, st, (k_vof_fused<<<grid, dim3(kVofTX, kVofTY), 0, st>>>(g, C, uG, vG, wG, dt, dst)));
  if (in_place && cudaMemcpyAsync(C_out, work, cells * sizeof(double), cudaMemcpyDeviceToDevice, st) != cudaSuccess)
    return VOFP_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? VOFP_OK : VOFP_ERR_CUDA;
}
