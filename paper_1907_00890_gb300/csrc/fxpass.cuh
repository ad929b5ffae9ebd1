// Host side of the fixed-point transform passes (fxfft.cuh): which kernel, tile and scaling a launch takes.  Included
// by one translation unit per spectrum type (the kernels compile side by side).
#pragma once

#include "fxfft.cuh"
#include "solve_internal.h"

namespace vofp {

template <typename K>
static void fx_allow_smem(K kern) {
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
}

// The kernel of a pass for a tile: compiled for lines of 32 .. 512 samples at their usual tile width, else the run-time
// one.
template <typename T>
static int fx_lgn(const FxTables& f) {
  const int n = f.fd.n;
  // (FP32-pair plans leave the grids of one-warp tiles of 32 samples to the floating-point passes, see fx_takes)
  if ((n & (n - 1)) || n < (std::is_same<T, double>::value ? 32 : 64) || n > 512) return 0;
  const int lgn = 31 - __builtin_clz((unsigned)n);
  return f.lgB == fx_ct_lgB(lgn) ? lgn : 0;  // (the stages are the plan's: see fx_radix)
}
typedef void (*FxXFwd)(const XArgs, const FxTables);
typedef void (*FxYPass)(const YArgs, const FxTables);
typedef void (*FxXInv)(const XInvArgs, const FxTables);
template <typename T, int LGN>
static FxXFwd fx_xfwd_mode(int mode) {
  switch (mode) {
    case RHS_F: return k_xfwd_fx<T, RHS_F, LGN>;
    case RHS_DIV: return k_xfwd_fx<T, RHS_DIV, LGN>;
    case RHS_DIV_STEFAN: return k_xfwd_fx<T, RHS_DIV_STEFAN, 0>;
    case RHS_RESID:  // (a refinement plan's)
      if constexpr (std::is_same<T, ff>::value) return k_xfwd_fx<T, RHS_RESID, LGN>;
      else return nullptr;
    default: return nullptr;
  }
}
template <typename T>
static FxXFwd fx_xfwd_kernel(int mode, int lgn) {
  switch (lgn) {
    case 5:
      if constexpr (std::is_same<T, double>::value) return fx_xfwd_mode<T, 5>(mode);
      else return nullptr;
    case 6: return fx_xfwd_mode<T, 6>(mode);
    case 7: return fx_xfwd_mode<T, 7>(mode);
    case 8: return fx_xfwd_mode<T, 8>(mode);
    case 9: return fx_xfwd_mode<T, 9>(mode);
    default: return fx_xfwd_mode<T, 0>(mode);
  }
}
template <typename T>
static FxYPass fx_ypass_kernel(bool inv, int lgn) {
  switch (lgn) {
    case 5:
      if constexpr (std::is_same<T, double>::value) return inv ? k_ypass_fx<T, true, 5> : k_ypass_fx<T, false, 5>;
      else return nullptr;
    case 6: return inv ? k_ypass_fx<T, true, 6> : k_ypass_fx<T, false, 6>;
    case 7: return inv ? k_ypass_fx<T, true, 7> : k_ypass_fx<T, false, 7>;
    case 8: return inv ? k_ypass_fx<T, true, 8> : k_ypass_fx<T, false, 8>;
    case 9: return inv ? k_ypass_fx<T, true, 9> : k_ypass_fx<T, false, 9>;
    default: return inv ? k_ypass_fx<T, true, 0> : k_ypass_fx<T, false, 0>;
  }
}
template <typename T, bool PLAIN>
static FxXInv fx_xinv_kernel(int lgn) {
  switch (lgn) {
    case 5:
      if constexpr (std::is_same<T, double>::value) return k_xinv_fx<T, 5, PLAIN>;
      else return nullptr;
    case 6: return k_xinv_fx<T, 6, PLAIN>;
    case 7: return k_xinv_fx<T, 7, PLAIN>;
    case 8: return k_xinv_fx<T, 8, PLAIN>;
    case 9: return k_xinv_fx<T, 9, PLAIN>;
    default: return k_xinv_fx<T, 0, PLAIN>;
  }
}
// (FP64 plans only ever write the potential)
template <typename T>
static FxXInv fx_xinv_kernel(int lgn, bool plain) {
  if constexpr (!std::is_same<T, double>::value)
    if (!plain) return fx_xinv_kernel<T, false>(lgn);
  return plain ? fx_xinv_kernel<T, true>(lgn) : nullptr;
}
template <typename T>
void init_fx_attributes() {
  for (int lgn : {0, 5, 6, 7, 8, 9}) {
    for (int mode : {RHS_F, RHS_DIV, RHS_DIV_STEFAN, RHS_RESID})
      if (fx_xfwd_kernel<T>(mode, lgn)) fx_allow_smem(fx_xfwd_kernel<T>(mode, lgn));
    for (bool inv : {false, true})
      if (fx_ypass_kernel<T>(inv, lgn)) fx_allow_smem(fx_ypass_kernel<T>(inv, lgn));
    for (bool plain : {true, false})
      if (fx_xinv_kernel<T>(lgn, plain)) fx_allow_smem(fx_xinv_kernel<T>(lgn, plain));
  }
}

// Tables and tile (at least 2^least lines) of axis ax and the kernel for it (*lgn: a compiled-in length, or 0 for the
// run-time one, which `rt` asks for); false: the axis' length has no fixed-point form.
template <typename T>
static bool fx_tables(const vofp_plan* pl, int ax, int least, bool rt, FxTables* f, int* lgn) {
  const AxisDev& a = pl->ax[ax];
  if (!a.twfx || !fx_desc(a.fd, &f->fd)) return false;
  f->tw = (const fxtw*)a.twfx;
  f->quart = (const fxq*)a.quartfx;
  f->lgB = fx_lgB(a.n, fx_tiles8(pl->n[0], pl->n[1], pl->n[2], ax == 1), least);
  *lgn = rt ? 0 : fx_lgn<T>(*f);
  // (the run-time kernels are bound to kFxMaxThreads: eight lines of 512 samples are a compiled-in kernel's tile only)
  while (fx_threads(a.n, f->lgB) > fx_bound(*lgn)) --f->lgB;
  f->st = (1 << f->lgB) + (ax == 0 ? 1 : 0);
  return true;
}

template <typename T>
bool fx_xfwd(vofp_plan* pl, int mode, const XArgs& xa, cudaStream_t st) {
  FxTables f;
  const long npairs = ((long)pl->n[1] * pl->n[2] + 1) / 2;
  int lgn;
  if (!fx_tables<T>(pl, 0, 0, mode == RHS_DIV_STEFAN, &f, &lgn)) return false;
  const int grid = (int)((npairs + (1 << f.lgB) - 1) >> f.lgB), th = fx_threads(f.fd, f.lgB, grid);
  const size_t sm = fx_smem(f.fd, f.lgB, f.st);
  const int kid = mode == RHS_F ? KID_XFWD : (mode == RHS_DIV ? KID_XFWD_DIV : (mode == RHS_RESID ? KID_RESID : KID_XFWD_DIVSTEF));
  const FxXFwd kern = mode == RHS_STEFAN ? nullptr : fx_xfwd_kernel<T>(mode, lgn);
  if (!kern) return false;
  VOFP_LAUNCH(kid, st, (kern<<<grid, th, sm, st>>>(xa, f)));
  return true;
}
template <typename T>
bool fx_ypass(vofp_plan* pl, const YArgs& ya, bool inv, cudaStream_t st) {
  FxTables f;
  int lgn;
  const int nx = pl->n[0], nz = pl->n[2];
  if (!fx_tables<T>(pl, 1, 1, false, &f, &lgn)) return false;
  const dim3 grid((nx + (2 << f.lgB) - 1) / (2 << f.lgB), nz);
  const int th = fx_threads(f.fd, f.lgB, (long)grid.x * nz);
  const size_t sm = fx_smem(f.fd, f.lgB, f.st);
  VOFP_LAUNCH(inv ? KID_YINV : KID_YFWD, st, (fx_ypass_kernel<T>(inv, lgn)<<<grid, th, sm, st>>>(ya, f)));
  return true;
}
template <typename T>
bool fx_xinv(vofp_plan* pl, const XInvArgs& xi, cudaStream_t st) {
  FxTables f;
  const long npairs = ((long)pl->n[1] * pl->n[2] + 1) / 2;
  int lgn;
  if (!fx_tables<T>(pl, 0, 0, false, &f, &lgn)) return false;
  const int grid = (int)((npairs + (1 << f.lgB) - 1) >> f.lgB), th = fx_threads(f.fd, f.lgB, grid);
  const size_t sm = fx_smem(f.fd, f.lgB, f.st);
  const FxXInv kern = fx_xinv_kernel<T>(lgn, xi.p && !xi.accumulate && !xi.mean_out && !xi.d2_out);
  if (!kern) return false;
  VOFP_LAUNCH(KID_XINV, st, (kern<<<grid, th, sm, st>>>(xi, f)));
  return true;
}

}  // namespace vofp
