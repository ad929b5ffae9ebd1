// z pass of a periodic axis with equal cell widths h: every system is a circulant one,
//     a (p_{k-1} - (2 + mu) p_k + p_{k+1}) = s r_k,   a = 1 / h^2,  mu = -(lx + ly) h^2 >= 0  (indices mod nz),
// and its operator factors into two first-order recurrences around the ring,
//     -(a / rho) (1 - rho E^-1) (1 - rho E),   rho = 1 / (1 + mu/2 + sqrt(mu + mu^2/4)) < 1,
// with E the shift by one row: y_k = rho y_{k-1} + r_k going up, x_k = rho x_{k+1} + y_k going down, each closed
// by its wrap-around value Y = Y' / (1 - rho^nz) (Y' from a zero start), and p = -(s rho / a) x.  No divisions, no
// factor table per row, five numbers per distinct eigenvalue pair (written at plan time); rho is relatively
// accurate and so is 1 - rho^nz (expm1 / log1p), so the error grows like 1 / (1 - rho) where eliminating the rows
// loses mu in 2 + mu, like 1 / (1 - rho)^2.
//
// The tile: `ti` neighbouring columns x all rows in shared memory, the rows cut into 256 / ti segments, one per
// thread; each recurrence runs per segment from zero, the segments' ends are folded in order (and around), and the
// segment is run again from its true start: five operations a value.  What bounds it is the FP64 pipe (two
// operations per SM and cycle): 320 x 320 x 640 in FP64, 65.5 M values, has a floor of 0.52 ms and takes 1.02 ms;
// the general column solver (divisions, one thread a column, 4 columns a block) took 39.9 ms there.  Unequal widths
// and fewer than 3 rows keep that solver.
// ti is the widest of 32, 16, 8, 4 whose tile leaves two blocks on an SM (110 KB): one block per SM would stop the
// SM's memory traffic while it computes.
#pragma once

#include "zsolve.cuh"

namespace vofp {

// Per distinct eigenvalue pair, in the plan's arithmetic type.
template <typename T>
struct ZCirc {
  T rho, pw, pwl;  // rho; rho^L and rho^(rows of the last segment)
  T g;             // 1 / (1 - rho^nz)
  T sc;            // -s rho / a
};

struct ZCircArgs {
  int Ux, bcx, bcy;
  int ti, L;          // columns per tile, rows per segment (the last one may be shorter, or empty)
  const void* tab;    // ZCirc<T>[Uy][Ux]
  const int* lowcut;  // refinement plans: column i of row j is a low mode iff i < lowcut[j]; NULL: none
};

constexpr int kZCircThreads = 256;
inline int zcirc_ti(int nz, size_t elem) {
  for (int ti = 32; ti > 4; ti >>= 1)
    if ((size_t)nz * ti * elem <= 96 * 1024) return ti;
  return 4;
}
inline int zcirc_rows(int nz, int ti) { return (nz + kZCircThreads / ti - 1) / (kZCircThreads / ti); }
// the tile, then the segments' ends (one per thread)
inline size_t zcirc_smem(int nz, int ti, size_t elem) { return ((size_t)nz * ti + kZCircThreads) * elem; }

// Factors of the pair with eigenvalue sum lam (not the singular one); `rows` and `last`: full and last segment.
__device__ __forceinline__ ZCirc<double> zcirc_factors(double lam, double h, double scale, int nz, int rows,
                                                       int last) {
  const double mu = -lam * h * h;
  const double q = sqrt(fma(0.25 * mu, mu, mu));
  const double lg = log1p(-(mu / (0.5 * mu + q)));  // log rho, from 1 - rho
  ZCirc<double> f;
  f.rho = 1.0 / (1.0 + 0.5 * mu + q);
  f.pw = exp(rows * lg);
  f.pwl = exp(last * lg);
  f.g = -1.0 / expm1(nz * lg);
  f.sc = -scale * f.rho * h * h;
  return f;
}

template <typename T>
static __global__ void k_zcirc_table(ZArgs a, ZCircArgs c, int Uy, double h, ZCirc<T>* tab) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= c.Ux * Uy) return;
  const int ux = t % c.Ux, uy = t / c.Ux;
  const int qx = c.bcx == VOFP_BC_P ? (ux ? 2 * ux - 1 : 0) : ux;
  const int qy = c.bcy == VOFP_BC_P ? (uy ? 2 * uy - 1 : 0) : uy;
  if (!VOFP_IN(qx, a.nx, CHK_Z_TABLE) || !VOFP_IN(qy, a.ny, CHK_Z_TABLE)) return;
  ZCirc<double> f = {0.0, 0.0, 0.0, 0.0, 0.0};  // (the singular pair: its column is solved by zcirc_singular)
  if (!(a.singular && t == 0)) {
    const int last = a.nz - (a.nz - 1) / c.L * c.L;
    f = zcirc_factors(a.lamx[qx] + a.lamy[qy], h, a.scale, a.nz, c.L, last);
  }
  tab[t] = {(T)f.rho, (T)f.pw, (T)f.pwl, (T)f.g, (T)f.sc};
}
static __global__ void k_zcirc_low_table(ZArgs a, const int2* __restrict__ modes, int nlow, double h,
                                         ZCirc<double>* tab) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nlow) return;
  const int2 md = modes[t];
  if (!VOFP_IN(md.x, a.nx, CHK_Z_TABLE) || !VOFP_IN(md.y, a.ny, CHK_Z_TABLE)) return;
  if (!(a.singular && md.x == 0 && md.y == 0))
    tab[t] = zcirc_factors(a.lamx[md.x] + a.lamy[md.y], h, a.scale, a.nz, 1, 1);
}

// The mean mode of a singular operator (mu = 0) by one warp, in FP64: remove the mean of its right-hand side (the
// compatibility defect), sum it up to the flux G_k + c through the ring (c such that the fluxes sum to zero), sum
// that to p and remove p's mean.  Lane l holds rows [l R, (l + 1) R).
template <typename TS>
__device__ void zcirc_singular(const ZArgs& a, TS* col, size_t plane, int lane) {
  const int nz = a.nz, R = (nz + 31) >> 5;
  const int k0 = lane * R < nz ? lane * R : nz;
  const int k1 = k0 + R < nz ? k0 + R : nz;
  const double h = __ldg(a.dz);
  const double sc = a.scale * h * h;
  double s = 0.0;
  for (int k = k0; k < k1; ++k) s += (double)col[k * plane];
  const double own = s;
  const double defect = warp_sum(s) / nz;
  if (lane == 0 && a.info) a.info->compat_defect = defect * a.scale;
  auto before = [&](double v) {  // sum of v over the lanes below
    double t = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double u = shfl_up_t(t, o);
      if (lane >= o) t += u;
    }
    return t - v;
  };
  const double G0 = before(own - defect * (k1 - k0));
  double G = G0, sg = 0.0;
  for (int k = k0; k < k1; ++k) {
    G += (double)col[k * plane] - defect;
    sg += G;
  }
  const double c = -warp_sum(sg) / nz;
  // p_k = sum over m < k of (G_m + c)
  const double P0 = before(fma(c, (double)(k1 - k0), sg));
  double P = P0, sp = 0.0;
  G = G0;
  for (int k = k0; k < k1; ++k) {
    sp += P;
    G += (double)col[k * plane] - defect;
    P += G + c;
  }
  const double mean = warp_sum(sp) / nz;
  bool bad = false;
  P = P0;
  G = G0;
  for (int k = k0; k < k1; ++k) {
    const double v = (P - mean) * sc;
    G += (double)col[k * plane] - defect;
    P += G + c;
    col[k * plane] = (TS)v;
    if (a.info) bad |= !isfinite(v);
  }
  if (bad) atomicOr(&a.info->nonfinite, 1u);
}

// ti columns from i0 = bx ti of y index by.  Thread t works on column t % ti, in the recurrences on the rows of
// segment t / ti.
template <typename T>
__device__ __forceinline__ void zcirc_block(const ZArgs& a, const ZCircArgs& z, int bx, int by,
                                            unsigned char* smem_raw) {
  if (block_skipped(a.skip_conv, a.skip_k, a.tol2)) return;
  const int TI = z.ti, nz = a.nz, NS = kZCircThreads / TI, L = z.L;
  const int c = threadIdx.x & (TI - 1), sg = threadIdx.x / TI;
  const int i = bx * TI + c, j = by;
  const size_t plane = (size_t)a.nx * a.ny;
  T* yv = reinterpret_cast<T*>(smem_raw) + c;                        // this column of the tile (stride TI)
  T* ends = reinterpret_cast<T*>(smem_raw) + (size_t)nz * TI + c;    // this column's segment ends (stride TI)
  const bool sing = a.singular && j == 0 && i == 0;
  const bool live = i < a.nx && !sing && !(z.lowcut && i < __ldg(z.lowcut + j)) &&
                    VOFP_IN((size_t)j * a.nx + i, plane, CHK_Z_COLUMN);
  T* col = reinterpret_cast<T*>(a.S) + (size_t)j * a.nx + (i < a.nx ? i : 0);
  const ZCirc<T> f = reinterpret_cast<const ZCirc<T>*>(
      z.tab)[(size_t)distinct_index(j, z.bcy) * z.Ux + distinct_index(i < a.nx ? i : 0, z.bcx)];
  if (live) {  // eight rows per thread in flight
    constexpr int UL = 8;
    for (int kb = sg; kb < nz; kb += UL * NS) {
      T r[UL];
#pragma unroll
      for (int u = 0; u < UL; ++u)
        if (kb + u * NS < nz) r[u] = col[(size_t)(kb + u * NS) * plane];
#pragma unroll
      for (int u = 0; u < UL; ++u)
        if (kb + u * NS < nz) yv[(kb + u * NS) * TI] = r[u] * f.sc;
    }
  }
  __syncthreads();
  const int k0 = sg * L < nz ? sg * L : nz;
  const int k1 = k0 + L < nz ? k0 + L : nz;
  const int nseg = (nz + L - 1) / L;  // segments with rows
  // Value entering segment sg of a recurrence whose segments ended (from zero) in `ends`, visited in the order
  // first, first + dir, ...: the segments before it in that order, and the whole ring's wrap-around value.
  auto enter = [&](int dir) {
    const int first = dir > 0 ? 0 : nseg - 1;
    T e = (T)0, in = (T)0, p = (T)1, pin = (T)1;
    for (int q = 0, s = first; q < nseg; ++q, s += dir) {
      if (s == sg) {
        in = e;
        pin = p;
      }
      const T w = s == nseg - 1 ? f.pwl : f.pw;
      e = fma_t(w, e, ends[s * TI]);
      p = p * w;
    }
    return fma_t(pin, e * f.g, in);
  };
  T v = (T)0;
  if (live)
#pragma unroll 4
    for (int k = k0; k < k1; ++k) v = fma_t(f.rho, v, yv[k * TI]);
  ends[sg * TI] = v;
  __syncthreads();
  if (live && k0 < k1) {
    v = enter(1);
#pragma unroll 4
    for (int k = k0; k < k1; ++k) {
      v = fma_t(f.rho, v, yv[k * TI]);
      yv[k * TI] = v;
    }
    v = (T)0;
#pragma unroll 4
    for (int k = k1 - 1; k >= k0; --k) v = fma_t(f.rho, v, yv[k * TI]);
  }
  __syncthreads();
  ends[sg * TI] = v;
  __syncthreads();
  bool bad = false;
  if (live && k0 < k1) {
    v = enter(-1);
#pragma unroll 4
    for (int k = k1 - 1; k >= k0; --k) {
      v = fma_t(f.rho, v, yv[k * TI]);
      yv[k * TI] = v;
    }
  }
  __syncthreads();
  if (live)
#pragma unroll 4
    for (int k = sg; k < nz; k += NS) {
      const T x = yv[k * TI];
      col[(size_t)k * plane] = x;
      if (a.info) bad |= !isfinite((double)x);
    }
  if (bad) atomicOr(&a.info->nonfinite, 1u);
  if (a.singular && bx == 0 && j == 0 && !z.lowcut && threadIdx.x < 32)
    zcirc_singular<T>(a, reinterpret_cast<T*>(a.S), plane, threadIdx.x);
}

template <typename T>
static __global__ void __launch_bounds__(kZCircThreads) k_zcirc(ZArgs a, ZCircArgs z) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  zcirc_block<T>(a, z, blockIdx.x, blockIdx.y, smem_raw);
}

// Refinement plans: the low-eigenvalue systems in FP64, one warp each: every lane runs its rows from zero, a warp
// scan of the lanes' maps (and the wrap-around value) gives each its start.  `scratch`: [nz][nlow].
template <typename TS>
static __global__ void __launch_bounds__(128) k_zcirc_low(ZArgs a, const int2* __restrict__ modes, int nlow,
                                                          const ZCirc<double>* __restrict__ tab, double* scratch) {
  if (block_skipped(a.skip_conv, a.skip_k, a.tol2)) return;
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (w >= nlow) return;  // uniform per warp
  const int2 md = modes[w];
  const size_t plane = (size_t)a.nx * a.ny;
  if (!VOFP_IN((size_t)md.y * a.nx + md.x, plane, CHK_Z_COLUMN)) return;
  TS* col = reinterpret_cast<TS*>(a.S) + (size_t)md.y * a.nx + md.x;
  if (a.singular && md.x == 0 && md.y == 0) {
    zcirc_singular<TS>(a, col, plane, lane);
    return;
  }
  const ZCirc<double> f = tab[w];
  double* scr = scratch + w;
  const int nz = a.nz, R = (nz + 31) >> 5;
  const int k0 = lane * R < nz ? lane * R : nz;
  const int k1 = k0 + R < nz ? k0 + R : nz;
  double A = 1.0, B = 0.0;
  for (int k = k0; k < k1; ++k) {
    B = fma(f.rho, B, (double)col[k * plane] * f.sc);
    A *= f.rho;
  }
  double A1 = A;
  affine_scan_up(A1, B, lane);
  double Y = __shfl_sync(0xffffffffu, B, 31) * f.g;
  double pa = shfl_up_t(A1, 1), pb = shfl_up_t(B, 1);
  double v = lane == 0 ? Y : fma(pa, Y, pb);
  for (int k = k0; k < k1; ++k) {
    v = fma(f.rho, v, (double)col[k * plane] * f.sc);
    scr[(size_t)k * nlow] = v;
  }
  B = 0.0;
  for (int k = k1 - 1; k >= k0; --k) B = fma(f.rho, B, scr[(size_t)k * nlow]);
  affine_scan_down(A, B, lane);
  Y = __shfl_sync(0xffffffffu, B, 0) * f.g;
  pa = shfl_down_t(A, 1);
  pb = shfl_down_t(B, 1);
  v = lane == 31 ? Y : fma(pa, Y, pb);
  bool bad = false;
  for (int k = k1 - 1; k >= k0; --k) {
    v = fma(f.rho, v, scr[(size_t)k * nlow]);
    col[k * plane] = (TS)v;
    if (a.info) bad |= !isfinite(v);
  }
  if (bad) atomicOr(&a.info->nonfinite, 1u);
}

}  // namespace vofp
