// Real-to-real x and y transforms of FP64 and FP32-pair spectra in 64-bit fixed point.
//
// An FP64 operation holds this GPU's FP64 pipe as long as 32 integer lanes hold theirs (2 against 64 operations per
// SM and cycle), so a transform pass in FP64 is bound by that pipe at a tenth of the copy bandwidth.  Here every pair
// of lines is scaled by one power of two (its largest exponent) to 64-bit integers as it is loaded, transformed
// with integer additions and 32 x 32-bit products, and turned back into doubles (or FP32 pairs) as it is stored;
// both conversions are integer operations too.
//
// Measured (CUDA events, FP64 spectra, P, P, NN; FP64 butterflies -> fixed point): 128^3 divergence + x 92.7 -> 55 us,
// x 69.5 -> 28.7, y 62.0 / 63.6 -> 20.4 / 23.4, inverse x 65.5 -> 24.8; 320 x 320 x 640 (run-time stages of radix 5, 8, 8)
// x 2.30 -> 1.28 ms, y 2.09 -> 0.68, inverse x 2.16 -> 0.81.  Bound now by the integer pipe, 52 to 57% busy over a whole
// pass (ncu at 128^3: 143 to 198 instructions a value, issue 38 to 46%), and by the latency of the 64-bit carry chains with a
// third of the warps that an SM can hold.
//
// Scaling.  A complex value z of a line satisfies |z| <= 2^61.5 throughout.  A twiddle product leaves a quarter of
// its exact value (two factors of 2^62 and the upper 64 bits of the product), a radix-R stage adds up R values, so
// after stage s the bound has grown by prod R / 4^(s-1) (and by R / 16 in a rolled odd-prime stage, whose own
// products leave a quarter again).  FxDesc::bits, the width of the scaled inputs, is what the largest of these
// growths leaves: 58 bits for 128 points, 56 for 512, against a double's 53.  Lines whose sums do not grow are scaled by
// their L1 norm instead (fx_settle).  Error of a forward transform against extended precision (host emulation; dense, smooth,
// sparse and dominated lines, steps and bumps): 0.4e-16 to 1.9e-16 up to 1024 points, to 3.5e-16 at 2048 and with many short odd stages
// (see fx_noise); FP64 butterflies 1.2e-16 to 5e-16, in Bluestein form 4e-16 to 7e-16.
//
// A line with an infinity or a NaN gives NaN on the whole pair of lines, as FP64 butterflies do.
//
// Layout.  A tile of 2^lgB complex lines (two real lines each) lies element-major in shared memory, element e of
// line b at e st + b: lanes run over the lines first, so that every butterfly reads and writes consecutive
// words.  Each thread holds at most ten values between two barriers and writes them back in place: one buffer per
// tile.  The y pass takes st = 2^lgB; the x pass, whose global accesses run along a line, st = 2^lgB + 1, which
// keeps those free of bank conflicts too.
#pragma once

#include "passes.cuh"

namespace vofp {

struct __align__(16) cfx {
  long long x, y;
};
struct fxw {  // a 64-bit weight w as two signed halves: w = hi 2^32 + lo
  int lo, hi;
};
struct __align__(16) fxtw {  // twiddle c + i d (Q62) for three products: c, d - c, c + d, and the roundings of the last two
  fxw c, dmc, cpd;
  int rdmc, rcpd;
};
struct __align__(16) fxq {
  fxw c, d;
};

constexpr int kFxStages = 12;
constexpr int kFxMaxPrime = 199;  // of a rolled stage
// Twiddles in shared memory up to this length (32 bytes each); beyond it they are read through L1.
constexpr int kFxTwSmem = 512;
struct FxDesc {
  int n, nst;
  int bits;   // width of the scaled inputs of a forward pass
  int shift;  // the transform's result is 2^-shift of the exact one
  int two;    // the largest radix of a rolled odd-prime stage, which needs a second buffer and its weights there; 0: none
  int radix[kFxStages];
  // per stage: butterflies per line n / radix, twiddle step n / (Ns radix), and ceil(2^32 / Ns): j / Ns =
  // umulhi(j, magic) for j < 2^16
  int nr[kFxStages], step[kFxStages];
  unsigned magic[kFxStages];
  unsigned magn, magh;  // the same for n and for (n + 1) / 2
};

// Stages, scaling and bounds of the length in fd; false: not handled (too long, too many stages).
inline bool fx_desc(const FftDesc& fd, FxDesc* fx) {
  if (fd.nst > kFxStages || fd.n > 2048) return false;
  fx->n = fd.n;
  fx->nst = fd.nst;
  fx->two = 0;
  fx->shift = 0;
  double grow = 1.0, most = 1.0;
  unsigned Ns = 1;
  for (int s = 0; s < fd.nst; ++s) {
    const int R = fd.radix[s];
    fx->radix[s] = R;
    fx->magic[s] = Ns == 1 ? 0u : (unsigned)((0x100000000ull + Ns - 1) / Ns);
    fx->nr[s] = fd.n / R;
    fx->step[s] = fd.n / ((int)Ns * R);
    if (s > 0) {
      grow *= 0.25;
      fx->shift += 2;
    }
    if (R > 5 && R != 8) {
      if (R > fx->two) fx->two = R;
      grow *= 0.25;
      fx->shift += 2;
    }
    grow *= R;
    if (grow > most) most = grow;
    Ns *= R;
  }
  int g = 0;
  while ((double)(1ull << g) < most) ++g;
  fx->bits = 61 - g;
  const unsigned h = (fd.n + 1) / 2;
  fx->magn = fd.n == 1 ? 0u : (unsigned)((0x100000000ull + fd.n - 1) / fd.n);
  fx->magh = h == 1 ? 0u : (unsigned)((0x100000000ull + h - 1) / h);
  return true;
}

// The rounding error of a transform of a dense line, relative (rms): the signal's and the noise's size stage by stage.  Each
// product takes two bits off that only a radix of 16 or more brings back, sums of random terms growing by sqrt(R) and not by
// the R that the scaling allows for: many short odd stages end with few bits.  Emulated on the host against extended
// precision for all lengths this may concern (383, seven kinds of line): the error is at most 1.05 times that of FP64 butterflies
// where this is below 1.45e-16 (2e-16 without a rolled stage), and up to 2.6 times it above (1029 = 3 7 7 7: 3.1e-16; 1715, 1764,
// 1911, 1944).
inline double fx_noise(const FftDesc& fd) {
  FxDesc fx;
  if (!fx_desc(fd, &fx)) return 1.0;
  double sig = ldexp(1.0, fx.bits) / 3, var = 0.1;
  for (int s = 0; s < fx.nst; ++s) {
    const int R = fx.radix[s];
    if (s > 0) {
      sig *= 0.25;
      var = var / 16 + 0.25;
    }
    if (R > 5 && R != 8) {
      sig *= 0.25 * sqrt((double)R);
      var = var / 16 * R + 0.1;
    } else {
      sig *= sqrt((double)R);
      var = var * R + (R == 2 || R == 4 ? 0.0 : 0.3);
    }
  }
  return sqrt(var) / sig;
}

// Lines of a compiled-in length's tile (2^lgn samples).
__host__ __device__ constexpr int fx_ct_lgB(int lgn) { return lgn == 5 ? 1 : 3; }
// Tile width, from the number of eight-line tiles: the widest of 8, 4, 2, 1 lines whose tile takes at most 256
// threads (512 for 512 samples),
// narrowed while tiles are fewer than SMs (but not below `least` lines, nor a warp with two values a lane).
inline int fx_lgB(int n, long tiles8, int least) {
  int lg = 3;
  while (lg > 0 && (n << lg) > ((n & (n - 1)) == 0 && n <= 512 ? 4096 : 2048)) --lg;
  while (lg > least && (tiles8 << (3 - lg)) < 152 && (n << lg) > 64) --lg;
  return lg;
}
// Eight-line tiles of the x, or the y pass.
inline long fx_tiles8(int nx, int ny, int nz, bool y) {
  return y ? (long)((nx + 15) / 16) * nz : (((long)ny * nz + 1) / 2 + 7) / 8;
}

// Does a plan (ff: of FP32-pair spectra) transform the x (or y) axis of the length in fd in fixed point?  Where it is the
// faster way, by cells.  Measured per axis, forward and inverse pass together, P and NN, floating point against fixed point (above 1:
// fixed point is faster).
// Powers of two.  FP64 from 64 on: 0.94-1.5 below 400,000 cells, 1.4-3.8 above; 32: 1.2-1.4 where the compiled-in kernel's one-warp
// tiles are what the grid has (16,000 and 32,000 cells), 0.79-0.97 from 64,000 to 256,000 with the run-time kernel, 1.1-2.0 from 512,000.
// FP32 pairs, x (their y pass takes TMA tiles): 64 0.87-1.06 below 480,000, 1.06-1.7 above; 128, 256, 512 0.73-0.99 up to 600,000,
// 1.0-1.15 at 720,000, 1.2-1.5 above a million.
// Other lengths.  A pass of a small grid is one short wave of blocks, bound by the latency of its chain, and that of the
// fixed-point passes is the longer one.  FP64: 0.70-0.99 at 128,000 cells on lines below 64, 1.0-1.4 at 200,000 to 250,000 -- but for
// three short stages (30: 0.74-0.87, 48: 0.9, 60: 0.84-1.0; 0.94-1.3 at 300,000) -- and 1.3-2.6 above 500,000; y of 256 and more
// 1.4-2.2 everywhere.  FP32 pairs, x: 0.6-0.95 up to 500,000 cells, 0.81-1.2 at 2,000,000, 0.87-1.16 at 2,400,000, 1.0-1.28 at
// 2,800,000, 1.1-1.4 at 12,000,000; y: up to 50 samples 1.0-1.28 from 2,400,000, 72 to 100 0.74-1.08 below 6,000,000 and 1.0-1.2 at 8 to 12
// million, beyond that 0.66-0.98 up to 6,000,000 and 0.87-1.1 at 8 to 12.
// Lengths with a prime above 13 (p to 199; FP32 pairs 53): a rolled stage costs p products a value, the floating-point passes'
// Bluestein form two transforms of two to three times the length.  FP64: x 0.99-2.3 at 16,000 to 125,000 cells (179: 0.99, 199: 1.11,
// 127: 1.27), 1.03-4.9 above, y 1.35-6.6; FP32 pairs 1.0-3.  (With an eighth of a tile's values in threads on small grids too: FP64
// x 0.54-1.0 for p from 127 on below 500,000 cells, FP32 pairs 0.76-1.1 for 47 and 53.  See fx_threads.)
// `force` (VOFP_FX=1 when the plan is created): fixed point whatever the grid, for comparisons.
inline bool fx_takes(const FftDesc& fd, bool ff, bool y, int nx, int ny, int nz, bool force) {
  FxDesc fx;
  for (int s = 0; s < fd.nst; ++s)
    if (fd.radix[s] > (ff ? 53 : kFxMaxPrime)) return false;
  if (!fx_desc(fd, &fx)) return false;
  // (stages of radix 3 err more in FP64 too; a Bluestein form by 4e-16 to 7e-16)
  if (!fd.bm && !ff && fx_noise(fd) > (fx.two ? 1.45e-16 : 2e-16)) return false;
  if (force || fd.bm) return true;
  const long cells = (long)nx * ny * nz;
  const int n = fd.n;
  const bool pow2 = (n & (n - 1)) == 0;
  if (pow2 && n >= 32 && n <= 512) {
    if (ff) return cells >= (n <= 64 ? 480000 : 700000);
    return n >= 64 || cells >= 480000 || fx_lgB(n, fx_tiles8(nx, ny, nz, y), y ? 1 : 0) == fx_ct_lgB(5);
  }
  if (ff) {
    if (y) return cells >= 2400000 && (n <= 50 || (n <= 100 && cells >= 8000000));
    return cells >= 2800000;
  }
  return cells >= (n < 64 && fd.nst >= 3 ? 300000 : 200000) || (y && n >= 256);
}

// ---- scalars ------------------------------------------------------------------------------------------------

// a w / 2^64 for |a| < 2^63: the product of the upper halves and the upper words of the two mixed products (the
// lower halves taken as signed numbers, so that every product is one signed instruction).  Each mixed product is
// rounded down, half a unit on average: rd = 1 centres the error.
__device__ __forceinline__ long long fx_mul(long long a, fxw w, int rd = 1) {
  const int al = (int)a;
  const int ah = (int)(a >> 32) + (int)((unsigned)al >> 31);
  const int lo = __mulhi(ah, w.lo) + __mulhi(al, w.hi) + rd;
  return (long long)ah * w.hi + lo;
}
// (a + i b)(c + i d) / 4 by three products.  Their roundings are centred in the sums (rcpd, rdmc: 0 and 2, less where a
// factor is 0 or 1 and its product is exact, see fx_twiddle): a constant error of one unit would be added up by the
// stages that follow into the lowest modes, whose errors the z solve magnifies most.
// ZERO: a product of zero is zero and needs no centring.  On lines longer than 512, one cell's source (zeros almost
// everywhere, until the last stage) came out of 2048 points with twice the error of FP64 butterflies in the lowest modes without it.
template <bool ZERO>
__device__ __forceinline__ cfx fx_cmul(cfx z, const fxtw& w) {
  const bool zero = ZERO && (z.x | z.y) == 0;
  const long long k = fx_mul(z.x + z.y, w.c, 0);
  cfx r;
  r.x = k - fx_mul(z.y, w.cpd, zero ? 0 : w.rcpd);
  r.y = k + fx_mul(z.x, w.dmc, zero ? 0 : w.rdmc);
  return r;
}
// z / 4, ties to even (also in the place of a product with 1).
__device__ __forceinline__ cfx fx_quarter(cfx z) {
  cfx r;
  r.x = (z.x + 1 + ((int)(z.x >> 2) & 1)) >> 2;
  r.y = (z.y + 1 + ((int)(z.y >> 2) & 1)) >> 2;
  return r;
}
__host__ __device__ __forceinline__ fxw fx_weight(long long w) {
  fxw f;
  f.lo = (int)(unsigned)(unsigned long long)w;
  f.hi = (int)((w - f.lo) >> 32);
  return f;
}
// Table entry of the twiddle c + i d.
inline fxtw fx_twiddle(long long c, long long d) {
  // how far below the exact value a product with w comes out on average
  auto low = [](long long w) { return w == 0 ? 0.0 : (w == 1ll << 62 || w == -(1ll << 62) ? 0.375 : 1.0); };
  auto nearest = [](double v) { return v < 0 ? -(int)(0.5 - v) : (int)(v + 0.5); };
  return {fx_weight(c), fx_weight(d - c), fx_weight(c + d), nearest(low(c) + low(d - c)), nearest(low(c + d) - low(c))};
}
// a c for a constant c = w / 2^63, |a| < 2^62
__device__ __forceinline__ long long fx_scale(long long a, long long w) {
  return fx_mul(a + a, fx_weight(w));
}

// Size of a value for the line's exponent: the upper word of its magnitude as a double (0x7ff00000: infinity or NaN) and
// the bits below, gathered by or.
__device__ __forceinline__ void fx_size(double d, int& top, unsigned& low) {
  top = max(top, __double2hiint(d) & 0x7fffffff);
  low |= (unsigned)__double2loint(d);
}
__device__ __forceinline__ void fx_size(ff f, int& top, unsigned&) {
  // (the pair's leading part: |pair| < 2^(e + 1 - 127) all the same)
  const int b = __float_as_int(f.hi) & 0x7fffffff;
  top = max(top, b >= 0x7f800000 ? 0x7ff00000 : (b ? (b >> 3) + ((1023 - 127) << 20) : 0));
}

// The double x scaled to 64 - rs0 bits below the exponent E of the line's largest value; E >= 66 (values below the
// normal range, like zeros, are shifted out; fx_transform lifts lines that consist of such).
__device__ __forceinline__ long long fx_of(double x, int E, int rs0, int flip) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  const unsigned mh = __funnelshift_l(lo, (unsigned)hi, 11) | 0x80000000u;
  unsigned long long m = ((unsigned long long)mh << 32) | (lo << 11);
  asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(rs0 + E - ((hi >> 20) & 0x7ff)));  // (a shift beyond 63 gives 0)
  return (hi ^ flip) < 0 ? -(long long)m : (long long)m;
}
__device__ __forceinline__ long long fx_of_f32(float x, int E, int rs0, int flip) {
  const int b = __float_as_int(x);
  const int e = (b >> 23) & 0xff;  // (0: subnormal, 2^-126 as the unit and no implicit bit)
  unsigned long long m = (unsigned long long)(((unsigned)b << 8) | (e ? 0x80000000u : 0u)) << 32;
  asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(rs0 + E - (max(e, 1) + 1023 - 127)));
  return (b ^ flip) < 0 ? -(long long)m : (long long)m;
}
__device__ __forceinline__ long long fx_of(ff x, int E, int rs0, int flip) {
  return fx_of_f32(x.hi, E, rs0, flip) + fx_of_f32(x.lo, E, rs0, flip);
}

// Exponent offsets K of a line's results (value = v 2^K) that stand for a line with an infinity or a NaN, and for a line
// of zeros (whose products come out as a unit or two).
constexpr int kFxNan = 1 << 20, kFxZero = -(1 << 20);
// v 2^K as a double, rounded to nearest (ties up): the rare cases ...
static __device__ __noinline__ double fx_to_rare(long long v, int K) {
  if (K == kFxNan) return __longlong_as_double(0x7ff8000000000000ll);
  // (two factors: |K| can pass 1022)
  const int k1 = K / 2, k2 = K - k1;
  return (double)v * __longlong_as_double((long long)(k1 + 1023) << 52) *
         __longlong_as_double((long long)(k2 + 1023) << 52);
}
// ... and the others: normalise, round at bit 11, put the exponent in.
__device__ __forceinline__ double fx_to(long long v, int K, int flip, double*) {
  const int vh = (int)(v >> 32);
  const unsigned long long a = (unsigned long long)(vh < 0 ? -v : v);
  unsigned h = (unsigned)(a >> 32), l = (unsigned)a;
  int e = 1085 + K;  // one below the biased exponent: the implicit bit adds it
  if (h == 0) {
    h = l;
    l = 0;
    e -= 32;
  }
  const int lz = __clz((int)h);
  e -= lz;
  if (h == 0 || (unsigned)e > 2044u) return ((v == 0 && K != kFxNan) || K == kFxZero) ? 0.0 : fx_to_rare(flip ? -v : v, K);
  const unsigned nh = __funnelshift_l(l, h, lz), nl = l << lz;
  const unsigned rh = (nh >> 11) + (((unsigned)e << 20) | ((unsigned)(vh ^ flip) & 0x80000000u));
  const unsigned rl = __funnelshift_r(nl, nh, 11);
  const unsigned long long r = (((unsigned long long)rh << 32) | rl) + ((nl >> 10) & 1u);
  return __longlong_as_double((long long)r);
}
// ... as an FP32 pair: the leading 24 bits rounded to nearest, then the next 23 of the signed remainder.
__device__ __forceinline__ ff fx_to(long long v, int K, int flip, ff*) {
  int s = (int)(v >> 63);
  unsigned long long u = (unsigned long long)((v ^ (long long)s) - (long long)s);
  if (u == 0 || K == kFxNan || K == kFxZero) {
    const float q = K == kFxNan ? __int_as_float(0x7fc00000) : 0.0f;
    return ff(q, 0.0f);
  }
  const int lz = __clzll((long long)u);
  u <<= lz;
  s ^= flip;  // (its sign bit from here on)
  const int e = 63 - lz + K;  // |value| = u / 2^63 2^e
  if (e < -78 || e > 126) {  // near the ends of the FP32 range
    const double d = fx_to(v, K, flip, (double*)nullptr);
    const float hi = (float)d;
    return ff(hi, isinf(hi) ? 0.0f : (float)(d - (double)hi));
  }
  const unsigned h = (unsigned)(u >> 32);
  const unsigned hr = ((h >> 8) + ((h >> 7) & 1u));  // 24 bits, or 2^24
  const int rem = (int)((unsigned)(u >> 16) - (hr << 24));  // the signed remainder in units of 2^-24 of the leading ulp
  const float hi = __int_as_float((int)(hr + ((unsigned)(e + 126) << 23)) | (s & 0x80000000));
  const float lo = (float)rem * __int_as_float((unsigned)(e - 47 + 127) << 23);
  return ff(hi, __int_as_float(__float_as_int(lo) ^ (s & 0x80000000)));
}

// ---- butterflies ----------------------------------------------------------------------------------------------

__device__ __forceinline__ void fx_dft(cfx* v, std::integral_constant<int, 2>) {
  const cfx t = v[0];
  v[0] = cadd(t, v[1]);
  v[1] = csub(t, v[1]);
}
__device__ __forceinline__ void fx_dft(cfx* v, std::integral_constant<int, 3>) {
  const long long h = 0x6ed9eba16132a9cfll;  // sin(2 pi / 3), Q63
  const cfx s = cadd(v[1], v[2]), d = csub(v[1], v[2]);
  const cfx m = cmk<cfx>(v[0].x - (s.x >> 1), v[0].y - (s.y >> 1));
  const cfx r = cmk<cfx>(fx_scale(d.y, h), -fx_scale(d.x, h));
  v[0] = cadd(v[0], s);
  v[1] = cadd(m, r);
  v[2] = csub(m, r);
}
__device__ __forceinline__ void fx_dft4(cfx& v0, cfx& v1, cfx& v2, cfx& v3) {
  const cfx a0 = cadd(v0, v2), a1 = csub(v0, v2), b0 = cadd(v1, v3), b1 = csub(v1, v3);
  v0 = cadd(a0, b0);
  v2 = csub(a0, b0);
  v1 = cmk<cfx>(a1.x + b1.y, a1.y - b1.x);  // a1 - i b1
  v3 = cmk<cfx>(a1.x - b1.y, a1.y + b1.x);
}
__device__ __forceinline__ void fx_dft(cfx* v, std::integral_constant<int, 4>) { fx_dft4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ void fx_dft(cfx* v, std::integral_constant<int, 5>) {
  const long long c1 = 0x278dde6e5fd29f05ll, c2 = -0x678dde6e5fd29f05ll;  // cos(2 pi / 5), cos(4 pi / 5), Q63
  const long long s1 = 0x79bc384d1153fd7all, s2 = 0x4b3c8c11d56977b7ll;   // sin
  const cfx a1 = cadd(v[1], v[4]), b1 = csub(v[1], v[4]);
  const cfx a2 = cadd(v[2], v[3]), b2 = csub(v[2], v[3]);
  const cfx m1 = cmk<cfx>(v[0].x + fx_scale(a1.x, c1) + fx_scale(a2.x, c2),
                          v[0].y + fx_scale(a1.y, c1) + fx_scale(a2.y, c2));
  const cfx m2 = cmk<cfx>(v[0].x + fx_scale(a1.x, c2) + fx_scale(a2.x, c1),
                          v[0].y + fx_scale(a1.y, c2) + fx_scale(a2.y, c1));
  const cfx t1 = cmk<cfx>(fx_scale(b1.x, s1) + fx_scale(b2.x, s2), fx_scale(b1.y, s1) + fx_scale(b2.y, s2));
  const cfx t2 = cmk<cfx>(fx_scale(b1.x, s2) - fx_scale(b2.x, s1), fx_scale(b1.y, s2) - fx_scale(b2.y, s1));
  v[0] = cmk<cfx>(v[0].x + a1.x + a2.x, v[0].y + a1.y + a2.y);
  v[1] = cmk<cfx>(m1.x + t1.y, m1.y - t1.x);
  v[4] = cmk<cfx>(m1.x - t1.y, m1.y + t1.x);
  v[2] = cmk<cfx>(m2.x + t2.y, m2.y - t2.x);
  v[3] = cmk<cfx>(m2.x - t2.y, m2.y + t2.x);
}
__device__ __forceinline__ void fx_dft(cfx* v, std::integral_constant<int, 8>) {
  const long long r2 = 0x5a827999fcef3242ll;  // 1 / sqrt(2), Q63
  fx_dft4(v[0], v[2], v[4], v[6]);
  fx_dft4(v[1], v[3], v[5], v[7]);
  const cfx o1 = cmk<cfx>(fx_scale(v[3].x + v[3].y, r2), fx_scale(v[3].y - v[3].x, r2));
  const cfx o3 = cmk<cfx>(fx_scale(v[7].y - v[7].x, r2), -fx_scale(v[7].x + v[7].y, r2));
  const cfx e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o2 = cmi(v[5]);
  v[0] = cadd(e0, o0);
  v[4] = csub(e0, o0);
  v[1] = cadd(e1, o1);
  v[5] = csub(e1, o1);
  v[2] = cadd(e2, o2);
  v[6] = csub(e2, o2);
  v[3] = cadd(e3, o3);
  v[7] = csub(e3, o3);
}

// The values of a line with little growth (see fx_settle) lifted by lam = 2 bits before a product takes them off.
__device__ __forceinline__ cfx fx_lift(cfx z, int lam) { return cmk<cfx>(z.x << lam, z.y << lam); }
template <int N>
__device__ __forceinline__ void fx_lift(cfx* v, int lam) {
  if (__any_sync(__activemask(), lam != 0)) {
#pragma unroll
    for (int r = 0; r < N; ++r) v[r] = fx_lift(v[r], lam);
  }
}

// Keeps the compiler from starting the loads of the next step before this one is done (the values in flight would
// spill).
__device__ __forceinline__ void fx_fence() { asm volatile("" ::: "memory"); }

// One radix-RAD stage in place (MAXIT butterflies a thread: blockDim.x >= 2^lgB n / 8) on the tile at byte offset
// `off` of the dynamic shared memory, twiddles at offset twoff there (TWS) or at twg.  A call: inlined side by side, the
// stages of all radices would share one register allocation and spill.
template <int RAD, int MAXIT, bool TWS>
__device__ __noinline__ void fx_stage(int off, int st, int lgB, int NR, int Ns, int twstep, unsigned magic, int twoff,
                                      const fxtw* __restrict__ twg, int lam) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cfx* buf = reinterpret_cast<cfx*>(smem_raw + off);
  const fxtw* tws = reinterpret_cast<const fxtw*>(smem_raw + twoff);
  const int total = NR << lgB;
  const int mB = (1 << lgB) - 1;
  cfx v[MAXIT][RAD];
#pragma unroll
  for (int it = 0; it < MAXIT; ++it) {
    const int t = threadIdx.x + it * blockDim.x;
    if (t < total) {
      const int j = t >> lgB;
      const cfx* s = buf + j * st + (t & mB);
#pragma unroll
      for (int r = 0; r < RAD; ++r) v[it][r] = s[r * NR * st];
      if (Ns > 1) {
        const int k = j - (int)__umulhi((unsigned)j, magic) * Ns;
        fx_lift<RAD>(v[it], lam);
        v[it][0] = fx_quarter(v[it][0]);
        if (k == 0) {
#pragma unroll
          for (int r = 1; r < RAD; ++r) v[it][r] = fx_quarter(v[it][r]);
        } else {
#pragma unroll
          for (int r = 1; r < RAD; ++r) {
            v[it][r] = fx_cmul<!TWS>(v[it][r], TWS ? tws[r * k * twstep] : twg[r * k * twstep]);
            fx_fence();
          }
        }
      }
      fx_dft(v[it], std::integral_constant<int, RAD>());
      fx_fence();
    }
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < MAXIT; ++it) {
    const int t = threadIdx.x + it * blockDim.x;
    if (t < total) {
      const int j = t >> lgB;
      const int q = Ns > 1 ? (int)__umulhi((unsigned)j, magic) : j;
      cfx* d = buf + (q * Ns * (RAD - 1) + j) * st + (t & mB);  // element (j - k) RAD + k
#pragma unroll
      for (int r = 0; r < RAD; ++r) d[r * Ns * st] = v[it][r];
    }
  }
  __syncthreads();
}

// The same for a power-of-two length 2^LGN, its tile width and threads known at compile time.
__host__ __device__ constexpr int fx_ct_threads(int lgn) {
  return (1 << (lgn + fx_ct_lgB(lgn))) / 8 < 32 ? 32 : (1 << (lgn + fx_ct_lgB(lgn))) / 8;
}
template <int RAD, int LGN, int LGNS, int PAD>
__device__ __forceinline__ void fx_stage_ct(cfx* buf, const fxtw* __restrict__ tw, int lam) {
  constexpr int lgR = RAD == 8 ? 3 : (RAD == 4 ? 2 : 1), LGB = fx_ct_lgB(LGN), ST = (1 << LGB) + PAD;
  constexpr int NR = 1 << (LGN - lgR), NT = fx_ct_threads(LGN), Ns = 1 << LGNS, TOTAL = NR << LGB;
  constexpr int IT = (TOTAL + NT - 1) / NT;
  cfx v[IT][RAD];
  const int b = threadIdx.x & ((1 << LGB) - 1);
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int j = (threadIdx.x + it * NT) >> LGB;
    if (TOTAL % NT != 0 && j >= NR) break;
    const cfx* s = buf + j * ST + b;
#pragma unroll
    for (int r = 0; r < RAD; ++r) v[it][r] = s[r * NR * ST];
    if (LGNS > 0) {
      const int k = j & (Ns - 1);
      fx_lift<RAD>(v[it], lam);
      v[it][0] = fx_quarter(v[it][0]);
      if (k == 0) {
#pragma unroll
        for (int r = 1; r < RAD; ++r) v[it][r] = fx_quarter(v[it][r]);
      } else {
#pragma unroll
        for (int r = 1; r < RAD; ++r) {
          v[it][r] = fx_cmul<false>(v[it][r], tw[(r * k) << (LGN - LGNS - lgR)]);
          fx_fence();
        }
      }
    }
    fx_dft(v[it], std::integral_constant<int, RAD>());
    fx_fence();
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int j = (threadIdx.x + it * NT) >> LGB;
    if (TOTAL % NT != 0 && j >= NR) break;
    const int k = j & (Ns - 1);
    cfx* d = buf + (((j - k) << lgR) + k) * ST + b;
#pragma unroll
    for (int r = 0; r < RAD; ++r) d[r * Ns * ST] = v[it][r];
  }
  __syncthreads();
}
__host__ __device__ constexpr int fx_radix(int lgn, int s) {  // (the plan's factorisation of a power of two)
  return lgn % 3 == 1 ? (lgn / 3 > 0 ? (s < 2 ? 4 : 8) : 2) : (lgn % 3 == 2 ? (s == 0 ? 4 : 8) : 8);
}
template <int LGN, int PAD, int S = 0, int LGNS = 0>
__device__ __forceinline__ void fx_fft_ct(cfx* buf, const fxtw* __restrict__ tw, int lam) {
  if constexpr (LGNS < LGN) {
    constexpr int R = fx_radix(LGN, S);
    fx_stage_ct<R, LGN, LGNS, PAD>(buf, tw, lam);
    fx_fft_ct<LGN, PAD, S + 1, LGNS + (R == 8 ? 3 : (R == 4 ? 2 : 1))>(buf, tw, lam);
  }
}

// A sum of products a w / 2^64 with the mixed products' lower words kept, h + s / 2^23: rounded once, and a zero adds
// nothing.  (With fx_mul's rounding in every product and half a unit of centring each, the (p - 1) / 2 products of a sparse
// line's zeros added up: 4e-15 at p = 151 .. 199; 0.5e-15 this way, and 0.7e-16, of 2e-16, on dense lines.)  Up to 99 products:
// |s| < 2^61.
struct FxSum {
  long long h, s;
};
__device__ __forceinline__ void fx_mac(FxSum& f, long long a, fxw w) {
  const int al = (int)a;
  const int ah = (int)(a >> 32) + (int)((unsigned)al >> 31);
  f.h += (long long)ah * w.hi;
  f.s += ((long long)ah * w.lo + (long long)al * w.hi) >> 9;
}
// a / 4, exactly, and the sum 2^lam times as a number
__device__ __forceinline__ FxSum fx_sum(long long a) { return {a >> 2, (a & 3) << 21}; }
__device__ __forceinline__ long long fx_value(const FxSum& f, int lam) {
  return (f.h << lam) + ((f.s + (1 << (22 - lam))) >> (23 - lam));
}

// A rolled stage of an odd prime RAD >= 7 from src into dst (see fft_stage_odd); src is scratch afterwards.  Bound by
// instruction issue: the weights lie in shared memory with their signs, and the lift of a line
// with little growth is applied to the sums.
template <bool TWS>
__device__ __noinline__ void fx_stage_odd(int so, int dof, int st, int lgB, int n, int Ns, unsigned magic, int RAD, int twoff,
                                          const fxtw* __restrict__ twg, int lam, int wo) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cfx *src = reinterpret_cast<cfx*>(smem_raw + so), *dst = reinterpret_cast<cfx*>(smem_raw + dof);
  const fxtw* tws = reinterpret_cast<const fxtw*>(smem_raw + twoff);
  fxq* wt = reinterpret_cast<fxq*>(smem_raw + wo);
  const int NR = n / RAD, H = (RAD - 1) / 2;
  const int mB = (1 << lgB) - 1;
  for (int a = threadIdx.x; a < RAD; a += blockDim.x) {
    const fxtw w = TWS ? tws[a * NR] : twg[a * NR];
    wt[a] = {w.c, fx_weight(((long long)(w.c.hi - w.cpd.hi) << 32) + ((long long)w.c.lo - w.cpd.lo))};
  }
  if (Ns > 1) {
    const int twstep = NR / Ns;
#pragma unroll 1
    for (int t = threadIdx.x; t < (n << lgB); t += blockDim.x) {
      const int e = t >> lgB;
      const int r = e / NR;
      const int j = e - r * NR;
      const int k = j - (int)__umulhi((unsigned)j, magic) * Ns;
      cfx* p = src + e * st + (t & mB);
      *p = r * k == 0 ? fx_quarter(fx_lift(*p, lam))
                      : fx_cmul<!TWS>(fx_lift(*p, lam), TWS ? tws[r * k * twstep] : twg[r * k * twstep]);
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int t = threadIdx.x; t < ((NR * (H + 1)) << lgB); t += blockDim.x) {
    const int it = t >> lgB;
    const int m = it / NR;
    const int j = it - m * NR;
    const int q = Ns > 1 ? (int)__umulhi((unsigned)j, magic) : j;
    const cfx* s = src + j * st + (t & mB);
    cfx* d = dst + (q * Ns * (RAD - 1) + j) * st + (t & mB);
    FxSum ax = fx_sum(s[0].x), ay = fx_sum(s[0].y);
    const int step = NR * st;
    if (m == 0) {
#pragma unroll 1
      for (int r = 1; r < RAD; ++r) {
        const cfx z = s[r * step];
        ax.h += z.x >> 2;
        ay.h += z.y >> 2;
        ax.s += (long long)((int)z.x & 3) << 21;
        ay.s += (long long)((int)z.y & 3) << 21;
      }
      d[0] = cmk<cfx>(fx_value(ax, lam), fx_value(ay, lam));
      continue;
    }
    FxSum bx = {0, 0}, by = {0, 0};
    int a = m;  // r m mod RAD
#pragma unroll 1
    for (int r = 1; r <= H; ++r) {
      const cfx lo = s[r * step], hi = s[(RAD - r) * step];
      const fxq w = wt[a];
      fx_mac(ax, lo.x + hi.x, w.c);
      fx_mac(ay, lo.y + hi.y, w.c);
      fx_mac(bx, lo.x - hi.x, w.d);
      fx_mac(by, lo.y - hi.y, w.d);
      a += m;
      if (a >= RAD) a -= RAD;
    }
    const long long px = fx_value(ax, lam), py = fx_value(ay, lam), qx = fx_value(bx, lam), qy = fx_value(by, lam);
    d[m * Ns * st] = cmk<cfx>(px + qy, py - qx);
    d[(RAD - m) * Ns * st] = cmk<cfx>(px - qy, py + qx);
  }
  __syncthreads();
}

// All stages on the tile in b0 (b1: the second buffer of a length with rolled stages; tw: the twiddles in shared
// memory, or in global memory for long lines); returns the result's buffer.  b0 starts the dynamic shared memory.
template <bool TWS>
__device__ __forceinline__ cfx* fx_fft_rt(cfx* b0, cfx* b1, int st, int lgB, const FxDesc& fd, const fxtw* tw,
                                          int lam) {
  int Ns = 1;
  const int o1 = (int)((unsigned char*)b1 - (unsigned char*)b0);
  const int to = TWS ? (int)((const unsigned char*)tw - (const unsigned char*)b0) : 0;
  int off = 0;
  for (int s = 0; s < fd.nst; ++s) {
    const int R = fd.radix[s];
    switch (R) {
      case 2: fx_stage<2, 4, TWS>(off, st, lgB, fd.nr[s], Ns, fd.step[s], fd.magic[s], to, tw, lam); break;
      case 3: fx_stage<3, 3, TWS>(off, st, lgB, fd.nr[s], Ns, fd.step[s], fd.magic[s], to, tw, lam); break;
      case 4: fx_stage<4, 2, TWS>(off, st, lgB, fd.nr[s], Ns, fd.step[s], fd.magic[s], to, tw, lam); break;
      case 5: fx_stage<5, 2, TWS>(off, st, lgB, fd.nr[s], Ns, fd.step[s], fd.magic[s], to, tw, lam); break;
      case 8: fx_stage<8, 1, TWS>(off, st, lgB, fd.nr[s], Ns, fd.step[s], fd.magic[s], to, tw, lam); break;
      default:
        fx_stage_odd<TWS>(off, o1 - off, st, lgB, fd.n, Ns, fd.magic[s], R, to, tw, lam,
                          o1 + fd.n * st * (int)sizeof(cfx) + (TWS ? fd.n * (int)sizeof(fxtw) : 0));
        off = o1 - off;
    }
    Ns *= R;
  }
  return off ? b1 : b0;
}
// LGN > 0: the length is 2^LGN and the tile fx_ct_lgB(LGN) wide, its stride PAD more.
template <int LGN, int PAD>
__device__ __forceinline__ cfx* fx_fft(cfx* b0, cfx* b1, int st, int lgB, const FxDesc& fd, const fxtw* tw, int lam) {
  if constexpr (LGN > 0) {
    fx_fft_ct<LGN, PAD>(b0, tw, lam);
    return b0;
  } else {
    if (fd.n <= kFxTwSmem) return fx_fft_rt<true>(b0, b1, st, lgB, fd, tw, lam);
    return fx_fft_rt<false>(b0, b1, st, lgB, fd, tw, lam);
  }
}

// ---- pre- and post-processing (as fwd_post / inv_pre / quarter_load, on fixed point) --------------------------------

__device__ __forceinline__ long long fx_neg_if(long long x, bool f) { return f ? -x : x; }

// Quarter-wave pre-twiddle of sample i of a pair: position and (a quarter of) the value.
__device__ __forceinline__ cfx fx_quarter_load(cfx z, int i, int n, int bc, const fxq* __restrict__ quart, int& pos) {
  const int s = bc == VOFP_BC_ND ? i : n - 1 - i;
  pos = dct_perm(s, n);
  const fxq w = quart[pos];
  const bool neg = s & 1;
  const long long a = fx_neg_if(z.x, neg), b = fx_neg_if(z.y, neg);
  return cmk<cfx>(fx_mul(a, w.c) - fx_mul(b, w.d), fx_mul(a, w.d) + fx_mul(b, w.c));
}

// Twice the transform (periodic) or half of it (the others: the quarter-wave product leaves a quarter) at spectral
// index q of both lines; Z element-major with stride st.
__device__ __forceinline__ cfx fx_post(const cfx* Z, int st, int n, int bc, int q, const fxq* __restrict__ quart) {
  if (bc == VOFP_BC_P) {
    const int m = (q + 1) >> 1;
    const cfx P = Z[m * st], Q = Z[(m == 0 ? 0 : n - m) * st];
    return ((q == 0) || (q & 1)) ? cmk<cfx>(P.x + Q.x, P.y + Q.y) : cmk<cfx>(P.y - Q.y, Q.x - P.x);
  }
  cfx P, Q;
  fxq w;
  bool neg = false;
  if (quarter_bc(bc)) {
    P = Z[q * st];
    Q = Z[(n - 1 - q) * st];
    w = quart[n + q];
    neg = bc == VOFP_BC_DN && (q & 1);
  } else {
    const int m = (bc == VOFP_BC_DD) ? (n - 1 - q) : q;
    P = Z[m * st];
    Q = Z[(m == 0 ? 0 : n - m) * st];
    w = quart[m];
  }
  const long long oa = fx_mul(P.x + Q.x, w.c) - fx_mul(P.y - Q.y, w.d);
  const long long ob = fx_mul(P.y + Q.y, w.c) - fx_mul(Q.x - P.x, w.d);
  return cmk<cfx>(fx_neg_if(oa, neg), fx_neg_if(ob, neg));
}

// FFT input (conjugated for the forward engine) at index m from the packed spectral lines in S; a quarter of it for
// DCT-II / DST-II.
__device__ __forceinline__ cfx fx_pre(const cfx* S, int st, int n, int bc, int m, const fxq* __restrict__ quart) {
  cfx Z;
  if (bc == VOFP_BC_P) {
    const bool conj = 2 * m > n;
    const int mm = conj ? n - m : m;
    if (m == 0 || 2 * mm == n) {
      const cfx r = S[(m == 0 ? 0 : n - 1) * st];
      Z = r;
    } else {
      const cfx re = S[(2 * mm - 1) * st], im = S[2 * mm * st];
      Z = conj ? cmk<cfx>(re.x + im.y, re.y - im.x) : cmk<cfx>(re.x - im.y, re.y + im.x);
    }
  } else {
    cfx X, Y = cmk<cfx>(0, 0);
    if (bc == VOFP_BC_DD) {
      X = S[(n - 1 - m) * st];
      if (m > 0) Y = S[(m - 1) * st];
    } else {
      X = S[m * st];
      if (m > 0) Y = S[(n - m) * st];
    }
    const fxq w = quart[m];  // (c, -s): V = (c X + s Y) + i (s X - c Y) for each line, Z = Va + i Vb
    const long long vax = fx_mul(X.x, w.c) - fx_mul(Y.x, w.d), vay = -fx_mul(X.x, w.d) - fx_mul(Y.x, w.c);
    const long long vbx = fx_mul(X.y, w.c) - fx_mul(Y.y, w.d), vby = -fx_mul(X.y, w.d) - fx_mul(Y.y, w.c);
    Z = cmk<cfx>(vax - vby, vay + vbx);
  }
  return cmk<cfx>(Z.x, -Z.y);
}

// Scaling around the FFT: the inputs are first scaled to `bits` bits (61, or 60 where an inverse pass adds two of them);
// `width` is what the first stage may take (of lines whose sums grow, see fx_settle), `wide` what the step before it hands
// over; the pre- and post-products leave the result 2^-shift of the exact one.
struct FxScale {
  int bits, wide, width, shift;
};
__device__ __forceinline__ FxScale fx_scale_of(const FxDesc& fd, int bc, bool inv) {
  FxScale s;
  const bool quarter = quarter_bc(bc), pre = quarter || (inv && bc != VOFP_BC_P);  // (a product before the FFT)
  // an inverse pass combines two spectra (up to 2 sqrt 2 times larger), or up to sqrt 2 after the product
  s.width = fd.bits - (inv && !quarter ? 1 : 0);
  s.bits = inv && !pre ? 60 : 61;
  s.wide = s.bits - (pre ? 2 : 0);
  s.shift = (bc != VOFP_BC_P ? 2 : 0) + (quarter ? 2 : 0);
  return s;
}

// Scaling of a line through the FFT, decided from its inputs v (this thread's, nv of at most eight, of line b), when they
// are about to be stored: they go in as v >> rho.  The quarter that each product leaves suits lines whose sums grow with
// every stage.  Where few values dominate -- the spectrum of a smooth line, a right-hand side that is zero but at the
// interface -- nothing grows past the line's L1 norm, and the quarters would cost accuracy: such a line, with an L1
// norm of at most 2^5 times its largest value and a larger result that way, goes in with its L1 norm below 2^60 and is
// lifted again before each product (lam = 2).  (2^60: a lifted value's two parts and their sum stay below 2^63.)  Lines are
// loaded with all the bits there are and shortened here: loaded at fd.bits, one with a dominating value kept the 5 or 6 bits
// of headroom it does not need, 4.5e-16 at 512 points and 9e-16 at 2048 where FP64 butterflies err by 2.6e-16 and 3.3e-16; 0.8e-16 and
// 2.9e-16 this way.  `l1`: per line, cleared; units of 2^44.
struct FxLine {
  int lam, rho;
};
__device__ __forceinline__ FxLine fx_settle(const cfx (&v)[8], int nv, int B, int b, const FxScale& sc, int shift,
                                            unsigned* l1) {
  unsigned acc = 0;
#pragma unroll
  for (int it = 0; it < 8; ++it)
    if (it < nv) acc += ((unsigned)abs((int)(v[it].x >> 32)) + (unsigned)abs((int)(v[it].y >> 32)) >> 4) + 1;
  acc = (acc >> 8) + 1;
  for (int o = B; o < 32; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) < B) atomicAdd(&l1[b], acc);
  __syncthreads();
  const int top = 76 - __clz((int)l1[b]);  // the L1 norm is below 2^top
  const int over = top > 60 ? top - 60 : 0;
  FxLine f;
  if (shift > 0 && top - sc.wide <= 5 && sc.wide - over > sc.width - shift) {
    f.lam = 2;
    f.rho = over;
  } else {
    f.lam = 0;
    f.rho = sc.wide > sc.width ? sc.wide - sc.width : 0;
  }
  return f;
}
// v 2^-rho, rounded.
__device__ __forceinline__ cfx fx_down(cfx v, int rho) {
  const long long h = (1ll << rho) >> 1;
  return cmk<cfx>((v.x + h) >> rho, (v.y + h) >> rho);
}

// Threads for a tile of 2^lgB lines of n: an eighth of its values, whole warps.
inline int fx_threads(int n, int lgB) { return (((n << lgB) + 7) / 8 + 31) / 32 * 32; }
// The same for `blocks` tiles: where they leave an SM less than half its warps, a length with a rolled stage takes more of them, down to
// a value a thread: the stage's items, p products each, are what such a pass waits for (x pass of 199 x 199 x 3 72 us with an eighth,
// 33 so).
inline int fx_threads(const FxDesc& fd, int lgB, long blocks) {
  int th = fx_threads(fd.n, lgB);
  if (fd.two)
    while (2 * th <= 256 && 2 * th < (fd.n << lgB) + 32 && blocks * (2 * th / 32) <= 152 * 32) th *= 2;
  return th;
}
constexpr int kFxMaxThreads = 256;  // (of the run-time lengths)
// Launch bounds.  The compiled-in lengths are held to 72 registers a thread (seven blocks of 128 threads an SM): more
// warps hide more of the integer carry chains' latency than the registers would save (y pass of 128^3: 25.0 us at 96
// registers, 22.1 at 72).
__host__ __device__ constexpr int fx_bound(int lgn) { return lgn > 0 ? fx_ct_threads(lgn) : kFxMaxThreads; }
__host__ __device__ constexpr int fx_blocks(int lgn) {
  return lgn > 0 ? (896 / fx_ct_threads(lgn) < 1 ? 1 : (896 / fx_ct_threads(lgn) > 24 ? 24 : 896 / fx_ct_threads(lgn))) : 3;
}
inline size_t fx_smem(const FxDesc& fd, int lgB, int st) {
  return (size_t)fd.n * st * sizeof(cfx) * (fd.two ? 2 : 1) + (fd.n <= kFxTwSmem ? (size_t)fd.n * sizeof(fxtw) : 0) +
         fd.two * sizeof(fxq);
}

// ---- passes ----------------------------------------------------------------------------------------------------

struct FxTables {
  FxDesc fd;
  const fxtw* tw;
  const fxq* quart;
  int lgB, st;
};

// Shared-memory set-up common to the passes: the twiddles' copy and the lines' largest exponents, cleared.
__device__ __forceinline__ const fxtw* fx_begin(const FxTables& f, unsigned char* smem, cfx*& b0, cfx*& b1, int* emax,
                                              unsigned* l1) {
  b0 = reinterpret_cast<cfx*>(smem);
  const int len = f.fd.n * f.st;
  b1 = b0 + (f.fd.two ? len : 0);
  if (threadIdx.x < (1 << f.lgB)) {
    emax[threadIdx.x] = 0;
    l1[threadIdx.x] = 0u;
  }
  if (f.fd.n > kFxTwSmem) return f.tw;
  int4* tws = reinterpret_cast<int4*>(b1 + len);
  const int4* src = reinterpret_cast<const int4*>(f.tw);
  for (int t = threadIdx.x; t < 2 * f.fd.n; t += blockDim.x) tws[t] = __ldg(src + t);
  return reinterpret_cast<const fxtw*>(tws);
}

// The transform of a tile from its raw values: this thread's are those of elements (threadIdx.x + it blockDim.x) >> lgB of
// line b = threadIdx.x mod 2^lgB (a block is a multiple of 2^lgB threads), nv of them.  Leaves the FFT's result in shared
// memory (returned) and sets the exponent offset K of line b's results.  flip: the sign bit, to transform -x (and negate
// the results): forward passes negate every other line pair, or plane, so that what error of a constant sign the
// roundings have left alternates from line to line -- and ends in the highest modes -- instead of adding up in the
// lowest ones.
template <typename T, bool INV, int LGN, int PAD>
__device__ __forceinline__ const cfx* fx_transform(T (&ra)[8], T (&rb)[8], int nv, int n, int lgB, int st, int bc,
                                                   const FxTables& f, cfx* b0, cfx* b1, const fxtw* tw, int* emax,
                                                   unsigned* l1, int flip, int& K) {
  const int B = 1 << lgB, b = threadIdx.x & (B - 1);
  {
    int e = 0;
    unsigned low = 0;
#pragma unroll
    for (int it = 0; it < 8; ++it) {
      fx_size(ra[it], e, low);
      fx_size(rb[it], e, low);
    }
    if (low != 0 && e == 0) e = 1;
    for (int o = B; o < 32; o <<= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    if ((threadIdx.x & 31) < B) atomicMax(&emax[b], e);
  }
  __syncthreads();
  int any = 0;
  for (int q = 0; q < B; ++q) any |= emax[q];
  if (any == 0) {  // a tile of zeros (a source that lives at the interface has many): so is its transform
#pragma unroll
    for (int it = 0; it < 8; ++it)
      if (it < nv) b0[((threadIdx.x + it * blockDim.x) >> lgB) * st + b] = cmk<cfx>(0, 0);
    K = 0;
    __syncthreads();
    return b0;
  }
  int E = emax[b] >> 20, tiny = 0;
  if constexpr (std::is_same<T, double>::value) {
    if (E < 66) {
      if (emax[b] == 0) {
        E = 66;  // (a line of zeros)
      } else {  // near the end of the range: lifted into it first
        tiny = 128;
        E += 128;
#pragma unroll
        for (int it = 0; it < 8; ++it) {
          ra[it] *= 0x1p128;
          rb[it] *= 0x1p128;
        }
      }
    }
  }
  const FxScale sc = fx_scale_of(f.fd, bc, INV);
  const int rs0 = 64 - sc.bits;
  cfx v[8];
  int pos[8];
#pragma unroll
  for (int it = 0; it < 8; ++it) {
    if (it < nv) {
      const int j = (threadIdx.x + it * blockDim.x) >> lgB;
      v[it] = cmk<cfx>(fx_of(ra[it], E, rs0, flip), fx_of(rb[it], E, rs0, flip));
      pos[it] = j;
      if (quarter_bc(bc)) {
        v[it] = fx_quarter_load(v[it], j, n, bc, f.quart, pos[it]);
      } else if (!INV && bc != VOFP_BC_P) {
        pos[it] = dct_perm(j, n);
        if (bc == VOFP_BC_DD && (j & 1)) v[it] = cmk<cfx>(-v[it].x, -v[it].y);
      }
    }
  }
  if (INV && !quarter_bc(bc)) {
#pragma unroll
    for (int it = 0; it < 8; ++it)
      if (it < nv) b0[pos[it] * st + b] = v[it];
    __syncthreads();
#pragma unroll
    for (int it = 0; it < 8; ++it)
      if (it < nv) v[it] = fx_pre(b0 + b, st, n, bc, pos[it], f.quart);
  }
  const FxLine ln = fx_settle(v, nv, B, b, sc, f.fd.shift, l1);  // (a barrier inside)
  if (__any_sync(0xffffffffu, ln.rho != 0)) {
#pragma unroll
    for (int it = 0; it < 8; ++it) v[it] = fx_down(v[it], ln.rho);
  }
#pragma unroll
  for (int it = 0; it < 8; ++it)
    if (it < nv) b0[pos[it] * st + b] = v[it];
  if (emax[b] == 0) K = kFxZero;
  else K = E == 0x7ff ? kFxNan : E - 1022 - sc.bits - tiny + sc.shift + ln.rho + (ln.lam ? 0 : f.fd.shift);
  __syncthreads();
  return fx_fft<LGN, PAD>(b0, b1, st, lgB, f.fd, tw, ln.lam);
}

// Spectral outputs of a forward pass, both lines of line pair b at once: store(q, value of the first, of the second).
// Periodic: the real and imaginary parts of a mode come from the same two FFT values.  Items run over the lines first
// (LINES_FIRST), else along the line.
template <typename T, int LGN, bool LINES_FIRST, typename STORE>
__device__ __forceinline__ void fx_spectrum(const cfx* Z, int n, int lgB, int st, int bc, const FxTables& f,
                                            STORE store) {
  constexpr bool CT = LGN > 0;
  const int B = 1 << lgB;
  if (bc == VOFP_BC_P) {
    const int items = (n + 1) >> 1;  // modes 0 (with n / 2 of an even n), 1, 2, ...
    for (int t = threadIdx.x; t < (items << lgB); t += blockDim.x) {
      int b, m;
      if constexpr (LINES_FIRST) {
        b = t & (B - 1);
        m = t >> lgB;
      } else if constexpr (CT) {
        b = t >> (LGN - 1);
        m = t & ((n >> 1) - 1);
      } else {
        b = items > 1 ? (int)__umulhi((unsigned)t, f.fd.magh) : t;
        m = t - b * items;
      }
      const cfx P = Z[m * st + b];
      if (m == 0) {
        store(b, 0, 2 * P.x, 2 * P.y);
        if (!(n & 1)) {
          const cfx H = Z[(n >> 1) * st + b];
          store(b, n - 1, 2 * H.x, 2 * H.y);
        }
      } else {
        const cfx Q = Z[(n - m) * st + b];
        store(b, 2 * m - 1, P.x + Q.x, P.y + Q.y);
        store(b, 2 * m, P.y - Q.y, Q.x - P.x);
      }
    }
    return;
  }
  for (int t = threadIdx.x; t < (n << lgB); t += blockDim.x) {
    int b, q;
    if (LINES_FIRST) {
      b = t & (B - 1);
      q = t >> lgB;
    } else {
      b = CT ? t >> LGN : (n > 1 ? (int)__umulhi((unsigned)t, f.fd.magn) : t);
      q = t - b * n;
    }
    const cfx o = fx_post(Z + b, st, n, bc, q, f.quart);
    store(b, q, o.x, o.y);
  }
}

// Right-hand side + forward x transform; block bx takes the line pairs [bx 2^lgB, (bx + 1) 2^lgB).  The right-hand side is
// formed along the lines (coalesced) and handed over through the tile.
template <typename T, int MODE, int LGN>
__global__ void __launch_bounds__(fx_bound(LGN), fx_blocks(LGN)) k_xfwd_fx(const __grid_constant__ XArgs a,
                                                                        const __grid_constant__ FxTables f) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  __shared__ int emax[8], kout[8], lk[16], lj[16];
  __shared__ unsigned l1[8];
  if (block_skipped(a.skip_conv, a.skip_k, a.tol2)) return;
  constexpr bool CT = LGN > 0;
  const int n = CT ? 1 << LGN : f.fd.n, lgB = CT ? fx_ct_lgB(LGN) : f.lgB, B = 1 << lgB;
  const int st = CT ? B + 1 : f.st;
  const int nlines = a.g.ny * a.g.nz;
  const int l00 = blockIdx.x * 2 * B;
  const int bc = a.g.bcx;
  cfx *b0, *b1;
  const fxtw* tw = fx_begin(f, smem_raw, b0, b1, emax, l1);
  if (threadIdx.x < 2 * B) {
    const int l = l00 + threadIdx.x;
    lk[threadIdx.x] = l / a.g.ny;
    lj[threadIdx.x] = l - lk[threadIdx.x] * a.g.ny;
  }
  __syncthreads();
  const bool stats = a.info || a.sq_out || a.fv_out || a.abs_out;
  constexpr bool f64 = std::is_same<T, double>::value;
  const double fbar = (MODE == RHS_RESID && a.defect_sum) ? *a.defect_sum * a.inv_volume : 0.0;
  constexpr bool fv = MODE != RHS_RESID;  // (a residual's sum is not asked for: no multiply-add predicated off)
  double acc_abs = 0, acc_sq = 0, acc_fv = 0;
  float accf_abs = 0.0f, accf_sq = 0.0f;
  const int total = n << lgB;
  // the loads of UL items are issued before any is used (a divergence takes seven for each of its two lines)
  constexpr int UL = MODE == RHS_F ? 4 : 2;
  for (int t0 = threadIdx.x; t0 < total; t0 += UL * blockDim.x) {
    double v[UL][2];
#pragma unroll
    for (int u = 0; u < UL; ++u) {
      const int t = t0 + u * blockDim.x;
      const int pb = CT ? t >> LGN : (n > 1 ? (int)__umulhi((unsigned)t, f.fd.magn) : t), i = t - pb * n;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        v[u][h] = 0.0;
        if (t < total && l00 + 2 * pb + h < nlines) v[u][h] = rhs_at<MODE>(a, i, lj[2 * pb + h], lk[2 * pb + h], fbar);
      }
    }
#pragma unroll
    for (int u = 0; u < UL; ++u) {
      const int t = t0 + u * blockDim.x;
      const int pb = CT ? t >> LGN : (n > 1 ? (int)__umulhi((unsigned)t, f.fd.magn) : t), i = t - pb * n;
      if (t >= total) break;
      if (a.fsave || stats) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int l = l00 + 2 * pb + h, k = lk[2 * pb + h];
          if (l >= nlines) break;
          const double r = v[u][h];
          const size_t o = (size_t)l * n + i;
          if (a.fsave && VOFP_IN(o, (size_t)nlines * n, CHK_XFWD_STORE)) a.fsave[o] = r;
          if (!stats) continue;
          if (f64) {
            const double vol = __ldg(a.g.vol + k);
            acc_abs = fma(fabs(r), vol, acc_abs);
            acc_sq = fma(r, r, acc_sq);
            acc_fv = fma(r, vol, acc_fv);
          } else {
            const float fs = f32_lead_bits(r);
            accf_abs = fmaf(fabsf(fs), __ldg(a.g.volf + k), accf_abs);
            accf_sq = fmaf(fs, fs, accf_sq);
            if (fv && a.fv_out) acc_fv = fma(r, __ldg(a.g.vol + k), acc_fv);
          }
        }
      }
      double2 w;
      w.x = v[u][0];
      w.y = v[u][1];
      *reinterpret_cast<double2*>(b0 + i * st + pb) = w;
    }
  }
  if (stats) {
    if (a.info || a.abs_out) {
      const double s1 = f64 ? block_sum(acc_abs, red) : block_sum(accf_abs, red);
      if (threadIdx.x == 0 && s1 != 0) {
        if (a.info) atomicAdd(&a.info->abs_sum, s1);
        if (a.abs_out) atomicAdd(a.abs_out, s1);
      }
    }
    if (a.sq_out) {
      const double s2 = f64 ? block_sum(acc_sq, red) : block_sum(accf_sq, red);
      if (threadIdx.x == 0 && s2 != 0) atomicAdd(a.sq_out, s2);
    }
    if (fv && a.fv_out) {
      const double s3 = block_sum(acc_fv, red);
      if (threadIdx.x == 0 && s3 != 0) atomicAdd(a.fv_out, s3);
    }
  }
  __syncthreads();
  const int nv = (total - (int)threadIdx.x + (int)blockDim.x - 1) / (int)blockDim.x;
  double ra[8], rb[8];
#pragma unroll
  for (int it = 0; it < 8; ++it) {
    ra[it] = rb[it] = 0.0;
    if (it < nv) {
      const double2 w =
          *reinterpret_cast<const double2*>(b0 + ((threadIdx.x + it * blockDim.x) >> lgB) * st + (threadIdx.x & (B - 1)));
      ra[it] = w.x;
      rb[it] = w.y;
    }
  }
  // (the parity of the line pair; a tile starts at a multiple of its width)
  const int par = B > 1 ? 0 : blockIdx.x;
  int K;
  const cfx* Z = fx_transform<double, false, LGN, 1>(ra, rb, nv, n, lgB, st, bc, f, b0, b1, tw, emax, l1,
                                                     ((threadIdx.x & (B - 1)) + par) << 31, K);
  if (threadIdx.x < B) kout[threadIdx.x] = K;
  __syncthreads();
  T* S = reinterpret_cast<T*>(a.S);
  fx_spectrum<T, LGN, false>(Z, n, lgB, st, bc, f, [&](int b, int q, long long oa, long long ob) {
    const int l = l00 + 2 * b, Kb = kout[b], fl = (b + par) << 31;
    const size_t w = (size_t)l * n + q;
    if (l < nlines && VOFP_IN(w, (size_t)nlines * n, CHK_XFWD_STORE)) S[w] = fx_to(oa, Kb, fl, (T*)nullptr);
    if (l + 1 < nlines && VOFP_IN(w + n, (size_t)nlines * n, CHK_XFWD_STORE)) S[w + n] = fx_to(ob, Kb, fl, (T*)nullptr);
  });
}

// y transform of the column tile blockIdx.x (2^(lgB+1) columns) of plane blockIdx.y, forward or inverse, in place in the
// spectrum.
template <typename T, bool INV, int LGN>
__global__ void __launch_bounds__(fx_bound(LGN), fx_blocks(LGN)) k_ypass_fx(const __grid_constant__ YArgs a,
                                                                         const __grid_constant__ FxTables f) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int emax[8];
  __shared__ unsigned l1[8];
  if (block_skipped(a.skip_conv, a.skip_k, a.tol2)) return;
  constexpr bool CT = LGN > 0;
  const int n = CT ? 1 << LGN : f.fd.n, lgB = CT ? fx_ct_lgB(LGN) : f.lgB, B = 1 << lgB;
  const int st = CT ? B : f.st;
  const int total = n << lgB;
  const int b = threadIdx.x & (B - 1);
  const int i = blockIdx.x * 2 * B + 2 * b;
  const size_t base = (size_t)blockIdx.y * n * a.nx + i;
  [[maybe_unused]] const size_t cells = (size_t)a.nx * a.ny * a.nz;  // (bounds-checked builds)
  T* S = reinterpret_cast<T*>(a.S) + base;
  const int bc = a.bc;
  const bool in0 = i < a.nx, in1 = i + 1 < a.nx;
  cfx *b0, *b1;
  const fxtw* tw = fx_begin(f, smem_raw, b0, b1, emax, l1);
  const int nv = (total - (int)threadIdx.x + (int)blockDim.x - 1) / (int)blockDim.x;
  T ra[8], rb[8];
#pragma unroll
  for (int it = 0; it < 8; ++it) {
    ra[it] = rb[it] = (T)0;
    if (it < nv) {
      const size_t o = (size_t)((threadIdx.x + it * blockDim.x) >> lgB) * a.nx;
      if (in0 && VOFP_IN(base + o, cells, CHK_Y_PASS)) ra[it] = S[o];
      if (in1 && VOFP_IN(base + o + 1, cells, CHK_Y_PASS)) rb[it] = S[o + 1];
    }
  }
  __syncthreads();  // (emax, l1 cleared)
  const int flip = INV ? 0 : (int)(blockIdx.y << 31);
  int K;
  const cfx* Z = fx_transform<T, INV, LGN, 0>(ra, rb, nv, n, lgB, st, bc, f, b0, b1, tw, emax, l1, flip, K);
  auto store = [&](int, int q, long long oa, long long ob) {  // (a thread stays on its column pair)
    const size_t w = (size_t)q * a.nx;
    if (in0 && VOFP_IN(base + w, cells, CHK_Y_PASS)) S[w] = fx_to(oa, K, flip, (T*)nullptr);
    if (in1 && VOFP_IN(base + w + 1, cells, CHK_Y_PASS)) S[w + 1] = fx_to(ob, K, flip, (T*)nullptr);
  };
  if (!INV || quarter_bc(bc)) {
    fx_spectrum<T, LGN, true>(Z, n, lgB, st, bc, f, store);
  } else {
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
      const int q = t >> lgB;
      int idx = q;
      bool fl = false;
      if (bc != VOFP_BC_P) {
        idx = dct_perm(q, n);
        fl = bc == VOFP_BC_DD && (q & 1);
      }
      const cfx y = Z[idx * st + b];
      store(b, q, fx_neg_if(y.x, fl), fx_neg_if(y.y, !fl));
    }
  }
}

// Inverse x transform into the FP64 cell array p.  PLAIN: written, and nothing else; otherwise written or added to (NULL:
// only its size in d2_out) with the sums asked for (as FP64 instructions that are predicated off, they cost the plain
// pass three turns of the FP64 pipe a value: 24.8 -> 22.6 us at 128^3).
template <typename T, int LGN, bool PLAIN>
__global__ void __launch_bounds__(fx_bound(LGN), fx_blocks(LGN)) k_xinv_fx(const __grid_constant__ XInvArgs a,
                                                                        const __grid_constant__ FxTables f) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  __shared__ int emax[8], kout[8];
  __shared__ unsigned l1[8];
  if (block_skipped(a.skip_conv, a.skip_k, a.tol2)) return;
  constexpr bool CT = LGN > 0;
  const int n = CT ? 1 << LGN : f.fd.n, lgB = CT ? fx_ct_lgB(LGN) : f.lgB, B = 1 << lgB;
  const int st = CT ? B + 1 : f.st;
  const int nlines = a.ny * a.nz;
  const int l00 = blockIdx.x * 2 * B;
  const int bc = a.bc;
  const int total = n << lgB;
  cfx *b0, *b1;
  const fxtw* tw = fx_begin(f, smem_raw, b0, b1, emax, l1);
  const T* S = reinterpret_cast<const T*>(a.S);
  const int nv = (total - (int)threadIdx.x + (int)blockDim.x - 1) / (int)blockDim.x;
  T ra[8], rb[8];
#pragma unroll
  for (int it = 0; it < 8; ++it) {
    const int t = threadIdx.x + it * blockDim.x;
    const int pb = CT ? t >> LGN : (n > 1 ? (int)__umulhi((unsigned)t, f.fd.magn) : t), q = t - pb * n;
    const int l = l00 + 2 * pb;
    ra[it] = rb[it] = (T)0;
    if (it < nv) {
      const size_t o = (size_t)l * n + q;
      if (l < nlines && VOFP_IN(o, (size_t)nlines * n, CHK_XINV)) ra[it] = S[o];
      if (l + 1 < nlines && VOFP_IN(o + n, (size_t)nlines * n, CHK_XINV)) rb[it] = S[o + n];
    }
  }
  struct __align__(16) Raw {
    T x, y;
  };
#pragma unroll
  for (int it = 0; it < 8; ++it) {
    const int t = threadIdx.x + it * blockDim.x;
    const int pb = CT ? t >> LGN : (n > 1 ? (int)__umulhi((unsigned)t, f.fd.magn) : t), q = t - pb * n;
    if (it < nv) *reinterpret_cast<Raw*>(b0 + q * st + pb) = {ra[it], rb[it]};
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < 8; ++it) {
    if (it < nv) {
      const Raw w =
          *reinterpret_cast<const Raw*>(b0 + ((threadIdx.x + it * blockDim.x) >> lgB) * st + (threadIdx.x & (B - 1)));
      ra[it] = w.x;
      rb[it] = w.y;
    }
  }
  int K;
  const cfx* Z = fx_transform<T, true, LGN, 1>(ra, rb, nv, n, lgB, st, bc, f, b0, b1, tw, emax, l1, 0, K);
  if (threadIdx.x < B) kout[threadIdx.x] = K;
  __syncthreads();
  double acc = 0, acc2 = 0;
  auto store = [&](int pb, int i, long long oa, long long ob) {
    const int l = l00 + 2 * pb, Kb = kout[pb];
    const size_t w = (size_t)l * n + i;
    const long long ov[2] = {oa, ob};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (l + h >= nlines || !VOFP_IN(w + h * n, (size_t)nlines * n, CHK_XINV)) continue;
      const double v = fx_to(ov[h], Kb, 0, (double*)nullptr);
      if (PLAIN) {
        a.p[w + h * n] = v;
        continue;
      }
      if (a.p && !a.accumulate) a.p[w + h * n] = v;
      else if (a.p) a.p[w + h * n] += v;
      if (a.mean_out) acc = fma(v, __ldg(a.dz + (l + h) / a.ny), acc);
      if (a.d2_out) acc2 = fma(v, v, acc2);
    }
  };
  if (quarter_bc(bc)) {
    fx_spectrum<T, LGN, false>(Z, n, lgB, st, bc, f, store);
  } else {
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
      const int pb = CT ? t >> LGN : (n > 1 ? (int)__umulhi((unsigned)t, f.fd.magn) : t), i = t - pb * n;
      int idx = i;
      bool fl = false;
      if (bc != VOFP_BC_P) {
        idx = dct_perm(i, n);
        fl = bc == VOFP_BC_DD && (i & 1);
      }
      const cfx y = Z[idx * st + pb];
      store(pb, i, fx_neg_if(y.x, fl), fx_neg_if(y.y, !fl));
    }
  }
  if (PLAIN) return;
  if (a.mean_out) {
    const double s = block_sum(acc, red);
    if (threadIdx.x == 0 && s != 0) atomicAdd(a.mean_out, s);
  }
  if (a.d2_out) {
    const double s = block_sum(acc2, red);
    if (threadIdx.x == 0 && s != 0) atomicAdd(a.d2_out, s);
  }
}

}  // namespace vofp
