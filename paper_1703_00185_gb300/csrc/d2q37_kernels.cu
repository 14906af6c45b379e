// sm_103a kernels of one thermal D2Q37 time step, FP64 populations.
//
// Layout (Sec. "Data Structure Analysis"): structure of arrays, one plane per
// population, each plane column-major in y (y contiguous), in a halo frame of
// (Lx + 2*3) columns by NY rows, physical site (x, y) at
// (x + 3) * NY + (y + 16).  NY = Ly + 32 rounded up to a multiple of 16, so every
// column starts on a 128-byte boundary.  Two frames are double-buffered.
//
// Kernels and the step sequence (Sec. "Code Organization"):
//   wrap      pbc: fill the 3-column x halos (and y halos when y is periodic);
//             needed only after a state is uploaded or after a propagate
//             without collide, because collide and fused write the halo
//             images of the edge columns themselves (store_images)
//   propagate pull form of Eq. master2: dst_l(x,y) = src_l(x - c_lx, y - c_ly)
//   bc        diffuse walls on rows 0..2 and Ly-3..Ly-1
//   collide   BGK relaxation (Eq. discrete) to the shifted equilibrium of
//             Eq. MASTERSHIFT3, in place on dst
//   fused     propagate + bc + collide in one pass, src -> dst
//
// Threads: one per lattice site, blocks of 256 consecutive y of one column
// (the paper's 1-D blocks along y, Sec. "The propagate and bc Kernels").
// Every warp reads 32 consecutive doubles of each population plane, so each
// gather is a coalesced 256-byte row shifted by at most 3 elements.
#include <atomic>

#include <cuda_runtime.h>

#include "d2q37_launch.h"

namespace d2q37 {

__constant__ ShellConsts c_shell;

namespace {

constexpr int kBlockY = 256;
constexpr int kWallBlock = 128;

// The batched kernel (D2Q37_BATCH_MIN_BLOCKS x 128 threads per SM, whatever
// its block_y) reads its parameters from memory instead of the constant bank
// and spills a little at 128 registers (56 to 84 bytes per thread); with 3 blocks of
// 128 and no spills it was slower (2970 MLUPS against 3150 for 4, an earlier
// form of the kernel).  On large batches the tile kernels and the per-lattice
// shape (block_y = 0), which runs the single-lattice kernels, are faster.
#ifndef D2Q37_BATCH_MIN_BLOCKS
#define D2Q37_BATCH_MIN_BLOCKS 4
#endif

// P: StepParams or BatchGeo (NY, Hy)
template <class P>
__device__ __forceinline__ long long site_index(const P& p, int x, int y) {
  return (long long)(x + kHx) * p.NY + (y + p.Hy);
}

// Where a site's populations are: in registers, or in the block's shared
// memory (RowPops), read again each time they are needed.
struct RegPops {
  static constexpr bool kSelect = false;  // see largest_high
  const double (&f)[kQ];
  __device__ __forceinline__ double get(int l) const { return f[l]; }
};

// rho, u and T of one site (Sec. "Lattice Boltzmann methods"):
// rho = sum f, rho u = s sum c f, D rho T = sum |xi|^2 f - rho |u|^2 (D = 2),
// the last being sum |xi - u|^2 f expanded.  Pair sums and differences carry
// the even and odd moments.  FP64 arithmetic throughout (the fallback of
// site_moments below).
__device__ __forceinline__ void site_moments_fp64(const double (&f)[kQ], double& rho, double& ux, double& uy,
                                                  double& T) {
  double sh[kShells];
  sh[0] = f[0];
#pragma unroll
  for (int k = 1; k < kShells; ++k) sh[k] = 0.0;
  double jx = 0.0, jy = 0.0;
#pragma unroll
  for (int p = 0; p < kPairs; ++p) {
    const double sum = f[1 + 2 * p] + f[2 + 2 * p];
    const double dif = f[1 + 2 * p] - f[2 + 2 * p];
    sh[pair_shell(p)] += sum;
    if (pair_cx(p) != 0) jx += (double)pair_cx(p) * dif;
    if (pair_cy(p) != 0) jy += (double)pair_cy(p) * dif;
  }
  rho = sh[0];
  double e = 0.0;
#pragma unroll
  for (int k = 1; k < kShells; ++k) {
    rho += sh[k];
    e += (double)shell_c2(k) * sh[k];
  }
  const double inv_rho = 1.0 / rho;
  ux = c_shell.s * jx * inv_rho;
  uy = c_shell.s * jy * inv_rho;
  T = 0.5 * (c_shell.s2 * e * inv_rho - (ux * ux + uy * uy));
}

// The same moments with the sums done in 64-bit integers, off the FP64 pipe
// (GB300 issues 2 FP64 operations per SM per clock but 64+ integer ones).
// Every population is rounded down to the grid of the site's largest
// exponent, 2^(emax - 1075), i.e. to 53 bits relative to the largest
// population, and summed exactly: rho and the moment sums carry one rounding
// per term at that grid (comparable to an FP64 sum) and none from the
// additions.  The roundings are floors, on average 0.5 below for a term whose
// shift drops many bits and less for the largest populations; the sums of r
// and e get a constant back (kFloorR, kFloorE: the mean deficits over
// near-equilibrium states, 16.3 and 104.8 grid units), and those of jx, jy
// need none (sum c = 0).  The remaining -0.3 units of r (-1.2e-17 of rho)
// offset most of the equilibrium's +1.7e-17 (see fx_d0).
// Headroom: |term| < 2^53, |c|^2 <= 10 and 37 terms keep every sum < 2^62.
// Sites with a population that is zero-exponent tiny (< 2^-960), infinite or
// NaN take the FP64 form.
constexpr long long kFloorR = 16, kFloorE = 105;

// top2 = 2 (2^20 emax + 2^20 - 1): the shift emax - e in two instructions, the
// doubling dropping the sign bit (the mantissa bits borrow nothing).
__device__ __forceinline__ long long fixed_term(double v, unsigned top2, unsigned& wrap) {
  const int hi = __double2hiint(v);
  const unsigned d = top2 - 2u * (unsigned)hi;
  wrap = max(wrap, d);  // above top2: v has a larger exponent than emax
  const unsigned sh = d >> 21;
  const int s = hi >> 31;  // 0 or -1
  // the implicit one is set for zero and subnormal inputs too: with emax >= 64
  // their shift is above 62 and they round to 0 (-1 for a negative zero).  A
  // negative v enters as the one's complement of its magnitude, -mant - 1: its
  // arithmetic shift is floor(v 2^-sh) or, when the dropped bits are all zero,
  // one below it
  const int mh = ((hi & 0xFFFFF) | 0x100000) ^ s;
  const int ml = __double2loint(v) ^ s;
  long long r;  // PTX clamps shifts above 63 (C++ leaves them undefined)
  asm("{\n\t.reg .b64 m;\n\tmov.b64 m, {%1, %2};\n\tshr.s64 %0, m, %3;\n\t}" : "=l"(r) : "r"(ml), "r"(mh), "r"(sh));
  return r;
}

// The high word of the population of the largest magnitude: its exponent field
// is the largest exponent.  Two ways, the same result: the maximum of the high
// words, or (F::kSelect) the population itself, selected by its high word.  The
// second costs more, but it is off the common path in the staged kernels, and the
// pulling ones get a better register allocation with it (2048 x 8192 step 2.411 ->
// 2.395 ms; 64 lattices with their own tau in tiles of 128 rows 7.08 -> 6.96 ms); in
// place and in registers the first is faster (separate steps of 1000 x 2050 0.566
// -> 0.544 ms).
template <class F>
__device__ __forceinline__ int largest_high(const F& f) {
  if constexpr (F::kSelect) {
    double m = 0.0;
#pragma unroll
    for (int l = 0; l < kQ; ++l) {
      const double v = f.get(l);
      if ((__double2hiint(v) & 0x7FFFFFFF) > (__double2hiint(m) & 0x7FFFFFFF)) m = v;
    }
    return __double2hiint(m);
  }
  int m = 0;
#pragma unroll
  for (int l = 0; l < kQ; ++l) m = max(m, __double2hiint(f.get(l)) & 0x7FFFFFFF);
  return m;
}

// The exact sums r = sum f, jx, jy = sum c f, e = sum |c|^2 f on the grid
// 2^(emax - 1075), emax the largest exponent.  ANY = false takes the rest
// population's for it, which near equilibrium it is (w_0 is twice the next
// weight), and returns false when it is not; then, with ANY = true, false is
// left for the sites that take the FP64 sums.
template <bool ANY, class F>
__device__ __forceinline__ bool site_sums(const F& f, long long& r, long long& jx, long long& jy,
                                          long long& e, int& emax) {
  const int top = ANY ? largest_high(f) : __double2hiint(f.get(0));
  emax = top >> 20 & 0x7FF;
  const unsigned top2 = 2u * (unsigned)(top | 0xFFFFF);
  unsigned wrap = 0;
  long long sh[kShells];
  sh[0] = fixed_term(f.get(0), top2, wrap);
#pragma unroll
  for (int k = 1; k < kShells; ++k) sh[k] = 0;
  jx = jy = 0;
#pragma unroll
  for (int p = 0; p < kPairs; ++p) {
    const long long vp = fixed_term(f.get(1 + 2 * p), top2, wrap);
    const long long vm = fixed_term(f.get(2 + 2 * p), top2, wrap);
    sh[pair_shell(p)] += vp + vm;
    const long long d = vp - vm;
    jx += pair_cx(p) * d;
    jy += pair_cy(p) * d;
  }
  r = sh[0] + kFloorR;
  e = kFloorE;
#pragma unroll
  for (int k = 1; k < kShells; ++k) {
    r += sh[k];
    e += shell_c2(k) * sh[k];
  }
  return wrap <= top2 && emax >= 64 && emax <= 2046;
}

__device__ __forceinline__ void moments_from_sums(long long r, long long jx, long long jy, long long e, int emax,
                                                  double& rho, double& ux, double& uy, double& T) {
  const double rd = (double)r;
  const double inv = 1.0 / rd;  // the grid scale cancels in u and T
  ux = c_shell.s * (double)jx * inv;
  uy = c_shell.s * (double)jy * inv;
  T = 0.5 * (c_shell.s2 * (double)e * inv - (ux * ux + uy * uy));
  rho = rd * __hiloint2double((emax - 52) << 20, 0);  // 2^(emax - 1075)
}

__device__ __forceinline__ void site_moments(const double (&f)[kQ], double& rho, double& ux, double& uy,
                                             double& T) {
  long long r, jx, jy, e;
  int emax;
  if (site_sums<true>(RegPops{f}, r, jx, jy, e, emax))
    moments_from_sums(r, jx, jy, e, emax, rho, ux, uy, T);
  else
    site_moments_fp64(f, rho, ux, uy, T);
}

// c v for a hop component c in -3..3 given the multiples m = {v, 2v, 3v}.
__device__ __forceinline__ double hop_term(int c, const double (&m)[3]) {
  return c > 0 ? m[c - 1] : -m[-c - 1];
}

// cx ux + cy uy from precomputed multiples: one addition at most.
__device__ __forceinline__ double hop_dot(int cx, int cy, const double (&mx)[3], const double (&my)[3]) {
  if (cx == 0) return hop_term(cy, my);
  if (cy == 0) return hop_term(cx, mx);
  return hop_term(cx, mx) + hop_term(cy, my);
}

// ---- the equilibrium in 64-bit fixed point ---------------------------------
//
// GB300 issues 2 FP64 operations per SM per clock, while the high 64 bits of
// a 64 x 64-bit integer product take about four IMAD.WIDE on the integer
// pipes.  So the equilibrium of the FP64 step is evaluated in fixed point:
// each quantity is an int64 scaled by its own power of two ("Qn": v 2^-n),
// chosen from its range so that every product is the high word of a 128-bit
// product and keeps 2^-55 or better absolute precision on the order-1
// quantities; exact integer sums remove the cancellation that
// limits the FP64 form near T = 0.5 for the outer shells.  Per population
// the result is turned into an FP64 number (fx_convert: the FP64 pipe's integer
// conversion, or integer operations for the last shell) and relaxed with one FP64 FMA.  The shell factor omega w_k is carried as
// c_k 2^E_k with c_k in [0.5, 1).  The ranges that keep every intermediate
// inside its format hold for rho in (0, 4), |T_bar - 1| < 1 and |u_bar| < 0.35
// per component; other sites take the FP64 evaluation.
//
// With K0 = rho (A0 - theta + theta q + theta^2), K1 = rho (theta/2 - theta q/4
// - theta^2), K2 = rho theta^2 / 8, L0 = rho (B1 - 2 theta), L1 = rho theta / 2,
// M0 = rho (B2 - 3 theta / 2), M1 = rho theta / 4 (site values), the shell
// coefficients of collide_site times c_k rho are
//   R0 = c (K0 + x2 K1 + x2^2 K2),  R1 = c (L0 + x2 L1),  R2 = c (M0 + x2 M1),
//   R3 = c rho / 6,  R4 = c rho / 24 (one product: (c/6) 2^64 is (c/24) 2^66),
// and per pair even = R0 + b (R2 + b R4), odd = a (R1 + b R3), b = a^2.
// A signed site value x meets the unsigned shell constants as x + 2^63 (its
// sign bit flipped), which needs no sign fix: x y 2^-64 = (x + 2^63) y 2^-64
// - y / 2, and the y / 2 terms of a shell are one constant subtracted from R0,
// R1 and R2 (fx_d0, fx_d1, fx_d2), together with corrections for the
// roundings of its sums and per-pair products (0.5 below on average for an
// exact high word, 0.75 for umulhi_t).  K0 > 0.74 rho inside the ranges and
// needs no shift.  With the set lowest bit of the conversion (+0.5 on
// average) and two corrections in fx_d0, the equilibrium's mass bias is
// +1.7e-17 per collision relative to omega rho (without the corrections:
// -7.6e-17), which the moment sums' -1.2e-17 nearly cancels.
// The odd part takes a rounded product: a bias there would act on the
// momentum the same way every step.

using u64 = unsigned long long;

// floor(x y 2^-64) for signed x, unsigned y
__device__ __forceinline__ long long mulhi_su(long long x, u64 y) {
  return (long long)(__umul64hi((u64)x, y) - (y & (u64)(x >> 63)));  // x >> 63: 0 or all ones
}

// The high word of a y with the low-by-low partial product left out, the floor
// of a y 2^-64 or one below it (0.75 below on average).
__device__ __forceinline__ u64 umulhi_t(u64 a, u64 y) {
  const unsigned al = (unsigned)a, ah = (unsigned)(a >> 32);
  const unsigned yl = (unsigned)y, yh = (unsigned)(y >> 32);
  const u64 lh = (u64)al * yh;
  const u64 hl = (u64)ah * yl + (lh & 0xFFFFFFFFull);  // < 2^64
  return (u64)ah * yh + (lh >> 32) + (hl >> 32);
}

// The same for a, y < 2^63, whose cross sum fits 64 bits: three 32 x 32 ->
// 64-bit multiply-adds (the per-pair products, which form one chain per pair).
__device__ __forceinline__ u64 umulhi_t63(u64 a, u64 y) {
  const unsigned al = (unsigned)a, ah = (unsigned)(a >> 32);
  const unsigned yl = (unsigned)y, yh = (unsigned)(y >> 32);
  u64 r;
  asm("{\n\t.reg .b64 m;\n\tmul.wide.u32 m, %1, %4;\n\tmad.wide.u32 m, %2, %3, m;\n\tshr.u64 m, m, 32;\n\t"
      "mad.wide.u32 %0, %2, %4, m;\n\t}"
      : "=l"(r)
      : "r"(al), "r"(ah), "r"(yl), "r"(yh));
  return r;
}

// umulhi_t for signed x: x y = (x mod 2^64) y - 2^64 y [x < 0]
__device__ __forceinline__ long long mulhi_su_t(long long x, u64 y) {
  return (long long)(umulhi_t((u64)x, y) - (y & (u64)(x >> 63)));
}

// round(x y 2^-64) (half up) for signed x, unsigned y.  Used where a biased
// rounding would act the same way every step: the odd part of a pair, whose
// magnitude a floor after the sign split would always shrink (a momentum
// damping of 2^-56 per step relative to the odd part).
// The four 32 x 32-bit partial products are independent; the rounding half
// (2^63 of the 128-bit product) enters the middle column as 2^31.
__device__ __forceinline__ long long mulhi_su_rn(long long x, u64 y) {
  const unsigned xl = (unsigned)x, xh = (unsigned)((u64)x >> 32);
  const unsigned yl = (unsigned)y, yh = (unsigned)(y >> 32);
  const u64 ll = (u64)xl * yl, lh = (u64)xl * yh, hl = (u64)xh * yl, hh = (u64)xh * yh;
  const u64 mid = (ll >> 32) + (lh & 0xFFFFFFFFull) + (hl & 0xFFFFFFFFull) + 0x80000000ull;  // < 2^34
  const u64 hi = hh + (lh >> 32) + (hl >> 32) + (mid >> 32);  // floor(((x mod 2^64) y + 2^63) 2^-64)
  return (long long)(hi - (y & (u64)(x >> 63)));
}

// floor(x y 2^-sh) for signed x, y and 0 < sh < 64 (the result fits 64 bits)
__device__ __forceinline__ long long mul_shift(long long x, long long y, int sh) {
  const u64 h = (u64)__mul64hi(x, y);
  const u64 l = (u64)x * (u64)y;
  return (long long)((h << (64 - sh)) | (l >> sh));
}

// g 2^(E - 55) as an FP64 number for odd g, es = (E - 55) 2^20 added to the
// exponent field, two ways: the FP64 pipe's 64-bit integer conversion (round
// to nearest even), or integer operations only (half away from zero).  The
// last shell's 8 populations take the integer form: the FP64 pipe is the
// busiest unit (72 %) and the ALU second (54 %).  2048 x 8192 step 2.412 ms, the
// last two shells 2.394 ms (both before largest_high's last change), the last four and all of them slower (2.49, 2.61
// beside 2.46).  The split stays at one: ties round differently, so moving a
// shell changes the last bits of results.
__device__ __forceinline__ double fx_to_double_fp64(long long g, int es) {
  const double d = (double)g;  // exact up to its one rounding
  return __hiloint2double(__double2hiint(d) + es, __double2loint(d));
}

// |g| >= 2^32
__device__ __forceinline__ double fx_to_double_int(long long g, int es) {
  const int gh = (int)(g >> 32), sm = gh >> 31;
  const unsigned mh = (unsigned)(gh ^ sm), ml = ((unsigned)g ^ (unsigned)sm) | 1u;  // |g|: odd
  // the leading one moved to bit 62 (|g| < 2^63), rounded to 53 bits, 54 when
  // the rounding carries; it adds 1 to the exponent field, a carry one more
  const int lz = __clz((int)mh) - 1;
  const u64 n = ((u64)__funnelshift_l(ml, mh, lz) << 32 | (ml << lz)) + 0x200;
  const u64 mant = n >> 10;
  const int hi = (int)(mant >> 32) + (es + ((1023 + 61) << 20)) - (lz << 20);
  return __hiloint2double(hi | (sm & (int)0x80000000), (int)mant);
}

// The same for any odd g.
__device__ __forceinline__ double fx_to_double_int_any(long long g, int es) {
  const u64 m = g < 0 ? 0ull - (u64)g : (u64)g;
  const int lz = __clzll((long long)m) - 1;
  const u64 mant = ((m << lz) + 0x200) >> 10;
  const int hi = (int)(mant >> 32) + es + ((1023 + 61 - lz) << 20);
  return __hiloint2double(g < 0 ? hi | (int)0x80000000 : hi, (int)mant);
}

// The equilibrium of a population of shell k from its fixed-point value, whose
// lowest bit is set first: it is never zero, and 0.5 larger on average, which
// the per-shell corrections of the equilibrium take into account.  ANY =
// false: the integer form's short version, keeping in `low` the smallest |high
// word| (0: some value needed the other).
template <bool ANY>
__device__ __forceinline__ double fx_convert(int k, long long g, int es, int& low) {
  if (k != kShells - 1) return fx_to_double_fp64(g | 1, es);
  if (ANY) return fx_to_double_int_any(g | 1, es);
  low = min(low, (int)(g >> 32) ^ (int)(g >> 63));
  return fx_to_double_int(g, es);
}

// c v for a hop component c in -3..3 given the multiples m = {v, 2v, 3v}.
__device__ __forceinline__ long long fx_hop_term(int c, const long long (&m)[3]) {
  return c > 0 ? m[c - 1] : -m[-c - 1];
}

__device__ __forceinline__ long long fx_hop_dot(int cx, int cy, const long long (&mx)[3],
                                                const long long (&my)[3]) {
  if (cx == 0) return fx_hop_term(cy, my);
  if (cy == 0) return fx_hop_term(cx, mx);
  return fx_hop_term(cx, mx) + fx_hop_term(cy, my);
}

// Fixed-point site values: rho (Q61), u_x and u_bar_y = u_y + tau g_y (Q64),
// theta = T_bar - 1 (Q62).
struct FxSite {
  u64 R;
  long long UX, UY, TH;
};

// The fixed-point site values straight from the exact moment sums (no FP64
// arithmetic): with r normalised to rn = r 2^n in [2^63, 2^64), X = 2^126 / rn
// from a float seed and two Newton steps (about 2^-60 relative), then
// j / r = (j 2^n) X 2^-126, u = s j / r, 2 T = s^2 e / r - |u|^2 (unshifted u,
// reading R6), rho = r 2^(emax - 1075).  False when the site is outside the
// fixed-point ranges (rho in (0, 4), |u_x|, |u_bar_y| < 0.35, |theta| < 1) or
// its sums do not fit the scaled forms; those sites take the FP64 collision.
template <class P>
__device__ __forceinline__ bool fx_site_from_sums(long long r, long long jx, long long jy, long long e, int emax,
                                                  const P& p, FxSite& o) {
  if (!p.fx_on || r <= 0 || e < 0) return false;
  const u64 ur = (u64)r;
  const u64 ajx = jx < 0 ? 0ull - (u64)jx : (u64)jx, ajy = jy < 0 ? 0ull - (u64)jy : (u64)jy;
  // |j| < r / 2 and e < 3 r keep the scaled sums inside 64 bits (r < 37 2^53)
  if ((ajx << 1) >= ur || (ajy << 1) >= ur || (u64)e >= ur + ur + ur) return false;
  const int n = __clzll(r);  // >= 5
  const u64 rn = ur << n;
  const unsigned top = (unsigned)(rn >> 40);  // [2^23, 2^24), exactly a float below
  const unsigned rb = __float_as_uint(__frcp_rn(__int_as_float(0x4B000000 | (int)(top & 0x7FFFFF))));
  u64 X = (u64)((rb & 0x7FFFFF) | 0x800000) << (((rb >> 23) & 0xFF) - 64);  // 1/top 2^86, Q62 of 2^64/rn
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const u64 pq = __umul64hi(rn, X);          // Q62 of rn X, about 1
    X = __umul64hi(X, (1ull << 63) - pq) << 2;  // X (2 - rn X), Q62; never above 2^64 / rn
  }
  const long long qx = mulhi_su((long long)((u64)jx << n), X);  // Q62 of jx / r
  const long long qy = mulhi_su((long long)((u64)jy << n), X);
  const long long ux61 = mulhi_su(qx, p.fx_s63);  // Q61 of u_x = s jx / r
  const long long uy61 = mulhi_su(qy, p.fx_s63);
  constexpr long long kU = 0x0B33333333333333LL;  // 0.35 2^61
  if (ux61 >= kU || ux61 <= -kU) return false;
  const long long UX = (long long)((u64)ux61 << 3);                      // Q64
  const long long UY0 = (long long)((u64)uy61 << 3);                     // Q64, unshifted
  const long long UY = UY0 + p.fx_uy_shift;                              // Q64 of u_bar_y
  if (UY >= 0x5999999999999999LL || UY <= -0x5999999999999999LL) return false;  // 0.35 2^64
  const u64 aux = UX < 0 ? 0ull - (u64)UX : (u64)UX, auy = UY0 < 0 ? 0ull - (u64)UY0 : (u64)UY0;
  const u64 er = __umul64hi((u64)e << (n - 2), X);                      // Q60 of e / r (< 3)
  const u64 s2er = __umul64hi(er, p.fx_s2_63);                           // Q59 of s^2 e / r
  const u64 q0 = __umul64hi(aux, aux) + __umul64hi(auy, auy);            // Q64 of |u|^2
  const long long th60 = (long long)s2er - (long long)(q0 >> 5) + p.fx_th_shift;  // Q60 of T + shift
  if (th60 >= (1LL << 60) || th60 <= -(1LL << 60)) return false;
  const int sR = emax - 1014;  // rho 2^61 = r 2^sR
  u64 R;
  if (sR >= 0) {
    if (sR >= n) return false;
    R = ur << sR;
  } else {
    const int rs = min(-sR, 63);
    R = (ur + (1ull << (rs - 1))) >> rs;
  }
  if (R == 0 || R >= (1ull << 63)) return false;
  o.R = R;
  o.UX = UX;
  o.UY = UY;
  o.TH = (long long)((u64)th60 << 2);
  return true;
}

// Where a collision puts the relaxed populations: straight into the site's
// planes of the destination, so that each pair's registers are free once it
// is relaxed.
struct ToPlanes {
  char* d;              // the site's element of plane 0
  const StepParams& p;  // plane_off
  __device__ __forceinline__ void put(int l, double v) const { *(double*)(d + p.plane_off[l]) = v; }
};
struct ToPlanesStride {  // the same with the planes addressed as multiples of the stride
  double* d;
  long long plane;
  __device__ __forceinline__ void put(int l, double v) const { d[l * plane] = v; }
};

// The collision of collide_site_fp64 below with the equilibrium in fixed
// point (formats in the comments), for a site inside the fixed-point ranges.
// ANY = false: false is returned when some equilibrium needs the general
// conversion (it is within 2^32 units of 0); the populations written are then
// to be written again with ANY = true.  One test a site: in each conversion it
// cost as much as the conversion.
template <bool ANY, class F, class P, class O>
__device__ __forceinline__ bool collide_site_fx(const F& f, const P& p, const FxSite& fs, const O& out) {
  const long long UX = fs.UX, UY = fs.UY;  // Q64
  const long long TH = fs.TH;              // Q62
  const u64 R = fs.R;                      // Q61
  const u64 AUX = UX < 0 ? 0ull - (u64)UX : (u64)UX, AUY = UY < 0 ? 0ull - (u64)UY : (u64)UY;
  const u64 q = __umul64hi(AUX, AUX) + __umul64hi(AUY, AUY);  // Q64
  const u64 q2 = __umul64hi(q, q);                            // Q64
  const u64 B1 = (1ull << 62) - (q >> 3);                     // Q62: 1 - q/2
  const u64 B2 = (1ull << 61) - (q >> 4);                     //      1/2 - q/4
  const u64 A0 = B1 + (q2 >> 5);                              //      1 - q/2 + q^2/8
  const long long SX = mulhi_su(UX, p.fx_s62), SY = mulhi_su(UY, p.fx_s62);  // Q62
  const long long rA0 = (long long)__umul64hi(R, A0);        // Q59
  const long long rB1 = (long long)__umul64hi(R, B1);        // Q59
  const long long rB2 = (long long)__umul64hi(R, B2);        // Q59
  const long long rth = mul_shift((long long)R, TH, 62);     // Q61: rho theta
  const long long rth2 = mul_shift(rth, TH, 62);             // Q61: rho theta^2
  const long long rthq = mulhi_su(rth, q);                   // Q61: rho theta q
  const long long K0 = rA0 - (rth >> 2) + (rthq >> 2) + (rth2 >> 2);  // Q59
  const long long K1 = (rth >> 2) - (rthq >> 3) - (rth2 >> 1);        // Q60
  const u64 K2 = (u64)rth2;                                           // Q64 (rho theta^2 / 8)
  const long long L0 = rB1 - (rth >> 1);                              // Q59
  const long long M0 = rB2 - (rth >> 2) - (rth >> 3);                 // Q59
  const long long mx[3] = {SX, SX + SX, SX + SX + SX};                // Q62
  const long long my[3] = {SY, SY + SY, SY + SY + SY};
  const u64 kSign = 1ull << 63;
  const u64 uK0 = (u64)K0, uK1 = (u64)K1 ^ kSign, uL0 = (u64)L0 ^ kSign;  // x + 2^63
  const u64 uM0 = (u64)M0 ^ kSign, uTH = (u64)rth ^ kSign;                // L1 = M1 = rth
  const double keep = p.one_minus_omega;
  int low = 0x7FFFFFFF;
  out.put(0, fma(keep, f.get(0),
                 fx_convert<ANY>(0, (long long)(__umul64hi(uK0, p.fx_c60[0]) - p.fx_d0[0]), p.fx_es[0], low)));  // x2 = 0
#pragma unroll
  for (int k = 1; k < kShells; ++k) {
    const long long R0 = (long long)(__umul64hi(uK0, p.fx_c60[k]) + __umul64hi(uK1, p.fx_cx2_59[k]) +
                                     __umul64hi(K2, p.fx_cx4_55[k]) - p.fx_d0[k]);  // Q55
    const long long R1 = (long long)(__umul64hi(uL0, p.fx_c62[k]) + __umul64hi(uTH, p.fx_cx2_59[k]) -
                                     p.fx_d1[k]);  // Q57
    const long long R2 = (long long)(__umul64hi(uM0, p.fx_c64[k]) + __umul64hi(uTH, p.fx_cx2_60[k]) -
                                     p.fx_d2[k]);  // Q59
    const u64 R3 = __umul64hi(R, p.fx_c6[k]);  // Q61 of c rho / 6, and Q63 of R4 = c rho / 24
    const int es = p.fx_es[k];
#pragma unroll
    for (int pr = 0; pr < kPairs; ++pr) {
      if (pair_shell(pr) != k) continue;
      const long long a = fx_hop_dot(pair_cx(pr), pair_cy(pr), mx, my);  // Q62
      const long long sa = a >> 63;                                      // 0 or -1
      const u64 A = (u64)((a ^ sa) - sa);
      const u64 b = umulhi_t63(A, A);                                    // Q60; A < 1.7 2^62
      const long long bR3 = (long long)umulhi_t63(b, R3);                // b < 2.9 2^60, R3 < 2^61
      const long long t = R2 + bR3;                                      // Q59: R2 + b R4
      const long long even = R0 + mulhi_su_t(t, b);                      // Q55
      const long long s = R1 + bR3;                                      // Q57
      const long long oa = mulhi_su_rn(s, A);                            // Q55: |a| (R1 + b R3)
      const long long odd = (oa ^ sa) - sa;                              // the sign of a
      const double gp = fx_convert<ANY>(k, even + odd, es, low);
      const double gm = fx_convert<ANY>(k, even - odd, es, low);
      out.put(1 + 2 * pr, fma(keep, f.get(1 + 2 * pr), gp));
      out.put(2 + 2 * pr, fma(keep, f.get(2 + 2 * pr), gm));
    }
  }
  return low > 0;
}

// BGK collision of one site, f <- f - (f - f^eq(rho, u_bar, T_bar)) / tau with
// u_bar = u + tau g, T_bar = T - tau^2 g^2 / D (Eq. MASTERSHIFT3, Eq. discrete).
// The equilibrium is evaluated per pair as even +- odd parts with per-shell
// coefficients (see ShellConsts), pre-scaled by omega rho w_shell.
template <class F, class P, class O>
__device__ __forceinline__ void collide_site_fp64(const F& f, const P& p, double rho, double ux,
                                                  double uy, double T, const O& out) {
  const double ubx = ux;
  const double uby = uy + p.uy_shift;
  const double q = ubx * ubx + uby * uby;
  const double th = T + p.theta_shift;
  const double A0 = 1.0 + q * (-0.5 + 0.125 * q);
  const double B1 = 1.0 - 0.5 * q;
  const double B2 = 0.5 - 0.25 * q;
  const double sux = c_shell.s * ubx, suy = c_shell.s * uby;
  // a = xi.u_bar = cx sux + cy suy with |cx|, |cy| <= 3: multiples formed once
  const double mx[3] = {sux, sux + sux, sux + sux + sux};
  const double my[3] = {suy, suy + suy, suy + suy + suy};
  const double wr = p.omega * rho;
  const double keep = p.one_minus_omega;
  {
    const double C0 = A0 + th * (c_shell.alpha[0] + q * c_shell.beta[0] + th * c_shell.gamma[0]);
    out.put(0, fma(keep, f.get(0), wr * c_shell.w[0] * C0));
  }
#pragma unroll
  for (int k = 1; k < kShells; ++k) {
    const double W = wr * c_shell.w[k];
    const double P0 = W * (A0 + th * (c_shell.alpha[k] + q * c_shell.beta[k] + th * c_shell.gamma[k]));
    const double P1 = W * (B1 + th * c_shell.delta[k]);
    const double P2 = W * (B2 + th * c_shell.eps[k]);
    const double P3 = W * (1.0 / 6.0);
    const double P4 = W * (1.0 / 24.0);
#pragma unroll
    for (int pr = 0; pr < kPairs; ++pr) {
      if (pair_shell(pr) != k) continue;
      const double a = hop_dot(pair_cx(pr), pair_cy(pr), mx, my);
      const double b = a * a;
      const double even = P0 + b * (P2 + b * P4);
      const double odd = a * (P1 + b * P3);
      out.put(1 + 2 * pr, fma(keep, f.get(1 + 2 * pr), even + odd));
      out.put(2 + 2 * pr, fma(keep, f.get(2 + 2 * pr), even - odd));
    }
  }
}

// One site's collision: moments as exact integer sums, then the fixed-point
// form inside its ranges, else the FP64 form; the relaxed populations to out.
// The common path ends before the rest, which starts again from the
// populations, so that it keeps nothing alive for it.  SHORT = false leaves the
// common path out: populations in registers stay alive for the rest, which 128
// registers do not hold (364 bytes of spills; 142 x 512 periodic 17.5 us a step,
// without 15.7).
template <bool SHORT, class F, class P, class O>
__device__ __forceinline__ void collide_site_to(const F& f, const P& p, const O& out) {
  long long r, jx, jy, e;
  int emax;
  if constexpr (SHORT) {
    FxSite v;
    if (site_sums<false>(f, r, jx, jy, e, emax) && fx_site_from_sums(r, jx, jy, e, emax, p, v) &&
        collide_site_fx<false>(f, p, v, out))
      return;
  }
  double rho, ux, uy, T;
  if (site_sums<true>(f, r, jx, jy, e, emax)) {
    FxSite v;
    if (fx_site_from_sums(r, jx, jy, e, emax, p, v)) {
      collide_site_fx<true>(f, p, v, out);
      return;
    }
    moments_from_sums(r, jx, jy, e, emax, rho, ux, uy, T);
  } else {
    double g[kQ];
#pragma unroll
    for (int l = 0; l < kQ; ++l) g[l] = f.get(l);
    site_moments_fp64(g, rho, ux, uy, T);
  }
  collide_site_fp64(f, p, rho, ux, uy, T, out);
}

// Wall bc for a site of a wall band, applied to its gathered populations:
// rows r = 0..2 from the wall; a population is missing when the pull took it
// from beyond the wall, outgoing when it leaves the column past the wall.
// Missing ones become rho_w f^eq_l(1, 0, T_wall), rho_w = outgoing mass of the
// column / sum of f^eq over the missing pairs, so the wall injects exactly the
// mass that left through it (reading of Sec. "The propagate and bc Kernels").
//
// The outgoing mass is summed row by row, each row's populations in index
// order, and the three row sums as (row 0 + row 1) + row 2: the same grouping
// whether one thread sums the column (wall_density) or the three threads of a
// column's wall rows each sum their own row and combine the sums by warp
// shuffles (wall_band_kernel), so both give the same bits.
// L2: the loads bypass L1 (see launch_pdl).
template <bool L2, class P>  // P: StepParams or BatchGeo (Ly, NY, Hy, plane)
__device__ __forceinline__ double wall_row_outgoing(const double* src, const P& p, int x, int wall, int r) {
  const int y = wall ? p.Ly - 1 - r : r;
  const long long i = site_index(p, x, y);
  double s = 0.0;
#pragma unroll
  for (int l = 0; l < kQ; ++l) {
    const int cy = vel_cy(l);
    if (wall ? (cy > r) : (cy < -r)) s += L2 ? __ldcg(src + (l * p.plane + i)) : src[l * p.plane + i];
  }
  return s;
}

__device__ __forceinline__ double wall_density(const double* src, const StepParams& p, int x, int wall) {
  const double s0 = wall_row_outgoing<false>(src, p, x, wall, 0);
  const double s1 = wall_row_outgoing<false>(src, p, x, wall, 1);
  const double s2 = wall_row_outgoing<false>(src, p, x, wall, 2);
  return ((s0 + s1) + s2) * p.inv_denom[wall];
}

// The missing populations of a wall-band site at row r from the wall; fw:
// the wall's equilibrium f^eq_l(1, 0, T_wall).
__device__ __forceinline__ void apply_wall(double (&f)[kQ], const double* fw, int wall, int r, double rho_w) {
#pragma unroll
  for (int l = 0; l < kQ; ++l) {
    const int cy = vel_cy(l);
    if (wall ? (cy < -r) : (cy > r)) f[l] = rho_w * fw[l];
  }
}

// Write the populations of physical site (x, y) and, for sites within 3 of a
// periodic edge, their halo images, so the next pull finds the halos filled
// (the pbc step folded into the writer; the halo columns see the same values
// the wrap kernel would copy).  x is uniform across a block, so the extra
// stores are divergence-free except on periodic y edges.
__global__ void __launch_bounds__(256) wrap_kernel(double* __restrict__ buf, StepParams p) {
  const int rows_a = p.periodic_y ? p.Ly + 2 * kHx : p.Ly;
  const int y0 = p.periodic_y ? -kHx : 0;
  const long long n_a = (long long)kQ * 6 * rows_a;
  const long long n_b = p.periodic_y ? (long long)kQ * p.Lx * 6 : 0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n_a + n_b;
       t += (long long)gridDim.x * blockDim.x) {
    int l, xd, yd, xs, ys;
    if (t < n_a) {  // x halo columns, whole height (corners included when y is periodic)
      const int yy = (int)(t % rows_a);
      const int h = (int)((t / rows_a) % 6);
      l = (int)(t / (6LL * rows_a));
      xd = h < 3 ? h - 3 : p.Lx + h - 3;
      xs = h < 3 ? p.Lx + h - 3 : h - 3;
      yd = y0 + yy;
      ys = yd < 0 ? yd + p.Ly : (yd >= p.Ly ? yd - p.Ly : yd);
    } else {  // y halo rows of the physical columns (periodic y only)
      const long long u = t - n_a;
      const int r = (int)(u % 6);
      xd = (int)((u / 6) % p.Lx);
      l = (int)(u / (6LL * p.Lx));
      xs = xd;
      yd = r < 3 ? r - 3 : p.Ly + r - 3;
      ys = r < 3 ? p.Ly + r - 3 : r - 3;
    }
    buf[l * p.plane + site_index(p, xd, yd)] = buf[l * p.plane + site_index(p, xs, ys)];
  }
}

__global__ void __launch_bounds__(kBlockY) propagate_kernel(const double* __restrict__ src,
                                                            double* __restrict__ dst, StepParams p) {
  const int x = blockIdx.x;
  const int y = blockIdx.y * kBlockY + threadIdx.x;
  if (y >= p.Ly) return;
  const long long i = site_index(p, x, y);
#pragma unroll
  for (int l = 0; l < kQ; ++l) dst[l * p.plane + i] = src[l * p.plane + i - vel_cx(l) * p.NY - vel_cy(l)];
}

__global__ void __launch_bounds__(128) bc_kernel(const double* __restrict__ src, double* __restrict__ dst,
                                                 StepParams p) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 2 * p.Lx) return;
  const int wall = t >= p.Lx;
  const int x = t - wall * p.Lx;
  const double rho_w = wall_density(src, p, x, wall);
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const int y = wall ? p.Ly - 1 - r : r;
    const long long i = site_index(p, x, y);
#pragma unroll
    for (int l = 0; l < kQ; ++l) {
      const int cy = vel_cy(l);
      if (wall ? (cy < -r) : (cy > r)) dst[l * p.plane + i] = rho_w * p.fw[wall][l];
    }
  }
}

// Byte offset of population plane l: from the parameters, or a multiple of the stride.
template <bool OFF, class P>
__device__ __forceinline__ long long plane_offset(const P& p, int l) {
  if constexpr (OFF)
    return p.plane_off[l];
  else
    return l * p.plane * 8;
}

// The halo images of a site whose populations are already in its own
// element of dst (written by this thread): read back and copied out.  OFF:
// the planes addressed with the byte offsets of p (read from the constant
// bank by the single-lattice kernels) instead of multiples of p.plane.
// PARTS: the populations copied in one go or in halves (where the kernel's 80 or
// 96 registers hold no more; a round trip to L2 longer for the edge sites).
template <bool OFF, int PARTS, class P>
__device__ __forceinline__ void store_images(double* __restrict__ dst, const P& p, int x, int y) {
  if (x >= kHx && x < p.Lx - kHx && (!p.periodic_y || (y >= kHx && y < p.Ly - kHx))) return;
  const char* const s = (const char*)(dst + site_index(p, x, y));
  int xs[3] = {x, 0, 0}, ys[3] = {y, 0, 0};
  int nx = 1, ny = 1;
  if (x < kHx) xs[nx++] = x + p.Lx;
  if (x >= p.Lx - kHx) xs[nx++] = x - p.Lx;
  if (p.periodic_y) {
    if (y < kHx) ys[ny++] = y + p.Ly;
    if (y >= p.Ly - kHx) ys[ny++] = y - p.Ly;
  }
#pragma unroll
  for (int part = 0; part < PARTS; ++part) {
    constexpr int kPart = (kQ + PARTS - 1) / PARTS;
    double f[kPart];
#pragma unroll
    for (int k = 0; k < kPart; ++k) {
      const int l = part * kPart + k;
      if (l < kQ) f[k] = *(const double*)(s + (plane_offset<OFF>(p, l)));
    }
#pragma unroll 1
    for (int ab = 1; ab < nx * ny; ++ab) {  // 0: the site's own element
      const int a = ab / ny, b = ab - a * ny;
      char* const d = (char*)(dst + site_index(p, a == 0 ? xs[0] : a == 1 ? xs[1] : xs[2],
                                               b == 0 ? ys[0] : b == 1 ? ys[1] : ys[2]));
#pragma unroll
      for (int k = 0; k < kPart; ++k) {
        const int l = part * kPart + k;
        if (l < kQ) *(double*)(d + (plane_offset<OFF>(p, l))) = f[k];
      }
    }
  }
}

// ---- populations staged in shared memory by bulk copies --------------------
//
// The blocks of the site kernels (one column x kStageRows rows) fetch their 37
// rows with one bulk copy each (cp.async.bulk, completion on an mbarrier)
// instead of 37 loads a thread.  The loads then need no registers, no address
// arithmetic and no issue slots of the threads, and the populations are read
// from shared memory twice, for the moment sums and for the relaxation, so
// that 24 warps per SM are resident with 80 registers (and a few spills)
// instead of 16 with 128.  Measured on the 2048 x 8192 fused step: 2.70 ms with
// the populations in registers, 2.42 ms this way (5 blocks of 128, 96
// registers: 2.56; 2 of 256, 128 registers: 2.86; 2 of 384: 2.64; 3 of 192:
// 2.61).  Persistent blocks that fetch the next tile into the slots the
// relaxation has finished with wait less for memory but run more instructions,
// and one warp per block lets the warps' code drift apart: both were slower.
constexpr int kStageRows = 256;
constexpr int kStageBlocks = 3;
// A slot holds one population's rows from a 16-byte boundary of the frame: one
// row early when its c_y is odd.
__host__ __device__ constexpr int slot_bytes(int rows) { return (rows + 2) * 8; }
__host__ __device__ constexpr int stage_bytes(int rows) { return kQ * slot_bytes(rows) + 16; }  // and the barrier
constexpr int kStageBytes = stage_bytes(kStageRows);
constexpr int kSharedPerSm = 228 * 1024, kSystemShared = 1024;  // the latter taken from it for every block
constexpr int kWaitLimit = 1 << 20;           // polls of the barrier, each of some microseconds at most

__host__ __device__ constexpr int odd_hops() {
  int n = 0;
  for (int l = 0; l < kQ; ++l) n += vel_cy(l) & 1;
  return n;
}

// One thread's row of the staged populations.  The reads are volatile, so
// that the compiler does not keep the first reading in registers.
template <bool PULL, int ROWS = kStageRows>
struct RowPopsOf {
  static constexpr bool kSelect = PULL;  // see largest_high
  unsigned a;  // shared address of the row in slot 0; 0: the copies did not land
  static __device__ __forceinline__ constexpr int at(int l) { return l * slot_bytes(ROWS) + (PULL ? vel_cy(l) & 1 : 0) * 8; }
  __device__ __forceinline__ double get(int l) const {
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a + at(l)));
    return v;
  }
};
using RowPops = RowPopsOf<true>;

__device__ __forceinline__ bool mbar_wait(unsigned bar) {
  for (int i = 0; i < kWaitLimit; ++i) {
    int ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\tselp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// 3-bit fields of c + 3 of the populations, 21 to a word.
__host__ __device__ constexpr unsigned long long hop_fields(int (*c)(int), int first) {
  unsigned long long w = 0;
  for (int l = first; l < kQ && l < first + 21; ++l) w |= (unsigned long long)(c(l) + 3) << (3 * (l - first));
  return w;
}

// The block's barrier, for the copies of `rows` rows of every population.
template <int ROWS = kStageRows>
__device__ __forceinline__ void stage_init(unsigned char* stage, bool pull, int rows) {
  const unsigned bar = (unsigned)__cvta_generic_to_shared(stage) + kQ * slot_bytes(ROWS);
  const int n_odd = pull ? odd_hops() : 0;
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                 "r"((kQ - n_odd) * ((rows * 8 + 15) & ~15) + n_odd * ((rows * 8 + 23) & ~15))
                 : "memory");
  }
  __syncthreads();
}

// After stage_init: copy `rows` rows from `site` (16-byte aligned) of every
// population into the block's slots, pulled (PULL) or in place, and wait for them.  g: the
// lattice's plane, NY and late.  The hops come from packed fields and the copies are
// spread over the warps: each is started by one lane after the other, and the
// offsets read from the constant bank with an index per lane take as long.
template <bool PULL, int ROWS = kStageRows, class G>
__device__ __forceinline__ RowPopsOf<PULL, ROWS> stage_rows(unsigned char* stage, const char* site, const G& g, int rows) {
  const unsigned slots = (unsigned)__cvta_generic_to_shared(stage);
  const unsigned bar = slots + kQ * slot_bytes(ROWS);
  const int even = (rows * 8 + 15) & ~15, odd = (rows * 8 + 23) & ~15;
  constexpr int per_warp = (kQ + ROWS / 32 - 1) / (ROWS / 32);
  const int lane = threadIdx.x & 31, l = (threadIdx.x >> 5) * per_warp + lane;
  if (lane < per_warp && l < kQ) {
    const char* from = site + l * (g.plane * 8);
    if (PULL) {
      constexpr unsigned long long x0 = hop_fields(vel_cx, 0), x1 = hop_fields(vel_cx, 21);
      constexpr unsigned long long y0 = hop_fields(vel_cy, 0), y1 = hop_fields(vel_cy, 21);
      const int k = 3 * (l < 21 ? l : l - 21);
      const int cx = (int)((l < 21 ? x0 : x1) >> k & 7) - 3, cy = (int)((l < 21 ? y0 : y1) >> k & 7) - 3;
      from -= ((long long)cx * g.NY + cy) * 8;
    }
    const unsigned long long at = (unsigned long long)from;
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     slots + l * slot_bytes(ROWS)),
                 "l"(at & ~15ull), "r"((at & 8) ? odd : even), "r"(bar)
                 : "memory");
  }
  if (!mbar_wait(bar)) {
    // never seen: every thread that ran out tells the host (the next call on the
    // handle returns LBM_ETIMEOUT) and gives the copies in flight the same time
    // again; its row stays unwritten if they do not land then either
    *(volatile unsigned*)g.late = 1u;
    if (!mbar_wait(bar)) return {0u};
  }
  return {slots + threadIdx.x * 8};
}

__global__ void __launch_bounds__(kStageRows, kStageBlocks) collide_kernel(double* __restrict__ buf, StepParams p) {
  extern __shared__ __align__(128) unsigned char stage[];
  const int x = blockIdx.x;
  const int y0 = blockIdx.y * kStageRows;
  const int y = y0 + threadIdx.x;
  const long long i0 = site_index(p, x, y0);
  stage_init(stage, false, min(kStageRows, p.Ly - y0));
  const RowPopsOf<false> f = stage_rows<false>(stage, (const char*)(buf + i0), p, min(kStageRows, p.Ly - y0));
  if (f.a == 0 || y >= p.Ly) return;
  collide_site_to<true>(f, p, ToPlanes{(char*)(buf + i0) + threadIdx.x * 8u, p});
  store_images<true, 2>(buf, p, x, y);
}

// One site of the fused step: gather (pull), wall bc on the wall bands,
// collide, store with halo images.
// p: the lattice (geometry, walls); px: the constants of its collision (tau,
// g: the fixed-point tables, omega, the field shifts), the same object for a
// single lattice.  OFF: addresses from the byte offsets of p (see store_images),
// and loads of the source from L2 (see launch_pdl).
// WALLS = false: the caller never passes a wall-band site.
template <bool OFF, bool WALLS = true, bool SHORT = false>
__device__ __forceinline__ void fused_site(const double* src, double* __restrict__ dst, const StepParams& p,
                                           const Collision& px, int x, int y) {
  const long long i = site_index(p, x, y);
  double f[kQ];
  if constexpr (OFF) {
    const char* s = (const char*)(src + i);
#pragma unroll
    for (int l = 0; l < kQ; ++l) f[l] = __ldcg((const double*)(s + p.pull_off[l]));
  } else {
#pragma unroll
    for (int l = 0; l < kQ; ++l) f[l] = src[l * p.plane + i - vel_cx(l) * p.NY - vel_cy(l)];
  }
  if (WALLS && !p.periodic_y && (y < 3 || y >= p.Ly - 3)) {
    const int wall = y >= p.Ly - 3;
    apply_wall(f, p.fw[wall], wall, wall ? p.Ly - 1 - y : y, wall_density(src, p, x, wall));
  }
  // each pair straight to the site's planes, then the halo images, if any
  if constexpr (OFF)
    collide_site_to<SHORT>(RegPops{f}, px, ToPlanes{(char*)(dst + i), p});
  else
    collide_site_to<SHORT>(RegPops{f}, px, ToPlanesStride{dst + i, p.plane});
  store_images<OFF, OFF ? 1 : 2>(dst, p, x, y);
}

__global__ void __launch_bounds__(kStageRows, kStageBlocks) fused_kernel(const double* src, double* dst,
                                                                        StepParams p) {
  extern __shared__ __align__(128) unsigned char stage[];
  const int x = blockIdx.x;
  const int y0 = blockIdx.y * kStageRows;
  const int y = y0 + threadIdx.x;
  stage_init(stage, true, min(kStageRows, p.Ly - y0));
  // launched with programmatic stream serialization this kernel starts in the
  // tail of the one before it (the previous step's): wait for that grid to
  // complete before the first access
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // the wall-band kernel, launched next the same way, reads and writes nothing
  // this kernel writes, and the previous step is complete here: it may start
  // once every block of this one has come this far, and fill the tail
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const long long i0 = site_index(p, x, y0);
  const RowPops f = stage_rows<true>(stage, (const char*)(src + i0), p, min(kStageRows, p.Ly - y0));
  if (f.a == 0 || y >= p.Ly) return;
  if (!p.periodic_y && (y < 3 || y >= p.Ly - 3)) return;  // wall_band_kernel's
  collide_site_to<true>(f, p, ToPlanes{(char*)(dst + i0) + threadIdx.x * 8u, p});
  store_images<true, 2>(dst, p, x, y);
}

// The same with the populations straight into registers, WARPS resident warps
// per SM: for lattices of few sites, where the length of one site's chain counts
// and not room for other warps, and for columns that fill tiles of 256 rows badly
// (see SiteForm).
template <int ROWS, int WARPS>
__global__ void __launch_bounds__(ROWS, WARPS * 32 / ROWS) fused_reg_kernel(const double* src, double* dst,
                                                                            StepParams p) {
  const int x = blockIdx.x;
  const int y = blockIdx.y * ROWS + threadIdx.x;
  asm volatile("griddepcontrol.wait;" ::: "memory");  // as fused_kernel
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (y >= p.Ly) return;
  if (!p.periodic_y && (y < 3 || y >= p.Ly - 3)) return;  // wall_band_kernel's
  fused_site<true, false, WARPS == 8>(src, dst, p, p, x, y);
}

template <int ROWS>
__global__ void __launch_bounds__(ROWS, 16 * 32 / ROWS) collide_reg_kernel(double* buf, StepParams p) {
  const int x = blockIdx.x;
  const int y = blockIdx.y * ROWS + threadIdx.x;
  if (y >= p.Ly) return;
  char* const b = (char*)(buf + site_index(p, x, y));
  double f[kQ];
#pragma unroll
  for (int l = 0; l < kQ; ++l) f[l] = *(const double*)(b + p.plane_off[l]);
  // in place: every population is read above before its pair is written back
  collide_site_to<false>(RegPops{f}, p, ToPlanes{b, p});
  store_images<true, 1>(buf, p, x, y);
}

// The fused step of the six wall-band rows of every column (y = 0..2 and
// Ly - 3..Ly - 1, walls only), packed into full warps so that the wall bc's
// work runs at warp width instead of in three lanes of a fused_kernel warp (a
// warp holding wall rows cost about three ordinary warps there).  Each warp
// takes ten (column, wall) groups of three lanes, one lane per wall row (lanes
// 30 and 31 idle); every lane sums the populations of its own row that leave
// through the wall, and the group's three row sums meet by warp shuffles, so
// the column's outgoing mass is read once instead of once per wall site.
// Its loads of the source go to L2 (ld.global.cg): no line that this SM's L1
// may hold from an earlier step.
// When it is launched as a programmatic dependent of fused_kernel it may run
// while that kernel's last blocks still run; every thread then waits for the
// sites kernel to complete (griddepcontrol.wait: the prerequisite grid has
// finished and its writes are visible) before it exits.  So this grid never
// completes before the sites kernel, and whatever the stream runs after it
// (the next step's sites kernel reads both kernels' rows) is ordered after
// both, in a stream and in a captured graph alike.  Launched normally, the
// wait returns at once.
constexpr int kWallGroupsPerWarp = 10;

__global__ void __launch_bounds__(kWallBlock) wall_band_kernel(const double* src, double* dst, StepParams p) {
  // the next step's sites kernel may start in this one's tail (it waits for it)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int lane = threadIdx.x & 31;
  const int g = (blockIdx.x * (kWallBlock / 32) + (threadIdx.x >> 5)) * kWallGroupsPerWarp + lane / 3;
  const int r = lane - 3 * (lane / 3);  // row from the wall
  const bool active = lane < 3 * kWallGroupsPerWarp && g < 2 * p.Lx;
  const int x = g >> 1, wall = g & 1;
  const double s = active ? wall_row_outgoing<true>(src, p, x, wall, r) : 0.0;
  const int base = lane - r;  // the group's row-0 lane (idle lanes read lanes 30, 31, 32 mod 32)
  const double s0 = __shfl_sync(0xffffffffu, s, base);
  const double s1 = __shfl_sync(0xffffffffu, s, base + 1);
  const double s2 = __shfl_sync(0xffffffffu, s, base + 2);
  if (active) {
    const int y = wall ? p.Ly - 1 - r : r;
    const long long i = site_index(p, x, y);
    double f[kQ];
    const char* sp = (const char*)(src + i);
#pragma unroll
    for (int l = 0; l < kQ; ++l) f[l] = __ldcg((const double*)(sp + p.pull_off[l]));
    apply_wall(f, p.fw[wall], wall, r, ((s0 + s1) + s2) * p.inv_denom[wall]);
    collide_site_to<true>(RegPops{f}, p, ToPlanes{(char*)(dst + i), p});
    store_images<true, 1>(dst, p, x, y);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Many lattices in one launch: block-sized tiles (one column x, BY
// consecutive y) of every lattice in the table, walked by a grid-stride loop
// (persistent when the grid is sized to the resident blocks).  Lattice i
// reads buffer cur_i ^ parity and writes the other one.
// UNIFORM: every lattice of the launch shares tau and g, so the collision
// constants come from the kernel argument `common` (constant bank, like the
// single-lattice kernel) instead of each lattice's entry.
template <int BY, bool UNIFORM>
__global__ void __launch_bounds__(BY, (D2Q37_BATCH_MIN_BLOCKS * 128) / BY > 0 ? (D2Q37_BATCH_MIN_BLOCKS * 128) / BY : 1)
    batch_fused_kernel(const BatchEntry* __restrict__ tab, const int* __restrict__ tile_entry, int n, long long tiles,
                       int parity, Collision common) {
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
    // owning lattice: per-tile table when given, else binary search; its
    // parameters are read in place (read-only, cached)
    const BatchEntry& e = tab[tile_entry ? tile_entry[t] : batch_entry_of(tab, n, t)];
    const int local = (int)(t - e.tile0);  // tiles of one lattice < 2^31: 32-bit division
    const int x = local / e.ytiles;
    const int y = (local - x * e.ytiles) * BY + threadIdx.x;
    const int c = e.cur ^ parity;
    if (y < e.p.Ly)
      fused_site<false>((const double*)e.buf[c], (double*)e.buf[c ^ 1], e.p,
                        UNIFORM ? common : static_cast<const Collision&>(e.p), x, y);
  }
}

// ---- many lattices in one launch, one block per tile ----------------------
//
// The blocks of site tiles (one column x ROWS rows, the wall rows left out) run
// fused_kernel's per-site work, and the blocks of wall tiles run
// wall_band_kernel's (three lanes per column and wall, the outgoing mass
// combined by warp shuffles), so that no warp of the launch holds a few wall
// rows among ordinary ones.  Geometry comes from the launch's parameter space
// (BatchLaunch, through the constant cache); the collision constants too when
// every lattice shares tau and g (UNIFORM), else each block copies its
// lattice's (BatchEntry) to shared memory.  The owner of a site tile comes from
// a per-tile table or, without one, from a search over the launch's lattices.
// The per-site arithmetic is the single-lattice kernels', so results are the
// same bit for bit.  64 uneven lattices (42.3 M sites), milliseconds a step:
// 7.36 with the populations in registers, 6.62 staged (256 rows, 3 blocks per
// SM); 100 lattices of 60-400 columns, each with its own tau and g: 1.86 as a
// table walked by grid-stride blocks, 1.33 staged (128 rows, 5 blocks per SM).
// Tiles of 256 rows with their own constants are never staged (own_staged).
static_assert(sizeof(BatchLaunch) <= 32700, "BatchLaunch must fit the kernel parameter space");

template <int ROWS, int BLOCKS, bool UNIFORM, bool STAGED>
__global__ void __launch_bounds__(ROWS, BLOCKS)
    batch_tile_kernel(const __grid_constant__ BatchLaunch L, const BatchEntry* __restrict__ tab,
                      const int* __restrict__ tile_entry, int parity) {
  static_assert(!STAGED || BLOCKS * (stage_bytes(ROWS) + (UNIFORM ? 0 : (int)sizeof(Collision)) + kSystemShared) <=
                               kSharedPerSm,
                "blocks per SM that do not fit its shared memory");
  extern __shared__ __align__(128) unsigned char stage[];
  __shared__ Collision own;
  static_assert(sizeof(Collision) % 8 == 0, "Collision is copied in 8-byte words");
  const int b = blockIdx.x;
  if (b < L.site_tiles) {
    const int i = tile_entry ? tile_entry[b] : batch_owner(L, b);
    const BatchGeo& g = L.g[i];
    // x fastest, as in fused_kernel: the columns a tile pulls from run at the same time
    const int local = b - g.tile0;
    const int yt = local / g.Lx;
    const int x = local - yt * g.Lx;
    const int y0 = yt * ROWS, y = y0 + threadIdx.x;
    if (!UNIFORM) {
      const long long* from = (const long long*)static_cast<const Collision*>(&tab[i].p);
      for (int k = threadIdx.x; k < (int)(sizeof(Collision) / 8); k += ROWS) ((long long*)&own)[k] = from[k];
    }
    if constexpr (STAGED) {
      stage_init<ROWS>(stage, true, min(ROWS, g.Ly - y0));
      const int c = g.cur ^ parity;
      const double* src = (const double*)g.buf[c];
      double* dst = (double*)g.buf[c ^ 1];
      const long long at = site_index(g, x, y0);
      const RowPopsOf<true, ROWS> f = stage_rows<true, ROWS>(stage, (const char*)(src + at), g, min(ROWS, g.Ly - y0));
      if (f.a == 0 || y >= g.Ly) return;
      if (!g.periodic_y && (y < 3 || y >= g.Ly - 3)) return;  // the wall tiles'
      const ToPlanesStride out{dst + at + threadIdx.x, g.plane};
      if constexpr (UNIFORM)
        collide_site_to<true>(f, L.common, out);
      else
        collide_site_to<true>(f, own, out);
      store_images<false, 2>(dst, g, x, y);
    } else {
      if (!UNIFORM) __syncthreads();
      if (y >= g.Ly) return;
      if (!g.periodic_y && (y < 3 || y >= g.Ly - 3)) return;
      const int c = g.cur ^ parity;
      const double* src = (const double*)g.buf[c];
      double* dst = (double*)g.buf[c ^ 1];
      const long long at = site_index(g, x, y);
      double f[kQ];
#pragma unroll
      for (int l = 0; l < kQ; ++l) f[l] = src[l * g.plane + at - vel_cx(l) * g.NY - vel_cy(l)];
      const ToPlanesStride out{dst + at, g.plane};
      if constexpr (UNIFORM)
        collide_site_to<false>(RegPops{f}, L.common, out);
      else
        collide_site_to<false>(RegPops{f}, own, out);
      store_images<false, 1>(dst, g, x, y);
    }
    return;
  }
  // wall tile: kWallGroupsPerWarp (column, wall) groups per warp, one lane per wall row
  const int w = b - L.site_tiles;
  int i = 0;
  for (int hi = L.n - 1; i < hi;) {  // lattices without walls own no wall tiles: the last with wtile0 <= w
    const int mid = (i + hi + 1) >> 1;
    if (L.g[mid].wtile0 <= w)
      i = mid;
    else
      hi = mid - 1;
  }
  const BatchGeo& g = L.g[i];
  const int lane = threadIdx.x & 31;
  const int grp = ((w - g.wtile0) * (ROWS / 32) + (threadIdx.x >> 5)) * kWallGroupsPerWarp + lane / 3;
  const int r = lane - 3 * (lane / 3);
  const bool active = lane < 3 * kWallGroupsPerWarp && grp < 2 * g.Lx;
  const int x = grp >> 1, wall = grp & 1;
  const int c = g.cur ^ parity;
  const double* src = (const double*)g.buf[c];
  const double sum = active ? wall_row_outgoing<false>(src, g, x, wall, r) : 0.0;
  const int base = lane - r;
  const double s0 = __shfl_sync(0xffffffffu, sum, base);
  const double s1 = __shfl_sync(0xffffffffu, sum, base + 1);
  const double s2 = __shfl_sync(0xffffffffu, sum, base + 2);
  if (!active) return;
  const int y = wall ? g.Ly - 1 - r : r;
  const long long at = site_index(g, x, y);
  double f[kQ];
#pragma unroll
  for (int l = 0; l < kQ; ++l) f[l] = src[l * g.plane + at - vel_cx(l) * g.NY - vel_cy(l)];
  const StepParams& p = tab[i].p;
  apply_wall(f, p.fw[wall], wall, r, ((s0 + s1) + s2) * g.inv_denom[wall]);
  double* dst = (double*)g.buf[c ^ 1];
  const ToPlanesStride out{dst + at, g.plane};
  if constexpr (UNIFORM)
    collide_site_to<false>(RegPops{f}, L.common, out);
  else
    collide_site_to<false>(RegPops{f}, p, out);
  store_images<false, 2>(dst, g, x, y);
}

__global__ void __launch_bounds__(kBlockY) fields_kernel(const double* buf, double* rho, double* u, double* T,
                                                         StepParams p) {
  asm volatile("griddepcontrol.wait;" ::: "memory");  // chained to the step before it (see fused_kernel)
  const int x = blockIdx.x;
  const int y = blockIdx.y * kBlockY + threadIdx.x;
  if (y >= p.Ly) return;
  const long long i = site_index(p, x, y);
  double f[kQ];
#pragma unroll
  for (int l = 0; l < kQ; ++l) f[l] = __ldcg(buf + (l * p.plane + i));  // see launch_pdl
  double r, ux, uy, t;
  site_moments(f, r, ux, uy, t);
  const long long o = (long long)x * p.Ly + y;
  const long long n = (long long)p.Lx * p.Ly;
  rho[o] = r;
  u[o] = ux;
  u[n + o] = uy;
  T[o] = t;
}

// SplitMix64 (Steele, Lea & Flood, OOPSLA 2014): the finaliser applied to
// state v + 0x9e3779b97f4a7c15.
__device__ __forceinline__ u64 splitmix64(u64 v) {
  u64 z = v + 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

// The Rayleigh-Taylor initial state: the temperature of a site from its side
// of the interface yi[x] (host, one sine a column) and its noise, each
// operation rounded on its own, rho = 1/T, populations f^eq(rho, 0, T) or, in
// FP32 storage, their deviations from the weights.  At u = 0 every population
// of a shell is rho w C0, C0 = 1 + theta (alpha + theta gamma).  1024 x 4096
// FP64: 8.8 ms for the call with the temperatures made by one host core
// (2.1 ns a site) and uploaded, 0.41 ms this way (the kernel 0.39, of which 0.18
// are HBM writes; the rest is FP64, mostly the division).
template <class T>
__global__ void __launch_bounds__(kBlockY) init_rayleigh_taylor_kernel(T* __restrict__ buf, const double* __restrict__ yi,
                                                                       double T_top, double T_bot, u64 seed,
                                                                       StepParams p) {
  const int x = blockIdx.x;
  const int y = blockIdx.y * kBlockY + threadIdx.x;
  if (y >= p.Ly) return;
  const double U = __dmul_rn((double)(splitmix64(seed + (u64)x * (u64)p.Ly + (u64)y) >> 11), 0x1.0p-53);
  const double T0 = (double)y + 0.5 < yi[x] ? T_bot : T_top;
  const double t = __dmul_rn(T0, __dadd_rn(1.0, __dmul_rn(1e-3, __dsub_rn(__dmul_rn(2.0, U), 1.0))));
  const double rho = 1.0 / t, th = t - 1.0;
  T* const f = buf + site_index(p, x, y);
#pragma unroll
  for (int k = 0; k < kShells; ++k) {
    const double C0 = fma(th, fma(th, c_shell.gamma[k], c_shell.alpha[k]), 1.0);
    const double W = rho * c_shell.w[k];
    const T v = sizeof(T) == sizeof(float) ? (T)fma(W, C0, -c_shell.w[k]) : (T)(W * C0);
#pragma unroll
    for (int l = 0; l < kQ; ++l)
      if (vel_shell(l) == k) f[l * p.plane] = v;
  }
}

dim3 site_grid(const StepParams& p) { return dim3(p.Lx, (p.Ly + kBlockY - 1) / kBlockY); }

// (column, wall) groups of the wall-band kernel: 2 Lx, ten per warp
int wall_grid(const StepParams& p) {
  constexpr int per_block = kWallGroupsPerWarp * (kWallBlock / 32);
  return (2 * p.Lx + per_block - 1) / per_block;
}

int done(int n) { return cudaGetLastError() == cudaSuccess ? n : -1; }

}  // namespace

// SMs of the current device, looked up once per device.
int sm_count() {
  static std::atomic<int> known[256];
  int dev = 0, v = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return 152;
  if ((v = known[dev].load(std::memory_order_relaxed)) > 0) return v;
  if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) return 152;
  known[dev].store(v, std::memory_order_relaxed);
  return v;
}

int launch_wrap(double* buf, const StepParams& p, cudaStream_t stream) {
  const long long n = (long long)kQ * 6 * (p.periodic_y ? p.Ly + 2 * kHx : p.Ly) +
                      (p.periodic_y ? (long long)kQ * p.Lx * 6 : 0);
  long long blocks = (n + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  wrap_kernel<<<(unsigned)blocks, 256, 0, stream>>>(buf, p);
  return done(1);
}

int launch_propagate(const double* src, double* dst, const StepParams& p, cudaStream_t stream) {
  propagate_kernel<<<site_grid(p), kBlockY, 0, stream>>>(src, dst, p);
  return done(1);
}

int launch_bc(const double* src, double* dst, const StepParams& p, cudaStream_t stream) {
  bc_kernel<<<(2 * p.Lx + 127) / 128, 128, 0, stream>>>(src, dst, p);
  return done(1);
}

// The form of a sites kernel: rows per block and warps per SM of a register form
// (255 registers with 8 warps, 128 with 16), or the staged one (rows = 0).
// Microseconds a step, "w" = warps of 32 rows per SM; the best of blocks of 32
// and 128 rows; chained or not as launch_fused has it:
//                           staged  255 regs  128 regs   before the staged form
//  walls     38 x 512   4 w   14.3      12.8      14.3
//            76 x 512   8 w   17.3      21.3      15.9
//           142 x 512  15 w   22.3      22.9      17.8    18.9
//           185 x 512  19 w   24.0      31.2      25.1
//           570 x 512  60 w   64.5      85.7      61.4    68.6
//          1500 x 512 158 w  139.2     191.8     135.9
//          2375 x 512 250 w  207.1     291.4     205.6   220.0
//          8000 x 512 842 w  662.9     949.2     673.3
//           256 x 8192 431 w 324.1     480.6     338.1
//  periodic  64 x 64          9.8       8.6       8.4     8.8
//           142 x 512  15 w   18.3      19.4      15.6    17.1
//           285 x 512  30 w   30.5      37.5      27.7    30.3
//           570 x 512  60 w   59.0      77.8      55.3    60.0
//          1140 x 512 120 w  102.5     143.5     101.1   106.5
//          1900 x 512 200 w  159.2     231.0     161.0
struct SiteForm {
  int rows, warps;
};
constexpr SiteForm kStaged = {0, 0};

// 128 registers: blocks of 32 rows leave the fewest threads idle (512 x 257
// periodic 27.6 us, of 128 rows 32.4).  Blocks of 128 have fewer warps with edge
// rows and are fewer to start: 60 lattices of 120 x 240 on four streams 347 us, of
// 32 rows 369.
SiteForm reg_form(int rows) {
  const bool one = rows > 32 && rows <= 128, full = rows * 10LL >= 9 * 128LL * ((rows + 127) / 128);
  return {one || full ? 128 : 32, 16};
}

// Whether a register form's blocks over Lx columns of `rows` rows and `walls`
// blocks of the wall-band kernel (246 registers) are all resident at once.
bool form_resident(SiteForm f, int Lx, int rows, int walls) {
  const long long warps = (long long)Lx * ((rows + f.rows - 1) / f.rows) * (f.rows / 32);
  return warps + walls * (kWallBlock / 32) * (f.warps / 8) <= (long long)f.warps * sm_count();
}

long long stage_tiles(int Lx, int rows) { return (long long)Lx * ((rows + kStageRows - 1) / kStageRows); }

// Whether the staged tiles take no more than nine tenths of the room.
bool one_wave(int Lx, int rows) { return stage_tiles(Lx, rows) * 10 <= 9LL * kStageBlocks * sm_count(); }

// Whether the staged tiles hold so few rows that 128 registers win at any size
// (their idle warps keep a third of the SM's warps from running): below 0.92 of
// 256 rows a tile, below a half where the staged tiles are one wave.  Staged / 128
// registers, walls: 1500 x 300 (0.58) 113.6 / 91.3 us, 4000 x 640 (0.83) 437.5 /
// 414.6, 4000 x 700 (0.91) 458 / 452, 3000 x 1200 (0.935) 568 / 574, 4000 x 1000
// (0.97) 622 / 644; periodic 1500 x 300 117.7 / 85.0, 4000 x 640 432 / 408, 4000 x 700
// 456 / 446, 4000 x 480 (0.94) 304 / 311; one wave: 256 x 196 (0.75) not chained 17.5 /
// 21.0, 400 x 100 (0.38) 24.3 / 18.3.  Beside other streams' grids below 0.8 (a
// server's 16 jobs of 200 to 500 columns 54.7 ms, with 0.92 57.5).
bool poor_fill(int Lx, int rows, bool alone) {
  const long long room = stage_tiles(1, rows) * kStageRows;
  return rows * 100LL < (one_wave(Lx, rows) ? 50 : alone ? 92 : 80) * room;
}

// Up to this many warps of rows per SM 128 registers win (the table above); beside
// other streams' grids less.
constexpr int kRegWarps = 150, kRegWarpsShared = 40;
bool few_warps(int Lx, int rows, bool alone) {
  return (long long)Lx * ((rows + 31) / 32) <= (long long)(alone ? kRegWarps : kRegWarpsShared) * sm_count();
}

// alone: no other stream's grids beside this one.  Beside others, walled lattices
// that do not fill the GPU many times over keep the staged form, which leaves room
// (a server's burst of 12 jobs 17.5 ms, 19.3 with tiles filled badly in 128
// registers; 16 jobs of 200 to 500 columns 54.7, 59.6), and no lattice takes 255
// registers.  Walled lattices of one wave take a register form only where the
// wall-band kernel has room beside it; else staged blocks leave it some (142 x 512 not
// chained 18.6 us, 21.9 in 128 registers).
SiteForm fused_form(const StepParams& p, int rows, int walls, bool chain, bool alone) {
  const SiteForm reg = reg_form(rows);
  if (p.periodic_y ? alone : chain)
    for (const SiteForm f : {SiteForm{rows > 32 ? 128 : 32, 8}, SiteForm{32, 8}})
      if (form_resident(f, p.Lx, rows, walls)) return f;
  const bool few = few_warps(p.Lx, rows, alone);
  if (p.periodic_y) return few || poor_fill(p.Lx, rows, alone) ? reg : kStaged;
  if (!alone && few) return kStaged;
  if (chain && form_resident(reg, p.Lx, rows, walls)) return reg;
  if (poor_fill(p.Lx, rows, alone)) return reg;
  return alone && few && !one_wave(p.Lx, rows) ? reg : kStaged;
}

int launch_collide(double* buf, const StepParams& p, cudaStream_t stream) {
  const SiteForm form = poor_fill(p.Lx, p.Ly, true) || few_warps(p.Lx, p.Ly, true) ? reg_form(p.Ly) : kStaged;
  void (*const kernel)(double*, StepParams) =
      !form.rows ? collide_kernel : form.rows == 128 ? collide_reg_kernel<128> : collide_reg_kernel<32>;
  const int rows = form.rows ? form.rows : kStageRows;
  kernel<<<dim3(p.Lx, (p.Ly + rows - 1) / rows), rows, form.rows ? 0 : kStageBytes, stream>>>(buf, p);
  return done(1);
}

int launch_fused(const double* src, double* dst, const StepParams& p, cudaStream_t stream, bool overlap, bool chain,
                 bool alone) {
  // the last three rows of a walled lattice are the wall-band kernel's
  const int Ly = p.periodic_y ? p.Ly : p.Ly - 3, walls = p.periodic_y ? 0 : wall_grid(p);
  const SiteForm form = fused_form(p, Ly, walls, chain, alone);
  void (*const sites)(const double*, double*, StepParams) =
      !form.rows         ? fused_kernel
      : form.warps == 8  ? (form.rows == 128 ? fused_reg_kernel<128, 8> : fused_reg_kernel<32, 8>)
      : form.rows == 128 ? fused_reg_kernel<128, 16>
                         : fused_reg_kernel<32, 16>;
  const int rows = form.rows ? form.rows : kStageRows;
  const dim3 grid(p.Lx, (Ly + rows - 1) / rows);
  // The next step's blocks wait where this one's leave room.  With 255 registers
  // that hides the launch.  Between half and all of the room they pile up on some
  // SMs, and the step after runs unevenly (100 x 512 periodic 15.0 us, not chained
  // 13.1); with walls and more than one wave they keep the wall-band kernel
  // from its room (2375 x 512 210.6 us, 207.1; 185 x 512, one wave, 24.0, 27.4).
  const long long used = (long long)grid.x * grid.y * (rows / 32), room = (long long)form.warps * sm_count();
  if (p.periodic_y)
    chain = chain && (form.warps != 16 || used * 12 <= room * 5 || used * 10 >= room * 9);
  else
    chain = chain && (form.rows ? form_resident(form, p.Lx, Ly, walls) : one_wave(p.Lx, Ly));
  if (!launch_pdl(sites, grid, rows, form.rows ? 0 : kStageBytes, stream, chain, src, dst, p)) return -1;
  if (p.periodic_y) return done(1);
  if (!launch_pdl(wall_band_kernel, dim3(walls), kWallBlock, 0, stream, overlap, src, dst, p)) return -1;
  return done(2);
}

template <int BY>
int batch_launch(const BatchEntry* tab, const int* tile_entry, int n, long long tiles, int parity, int grid,
                 const Collision* common, cudaStream_t stream) {
  if (common)
    batch_fused_kernel<BY, true><<<grid, BY, 0, stream>>>(tab, tile_entry, n, tiles, parity, *common);
  else
    batch_fused_kernel<BY, false><<<grid, BY, 0, stream>>>(tab, tile_entry, n, tiles, parity, Collision{});
  return done(1);
}

template <int BY>
int batch_occupancy() {
  int b = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, batch_fused_kernel<BY, true>, BY, 0);
  return b;
}

int launch_batch_fused(const BatchEntry* tab, const int* tile_entry, int n, long long tiles, int parity,
                       int block_y, int grid, const Collision* common, cudaStream_t stream) {
  switch (block_y) {
    case 64: return batch_launch<64>(tab, tile_entry, n, tiles, parity, grid, common, stream);
    case 128: return batch_launch<128>(tab, tile_entry, n, tiles, parity, grid, common, stream);
    case 256: return batch_launch<256>(tab, tile_entry, n, tiles, parity, grid, common, stream);
    default: return -1;
  }
}

namespace {

// Whether BLOCKS staged blocks and their copies of the collision constants fit an
// SM.  Three of 256 rows do not (352 bytes short); two of them took the same 80
// registers: 24 lattices of 1024 x 1024 4.69 ms a step, in registers 4.53.
constexpr bool own_staged(int rows, int blocks) {
  return blocks * (stage_bytes(rows) + (int)sizeof(Collision) + kSystemShared) <= kSharedPerSm;
}

template <int ROWS, int BLOCKS>
cudaError_t allow_tile_memory() {
  cudaError_t e = cudaFuncSetAttribute(batch_tile_kernel<ROWS, BLOCKS, true, true>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, stage_bytes(ROWS));
  if constexpr (own_staged(ROWS, BLOCKS))
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(batch_tile_kernel<ROWS, BLOCKS, false, true>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, stage_bytes(ROWS));
  return e;
}

// Up to this many warps of sites per SM (some waves) the register form (128
// registers, 16 warps per SM) is the faster one: a wave is one site's chain
// long, and the bulk copies add theirs.  Microseconds a step in registers /
// staged, 128 rows, walls: shared tau and g 3 lattices of 40 x 80 (2 warps) 17.0 /
// 21.1, 10 of 120 x 240 (63) 81.7 / 83.4, 14 (88) 105.5 / 104.7, 20 (126) 139 /
// 137, 40 of 100 x 97 (105) 121 / 126, 60 of 120 x 240 (379) 372 / 359, 24 of
// 1024 x 1024 (5174) 4449 / 4084; their own 10 (63) 85 / 93, 20 (126) 145 / 151,
// 30 (189) 207 / 210, 60 (379) 394 / 384.
constexpr int kBatchFewWarps = 120, kBatchFewWarpsOwn = 250;

template <int ROWS, int BLOCKS>
int tile_launch(const BatchLaunch& L, bool uniform, const BatchEntry* tab, const int* tile_entry, int parity,
                cudaStream_t stream) {
  constexpr int kRegBlocks = 4 * 128 / ROWS;
  const int grid = L.site_tiles + L.wall_tiles;
  const bool staged =
      (uniform || own_staged(ROWS, BLOCKS)) &&
      L.site_warps > (long long)(uniform ? kBatchFewWarps : kBatchFewWarpsOwn) * sm_count();
  void (*kernel)(BatchLaunch, const BatchEntry*, const int*, int) =
      uniform ? batch_tile_kernel<ROWS, kRegBlocks, true, false> : batch_tile_kernel<ROWS, kRegBlocks, false, false>;
  if (staged && uniform) kernel = batch_tile_kernel<ROWS, BLOCKS, true, true>;
  if constexpr (own_staged(ROWS, BLOCKS))
    if (staged && !uniform) kernel = batch_tile_kernel<ROWS, BLOCKS, false, true>;
  kernel<<<grid, ROWS, staged ? stage_bytes(ROWS) : 0, stream>>>(L, tab, tile_entry, parity);
  return done(1);
}

// With walls and up to 8 warps of sites per SM the table kernel is faster: its wall
// rows are a few lanes' longer chain in a block of sites, where a wall tile's
// chain waits for its row sums first.  So it is where the wall tiles alone would
// start a second or third wave.  Microseconds a step, tiles / table, 128 rows: 2
// lattices of 16 x 40 18.0 / 13.6, 6 of 40 x 80 (5 warps) 18.0 / 14.8, 5 of 60 x 120
// (8) 20.9 / 16.6, 6 (9.5) 21.0 / 18.9, 8 (13) 23.6 / 24.0, 3 of 120 x 240 (19) 31.2 /
// 35.9, 5 (32, two waves and the wall tiles) 50.2 / 44.2; with their own tau and g
// 18.9 / 14.8, 18.7 / 15.5, 22.9 / 16.7, 22.0 / 18.8, 24.0 / 23.3, 32.1 / 36.3, 53.1 /
// 46.3 (64 rows 51.7 / 53.1).  Without walls tiles win: 10.7 / 11.5 on the first.
constexpr int kBatchTableWarps = 8;

bool table_is_faster(const BatchLaunch& L, int block_y) {
  if (!L.wall_tiles) return false;
  if (L.site_warps <= (long long)kBatchTableWarps * sm_count()) return true;
  const long long slots = (long long)(16 * 32 / block_y) * sm_count();
  const long long sites = (L.site_tiles + slots - 1) / slots, all = (L.site_tiles + L.wall_tiles + slots - 1) / slots;
  return block_y >= 128 && sites <= 2 && all > sites;
}

}  // namespace

int launch_batch_tiles(const BatchLaunch& L, bool uniform, const BatchEntry* tab, const int* tile_entry, int parity,
                       int block_y, cudaStream_t stream) {
  if (table_is_faster(L, block_y))
    return launch_batch_fused(tab, tile_entry, L.n, L.site_tiles, parity, block_y, L.site_tiles,
                              uniform ? &L.common : nullptr, stream);
  switch (block_y) {
    case 64: return tile_launch<64, 10>(L, uniform, tab, tile_entry, parity, stream);
    case 128: return tile_launch<128, 5>(L, uniform, tab, tile_entry, parity, stream);
    case 256: return tile_launch<256, 3>(L, uniform, tab, tile_entry, parity, stream);
    default: return -1;
  }
}

cudaError_t upload_shell_consts(const ShellConsts& c) {
  cudaError_t e = cudaFuncSetAttribute(fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kStageBytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(collide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kStageBytes);
  if (e == cudaSuccess) e = allow_tile_memory<64, 10>();
  if (e == cudaSuccess) e = allow_tile_memory<128, 5>();
  if (e == cudaSuccess) e = allow_tile_memory<256, 3>();
  return e == cudaSuccess ? cudaMemcpyToSymbol(c_shell, &c, sizeof(c)) : e;
}

int batch_wall_groups_per_tile(int block_y) { return (block_y / 32) * kWallGroupsPerWarp; }

int batch_blocks_per_sm(int block_y) {
  switch (block_y) {
    case 64: return batch_occupancy<64>();
    case 128: return batch_occupancy<128>();
    case 256: return batch_occupancy<256>();
    default: return 0;
  }
}

int launch_fields(const double* buf, double* rho, double* u, double* T, const StepParams& p, cudaStream_t stream,
                  bool chain) {
  return launch_pdl(fields_kernel, site_grid(p), kBlockY, 0, stream, chain, buf, rho, u, T, p) ? done(1) : -1;
}

int launch_init_rayleigh_taylor(void* buf, bool fp32, const double* yi, double T_top, double T_bot,
                                unsigned long long seed, const StepParams& p, cudaStream_t stream) {
  if (fp32)
    init_rayleigh_taylor_kernel<<<site_grid(p), kBlockY, 0, stream>>>((float*)buf, yi, T_top, T_bot, seed, p);
  else
    init_rayleigh_taylor_kernel<<<site_grid(p), kBlockY, 0, stream>>>((double*)buf, yi, T_top, T_bot, seed, p);
  return done(1);
}

}  // namespace d2q37
