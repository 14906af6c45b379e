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
#include <cuda_runtime.h>

#include "d2q37_launch.h"

namespace d2q37 {

__constant__ ShellConsts c_shell;

namespace {

constexpr int kBlockY = 256;
constexpr int kWallBlock = 128;

// Minimum resident blocks per SM requested for the FP64 site kernels (caps
// their registers at 65536 / (kBlockY * blocks)); tuned on GB300: 2 blocks of
// 256 (128 registers) ran the 2048 x 8192 fused step in 2.79 ms, against
// 2.84 ms with 8 of 64, 2.87 ms with 4 of 128 and 3.53 ms with 1 of 512.
#ifndef D2Q37_SITE_MIN_BLOCKS
#define D2Q37_SITE_MIN_BLOCKS 2
#endif
// The batched kernel (D2Q37_BATCH_MIN_BLOCKS x 128 threads per SM, whatever
// its block_y) reads its parameters from memory instead of the constant bank
// and spills a little at 128 registers (20 bytes per thread); with 3 blocks of
// 128 and no spills it was slower (2970 MLUPS against 3150 for 4, an earlier
// form of the kernel).  The batch's per-lattice shape (block_y = 0), which
// runs the single-lattice kernels, is faster still on the 64-lattice workload.
#ifndef D2Q37_BATCH_MIN_BLOCKS
#define D2Q37_BATCH_MIN_BLOCKS 4
#endif

// P: StepParams or BatchGeo (NY, Hy)
template <class P>
__device__ __forceinline__ long long site_index(const P& p, int x, int y) {
  return (long long)(x + kHx) * p.NY + (y + p.Hy);
}

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
__device__ __forceinline__ long long fixed_term(double v, unsigned top2) {
  const int hi = __double2hiint(v);
  const unsigned sh = (top2 - 2u * (unsigned)hi) >> 21;
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

// The exact sums r = sum f, jx, jy = sum c f, e = sum |c|^2 f on the grid
// 2^(emax - 1075); false for the sites that take the FP64 sums.
__device__ __forceinline__ bool site_sums(const double (&f)[kQ], long long& r, long long& jx, long long& jy,
                                          long long& e, int& emax) {
  // the largest |high word| (its exponent field is the largest exponent): the
  // signed maximum finds the largest positive one, the unsigned one the
  // largest negative one
  int hs = 0;
  unsigned hu = 0;
#pragma unroll
  for (int l = 0; l < kQ; ++l) {
    hs = max(hs, __double2hiint(f[l]));
    hu = max(hu, (unsigned)__double2hiint(f[l]));
  }
  const int hmax = max(hs, (int)(hu & 0x7FFFFFFFu));
  emax = hmax >> 20;
  if (emax < 64 || emax > 2046) return false;
  const unsigned top2 = 2u * (unsigned)(hmax | 0xFFFFF);
  long long sh[kShells];
  sh[0] = fixed_term(f[0], top2);
#pragma unroll
  for (int k = 1; k < kShells; ++k) sh[k] = 0;
  jx = jy = 0;
#pragma unroll
  for (int p = 0; p < kPairs; ++p) {
    const long long vp = fixed_term(f[1 + 2 * p], top2);
    const long long vm = fixed_term(f[2 + 2 * p], top2);
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
  return true;
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
  if (site_sums(f, r, jx, jy, e, emax))
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
// GB300 issues 2 FP64 operations per SM per clock, while a 32 x 32 -> 64-bit
// multiply-add (IMAD.WIDE) runs at about 32.  So the equilibrium of the FP64
// step is evaluated in fixed point: each quantity is a signed 64-bit integer
// scaled by its own power of two ("Qn": v 2^-n), and a product is the high
// word of a 128-bit product (fx_mul: three multiply-adds).
//
// The equilibrium is a polynomial of degree 4 in the integer hop c = (cx, cy),
//   f^eq_l = w_l rho P(c_l),   P(c) = sum_{i+j<=4} p_ij cx^i cy^j,
// whose 15 coefficients are site values.  With U = s u_x, V = s u_bar_y,
// A = U^2, B = V^2, theta = T_bar - 1 and q = (A + B) / s^2:
//   L0 = 1 - q/2 - 2 theta,  M0 = (L0 - theta) / 2,  G = s^2 theta / 2,
//   p00 = 1 - q/2 + q^2/8 - theta + theta q + theta^2,
//   p20 = K1 + A M0,  p02 = K1 + B M0,  p11 = 2 U V M0,
//   p40 = K2 + A (G/2 + A/24),  p04 = K2 + B (G/2 + B/24),
//   p22 = 2 K2 + A (G/2 + B/4) + B G/2,
//   p10 = U L0,  p30 = U (G + A/6),  p12 = U (G + B/2),
//   p01 = V L0,  p03 = V (G + B/6),  p21 = V (G + A/2),
//   p31 = V p30,  p13 = U p03,
//   K1 = s^2 (theta/2 - theta q/4 - theta^2),  K2 = s^4 theta^2 / 8,
// all times rho below.  The hops of one class (|cx|, |cy|) differ by signs
// only: with the parts of P even in both components (ee), odd in cx (oe), odd
// in cy (eo) and odd in both (oo), their four values are (ee +- oo) +- (oe +-
// eo), and every part is one or two products with the class's weight, the
// powers of a hop of 2 or 3 folded into it.  So the 37 equilibria take 42
// products with constants after about 40 site products; a chain per pair of
// opposite hops (Horner in a = xi.u, after eight products per shell) took
// about 165 products and a longer dependency chain: 2048 x 8192 step 2.71 ms
// against 2.16 ms with this form.
//
// rho enters as rho^ in [0.5, 1) (the moment sum shifted to its leading one,
// a power of two taken out that joins the result's exponent).  The ranges
// |theta| < 1 and |u_bar| < 0.35 per component keep every value inside its
// format; other sites take the FP64 evaluation.  Products round to nearest
// (within 0.75 of the last place, no bias: both low words are signed and the
// half is added), so neither the momentum nor the energy drifts.
// tests/test_hop_moment_formats.py restates these integers and holds them
// to 2^-52 of omega w rho against rational arithmetic (the FP64 evaluation
// loses about 1e-14 for the outer shells near T = 0.5).
using u64 = unsigned long long;

// hi 2^32 + lo with a signed low word, the operand form of fx_mul
struct FxOp {
  int lo, hi;
};

// |v| < 2^63 - 2^31
__device__ __forceinline__ FxOp fx_op(long long v) {
  const int lo = (int)v;
  return {lo, (int)((u64)v >> 32) + (int)((unsigned)lo >> 31)};
}

__device__ __forceinline__ FxOp fx_op(const FxConst& c) { return {c.lo, c.hi}; }

// x y 2^-64 to within 1.25 of the last place, unbiased: the high word of each
// cross product is a floor (0.5 low on average, together one) and `one` = 1
// takes that back; the product of the low words (below 2^62, signed) is left
// out.  One comes from the launch's parameters: as a value the compiler does
// not know it enters the multiply-add as its addend, while a literal 1 cost an
// addition of its own.  Five instructions, three of them 32-bit multiplies;
// with 64-bit cross sums rounded by 2^31 (error 0.75) seven to fourteen.
__device__ __forceinline__ long long fx_mul(FxOp x, FxOp y, int one) {
  const int t = __mulhi(x.lo, y.hi) + (__mulhi(x.hi, y.lo) + one);
  return (long long)x.hi * y.hi + t;
}

// (x y + z w) 2^-64, two = 2
__device__ __forceinline__ long long fx_mul2(FxOp x, FxOp y, FxOp z, FxOp w, int two) {
  const int t = __mulhi(z.lo, w.hi) + (__mulhi(z.hi, w.lo) + (__mulhi(x.lo, y.hi) + (__mulhi(x.hi, y.lo) + two)));
  return (long long)x.hi * y.hi + ((long long)z.hi * w.hi + t);
}

// v 2^n without undefined behaviour for negative v
__device__ __forceinline__ long long fx_shl(long long v, int n) { return (long long)((u64)v << n); }

// g 2^E as an FP64 number by integer operations (round half away from zero),
// es = E 2^20.  The FP64 pipe converts too (I2F, one of its slots, as long as
// an FMA's), but it is the busiest unit and the integer pipes have room: 2048
// x 8192 step 2.16 ms with every population converted here, 2.27-2.34 ms with
// half of them, 2.51 ms with none.
// |g| < 2^32 (including 0): the general normalisation
__device__ __noinline__ double fx_to_double_small(unsigned m, int es, int sign) {
  if (!m) return 0.0;
  const int lz = __clz((int)m);
  const u64 mant = (u64)(m << lz) << 21;  // leading one at bit 52
  const int hi = (int)(mant >> 32) + es + ((1023 + 31 - lz - 1) << 20);
  return __hiloint2double(hi | sign, (int)mant);
}

// The magnitude is the one's complement for negative g: one less than |g|.
__device__ __forceinline__ double fx_to_double(long long g, int es) {
  const int gh = (int)(g >> 32), sm = gh >> 31;
  const unsigned mh = (unsigned)(gh ^ sm), ml = (unsigned)g ^ (unsigned)sm;
  const int sign = sm & (int)0x80000000;
  if (mh == 0u) return fx_to_double_small(ml, es, sign);
  // the leading one moved to bit 62 (|g| < 2^63), rounded to 53 bits, 54 when
  // the rounding carries; it adds 1 to the exponent field, a carry one more
  const int lz = __clz((int)mh) - 1;
  const u64 n = ((u64)__funnelshift_l(ml, mh, lz) << 32 | (ml << lz)) + 0x200;
  const u64 mant = n >> 10;
  const int hi = (int)(mant >> 32) + es + ((1023 + 61 - lz) << 20);
  return __hiloint2double(hi | sign, (int)mant);
}

// The site values the equilibrium starts from (formats beside each).
struct FxSite {
  long long R61;         // rho^
  long long mx, my;      // Q64: rho^ U, rho^ V
  long long U, V;        // Q64
  long long rA, rB, AB;  // Q64: rho^ A, rho^ B, A + B
  long long rq63;        // rho^ q
  long long rth60;       // rho^ theta
  long long X61;         // 1 / rho^
  FxOp A, B;             // Q64
  long long A64, B64;
  int es;                // 2^20 log2(rho / rho^)
};

// 2^125 / rn for rn in [2^63, 2^64), within 3: the float reciprocal r0 of the
// top 24 bits (24 bits, as an integer), e = 1 - rn r0 exactly, r0 (1 + e + e^2).
__device__ __forceinline__ long long fx_recip61(u64 rn) {
  const unsigned hi = (unsigned)(rn >> 32), lo = (unsigned)rn;
  const unsigned rb = __float_as_uint(__frcp_rn(__int_as_float(0x4B000000 | (int)((hi >> 8) & 0x7FFFFF))));
  // 2^47 / top: top = 2^23 gives 2^24, else below it
  const unsigned s = ((rb & 0x7FFFFF) | 0x800000) << ((rb >> 23) - 103);
  long long e = -(long long)((((u64)hi * s) << 24) + (((u64)lo * s) >> 8));  // Q79, mod 2^64; |e| < 2^57
  const int eh = (int)(e >> 32);
  e += ((long long)eh * eh) >> 15;
  return (long long)((u64)s << 38) + (((e >> 18) * (long long)s) >> 23);
}

// The fixed-point site values from the exact moment sums (no FP64
// arithmetic): rho^ = r 2^n 2^-64, rho^ U = s^2 jx / r rho^, 2 rho^ theta =
// s^2 e - rho^ (|u|^2 + ...) with the shifts of Eq. MASTERSHIFT3 (unshifted u
// in T, reading R6).  False when the site is outside the fixed-point ranges
// (|u_x|, |u_bar_y| < 0.35, |theta| < 1) or its sums do not fit the scaled
// forms; those sites take the FP64 collision.
__device__ __forceinline__ bool fx_site_from_sums(long long r, long long jx, long long jy, long long e, int emax,
                                                  const StepParams& p, FxSite& o) {
  if (!p.fx_on || r <= 0) return false;
  const u64 ur = (u64)r;
  const long long h = (r >> 1) - (r >> 4);
  const u64 h2 = 2 * (u64)h;
  // |j| <= 7/16 r and 0 <= e < 3 r keep the scaled sums inside an fx_op (r <
  // 37 2^53); the exponents leave room for those of the weights
  if ((u64)(jx + h) >= h2 || (u64)(jy + h) >= h2 || (u64)e >= ur + ur + ur || emax < 256 || emax > 1792)
    return false;
  const int one = p.fx_one;
  const int n = __clzll(r);  // >= 5
  const u64 rn = ur << n;    // Q64
  const long long R60 = (long long)(rn >> 4);
  const FxOp R62 = fx_op((long long)(rn >> 2));
  const FxOp jnx = fx_op(fx_shl(jx, n)), jny = fx_op(fx_shl(jy, n));  // Q64
  const FxOp s2 = fx_op(p.fx_s2_62);
  const long long mx62 = fx_mul(jnx, s2, one);
  const long long my62 = fx_mul(jny, s2, one) + fx_mul(R62, fx_op(p.fx_sd_64), one);
  const long long lim = fx_shl(fx_mul(R62, fx_op(p.fx_lim_63), one), 1);  // Q62: 0.35 s rho^
  if (mx62 >= lim || mx62 <= -lim || my62 >= lim || my62 <= -lim) return false;
  o.X61 = fx_recip61(rn);
  const FxOp X = fx_op(o.X61);
  o.mx = fx_shl(mx62, 2);
  o.my = fx_shl(my62, 2);
  const FxOp mx = fx_op(o.mx), my = fx_op(o.my);
  o.U = fx_shl(fx_mul(mx, X, one), 3);
  o.V = fx_shl(fx_mul(my, X, one), 3);
  const FxOp U = fx_op(o.U), V = fx_op(o.V);
  o.A64 = fx_mul(U, U, one);
  o.B64 = fx_mul(V, V, one);
  o.AB = o.A64 + o.B64;
  o.rA = fx_mul(mx, U, one);
  o.rB = fx_mul(my, V, one);
  o.rq63 = fx_mul(fx_op(o.rA + o.rB), fx_op(p.fx_is2_63), one);
  // rho theta = s^2 e / 2 - rho q / 2 + tau g_y rho u_y - rho (u_y unshifted)
  o.rth60 = fx_mul(fx_op(fx_shl(e, n - 3)), s2, one) - (o.rq63 >> 4) + fx_mul(jny, fx_op(p.fx_sd_60), one) - R60;
  const long long tl = R60 - (1LL << 29);  // a margin that keeps 8 rho^ theta an fx_op
  if (o.rth60 >= tl || o.rth60 <= -tl) return false;
  o.R61 = (long long)(rn >> 3);
  o.es = (emax - 1011 - n) << 20;  // rho = r 2^(emax - 1075) = rho^ 2^(64 - n + emax - 1075)
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

// The relaxation of population l towards the equilibrium g 2^(es / 2^20).
template <class O>
__device__ __forceinline__ void fx_relax(const double (&f)[kQ], double keep, int es, int l, long long g, const O& out) {
  out.put(l, fma(keep, f[l], fx_to_double(g, es)));
}

// The populations of one class of hops (shell K) from its parts; PX: the pair
// of (cx, cy) (or of (cx, 0)), PY: the pair of (cx, -cy) (or of (0, cy)).
// (cx, 0), (-cx, 0), (0, cy), (0, -cy)
template <int K, int PX, int PY, class O>
__device__ __forceinline__ void fx_axis(const double (&f)[kQ], const StepParams& p, int es0, long long ex, long long ox,
                                        long long ey, long long oy, const O& out) {
  const int es = es0 + p.fx_es[K];
  const double keep = p.one_minus_omega;
  fx_relax(f, keep, es, 1 + 2 * PX, ex + ox, out);
  fx_relax(f, keep, es, 2 + 2 * PX, ex - ox, out);
  fx_relax(f, keep, es, 1 + 2 * PY, ey + oy, out);
  fx_relax(f, keep, es, 2 + 2 * PY, ey - oy, out);
}

// (cx, cy), (-cx, -cy), (cx, -cy), (-cx, cy)
template <int K, int PX, int PY, class O>
__device__ __forceinline__ void fx_diag(const double (&f)[kQ], const StepParams& p, int es0, long long ee, long long oe,
                                        long long eo, long long oo, const O& out) {
  const int es = es0 + p.fx_es[K];
  const double keep = p.one_minus_omega;
  const long long s = ee + oo, d = ee - oo, t = oe + eo, u = oe - eo;
  fx_relax(f, keep, es, 1 + 2 * PX, s + t, out);
  fx_relax(f, keep, es, 2 + 2 * PX, s - t, out);
  fx_relax(f, keep, es, 1 + 2 * PY, d + u, out);
  fx_relax(f, keep, es, 2 + 2 * PY, d - u, out);
}

// The collision of collide_site_fp64 below with the equilibrium in fixed
// point, for a site inside the fixed-point ranges.  Every p is Q61; a part's
// product with fx_w (c_k h^m 2^(fx_q(k) + 3), h the class's larger hop) is at
// Q fx_q(k).
template <class O>
__device__ __forceinline__ void collide_site_fx(const double (&f)[kQ], const StepParams& p, const FxSite& v,
                                                const O& out) {
  const int one = p.fx_one, two = p.fx_two;
  const FxOp mx = fx_op(v.mx), my = fx_op(v.my), U = fx_op(v.U), V = fx_op(v.V);
  const FxOp rA = fx_op(v.rA), rB = fx_op(v.rB), s2 = fx_op(p.fx_s2_62);
  const long long rC = fx_mul(mx, V, one);
  const long long q61 = fx_mul(fx_op(v.AB), fx_op(p.fx_is2_61), one);
  const FxOp rth63 = fx_op(fx_shl(v.rth60, 3)), rq = fx_op(v.rq63);
  const long long th62 = fx_shl(fx_mul(rth63, fx_op(v.X61), one), 2);
  const FxOp th = fx_op(th62);
  const long long Pq = fx_mul(rq, th, one), Pt = fx_mul(rth63, th, one);  // Q61: rho theta q, rho theta^2
  const long long qq = fx_mul(rq, fx_op(q61), one);                 // Q60: rho q^2
  const long long p00 = v.R61 - (v.rq63 >> 3) - fx_shl(v.rth60, 1) + (qq >> 2) + Pq + Pt;
  const long long G = fx_mul(th, fx_op(p.fx_hs2_63), one), G2 = G >> 1;
  const long long K1 = fx_shl(fx_mul(fx_op(fx_shl(v.rth60, 1) - (Pq >> 1) - fx_shl(Pt, 1)), s2, one), 1);
  const long long K2 = fx_mul(fx_op(Pt), fx_op(p.fx_s4_64), one);
  const long long L0 = (1LL << 61) - (q61 >> 1) - th62;
  const FxOp M0 = fx_op((L0 - (th62 >> 1)) >> 1);
  const long long A6 = fx_mul(fx_op(v.A64), fx_op(p.fx_sixth_61), one), B6 = fx_mul(fx_op(v.B64), fx_op(p.fx_sixth_61), one);
  const long long p20 = K1 + fx_mul(rA, M0, one), p02 = K1 + fx_mul(rB, M0, one);
  const long long p11 = fx_shl(fx_mul(fx_op(rC), M0, one), 1);
  const long long p40 = K2 + fx_mul(rA, fx_op(G2 + (A6 >> 2)), one), p04 = K2 + fx_mul(rB, fx_op(G2 + (B6 >> 2)), one);
  const long long p22 = fx_shl(K2, 1) + fx_mul2(rA, fx_op(G2 + (v.B64 >> 5)), rB, fx_op(G2), two);
  const long long p30 = fx_mul(mx, fx_op(G + A6), one), p12 = fx_mul(mx, fx_op(G + (v.B64 >> 4)), one);
  const long long p03 = fx_mul(my, fx_op(G + B6), one), p21 = fx_mul(my, fx_op(G + (v.A64 >> 4)), one);
  const long long p31 = fx_mul(V, fx_op(p30), one), p13 = fx_mul(U, fx_op(p03), one);
  const long long p10 = fx_mul(mx, fx_op(L0), one), p01 = fx_mul(my, fx_op(L0), one);
  const int es = v.es;
#define W(k, m) fx_op(p.fx_w[k][m])
#define EE(k, t) fx_mul(fx_op(t), W(k, 0), one)
#define EE2(k, t, t2) fx_mul2(fx_op(t), W(k, 0), fx_op(t2), W(k, 2), two)
#define OD(k, m, t) fx_mul(fx_op(t), W(k, m), one)
  fx_relax(f, p.one_minus_omega, es + p.fx_es[0], 0, EE(0, p00), out);
  const long long ex1 = p00 + p20 + p40, ey1 = p00 + p02 + p04;  // p00 + X1, p00 + Y1
  {
    const long long a = p10 + p30, b = p01 + p03;
    fx_axis<1, 0, 1>(f, p, es, EE(1, ex1), OD(1, 0, a), EE(1, ey1), OD(1, 0, b), out);
    fx_diag<2, 2, 3>(f, p, es, EE(2, ex1 + p02 + p04 + p22), OD(2, 0, a + p12), OD(2, 0, b + p21),
                     OD(2, 0, p11 + p31 + p13), out);
  }
  const long long a1 = p10 + p30, a2 = p10 + 4 * p30, b1 = p01 + p03, b2 = p01 + 4 * p03;
  const long long x2 = p20 + 4 * p40, y2 = p02 + 4 * p04;
  fx_axis<3, 4, 5>(f, p, es, EE2(3, p00, x2), OD(3, 1, a2), EE2(3, p00, y2), OD(3, 1, b2), out);
  fx_diag<4, 6, 7>(f, p, es, EE2(4, ey1, x2 + p22), OD(4, 1, a2 + p12), OD(4, 0, b1 + 4 * p21),
                   OD(4, 1, p11 + 4 * p31 + p13), out);
  fx_diag<4, 8, 9>(f, p, es, EE2(4, ex1, y2 + p22), OD(4, 0, a1 + 4 * p12), OD(4, 1, b2 + p21),
                   OD(4, 1, p11 + p31 + 4 * p13), out);
  fx_diag<5, 10, 11>(f, p, es, EE2(5, p00, x2 + y2 + 4 * p22), OD(5, 1, a2 + 4 * p12), OD(5, 1, b2 + 4 * p21),
                     OD(5, 2, p11 + 4 * (p31 + p13)), out);
  const long long a3 = p10 + 9 * p30, b3 = p01 + 9 * p03, x3 = p20 + 9 * p40, y3 = p02 + 9 * p04;
  fx_axis<6, 12, 13>(f, p, es, EE2(6, p00, x3), OD(6, 1, a3), EE2(6, p00, y3), OD(6, 1, b3), out);
  fx_diag<7, 14, 15>(f, p, es, EE2(7, ey1, x3 + p22), OD(7, 1, a3 + p12), OD(7, 0, b1 + 9 * p21),
                     OD(7, 1, p11 + 9 * p31 + p13), out);
  fx_diag<7, 16, 17>(f, p, es, EE2(7, ex1, y3 + p22), OD(7, 0, a1 + 9 * p12), OD(7, 1, b3 + p21),
                     OD(7, 1, p11 + p31 + 9 * p13), out);
#undef W
#undef EE
#undef EE2
#undef OD
}

// BGK collision of one site, f <- f - (f - f^eq(rho, u_bar, T_bar)) / tau with
// u_bar = u + tau g, T_bar = T - tau^2 g^2 / D (Eq. MASTERSHIFT3, Eq. discrete).
// The equilibrium is evaluated per pair as even +- odd parts with per-shell
// coefficients (see ShellConsts), pre-scaled by omega rho w_shell.
template <class O>
__device__ __forceinline__ void collide_site_fp64(const double (&f)[kQ], const StepParams& p, double rho, double ux,
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
    out.put(0, fma(keep, f[0], wr * c_shell.w[0] * C0));
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
      out.put(1 + 2 * pr, fma(keep, f[1 + 2 * pr], even + odd));
      out.put(2 + 2 * pr, fma(keep, f[2 + 2 * pr], even - odd));
    }
  }
}

// One site's collision: moments as exact integer sums, then the fixed-point
// form inside its ranges, else the FP64 form; the relaxed populations to out.
template <class O>
__device__ __forceinline__ void collide_site_to(double (&f)[kQ], const StepParams& p, const O& out) {
  long long r, jx, jy, e;
  int emax;
  FxSite fs;
  const bool sums = site_sums(f, r, jx, jy, e, emax);
  if (sums && fx_site_from_sums(r, jx, jy, e, emax, p, fs)) {
    collide_site_fx(f, p, fs, out);
    return;
  }
  double rho, ux, uy, T;
  if (sums)
    moments_from_sums(r, jx, jy, e, emax, rho, ux, uy, T);
  else
    site_moments_fp64(f, rho, ux, uy, T);
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
template <class P>  // StepParams or BatchGeo (Ly, NY, Hy, plane)
__device__ __forceinline__ double wall_row_outgoing(const double* __restrict__ src, const P& p, int x, int wall,
                                                    int r) {
  const int y = wall ? p.Ly - 1 - r : r;
  const long long i = site_index(p, x, y);
  double s = 0.0;
#pragma unroll
  for (int l = 0; l < kQ; ++l) {
    const int cy = vel_cy(l);
    if (wall ? (cy > r) : (cy < -r)) s += src[l * p.plane + i];
  }
  return s;
}

__device__ __forceinline__ double wall_density(const double* __restrict__ src, const StepParams& p, int x,
                                               int wall) {
  const double s0 = wall_row_outgoing(src, p, x, wall, 0);
  const double s1 = wall_row_outgoing(src, p, x, wall, 1);
  const double s2 = wall_row_outgoing(src, p, x, wall, 2);
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

// The halo images of a site whose populations are already in its own
// element of dst (written by this thread): read back and copied out.  OFF:
// the planes addressed with the byte offsets of p (read from the constant
// bank by the single-lattice kernels) instead of multiples of p.plane.
template <bool OFF>
__device__ __forceinline__ void store_images(double* __restrict__ dst, const StepParams& p, int x, int y) {
  if (x >= kHx && x < p.Lx - kHx && (!p.periodic_y || (y >= kHx && y < p.Ly - kHx))) return;
  const double* s = dst + site_index(p, x, y);
  double f[kQ];
#pragma unroll
  for (int l = 0; l < kQ; ++l)
    f[l] = OFF ? *(const double*)((const char*)s + p.plane_off[l]) : s[l * p.plane];
  int xs[3] = {x, 0, 0}, ys[3] = {y, 0, 0};
  int nx = 1, ny = 1;
  if (x < kHx) xs[nx++] = x + p.Lx;
  if (x >= p.Lx - kHx) xs[nx++] = x - p.Lx;
  if (p.periodic_y) {
    if (y < kHx) ys[ny++] = y + p.Ly;
    if (y >= p.Ly - kHx) ys[ny++] = y - p.Ly;
  }
  for (int a = 0; a < nx; ++a)
    for (int b = 0; b < ny; ++b) {
      if (a == 0 && b == 0) continue;  // the site's own element
      double* d = dst + site_index(p, xs[a], ys[b]);
#pragma unroll
      for (int l = 0; l < kQ; ++l) {
        if (OFF)
          *(double*)((char*)d + p.plane_off[l]) = f[l];
        else
          d[l * p.plane] = f[l];
      }
    }
}

__global__ void __launch_bounds__(kBlockY, D2Q37_SITE_MIN_BLOCKS) collide_kernel(double* __restrict__ buf, StepParams p) {
  const int x = blockIdx.x;
  const int y = blockIdx.y * kBlockY + threadIdx.x;
  if (y >= p.Ly) return;
  double* const b = buf + site_index(p, x, y);
  double f[kQ];
#pragma unroll
  for (int l = 0; l < kQ; ++l) f[l] = *(const double*)((const char*)b + p.plane_off[l]);
  // in place: every population is read above before its pair is written back
  collide_site_to(f, p, ToPlanes{(char*)b, p});
  store_images<true>(buf, p, x, y);
}

// One site of the fused step: gather (pull), wall bc on the wall bands,
// collide, store with halo images.
// p: the lattice (geometry, walls); px: the constants of its collision (tau,
// g: the fixed-point tables, omega, the field shifts), the same object for a
// single lattice.  OFF: addresses from the byte offsets of p (see store_images).
// WALLS = false: the caller never passes a wall-band site.
template <bool OFF, bool WALLS = true>
__device__ __forceinline__ void fused_site(const double* __restrict__ src, double* __restrict__ dst,
                                           const StepParams& p, const StepParams& px, int x, int y) {
  const long long i = site_index(p, x, y);
  double f[kQ];
  if constexpr (OFF) {
    const char* s = (const char*)(src + i);
#pragma unroll
    for (int l = 0; l < kQ; ++l) f[l] = *(const double*)(s + p.pull_off[l]);
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
    collide_site_to(f, px, ToPlanes{(char*)(dst + i), p});
  else
    collide_site_to(f, px, ToPlanesStride{dst + i, p.plane});
  store_images<OFF>(dst, p, x, y);
}

__global__ void __launch_bounds__(kBlockY, D2Q37_SITE_MIN_BLOCKS) fused_kernel(const double* __restrict__ src, double* __restrict__ dst,
                                                        StepParams p) {
  const int x = blockIdx.x;
  const int y = blockIdx.y * kBlockY + threadIdx.x;
  // the wall-band kernel, launched next with programmatic stream
  // serialization, reads and writes nothing this kernel writes: it may start
  // once every block of this one has started, and fill the tail
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (y >= p.Ly) return;
  if (!p.periodic_y && (y < 3 || y >= p.Ly - 3)) return;  // wall_band_kernel's
  fused_site<true, false>(src, dst, p, p, x, y);
}

// The fused step of the six wall-band rows of every column (y = 0..2 and
// Ly - 3..Ly - 1, walls only), packed into full warps so that the wall bc's
// work runs at warp width instead of in three lanes of a fused_kernel warp (a
// warp holding wall rows cost about three ordinary warps there).  Each warp
// takes ten (column, wall) groups of three lanes, one lane per wall row (lanes
// 30 and 31 idle); every lane sums the populations of its own row that leave
// through the wall, and the group's three row sums meet by warp shuffles, so
// the column's outgoing mass is read once instead of once per wall site.
// When it is launched as a programmatic dependent of fused_kernel it may run
// while that kernel's last blocks still run; every thread then waits for the
// sites kernel to complete (griddepcontrol.wait: the prerequisite grid has
// finished and its writes are visible) before it exits.  So this grid never
// completes before the sites kernel, and whatever the stream runs after it
// (the next step's sites kernel reads both kernels' rows) is ordered after
// both, in a stream and in a captured graph alike.  Launched normally, the
// wait returns at once.
constexpr int kWallGroupsPerWarp = 10;

__global__ void __launch_bounds__(kWallBlock) wall_band_kernel(const double* __restrict__ src,
                                                              double* __restrict__ dst, StepParams p) {
  const int lane = threadIdx.x & 31;
  const int g = (blockIdx.x * (kWallBlock / 32) + (threadIdx.x >> 5)) * kWallGroupsPerWarp + lane / 3;
  const int r = lane - 3 * (lane / 3);  // row from the wall
  const bool active = lane < 3 * kWallGroupsPerWarp && g < 2 * p.Lx;
  const int x = g >> 1, wall = g & 1;
  const double s = active ? wall_row_outgoing(src, p, x, wall, r) : 0.0;
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
    for (int l = 0; l < kQ; ++l) f[l] = *(const double*)(sp + p.pull_off[l]);
    apply_wall(f, p.fw[wall], wall, r, ((s0 + s1) + s2) * p.inv_denom[wall]);
    collide_site_to(f, p, ToPlanes{(char*)(dst + i), p});
    store_images<true>(dst, p, x, y);
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
                       int parity, StepParams common) {
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
    // owning lattice: per-tile table when given, else binary search; its
    // parameters are read in place (read-only, cached)
    const BatchEntry& e = tab[tile_entry ? tile_entry[t] : batch_entry_of(tab, n, t)];
    const int local = (int)(t - e.tile0);  // tiles of one lattice < 2^31: 32-bit division
    const int x = local / e.ytiles;
    const int y = (local - x * e.ytiles) * BY + threadIdx.x;
    const int c = e.cur ^ parity;
    if (y < e.p.Ly)
      fused_site<false>((const double*)e.buf[c], (double*)e.buf[c ^ 1], e.p, UNIFORM ? common : e.p, x, y);
  }
}

// ---- many lattices in one launch, split into site tiles and wall tiles ----
//
// One block per tile, no grid-stride loop: the blocks of site tiles (one
// column x BY rows, the wall rows left out) run fused_kernel's per-site work,
// and the blocks of wall tiles run wall_band_kernel's (three lanes per
// column and wall, the outgoing mass combined by warp shuffles), so that no
// warp of the launch holds a few wall rows among ordinary ones.  Every
// lattice's offsets come from the launch's parameter space (BatchLaunch,
// through the constant cache) and its collision constants from `common`; the
// per-site arithmetic is the single-lattice kernels', so results are the same
// bit for bit.  Requires walls, the same tau and g for every lattice and
// offsets that fit 32 bits (checked on the host).
static_assert(sizeof(BatchLaunch) <= 32764, "BatchLaunch must fit the kernel parameter space");


struct GeoPlanes {
  char* d;  // the site's element of plane 0
  const BatchGeo& g;
  __device__ __forceinline__ void put(int l, double v) const { *(double*)(d + g.plane_off[l]) = v; }
};

// The same with the plane offsets from a shared-memory copy.
struct SharedPlanes {
  char* d;
  const int* off;  // shared memory: plane offsets of the block's lattice
  __device__ __forceinline__ void put(int l, double v) const { *(double*)(d + off[l]) = v; }
};

// The lattice owning block b of the site tiles (wall = false) or wall tiles.
__device__ __forceinline__ int split_owner(const BatchLaunch& L, int b, bool wall) {
  int lo = 0, hi = L.n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if ((wall ? L.g[mid].wtile0 : L.g[mid].tile0) <= b)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

// The x halo image(s) of a site of a walled lattice (copied from dst[i]).
__device__ __forceinline__ void split_images(double* __restrict__ dst, const BatchGeo& g, int x, long long i) {
  if (x >= kHx && x < g.Lx - kHx) return;
  const char* s = (const char*)(dst + i);
  double f[kQ];
#pragma unroll
  for (int l = 0; l < kQ; ++l) f[l] = *(const double*)(s + g.plane_off[l]);
  const long long shift = (long long)g.Lx * g.NY;
  if (x < kHx) {
    char* d = (char*)(dst + i + shift);
#pragma unroll
    for (int l = 0; l < kQ; ++l) *(double*)(d + g.plane_off[l]) = f[l];
  }
  if (x >= g.Lx - kHx) {
    char* d = (char*)(dst + i - shift);
#pragma unroll
    for (int l = 0; l < kQ; ++l) *(double*)(d + g.plane_off[l]) = f[l];
  }
}

template <int BY>
__global__ void __launch_bounds__(BY, (D2Q37_BATCH_MIN_BLOCKS * 128) / BY > 0 ? (D2Q37_BATCH_MIN_BLOCKS * 128) / BY : 1)
    batch_split_kernel(const __grid_constant__ BatchLaunch L, const BatchEntry* __restrict__ tab,
                       const int* __restrict__ tile_entry, int parity) {
  const int b = blockIdx.x;
  if (b < L.site_tiles) {
    const BatchGeo& g = L.g[tile_entry[b]];
    // the lattice's 74 offsets in shared memory: the blocks of an SM serve
    // different lattices, whose parameter slices crowd the constant cache
    // (read from there: 5796 MLUPS on the 64-lattice workload, against 5881)
    __shared__ int off[2 * kQ];
    for (int k = threadIdx.x; k < 2 * kQ; k += BY) off[k] = k < kQ ? g.pull_off[k] : g.plane_off[k - kQ];  // BY may be < 74
    __syncthreads();
    // x fastest, as in fused_kernel: the columns a tile pulls from run at the same time
    const int local = b - g.tile0;
    const int yt = local / g.Lx;
    const int x = local - yt * g.Lx;
    const int y = yt * BY + threadIdx.x;
    if (y < 3 || y >= g.Ly - 3) return;  // the wall tiles'
    const int c = g.cur ^ parity;
    const long long i = site_index(g, x, y);
    const char* s = (const char*)((const double*)g.buf[c] + i);
    double f[kQ];
    double* dst = (double*)g.buf[c ^ 1];
#pragma unroll
    for (int l = 0; l < kQ; ++l) f[l] = *(const double*)(s + off[l]);
    collide_site_to(f, L.common, SharedPlanes{(char*)(dst + i), off + kQ});
    split_images(dst, g, x, i);
    return;
  }
  // wall tile: kWallGroupsPerWarp (column, wall) groups per warp, one lane per wall row
  const int w = b - L.site_tiles;
  const BatchGeo& g = L.g[split_owner(L, w, true)];
  const int lane = threadIdx.x & 31;
  const int grp = ((w - g.wtile0) * (BY / 32) + (threadIdx.x >> 5)) * kWallGroupsPerWarp + lane / 3;
  const int r = lane - 3 * (lane / 3);
  const bool active = lane < 3 * kWallGroupsPerWarp && grp < 2 * g.Lx;
  const int x = grp >> 1, wall = grp & 1;
  const int c = g.cur ^ parity;
  const double* src = (const double*)g.buf[c];
  const double sum = active ? wall_row_outgoing(src, g, x, wall, r) : 0.0;
  const int base = lane - r;
  const double s0 = __shfl_sync(0xffffffffu, sum, base);
  const double s1 = __shfl_sync(0xffffffffu, sum, base + 1);
  const double s2 = __shfl_sync(0xffffffffu, sum, base + 2);
  if (!active) return;
  const int y = wall ? g.Ly - 1 - r : r;
  const long long i = site_index(g, x, y);
  const char* s = (const char*)(src + i);
  double f[kQ];
#pragma unroll
  for (int l = 0; l < kQ; ++l) f[l] = *(const double*)(s + g.pull_off[l]);
  apply_wall(f, tab[g.entry].p.fw[wall], wall, r, ((s0 + s1) + s2) * g.inv_denom[wall]);
  double* dst = (double*)g.buf[c ^ 1];
  collide_site_to(f, L.common, GeoPlanes{(char*)(dst + i), g});
  split_images(dst, g, x, i);
}

__global__ void __launch_bounds__(kBlockY) fields_kernel(const double* __restrict__ buf, double* __restrict__ rho,
                                                         double* __restrict__ u, double* __restrict__ T,
                                                         StepParams p) {
  const int x = blockIdx.x;
  const int y = blockIdx.y * kBlockY + threadIdx.x;
  if (y >= p.Ly) return;
  const long long i = site_index(p, x, y);
  double f[kQ];
#pragma unroll
  for (int l = 0; l < kQ; ++l) f[l] = buf[l * p.plane + i];
  double r, ux, uy, t;
  site_moments(f, r, ux, uy, t);
  const long long o = (long long)x * p.Ly + y;
  const long long n = (long long)p.Lx * p.Ly;
  rho[o] = r;
  u[o] = ux;
  u[n + o] = uy;
  T[o] = t;
}

__global__ void __launch_bounds__(kBlockY) init_equilibrium_kernel(double* __restrict__ buf,
                                                                   const double* __restrict__ T, StepParams p) {
  const int x = blockIdx.x;
  const int y = blockIdx.y * kBlockY + threadIdx.x;
  if (y >= p.Ly) return;
  const double t = T[(long long)x * p.Ly + y];
  double feq[kQ];
  equilibrium(c_shell, 1.0 / t, 0.0, 0.0, t, feq);
  const long long i = site_index(p, x, y);
#pragma unroll
  for (int l = 0; l < kQ; ++l) buf[l * p.plane + i] = feq[l];
}

// The same initial state stored as FP32 deviations d_l = f_l - w_l.
__global__ void __launch_bounds__(kBlockY) init_equilibrium32_kernel(float* __restrict__ buf,
                                                                     const double* __restrict__ T, StepParams p) {
  const int x = blockIdx.x;
  const int y = blockIdx.y * kBlockY + threadIdx.x;
  if (y >= p.Ly) return;
  const double t = T[(long long)x * p.Ly + y];
  double feq[kQ];
  equilibrium(c_shell, 1.0 / t, 0.0, 0.0, t, feq);
  const long long i = site_index(p, x, y);
#pragma unroll
  for (int l = 0; l < kQ; ++l) buf[l * p.plane + i] = (float)(feq[l] - c_shell.w[vel_shell(l)]);
}

dim3 site_grid(const StepParams& p) { return dim3(p.Lx, (p.Ly + kBlockY - 1) / kBlockY); }

// (column, wall) groups of the wall-band kernel: 2 Lx, ten per warp
int wall_grid(const StepParams& p) {
  constexpr int per_block = kWallGroupsPerWarp * (kWallBlock / 32);
  return (2 * p.Lx + per_block - 1) / per_block;
}

int done(int n) { return cudaGetLastError() == cudaSuccess ? n : -1; }

}  // namespace

cudaError_t upload_shell_consts(const ShellConsts& c) { return cudaMemcpyToSymbol(c_shell, &c, sizeof(c)); }

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

int launch_collide(double* buf, const StepParams& p, cudaStream_t stream) {
  collide_kernel<<<site_grid(p), kBlockY, 0, stream>>>(buf, p);
  return done(1);
}

int launch_fused(const double* src, double* dst, const StepParams& p, cudaStream_t stream, bool overlap) {
  fused_kernel<<<site_grid(p), kBlockY, 0, stream>>>(src, dst, p);
  if (p.periodic_y) return done(1);
  if (!overlap) {
    wall_band_kernel<<<wall_grid(p), kWallBlock, 0, stream>>>(src, dst, p);
    return done(2);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(wall_grid(p));
  cfg.blockDim = dim3(kWallBlock);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, wall_band_kernel, src, dst, p) != cudaSuccess) return -1;
  return done(2);
}

template <int BY>
int batch_launch(const BatchEntry* tab, const int* tile_entry, int n, long long tiles, int parity, int grid,
                 const StepParams* common, cudaStream_t stream) {
  if (common)
    batch_fused_kernel<BY, true><<<grid, BY, 0, stream>>>(tab, tile_entry, n, tiles, parity, *common);
  else
    batch_fused_kernel<BY, false><<<grid, BY, 0, stream>>>(tab, tile_entry, n, tiles, parity, StepParams{});
  return done(1);
}

template <int BY>
int batch_occupancy() {
  int b = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, batch_fused_kernel<BY, true>, BY, 0);
  return b;
}

int launch_batch_fused(const BatchEntry* tab, const int* tile_entry, int n, long long tiles, int parity,
                       int block_y, int grid, const StepParams* common, cudaStream_t stream) {
  switch (block_y) {
    case 64: return batch_launch<64>(tab, tile_entry, n, tiles, parity, grid, common, stream);
    case 128: return batch_launch<128>(tab, tile_entry, n, tiles, parity, grid, common, stream);
    case 256: return batch_launch<256>(tab, tile_entry, n, tiles, parity, grid, common, stream);
    default: return -1;
  }
}

int launch_batch_split(const BatchLaunch& L, const BatchEntry* tab, const int* tile_entry, int parity, int block_y,
                       cudaStream_t stream) {
  const int grid = L.site_tiles + L.wall_tiles;
  switch (block_y) {
    case 64: batch_split_kernel<64><<<grid, 64, 0, stream>>>(L, tab, tile_entry, parity); break;
    case 128: batch_split_kernel<128><<<grid, 128, 0, stream>>>(L, tab, tile_entry, parity); break;
    case 256: batch_split_kernel<256><<<grid, 256, 0, stream>>>(L, tab, tile_entry, parity); break;
    default: return -1;
  }
  return done(1);
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

int launch_fields(const double* buf, double* rho, double* u, double* T, const StepParams& p, cudaStream_t stream) {
  fields_kernel<<<site_grid(p), kBlockY, 0, stream>>>(buf, rho, u, T, p);
  return done(1);
}

int launch_init_equilibrium(double* buf, const double* T, const StepParams& p, cudaStream_t stream) {
  init_equilibrium_kernel<<<site_grid(p), kBlockY, 0, stream>>>(buf, T, p);
  return done(1);
}

int launch_init_equilibrium32(float* buf, const double* T, const StepParams& p, cudaStream_t stream) {
  init_equilibrium32_kernel<<<site_grid(p), kBlockY, 0, stream>>>(buf, T, p);
  return done(1);
}

}  // namespace d2q37
