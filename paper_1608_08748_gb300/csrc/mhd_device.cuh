// mhd_device.cuh -- device arithmetic of one time step of the MHD + H/H2 chemistry method of
// arXiv:1608.08748 (Kulikov, Chernykh & Protasov).  Templated on the bulk type T (double for the
// FP64 path, float for the FP32-bulk path); the CFL reduction and the chemistry are FP64 always.
//
// The formulas follow the paper section by section.  On GB300 the FP64 pipe is the bound of the FP64
// path, so the work that need not be FP64 arithmetic leaves it: the limiter's sign tests, minima,
// orderings and power-of-two scalings run on the integer pipes (inline PTX on the halves of the
// doubles), quotients and roots take one Newton-Raphson step from the hardware seeds, and the
// Riemann solver forms its speeds and eigenvector rows with few divisions and square roots.  The
// parabolas are held as the deviations of their edges from the cell's value; the FP64 build contracts
// a*b+c into one FMA.  The FP64 path agrees with a plain evaluation to a few ulp per operation (about
// 1e-15 relative L1 after 50 steps of the 128^3 turbulence box).
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

// one body per translation unit, whatever the kernel that calls it
#ifdef __CUDACC__
#define MHD_NOINLINE __noinline__
#else
#define MHD_NOINLINE
#endif

namespace mhd {

// ------------------------------------------------------------------------------------------------
// Geometry and parameters (passed by value to every kernel)
// Division of a non-negative 32-bit index by an invariant divisor d >= 1 with a multiply-high, two
// shifts and two additions instead of the integer division's dozen-odd instructions (the
// round-up method with an add indicator of Granlund & Montgomery, 1994): l = ceil(log2 d),
// m = floor(2^32 (2^l - d) / d) + 1 (below 2^32), and for every t < 2^32 the quotient is
// (hi + ((t - hi) >> min(l, 1))) >> max(l - 1, 0) with hi = floor(m t / 2^32).
struct FastDiv {
  unsigned d, m;
  int s1, s2;
};
inline FastDiv make_fastdiv(unsigned d) {
  int l = 0;
  while ((1ull << l) < d) ++l;
  const unsigned long long m = (((1ull << 32) * ((1ull << l) - d)) / d) + 1;
  return FastDiv{d, (unsigned)m, l < 1 ? l : 1, l > 1 ? l - 1 : 0};
}

struct Geom {
  int n[3];          // cells per axis
  int bc[3];         // 0 periodic, 1 outflow (zero-gradient)
  long long N;       // cells
  long long NF;      // (nx+1)(ny+1)(nz+1): size of face / edge scratch arrays
  FastDiv dn[2];     // division by n_x, n_y (cell indices)
  FastDiv dn1[2];    // division by n_x + 1, n_y + 1 (face and lattice indices)
};

// the divisors of a grid of nx x ny x nz cells
inline void set_divisors(Geom& g) {
  for (int d = 0; d < 2; ++d) {
    g.dn[d] = make_fastdiv((unsigned)g.n[d]);
    g.dn1[d] = make_fastdiv((unsigned)g.n[d] + 1u);
  }
}

struct Phys {
  double gamma;      // scalar adiabatic index (chemistry off)
  double dx, ih;     // cell width and 1/dx
  int chem;          // H/H2 network on
  int regul_mode;    // Sec. 2.9 reading: 0 max form, 1 unconditional, 2 literal branch order
  double lshield;    // shielding length, code units
  double bdop, xnorm, taud;
  double ibdop, ixnorm;  // 1 / bdop, 1 / xnorm
  double taud_ls, ls_ixnorm;  // taud L_s and L_s / xnorm, L_s the shielding length in cm (set_shielding)
  float taud_ls_f[2], ls_ixnorm_f[2], ibdop_f[2];  // taud_ls, ls_ixnorm, ibdop as float pairs (set_shielding)
  int heatcool;          // Sec. 2.8 heating/cooling stage on (needs chem)
  double grav_g;         // gravitational constant in code units (0: no self-gravity)
  int ions;              // reactions 5-8 with H+ and electrons on (needs chem)
};

// Device-resident scalars of a simulation: tau never crosses to the host inside a step.
struct Scalars {
  double cfl, t_end;       // set by the host with a kernel launch (graph-safe)
  double tau, tau_h;       // this step's tau and tau / dx
  double gth[3];           // g tau / dx of the three substages (Sec. 2.2)
  float tau_h32;           // tau / dx in float (a conversion takes the FP64 pipe as long as an FMA)
  float ts[2];             // tau in seconds as a float pair (the FP32 path's chemistry)
  double t;                // simulated time
  unsigned long long dmax; // bits of max CFL denominator of the current state (positive double)
  int dlow;                // bits of a lower bound of that maximum (non-negative float), see post_cell
  unsigned long long vel_branch;
  long long steps;
  int flags;               // bit 0: non-physical state, bit 1: tau <= 0
  int fixed_tau;           // 1: tau was given by the host (stage calls)
};

template <typename T>
struct State {
  T* rho;
  T* m[3];
  T* E;
  T* eint;
  T* rh2;  // may be unused when chemistry is off
  T* rhp;  // rho_H+ = n_H+ = n_e; used when the ions are on
  T* b[3];
};

// ------------------------------------------------------------------------------------------------
// indexing: cells [k][j][i]; face / edge scratch arrays on the (n+1)^3 lattice
__device__ __forceinline__ int wrap(int i, int n, int bc) {
  if ((unsigned)i < (unsigned)n) return i;  // interior: no integer division
  if (bc == 0) {
    int r = i % n;
    return r < 0 ? r + n : r;
  }
  return i < 0 ? 0 : n - 1;
}
// Cell, face and lattice indices are 32-bit: mhd_create rejects grids whose (n+1)^3 lattice does
// not fit (512^3 needs 1.35e8).
typedef int idx_t;

// Index-checked build (compiled with -DMHD_CHECK; build.build(check=True) makes libmhd_check.so):
// every computed cell index is tested against the cells [0, N) and every face or lattice index
// against [0, NF); a bad one sets a bit of this translation unit's flag word (1: cell, 2: lattice)
// and is replaced by 0, so that the access stays inside its array.  mhd_check_flags reads the
// words.  The plain build compiles the checks away.
#ifdef MHD_CHECK
static __device__ unsigned int g_check_flags;
__device__ __forceinline__ idx_t checked_index(idx_t i, long long n, unsigned bit) {
  if (i < 0 || (long long)i >= n) {
    atomicOr(&g_check_flags, bit);
    return 0;
  }
  return i;
}
#define MHD_CELL(g, i) ::mhd::checked_index((i), (g).N, 1u)
#define MHD_LATTICE(g, i) ::mhd::checked_index((i), (g).NF, 2u)
#else
#define MHD_CELL(g, i) (i)
#define MHD_LATTICE(g, i) (i)
#endif

__device__ __forceinline__ idx_t cidx(const Geom& g, int i, int j, int k) {
  return MHD_CELL(g, (k * g.n[1] + j) * g.n[0] + i);
}
__device__ __forceinline__ idx_t fidx(const Geom& g, int i, int j, int k) {
  return MHD_LATTICE(g, (k * (g.n[1] + 1) + j) * (g.n[0] + 1) + i);
}
// cell index of (c[0], c[1], c[2]) after the boundary map on each axis
__device__ __forceinline__ idx_t cmap(const Geom& g, int c0, int c1, int c2) {
  return cidx(g, wrap(c0, g.n[0], g.bc[0]), wrap(c1, g.n[1], g.bc[1]), wrap(c2, g.n[2], g.bc[2]));
}

// ------------------------------------------------------------------------------------------------
// Sec. 2.1: local parabola.  Delta q = q^R - q^L (the parabola's endpoints q(0) = q^L, q(1) = q^R).
template <typename T>
struct Para {
  T L, R, d, q6;
};

// 2^(j/32) for j = 0 .. 31, correctly rounded (the table of the exponential exp_tang below)
__device__ const double kExp2Frac32[32] = {
    0x1.0000000000000p+0, 0x1.059b0d3158574p+0, 0x1.0b5586cf9890fp+0, 0x1.11301d0125b51p+0,
    0x1.172b83c7d517bp+0, 0x1.1d4873168b9aap+0, 0x1.2387a6e756238p+0, 0x1.29e9df51fdee1p+0,
    0x1.306fe0a31b715p+0, 0x1.371a7373aa9cbp+0, 0x1.3dea64c123422p+0, 0x1.44e086061892dp+0,
    0x1.4bfdad5362a27p+0, 0x1.5342b569d4f82p+0, 0x1.5ab07dd485429p+0, 0x1.6247eb03a5585p+0,
    0x1.6a09e667f3bcdp+0, 0x1.71f75e8ec5f74p+0, 0x1.7a11473eb0187p+0, 0x1.82589994cce13p+0,
    0x1.8ace5422aa0dbp+0, 0x1.93737b0cdc5e5p+0, 0x1.9c49182a3f090p+0, 0x1.a5503b23e255dp+0,
    0x1.ae89f995ad3adp+0, 0x1.b7f76f2fb5e47p+0, 0x1.c199bdd85529cp+0, 0x1.cb720dcef9069p+0,
    0x1.d5818dcfba487p+0, 0x1.dfc97337b9b5fp+0, 0x1.ea4afa2a490dap+0, 0x1.f50765b6e4540p+0};

// ---- begin inline-PTX helpers ----
// Sign tests, absolute values, minima and comparisons of doubles on the integer pipes.  On sm_103
// the FP64 pipe issues two instructions per clock per SM and the integer pipes 64, and the PPM
// limiter is mostly such tests.  They work on the two 32-bit halves in inline PTX, so that the
// compiler does not turn them back into floating-point negations, absolute values or compares.
// For non-NaN operands they give the IEEE answer, with two exceptions that cannot change a
// limited value: -0 and +0 are told apart, and a product of two differences that underflows to
// zero is not formed (the test "a b > 0" is taken on the signs).  The float overloads are the plain
// operations.
__device__ __forceinline__ double abs_b(double x) {
  double r;
  asm("{\n\t.reg .b32 lo, hi;\n\tmov.b64 {lo, hi}, %1;\n\tand.b32 hi, hi, 0x7fffffff;\n\t"
      "mov.b64 %0, {lo, hi};\n\t}" : "=d"(r) : "d"(x));
  return r;
}
__device__ __forceinline__ float abs_b(float x) { return fabsf(x); }
__device__ __forceinline__ double neg_b(double x) {
  double r;
  asm("{\n\t.reg .b32 lo, hi;\n\tmov.b64 {lo, hi}, %1;\n\txor.b32 hi, hi, 0x80000000;\n\t"
      "mov.b64 %0, {lo, hi};\n\t}" : "=d"(r) : "d"(x));
  return r;
}
__device__ __forceinline__ float neg_b(float x) { return -x; }
// m (>= 0) with the sign of s
__device__ __forceinline__ double with_sign_b(double m, double s) {
  double r;
  asm("{\n\t.reg .b32 lo, hi, hs, ls;\n\tmov.b64 {lo, hi}, %1;\n\tmov.b64 {ls, hs}, %2;\n\t"
      "and.b32 hs, hs, 0x80000000;\n\tor.b32 hi, hi, hs;\n\tmov.b64 %0, {lo, hi};\n\t}"
      : "=d"(r) : "d"(m), "d"(s));
  return r;
}
__device__ __forceinline__ float with_sign_b(float m, float s) { return copysignf(m, s); }
// the smaller of a, b >= 0
__device__ __forceinline__ double min_nn(double a, double b) {
  double r;
  asm("{\n\t.reg .s64 ia, ib;\n\t.reg .pred p;\n\tmov.b64 ia, %1;\n\tmov.b64 ib, %2;\n\t"
      "setp.lt.s64 p, ia, ib;\n\tselp.b64 %0, %1, %2, p;\n\t}" : "=d"(r) : "d"(a), "d"(b));
  return r;
}
__device__ __forceinline__ float min_nn(float a, float b) { return fminf(a, b); }  // one FMNMX
// the larger of a, b >= 0
__device__ __forceinline__ double max_nn(double a, double b) {
  double r;
  asm("{\n\t.reg .s64 ia, ib;\n\t.reg .pred p;\n\tmov.b64 ia, %1;\n\tmov.b64 ib, %2;\n\t"
      "setp.gt.s64 p, ia, ib;\n\tselp.b64 %0, %1, %2, p;\n\t}" : "=d"(r) : "d"(a), "d"(b));
  return r;
}
__device__ __forceinline__ float max_nn(float a, float b) { return a > b ? a : b; }
// a > b for b >= 0
__device__ __forceinline__ bool gt_nn(double a, double b) {
  unsigned r;
  asm("{\n\t.reg .s64 ia, ib;\n\t.reg .pred p;\n\tmov.b64 ia, %1;\n\tmov.b64 ib, %2;\n\t"
      "setp.gt.s64 p, ia, ib;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r) : "d"(a), "d"(b));
  return r != 0;
}
__device__ __forceinline__ bool gt_nn(float a, float b) { return a > b; }
// a b > 0: both nonzero, one sign
__device__ __forceinline__ bool same_sign(double a, double b) {
  unsigned r;
  asm("{\n\t.reg .b32 la, ha, lb, hb, t;\n\t.reg .pred p;\n\t"
      "mov.b64 {la, ha}, %1;\n\tmov.b64 {lb, hb}, %2;\n\t"
      "and.b32 t, ha, 0x7fffffff;\n\tor.b32 t, t, la;\n\tsetp.ne.u32 p, t, 0;\n\t"
      "and.b32 t, hb, 0x7fffffff;\n\tor.b32 t, t, lb;\n\tsetp.ne.and.u32 p, t, 0, p;\n\t"
      "xor.b32 t, ha, hb;\n\tsetp.ge.and.s32 p, t, 0, p;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r) : "d"(a), "d"(b));
  return r != 0;
}
__device__ __forceinline__ bool same_sign(float a, float b) { return a * b > 0.f; }
// the sign bit
__device__ __forceinline__ bool sign_bit_b(double x) {
  unsigned r;
  asm("{\n\t.reg .b32 lo, hi;\n\tmov.b64 {lo, hi}, %1;\n\tshr.u32 %0, hi, 31;\n\t}" : "=r"(r) : "d"(x));
  return r != 0;
}
__device__ __forceinline__ bool sign_bit_b(float x) { return signbit(x); }

// Ordered key of a double: the signed 64-bit order of the keys is the order of the values, with
// -0 below +0 (the magnitude bits of a negative value flipped).  Comparisons of keys run on the
// integer pipe.
__device__ __forceinline__ long long okey(double x) {
  long long k;
  asm("{\n\t.reg .s64 m;\n\tmov.b64 %0, %1;\n\tshr.s64 m, %0, 63;\n\t"
      "and.b64 m, m, 0x7fffffffffffffff;\n\txor.b64 %0, %0, m;\n\t}" : "=l"(k) : "d"(x));
  return k;
}

// x 2^-K (K = 1, 2) on the integer pipe: the exponent field lowered by K.  Equal to the FP64
// product wherever that is a normal double, a zero, an infinity or a NaN; a product below the
// normal range (|x| < 2^(K-1021)) is taken as the zero of the sign of x.
template <int K>
__device__ __forceinline__ double scale_down_b(double x) {
  double r;
  asm("{\n\t.reg .b32 lo, hi, e, s, t, l;\n\t.reg .pred p, q;\n\tmov.b64 {lo, hi}, %1;\n\t"
      "bfe.u32 e, hi, 20, 11;\n\tsetp.gt.u32 p, e, %2;\n\tsetp.eq.u32 q, e, 2047;\n\t"
      "and.b32 s, hi, 0x80000000;\n\tsub.u32 t, hi, %3;\n\tselp.b32 t, t, s, p;\n\t"
      "selp.b32 l, lo, 0, p;\n\tselp.b32 t, hi, t, q;\n\tselp.b32 l, lo, l, q;\n\t"
      "mov.b64 %0, {l, t};\n\t}"
      : "=d"(r) : "d"(x), "n"(K), "n"(K << 20));
  return r;
}
template <int K>
__device__ __forceinline__ float scale_down_b(float x) { return x * (1.0f / (float)(1 << K)); }

// Approximate reciprocal and reciprocal square root of a double (PTX rcp.approx.ftz.f64,
// rsqrt.approx.ftz.f64): seeds for the Newton-Raphson steps below.  Subnormal arguments count as 0.
__device__ __forceinline__ double rcp_seed(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  return r;
}
__device__ __forceinline__ double rsqrt_seed(double x) {
  double r;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  return r;
}

// high 32 bits of the 64-bit product (the fast index divisions)
__device__ __forceinline__ unsigned umulhi32(unsigned a, unsigned b) { return __umulhi(a, b); }

// Device intrinsics, grouped here with the other device-only helpers.  The pieces of exp_tang below
// that act on bit patterns: the range test of its argument (-707 <= x
// <= -0 or +0 <= x < 707; NaNs and infinities fail), the low word of a double, 2^m y for y in
// [0.5, 4) and |m| <= 1020 by an addition to the exponent field, and the table read.
__device__ __forceinline__ bool exp_fast_range(double x) {
  const unsigned long long ux = (unsigned long long)__double_as_longlong(x);
  return ux <= 0xc086180000000000ull && (ux >= 0x8000000000000000ull || ux < 0x4086180000000000ull);
}
__device__ __forceinline__ int lo_word(double x) { return __double2loint(x); }
__device__ __forceinline__ double scale_pow2(double y, int m) {
  return __hiloint2double(__double2hiint(y) + (int)((unsigned)m << 20), __double2loint(y));
}
__device__ __forceinline__ double exp2_frac32(int j) { return __ldg(&kExp2Frac32[j]); }

// FP32 operations rounded to nearest whatever the build's FP32 flags (the CFL screen's error bound
// assumes them), and +inf
__device__ __forceinline__ float fsqrt_rn(float x) { return __fsqrt_rn(x); }
__device__ __forceinline__ float frsqrt_rn(float x) { return __frsqrt_rn(x); }
__device__ __forceinline__ float fdiv_rn(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ float fmul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float f_inf() { return __int_as_float(0x7f800000); }

// ---- end inline-PTX helpers ----

// t / f.d for t < 2^32 (FastDiv)
__device__ __forceinline__ unsigned fdiv(unsigned t, const FastDiv& f) {
  const unsigned hi = umulhi32(f.m, t);
  return (hi + ((t - hi) >> f.s1)) >> f.s2;
}

__device__ __forceinline__ double rsqrt_t(double x) { return rsqrt(x); }
__device__ __forceinline__ float rsqrt_t(float x) { return rsqrtf(x); }

// A double in a vector register whose value the compiler does not know: FP64 instructions with an
// immediate, constant-bank or missing operand take 19 SM clocks on GB300, a DFMA of three vector
// registers 16 (measured with four independent chains per warp at 4 to 32 warps per SM; a product or a
// sum alone counts as an instruction with a missing operand).  z is 0 at run time.
__device__ __forceinline__ double in_register(double c) {
#ifdef __CUDA_ARCH__
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));  // bit 31 is clear in every lane
  return __hiloint2double(__double2hiint(c) | (int)(m >> 31), __double2loint(c));
#else
  return c;
#endif
}
__device__ __forceinline__ float in_register(float c) { return c; }

// Sums and products of the bulk type where no FMA takes both (the kernels write their FMAs out).  The FP32
// ones are the rounded operations that the compiler does not contract: a kernel has an instance for one
// box and one for many, and a box's results must not depend on which of them contracts what.
// In FP64 they are FMAs with 1 or -0 in a register, exact and by the figures above 16 % faster: 128^3
// FP64 step 19.4 -> 17.9 ms (Eulerian faces 12.8 -> 11.9, Lagrangian 5.6 -> 5.1 ms).
__device__ __forceinline__ float add_t(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  return a + b;
#endif
}
__device__ __forceinline__ float sub_t(float a, float b) { return add_t(a, -b); }
__device__ __forceinline__ float mul_t(float a, float b) { return fmul_rn(a, b); }
__device__ __forceinline__ double add_t(double a, double b) { return fma(a, in_register(1.0), b); }
__device__ __forceinline__ double sub_t(double a, double b) { return fma(-b, in_register(1.0), a); }
__device__ __forceinline__ double mul_t(double a, double b) { return fma(a, b, in_register(-0.0)); }

// FP64 reciprocal, quotient and square root in few FP64 instructions, by one third-order
// Newton-Raphson step (the series of the inverse function) from the seeds above; a correctly
// rounded FP64 division or square root takes about twice the FP64-pipe slots.
//   1/x: with e = 1 - x r0, 1/x = r0 / (1 - e) = r0 (1 + e + e^2 + e^3 + ...); keeping 1 + e + e^2
//        leaves a relative error of about e^3, below the double's rounding for the seed's error.
//   1/sqrt(x): with e = 1 - x y0^2, 1/sqrt(x) = y0 (1 - e)^(-1/2) = y0 (1 + e/2 + 3 e^2 / 8 + ...).
//   sqrt(x) = x (1/sqrt(x)).
// Each is within 2 ulp of the correctly rounded value for finite normal arguments (x != 0); sqrt_nr
// takes 0 and subnormal arguments through the library square root.
__device__ __forceinline__ double rcp_nr(double x) {
  const double r = rcp_seed(x);
  const double e = fma(-x, r, in_register(1.0));
  return fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ double rsqrt_nr(double x) {
  const double y = rsqrt_seed(x);
  const double e = fma(-x, mul_t(y, y), in_register(1.0));
  return fma(y, mul_t(e, fma(in_register(0.375), e, in_register(0.5))), y);
}
__device__ __forceinline__ double sqrt_nr(double x) {
  // the range test on the integer pipe (x >= 0 or NaN here; -0 and negative x take the library)
  if (__builtin_expect(!gt_nn(2.2250738585072014e-308, x), 1)) return x * rsqrt_nr(x);
  return sqrt(x);
}
// 1/sqrt of a positive normal value in the bulk type (FP64: the step above)
__device__ __forceinline__ double rsqrt_n(double x) { return rsqrt_nr(x); }
__device__ __forceinline__ float rsqrt_n(float x) { return rsqrtf(x); }
// bulk-type forms: FP64 by the steps above; FP32 by the plain operations (the FP32 build already
// takes the hardware-approximate division and square root)
__device__ __forceinline__ double rcp_t(double x) { return rcp_nr(x); }
__device__ __forceinline__ float rcp_t(float x) { return 1.0f / x; }
__device__ __forceinline__ double sqrt_t(double x) { return sqrt_nr(x); }
__device__ __forceinline__ float sqrt_t(float x) { return sqrtf(x); }

// e^x in FP64 by the table-driven method of P. T. P. Tang (ACM TOMS 15, 144-157, 1989), for the
// arguments of the H/H2 rates (x <= 0).  With k the integer nearest to 32 x / ln 2, k = 32 m + j
// (0 <= j < 32) and r = x - k ln2/32 (|r| <= ln2/64), e^x = 2^m 2^(j/32) e^r; e^r - 1 is its
// Taylor polynomial of degree 6 (the remainder r^7/7! stays below 4e-18), 2^(j/32) comes from a
// table of correctly rounded doubles, and 2^m is added to the exponent field on the integer pipe.
// ln2/32 is split in a 36-bit head, whose products with |k| < 2^15 are exact, and a tail.  The
// result lies within 1.01 ulp of e^x (half an ulp of the table entry, scaled by e^r, and half an ulp
// of the last rounding); it takes 11 FP64-pipe instructions.  Arguments outside
// [-707, 707] (where 2^m or the result leaves the normal range), infinities and NaNs take the
// library exp; the range test runs on the integer pipe.
__device__ __forceinline__ double exp_tang(double x) {
  if (!exp_fast_range(x)) return exp(x);
  const double INV_L = 0x1.71547652b82fep+5;                 // 32 / ln 2
  const double L_HI = 0x1.62e42fefa0000p-6, L_LO = 0x1.cf79abc9e3b3ap-45;  // ln2/32 = L_HI + L_LO
  const double SHIFTER = 0x1.8p52;                           // adding it rounds to an integer
  const double t = fma(x, INV_L, SHIFTER);
  const double kd = t - SHIFTER;
  const int k = lo_word(t);                                  // k in the low word, two's complement
  const double r = fma(-kd, L_LO, fma(-kd, L_HI, x));
  double p = fma(r, 1.0 / 720.0, 1.0 / 120.0);
  p = fma(r, p, 1.0 / 24.0);
  p = fma(r, p, 1.0 / 6.0);
  p = fma(r, p, 0.5);
  p = fma(r, p, 1.0);
  p = r * p;                                                 // e^r - 1
  const double tj = exp2_frac32(k & 31);
  const double y = fma(tj, p, tj);                           // 2^(j/32) e^r, in [0.98, 2.03)
  return scale_pow2(y, k >> 5);
}

// The bit pattern of a double as two 32-bit words and back, and the powers of two that the limiter
// takes on the integer pipe for magnitudes of normal doubles: 2 |x| (|x| + |x| for every finite
// |x| from the normal range on) and |x| / 4 (below 2^-1020 the exponent is held at zero: a value
// under the normal range, as good as the zero it stands for).
__device__ __forceinline__ int hi_of(double x) {
#ifdef __CUDA_ARCH__
  return __double2hiint(x);
#else
  long long k;
  __builtin_memcpy(&k, &x, 8);
  return (int)(k >> 32);
#endif
}
__device__ __forceinline__ double with_hi(double x, int hi) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(hi, __double2loint(x));
#else
  long long k;
  __builtin_memcpy(&k, &x, 8);
  k = (long long)(((unsigned long long)(unsigned)hi << 32) | ((unsigned long long)k & 0xffffffffull));
  __builtin_memcpy(&x, &k, 8);
  return x;
#endif
}
__device__ __forceinline__ double twice_b(double x) { return with_hi(x, hi_of(x) + (1 << 20)); }
__device__ __forceinline__ float twice_b(float x) { return x + x; }
__device__ __forceinline__ double quarter_nn(double x) {
  const int h = hi_of(x) - (2 << 20);
  return with_hi(x, h > 0 ? h : 0);
}
__device__ __forceinline__ float quarter_nn(float x) { return 0.25f * x; }
// x / 2 for x >= 0, likewise, and 4 x for a normal x
__device__ __forceinline__ double half_nn(double x) {
  const int h = hi_of(x) - (1 << 20);
  return with_hi(x, h > 0 ? h : 0);
}
__device__ __forceinline__ float half_nn(float x) { return 0.5f * x; }
__device__ __forceinline__ double four_b(double x) { return with_hi(x, hi_of(x) + (2 << 20)); }
__device__ __forceinline__ float four_b(float x) { return 4.0f * x; }

// A sufficient test of x > 2^-K s for x >= 0 and s > 0 on the high words (K exponents below s or more
// fails, and so does a value under 2^-1022); FP32 takes the comparison it guards.
template <int K>
__device__ __forceinline__ bool surely_above(double x, double s) {
  const int t = hi_of(s) - (K << 20);
  return hi_of(x) > (t > 0 ? t : 0);
}
template <int K>
__device__ __forceinline__ bool surely_above(float, float) { return false; }

// Half the limited slope of Sec. 2.1 Step 1 for a cell with differences dn = q_0 - q_-1,
// dp = q_1 - q_0 and s = q_1 - q_-1: the slope is min(|s|/2, 2|dp|, 2|dn|) with the sign of s where
// dn and dp have one sign, else 0; halving it is exact, and saves the doublings.  Selects, not
// branches (in FP64 on the integer pipe; in FP32 the minima are single instructions).
template <typename T>
__device__ __forceinline__ T half_slope(T s, T dn, T dp) {
  const T m = min_nn(min_nn(quarter_nn(abs_b(s)), abs_b(dp)), abs_b(dn));
  return same_sign(dn, dp) ? with_sign_b(m, s) : T(0);
}

// Sec. 2.1 in deviations.  A cell's parabola is held as its value q and A = 2 (q - q^L),
// B = 2 (q^R - q), twice the deviations of its edges.  With the halved slopes h and the difference
// d = q_{j+1} - q_j the edge between the cells j and j+1 (Step 1) gives B_j = d - (2/3)(h_{j+1} - h_j)
// and A_{j+1} = d + (2/3)(h_{j+1} - h_j): one subtraction and two FMAs for both.  In A and B the rest
// of the method is short:
//   Step 2: an extremum is A B <= 0 (then A = B = 0); Delta q q6 > (Delta q)^2 is |A| > 2 |B|, and its
//           fix q^L = 3 q - 2 q^R is A = 2 B; the mirrored case is |B| > 2 |A|, B = 2 A.  No sum or
//           product: comparisons and doublings.
//   Step 4: the flattened edges q -+ (slope)/4 are A = B = h, so the blend is A += hbar (h - A),
//           B += hbar (h - B).
//   Step 5: Delta q = (A + B)/2 and q6 = 3 (A - B)/2 are not formed: the averages of Sec. 2.4 over
//           the fraction y next to the right or the left edge are
//             q + y u A/2 + u^2 B/2   and   q - u^2 A/2 - y u B/2   with u = 1 - y.
// A streamed parabola takes 7 floating-point instructions besides Step 4's blend (with edge values, Delta q
// and q6 it took 17), and an average the same two FMAs; the FP64 faces form the same deviations in fixed
// point (fix_dev below).  The deviations also round less: no edge value is formed from which q is subtracted
// again.  With the Riemann solve below, one step of the turbulence box went from 25.6 to 19.4 ms at 128^3
// in FP64 (then still with FP64 parabolas) and from 15.9 to 14.5 ms at 256^3 in FP32 (Eulerian faces
// 5.2 -> 4.5, Lagrangian 4.1 -> 3.4 ms).
template <typename T>
struct Dev {
  T A, B;
};

// Steps 2 and 4 for a cell with unlimited deviations A, B, halved slope h0, second differences D+ and
// D-, s0 = q_{+1} - q_{-1} and the two neighbours' values.  Step 4's eta = -(D+ - D-)/(3 s0) acts where
// |s0| > min(|q_{+1}|, |q_{-1}|)/100 (the smaller of the paper's three values is one of the two) and
// D+ D- <= 0; hbar = 20 (eta - 1/20) = (20/3)(D- - D+)/s0 - 1, clamped to [0, 1].
// In FP64 (only the wide stencils of the fixed-point form below come here): hbar is continuous where it
// crosses 0 and 1, so the clamps' rounding cannot move the result.
__device__ __forceinline__ Dev<double> dev_limit(double A, double B, double h0, double Dp, double Dm, double s0,
                                                 double qp1, double qm1) {
  const bool mono = same_sign(A, B);
  const double mA = min_nn(abs_b(A), abs_b(twice_b(B))), mB = min_nn(abs_b(B), abs_b(twice_b(A)));
  A = mono ? with_sign_b(mA, A) : 0.0;
  B = mono ? with_sign_b(mB, B) : 0.0;
  if (!same_sign(Dp, Dm) && gt_nn(abs_b(s0), mul_t(0.01, min_nn(abs_b(qp1), abs_b(qm1))))) {
    const double hb = min_nn(fma(mul_t(20.0 / 3.0, sub_t(Dm, Dp)), rcp_nr(s0), -1.0), 1.0);
    if (!sign_bit_b(hb)) {
      A = fma(hb, sub_t(h0, A), A);
      B = fma(hb, sub_t(h0, B), B);
    }
  }
  return Dev<double>{A, B};
}
// FP32: bound by instruction issue, so selects instead of branches, and the reciprocal is taken
// everywhere and discarded where the detector is off (s0 may be 0 there); the clamp is the FMA's own
// saturation.
__device__ __forceinline__ unsigned bits_f(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  unsigned b;
  __builtin_memcpy(&b, &x, 4);
  return b;
#endif
}
__device__ __forceinline__ float float_of(unsigned b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float x;
  __builtin_memcpy(&x, &b, 4);
  return x;
#endif
}
__device__ __forceinline__ float saturate_f(float x) {
#ifdef __CUDA_ARCH__
  return __saturatef(x);
#else
  return x > 0.0f ? (x < 1.0f ? x : 1.0f) : 0.0f;
#endif
}
__device__ __forceinline__ Dev<float> dev_limit(float A, float B, float h0, float Dp, float Dm, float s0, float qp1,
                                                float qm1) {
  const bool mono = A * B > 0.0f;
  const float mA = min_nn(abs_b(A), 2.0f * abs_b(B)), mB = min_nn(abs_b(B), 2.0f * abs_b(A));
  A = mono ? with_sign_b(mA, A) : 0.0f;
  B = mono ? with_sign_b(mB, B) : 0.0f;
  const bool det = gt_nn(abs_b(s0), 0.01f * min_nn(abs_b(qp1), abs_b(qm1))) && !(Dp * Dm > 0.0f);
  const float hb = det ? saturate_f(fma((20.0f / 3.0f) * (Dm - Dp), rcp_t(s0), -1.0f)) : 0.0f;
  return Dev<float>{fma(hb, h0 - A, A), fma(hb, h0 - B, B)};
}

// the deviations of the cell in the middle of q_{-2} .. q_{+2}; in FP32 with the sign of q_0 - q_{-1} taken off
// and put back at the end: the halved slopes are then minima clamped at 0, without tests of signs.  The same bits as
// DevStream's.  The FP32 Lagrangian faces are bound by instruction issue (78 %): 256^3 step 3.34 -> 3.25 ms
__device__ __forceinline__ Dev<float> dev_of_f(float qm2, float qm1, float qc, float qp1, float qp2) {
  const float d1s = sub_t(qc, qm1);
  const unsigned sg = bits_f(d1s) & 0x80000000u;
  auto flip = [&](float x) { return float_of(bits_f(x) ^ sg); };
  const float d0 = flip(sub_t(qm1, qm2)), d1 = abs_b(d1s), d2 = flip(sub_t(qp1, qc)), d3 = flip(sub_t(qp2, qp1));
  const float s0 = flip(sub_t(qp1, qm1));
  auto slope = [](float a, float b, float s) { return fmaxf(fminf(fminf(a, b), 0.25f * abs_b(s)), 0.0f); };
  const float hm = slope(d0, d1, sub_t(qc, qm2)), h0 = slope(d1, d2, s0), hp = slope(d2, d3, sub_t(qp2, qc));
  float A = fma(2.0f / 3.0f, sub_t(h0, hm), d1), B = fma(-2.0f / 3.0f, sub_t(hp, h0), d2);
  const bool mono = A * B > 0.0f;
  const float mA = min_nn(A, 2.0f * B), mB = min_nn(B, 2.0f * A);
  A = mono ? mA : 0.0f;
  B = mono ? mB : 0.0f;
  const float Dp = sub_t(d3, d2), Dm = sub_t(d1, d0);
  const bool det = gt_nn(abs_b(s0), 0.01f * min_nn(abs_b(qp1), abs_b(qm1))) && !(Dp * Dm > 0.0f);
  const float hb = det ? saturate_f(fma((20.0f / 3.0f) * (Dm - Dp), rcp_t(s0), -1.0f)) : 0.0f;
  return Dev<float>{flip(fma(hb, h0 - A, A)), flip(fma(hb, h0 - B, B))};
}
template <typename T>
__device__ __forceinline__ Dev<T> dev_of(T qm2, T qm1, T qc, T qp1, T qp2) {
  if constexpr (sizeof(T) == 4) return dev_of_f(qm2, qm1, qc, qp1, qp2);
  const T d0 = sub_t(qm1, qm2), d1 = sub_t(qc, qm1), d2 = sub_t(qp1, qc), d3 = sub_t(qp2, qp1);
  const T sm = sub_t(qc, qm2), s0 = sub_t(qp1, qm1), sp = sub_t(qp2, qc);
  const T hm = half_slope(sm, d0, d1), h0 = half_slope(s0, d1, d2), hp = half_slope(sp, d2, d3);
  const T A = fma(in_register(T(2.0 / 3.0)), sub_t(h0, hm), d1), B = fma(-in_register(T(2.0 / 3.0)), sub_t(hp, h0), d2);
  return dev_limit(A, B, h0, sub_t(d3, d2), sub_t(d1, d0), s0, qp1, qm1);
}

// The deviations of consecutive cells j, j+1, ... along a line, each from the quantities dev_of forms
// for it (so bit for bit the same), where the difference q_{j+1} - q_j, the halved slope, the edge and
// the second difference centred on a cell are formed once and shared by the neighbours that use them.
// Prime with q_{J-2} .. q_{J+1}; each next(q_{j+2}) then returns cell j = J, J+1, ..., whose value is
// left in qm.  FP32 forms the differences dp and s0 again instead of carrying them (two instructions
// against two registers).
template <typename T>
struct DevStream {
  T qm, q0, qp;  // q_{j-1}, q_j, q_{j+1}
  T dp;          // q_{j+1} - q_j
  T h0;          // halved slope of cell j
  T A;           // unlimited A of cell j
  T Cm, C0;      // second differences centred on j-1 and j
  T s0;          // q_{j+1} - q_{j-1}

  __device__ __forceinline__ void prime(T qa, T qb, T qc, T qd) {  // q_{J-2} .. q_{J+1}
    const T d0 = sub_t(qb, qa), d1 = sub_t(qc, qb), d2 = sub_t(qd, qc);
    const T hm = half_slope(sub_t(qc, qa), d0, d1);
    s0 = sub_t(qd, qb);
    h0 = half_slope(s0, d1, d2);
    A = fma(in_register(T(2.0 / 3.0)), sub_t(h0, hm), d1);
    Cm = sub_t(d1, d0);
    C0 = sub_t(d2, d1);
    qm = qb;
    q0 = qc;
    qp = qd;
    dp = d2;
  }
  // The unlimited deviations A, B of cell j and what the limits take besides: limit(A, B, h0, Dp, Dm,
  // s0, q_{j+1}, q_{j-1}).  Moves on to cell j + 1.
  template <typename F>
  __device__ __forceinline__ void next(T qn, F limit) {  // qn = q_{j+2}
    if constexpr (sizeof(T) == 4) {
      dp = qp - q0;
      s0 = qp - qm;
    }
    const T d2 = sub_t(qn, qp), s1 = sub_t(qn, q0);
    const T h1 = half_slope(s1, dp, d2);
    const T C1 = sub_t(d2, dp), t = sub_t(h1, h0);
    limit(A, fma(-in_register(T(2.0 / 3.0)), t, dp), h0, C1, Cm, s0, qp, qm);
    A = fma(in_register(T(2.0 / 3.0)), t, dp);
    qm = q0;
    q0 = qp;
    qp = qn;
    dp = d2;
    h0 = h1;
    Cm = C0;
    C0 = C1;
    s0 = s1;
  }
  __device__ __forceinline__ Dev<T> next(T qn) {
    Dev<T> P;
    next(qn, [&](T a, T b, T h, T Dp, T Dm, T s, T qp1, T qm1) { P = dev_limit(a, b, h, Dp, Dm, s, qp1, qm1); });
    return P;
  }
};

// ------------------------------------------------------------------------------------------------
// The FP64 parabolas in fixed point.  Steps 1 and 2 of Sec. 2.1 are differences, minima, small integer
// multiples and comparisons, so within one stencil they need no floating point: the five values are
// aligned to the largest exponent among them as 64-bit integers with 59 bits for the magnitude (the
// largest value keeps all its 53 bits and 6 to spare; a smaller one is cut at 2^-59 of the largest), and the
// work runs on the integer pipes, which issue 32 instructions in the time the FP64 pipe takes one.
// A stencil's result depends on nothing else, so a pencil's length does not show.  Results are held as 3 A
// and 3 B (no division by 3; the averages' coefficients carry the third), rounded once from the integers: against
// 113-bit arithmetic the error of A is 0.4 to 1.3 times that of the FP64 form (r.m.s. over smooth, steep and rough
// stencils) and that of a whole step the same (8.6e-17 of the density at 96^3).  A streamed parabola
// took 7 FP64 instructions besides Step 4; here it takes none.  128^3 FP64 step at the developed flow, with the
// pencils in blocks of 64 threads: 16.5 -> 14.2 ms (Eulerian faces 10.3 -> 9.3, Lagrangian 4.1 -> 2.8 ms).
// Its callers keep their loops rolled: unrolled over cells the Lagrangian faces take 3.1 / 3.3 / 3.6 ms for 1, 2
// and 3 cells (128-thread blocks).
struct FixCell {
  long long n;  // value 2^(1081 - e), |n| < 2^59
  int e;        // biased exponent, at least 1
};
__device__ __forceinline__ long long bits_of(double q) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(q);
#else
  long long b;
  __builtin_memcpy(&b, &q, 8);
  return b;
#endif
}
__device__ __forceinline__ double dbl_of(long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double q;
  __builtin_memcpy(&q, &b, 8);
  return q;
#endif
}
__device__ __forceinline__ int min_i(int a, int b) { return a < b ? a : b; }
__device__ __forceinline__ int max_i(int a, int b) { return a > b ? a : b; }
__device__ __forceinline__ FixCell fix_cell(double q) {
  const long long b = bits_of(q);
  const int f = (int)((unsigned long long)b >> 52) & 0x7ff;
  FixCell c;
  c.e = f > 0 ? f : 1;
  const long long m = ((b & 0xfffffffffffffll) | (f > 0 ? 1ll << 52 : 0)) << 6;
  c.n = b < 0 ? -m : m;
  return c;
}
__device__ __forceinline__ int leading_zeros(unsigned long long x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}
// sgn m 2^(E - 1081) as a double, m < 2^63, rounded to nearest (0 below 2^-1022); neg is 0 or -1
__device__ __forceinline__ double fix_to_double(unsigned long long m, long long neg, int E) {
  const int z = leading_zeros(m), e = E + 4 - z;  // the biased exponent less one
  const unsigned long long f = ((m << (z - 1)) + 0x200) >> 10;
  const unsigned long long b = f + ((unsigned long long)(unsigned)e << 52) + (neg & (1ull << 63));
  return m != 0 && e >= 0 ? dbl_of((long long)b) : 0.0;
}
__device__ __forceinline__ unsigned long long uabs64(long long a) { return (unsigned long long)(a < 0 ? -a : a); }
__device__ __forceinline__ double fix_value(FixCell c) { return fix_to_double(uabs64(c.n), c.n >> 63, c.e); }
// min(a, b, (a + b)/4): the halved slope of a cell whose two differences a and b are not negative, negative where
// one of them is
__device__ __forceinline__ long long fix_half_slope(long long a, long long b) {
  const long long m = a < b ? a : b, t = (a + b) >> 2;
  return m < t ? m : t;
}
__device__ __forceinline__ long long not_negative(long long a) { return a & ~(a >> 63); }
__device__ __forceinline__ int hi_word(long long a) { return (int)(a >> 32); }
// What Step 4 takes of a cell: |num| = |D- - D+|, |s0|, three times the halved slope's magnitude and min(|q_{+1}|,
// |q_{-1}|), all times 2^(1081 - E); the sign of the parabola is that of its deviations
struct FixStep4 {
  long long num, s0, h3, ql, qr;  // (ql, qr) = q_{-1}, q_{+1}
  int E;
};
// Steps 1 and 2 of the cell in the middle of q_{-2} .. q_{+2}: 3 A and 3 B (left: q_0 - q_{-1}, for the
// Riemann solve).  All is done with the sign of
// q_0 - q_{-1} taken off: where q_{+1} - q_0 is then negative the cell is an extremum, and else the
// cell's own slope and A and B are not negative, and a neighbour's slope counts only where it is not.  Returns
// whether Step 4 may act (never false where it does): D- >= 0 >= D+, and by the high words |num| > 3 |s0| / 20
// and |s0| > mn / 128.  A wide stencil, where the largest exponent is more than 5 above that of the cell and of one
// of its neighbours (the results are at most a few times the smaller of the two differences, so the cut
// would show), or with an infinity, a NaN or a value of 2^1019 or more (3 A could overflow), is done as a whole in
// FP64.
__device__ __forceinline__ bool fix_dev(const FixCell c[5], Dev<double>& P, double& left, FixStep4& st) {
  const int near = max_i(c[2].e, min_i(c[1].e, c[3].e));
  const int E = max_i(max_i(max_i(c[0].e, c[1].e), max_i(c[3].e, c[4].e)), c[2].e);
  const bool wide = E > near + 5 || E >= 0x7fa;
  long long q[5], d[4];
#pragma unroll
  for (int k = 0; k < 5; ++k) q[k] = c[k].n >> min_i(E - c[k].e, 63);
  const long long neg = (q[2] - q[1]) >> 63;
#pragma unroll
  for (int k = 0; k < 4; ++k) d[k] = ((q[k + 1] - q[k]) ^ neg) - neg;
  const long long h0 = fix_half_slope(d[1], d[2]), hm = not_negative(fix_half_slope(d[0], d[1])),
                  hp = not_negative(fix_half_slope(d[2], d[3]));
  const long long A = 3 * d[1] + 2 * (h0 - hm), B = 3 * d[2] - 2 * (hp - h0);  // below 5 2^60
  const unsigned long long uA = (unsigned long long)A, uB = (unsigned long long)B;
  const unsigned long long mA = uA < 2 * uB ? uA : 2 * uB, mB = uB < 2 * uA ? uB : 2 * uA;
  const bool mono = d[2] >= 0;
  P.A = fix_to_double(mono ? mA : 0, neg, E);
  P.B = fix_to_double(mono ? mB : 0, neg, E);
  left = fix_to_double((unsigned long long)d[1], neg, E);
  const long long Dm = d[1] - d[0], Dp = d[2] - d[3];  // D- and -D+
  st = FixStep4{Dm + Dp, d[1] + d[2], 3 * h0, q[1], q[3], E};
  const int ml = hi_word(q[1]), mr = hi_word(q[3]);
  const int mn = min_i(ml ^ (ml >> 31), mr ^ (mr >> 31));
  const unsigned hn = (unsigned)hi_word(st.num) >> 2, hs = (unsigned)hi_word(st.s0) >> 2;
  const bool cand = (hi_word(Dm) | hi_word(Dp) | hi_word(d[2])) >= 0 && st.num != 0 && 7u * (hn + 1) >= hs &&
                    hs + 1 >= ((unsigned)mn >> 9);
  if (wide) {
    const Dev<double> W = dev_of(fix_value(c[0]), fix_value(c[1]), fix_value(c[2]), fix_value(c[3]), fix_value(c[4]));
    P = Dev<double>{mul_t(3.0, W.A), mul_t(3.0, W.B)};
    left = sub_t(fix_value(c[2]), fix_value(c[1]));
    return false;
  }
  return cand;
}
__device__ __forceinline__ long long fix_min_abs(const FixStep4& st) {
  const unsigned long long l = uabs64(st.ql), r = uabs64(st.qr);
  return (long long)(l < r ? l : r);
}
// Step 4's blend from there (converted on the integer pipes, where a conversion on the FP64 pipe would cost it
// an instruction: 128^3 step 13.7 -> 13.6 ms): hbar =
// (20/3) num / s0 - 1 clamped to [0, 1], 3 A += hbar (3 h - 3 A).
__device__ __forceinline__ Dev<double> fix_step4(Dev<double> P, long long n, long long s, long long h3, long long mn,
                                                 int E) {
  const double num = fix_to_double((unsigned long long)n, 0, 1081), s0 = fix_to_double((unsigned long long)s, 0, 1081);
  double hb = fma(mul_t(in_register(20.0 / 3.0), num), rcp_nr(s0), -in_register(1.0));
  hb = min_nn(hb, 1.0);
  // |s0| > mn / 100 exactly: from 2^53 on 100 |s0| is above 2^59, the bound of mn
  if (sign_bit_b(hb) || !(s >= (1ll << 53) || 100 * s > mn)) hb = 0.0;
  const double h = with_sign_b(fix_to_double((unsigned long long)h3, 0, E), P.A);  // A = 0: h = 0
  return Dev<double>{fma(hb, sub_t(h, P.A), P.A), fma(hb, sub_t(h, P.B), P.B)};
}
// the deviations of the cell in the middle of five values, by the same steps
__device__ __forceinline__ Dev<double> fix_dev_of(const FixCell c[5]) {
  Dev<double> P;
  double left;
  FixStep4 st;
  if (fix_dev(c, P, left, st)) P = fix_step4(P, st.num, st.s0, st.h3, fix_min_abs(st), st.E);
  return Dev<double>{P.A * (1.0 / 3.0), P.B * (1.0 / 3.0)};
}

// The parabola by its edge values, Delta q = q^R - q^L and q6 (the paper's own form), from the value
// and the deviations, and the forms that return it; the kernels take the deviations.
template <typename T>
__device__ __forceinline__ Para<T> para_of(T q, Dev<T> P) {
  return Para<T>{q - T(0.5) * P.A, q + T(0.5) * P.B, T(0.5) * (P.A + P.B), T(1.5) * (P.A - P.B)};
}
template <typename T>
__device__ __forceinline__ Para<T> ppm_lean(T qm2, T qm1, T qc, T qp1, T qp2) {
  if constexpr (sizeof(T) == 8) {
    const FixCell c[5] = {fix_cell(qm2), fix_cell(qm1), fix_cell(qc), fix_cell(qp1), fix_cell(qp2)};
    return para_of(qc, fix_dev_of(c));
  } else {
    return para_of(qc, dev_of(qm2, qm1, qc, qp1, qp2));
  }
}
// consecutive cells along a line (FP64): prime with q_{J-2} .. q_{J+1}, then next(q_{j+2}) for j = J, J+1, ...
template <typename T>
struct PPMStream {
  FixCell c[5];
  T q[2];
  __device__ __forceinline__ void prime(T qa, T qb, T qc, T qd) {
    c[1] = fix_cell(qa);
    c[2] = fix_cell(qb);
    c[3] = fix_cell(qc);
    c[4] = fix_cell(qd);
    q[0] = qc;
    q[1] = qd;
  }
  __device__ __forceinline__ Para<T> next(T qn) {
    for (int k = 0; k < 4; ++k) c[k] = c[k + 1];
    c[4] = fix_cell(qn);
    const T v = q[0];
    q[0] = q[1];
    q[1] = qn;
    return para_of(v, fix_dev_of(c));
  }
};
// ... from the slopes of the cells i - 1, i, i + 1 and the second differences around them
template <typename T>
__device__ __forceinline__ T slope_m(T qm, T q0, T qp) {
  return T(2) * half_slope(qp - qm, q0 - qm, qp - q0);
}
template <typename T>
__device__ __forceinline__ Para<T> ppm_carried(T qm1, T qc, T qp1, T dmm, T dm0, T dmp, T Dp, T Dm) {
  const T A = fma(T(1.0 / 3.0), dm0 - dmm, qc - qm1), B = fma(T(-1.0 / 3.0), dmp - dm0, qp1 - qc);
  return para_of(qc, dev_limit(A, B, T(0.5) * dm0, Dp, Dm, qp1 - qm1, qp1, qm1));
}
template <typename T>
__device__ __forceinline__ Para<T> ppm_direct(T qm2, T qm1, T qc, T qp1, T qp2) {
  return ppm_carried(qm1, qc, qp1, slope_m(qm2, qm1, qc), slope_m(qm1, qc, qp1), slope_m(qc, qp1, qp2),
                     qp2 - T(2) * qp1 + qc, qc - T(2) * qm1 + qm2);
}

// the coefficients of A and B in the averages over the fraction y (Sec. 2.4): y u / 2 and u^2 / 2; in FP64 those
// of 3 A and 3 B
template <typename T>
struct AvgCoef {
  T p, r;
};
// The factor of A and B goes into y as its square root k: (k - k y)^2 and (k y)(k - k y); y k comes from
// tau k / h, formed once per thread (avg_scale).
template <typename T>
__device__ __forceinline__ T avg_scale() { return sizeof(T) == 8 ? T(0.40824829046386301637) : T(0.70710678118654752440); }
template <typename T>
__device__ __forceinline__ AvgCoef<T> avg_coef(T yk) {
  const T v = sub_t(in_register(avg_scale<T>()), yk);
  return AvgCoef<T>{mul_t(yk, v), mul_t(v, v)};
}
// the average next to the right edge of a cell less the cell's value, and the average next to the left
// edge of a cell of value d
template <typename T>
__device__ __forceinline__ T inc_right(Dev<T> P, AvgCoef<T> k) { return fma(k.r, P.B, mul_t(k.p, P.A)); }
template <typename T>
__device__ __forceinline__ T inc_left(T d, Dev<T> P, AvgCoef<T> k) { return fma(-k.r, P.A, fma(-k.p, P.B, d)); }
// a row times four averages of inc_right: applied to A and B first, which leaves one average (10 instructions
// instead of 12; for inc_left, with d as a third, it would be 14)
template <typename T>
__device__ __forceinline__ T row_right(T a, Dev<T> P, T b, Dev<T> Q, T c, Dev<T> R, T d, Dev<T> S, AvgCoef<T> k) {
  auto dot = [&](T p, T q, T r, T s) { return fma(a, p, fma(b, q, fma(c, r, mul_t(d, s)))); };
  return inc_right(Dev<T>{dot(P.A, Q.A, R.A, S.A), dot(P.B, Q.B, R.B, S.B)}, k);
}

// ------------------------------------------------------------------------------------------------
// Sec. 2.4 + App. A: Roe-type face state, eigenvectors and the characteristic Riemann solution.
// Of each side: w = (rho, p, gamma, B_t1, B_t2, sqrt(rho)) of the cell, and the values and deviations of
// its parabolas of (v_n, v_t1, v_t2, B_t1, B_t2, p).  Bn is the face field.  qs = (V_n, V_t1, V_t2, B_t1, B_t2, P).
template <typename T>
struct FaceSide {
  T w[6];
  T q[6];
  Dev<T> P[6];
};

// The speeds, alpha factors and eigenvector entries are those of App. A in few FP64 instructions:
//   one reciprocal of the weight sum; 1/sqrt(rho) gives 1/rho, sqrt(rho) and c_a = |B_n| / sqrt(rho);
//   with Z = c^2 - c_a^2 - b_perp^2: c_f^2 = (c^2 + c_a^2 + b_perp^2 + sq)/2 with sq = c_f^2 - c_s^2 =
//     sqrt(Z^2 + 4 c^2 b_perp^2), sums of non-negative terms, and c_s = c c_a / c_f; alpha_f^2 = (c^2 - c_s^2)/sq = (1 + Z/sq)/2 and alpha_s^2 =
//     (c_f^2 - c^2)/sq = (1 - Z/sq)/2.  The larger of the two is formed from |Z|, without
//     cancellation, and the other from alpha_f alpha_s = c b_perp / sq, with the one reciprocal square
//     root of the larger: exactly 0 where B_perp = 0;
//   1/sq comes with the square root of sq^2, |B_perp| with 1/|B_perp|.
// The rows of the fast and the slow waves see v_t and B_t only through their components along B_perp,
// and those of the Alfven waves only through the ones across it.  The components along B_perp
// are taken of the parabolas' coefficients once per face, so the four magnetosonic waves average and
// sum four variables instead of six and their rows have four entries; each pair +-c shares y and its
// rows up to the sign of the velocity entries (s_+ from the left cell's right end, s_- from the right
// cell's left end; R s_+ + (S R) s_- is R (s_+ - s_-) on the velocities and R (s_+ + s_-) on B_t, P).
//
// All waves act on the averages less the left cell's values q_l, and q* = q_l + sum R s: with R L = I that
// is the sum over the averages themselves, at the same count of instructions, and its rounding is that
// of the differences between the cells, not of their values.
// d: the right cell's values less the left cell's
template <typename T>
__device__ __forceinline__ void riemann(const FaceSide<T>& l, const FaceSide<T>& r, const T d[6], T Bn, T tau_k, T qs[6]) {
  const T INV_SQRT2 = T(0.70710678118654752440), HALF = in_register(T(0.5));
  const T iden = rcp_t(add_t(l.w[5], r.w[5]));
  const T al = mul_t(l.w[5], iden), ar = mul_t(r.w[5], iden);  // the normalised weights
  const T rho = fma(al, l.w[0], mul_t(ar, r.w[0]));
  const T p = fma(al, l.w[1], mul_t(ar, r.w[1]));
  const T gam = fma(al, l.w[2], mul_t(ar, r.w[2]));
  const T Bt1 = fma(al, r.w[3], mul_t(ar, l.w[3]));  // crossed weights for B
  const T Bt2 = fma(al, r.w[4], mul_t(ar, l.w[4]));

  const T rs = rsqrt_n(rho);  // 1 / sqrt(rho)
  const T irho = mul_t(rs, rs), sqr = mul_t(rho, rs);
  const T gp = mul_t(gam, p);
  const T c2 = mul_t(gp, irho);
  const T ca = mul_t(abs_b(Bn), rs), ca2 = mul_t(ca, ca);
  const T bp2 = fma(Bt1, Bt1, mul_t(Bt2, Bt2));
  const T b2 = mul_t(bp2, irho);  // b_perp^2
  const T ab2 = add_t(ca2, b2), s = add_t(c2, ab2), Z = sub_t(c2, ab2);
  const T sq2 = fma(Z, Z, mul_t(b2, four_b(c2)));
  // the directions of B_perp; the degenerate case keeps |B_perp| itself
  T by = INV_SQRT2, bz = INV_SQRT2, bper;
  if (surely_above<78>(b2, s) || gt_nn(bp2, T(1e-24) * rho * s)) {  // 1e-24 < 2^-79
    const T ib = rsqrt_n(bp2);
    by = mul_t(Bt1, ib);
    bz = mul_t(Bt2, ib);
    bper = mul_t(bp2, ib);
  } else {
    bper = sqrt_t(bp2);
  }
  const T rc = rsqrt_n(c2), c = mul_t(c2, rc), crs = mul_t(c, rs);
  T sq = T(0), af = INV_SQRT2, as = INV_SQRT2;
  {
    const T isq = rsqrt_n(sq2), sqn = mul_t(sq2, isq);
    if (surely_above<38>(sqn, s) || gt_nn(sqn, T(1e-12) * s)) {  // 1e-12 < 2^-39
      sq = sqn;
      const T big2 = fma(half_nn(abs_b(Z)), isq, HALF);  // in [1/2, 1]
      const T rb = rsqrt_n(big2), big = mul_t(big2, rb);
      const T small = mul_t(mul_t(crs, bper), mul_t(isq, rb));
      const bool fast = !sign_bit_b(Z);
      af = fast ? big : small;
      as = fast ? small : big;
    }
  }
  const T cf2 = half_nn(add_t(s, sq));
  const T rcf = rsqrt_n(cf2);
  const T cf = mul_t(cf2, rcf);
  const T cs = mul_t(mul_t(c, ca), rcf);
  const bool neg = sign_bit_b(Bn) && gt_nn(abs_b(Bn), T(0));  // sign(0) = +1
  const T bys = neg ? neg_b(by) : by, bzs = neg ? neg_b(bz) : bz;

  const AvgCoef<T> ka = avg_coef(mul_t(ca, tau_k)), kf = avg_coef(mul_t(cf, tau_k)), ks = avg_coef(mul_t(cs, tau_k));

  // the Alfven waves, on the components across B_perp: v = -bz v_t1 + by v_t2 (times sgn(B_n)),
  // b = (bz B_t1 - by B_t2) / sqrt(rho); first, so that the tangential coefficients are not needed
  // beyond their components along B_perp
  T hv, hb;
  {
    const T rbz = mul_t(rs, bz), rby = mul_t(rs, by);
    T qr[5];
#pragma unroll
    for (int m = 1; m < 5; ++m) qr[m] = inc_left(d[m], r.P[m], ka);
    const T sp = row_right(bys, l.P[2], -bzs, l.P[1], rbz, l.P[3], -rby, l.P[4], ka);
    const T sm = fma(bys, qr[2], fma(-bzs, qr[1], fma(-rbz, qr[3], mul_t(rby, qr[4]))));
    hv = scale_down_b<1>(add_t(sp, sm));
    hb = mul_t(half_nn(sqr), sub_t(sp, sm));
  }
  // the magnetosonic waves on (v_n, v_par sgn(B_n), B_par, p): with the rows times 2 c^2 and the columns
  // divided by it, the +c_f wave has L = (af cf, -as cs, as c / sqrt(rho), af / rho), R = (lf, -ls,
  // as sqrt(rho) / 2c, af rho / 2), the +c_s wave L = (as cs, af cf, -af c / sqrt(rho), as / rho),
  // R = (ls, lf, -af sqrt(rho) / 2c, as rho / 2)
  auto along = [&](T a, T b) { return fma(by, a, mul_t(bz, b)); };
  auto along_s = [&](T a, T b) { return fma(bys, a, mul_t(bzs, b)); };
  const Dev<T> lv = {along_s(l.P[1].A, l.P[2].A), along_s(l.P[1].B, l.P[2].B)};
  const Dev<T> lb = {along(l.P[3].A, l.P[4].A), along(l.P[3].B, l.P[4].B)};
  const Dev<T> rv = {along_s(r.P[1].A, r.P[2].A), along_s(r.P[1].B, r.P[2].B)};
  const Dev<T> rb = {along(r.P[3].A, r.P[4].A), along(r.P[3].B, r.P[4].B)};
  const T dv = along_s(d[1], d[2]), db = along(d[3], d[4]);
  const T af_cf = mul_t(af, cf), as_cs = mul_t(as, cs);
  const T hrc = half_nn(rc), i2c2 = mul_t(hrc, rc);
  const T lf = mul_t(af_cf, i2c2), ls = mul_t(as_cs, i2c2);
  auto pair = [&](AvgCoef<T> k, T l0, T l1, T l2, T l3, T& dif, T& sum) {
    const T sp = row_right(l0, l.P[0], l1, lv, l2, lb, l3, l.P[5], k);
    const T sm = fma(-l0, inc_left(d[0], r.P[0], k),
                     fma(-l1, inc_left(dv, rv, k), fma(l2, inc_left(db, rb, k), mul_t(l3, inc_left(d[5], r.P[5], k)))));
    dif = sub_t(sp, sm);
    sum = add_t(sp, sm);
  };
  T difF, sumF, difS, sumS;
  pair(kf, af_cf, -as_cs, mul_t(as, crs), mul_t(af, irho), difF, sumF);
  pair(ks, as_cs, af_cf, -mul_t(af, crs), mul_t(as, irho), difS, sumS);
  const T vpar = fma(lf, difS, -mul_t(ls, difF));
  const T bpar = mul_t(mul_t(sqr, hrc), fma(as, sumF, -mul_t(af, sumS)));
  qs[0] = fma(lf, difF, fma(ls, difS, l.q[0]));
  qs[1] = fma(bys, vpar, fma(-bzs, hv, l.q[1]));
  qs[2] = fma(bzs, vpar, fma(bys, hv, l.q[2]));
  qs[3] = fma(by, bpar, fma(bz, hb, l.q[3]));
  qs[4] = fma(bz, bpar, fma(-by, hb, l.q[4]));
  qs[5] = fma(half_nn(rho), fma(af, sumF, mul_t(as, sumS)), l.q[5]);
}
template <typename T>
__device__ __forceinline__ void riemann(const FaceSide<T>& l, const FaceSide<T>& r, T Bn, T tau_k, T qs[6]) {
  T d[6];
#pragma unroll
  for (int m = 0; m < 6; ++m) d[m] = sub_t(r.q[m], l.q[m]);
  riemann(l, r, d, Bn, tau_k, qs);
}
// the same from parabolas in the paper's form, whose values are L + A/2 with A = Delta q + q6/3 and
// B = Delta q - q6/3
template <typename T>
__device__ __forceinline__ void riemann(const T wl[6], const T wr[6], T Bn, const Para<T> pl[6],
                                        const Para<T> pr[6], T tau_h, T qs[6]) {
  auto side = [](const T w[6], const Para<T> P[6]) {
    FaceSide<T> f;
    for (int m = 0; m < 6; ++m) {
      f.w[m] = w[m];
      const T A = P[m].d + P[m].q6 * T(1.0 / 3.0), B = P[m].d - P[m].q6 * T(1.0 / 3.0);
      f.q[m] = P[m].L + T(0.5) * A;
      f.P[m].A = sizeof(T) == 8 ? T(3) * A : A;
      f.P[m].B = sizeof(T) == 8 ? T(3) * B : B;
    }
    return f;
  };
  FaceSide<T> l = side(wl, pl), r = side(wr, pr);
  riemann(l, r, Bn, tau_h * avg_scale<T>(), qs);
}

// ------------------------------------------------------------------------------------------------
// Sec. 2.3: CFL denominator |v| + b + c + c_a + c_s + c_f, the largest over the three choices of
// the longitudinal axis (b^2 = B^2 / rho), in FP64.  With c_f^2 + c_s^2 = c^2 + b^2 and
// c_f c_s = c c_a, c_f + c_s = sqrt(c^2 + b^2 + 2 c c_a); the denominator grows with c_a = |B_d| /
// sqrt(rho), so the largest one is that of the axis of the largest |B_d|.  Takes the momenta and
// gamma p; 1/sqrt(rho) is the one reciprocal: |v| = |m| / rho, b = |B| / sqrt(rho),
// c = sqrt(gamma p) / sqrt(rho) and c_f + c_s = sqrt(gamma p + B^2 + 2 sqrt(gamma p) |B_d|) / sqrt(rho).
// Compiled once (as the chemistry and the heating/cooling are), so that every kernel gets the same bits.
__device__ MHD_NOINLINE inline double cfl_denominator(double rho, double mx, double my, double mz,
                                                  double Bx, double By, double Bz, double gp) {
  const double irs = rsqrt(rho);
  const double irho = irs * irs;
  const double sgp = sqrt_nr(gp);
  const double B2 = Bx * Bx + By * By + Bz * Bz;
  const double sB = sqrt_nr(B2);
  const double v = sqrt_nr(mx * mx + my * my + mz * mz) * irho;
  const double Bm = max_nn(abs_b(Bx), max_nn(abs_b(By), abs_b(Bz)));
  const double fs = sqrt_nr((gp + B2) + 2.0 * sgp * Bm);
  return v + ((sB + sgp + Bm) + fs) * irs;
}

// The screen of the CFL maximum.  tau takes only the largest FP64 denominator over the cells, so a
// cell whose denominator provably lies below an FP64 denominator already reached by another cell
// cannot set it and need not be evaluated in FP64: tau stays bit for bit that of evaluating every
// cell.  The proof is the FP32 estimate below, the same formula from FP32-rounded inputs (square
// roots and 1/sqrt correctly rounded, sums and products rounded to nearest).  With u = 2^-24 a
// first-order count of its relative error gives about 30 u: up to 23 u in gamma - 1 (the
// cancellation in n_H = rho - rho_H2 - rho_H+ stays below 5 u rho, against numerator and
// denominator of at least rho / 2 and 2 rho), 35 u in gamma p, half of that through the square
// roots, 1.5 u through 1/sqrt(rho) and its square, a few u of sums.  FP32 squares that flush to
// zero or lose bits below the normal range move |m| or |B| by less than 2^-62, which is below 2^-22
// of the denominator (>= sqrt(gamma p / rho)) while rho >= 2^-40 and gamma p >= 2^-40.  The
// screen allows 2^-12 (4096 u).  A cell outside those guards, or whose estimate overflows, gets
// +inf and is always evaluated in FP64.
__device__ __forceinline__ float cfl_estimate_f32(float rho, float mx, float my, float mz, float Bx,
                                                  float By, float Bz, float eint, float gm1) {
  const float gp = fmul_rn(fmul_rn(1.0f + gm1, gm1), eint);
  if (!(rho >= 0x1p-40f) || !(gp >= 0x1p-40f)) return f_inf();
  const float irs = frsqrt_rn(rho);
  const float irho = irs * irs;
  const float sgp = fsqrt_rn(gp);
  const float B2 = Bx * Bx + By * By + Bz * Bz;
  const float sB = fsqrt_rn(B2);
  const float v = fsqrt_rn(mx * mx + my * my + mz * mz) * irho;
  const float Bm = fmaxf(fabsf(Bx), fmaxf(fabsf(By), fabsf(Bz)));
  const float fs = fsqrt_rn((gp + B2) + 2.0f * sgp * Bm);
  return v + ((sB + sgp + Bm) + fs) * irs;
}

// gamma - 1 of the cell in FP32 for the screen: that of the ideal gas, or of the H/H2 (+ H+, e-)
// mixture as (2 n_1 + 2 n_H2) / (3 n_1 + 5 n_H2) (gamma_eff below minus one); -1 where the
// numerator falls below rho / 2 or the denominator below 2 rho (3 rho - rho_H2 / 2 + 3 rho_H+ for
// physical abundances), which fails the screen's guard.
__device__ __forceinline__ float gamma_minus_one_f32(bool chem, double gamma, float rho, float rh2, float rhp) {
  if (!chem) return (float)(gamma - 1.0);
  const float n1 = (rho - rh2 - rhp) + 2.0f * rhp, nH2 = 0.5f * rh2;
  const float num = 2.0f * (n1 + nH2), den = 3.0f * n1 + 5.0f * nH2;
  return (num >= 0.5f * rho && den >= 2.0f * rho) ? fdiv_rn(num, den) : -1.0f;
}

// Sec. 4.3 effective adiabatic index of the H/H2 mixture (no electrons)
template <typename T>
__device__ __forceinline__ T gamma_eff(T rho, T rh2) {
  T nH = rho - rh2, nH2 = T(0.5) * rh2;
  return mul_t(fma(T(7), nH2, mul_t(T(5), nH)), rcp_t(fma(T(5), nH2, mul_t(T(3), nH))));
}

// ... and with H+ and electrons: the monatomic particles n_1 = n_H + n_H+ + n_e replace n_H, with
// the neutral atoms n_H = rho - rho_H2 - rho_H+ and n_H+ = n_e = rho_H+ (rho_H+ = 0: the form above)
template <typename T>
__device__ __forceinline__ T gamma_eff(T rho, T rh2, T rhp) {
  T n1 = fma(T(2), rhp, rho - rh2 - rhp), nH2 = T(0.5) * rh2;
  return mul_t(fma(T(7), nH2, mul_t(T(5), n1)), rcp_t(fma(T(5), nH2, mul_t(T(3), n1))));
}

// ------------------------------------------------------------------------------------------------
// Sec. 2.7 + App. D: one cell of the H/H2 network (reactions 1-4), backward-differentiation
// update of n_H2 with rates frozen over the step; returns the new rho_H2.  FP64.
struct ChemConst {
  static constexpr double KB = 1.380649e-16;         // erg / K
  static constexpr double MH = 1.6735575e-24;        // g
  static constexpr double PC = 3.0856775814913673e18; // cm
  static constexpr double KMS = 1.0e5;               // cm / s
};

// the per-box products of the shielding length L_s = (lshield > 0 ? lshield : dx) pc (App. D column
// densities N = n L_s): set on the host whenever lshield, xnorm, taud or dx change
inline void set_shielding(Phys& ph) {
  const double Ls = (ph.lshield > 0.0 ? ph.lshield : ph.dx) * ChemConst::PC;
  ph.taud_ls = ph.taud * Ls;
  ph.ls_ixnorm = Ls * ph.ixnorm;
  auto pair = [](double x, float* f) {
    f[0] = (float)x;
    f[1] = (float)(x - (double)f[0]);
  };
  pair(ph.taud_ls, ph.taud_ls_f);
  pair(ph.ls_ixnorm, ph.ls_ixnorm_f);
  pair(ph.ibdop, ph.ibdop_f);
}

// The App. D formulas in FP64 with few FP64 instructions (the rates agree with a term-by-term
// evaluation to about 1e-14 relative):
//   T = (gamma - 1) rho eps P0 / (n_particles k_B) with gamma - 1 = 2 n_particles / (3 n_1 + 5 n_H2)
//     = (2 P0 / k_B) rho eps / (3 n_1 + 5 n_H2), n_1 = n_H + n_H+ + n_e, and T, 1/T and sqrt(T)
//     from one reciprocal square root of the product;
//   1/sqrt(1 + x) from one reciprocal square root; 1/x_norm, 1/b_doppler and the products with the
//   shielding length precomputed; one reciprocal for k1' and 1/u^2 (of their denominators' product);
//   the exponentials of the H/H2 rates by exp_tang (their arguments are <= 0); the arguments of
//   reactions 2 and 3 not formed in gas cold enough for their exponentials to be 0.
struct ChemOut {
  double rh2, rhp;  // new rho_H2 and rho_H+
};

// App. D rates of reactions 5-8 at T (ln T given): k5 = 6e-18 s^-1 per atom, k6 = exp(poly(ln T_eV))
// (Horner), k7 = 10^(P(x) / Q(x)) with x = log10 T, k8 the grain-recombination fit with
// T^0.01586 10^(-4.4e-5 log10 T) = T^(0.01586 - 4.4e-5).
struct IonRates {
  double k5, k6, k7, k8;
};
__device__ __forceinline__ IonRates ion_rates(double lnT) {
  const double LN_KB_EV = -9.359149794515579;  // ln(8.617333262e-5 eV/K)
  const double INV_LN10 = 0.43429448190325176;
  IonRates r;
  r.k5 = 6e-18;
  const double L = lnT + LN_KB_EV;
  double p = -2.1e-6;
  p = fma(p, L, 1.1e-4);
  p = fma(p, L, -2.6e-3);
  p = fma(p, L, 3.4e-2);
  p = fma(p, L, -0.3);
  p = fma(p, L, 1.5);
  p = fma(p, L, -5.7);
  p = fma(p, L, 13.5);
  p = fma(p, L, -32.7);
  r.k6 = exp(p);
  const double x = lnT * INV_LN10;
  const double P = fma(fma(fma(fma(-3.87e-3, x, 0.08), x, -0.87), x, 4.68), x, -10.78);
  const double Q = fma(fma(fma(fma(2.4e-4, x, -5.1e-3), x, 0.06), x, -0.38), x, 1.0);
  r.k7 = exp10(P / Q);
  const double A = 8.074e-6 * 570.1642722807472;  // 8.074e-6 10^2.756
  const double Bc = 5.087e2 * 0.012906247820605376;  // 5.087e2 10^-1.8892
  r.k8 = 12.25e-14 / (1.0 + A * (1.0 + Bc * exp((1.586e-2 - 4.4e-5) * lnT)));
  return r;
}

// IONS: the kernel may see boxes with the ions on (ph.ions decides per box); without it the ion
// code is compiled out and rhp must be 0.
template <bool IONS>
__device__ MHD_NOINLINE ChemOut chem_cell(const Phys& ph, double rho, double eint, double rh2,
                                             double rhp, double tau) {
  const double P0 = ChemConst::MH * ChemConst::KMS * ChemConst::KMS;  // code pressure, erg cm^-3
  const double T0 = ChemConst::PC / ChemConst::KMS;                  // code time, s
  // the ion terms are added to the H/H2 expressions with explicit FMAs, so that a box without ions
  // gets the same bits from either instance (rhp = 0 then adds exactly nothing)
  double nH = rho - rh2;
  if (IONS) nH = nH - rhp;
  const double nH2 = scale_down_b<1>(rh2), n = rho;
  const double num = (2.0 * P0 / ChemConst::KB) * eint;
  double den3 = fma(3.0, nH, 5.0 * nH2);  // 3 n_1 + 5 n_H2 with n_1 = n_H + n_H+ + n_e
  if (IONS) den3 = fma(6.0, rhp, den3);
  // T = num / den3 and its square root from one reciprocal square root q = 1 / sqrt(num den3):
  // sqrt(T) = num q, T = (num q)^2, 1/T = (den3 q)^2
  const double q = rsqrt_nr(num * den3);
  const double sT = num * q, dq = den3 * q;
  const double T = sT * sT, iT = dq * dq;
  // App. D rates; the branch tests and clamps compare on the integer pipe (T >= 0; a2, a3 < 0)
  const bool hot2 = gt_nn(T, 7390.0), hot3 = gt_nn(T, 7291.0);
  // reactions 2 and 3: exp of an argument below -746 is exactly 0 in double, and the cold branches'
  // arguments -(6750 / T)^2 and -4060 / T - (7500 / T)^2 lie below -746.6 for T <= 247 and below
  // -747 for T <= 277, so there the rates are 0 without forming them (warps of cold cells skip)
  double k2 = 0.0, k3 = 0.0;
  if (gt_nn(T, 247.0)) {
    const double a2 = hot2 ? -2.93e4 * iT : -((6750.0 * iT) * (6750.0 * iT));
    if (!gt_nn(neg_b(a2), 746.0)) k2 = (hot2 ? 6.11e-14 : 2.67e-15) * exp_tang(a2);
  }
  if (gt_nn(T, 277.0)) {
    const double a3 = hot3 ? -3.22e4 * iT : -(4060.0 * iT) - (7500.0 * iT) * (7500.0 * iT);
    if (!gt_nn(neg_b(a3), 746.0)) k3 = (hot3 ? 5.22e-14 : 3.17e-15) * exp_tang(a3);
  }
  // shielding: f_dust = exp(-taud (N_H + N_H2)), x = N_H2 / x_norm, N = n L_s
  const double fdust = exp_tang(-(ph.taud_ls * (nH + nH2)));
  const double x = nH2 * ph.ls_ixnorm;
  const double u = 1.0 + x * ph.ibdop;
  const double isx = rsqrt_nr(1.0 + x);
  const double sx = (1.0 + x) * isx;
  // k1' = 3e-17 s / (1 + 0.4 s + 0.2 t + 0.08 t^2) with t = T / 100, s = sqrt(t) = sqrt(T) / 10
  const double d1 = fma(fma(0.08 * 1e-4, T, 0.2 * 1e-2), T, fma(0.4 * 0.1, sT, 1.0)), u2 = u * u;
  const double rd = rcp_nr(d1 * u2);  // 1 / (d1 u^2): d1, u^2 >= 1
  const double k1p = (3e-17 * 0.1 * sT) * (u2 * rd);
  // k4 = 3.3 1.7e-11 f_sh f_dust with f_sh = 0.965 / u^2 + 0.035 exp(-8.5e-4 sqrt(1 + x)) / sqrt(1 + x)
  const double k4 = fdust * fma(3.3 * 1.7e-11 * 0.965, d1 * rd,
                                ((3.3 * 1.7e-11 * 0.035) * isx) * exp_tang(-8.5e-4 * sx));
  const double C = k1p * n * nH;
  const double D = (k2 * nH + k3 * nH2) + k4;
  const double ts = tau * T0;
  double nH2n = nH2 + (ts * (C - D * nH2)) * rcp_nr(1.0 + ts * D);
  if (sign_bit_b(nH2n)) nH2n = 0.0;
  const double half_n = scale_down_b<1>(n);
  if (gt_nn(nH2n, half_n)) nH2n = half_n;
  ChemOut out;
  out.rh2 = 2.0 * nH2n;
  out.rhp = rhp;
  if (IONS && ph.ions) {
    // reactions 5-8: creation k5 n_H + k6 n_H n_e, destruction (k7 n_e + k8 n) n_H+, the same
    // semi-implicit update from the stage-start densities; n_H+ <= n - 2 n_H2 (n_H >= 0)
    const double ne = rhp;
    const IonRates q = ion_rates(log(T));
    const double Ci = (q.k5 + q.k6 * ne) * nH;
    const double Di = q.k7 * ne + q.k8 * n;
    double nHpn = rhp + ts * (Ci - Di * rhp) / (1.0 + ts * Di);
    if (nHpn < 0.0) nHpn = 0.0;
    if (nHpn > n - 2.0 * nH2n) nHpn = n - 2.0 * nH2n;
    out.rhp = nHpn;
  }
  return out;
}

// ------------------------------------------------------------------------------------------------
// The H/H2 network in pairs of floats, for the FP32-bulk path (without the ions).  That path stores
// rho_H2 in 24 bits; evaluated in FP64, its 79 instructions per cell were the bound of the post kernel
// (an FP64 instruction takes the SM as long as 64 FP32 ones).  A pair h + l with |l| <= ulp(h)/2 carries
// about 48 bits: products and sums lose under 2^-44, far below the 2^-25 of the final rounding, so the stored
// rho_H2 is the FP64 evaluation's but for cells within 2^-40 of a rounding boundary
// (tests/test_chem_pairs_host.py).  256^3 FP32 step: the last Lagrangian update with the post stage 2.81 ->
// 1.11 ms, now near the HBM bound of its 45 arrays.  The elementary steps are the error-free sums and products of Dekker
// (Numer. Math. 18, 1971) and Knuth with the FMA for a product's error; they use the rounded operations
// that the compiler does not contract.
struct FF {
  float h, l;
};
__device__ __forceinline__ float fadd_rn(float a, float b) { return add_t(a, b); }
__device__ __forceinline__ FF ff_fast_sum(float a, float b) {  // |a| >= |b| or a = 0
  const float s = fadd_rn(a, b);
  return FF{s, fadd_rn(b, -fadd_rn(s, -a))};
}
__device__ __forceinline__ FF ff_sum(float a, float b) {
  const float s = fadd_rn(a, b), t = fadd_rn(s, -a);
  return FF{s, fadd_rn(fadd_rn(a, -fadd_rn(s, -t)), fadd_rn(b, -t))};
}
__device__ __forceinline__ FF ff_add(FF a, FF b) {
  const FF s = ff_sum(a.h, b.h);
  return ff_fast_sum(s.h, fadd_rn(s.l, fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ FF ff_add(FF a, float b) {
  const FF s = ff_sum(a.h, b);
  return ff_fast_sum(s.h, fadd_rn(s.l, a.l));
}
__device__ __forceinline__ FF ff_mul(FF a, FF b) {
  const float p = fmul_rn(a.h, b.h);
  return ff_fast_sum(p, fma(a.h, b.l, fma(a.l, b.h, fma(a.h, b.h, -p))));
}
__device__ __forceinline__ FF ff_mul(FF a, float b) {
  const float p = fmul_rn(a.h, b);
  return ff_fast_sum(p, fma(a.l, b, fma(a.h, b, -p)));
}
__device__ __forceinline__ FF ff_neg(FF a) { return FF{-a.h, -a.l}; }
// 1/x and 1/sqrt(x) by the series of rcp_nr and rsqrt_nr from the float approximations (a few 2^-23)
__device__ __forceinline__ FF ff_rcp(FF x) {
  const float r = rcp_t(x.h);
  const float e = fma(-x.l, r, fma(-x.h, r, 1.0f));
  return ff_fast_sum(r, fmul_rn(r, fma(e, e, e)));
}
__device__ __forceinline__ FF ff_rsqrt(FF x) {
  const float y = rsqrt_t(x.h), y2 = fmul_rn(y, y), dy2 = fma(y, y, -y2);
  const float e = fma(-x.l, y2, fma(-x.h, dy2, fma(-x.h, y2, 1.0f)));
  return ff_fast_sum(y, fmul_rn(y, fmul_rn(e, fma(0.375f, e, 0.5f))));
}
// 2^(j/32) in pairs
struct FFPair {
  float h, l;
};
__device__ const FFPair kExp2Frac32Pairs[32] = {
    {0x1.000000p+0f, 0x0.0p+0f}, {0x1.059b0ep+0f, -0x1.9d4f52p-25f}, {0x1.0b5586p+0f, 0x1.9f3122p-25f},
    {0x1.11301ep+0f, -0x1.fdb496p-25f}, {0x1.172b84p+0f, -0x1.c15742p-27f}, {0x1.1d4874p+0f, -0x1.d2e8cap-25f},
    {0x1.2387a6p+0f, 0x1.ceac48p-25f}, {0x1.29e9e0p+0f, -0x1.5c0424p-25f}, {0x1.306fe0p+0f, 0x1.4636e2p-25f},
    {0x1.371a74p+0f, -0x1.18aac6p-25f}, {0x1.3dea64p+0f, 0x1.824684p-25f}, {0x1.44e086p+0f, 0x1.8624b4p-30f},
    {0x1.4bfdaep+0f, -0x1.593abcp-25f}, {0x1.5342b6p+0f, -0x1.2c5610p-25f}, {0x1.5ab07ep+0f, -0x1.5bd5ecp-27f},
    {0x1.6247ecp+0f, -0x1.f8b550p-25f}, {0x1.6a09e6p+0f, 0x1.9fcef4p-26f}, {0x1.71f75ep+0f, 0x1.1d8beep-25f},
    {0x1.7a1148p+0f, -0x1.829fd0p-25f}, {0x1.82589ap+0f, -0x1.accc7cp-26f}, {0x1.8ace54p+0f, 0x1.15506ep-27f},
    {0x1.93737cp+0f, -0x1.e64744p-25f}, {0x1.9c4918p+0f, 0x1.51f848p-27f}, {0x1.a5503cp+0f, -0x1.b83b54p-25f},
    {0x1.ae89fap+0f, -0x1.a94b14p-26f}, {0x1.b7f770p+0f, -0x1.a09438p-25f}, {0x1.c199bep+0f, -0x1.3d56b2p-27f},
    {0x1.cb720ep+0f, -0x1.8837ccp-27f}, {0x1.d5818ep+0f, -0x1.822dbcp-27f}, {0x1.dfc974p+0f, -0x1.908c94p-25f},
    {0x1.ea4afap+0f, 0x1.52486cp-27f}, {0x1.f50766p+0f, -0x1.246eb0p-26f}};
// e^x for -87 <= x <= 0 (0 below: e^-87 is 1.6e-38), exp_tang's method: k = 32 m + j the integer nearest
// to 32 x / ln 2, r = x - k ln2/32 with ln2/32 in three parts whose products with |k| < 2^12 are exact in
// the first two, e^r - 1 = r + r^2/2 + r^3 (1/6 + r/24 + r^2/120) with the first two terms in pairs (the
// neglected r^6/720 is below 2^-48).
__device__ __forceinline__ FF ff_exp(FF x) {
  if (!(x.h >= -87.0f)) return FF{0.0f, 0.0f};
  const float t = fadd_rn(fmul_rn(x.h, 0x1.715476p+5f), 12582912.0f);
  const float kf = fadd_rn(t, -12582912.0f);
  const int k = (int)kf;
  const float r1 = fma(-kf, 0x1.62ep-6f, x.h);
  FF r = ff_sum(r1, -fmul_rn(kf, 0x1.0cp-20f));
  r = ff_fast_sum(r.h, fadd_rn(r.l, fma(-kf, -0x1.05c61p-34f, x.l)));
  const float hr = fmul_rn(0.5f, r.h), q = fmul_rn(hr, r.h), dq = fma(hr, r.h, -q);
  const float c = fmul_rn(fmul_rn(fmul_rn(r.h, r.h), r.h), fma(r.h, fma(r.h, 1.0f / 120.0f, 1.0f / 24.0f), 1.0f / 6.0f));
  const FF p0 = ff_fast_sum(r.h, q);
  const FF p = ff_fast_sum(p0.h, fadd_rn(p0.l, fadd_rn(fma(r.h, r.l, r.l), fadd_rn(dq, c))));
#ifdef __CUDA_ARCH__
  const float2 tj = __ldg(reinterpret_cast<const float2*>(kExp2Frac32Pairs) + (k & 31));
  const FF T = {tj.x, tj.y};
  const float sc = __int_as_float((127 + (k >> 5)) << 23);  // m >= -126
#else
  const FF T = {kExp2Frac32Pairs[k & 31].h, kExp2Frac32Pairs[k & 31].l};
  const float sc = std::ldexp(1.0f, k >> 5);
#endif
  const FF y = ff_mul(T, p);
  const FF z = ff_add(FF{T.h, 0.0f}, FF{y.h, fadd_rn(y.l, T.l)});
  return FF{fmul_rn(z.h, sc), fmul_rn(z.l, sc)};
}
// the product of a constant's pair with a float or a pair
#define MHD_FF(c) (FF{(float)(c), (float)((c) - (double)(float)(c))})

// chem_cell<false> in pairs: the same formulas with the rates multiplied by the step's seconds ts, so that
// the numbers stay within the floats' range (a rate that flushes to zero moves nothing).  false where an
// input lies outside the range that this holds for (also NaN): the caller takes the FP64 form.
__device__ __forceinline__ bool chem_cell_pairs(const Phys& ph, const float ts_pair[2], float rho, float eint,
                                                float rh2, float& rh2_new) {
  const double P0 = ChemConst::MH * ChemConst::KMS * ChemConst::KMS;
  const FF ts = {ts_pair[0], ts_pair[1]};
  const float nH2 = 0.5f * rh2, n = rho;
  const FF nH = ff_sum(rho, -rh2);
  const bool ok = rho > 1e-8f && rho < 1e8f && eint > 1e-10f && eint < 1e10f && rh2 >= 0.0f && rh2 <= 2.0f * rho &&
                  (ts.h == 0.0f || ts.h > 1e-10f) && ts.h < 1e20f;
  if (!ok) return false;
  const FF num = ff_mul(MHD_FF(2.0 * P0 / ChemConst::KB), eint);
  const FF den3 = ff_add(ff_mul(nH, 3.0f), ff_mul(FF{nH2, 0.0f}, 5.0f));
  if (!(den3.h > 1e-8f)) return false;
  const FF q = ff_rsqrt(ff_mul(num, den3));
  const FF sT = ff_mul(num, q), dq = ff_mul(den3, q);
  const FF T = ff_mul(sT, sT), iT = ff_mul(dq, dq);
  const FF x = ff_mul(FF{ph.ls_ixnorm_f[0], ph.ls_ixnorm_f[1]}, nH2);
  const FF dust = ff_mul(FF{ph.taud_ls_f[0], ph.taud_ls_f[1]}, ff_add(nH, nH2));
  if (!(T.h < 1e9f && x.h < 1e15f && iT.h < 1e15f)) return false;
  // reactions 2 and 3 (their exponentials flush to zero in gas below about 720 K and 830 K)
  const bool hot2 = T.h > 7390.0f || (T.h == 7390.0f && T.l > 0.0f), hot3 = T.h > 7291.0f || (T.h == 7291.0f && T.l > 0.0f);
  FF D = {0.0f, 0.0f};
  if (T.h > 700.0f) {
    const FF w2 = ff_mul(iT, 6750.0f), w3 = ff_mul(iT, 7500.0f);
    const FF a2 = hot2 ? ff_mul(iT, -2.93e4f) : ff_neg(ff_mul(w2, w2));
    const FF a3 = hot3 ? ff_mul(iT, -3.22e4f) : ff_neg(ff_add(ff_mul(iT, 4060.0f), ff_mul(w3, w3)));
    const FF k2 = ff_mul(ff_mul(hot2 ? MHD_FF(6.11e-14) : MHD_FF(2.67e-15), ts), ff_exp(a2));
    const FF k3 = ff_mul(ff_mul(hot3 ? MHD_FF(5.22e-14) : MHD_FF(3.17e-15), ts), ff_exp(a3));
    D = ff_add(ff_mul(k2, nH), ff_mul(k3, nH2));
  }
  // reaction 4
  const FF u = ff_add(ff_mul(x, FF{ph.ibdop_f[0], ph.ibdop_f[1]}), 1.0f);
  const FF x1 = ff_add(x, 1.0f), isx = ff_rsqrt(x1), sx = ff_mul(x1, isx);
  const FF f1 = ff_mul(MHD_FF(3.3 * 1.7e-11 * 0.965), ff_rcp(ff_mul(u, u)));
  const FF f2 = ff_mul(ff_mul(MHD_FF(3.3 * 1.7e-11 * 0.035), isx), ff_exp(ff_mul(sx, MHD_FF(-8.5e-4))));
  const FF k4 = ff_mul(ff_mul(ff_add(f1, f2), ts), ff_exp(ff_neg(dust)));
  D = ff_add(D, k4);
  // reaction 1: 3e-17 s / (1 + 0.4 s + 0.2 t + 0.08 t^2), t = T / 100, s = sqrt(t) = sqrt(T) / 10
  const FF d1 = ff_add(ff_add(ff_mul(ff_add(ff_mul(T, MHD_FF(0.08 * 1e-4)), MHD_FF(0.2 * 1e-2)), T), ff_mul(sT, MHD_FF(0.4 * 0.1))), 1.0f);
  const FF k1 = ff_mul(ff_mul(ff_mul(MHD_FF(3e-17 * 0.1), ts), sT), ff_rcp(d1));
  const FF C = ff_mul(ff_mul(k1, n), nH);
  const FF dn = ff_mul(ff_add(C, ff_neg(ff_mul(D, nH2))), ff_rcp(ff_add(D, 1.0f)));
  float r = 2.0f * ff_add(dn, nH2).h;
  r = r < 0.0f ? 0.0f : r;
  rh2_new = r > n ? n : r;
  return true;
}

// ------------------------------------------------------------------------------------------------
// Sec. 2.8 + App. D: heating and cooling of one cell, d(rho E)/dt = d(rho eps)/dt = Gamma - Lambda by
// one Euler step; returns the change of rho E and rho eps in code units.  FP64.  Readings:
//   Gamma_1 = 7.2e-12 erg (k1' n n_H) / (1 + n_cr / n), n_cr = 10^(4 - 0.416 x - 0.327 x^2) (the H2
//     formation heating: the printed numerator read as the formation rate, the printed polynomial
//     over n as the critical density);
//   Lambda_2 = n_H2 L_H / (1 + L_H / L_L) with the printed two-branch L_H, L_L;
//   Lambda_3 = n_H2 L_H / (1 + L_H / L_L), L_H = 1.1e-13 exp(-6744 / T),
//     L_L = 8.18e-13 (n_H + n_H2) k_H2 (k_H, undefined in the paper, read as k_H2),
//     k_H2 = 6.29e-15 1.38 f(T) / f(4500), f(T) = sqrt(T) a e^a, a = 1 + 1 / (k_B T), k_B in eV/K;
//   Gamma_4 = 6.4e-13 erg k4 n_H2;
//   x = log10(T / 1e4); T, k1' and k4 as in chem_cell, from the state after the chemistry update;
//   the change is limited to at most half of rho eps (the explicit step of a cooling time shorter
//   than tau would drive rho eps negative).
// Bound by the FP64 pipe.  f(T) without logarithms, the quotients that stay finite by rcp_nr, the exponentials by
// exp_tang (its arguments outside +-707, where it takes the library's, are rare): post stage of a 128^3 FP64 step
// 3.05 -> 2.49 ms, with ions 4.05 -> 3.60 ms; the same worst error against the oracle (2.8e-14).
template <bool IONS>
__device__ MHD_NOINLINE double heatcool_delta(const Phys& ph, double rho, double eint, double rh2,
                                                 double rhp, double tau) {
  const double P0 = ChemConst::MH * ChemConst::KMS * ChemConst::KMS;  // erg cm^-3
  const double T0 = ChemConst::PC / ChemConst::KMS;                  // s
  const double KB_EV = 8.617333262e-5;                               // eV / K
  double nH = rho - rh2;
  if (IONS) nH = nH - rhp;
  const double nH2 = 0.5 * rh2, n = rho;
  double den3 = fma(3.0, nH, 5.0 * nH2);
  if (IONS) den3 = fma(6.0, rhp, den3);
  const double T = ((2.0 * P0) * eint) / (den3 * ChemConst::KB), iT = rcp_nr(T);
  const double x = log10(T * 1e-4);
  // k1' and k4 (App. D, as in chem_cell)
  const double t2 = T * 0.01, s2 = sqrt(t2);
  const double k1p = (3e-17 * s2) * rcp_nr(((1.0 + 0.4 * s2) + 0.2 * t2) + 0.08 * (t2 * t2));
  const double Ls = (ph.lshield > 0.0 ? ph.lshield : ph.dx) * ChemConst::PC;
  const double NH = nH * Ls, NH2 = nH2 * Ls;
  const double fdust = exp_tang(-(ph.taud * (NH + NH2)));
  const double xs = NH2 * ph.ixnorm;
  const double u = 1.0 + xs * ph.ibdop;
  const double isx = rsqrt(1.0 + xs);
  const double fsh = 0.965 * rcp_nr(u * u) + (0.035 * isx) * exp_tang(-8.5e-4 * ((1.0 + xs) * isx));
  const double k4 = (3.3 * 1.7e-11) * fsh * fdust;
  // Gamma_1
  const double ncr = exp10(4.0 - 0.416 * x - 0.327 * x * x);
  const double G1 = 7.2e-12 * (k1p * n * nH) / (1.0 + ncr / n);
  // Lambda_2
  const double LH2 = T > 1087.0 ? 3.9e-19 * exp_tang(-6118.0 * iT) : exp10(-19.24 + 0.474 * x - 1.247 * x * x);
  const double LL2 = (pow(nH2, 0.77) + 1.2 * pow(nH, 0.77)) *
                     (T > 4031.0 ? 1.38e-22 * exp_tang(-9243.0 * iT) : exp10(-22.9 - 0.553 * x - 1.148 * x * x));
  const double L2 = nH2 * LH2 / (1.0 + LH2 / LL2);
  // Lambda_3
  const double LH3 = 1.1e-13 * exp_tang(-6744.0 * iT);
  // f(T) / f(4500 K) of f = sqrt(T) a e^a, a = 1 + 1 / (k_B T)
  const double a = 1.0 + (1.0 / KB_EV) * iT, a0 = 1.0 + 1.0 / (KB_EV * 4500.0);
  const double kH2 = ((6.29e-15 * 1.38) / (6.7082039324993690892 * a0)) * (s2 * a) * exp_tang(a - a0);  // sqrt(45)
  const double LL3 = 8.18e-13 * ((nH + nH2) * kH2);
  const double L3 = nH2 * LH3 / (1.0 + LH3 / LL3);
  // Gamma_4
  const double G4 = 6.4e-13 * k4 * nH2;
  double net = (G1 + G4) - (L2 + L3);
  if (IONS && ph.ions) {
    // Gamma_5 = 1.92e-28 n; Lambda_6 = 2.18e-11 k6 n_H n_e; Lambda_7 = 4.65e-30 T^0.94 psi^beta n_e n_H+
    // with psi = exp(-0.75e-20 (N_H + N_H2)) sqrt(T) / n_e and beta = 0.74 / T^0.068 (0 where
    // n_e = 0); Lambda_8 = 5.7e-26 (T / 1e4)^0.8 n_e n_H+
    const double ne = rhp, lnT = log(T);
    const IonRates q = ion_rates(lnT);
    const double G5 = 1.92e-28 * n;
    const double L6 = 2.18e-11 * q.k6 * nH * ne;
    double L7 = 0.0;
    if (ne > 0.0) {
      const double lnpsi = (-0.75e-20 * (NH + NH2) + 0.5 * lnT) - log(ne);
      const double beta = 0.74 * exp(-0.068 * lnT);
      L7 = 4.65e-30 * exp(0.94 * lnT + beta * lnpsi) * ne * rhp;
    }
    const double L8 = 5.7e-26 * exp(0.8 * (lnT - 9.210340371976184)) * ne * rhp;  // ln 1e4
    net = (net + G5) - ((L6 + L7) + L8);
  }
  double d = (tau * T0) * net / P0;
  if (d < -0.5 * eint) d = -0.5 * eint;
  return d;
}

}  // namespace mhd
