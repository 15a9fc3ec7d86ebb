// Device-side ideal-MHD building blocks (templated on the working precision).
//
// Method (arXiv 2211.12867, Sect. 2.1): ideal MHD solved in the frame
// co-rotating with the Sun with the TVDLF scheme and the Woodward limiter.
// The limiter is the monotonised-central slope applied to the primitive
// variables in index space; a face whose reconstructed density or pressure is
// not positive falls back to the cell values; the TVDLF flux is
// F = (F_L + F_R)/2 - c_max (U_R - U_L)/2 with c_max the larger |v_n| + c_f of
// the two face states; the normal magnetic flux is zero.
#pragma once
#include "icarus_internal.h"

template <typename real> struct RT;
// FP64 mode: an FP64-pipe instruction of a warp takes 71 to 83 cycles of its
// scheduler (measured; 16 to 20 of the SM), an integer one 1 to 2, so the number
// of FP64-pipe instructions is the time of every FP64 kernel, and comparisons,
// minima and sign tests (each a DSETP, 80 cycles) go through the bit patterns.
// Reciprocal and square root: the hardware approximation (20 bits) and one
// step of third order, 1 + e + e^2 and 1 + e/2 + 3 e^2/8 with e the residual
// (Householder's iteration; the error e^3 is below 2^-56).  Over 4 M arguments
// of 2^-900 .. 2^900 both are within 1 ulp of the correctly rounded functions
// (the reciprocal differs in 0.03 % of them, the root in 12 %), at 3 and 5
// FP64-pipe instructions instead of 5 and 8.  1/0, 1/inf and sqrt(inf) are NaN
// (a step of a state with zero density or an infinite value ends as non-physical
// in IEEE arithmetic as well), the root of zero and of subnormal numbers is zero.
template <> struct RT<double> {
  static __device__ __forceinline__ double sqrt_(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double g = x * y, e = fma(-g, y, 1.0);
    const double r = fma(g * e, fma(e, 0.375, 0.5), g);
    // zero and subnormals, where the approximation is infinite
    return (__double2hiint(x) & 0x7fffffff) < 0x00100000 ? 0.0 : r;
  }
  static __device__ __forceinline__ double abs_(double x) { return fabs(x); }
  // minimum and maximum of numbers that are not negative
  static __device__ __forceinline__ double min_(double a, double b) {
    return __double_as_longlong(a) < __double_as_longlong(b) ? a : b;
  }
  static __device__ __forceinline__ double max_(double a, double b) {
    return __double_as_longlong(a) > __double_as_longlong(b) ? a : b;
  }
  static __device__ __forceinline__ double rcp_(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
  }
  // the same with IEEE's 1/0, 1/inf and sqrt(inf)
  static __device__ __forceinline__ double sqrt_inf_(double x) {
    return __double2hiint(x) == 0x7ff00000 ? x : sqrt_(x);
  }
  static __device__ __forceinline__ double rcp_inf_(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));   // infinite or zero: the result
    return ((unsigned)__double2hiint(y) & 0x7fffffffu) - 0x00100000u < 0x7fe00000u ? rcp_(x) : y;
  }
  // x > 0; not for NaN
  static __device__ __forceinline__ bool pos_(double x) {
    return (unsigned long long)(__double_as_longlong(x) - 1) < 0x7ff0000000000000ull;
  }
  // (magnitudes from the high words: a mask over all 64 bits is compiled to a
  // floating-point absolute value, which is an FP64-pipe addition)
  static __device__ __forceinline__ bool nan_(double x) {
    const unsigned h = (unsigned)__double2hiint(x) << 1;
    return h > 0xffe00000u || (h == 0xffe00000u && __double2loint(x) != 0);
  }
  // a < b; not for NaN (-0 counts as below +0)
  static __device__ __forceinline__ bool less_(double a, double b) {
    const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    const long long m = 0x7fffffffffffffffll;
    return (x ^ ((x >> 63) & m)) < (y ^ ((y >> 63) & m)) && !nan_(a) && !nan_(b);
  }
};
// FP32 mode: reciprocal and square root are the hardware approximations
// (PTX rcp.approx / sqrt.approx, relative error within about 1 ulp); the
// FP32 stencil is an approximation of the FP64 one at the 1e-6 level anyway
// and the correctly rounded forms cost several dependent instructions each.
template <> struct RT<float> {
  static __device__ __forceinline__ float sqrt_(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
  }
  static __device__ __forceinline__ float abs_(float x) { return fabsf(x); }
  static __device__ __forceinline__ float min_(float a, float b) { return fminf(a, b); }
  static __device__ __forceinline__ float max_(float a, float b) { return fmaxf(a, b); }
  static __device__ __forceinline__ float rcp_(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
  }
  static __device__ __forceinline__ bool pos_(float x) { return x > 0.f; }
  static __device__ __forceinline__ bool nan_(float x) { return !(x == x); }
  static __device__ __forceinline__ bool less_(float a, float b) { return a < b; }
};

// Exact conversion to FP64.  From FP32 by integer operations for zero and
// normal numbers: the conversion instruction runs at the FP64 pipe's rate (19
// cycles of an SM per warp).
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) {
  const unsigned b = __float_as_uint(x), e = (b >> 23) & 255u;
  if (e - 1u < 254u) return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
  if ((b << 1) == 0u) return __hiloint2double((int)b, 0);
  return (double)x;
}

// ---- the padded state ----
// A slot holds its cells' eight variables side by side, [cell][8] (32 bytes in
// FP32, one DRAM sector; 64 in FP64), and behind them, when the CME tracer is
// stored, one value per cell.  A cell is one 256-bit access in FP32 and two in
// FP64 wherever it lies, so the scattered reads of the ghost fills (7 cells per
// prolonged group) take one sector each instead of eight, and a stage kernel
// copies a cell with 16-byte asynchronous copies instead of 4-byte ones.
__device__ __forceinline__ size_t slot_base(const KParams &kp, int slot) {
  return (size_t)slot * kp.nvs * kp.pcells;
}
__device__ __forceinline__ int pad_cell(const KParams &kp, int p0, int p1, int p2) {
  return (p0 * kp.P[1] + p1) * kp.P[2] + p2;
}
// index of variable 0 of a cell; of its tracer
__device__ __forceinline__ size_t cell_index(const KParams &kp, int slot, int p0, int p1, int p2) {
  return slot_base(kp, slot) + (size_t)NVAR * pad_cell(kp, p0, p1, p2);
}
__device__ __forceinline__ size_t tracer_index(const KParams &kp, int slot, int p0, int p1, int p2) {
  return slot_base(kp, slot) + (size_t)NVAR * kp.pcells + pad_cell(kp, p0, p1, p2);
}
__device__ __forceinline__ void ld_cell(const float *p, float *u) {
  asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(u[0]), "=f"(u[1]), "=f"(u[2]), "=f"(u[3]), "=f"(u[4]), "=f"(u[5]), "=f"(u[6]), "=f"(u[7])
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ void ld_cell(const double *p, double *u) {
#pragma unroll
  for (int h = 0; h < NVAR; h += 4)
    asm volatile("ld.global.v4.f64 {%0,%1,%2,%3}, [%4];"
                 : "=d"(u[h]), "=d"(u[h + 1]), "=d"(u[h + 2]), "=d"(u[h + 3])
                 : "l"(p + h)
                 : "memory");
}
__device__ __forceinline__ void st_cell(float *p, const float *u) {
  asm volatile("st.global.v8.f32 [%8], {%0,%1,%2,%3,%4,%5,%6,%7};" ::"f"(u[0]), "f"(u[1]), "f"(u[2]), "f"(u[3]),
               "f"(u[4]), "f"(u[5]), "f"(u[6]), "f"(u[7]), "l"(p)
               : "memory");
}
__device__ __forceinline__ void st_cell(double *p, const double *u) {
#pragma unroll
  for (int h = 0; h < NVAR; h += 4)
    asm volatile("st.global.v4.f64 [%4], {%0,%1,%2,%3};" ::"d"(u[h]), "d"(u[h + 1]), "d"(u[h + 2]), "d"(u[h + 3]),
                 "l"(p + h)
                 : "memory");
}

// a cell's sector(s) into L2
__device__ __forceinline__ void prefetch_cell(const float *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ void prefetch_cell(const double *p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p + 4));
}

// Pressure from conserved variables.  In the mixed-precision mode the FP32
// result is replaced by an FP64 recomputation from the same (FP32-stored)
// conserved variables where the thermal energy is a small remainder of the
// total: p < pe * e or plasma beta = p / (B^2/2) < beta (settable; the
// library's defaults are pe = 0.002 and beta = 0.1).
struct Isl {
  float pe, beta;
};

template <typename real>
__device__ __forceinline__ real pressure_of(const real *u, real gamma, Isl) {
  real ir = RT<real>::rcp_(u[0]);
  real msq = u[1] * u[1] + u[2] * u[2] + u[3] * u[3];
  real me = real(0.5) * (u[5] * u[5] + u[6] * u[6] + u[7] * u[7]);
  real p = (gamma - real(1)) * (u[4] - real(0.5) * msq * ir - me);
  return p;
}

// FP64 pressure from FP32-stored variables.  The product of two floats is
// exact in double, so m.m and B.B carry no rounding beyond the double sums;
// 1/rho starts from the float reciprocal and one Newton step in double brings
// it to double accuracy (no FP64 division).
__device__ __forceinline__ float pressure_fp64_island(const float *u, float gamma) {
  const double r = u[0];
  double ri = (double)__frcp_rn(u[0]);
  ri = fma(ri, fma(-r, ri, 1.0), ri);
  const double m1 = u[1], m2 = u[2], m3 = u[3], b1 = u[5], b2 = u[6], b3 = u[7];
  const double ms = fma(m1, m1, fma(m2, m2, m3 * m3));
  const double bs = fma(b1, b1, fma(b2, b2, b3 * b3));
  const double h = fma(-0.5, bs, (double)u[4]);
  return (float)(((double)gamma - 1.0) * fma(-0.5 * ms, ri, h));
}

// float pressure without the island (accurate to ~1e-6 e; 1/rho is the
// approximate reciprocal, relative error below 2^-22, so the kinetic energy
// is off by at most ~3e-7 of e)
__device__ __forceinline__ float pressure_fp32(const float *u, float gamma) {
  const float ir = RT<float>::rcp_(u[0]);
  float msq = u[1] * u[1] + u[2] * u[2] + u[3] * u[3];
  float me = 0.5f * (u[5] * u[5] + u[6] * u[6] + u[7] * u[7]);
  return (gamma - 1.0f) * (u[4] - 0.5f * msq * ir - me);
}

template <>
__device__ __forceinline__ float pressure_of<float>(const float *u, float gamma, Isl isl) {
  float p = pressure_fp32(u, gamma);
  const float me = 0.5f * (u[5] * u[5] + u[6] * u[6] + u[7] * u[7]);
  if (p < isl.pe * u[4] || p < isl.beta * me) p = pressure_fp64_island(u, gamma);
  return p;
}

// pressure for the CFL wave speed: the float value suffices (relative error
// ~1e-6 e / p on a time-step bound taken with a 0.8 safety factor)
template <typename real>
__device__ __forceinline__ real pressure_for_speed(const real *u, real gamma) {
  return pressure_of<real>(u, gamma, Isl{0.f, 0.f});
}
template <>
__device__ __forceinline__ float pressure_for_speed<float>(const float *u, float gamma) {
  return pressure_fp32(u, gamma);
}

// U -> W with the pressure floor of the stage operator.
template <typename real>
__device__ __forceinline__ void cons2prim(const real *u, real *w, real gamma, real pfloor, Isl isl) {
  real ir = RT<real>::rcp_(u[0]);
  w[0] = u[0];
  w[1] = u[1] * ir;
  w[2] = u[2] * ir;
  w[3] = u[3] * ir;
  real p = pressure_of<real>(u, gamma, isl);
  w[4] = RT<real>::less_(p, pfloor) ? pfloor : p;
  w[5] = u[5];
  w[6] = u[6];
  w[7] = u[7];
}
// FP64: the two energies in one chain of products (14 FP64-pipe instructions),
// the radial one, the largest in the wind, last: only it then rounds at the size
// of the sum, which the pressure is the small difference to.
template <>
__device__ __forceinline__ void cons2prim<double>(const double *u, double *w, double gamma, double pfloor, Isl) {
  const double ir = RT<double>::rcp_(u[0]);
  w[0] = u[0];
  w[1] = u[1] * ir;
  w[2] = u[2] * ir;
  w[3] = u[3] * ir;
  const double t = fma(u[1], w[1], fma(u[2], w[2], fma(u[3], w[3], u[5] * u[5] + u[6] * u[6] + u[7] * u[7])));
  const double p = (gamma - 1.0) * fma(-0.5, t, u[4]);
  w[4] = RT<double>::less_(p, pfloor) ? pfloor : p;
  w[5] = u[5];
  w[6] = u[6];
  w[7] = u[7];
}

// primitives for the CFL speed (no FP64 island in the FP32 mode)
template <typename real>
__device__ __forceinline__ void cons2prim_speed(const real *u, real *w, real gamma, real pfloor) {
  real ir = RT<real>::rcp_(u[0]);
  w[0] = u[0];
  w[1] = u[1] * ir;
  w[2] = u[2] * ir;
  w[3] = u[3] * ir;
  real p = pressure_for_speed<real>(u, gamma);
  w[4] = RT<real>::less_(p, pfloor) ? pfloor : p;
  w[5] = u[5];
  w[6] = u[6];
  w[7] = u[7];
}

template <typename real>
__device__ __forceinline__ void prim2cons(const real *w, real *u, real igm1) {
  real v2 = w[1] * w[1] + w[2] * w[2] + w[3] * w[3];
  real b2 = w[5] * w[5] + w[6] * w[6] + w[7] * w[7];
  u[0] = w[0];
  u[1] = w[0] * w[1];
  u[2] = w[0] * w[2];
  u[3] = w[0] * w[3];
  u[4] = w[4] * igm1 + real(0.5) * w[0] * v2 + real(0.5) * b2;
  u[5] = w[5];
  u[6] = w[6];
  u[7] = w[7];
}

// fast magnetosonic speed along direction D
template <typename real, int D>
__device__ __forceinline__ real fast_speed(const real *w, real gamma) {
  real ir = RT<real>::rcp_(w[0]);
  real a2 = gamma * w[4] * ir;
  real b2 = (w[5] * w[5] + w[6] * w[6] + w[7] * w[7]) * ir;
  real bn2 = w[5 + D] * w[5 + D] * ir;
  real s = a2 + b2;
  real disc = s * s - real(4) * a2 * bn2;
  disc = disc < real(0) ? real(0) : disc;
  return RT<real>::sqrt_(real(0.5) * (s + RT<real>::sqrt_(disc)));
}

// Half the monotonised-central slope: min(|dm|, |dm + dp| / 4, |dp|) with the
// common sign, 0 at an extremum.  Equal, bit for bit, to 0.5 * mc_slope (the
// factors are powers of two), with two multiplications fewer.
template <typename real>
__device__ __forceinline__ real mc_half_slope(real um, real u0, real up) {
  real dm = u0 - um, dp = up - u0;
  real s = dm + dp;
  real lim = RT<real>::min_(RT<real>::min_(RT<real>::abs_(dm), RT<real>::abs_(dp)), real(0.25) * RT<real>::abs_(s));
  lim = s > real(0) ? lim : -lim;
  return dm * dp > real(0) ? lim : real(0);
}

__device__ __forceinline__ long long hilo(int hi, int lo) {
  return (long long)((unsigned long long)(unsigned)hi << 32 | (unsigned)lo);
}
// FP64: the minimum and the signs by bit patterns, the quarter by the exponent
// (three FP64-pipe instructions, the differences, instead of nine)
__device__ __forceinline__ double mc_half_of(double dm, double dp) {
  const double s = dm + dp;
  // magnitudes (see nan_ for the high words)
  const int ha = __double2hiint(dm), hb = __double2hiint(dp);
  const int qa = __double2hiint(s) & 0x7fffffff;
  const long long x = hilo(ha & 0x7fffffff, __double2loint(dm)), y = hilo(hb & 0x7fffffff, __double2loint(dp));
  const long long q = qa < 0x00300000 ? 0 : hilo(qa - 0x00200000, __double2loint(s));   // |s| / 4
  long long lim = x < y ? x : y;
  lim = q < lim ? q : lim;
  const int hl = (int)(lim >> 32) | (ha & 0x80000000);
  return (ha ^ hb) < 0 ? 0.0 : __hiloint2double(hl, (int)lim);
}
template <>
__device__ __forceinline__ double mc_half_slope<double>(double um, double u0, double up) {
  return mc_half_of(u0 - um, up - u0);
}

template <typename real>
__device__ __forceinline__ real mc_slope(real um, real u0, real up) {
  real dm = u0 - um, dp = up - u0;
  real dc = real(0.5) * (dm + dp);
  real lim = RT<real>::min_(real(2) * RT<real>::abs_(dm), real(2) * RT<real>::abs_(dp));
  lim = RT<real>::min_(lim, RT<real>::abs_(dc));
  real s = dc > real(0) ? lim : -lim;
  return dm * dp > real(0) ? s : real(0);
}

// physical flux along D from primitives (and the energy density e)
template <typename real, int D>
__device__ __forceinline__ void phys_flux(const real *w, real e, real *F) {
  real vn = w[1 + D], Bn = w[5 + D];
  real b2 = w[5] * w[5] + w[6] * w[6] + w[7] * w[7];
  real pt = w[4] + real(0.5) * b2;
  real vB = w[1] * w[5] + w[2] * w[6] + w[3] * w[7];
  real rvn = w[0] * vn;
  F[0] = rvn;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    F[1 + c] = rvn * w[1 + c] - w[5 + c] * Bn;
    F[5 + c] = vn * w[5 + c] - Bn * w[1 + c];
  }
  F[1 + D] += pt;
  F[5 + D] = real(0);
  F[4] = (e + pt) * vn - Bn * vB;
}

// Elementwise a + s * b over the 8 variables (s = +1 or -1).  FP32 mode uses
// the packed pair instructions of sm_100+ (two lanes per instruction, each
// rounded as the scalar operation would be).
template <typename real>
__device__ __forceinline__ void axpy8(const real *a, real s, const real *b, real *o) {
#pragma unroll
  for (int v = 0; v < NVAR; v++) o[v] = a[v] + s * b[v];
}
template <>
__device__ __forceinline__ void axpy8<float>(const float *a, float s, const float *b, float *o) {
  const float2 ss = make_float2(s, s);
#pragma unroll
  for (int v = 0; v < NVAR; v += 2) {
    const float2 r = __ffma2_rn(ss, make_float2(b[v], b[v + 1]), make_float2(a[v], a[v + 1]));
    o[v] = r.x;
    o[v + 1] = r.y;
  }
}

// Half MC slope from the one-sided differences dm, dp and q = (dm + dp) / 4:
// min(|dm|, |dp|) carries the product of their signs (min.xorsign.abs), so one
// maximum with zero clears an extremum; the result takes q's sign.  Four
// instructions (a scheduler issues this form in 9.4 cycles a slope in a loop
// of nothing else, sign flips of both differences in 13.7).
__device__ __forceinline__ float half_mc_signed(float dm, float dp, float q) {
  float t;
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(t) : "f"(dm), "f"(dp));
  const float m = fmaxf(fminf(t, fabsf(q)), 0.f);
  return __uint_as_float(__float_as_uint(m) | (__float_as_uint(q) & 0x80000000u));
}

// Half the monotonised-central slopes of the 8 variables at the middle of
// three cells (see mc_half_slope); the differences go in packed pairs in
// FP32 mode.
template <typename real>
__device__ __forceinline__ void mc_half_slopes8(const real *um, const real *u0, const real *up, real *out) {
#pragma unroll
  for (int v = 0; v < NVAR; v++) out[v] = mc_half_slope<real>(um[v], u0[v], up[v]);
}
template <>
__device__ __forceinline__ void mc_half_slopes8<float>(const float *um, const float *u0, const float *up,
                                                       float *out) {
#pragma unroll
  for (int v = 0; v < NVAR; v += 2) {
    const float2 c = make_float2(u0[v], u0[v + 1]);
    const float2 dm = __fadd2_rn(c, make_float2(-um[v], -um[v + 1]));
    const float2 dp = __fadd2_rn(make_float2(up[v], up[v + 1]), make_float2(-c.x, -c.y));
    const float2 sm = __fmul2_rn(make_float2(0.25f, 0.25f), __fadd2_rn(dm, dp));
    out[v] = half_mc_signed(dm.x, dp.x, sm.x);
    out[v + 1] = half_mc_signed(dm.y, dp.y, sm.y);
  }
}

// Flux balance of CH variables of a cell (FP64) with the areas over its volume:
// out[h] = rm Flo - rp Fhi + tm Ftl - tp Fth + pw (Fpl - Fph).
template <typename real, int CH>
__device__ __forceinline__ void flux_balance(const real *Fhi, const real *Flo, const real *fth, const real *ftl,
                                             const real *fph, const real *fpl, real rp, real rm, real tp, real tm,
                                             real pw, real *out) {
#pragma unroll
  for (int h = 0; h < CH; h++)
    out[h] = fma(pw, fpl[h] - fph[h], fma(-tp, fth[h], fma(tm, ftl[h], fma(-rp, Fhi[h], rm * Flo[h]))));
}
// FP32: out[h] = -((Arp Fhi - Arm Flo) + (Atp Fth - Atm Ftl) + Ap (Fph - Fpl)) iV
// from the areas, in packed pairs.
__device__ __forceinline__ void flux_balance32(const float *Fhi, const float *Flo, const float *fth, const float *ftl,
                                               const float *fph, const float *fpl, float Arp, float Arm, float Atp,
                                               float Atm, float Ap, float iV, float *out) {
  const float2 arp = make_float2(Arp, Arp), narm = make_float2(-Arm, -Arm), atp = make_float2(Atp, Atp),
               natm = make_float2(-Atm, -Atm), ap = make_float2(Ap, Ap), m1 = make_float2(-1.f, -1.f),
               niv = make_float2(-iV, -iV);
#pragma unroll
  for (int h = 0; h < 4; h += 2) {
    const float2 r = __ffma2_rn(narm, make_float2(Flo[h], Flo[h + 1]),
                                __fmul2_rn(arp, make_float2(Fhi[h], Fhi[h + 1])));
    const float2 t = __ffma2_rn(natm, make_float2(ftl[h], ftl[h + 1]),
                                __fmul2_rn(atp, make_float2(fth[h], fth[h + 1])));
    const float2 p = __ffma2_rn(m1, make_float2(fpl[h], fpl[h + 1]), make_float2(fph[h], fph[h + 1]));
    const float2 d = __ffma2_rn(ap, p, __fadd2_rn(r, t));
    const float2 o = __fmul2_rn(d, niv);
    out[h] = o.x;
    out[h + 1] = o.y;
  }
}

// Fast magnetosonic speed from 1/rho, gamma p, half gamma p, |B|^2 / 2 and the
// square bt2 of the field across the direction: the discriminant
// (a^2 + b^2)^2 - 4 a^2 b_n^2 as (a^2 - b^2)^2 + 4 a^2 b_t^2, which has no
// cancellation and no sign to test; halved, so that the root's sum needs no
// factor.
__device__ __forceinline__ double fast_speed_of(double ir, double gp, double hgp, double hb2, double bt2) {
  const double d = hgp - hb2;
  return RT<double>::sqrt_((hgp + hb2 + RT<double>::sqrt_(fma(d, d, gp * bt2))) * ir);
}

// The same from rho: sqrt(X / rho) = X / sqrt(X rho), one step of third order from
// the approximate reciprocal root (seven FP64-pipe instructions; reciprocal,
// product and root are nine).  Products below the normal range take the other
// form.
__device__ __forceinline__ double face_speed(double rho, double gp, double hgp, double hb2, double bt2) {
  const double d = hgp - hb2;
  const double X = hgp + hb2 + RT<double>::sqrt_(fma(d, d, gp * bt2)), m = X * rho;
  if (__double2hiint(m) < 0x00100000) return RT<double>::sqrt_(X * RT<double>::rcp_(rho));
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(m));
  const double e = fma(-(m * y), y, 1.0), g = X * y;
  return fma(g * e, fma(e, 0.375, 0.5), g);
}

// Sum over the directions of (|v_d| + c_f,d) / dx_d from 1/rho, the velocity,
// p and the field (ix: reciprocal widths)
__device__ __forceinline__ double cfl_rate(double ir, const double *v, double p, const double *B, double gamma,
                                           const double *ix) {
  const double gp = gamma * p, hgp = 0.5 * gp, q0 = B[0] * B[0], q1 = B[1] * B[1], q2 = B[2] * B[2];
  const double hb2 = 0.5 * (q0 + q1 + q2);
  return (fabs(v[0]) + fast_speed_of(ir, gp, hgp, hb2, q1 + q2)) * ix[0] +
         (fabs(v[1]) + fast_speed_of(ir, gp, hgp, hb2, q0 + q2)) * ix[1] +
         (fabs(v[2]) + fast_speed_of(ir, gp, hgp, hb2, q0 + q1)) * ix[2];
}

// Both sides' parts of the TVDLF flux, G_L + G_R with G = F(W) + sc U(W) and sc =
// +c_max on the left, -c_max on the right (the flux is half of it).  Per
// component with w = v_n + sc:
//   mass rho w;  momentum (rho w) v_k - B_n B_k (+ p_T along n);
//   energy e w + p_T v_n - B_n (v.B);  induction B_k w - B_n v_k (k != n).
// One chain of multiply-adds a component, the terms with w, the large ones in a
// fast wind, last: only they round at the size of the sum.  Against 80-bit
// arithmetic over 37 winds with CMEs on 12 x 16 x 32 cells, five steps, the state
// is off by 2.3e-16 of its norm (correctly rounded reciprocals and roots, sides
// added at the end: 2.7e-16).
template <int D>
__device__ __forceinline__ void sides_flux(const double *L, const double *R, double hbL, double hbR, double igm1,
                                           double cm, double *G) {
  const double vL = L[1 + D], vR = R[1 + D], bL = L[5 + D], bR = R[5 + D];
  const double wL = vL + cm, wR = vR - cm;
  const double pL = L[4] + hbL, pR = R[4] + hbR;
  const double qL = fma(L[1], L[1], fma(L[2], L[2], L[3] * L[3])), qR = fma(R[1], R[1], fma(R[2], R[2], R[3] * R[3]));
  const double eL = fma(L[4], igm1, fma(0.5 * L[0], qL, hbL)), eR = fma(R[4], igm1, fma(0.5 * R[0], qR, hbR));
  const double dL = L[1] * L[5] + L[2] * L[6] + L[3] * L[7], dR = R[1] * R[5] + R[2] * R[6] + R[3] * R[7];
  const double mL = L[0] * wL, mR = R[0] * wR;
  G[0] = fma(R[0], wR, mL);
#pragma unroll
  for (int k = 0; k < 3; k++) {
    double g = fma(-bR, R[5 + k], -(bL * L[5 + k]));
    if (k == D) g += pL + pR;
    G[1 + k] = fma(mR, R[1 + k], fma(mL, L[1 + k], g));
    if (k != D) G[5 + k] = fma(R[5 + k], wR, fma(L[5 + k], wL, fma(-bR, R[1 + k], -(bL * L[1 + k]))));
  }
  G[4] = fma(eR, wR, fma(eL, wL, fma(pR, vR, fma(pL, vL, fma(-bR, dR, -(bL * dL))))));
}

// TVDLF flux from reconstructed face states WL | WR (primitive variables),
// F = (F_L + F_R)/2 - c_max (U_R - U_L)/2, c_max the larger |v_n| + c_f of
// the two states; b, c are the two cell values the face falls back to when a
// reconstructed density or pressure is not positive.  F2 receives TWICE the
// numerical flux (the caller folds the 1/2 into its face areas); the normal
// magnetic flux is zero.
template <int D>
__device__ __forceinline__ void tvdlf_states(double *WL, double *WR, const double *b, const double *c, double gamma,
                                             double igm1, double *F2) {
  if (!RT<double>::pos_(WL[0]) || !RT<double>::pos_(WL[4]) || !RT<double>::pos_(WR[0]) || !RT<double>::pos_(WR[4])) {
#pragma unroll
    for (int v = 0; v < NVAR; v++) {
      WL[v] = b[v];
      WR[v] = c[v];
    }
  }
  constexpr int T1 = 5 + (D + 1) % 3, T2 = 5 + (D + 2) % 3;   // field across the direction
  const double tL = WL[T1] * WL[T1] + WL[T2] * WL[T2], tR = WR[T1] * WR[T1] + WR[T2] * WR[T2];
  const double hbL = 0.5 * (WL[5 + D] * WL[5 + D] + tL), hbR = 0.5 * (WR[5 + D] * WR[5 + D] + tR);
  const double hg = 0.5 * gamma;
  const double cl = RT<double>::abs_(WL[1 + D]) + face_speed(WL[0], gamma * WL[4], hg * WL[4], hbL, tL);
  const double cr = RT<double>::abs_(WR[1 + D]) + face_speed(WR[0], gamma * WR[4], hg * WR[4], hbR, tR);
  const double cm = RT<double>::max_(cl, cr);
  sides_flux<D>(WL, WR, hbL, hbR, igm1, cm, F2);
  F2[5 + D] = 0.0;
}

// FP32 TVDLF flux (twice, see tvdlf_states) with the two face states in
// the two lanes of packed pairs (lane x the left state b + hb, lane y the
// right state c - hc; hb, hc the half slopes of cells b | c): the fast speed
// and the per-side flux G = F(W) +- c_max U(W) are computed once for both
// sides with the f32x2 instructions, each lane rounded as the scalar
// operation, and the lanes are added at the end.  A face whose reconstructed
// density or pressure is not positive takes the cell values.
// D < 0: the direction is theta, or phi where `ph` is set (lanes of a warp may
// differ); the operations on a face are those of its direction's instance.
template <int D>
__device__ __forceinline__ void tvdlf_pair(const float *b, const float *c, const float *hb, const float *hc,
                                           float gamma, float igm1, float *F2, bool ph = false) {
  float2 W[NVAR];
  // the fallback multiplies the half slopes by zero: no branch
  const float m = fminf(fminf(b[0] + hb[0], c[0] - hc[0]), fminf(b[4] + hb[4], c[4] - hc[4]));
  const float on = m > 0.f ? 1.f : 0.f;
#pragma unroll
  for (int v = 0; v < NVAR; v++) W[v] = make_float2(fmaf(hb[v], on, b[v]), fmaf(-hc[v], on, c[v]));
  const float2 half = make_float2(0.5f, 0.5f);
  constexpr int N = D < 0 ? 1 : D;
  float2 vn = W[1 + N], Bn = W[5 + N];   // normal components
  if (D < 0) {
    vn = ph ? W[3] : vn;
    Bn = ph ? W[7] : Bn;
  }
  const float2 b2 = __ffma2_rn(W[7], W[7], __ffma2_rn(W[6], W[6], __fmul2_rn(W[5], W[5])));
  // fast magnetosonic speed along D of both states (as fast_speed)
  const float2 ir = make_float2(RT<float>::rcp_(W[0].x), RT<float>::rcp_(W[0].y));
  const float2 a2 = __fmul2_rn(__fmul2_rn(make_float2(gamma, gamma), W[4]), ir);
  const float2 bt2 = __fmul2_rn(b2, ir);
  const float2 bn2 = __fmul2_rn(__fmul2_rn(Bn, Bn), ir);
  const float2 sum = __fadd2_rn(a2, bt2);
  float2 disc = __ffma2_rn(sum, sum, __fmul2_rn(__fmul2_rn(make_float2(-4.f, -4.f), a2), bn2));
  disc.x = fmaxf(disc.x, 0.f);
  disc.y = fmaxf(disc.y, 0.f);
  const float2 cf2 =
      __fmul2_rn(half, __fadd2_rn(sum, make_float2(RT<float>::sqrt_(disc.x), RT<float>::sqrt_(disc.y))));
  const float cm = fmaxf(fabsf(vn.x) + RT<float>::sqrt_(cf2.x), fabsf(vn.y) + RT<float>::sqrt_(cf2.y));
  // per-side flux with w = v_n + c_max on the left, v_n - c_max on the right
  const float2 nBn = __fmul2_rn(Bn, make_float2(-1.f, -1.f));
  const float2 w = __fadd2_rn(vn, make_float2(cm, -cm));
  const float2 m1 = __fmul2_rn(W[0], W[1]), m2 = __fmul2_rn(W[0], W[2]), m3 = __fmul2_rn(W[0], W[3]);
  const float2 rv2 = __ffma2_rn(m3, W[3], __ffma2_rn(m2, W[2], __fmul2_rn(m1, W[1])));
  const float2 pt = __ffma2_rn(half, b2, W[4]);
  const float2 en = __ffma2_rn(W[4], make_float2(igm1, igm1), __fmul2_rn(half, __fadd2_rn(rv2, b2)));
  const float2 vB = __ffma2_rn(W[3], W[7], __ffma2_rn(W[2], W[6], __fmul2_rn(W[1], W[5])));
  float2 G[NVAR];
  G[0] = __fmul2_rn(W[0], w);
  G[1] = __ffma2_rn(m1, w, __fmul2_rn(nBn, W[5]));
  G[2] = __ffma2_rn(m2, w, __fmul2_rn(nBn, W[6]));
  G[3] = __ffma2_rn(m3, w, __fmul2_rn(nBn, W[7]));
  if (D < 0) {
    const float2 gt = __fadd2_rn(G[2], pt), gp = __fadd2_rn(G[3], pt);
    G[2] = ph ? G[2] : gt;
    G[3] = ph ? gp : G[3];
  } else {
    G[1 + N] = __fadd2_rn(G[1 + N], pt);
  }
  G[4] = __ffma2_rn(en, w, __ffma2_rn(pt, vn, __fmul2_rn(nBn, vB)));
#pragma unroll
  for (int k = 0; k < 3; k++)
    if (k != D) G[5 + k] = __ffma2_rn(W[5 + k], w, __fmul2_rn(nBn, W[1 + k]));
#pragma unroll
  for (int v = 0; v < NVAR; v++) F2[v] = D >= 0 && v == 5 + D ? 0.f : G[v].x + G[v].y;
  if (D < 0) {
    F2[6] = ph ? F2[6] : 0.f;
    F2[7] = ph ? 0.f : F2[7];
  }
}

// TVDLF face flux (twice, see tvdlf_states) from the four cells a, b | c, e
// around the face (primitive variables).  FP32: the difference c - b serves
// both half slopes, then tvdlf_pair.
template <typename real, int D>
__device__ __forceinline__ void tvdlf_face(const real *a, const real *b, const real *c, const real *e,
                                           real gamma, real igm1, real *F2, bool ph = false) {
  if constexpr (sizeof(real) == 4) {
    float hb[NVAR], hc[NVAR];
#pragma unroll
    for (int v = 0; v < NVAR; v += 2) {
      const float2 B = make_float2(b[v], b[v + 1]), C = make_float2(c[v], c[v + 1]);
      const float2 d1 = __fadd2_rn(B, make_float2(-a[v], -a[v + 1]));
      const float2 d2 = __fadd2_rn(C, make_float2(-B.x, -B.y));
      const float2 d3 = __fadd2_rn(make_float2(e[v], e[v + 1]), make_float2(-C.x, -C.y));
      const float2 quarter = make_float2(0.25f, 0.25f);
      const float2 s1 = __fmul2_rn(quarter, __fadd2_rn(d1, d2)), s2 = __fmul2_rn(quarter, __fadd2_rn(d2, d3));
      hb[v] = half_mc_signed(d1.x, d2.x, s1.x);
      hb[v + 1] = half_mc_signed(d1.y, d2.y, s1.y);
      hc[v] = half_mc_signed(d2.x, d3.x, s2.x);
      hc[v + 1] = half_mc_signed(d2.y, d3.y, s2.y);
    }
    tvdlf_pair<D>(b, c, hb, hc, gamma, igm1, F2, ph);
    return;
  }
  if constexpr (sizeof(real) == 8) {
    static_assert(D >= 0);
    real sb[NVAR], sc[NVAR], WL[NVAR], WR[NVAR];
    mc_half_slopes8<real>(a, b, c, sb);
    mc_half_slopes8<real>(b, c, e, sc);
    axpy8<real>(b, real(1), sb, WL);
    axpy8<real>(c, real(-1), sc, WR);
    tvdlf_states<D>(WL, WR, b, c, gamma, igm1, F2);
  }
}

// asynchronous global -> shared copies of 8 or 16 bytes (cp.async)
template <int BYTES>
__device__ __forceinline__ void cp_async(void *smem, const void *gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  if (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
  else if (BYTES == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem) : "memory");
}
// wait until at most N of this thread's most recent copy groups are pending
template <int N>
__device__ __forceinline__ void cp_async_wait_group() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// floors on a freshly updated cell; returns the number of floor hits
template <typename real>
__device__ __forceinline__ int apply_floors(real *u, real gamma, real pfloor, real rfloor, Isl isl) {
  int hits = 0;
  if (RT<real>::less_(u[0], rfloor)) {
    u[0] = rfloor;
    hits++;
  }
  // the plain-precision pressure is within ~1e-6 |e| of the exact one: only a
  // cell that might be below the floor pays for the precise recovery
  const real pq = pressure_for_speed<real>(u, gamma);
  const real margin = sizeof(real) == 4 ? real(1e-6) : real(0);
  if (pq > pfloor + margin * RT<real>::abs_(u[4])) return hits;
  real p = pressure_of<real>(u, gamma, isl);
  if (RT<real>::less_(p, pfloor)) {
    real ke = real(0.5) * (u[1] * u[1] + u[2] * u[2] + u[3] * u[3]) / u[0];
    real me = real(0.5) * (u[5] * u[5] + u[6] * u[6] + u[7] * u[7]);
    u[4] = pfloor / (gamma - real(1)) + ke + me;
    hits++;
  }
  return hits;
}

// The eight children of coarse cell Ic (global at level Lc) from its value and
// MC slopes, handed to store(child, variables); if any child's density or
// pressure is not positive all eight take the parent's value.  A first pass
// checks, a second one stores (the CME tracer follows the MHD variables).
template <typename real, typename Store>
__device__ __forceinline__ void prolong_children(const KParams &kp, const real *up, const real (*s)[NVAR + 1], int Lc,
                                                 const int *Ic, Store store) {
  const int nv = kp.nvs;
  const real *d0 = GeoSel<real>::dlt(kp.geo, Lc, 0), *d1 = GeoSel<real>::dlt(kp.geo, Lc, 1),
             *d2 = GeoSel<real>::dlt(kp.geo, Lc, 2);
  const real gamma = (real)kp.gamma;
  const real a0 = d0[2 * Ic[0]], a1 = d0[2 * Ic[0] + 1], b0 = d1[2 * Ic[1]], b1 = d1[2 * Ic[1] + 1],
             e0 = d2[2 * Ic[2]], e1 = d2[2 * Ic[2] + 1];
  bool ok = true;
  for (int c = 0; c < 8; c++) {
    const real a = (c & 4) ? a1 : a0, b = (c & 2) ? b1 : b0, e = (c & 1) ? e1 : e0;
    real u[NVAR];
#pragma unroll
    for (int v = 0; v < NVAR; v++) u[v] = ((up[v] + s[0][v] * a) + s[1][v] * b) + s[2][v] * e;
    if (!(u[0] > real(0)) || !(pressure_of<real>(u, gamma, Isl{(float)kp.isl_pe, (float)kp.isl_beta}) > real(0))) ok = false;
  }
  for (int c = 0; c < 8; c++) {
    const real a = (c & 4) ? a1 : a0, b = (c & 2) ? b1 : b0, e = (c & 1) ? e1 : e0;
    real u[NVAR + 1];
#pragma unroll
    for (int v = 0; v < NVAR + 1; v++)
      if (v < nv) u[v] = ok ? ((up[v] + s[0][v] * a) + s[1][v] * b) + s[2][v] * e : up[v];
    store(c, u);
  }
}

// atomic max of a non-negative double through its bit pattern
__device__ __forceinline__ void atomic_max_pos(unsigned long long *addr, double v) {
  atomicMax(addr, (unsigned long long)__double_as_longlong(v));
}
