// State transfer, refinement estimator, regrid data movement, probe and
// conservation sums.
//
// Refinement estimator (arXiv 2211.12867, Sect. 3: refinement is triggered by
// criteria on the local solution; blocks coarsen again when the criterion
// fails): Loehner's second-derivative estimator of density and pressure in
// its diagonal index-space form, gated by a radial speed above the relaxed
// background.  It is evaluated in FP64 with explicitly rounded operations in a
// fixed order (no contraction), so the block flags agree bit for bit with any
// IEEE FP64 evaluation of the same formula on the same stored state.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "mhd_device.cuh"

namespace cg = cooperative_groups;

namespace {

// variable v of a cell
template <typename real>
__device__ __forceinline__ size_t cidx(const KParams &kp, int slot, int v, int p0, int p1, int p2) {
  return v < NVAR ? cell_index(kp, slot, p0, p1, p2) + v : tracer_index(kp, slot, p0, p1, p2);
}

// the host's [slot][variable][i][j][k] in FP64 from and to the padded cells: a
// thread takes a cell, so its side of the state is one access and a warp's
// sides of the host array are eight runs of consecutive values
template <typename real>
__global__ void k_pack(const KParams kp, const real *U, int slot0, int nslots, double *out) {
  const size_t n = (size_t)nslots * kp.icells;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const int s = (int)(e / kp.icells), c = (int)(e - (size_t)s * kp.icells);
    const int k = c % kp.nb[2], j = (c / kp.nb[2]) % kp.nb[1], i = c / (kp.nb[2] * kp.nb[1]);
    real u[NVAR];
    ld_cell(U + cell_index(kp, slot0 + s, i + NGH, j + NGH, k + NGH), u);
#pragma unroll
    for (int v = 0; v < NVAR; v++) out[((size_t)s * NVAR + v) * kp.icells + c] = (double)u[v];
  }
}

template <typename real, bool PRIM>
__global__ void __launch_bounds__(256) k_unpack(const KParams kp, real *U, int slot0, int nslots, const double *in) {
  const size_t n = (size_t)nslots * kp.icells;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const int s = (int)(e / kp.icells), c = (int)(e - (size_t)s * kp.icells);
    double u[NVAR];
    if constexpr (PRIM) {
      double x[NVAR];
#pragma unroll
      for (int v = 0; v < NVAR; v++) x[v] = in[((size_t)s * NVAR + v) * kp.icells + c];
      prim2cons<double>(x, u, 1.0 / (kp.gamma - 1.0));
    } else {
#pragma unroll
      for (int v = 0; v < NVAR; v++) u[v] = in[((size_t)s * NVAR + v) * kp.icells + c];
    }
    const int k = c % kp.nb[2], j = (c / kp.nb[2]) % kp.nb[1], i = c / (kp.nb[2] * kp.nb[1]);
    real o[NVAR];
#pragma unroll
    for (int v = 0; v < NVAR; v++) o[v] = (real)u[v];
    st_cell(U + cell_index(kp, slot0 + s, i + NGH, j + NGH, k + NGH), o);
  }
}

// the tracer between the host's [slot][i][j][k] in FP64 and the padded planes
template <typename real>
__global__ void k_pack_tracer(const KParams kp, const real *U, int slot0, int nslots, double *out) {
  const size_t n = (size_t)nslots * kp.icells;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const int s = (int)(e / kp.icells), c = (int)(e - (size_t)s * kp.icells);
    const int k = c % kp.nb[2], j = (c / kp.nb[2]) % kp.nb[1], i = c / (kp.nb[2] * kp.nb[1]);
    out[e] = (double)U[tracer_index(kp, slot0 + s, i + NGH, j + NGH, k + NGH)];
  }
}
template <typename real>
__global__ void k_unpack_tracer(const KParams kp, real *U, int slot0, int nslots, const double *in) {
  const size_t n = (size_t)nslots * kp.icells;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const int s = (int)(e / kp.icells), c = (int)(e - (size_t)s * kp.icells);
    const int k = c % kp.nb[2], j = (c / kp.nb[2]) % kp.nb[1], i = c / (kp.nb[2] * kp.nb[1]);
    U[tracer_index(kp, slot0 + s, i + NGH, j + NGH, k + NGH)] = (real)in[e];
  }
}

// Padded planes [slot][variable][cell] (a checkpoint's order) from and to the
// cells; blockIdx.x is a leaf.  Bound by memory, and the copy over the link that
// goes with it takes ten times as long.
template <typename real, bool OUT>
__global__ void __launch_bounds__(256) k_planes(const KParams kp, real *U, int slot0, real *planes) {
  real *cells = U + slot_base(kp, slot0 + blockIdx.x), *p = planes + slot_base(kp, blockIdx.x);
  const size_t n = kp.pcells;
  for (size_t c = (size_t)blockIdx.y * blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.y * blockDim.x) {
    real u[NVAR];
    if (OUT) ld_cell(cells + NVAR * c, u);
#pragma unroll
    for (int v = 0; v < NVAR; v++) {
      if (OUT) p[v * n + c] = u[v];
      else u[v] = p[v * n + c];
    }
    if (!OUT) st_cell(cells + NVAR * c, u);
    if (kp.nvs > NVAR) {   // the tracer's plane is one in both
      if (OUT) p[NVAR * n + c] = cells[NVAR * n + c];
      else cells[NVAR * n + c] = p[NVAR * n + c];
    }
  }
}

// ---- estimator ----
__device__ __forceinline__ double est_pressure(const double *u, double gamma) {
  double msq = __dadd_rn(__dadd_rn(__dmul_rn(u[1], u[1]), __dmul_rn(u[2], u[2])), __dmul_rn(u[3], u[3]));
  double bsq = __dadd_rn(__dadd_rn(__dmul_rn(u[5], u[5]), __dmul_rn(u[6], u[6])), __dmul_rn(u[7], u[7]));
  double ke = __ddiv_rn(__dmul_rn(0.5, msq), u[0]);
  double me = __dmul_rn(0.5, bsq);
  return __dmul_rn(__dsub_rn(gamma, 1.0), __dsub_rn(__dsub_rn(u[4], ke), me));
}

__device__ __forceinline__ double loehner(const double *um, double u0, const double *up, double eps) {
  double num = 0.0, den = 0.0;
  for (int d = 0; d < 3; d++) {
    double t1 = __dsub_rn(up[d], u0);
    double t2 = __dsub_rn(u0, um[d]);
    double d2 = __dsub_rn(t1, t2);
    double w = __dadd_rn(__dadd_rn(fabs(up[d]), __dmul_rn(2.0, fabs(u0))), fabs(um[d]));
    double s = __dadd_rn(__dadd_rn(fabs(t1), fabs(t2)), __dmul_rn(eps, w));
    num = __dadd_rn(num, __dmul_rn(d2, d2));
    den = __dadd_rn(den, __dmul_rn(s, s));
  }
  if (den <= 0.0) return 0.0;
  return __dsqrt_rn(__ddiv_rn(num, den));
}

// E of a cell, every operation rounded on its own
template <typename real>
__device__ __forceinline__ double exact_E(const KParams &kp, const real *U, int slot, int p0, int p1, int p2, double eps) {
  auto get = [&](int a, int b, int c, double *u) {
    real x[NVAR];
    ld_cell(U + cell_index(kp, slot, a, b, c), x);
#pragma unroll
    for (int v = 0; v < NVAR; v++) u[v] = widen(x[v]);
  };
  double u0[NVAR], rm[3], rp[3], pm[3], pp[3];
  get(p0, p1, p2, u0);
#pragma unroll
  for (int d = 0; d < 3; d++) {
    double um[NVAR], up[NVAR];
    get(p0 - (d == 0), p1 - (d == 1), p2 - (d == 2), um);
    get(p0 + (d == 0), p1 + (d == 1), p2 + (d == 2), up);
    rm[d] = um[0];
    rp[d] = up[0];
    pm[d] = est_pressure(um, kp.gamma);
    pp[d] = est_pressure(up, kp.gamma);
  }
  const double er = loehner(rm, u0[0], rp, eps);
  const double ep = loehner(pm, est_pressure(u0, kp.gamma), pp, eps);
  return er > ep ? er : ep;
}

template <typename real>
__global__ void k_estimator(const KParams kp, const real *U, int slot0, double e_ref, double e_crs, double eps,
                            double dv, signed char *flags) {
  const int slot = slot0 + blockIdx.x;
  const DevBlock B = kp.blk[slot];
  const int L = B.level, sh = L - 1;
  const DevCme C = kp.cme[B.member];
  const bool has_bg = C.pad != 0;
  const size_t nbc = (size_t)kp.n_base_cells[0] * kp.n_base_cells[1] * kp.n_base_cells[2];
  const double *vbg = kp.vbg + (size_t)B.member * nbc;
  int refine = 0, keep = 0;
  // one refining cell settles the leaf's flag: the threads stop once any of
  // them has found one (s_refine), which leaves the flag unchanged
  __shared__ volatile int s_refine;
  if (threadIdx.x == 0) s_refine = 0;
  __syncthreads();
  // without a recorded background the gate is closed everywhere: no cell
  // counts and the block is flagged for coarsening
  for (int c = has_bg ? threadIdx.x : kp.icells; c < kp.icells && !s_refine; c += blockDim.x) {
    const int k = c % kp.nb[2], j = (c / kp.nb[2]) % kp.nb[1], i = c / (kp.nb[2] * kp.nb[1]);
    const int p0 = i + NGH, p1 = j + NGH, p2 = k + NGH;
    // the speed gate first: E only matters where it is open, and not at all
    // once this thread has found a refining cell (the flags are unchanged)
    real uc[NVAR];
    ld_cell(U + cell_index(kp, slot, p0, p1, p2), uc);
    const double r0 = widen(uc[0]), m0 = widen(uc[1]);
    {
      const int I = B.ix[0] * kp.nb[0] + i, J = B.ix[1] * kp.nb[1] + j, K = B.ix[2] * kp.nb[2] + k;
      const double vb = vbg[((size_t)(I >> sh) * kp.n_base_cells[1] + (J >> sh)) * kp.n_base_cells[2] + (K >> sh)];
      // The gate compares the rounded quotient m / rho.  The sign of m - g rho is
      // exact after its one rounding, and where it is not positive the rounded
      // quotient cannot exceed g either: most cells need no division.
      const double gate = __dadd_rn(vb, dv);
      if (r0 > 0.0 && !(__fma_rn(-gate, r0, m0) > 0.0)) continue;
      const double vr = __ddiv_rn(m0, r0);
      if (!(vr > gate) || refine) continue;
    }
    const double E = exact_E(kp, U, slot, p0, p1, p2, eps);
    if (E > e_ref) {
      refine = 1;
      s_refine = 1;
    }
    if (E > e_crs) keep = 1;
  }
  refine = __syncthreads_or(refine);
  keep = __syncthreads_or(keep);
  if (threadIdx.x == 0) flags[blockIdx.x] = refine ? 1 : (keep ? 0 : -1);
}

// The same flags with the leaf's planes split over the four CTAs of a cluster
// and FP32 comparisons where they decide.  The FP64 pipe bounds the estimator
// (19 cycles of an SM per instruction of a warp; 280 instructions a cell with the
// speed gate open, seven pressures with a division each among them), and one
// CTA per leaf left the leaves inside the CME to few SMs.  Here a CTA rounds
// the density and pressure of its slab and one halo cell around it to FP32 in
// shared memory (from FP32 state without the FP64 pipe) and evaluates
// E = |second differences| / |s| there with a bound on the FP32 error; a cell
// whose comparison the bound leaves open takes the exact operations.  A slab
// without an open gate is done after its gate test.  Five CTAs per SM (48
// registers, spills on the exact path only): a slab is a chain of short phases,
// and two CTAs per SM at 108 registers took 201 us for 1914 leaves of 12^3 FP32
// cells on three levels; now 124 us, one CTA per leaf 367.  808 leaves: 50 to 62
// us, before 220.
constexpr int EST_CTAS = 4;

// Pressure to within one FP32 rounding of est_pressure's.  FP64 state: FP64
// operations in another order; with a thermal energy of at least 2^-26 e the
// two, each within 7 2^-53 e, differ by 2^-23 of it at most.  FP32 state: in
// pairs of FP32 numbers (exact products and sums by fused multiply-adds,
// Dekker's and Knuth's error-free transformations), whose error is below
// 2^-42 e.  NaN, which is not decided, where the thermal energy is below
// 2^-26 e, in FP32 states the pressure below 2^-16 e or the cell out of the
// range in which no product of the pairs overflows or loses its low part.
__device__ __forceinline__ float rounded_pressure(const double *u, double gamma, float) {
  const double ke2 = (u[1] * u[1] + u[2] * u[2] + u[3] * u[3]) * RT<double>::rcp_(u[0]);
  const double th = fma(-0.5, ke2 + (u[5] * u[5] + u[6] * u[6] + u[7] * u[7]), u[4]);
  return RT<double>::less_(0x1p-26 * fabs(u[4]), th) ? (float)((gamma - 1.0) * th) : nanf("");
}
__device__ __forceinline__ void pair_add(float a, float &h, float &l) {   // (h, l) += a
  const float s = __fadd_rn(h, a), t = __fsub_rn(s, h);
  l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(s, t)), __fsub_rn(a, t)));
  h = s;
}
__device__ __forceinline__ void pair_add_square(float x, float &h, float &l) {
  const float p = __fmul_rn(x, x);
  l = __fadd_rn(l, __fmaf_rn(x, x, -p));
  pair_add(p, h, l);
}
__device__ __forceinline__ float rounded_pressure(const float *u, double, float gm1) {
  float h = 0.f, l = 0.f;
  pair_add_square(u[1], h, l);
  pair_add_square(u[2], h, l);
  pair_add_square(u[3], h, l);
  const float r = RT<float>::rcp_(u[0]), q = __fmul_rn(h, r);   // (h, l) / rho
  l = __fmul_rn(__fadd_rn(__fmaf_rn(-q, u[0], h), l), r);
  h = q;
  pair_add_square(u[5], h, l);
  pair_add_square(u[6], h, l);
  pair_add_square(u[7], h, l);
  h *= -0.5f;
  l *= -0.5f;
  pair_add(u[4], h, l);
  const float p = __fmul_rn(gm1, __fadd_rn(h, l));
  const bool in = u[4] > 1e-20f && u[4] < 1e15f && u[0] > 1e-24f && u[0] < 1e15f && u[0] * u[4] > 1e-31f;
  return in && p > 1.52587890625e-5f * u[4] ? p : nanf("");
}

// E > e from FP32 values: 1 yes, 0 no, -1 not decided.  Inputs carry a relative
// error of 2^-22 (see rounded_pressure), each difference and sum one more per
// operation: |N_f - N| and |S_f - S| stay below 2^-20 (1 + eps) of the sum of the
// w, for N the norm of the second differences and S that of s.  NaN and
// infinities are not decided, nor are sums of the w so small or large that the
// squares are not normal numbers to that accuracy.
__device__ __forceinline__ void loehner32(const float *um, float u0, const float *up, float eps, float *N, float *S,
                                          float *W) {
  float n = 0.f, d = 0.f, t = 0.f;
#pragma unroll
  for (int e = 0; e < 3; e++) {
    const float t1 = up[e] - u0, t2 = u0 - um[e], d2 = t1 - t2;
    const float w = fabsf(up[e]) + 2.f * fabsf(u0) + fabsf(um[e]);
    const float s = fabsf(t1) + fabsf(t2) + eps * w;
    n = fmaf(d2, d2, n);
    d = fmaf(s, s, d);
    t += w;
  }
  *N = sqrtf(n);
  *S = sqrtf(d);
  t *= 1.f + eps;
  *W = t > 1e-15f && t < 1e18f ? t : nanf("");
}
__device__ __forceinline__ int decide(float N, float S, float W, float e) {
  const float x = N - e * S, tol = (1.f + e) * 9.5367431640625e-7f * W;
  return x > tol ? 1 : (x < -tol ? 0 : -1);
}

template <typename real>
__global__ void __cluster_dims__(EST_CTAS, 1, 1) __launch_bounds__(256, 5)
    k_estimator_slabs(const KParams kp, const real *U, int slot0, double e_ref, double e_crs, double eps, double dv,
                      signed char *flags) {
  extern __shared__ float est_sm[];
  __shared__ int s_any, s_code[EST_CTAS];   // s_code: of the cluster's CTAs, in its first one
  __shared__ volatile int s_refine;
  // another CTA's shared memory may be written only once that CTA runs: every
  // thread arrives here and waits ahead of the write
  cg::cluster_group cl = cg::this_cluster();
  cl.barrier_arrive();
  const int part = blockIdx.x % EST_CTAS, leaf = blockIdx.x / EST_CTAS, slot = slot0 + leaf;
  const DevBlock &B = kp.blk[slot];
  const int sh = B.level - 1, tid = threadIdx.x;
  const int n1 = kp.nb[1], n2 = kp.nb[2], rows = n1 * n2, h2 = n2 + 2, H = (n1 + 2) * h2;
  const int ns = (kp.nb[0] + EST_CTAS - 1) / EST_CTAS, i0 = part * ns, i1 = min(kp.nb[0], i0 + ns);
  const size_t nbc = (size_t)kp.n_base_cells[0] * kp.n_base_cells[1] * kp.n_base_cells[2];
  const double *vbg = kp.vbg + (size_t)B.member * nbc;
  float *rho = est_sm, *pr = est_sm + (size_t)(ns + 2) * H;
  unsigned char *open = reinterpret_cast<unsigned char *>(pr + (size_t)(ns + 2) * H);
  // without a recorded background the gate is closed everywhere
  const int cells = kp.cme[B.member].pad != 0 ? max(0, i1 - i0) * rows : 0;
  int code = 0, any = 0;   // code: 1 a cell keeps the leaf, 2 one refines it
  if (tid == 0) s_any = s_refine = 0;
  __syncthreads();
  for (int c = tid; c < cells; c += blockDim.x) {
    const int i = i0 + c / rows, r = c % rows, j = r / n2, k = r - (r / n2) * n2;
    const real *u = U + cell_index(kp, slot, i + NGH, j + NGH, k + NGH);
    const double r0 = widen(u[0]), m0 = widen(u[1]);
    const int I = B.ix[0] * kp.nb[0] + i, J = B.ix[1] * n1 + j, K = B.ix[2] * n2 + k;
    const double gate = __dadd_rn(vbg[((size_t)(I >> sh) * kp.n_base_cells[1] + (J >> sh)) * kp.n_base_cells[2] + (K >> sh)], dv);
    // see k_estimator; an excess of 4 ulp of the gate leaves no doubt either
    const double x = __fma_rn(-gate, r0, m0);
    bool on = !(r0 > 0.0) || x > 0.0;
    if (on && !(r0 > 0.0 && x > 1e-15 * fabs(gate) * r0)) on = __ddiv_rn(m0, r0) > gate;
    open[c] = on;
    any |= on;
  }
  if (any) s_any = 1;
  __syncthreads();
  if (s_any) {
    const float gm1 = (float)(kp.gamma - 1.0);
    for (int c = tid; c < (i1 - i0 + 2) * H; c += blockDim.x) {
      const int a = c / H, r = c - a * H, b = r / h2, e = r - b * h2;
      // edges and corners of the halo are not read
      if ((a == 0 || a == i1 - i0 + 1) + (b == 0 || b == n1 + 1) + (e == 0 || e == n2 + 1) > 1) continue;
      real x[NVAR];
      ld_cell(U + cell_index(kp, slot, i0 + a - 1 + NGH, b - 1 + NGH, e - 1 + NGH), x);
      rho[c] = (float)x[0];
      pr[c] = rounded_pressure(x, kp.gamma, gm1);
    }
    __syncthreads();
    // one refining cell settles the leaf's flag: the CTA stops at it
    const float epsf = (float)eps, refl = (float)e_ref, crsl = (float)e_crs;
    const bool fast = eps >= 0.0 && e_ref >= 0.0 && e_crs >= 0.0;
    for (int c = tid; c < cells && !s_refine; c += blockDim.x) {
      if (!open[c]) continue;
      const int a = c / rows, r = c - a * rows, j = r / n2, k = r - j * n2;
      const int at = (a + 1) * H + (j + 1) * h2 + k + 1;
      const float rm[3] = {rho[at - H], rho[at - h2], rho[at - 1]}, rp[3] = {rho[at + H], rho[at + h2], rho[at + 1]};
      const float pm[3] = {pr[at - H], pr[at - h2], pr[at - 1]}, pp[3] = {pr[at + H], pr[at + h2], pr[at + 1]};
      float Nr, Sr, Wr, Np, Sp, Wp;
      loehner32(rm, rho[at], rp, epsf, &Nr, &Sr, &Wr);
      loehner32(pm, pr[at], pp, epsf, &Np, &Sp, &Wp);
      const int r1 = decide(Nr, Sr, Wr, refl), p1 = decide(Np, Sp, Wp, refl);
      const int r2 = decide(Nr, Sr, Wr, crsl), p2 = decide(Np, Sp, Wp, crsl);
      if (!(fast && (r1 | p1 | r2 | p2) >= 0)) {
        const double E = exact_E(kp, U, slot, i0 + a + NGH, j + NGH, k + NGH, eps);
        code |= (E > e_ref ? 2 : 0) | (E > e_crs ? 1 : 0);
      } else {
        code |= (r1 | p1) << 1 | (r2 | p2);
      }
      if (code & 2) s_refine = 1;
    }
  }
  code = (__syncthreads_or(code & 2) ? 2 : 0) | (__syncthreads_or(code & 1) ? 1 : 0);
  cl.barrier_wait();
  if (tid == 0) *cl.map_shared_rank(&s_code[part], 0) = code;
  cl.sync();
  if (part == 0 && tid == 0) {
    int all = 0;
    for (int q = 0; q < EST_CTAS; q++) all |= s_code[q];
    flags[leaf] = all & 2 ? 1 : (all & 1 ? 0 : -1);
  }
}

// ---- shock criterion (Sect. 3.2) ----
// The paper refines where the velocity divergence is negative, inside
// windows around the Sun-Earth line and the CME's hemisphere, and coarsens
// once the criterion fails.  The divergence is the central difference at cell
// centres in spherical form; everything is FP64 with explicitly rounded
// operations in a fixed order, so the flags agree bit for bit with any IEEE
// FP64 evaluation of the same expression on the same stored state and
// geometry.
__device__ __forceinline__ double wrap_pi(double a) {
  const double pi = 3.14159265358979323846, tp = 2.0 * pi;
  return __dsub_rn(a, __dmul_rn(tp, floor(__ddiv_rn(__dadd_rn(a, pi), tp))));
}

template <typename real>
__device__ __forceinline__ double vel(const KParams &kp, const real *U, int slot, int v, int p0, int p1, int p2) {
  return __ddiv_rn((double)U[cidx<real>(kp, slot, v, p0, p1, p2)], (double)U[cidx<real>(kp, slot, 0, p0, p1, p2)]);
}

// which: 0 shock (div v < -div_thr), 1 tracer (X > x_thr), 2 combined
// (either), all inside the windows.  The tracer fraction X = (rho X) / rho is
// one correctly rounded division of the stored values.
template <typename real>
__global__ void k_shock_estimator(const KParams kp, const real *U, int slot0, double div_thr, double w_le,
                                  double w_ce, double w_lc, double x_thr, int which, signed char *flags) {
  const int slot = slot0 + blockIdx.x;
  const DevBlock B = kp.blk[slot];
  const LevelGeo<double> &G = kp.geo->d[B.level];
  const DevEarth E = kp.earth[B.member];
  const DevCme C = kp.cme[B.member];
  const double t = kp.t[B.member];
  const double lon_e = __dsub_rn(E.lon0, __dmul_rn(E.rate, __dsub_rn(t, E.t0)));
  const bool sph = kp.geometry == 0;
  int refine = 0;
  // one refining cell settles the leaf's flag (see k_estimator)
  __shared__ volatile int s_refine;
  if (threadIdx.x == 0) s_refine = 0;
  __syncthreads();
  for (int c = threadIdx.x; c < kp.icells && !refine && !s_refine; c += blockDim.x) {
    const int k = c % kp.nb[2], j = (c / kp.nb[2]) % kp.nb[1], i = c / (kp.nb[2] * kp.nb[1]);
    const int I = B.ix[0] * kp.nb[0] + i + NGH, J = B.ix[1] * kp.nb[1] + j + NGH, K = B.ix[2] * kp.nb[2] + k + NGH;
    const double th = G.tc[J], ph = G.pc[K];
    bool in = true;
    if (w_le > 0.0) in = in && E.set && fabs(wrap_pi(__dsub_rn(ph, lon_e))) <= w_le;
    if (w_ce > 0.0) in = in && E.set && fabs(__dsub_rn(th, E.colat)) <= w_ce;
    if (w_lc > 0.0) in = in && C.active && fabs(wrap_pi(__dsub_rn(ph, C.lon))) <= w_lc;
    if (!in) continue;
    const int p0 = i + NGH, p1 = j + NGH, p2 = k + NGH;
    if (which >= 1 && vel(kp, U, slot, TRV, p0, p1, p2) > x_thr) {
      refine = 1;
      s_refine = 1;
      continue;
    }
    if (which == 1) continue;
    const double vrm = vel(kp, U, slot, 1, p0 - 1, p1, p2), vrp = vel(kp, U, slot, 1, p0 + 1, p1, p2);
    const double vtm = vel(kp, U, slot, 2, p0, p1 - 1, p2), vtp = vel(kp, U, slot, 2, p0, p1 + 1, p2);
    const double vpm = vel(kp, U, slot, 3, p0, p1, p2 - 1), vpp = vel(kp, U, slot, 3, p0, p1, p2 + 1);
    const double rm = G.rc[I - 1], r0 = G.rc[I], rp = G.rc[I + 1];
    const double tm = G.tc[J - 1], tp = G.tc[J + 1], qm = G.pc[K - 1], qp = G.pc[K + 1];
    double a, b, e;
    if (sph) {
      const double sm = G.sintc[J - 1], s0 = G.sintc[J], sp = G.sintc[J + 1];
      a = __ddiv_rn(__dsub_rn(__dmul_rn(__dmul_rn(rp, rp), vrp), __dmul_rn(__dmul_rn(rm, rm), vrm)),
                    __dmul_rn(__dmul_rn(r0, r0), __dsub_rn(rp, rm)));
      const double rs = __dmul_rn(r0, s0);
      b = __ddiv_rn(__dsub_rn(__dmul_rn(sp, vtp), __dmul_rn(sm, vtm)), __dmul_rn(rs, __dsub_rn(tp, tm)));
      e = __ddiv_rn(__dsub_rn(vpp, vpm), __dmul_rn(rs, __dsub_rn(qp, qm)));
    } else {
      a = __ddiv_rn(__dsub_rn(vrp, vrm), __dsub_rn(rp, rm));
      b = __ddiv_rn(__dsub_rn(vtp, vtm), __dsub_rn(tp, tm));
      e = __ddiv_rn(__dsub_rn(vpp, vpm), __dsub_rn(qp, qm));
    }
    const double div = __dadd_rn(__dadd_rn(a, b), e);
    if (div < -div_thr) {
      refine = 1;
      s_refine = 1;
    }
  }
  refine = __syncthreads_or(refine);
  if (threadIdx.x == 0) flags[blockIdx.x] = refine ? 1 : -1;
}

// ---- regrid data movement ----
// the 2 x 2 x 2 cells of the new leaf (slot dst) at padded cell (p0, p1, p2)
// from the old parent's coarse cell Ic
template <typename real>
__device__ __forceinline__ void prolong_group(const KParams &kp, const real *U, real *Unew, int cs, const int *Ic, int dst, int p0,
                              int p1, int p2) {
  const DevBlock &C = kp.blk[cs];
  const int nv = kp.nvs;   // the MHD variables and, when stored, the CME tracer
  int pc[3];
#pragma unroll
  for (int d = 0; d < 3; d++) pc[d] = Ic[d] - C.ix[d] * kp.nb[d] + NGH;
  real up[NVAR + 1], s[3][NVAR + 1];
  auto get = [&](int q0, int q1, int q2, real *u) {
    ld_cell(U + cell_index(kp, cs, q0, q1, q2), u);
    if (nv > NVAR) u[TRV] = U[tracer_index(kp, cs, q0, q1, q2)];
  };
  get(pc[0], pc[1], pc[2], up);
  {
    real um[3][NVAR + 1], uq[3][NVAR + 1];
#pragma unroll
    for (int d = 0; d < 3; d++) {
      get(pc[0] - (d == 0), pc[1] - (d == 1), pc[2] - (d == 2), um[d]);
      get(pc[0] + (d == 0), pc[1] + (d == 1), pc[2] + (d == 2), uq[d]);
    }
#pragma unroll
    for (int d = 0; d < 3; d++)
#pragma unroll
      for (int v = 0; v < NVAR + 1; v++)
        if (v < nv) s[d][v] = mc_slope<real>(um[d][v], up[v], uq[d][v]);
  }
  prolong_children<real>(kp, up, s, C.level, Ic, [&](int c, const real *u) {
    const int q0 = p0 + ((c >> 2) & 1), q1 = p1 + ((c >> 1) & 1), q2 = p2 + (c & 1);
    st_cell(Unew + cell_index(kp, dst, q0, q1, q2), u);
    if (nv > NVAR) Unew[tracer_index(kp, dst, q0, q1, q2)] = u[TRV];
  });
}

// Bound by memory: one thread per 2 x 2 x 2 group of a prolonged leaf, per four
// cells of a copied one, per cell of a restricted one.  A thread per cell, which
// for a prolongation computed the eight children of its parent and kept one,
// took (between events) 120 us for 2481 leaves of 12^3 in FP32 most of whose
// parents were refined, 84 for 2005 mostly copied ones and 66 for 218 in FP64;
// now 51, 73 and 55.
template <typename real>
__global__ void __launch_bounds__(256, sizeof(real) == 4 ? 2 : 1) k_regrid_move(const KParams kpo, const real *Uold, real *Unew, const DevBlock *nblk,
                              const MoveOp *ops) {
  const MoveOp &op = ops[blockIdx.x];
  const int kind = op.kind;
  if (kind == 0) {   // four cells a thread in flight
    const int c0 = blockIdx.y * 1024 + threadIdx.x, src = op.src[0], dst = op.dst;
    real u[4][NVAR + 1];
    size_t to[4], tt[4];
#pragma unroll
    for (int n = 0; n < 4; n++) {
      const int c = c0 + 256 * n;
      if (c >= kpo.icells) continue;
      const int k = c % kpo.nb[2], j = (c / kpo.nb[2]) % kpo.nb[1], i = c / (kpo.nb[2] * kpo.nb[1]);
      ld_cell(Uold + cell_index(kpo, src, i + NGH, j + NGH, k + NGH), u[n]);
      to[n] = cell_index(kpo, dst, i + NGH, j + NGH, k + NGH);
      if (kpo.nvs > NVAR) {
        u[n][TRV] = Uold[tracer_index(kpo, src, i + NGH, j + NGH, k + NGH)];
        tt[n] = tracer_index(kpo, dst, i + NGH, j + NGH, k + NGH);
      }
    }
#pragma unroll
    for (int n = 0; n < 4; n++) {
      if (c0 + 256 * n >= kpo.icells) continue;
      st_cell(Unew + to[n], u[n]);
      if (kpo.nvs > NVAR) Unew[tt[n]] = u[n][TRV];
    }
    return;
  }
  const int c = blockIdx.y * 256 + threadIdx.x;
  if (c >= kpo.icells) return;
  const int k = c % kpo.nb[2], j = (c / kpo.nb[2]) % kpo.nb[1], i = c / (kpo.nb[2] * kpo.nb[1]);
  const DevBlock N = nblk[op.dst];
  real val[NVAR + 1];
  const int nv = kpo.nvs;
  if (kind == 1) {
    const int g2 = kpo.nb[2] / 2, g1 = kpo.nb[1] / 2, gk = c % g2, gj = (c / g2) % g1, gi = c / (g2 * g1);
    if (gi >= kpo.nb[0] / 2) return;
    const int Ic[3] = {N.ix[0] * kpo.nb[0] / 2 + gi, N.ix[1] * kpo.nb[1] / 2 + gj, N.ix[2] * kpo.nb[2] / 2 + gk};
    prolong_group<real>(kpo, Uold, Unew, op.src[0], Ic, op.dst, 2 * gi + NGH, 2 * gj + NGH, 2 * gk + NGH);
    return;
  } else {
    const LevelGeo<real> &FG = GeoSel<real>::get(kpo.geo, N.level + 1);
    const int G[3] = {N.ix[0] * kpo.nb[0] + i, N.ix[1] * kpo.nb[1] + j, N.ix[2] * kpo.nb[2] + k};
    real sum[NVAR + 1];
#pragma unroll
    for (int v = 0; v < NVAR + 1; v++) sum[v] = real(0);
    real vs = real(0);
    for (int ch = 0; ch < 8; ch++) {
      const int f[3] = {2 * G[0] + ((ch >> 2) & 1), 2 * G[1] + ((ch >> 1) & 1), 2 * G[2] + (ch & 1)};
      int cb[3];
#pragma unroll
      for (int d = 0; d < 3; d++) cb[d] = f[d] / kpo.nb[d] - 2 * N.ix[d];
      const int os = op.src[(cb[0] << 2) | (cb[1] << 1) | cb[2]];
      const int q0 = f[0] - (2 * N.ix[0] + cb[0]) * kpo.nb[0] + NGH;
      const int q1 = f[1] - (2 * N.ix[1] + cb[1]) * kpo.nb[1] + NGH;
      const int q2 = f[2] - (2 * N.ix[2] + cb[2]) * kpo.nb[2] + NGH;
      const real V = FG.dr3[f[0] + NGH] * FG.dcos[f[1] + NGH] * FG.dphi;
      real u[NVAR + 1];
      ld_cell(Uold + cell_index(kpo, os, q0, q1, q2), u);
      if (nv > NVAR) u[TRV] = Uold[tracer_index(kpo, os, q0, q1, q2)];
#pragma unroll
      for (int v = 0; v < NVAR + 1; v++)
        if (v < nv) sum[v] += V * u[v];
      vs += V;
    }
#pragma unroll
    for (int v = 0; v < NVAR + 1; v++) val[v] = sum[v] / vs;
  }
  st_cell(Unew + cell_index(kpo, op.dst, i + NGH, j + NGH, k + NGH), val);
  if (nv > NVAR) Unew[tracer_index(kpo, op.dst, i + NGH, j + NGH, k + NGH)] = val[TRV];
}

// ---- probe ----
__device__ int find_face(const double *f, int N, double x) {
  int lo = 0, hi = N;
  while (hi - lo > 1) {
    int m = (lo + hi) / 2;
    if (f[m + NGH] <= x) lo = m;
    else hi = m;
  }
  return lo;
}

template <typename real>
__global__ void k_probe(const KParams kp, const real *U, int member, int maxL, int npts, const double *pts,
                        double *out) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= npts) return;
  double p[3] = {pts[3 * n], pts[3 * n + 1], pts[3 * n + 2]};
  if (kp.bc_lo[2] == 0) {
    const LevelGeo<double> &G1 = kp.geo->d[1];
    const double lo = G1.pf[NGH], hi = G1.pf[NGH + G1.n[2]], span = hi - lo;
    p[2] = lo + fmod(fmod(p[2] - lo, span) + span, span);
  }
  const LevelGeo<double> &GM = kp.geo->d[maxL];
  const double *faces[3] = {GM.rf, GM.tf, GM.pf};
  int I[3];
  bool bad = false;
  for (int d = 0; d < 3; d++) {
    const int N = GM.n[d];
    if (p[d] < faces[d][NGH] || p[d] >= faces[d][NGH + N]) bad = true;
    I[d] = find_face(faces[d], N, p[d]);
  }
  if (bad) {
    for (int v = 0; v < NVAR; v++) out[n * NVAR + v] = nan("");
    return;
  }
  int L = maxL, slot = -1;
  while (L >= 1) {
    const int o = (int)0;
    (void)o;
    const long long off = kp.lmap_off[member * (MAXLEV + 1) + L];
    const int s = L - 1;
    const int b0 = I[0] / kp.nb[0], b1 = I[1] / kp.nb[1], b2 = I[2] / kp.nb[2];
    const int n1 = kp.nbase[1] << s, n2 = kp.nbase[2] << s;
    const int v = kp.lmap[off + ((long long)b0 * n1 + b1) * n2 + b2];
    if (v >= 0) {
      slot = v;
      break;
    }
    for (int d = 0; d < 3; d++) I[d] >>= 1;
    L--;
  }
  if (slot < 0) {
    for (int v = 0; v < NVAR; v++) out[n * NVAR + v] = nan("");
    return;
  }
  const DevBlock B = kp.blk[slot];
  const LevelGeo<double> &G = kp.geo->d[B.level];
  const double *cen[3] = {G.rc, G.tc, G.pc};
  int q[3];
  double w[3];
  for (int d = 0; d < 3; d++) {
    const int P = kp.P[d], g0 = B.ix[d] * kp.nb[d] - NGH;
    int kk = 0;
    for (int s = 0; s < P - 1; s++)
      if (cen[d][g0 + s + NGH] <= p[d]) kk = s;
    if (kk > P - 2) kk = P - 2;
    const double c0 = cen[d][g0 + kk + NGH], c1 = cen[d][g0 + kk + 1 + NGH];
    q[d] = kk;
    w[d] = (p[d] - c0) / (c1 - c0);
  }
  double acc[NVAR];
  for (int v = 0; v < NVAR; v++) acc[v] = 0.0;
  for (int a = 0; a < 2; a++)
    for (int b = 0; b < 2; b++)
      for (int c = 0; c < 2; c++) {
        double u[NVAR];
        for (int v = 0; v < NVAR; v++) u[v] = (double)U[cidx<real>(kp, slot, v, q[0] + a, q[1] + b, q[2] + c)];
        const double ir = 1.0 / u[0];
        double W[NVAR];
        W[0] = u[0];
        W[1] = u[1] * ir;
        W[2] = u[2] * ir;
        W[3] = u[3] * ir;
        W[4] = (kp.gamma - 1.0) * (u[4] - 0.5 * u[0] * (W[1] * W[1] + W[2] * W[2] + W[3] * W[3]) -
                                   0.5 * (u[5] * u[5] + u[6] * u[6] + u[7] * u[7]));
        W[5] = u[5];
        W[6] = u[6];
        W[7] = u[7];
        const double wt = (a ? w[0] : 1.0 - w[0]) * (b ? w[1] : 1.0 - w[1]) * (c ? w[2] : 1.0 - w[2]);
        for (int v = 0; v < NVAR; v++) acc[v] += wt * W[v];
      }
  for (int v = 0; v < NVAR; v++) out[n * NVAR + v] = acc[v];
}

// ---- conservation sums: per-block partials in a fixed order ----
template <typename real>
__global__ void k_sums(const KParams kp, const real *U, int slot0, double *partial) {
  __shared__ double sh[NVAR][256];
  const int slot = slot0 + blockIdx.x;
  const DevBlock B = kp.blk[slot];
  const LevelGeo<real> &G = GeoSel<real>::get(kp.geo, B.level);
  const LevelGeo<double> &GD = kp.geo->d[B.level];
  double acc[NVAR];
  for (int v = 0; v < NVAR; v++) acc[v] = 0.0;
  (void)G;
  for (int c = threadIdx.x; c < kp.icells; c += blockDim.x) {
    const int k = c % kp.nb[2], j = (c / kp.nb[2]) % kp.nb[1], i = c / (kp.nb[2] * kp.nb[1]);
    const int I = B.ix[0] * kp.nb[0] + i + NGH, J = B.ix[1] * kp.nb[1] + j + NGH;
    const double V = GD.dr3[I] * GD.dcos[J] * GD.dphi;
    real u[NVAR];
    ld_cell(U + cell_index(kp, slot, i + NGH, j + NGH, k + NGH), u);
    for (int v = 0; v < NVAR; v++) acc[v] += V * (double)u[v];
  }
  for (int v = 0; v < NVAR; v++) sh[v][threadIdx.x] = acc[v];
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s)
      for (int v = 0; v < NVAR; v++) sh[v][threadIdx.x] += sh[v][threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x < NVAR) partial[(size_t)blockIdx.x * NVAR + threadIdx.x] = sh[threadIdx.x][0];
}

template <typename real>
__global__ void k_vbg(const KParams kp, const real *U, int member, int slot0, double *vbg) {
  const int slot = slot0 + blockIdx.x;
  const DevBlock B = kp.blk[slot];
  for (int c = blockIdx.y * blockDim.x + threadIdx.x; c < kp.icells; c += gridDim.y * blockDim.x) {
    const int k = c % kp.nb[2], j = (c / kp.nb[2]) % kp.nb[1], i = c / (kp.nb[2] * kp.nb[1]);
    const int I = B.ix[0] * kp.nb[0] + i, J = B.ix[1] * kp.nb[1] + j, K = B.ix[2] * kp.nb[2] + k;
    const double m = (double)U[cidx<real>(kp, slot, 1, i + NGH, j + NGH, k + NGH)];
    const double r = (double)U[cidx<real>(kp, slot, 0, i + NGH, j + NGH, k + NGH)];
    vbg[((size_t)I * kp.n_base_cells[1] + J) * kp.n_base_cells[2] + K] = m / r;
  }
  (void)member;
}

}  // namespace

void pack_state_launch(const KParams &kp, const void *U, int precision, int slot0, int nslots, double *out,
                       cudaStream_t s) {
  if (nslots <= 0) return;
  if (precision)
    k_pack<float><<<1024, 256, 0, s>>>(kp, (const float *)U, slot0, nslots, out);
  else
    k_pack<double><<<1024, 256, 0, s>>>(kp, (const double *)U, slot0, nslots, out);
}

void pack_tracer_launch(const KParams &kp, const void *U, int precision, int slot0, int nslots, double *out,
                        cudaStream_t s) {
  if (nslots <= 0) return;
  if (precision)
    k_pack_tracer<float><<<1024, 256, 0, s>>>(kp, (const float *)U, slot0, nslots, out);
  else
    k_pack_tracer<double><<<1024, 256, 0, s>>>(kp, (const double *)U, slot0, nslots, out);
}

void unpack_tracer_launch(const KParams &kp, void *U, int precision, int slot0, int nslots, const double *in,
                          cudaStream_t s) {
  if (nslots <= 0) return;
  if (precision)
    k_unpack_tracer<float><<<1024, 256, 0, s>>>(kp, (float *)U, slot0, nslots, in);
  else
    k_unpack_tracer<double><<<1024, 256, 0, s>>>(kp, (double *)U, slot0, nslots, in);
}

void planes_launch(const KParams &kp, void *U, int precision, int slot0, int nslots, void *planes, bool out,
                   cudaStream_t s) {
  if (nslots <= 0) return;
  const dim3 grid(nslots, (unsigned)std::min((kp.pcells + 1023) / 1024, 65535));
  auto launch = [&](auto *u, auto *p) {
    using real = std::remove_pointer_t<decltype(u)>;
    if (out) k_planes<real, true><<<grid, 256, 0, s>>>(kp, u, slot0, p);
    else k_planes<real, false><<<grid, 256, 0, s>>>(kp, u, slot0, p);
  };
  if (precision) launch((float *)U, (float *)planes);
  else launch((double *)U, (double *)planes);
}

void unpack_state_launch(const KParams &kp, void *U, int precision, int slot0, int nslots, const double *in,
                         int is_prim, cudaStream_t s) {
  if (nslots <= 0) return;
  auto launch = [&](auto *u) {
    using real = std::remove_pointer_t<decltype(u)>;
    if (is_prim) k_unpack<real, true><<<1024, 256, 0, s>>>(kp, u, slot0, nslots, in);
    else k_unpack<real, false><<<1024, 256, 0, s>>>(kp, u, slot0, nslots, in);
  };
  if (precision) launch((float *)U);
  else launch((double *)U);
}

namespace {
template <typename real>
void estimator(const KParams &kp, const real *U, int slot0, int nslots, double e_ref, double e_crs, double eps, double dv,
               signed char *flags, cudaStream_t s) {
  // four slabs of a leaf in at most 100 KB each (two CTAs per SM): 12^3 blocks
  // take 8 KB; above, one CTA per leaf without shared planes
  constexpr size_t most = 100 * 1024;
  const size_t ns = (kp.nb[0] + EST_CTAS - 1) / EST_CTAS, H = (size_t)(kp.nb[1] + 2) * (kp.nb[2] + 2);
  const size_t smem = 2 * sizeof(float) * (ns + 2) * H + ns * kp.nb[1] * kp.nb[2];
  if (smem > most) {
    k_estimator<real><<<nslots, 256, 0, s>>>(kp, U, slot0, e_ref, e_crs, eps, dv, flags);
    return;
  }
  raise_smem_limit<k_estimator_slabs<real>, most>();
  k_estimator_slabs<real><<<nslots * EST_CTAS, 256, smem, s>>>(kp, U, slot0, e_ref, e_crs, eps, dv, flags);
}
}  // namespace

void estimator_launch(const KParams &kp, const void *U, int precision, int slot0, int nslots, double e_ref,
                      double e_crs, double eps, double dv, signed char *flags, cudaStream_t s) {
  if (nslots <= 0) return;
  if (precision)
    estimator<float>(kp, (const float *)U, slot0, nslots, e_ref, e_crs, eps, dv, flags, s);
  else
    estimator<double>(kp, (const double *)U, slot0, nslots, e_ref, e_crs, eps, dv, flags, s);
}

void shock_estimator_launch(const KParams &kp, const void *U, int precision, int slot0, int nslots,
                            const double *crit, signed char *flags, cudaStream_t s) {
  if (nslots <= 0) return;
  const int which = (int)crit[5];
  if (precision)
    k_shock_estimator<float><<<nslots, 256, 0, s>>>(kp, (const float *)U, slot0, crit[0], crit[1], crit[2], crit[3],
                                                     crit[4], which, flags);
  else
    k_shock_estimator<double><<<nslots, 256, 0, s>>>(kp, (const double *)U, slot0, crit[0], crit[1], crit[2],
                                                      crit[3], crit[4], which, flags);
}

void regrid_move_launch2(const KParams &kp_old, const void *Uold, void *Unew, const DevBlock *nblk, int precision,
                         const MoveOp *ops, int nops, cudaStream_t s) {
  if (nops <= 0) return;
  dim3 grid(nops, (kp_old.icells + 255) / 256);
  if (precision)
    k_regrid_move<float><<<grid, 256, 0, s>>>(kp_old, (const float *)Uold, (float *)Unew, nblk, ops);
  else
    k_regrid_move<double><<<grid, 256, 0, s>>>(kp_old, (const double *)Uold, (double *)Unew, nblk, ops);
}

void probe_launch2(const KParams &kp, const void *U, int precision, int member, int maxL, int npts, const double *pts,
                   double *out, cudaStream_t s) {
  if (npts <= 0) return;
  if (precision)
    k_probe<float><<<(npts + 127) / 128, 128, 0, s>>>(kp, (const float *)U, member, maxL, npts, pts, out);
  else
    k_probe<double><<<(npts + 127) / 128, 128, 0, s>>>(kp, (const double *)U, member, maxL, npts, pts, out);
}

void sums_launch(const KParams &kp, const void *U, int precision, int slot0, int nslots, double *partial,
                 cudaStream_t s) {
  if (nslots <= 0) return;
  if (precision)
    k_sums<float><<<nslots, 256, 0, s>>>(kp, (const float *)U, slot0, partial);
  else
    k_sums<double><<<nslots, 256, 0, s>>>(kp, (const double *)U, slot0, partial);
}

void vbg_launch(const KParams &kp, const void *U, int precision, int member, int slot0, int nslots, double *vbg,
                cudaStream_t s) {
  if (nslots <= 0) return;
  if (precision)
    k_vbg<float><<<dim3(nslots, (kp.icells + 4095) / 4096), 256, 0, s>>>(kp, (const float *)U, member, slot0, vbg);
  else
    k_vbg<double><<<dim3(nslots, (kp.icells + 4095) / 4096), 256, 0, s>>>(kp, (const double *)U, member, slot0, vbg);
}
