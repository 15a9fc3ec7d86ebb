// Learned refinement pre-flagger: features, forward, backward and Adam.
//
// The paper refines with criteria evaluated on the solution (Sect. 3); this
// predictor anticipates the estimator's next decision.  Per block: the
// index-space gradient magnitude of density, radial speed and pressure, each
// divided by the cell's magnitude, averaged over the three variables and over
// 4 x 4 x 4 sub-cubes -> 64 inputs; MLP 64 -> 128 (ReLU) -> 128 (ReLU) -> 1
// (sigmoid); binary cross-entropy; Adam.  FP32 storage and accumulation.
//
// A training batch is two launches.  k_mlp holds both weight matrices in shared
// memory and takes groups of 8 samples through the forward pass, the backward
// pass and the outer products of the weight gradients, which stay in registers
// (96 per thread) until the CTA has done its groups; k_reduce adds the CTAs'
// partial gradients in a fixed order (the gradient is the same bits on every
// call) and takes the Adam step.  Latency bounds both (50 MFLOP and 13 MB of
// partial gradients for a batch of 1024): 15 and 7 us, beginnings and ends
// overlapping (four launches with the activations in global memory and one
// thread per parameter summing over the batch took 120 us; weights copied and
// partial gradients written word by word 25 and 8 us).
#include "mhd_device.cuh"

#define MLP_IN 64
#define MLP_H 128

namespace {

struct MlpView {
  const float *W1, *b1, *W2, *b2, *w3, *b3;
};

__host__ __device__ inline MlpView mlp_view(const float *th) {
  MlpView m;
  m.W1 = th;
  m.b1 = m.W1 + MLP_H * MLP_IN;
  m.W2 = m.b1 + MLP_H;
  m.b2 = m.W2 + MLP_H * MLP_H;
  m.w3 = m.b2 + MLP_H;
  m.b3 = m.w3 + MLP_H;
  return m;
}

// rho, v_r and p of a cell in FP64
template <typename real>
__device__ __forceinline__ void feature_prims(const KParams &kp, const real *U, int slot, int i, int j, int k, double *w) {
  real u[NVAR];
  ld_cell(U + cell_index(kp, slot, i, j, k), u);
  const double r = widen(u[0]), m1 = widen(u[1]), m2 = widen(u[2]), m3 = widen(u[3]);
  const double b1 = widen(u[5]), b2 = widen(u[6]), b3 = widen(u[7]);
  const double ir = RT<double>::rcp_inf_(r);
  w[0] = r;
  // the quotient with its remainder: equal speeds come out equal whatever the
  // densities (infinite and zero ones as they are)
  const double v = m1 * ir;
  const bool normal = ((unsigned)__double2hiint(v) & 0x7fffffffu) - 0x00100000u < 0x7fe00000u;
  w[1] = normal ? fma(fma(-v, r, m1), ir, v) : v;
  w[2] = (kp.gamma - 1.0) * fma(-0.5, (m1 * m1 + m2 * m2 + m3 * m3) * ir + (b1 * b1 + b2 * b2 + b3 * b3), widen(u[4]));
}

// Sum over the three primitives of the index-space gradient magnitude over the
// cell's magnitude: w0 the cell, d the differences of its neighbours per
// direction and primitive
__device__ __forceinline__ double feature_of(const double *w0, const double (*d)[3]) {
  double g = 0.0;
#pragma unroll
  for (int q = 0; q < 3; q++) {
    const double s = d[0][q] * d[0][q] + d[1][q] * d[1][q] + d[2][q] * d[2][q];
    g += RT<double>::sqrt_inf_(s) * RT<double>::rcp_inf_(fabs(w0[q]) + 1e-30);
  }
  return g;   // of doubled differences: the caller divides by 2 and by 3
}

// Features of 4 x 4 x 4 sub-cubes of s0 x s1 x s2 cells with s = n / 4.  One
// CTA per leaf marches along r with the primitives of three planes (and one
// halo cell around them) in shared memory, so a cell is converted 1.6 times
// (12^3 block) instead of 7.  Each column sums its cells along r, then one warp
// per sub-cube its columns in a fixed lane stride and shuffle tree: the
// features are the same bits on every run and for every member.
// FP64 states: the FP64 pipe bounds this kernel (one instruction of a warp per
// 19 cycles of an SM), with 72 such instructions a cell.
__global__ void __launch_bounds__(256) k_features(const KParams kp, const double *U, int slot0, float *out) {
  extern __shared__ double smd[];
  const int slot = slot0 + blockIdx.x;
  const int n1 = kp.nb[1], n2 = kp.nb[2], h2 = n2 + 2, H = (n1 + 2) * h2;
  const int s0 = kp.nb[0] / 4, s1 = n1 / 4, s2 = n2 / 4, per = s0 * s1 * s2;
  double *acc = smd + 9 * H;   // [ring plane][primitive][cell], then per column
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto plane = [&](int i) {   // primitives of padded plane i
    double *P = smd + (i % 3) * 3 * H;
    for (int c = threadIdx.x; c < H; c += blockDim.x) {
      double w[3];
      feature_prims(kp, U, slot, i, NGH - 1 + c / h2, NGH - 1 + c % h2, w);
      P[c] = w[0];
      P[H + c] = w[1];
      P[2 * H + c] = w[2];
    }
  };
  plane(NGH - 1);
  plane(NGH);
  for (int a = 0; a < 4; a++) {
    for (int t = threadIdx.x; t < n1 * n2; t += blockDim.x) acc[t] = 0.0;
    for (int i = NGH + a * s0; i < NGH + (a + 1) * s0; i++) {
      plane(i + 1);
      __syncthreads();
      const double *Pm = smd + ((i - 1) % 3) * 3 * H, *P = smd + (i % 3) * 3 * H, *Pp = smd + ((i + 1) % 3) * 3 * H;
      for (int t = threadIdx.x; t < n1 * n2; t += blockDim.x) {
        const int c = (t / n2 + 1) * h2 + t % n2 + 1;
        double w0[3], d[3][3];
#pragma unroll
        for (int q = 0; q < 3; q++) {
          w0[q] = P[q * H + c];
          d[0][q] = Pp[q * H + c] - Pm[q * H + c];
          d[1][q] = P[q * H + c + h2] - P[q * H + c - h2];
          d[2][q] = P[q * H + c + 1] - P[q * H + c - 1];
        }
        acc[t] += feature_of(w0, d);
      }
      __syncthreads();   // plane i - 1 is read no more
    }
    for (int sc = warp; sc < 16; sc += (int)blockDim.x >> 5) {
      const int b = sc / 4, cc = sc % 4;
      double s = 0.0;
      for (int t = lane; t < s1 * s2; t += 32) s += acc[(b * s1 + t / s2) * n2 + cc * s2 + t % s2];
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) out[(size_t)blockIdx.x * 64 + a * 16 + sc] = (float)(s / (6.0 * per));
    }
    __syncthreads();
  }
}

// Sum over a sub-cube in FP64 by one warp, every cell converting its six
// neighbours.
template <typename real>
__device__ __forceinline__ double subcube_sum(const KParams &kp, const real *U, int slot, int sc, int lane) {
  const int s0 = kp.nb[0] / 4, s1 = kp.nb[1] / 4, s2 = kp.nb[2] / 4, per = s0 * s1 * s2;
  const int a = sc / 16, b = (sc / 4) % 4, cc = sc % 4;
  double acc = 0.0;
  for (int t = lane; t < per; t += 32) {
    const int p0 = NGH + a * s0 + t / (s1 * s2), p1 = NGH + b * s1 + (t / s2) % s1, p2 = NGH + cc * s2 + t % s2;
    double w0[3], d[3][3];
    feature_prims(kp, U, slot, p0, p1, p2, w0);
#pragma unroll
    for (int e = 0; e < 3; e++) {
      double wm[3], wp[3];
      feature_prims(kp, U, slot, p0 - (e == 0), p1 - (e == 1), p2 - (e == 2), wm);
      feature_prims(kp, U, slot, p0 + (e == 0), p1 + (e == 1), p2 + (e == 2), wp);
#pragma unroll
      for (int q = 0; q < 3; q++) d[e][q] = wp[q] - wm[q];
    }
    acc += feature_of(w0, d);
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return acc;
}

// The same features where three planes do not fit in shared memory: one warp
// per sub-cube.
template <typename real>
__global__ void __launch_bounds__(256) k_features_large(const KParams kp, const real *U, int slot0, float *out) {
  const int slot = slot0 + blockIdx.x, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int per = (kp.nb[0] / 4) * (kp.nb[1] / 4) * (kp.nb[2] / 4);
  for (int sc = threadIdx.x >> 5; sc < 64; sc += nw) {
    const double acc = subcube_sum(kp, U, slot, sc, lane);
    if (lane == 0) out[(size_t)blockIdx.x * 64 + sc] = (float)(acc / (6.0 * per));
  }
}

// ---- FP32 states: the same sums in pairs of floats ----
//
// A number is h + l with |l| about half an ulp of h: 48 bits, by the
// error-free sums and products of Dekker (1971) and Knuth.  A cell takes 430
// instructions of the FP32 pipe instead of 72 of the FP64 pipe, of which each
// costs 61 times as much.  Results are rounded to FP32 (2^-24), and the pairs'
// errors stay below that (see FEAT_REL): against 80-bit arithmetic the largest
// and mean errors on winds with and without CMEs are the FP64 kernel's to ten
// digits (5.84e-8, 2.28e-8).  808 leaves of 12^3 on three levels: FP64 290 us
// (the FP64 pipe 86 % busy), pairs 67 us; features with the ghost fill and
// the copy to the host 390 -> 169 us.
__device__ __forceinline__ float2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return make_float2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t)));
}
__device__ __forceinline__ float2 renorm(float h, float l) {   // |h| >= |l|
  const float s = __fadd_rn(h, l);
  return make_float2(s, __fsub_rn(l, __fsub_rn(s, h)));
}
__device__ __forceinline__ float2 pair_add(float2 a, float2 b) {
  const float2 s = two_sum(a.x, b.x);
  return renorm(s.x, __fadd_rn(s.y, __fadd_rn(a.y, b.y)));
}
__device__ __forceinline__ float2 pair_mul(float2 a, float2 b) {   // not renormalised
  const float p = __fmul_rn(a.x, b.x);
  return make_float2(p, __fmaf_rn(a.y, b.x, __fmaf_rn(a.x, b.y, __fmaf_rn(a.x, b.x, -p))));
}
__device__ __forceinline__ float2 pair_rcp(float2 a) {
  float y;
  asm("rcp.approx.f32 %0, %1;" : "=f"(y) : "f"(a.x));
  const float e = __fmaf_rn(-a.y, y, __fmaf_rn(-a.x, y, 1.f));
  return make_float2(y, __fmul_rn(y, __fmaf_rn(e, e, e)));
}
// a^2 + b^2 + c^2 of pairs
__device__ __forceinline__ float2 pair_norm2(float2 a, float2 b, float2 c) {
  const float p = __fmul_rn(a.x, a.x), q = __fmul_rn(b.x, b.x), r = __fmul_rn(c.x, c.x);
  const float ep = __fmaf_rn(a.x + a.x, a.y, __fmaf_rn(a.x, a.x, -p));
  const float eq = __fmaf_rn(b.x + b.x, b.y, __fmaf_rn(b.x, b.x, -q));
  const float er = __fmaf_rn(c.x + c.x, c.y, __fmaf_rn(c.x, c.x, -r));
  const float2 s = two_sum(p, q), t = two_sum(s.x, r);
  return renorm(t.x, __fadd_rn(t.y, __fadd_rn(s.y, __fadd_rn(ep, __fadd_rn(eq, er)))));
}

// A cell's primitives carry relative errors of about 2^-46, the pressure
// 2^-46 E / p from the difference that it is.  Cells with p < 2^-12 E, or out
// of the range in which no product of theirs overflows or loses its low part,
// are converted in FP64.  ratio: at least E / p of the others.
__device__ __forceinline__ void pair_prims(const KParams &kp, const float *U, int slot, int i, int j, int k, float2 gm1,
                                           float2 *w, float &ratio) {
  float u[NVAR];
  ld_cell(U + cell_index(kp, slot, i, j, k), u);
  const float r = u[0], E = u[4];
  const float2 z = make_float2(0.f, 0.f);
  const float2 ir = pair_rcp(make_float2(r, 0.f));
  const float2 M = pair_norm2(make_float2(u[1], 0.f), make_float2(u[2], 0.f), make_float2(u[3], 0.f));
  const float2 B = pair_norm2(make_float2(u[5], 0.f), make_float2(u[6], 0.f), make_float2(u[7], 0.f));
  const float2 K = pair_add(pair_mul(M, ir), B);
  const float2 P = pair_add(make_float2(E, 0.f), make_float2(-0.5f * K.x, -0.5f * K.y));
  if (P.x >= 0x1p-12f * E && E > 1e-20f && E < 1e15f && r > 1e-24f && r < 1e15f && r * E > 1e-31f) {
    const float2 p = pair_mul(P, gm1);
    const float v = __fmul_rn(u[1], ir.x);   // and its remainder, as in feature_prims
    w[0] = make_float2(r, 0.f);
    w[1] = renorm(v, __fmul_rn(__fmaf_rn(-v, r, u[1]), ir.x));
    w[2] = renorm(p.x, p.y);
    ratio = fmaxf(ratio, __fdividef(E, P.x));
  } else {
    double x[3];
    feature_prims(kp, U, slot, i, j, k, x);
#pragma unroll
    for (int q = 0; q < 3; q++) {
      w[q] = z;
      w[q].x = (float)x[q];
      w[q].y = (float)(x[q] - (double)w[q].x);
    }
  }
}

// A sub-cube whose feature is below FEAT_REL E / p (its differences are within
// the pairs' last 26 bits) is done again in FP64: the feature's relative
// error is 2^-46 (E / p) / f at most, 2^-26 where the pairs are kept, a
// quarter of the final rounding.  Smooth wind has features of 1e-3 and more
// and E / p of 100 to 300.
// That is for neighbours of the cell's own size, up to twice it.  Where they are
// c times it, their errors count c times: a cell whose own term is below FEAT_REL
// c, in the pressure, whose E / p is 2^12 at most, 2^12 times that, sends its
// sub-cube to FP64 as well.
constexpr float FEAT_REL = 0x1p-20f;

// feature_of in pairs, of the cell at P[q stride] (planes before, of and behind
// it; rows of h2); the differences are taken relative to the cell first, so
// that their squares stay in range whatever the units
__device__ __forceinline__ float2 pair_feature(const float2 *Pm, const float2 *P, const float2 *Pp, int stride, int h2) {
  float2 g = make_float2(0.f, 0.f);
#pragma unroll
  for (int q = 0; q < 3; q++) {
    const float2 *C = P + q * stride;
    auto diff = [](float2 a, float2 b) { return pair_add(a, make_float2(-b.x, -b.y)); };
    const float2 p0 = Pp[q * stride], p1 = C[h2], p2 = C[1];
    const float2 d0 = diff(p0, Pm[q * stride]), d1 = diff(p1, C[-h2]), d2 = diff(p2, C[-1]);
    // the others are as large, or d tells
    auto top = [&] { return fmaxf(fmaxf(fabsf(p0.x), fabsf(p1.x)), fabsf(p2.x)); };
    const float sg = C->x < 0.f ? -1.f : 1.f;
    float2 w = make_float2(sg * C->x, sg * C->y);
    if (w.x < 1e-15f) {   // where the 1e-30 that the magnitude is raised by counts
      w = pair_add(w, make_float2(1e-30f, 0.f));
      // too small for a pair: nothing if the neighbours are equal and as small,
      // else FP64
      if (w.x < 1e-22f) {
        if (!(d0.x == 0.f && d1.x == 0.f && d2.x == 0.f && top() <= 2.f * w.x)) g.x = INFINITY;
        continue;
      }
    }
    const float2 y = pair_rcp(w);
    const float2 s = pair_norm2(pair_mul(d0, y), pair_mul(d1, y), pair_mul(d2, y));
    float f = 0.f;
    if (s.x != 0.f) {
      float t;
      asm("rsqrt.approx.f32 %0, %1;" : "=f"(t) : "f"(s.x));
      f = __fmul_rn(s.x, t);
      const float e = __fadd_rn(__fmaf_rn(-f, f, s.x), s.y);
      g = pair_add(g, make_float2(f, __fmul_rn(0.5f * t, e)));
    }
    // neighbours far above the cell that nearly agree (see FEAT_REL; densities
    // are exact): FP64
    if (q > 0) {
      const float c = top() * y.x;
      if (c > 2.f && !(f >= (q == 2 ? 4096.f * FEAT_REL : FEAT_REL) * c)) g.x = INFINITY;
    }
  }
  return g;
}

// k_features for FP32 states.  The halo cells at a plane's corners are not
// read: a 12 x 12 plane takes the 192 threads once.  A sub-cube's sum and its
// shuffles stay in pairs; the 64 divisions come at the end.
constexpr int FEAT_NT = 192;
__global__ void __launch_bounds__(FEAT_NT, 6) k_features_pairs(const KParams kp, const float *U, int slot0,
                                                               float *out) {
  extern __shared__ double smd[];
  __shared__ unsigned worst;   // bits of the leaf's largest E / p
  __shared__ float2 sums[64];
  __shared__ float feat[64];
  const int slot = slot0 + blockIdx.x;
  const int n1 = kp.nb[1], n2 = kp.nb[2], h2 = n2 + 2, H = (n1 + 2) * h2;
  const int s0 = kp.nb[0] / 4, s1 = n1 / 4, s2 = n2 / 4;
  float2 *sm = reinterpret_cast<float2 *>(smd), *acc = sm + 9 * H;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const double gd = kp.gamma - 1.0;
  const float2 gm1 = make_float2((float)gd, (float)(gd - (double)(float)gd));
  float ratio = 1.f;
  // the c-th cell of a plane and its halo: the rows of the block, then those
  // before and behind it; the halo index of column t
  const int mid = n1 * h2, cells = mid + 2 * n2;
  auto halo = [&](int c) { return c < mid ? c + h2 : (c < mid + n2 ? c - mid + 1 : c - n2 + h2 + 1); };
  auto column = [&](int t) { return (t / n2 + 1) * h2 + t % n2 + 1; };
  const int hc = halo(tid), tc = column(tid), h_row = hc / h2, h_col = hc - h_row * h2;
  auto plane = [&](int i) {   // primitives of padded plane i
    float2 *P = sm + (i % 3) * 3 * H;
    for (int c = tid; c < cells; c += FEAT_NT) {
      int h = hc, row = h_row, col = h_col;
      if (c != tid) {
        h = halo(c);
        row = h / h2;
        col = h - row * h2;
      }
      float2 w[3];
      pair_prims(kp, U, slot, i, NGH - 1 + row, NGH - 1 + col, gm1, w, ratio);
      P[h] = w[0];
      P[H + h] = w[1];
      P[2 * H + h] = w[2];
    }
  };
  if (tid == 0) worst = 0;
  plane(NGH - 1);
  plane(NGH);
  for (int a = 0; a < 4; a++) {
    for (int t = tid; t < n1 * n2; t += FEAT_NT) acc[t] = make_float2(0.f, 0.f);
    for (int i = NGH + a * s0; i < NGH + (a + 1) * s0; i++) {
      plane(i + 1);
      __syncthreads();
      const float2 *Pm = sm + ((i - 1) % 3) * 3 * H, *P = sm + (i % 3) * 3 * H, *Pp = sm + ((i + 1) % 3) * 3 * H;
      for (int t = tid; t < n1 * n2; t += FEAT_NT) {
        const int c = t == tid ? tc : column(t);
        acc[t] = pair_add(acc[t], pair_feature(Pm + c, P + c, Pp + c, H, h2));
      }
      __syncthreads();   // plane i - 1 is read no more
    }
    for (int sc = warp; sc < 16; sc += FEAT_NT / 32) {
      const int b = sc / 4, cc = sc % 4;
      float2 s = make_float2(0.f, 0.f);
      for (int t = lane; t < s1 * s2; t += 32) s = pair_add(s, acc[(b * s1 + t / s2) * n2 + cc * s2 + t % s2]);
      for (int o = 16; o > 0; o >>= 1)
        s = pair_add(s, make_float2(__shfl_xor_sync(0xffffffffu, s.x, o), __shfl_xor_sync(0xffffffffu, s.y, o)));
      if (lane == 0) sums[a * 16 + sc] = s;
    }
    if (a < 3) __syncthreads();
  }
  {
    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(ratio));
    if (lane == 0) atomicMax(&worst, m);
  }
  __syncthreads();
  const double n6 = 6.0 * (s0 * s1 * s2);
  if (tid < 64) {
    const float2 s = sums[tid];
    const float f = (float)(((double)s.x + (double)s.y) / n6);
    feat[tid] = f;
    out[(size_t)blockIdx.x * 64 + tid] = f;
  }
  __syncthreads();
  const float least = FEAT_REL * __uint_as_float(worst);
  for (int sc = warp; sc < 64; sc += FEAT_NT / 32) {
    const float f = feat[sc];
    if (f != 0.f && !(f >= least && f < 1e15f)) {   // NaN and overflow among them
      const float x = (float)(subcube_sum(kp, U, slot, sc, lane) / n6);
      if (lane == 0) out[(size_t)blockIdx.x * 64 + sc] = x;
    }
  }
}

constexpr int NT = 256;          // threads of k_mlp
constexpr int GS = 8;            // samples of a group: two quads
// row strides in shared memory: 16-byte rows, and an odd number of 16-byte
// units, so neither four columns of 32 rows nor one row of 32 columns conflict
constexpr int S1 = MLP_IN + 4, S2 = MLP_H + 4;
constexpr int NW = MLP_H * (MLP_IN + MLP_H);   // weights
constexpr int NPAR = NW + MLP_H + MLP_H + MLP_H + 1;
// A CTA's partial gradient in the order its threads hold it: the weights as
// [4 columns of a tile's row][thread][4], W2 first, then b1, b2, w3, b3, the
// loss, rounded up to 16 bytes
constexpr int PART = (NPAR + 1 + 3) / 4 * 4;
constexpr int MLP_SMEM = (MLP_H * S1 + MLP_H * S2 + GS * (MLP_IN + 3 * MLP_H) + GS * (NT / 32) + 2 * GS) * 4;

// Forward pass of the rows of X (row index list `idx` or identity), and with
// GRAD the gradient of the mean cross-entropy over the batch: every CTA's share
// of it, and of the summed cross-entropy, to part[CTA].  Per group a thread
// has one hidden unit and one quad of samples; vectors over units lie in
// shared memory as [quad][unit][4], so a weight meets four samples per load.
// The weight gradients are 8 x 8 and 8 x 4 tiles of outer products per thread.
// Programmatic dependent launch: waits until the kernel before in the stream
// has completed, and lets the next one be launched (both without effect in a
// plain launch)
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <bool GRAD>
__global__ void __launch_bounds__(NT) k_mlp(const float *theta, const float *X, const float *T, const int *idx, int B,
                                            float *y, float *part) {
  extern __shared__ __align__(16) float sm[];
  float *xs = sm, *h1s = xs + GS * MLP_IN, *d2s = h1s + GS * MLP_H, *d1s = d2s + GS * MLP_H;
  float *red = d1s + GS * MLP_H, *dzs = red + GS * (NT / 32), *W1s = dzs + 2 * GS, *W2s = W1s + MLP_H * S1;
  const MlpView m = mlp_view(theta);
  const int tid = threadIdx.x, j = tid & (MLP_H - 1), q = tid >> 7, warp = tid >> 5;
  auto gather = [&](int s0) {
    for (int e = tid; e < GS * MLP_IN; e += NT) {
      const int s = e / MLP_IN, i = e % MLP_IN;
      const int row = s0 + s < B ? (idx ? idx[s0 + s] : s0 + s) : -1;
      xs[((s >> 2) * MLP_IN + i) * 4 + (s & 3)] = row >= 0 ? X[(size_t)row * MLP_IN + i] : 0.f;
    }
  };
  // the first group's samples while the step of the batch before may still run
  // (see mlp_step_launch), then the weights that it leaves
  gather(blockIdx.x * GS);
  grid_wait();
  for (int e = 4 * tid; e < MLP_H * MLP_IN; e += 4 * NT) cp_async<16>(W1s + (e / MLP_IN) * S1 + e % MLP_IN, m.W1 + e);
  for (int e = 4 * tid; e < MLP_H * MLP_H; e += 4 * NT) cp_async<16>(W2s + (e / MLP_H) * S2 + e % MLP_H, m.W2 + e);
  cp_async_commit();
  const float b1 = m.b1[j], b2 = m.b2[j], w3 = m.w3[j], b3 = m.b3[0];
  const int tj = tid >> 4, tk = tid & 15;   // gradient tile: rows tj + 16 a, columns tk + 16 b
  float g2[8][8], g1[8][4], gb1 = 0.f, gb2 = 0.f, gw3 = 0.f, gb3 = 0.f, loss = 0.f;
  if (GRAD) {
#pragma unroll
    for (int a = 0; a < 8; a++) {
#pragma unroll
      for (int b = 0; b < 8; b++) g2[a][b] = 0.f;
#pragma unroll
      for (int b = 0; b < 4; b++) g1[a][b] = 0.f;
    }
  }
  auto quad = [](const float *v, int n, int unit, int qd) -> float4 {
    return *reinterpret_cast<const float4 *>(v + (qd * n + unit) * 4);
  };
  for (int s0 = blockIdx.x * GS; s0 < B; s0 += gridDim.x * GS) {
    if (s0 != (int)blockIdx.x * GS) {
      __syncthreads();   // the previous group's vectors
      gather(s0);
    }
    cp_async_wait_all();
    __syncthreads();
    float a0 = b1, a1 = b1, a2 = b1, a3 = b1;
    auto rows = [&](const float *W, const float *v, int n) {   // four columns of the thread's row at a time
#pragma unroll 4
      for (int i = 0; i < n; i += 4) {
        const float4 w4 = *reinterpret_cast<const float4 *>(W + i);
        const float w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int c = 0; c < 4; c++) {
          const float4 x = quad(v, n, i + c, q);
          a0 = fmaf(w[c], x.x, a0);
          a1 = fmaf(w[c], x.y, a1);
          a2 = fmaf(w[c], x.z, a2);
          a3 = fmaf(w[c], x.w, a3);
        }
      }
    };
    rows(W1s + j * S1, xs, MLP_IN);
    const float4 h1 = make_float4(fmaxf(a0, 0.f), fmaxf(a1, 0.f), fmaxf(a2, 0.f), fmaxf(a3, 0.f));
    *reinterpret_cast<float4 *>(h1s + (q * MLP_H + j) * 4) = h1;
    __syncthreads();
    a0 = a1 = a2 = a3 = b2;
    rows(W2s + j * S2, h1s, MLP_H);
    const float4 h2 = make_float4(fmaxf(a0, 0.f), fmaxf(a1, 0.f), fmaxf(a2, 0.f), fmaxf(a3, 0.f));
    float z[4] = {w3 * h2.x, w3 * h2.y, w3 * h2.z, w3 * h2.w};
#pragma unroll
    for (int s = 0; s < 4; s++) {
      for (int o = 16; o > 0; o >>= 1) z[s] += __shfl_xor_sync(0xffffffffu, z[s], o);
      if ((tid & 31) == 0) red[s * (NT / 32) + warp] = z[s];
    }
    __syncthreads();
    if (tid < GS) {
      float zz = b3, dz = 0.f;
      for (int w = 0; w < MLP_H / 32; w++) zz += red[(tid & 3) * (NT / 32) + (tid >> 2) * (MLP_H / 32) + w];
      if (s0 + tid < B) {
        const float yy = 1.f / (1.f + expf(-zz));
        if (y) y[s0 + tid] = yy;
        if (GRAD) {
          const float t = T[idx ? idx[s0 + tid] : s0 + tid];
          dz = (yy - t) / (float)B;
          const float yc = fminf(fmaxf(yy, 1e-7f), 1.f - 1e-7f);
          loss += -(t * logf(yc) + (1.f - t) * logf(1.f - yc));
          gb3 += dz;
        }
      }
      dzs[tid] = dz;
    }
    if (!GRAD) continue;
    __syncthreads();
    const float4 dz = *reinterpret_cast<const float4 *>(dzs + 4 * q);
    const float4 d2 = make_float4(h2.x > 0.f ? dz.x * w3 : 0.f, h2.y > 0.f ? dz.y * w3 : 0.f,
                                  h2.z > 0.f ? dz.z * w3 : 0.f, h2.w > 0.f ? dz.w * w3 : 0.f);
    *reinterpret_cast<float4 *>(d2s + (q * MLP_H + j) * 4) = d2;
    gb2 += (d2.x + d2.y) + (d2.z + d2.w);
    gw3 = fmaf(dz.x, h2.x, fmaf(dz.y, h2.y, fmaf(dz.z, h2.z, fmaf(dz.w, h2.w, gw3))));
    __syncthreads();
    a0 = a1 = a2 = a3 = 0.f;
#pragma unroll 8
    for (int i = 0; i < MLP_H; i++) {
      const float w = W2s[i * S2 + j];
      const float4 x = quad(d2s, MLP_H, i, q);
      a0 = fmaf(w, x.x, a0);
      a1 = fmaf(w, x.y, a1);
      a2 = fmaf(w, x.z, a2);
      a3 = fmaf(w, x.w, a3);
    }
    const float4 d1 = make_float4(h1.x > 0.f ? a0 : 0.f, h1.y > 0.f ? a1 : 0.f, h1.z > 0.f ? a2 : 0.f,
                                  h1.w > 0.f ? a3 : 0.f);
    *reinterpret_cast<float4 *>(d1s + (q * MLP_H + j) * 4) = d1;
    gb1 += (d1.x + d1.y) + (d1.z + d1.w);
    __syncthreads();
    for (int qd = 0; qd < GS / 4; qd++) {
      float4 c[8];
#pragma unroll
      for (int b = 0; b < 8; b++) c[b] = quad(h1s, MLP_H, tk + 16 * b, qd);
#pragma unroll
      for (int a = 0; a < 8; a++) {
        const float4 r = quad(d2s, MLP_H, tj + 16 * a, qd);
#pragma unroll
        for (int b = 0; b < 8; b++)
          g2[a][b] = fmaf(r.x, c[b].x, fmaf(r.y, c[b].y, fmaf(r.z, c[b].z, fmaf(r.w, c[b].w, g2[a][b]))));
      }
#pragma unroll
      for (int b = 0; b < 4; b++) c[b] = quad(xs, MLP_IN, tk + 16 * b, qd);
#pragma unroll
      for (int a = 0; a < 8; a++) {
        const float4 r = quad(d1s, MLP_H, tj + 16 * a, qd);
#pragma unroll
        for (int b = 0; b < 4; b++)
          g1[a][b] = fmaf(r.x, c[b].x, fmaf(r.y, c[b].y, fmaf(r.z, c[b].z, fmaf(r.w, c[b].w, g1[a][b]))));
      }
    }
  }
  if (GRAD) {
    grid_launch_next();
    float *p = part + (size_t)blockIdx.x * PART;
    float *pb1 = p + NW, *pb2 = pb1 + MLP_H, *pw3 = pb2 + MLP_H, *pb3 = pw3 + MLP_H;
    float4 *pv = reinterpret_cast<float4 *>(p) + tid;
#pragma unroll
    for (int a = 0; a < 8; a++) {
      pv[(2 * a) * NT] = make_float4(g2[a][0], g2[a][1], g2[a][2], g2[a][3]);
      pv[(2 * a + 1) * NT] = make_float4(g2[a][4], g2[a][5], g2[a][6], g2[a][7]);
      pv[(16 + a) * NT] = make_float4(g1[a][0], g1[a][1], g1[a][2], g1[a][3]);
    }
    // the two quads of a unit, and the samples of b3 and the loss
    __syncthreads();
    float *v = xs;
    if (q == 1) {
      v[j] = gb1;
      v[MLP_H + j] = gb2;
      v[2 * MLP_H + j] = gw3;
    }
    if (tid < GS) {
      dzs[tid] = gb3;
      dzs[GS + tid] = loss;
    }
    __syncthreads();
    if (q == 0) {
      pb1[j] = gb1 + v[j];
      pb2[j] = gb2 + v[MLP_H + j];
      pw3[j] = gw3 + v[2 * MLP_H + j];
    }
    if (tid < 2) {
      float t = 0.f;
      for (int i = 0; i < GS; i++) t += dzs[tid * GS + i];
      pb3[tid] = t;
    } else if (tid < 2 + PART - NPAR - 1) {
      pb3[tid] = 0.f;
    }
  }
}

// the parameter that a partial gradient's element is of; NPAR: the loss
__device__ __forceinline__ int param_of(int e) {
  if (e >= NW) {
    e -= NW;   // b1, b2, w3, b3: around W2 in the parameters
    return e < MLP_H ? MLP_H * MLP_IN + e : NW + e;
  }
  const int v = e >> 2, c = e & 3, tid = v % NT, g = v / NT, tj = tid >> 4, tk = tid & 15;
  return g < 16 ? MLP_H * MLP_IN + MLP_H + (tj + 16 * (g >> 1)) * MLP_H + tk + 16 * (4 * (g & 1) + c)
                : (tj + 16 * (g - 16)) * MLP_IN + tk + 16 * c;
}

// Sum of the CTAs' partial gradients (16 threads for four parameters, each a
// fixed part of the CTAs), then the Adam step if theta is given, else the
// gradient to grad; the loss adds to *loss.
__global__ void __launch_bounds__(256) k_reduce(const float *part, int nparts, float *grad, float *loss, float *theta,
                                                float *m, float *v, float lr, float b1, float b2, float eps, float bc1,
                                                float bc2) {
  __shared__ float sh[16][64];
  const int c = threadIdx.x & 15, sl = threadIdx.x >> 4, e0 = blockIdx.x * 64 + 4 * c;
  grid_wait();
  grid_launch_next();
  // the parameter's state is on its way while the partial sums are read
  const int e = blockIdx.x * 64 + threadIdx.x, p = threadIdx.x < 64 && e < NPAR + 1 ? param_of(e) : -1;
  const bool adam = theta && p >= 0 && p < NPAR;
  const float m0 = adam ? m[p] : 0.f, v0 = adam ? v[p] : 0.f, t0 = adam ? theta[p] : 0.f;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  if (e0 < PART) {
    const int per = (nparts + 15) / 16, end = min(nparts, (sl + 1) * per);
#pragma unroll 8
    for (int n = sl * per; n < end; n++) {
      const float4 x = *reinterpret_cast<const float4 *>(part + (size_t)n * PART + e0);
      s.x += x.x;
      s.y += x.y;
      s.z += x.z;
      s.w += x.w;
    }
  }
  *reinterpret_cast<float4 *>(&sh[sl][4 * c]) = s;
  __syncthreads();
  if (p < 0) return;
  float g = 0.f;
#pragma unroll
  for (int q = 0; q < 16; q++) g += sh[q][threadIdx.x];
  if (p == NPAR) {
    *loss += g;
    return;
  }
  if (!theta) {
    grad[p] = g;
    return;
  }
  const float mm = b1 * m0 + (1.f - b1) * g;
  const float vv = b2 * v0 + (1.f - b2) * g * g;
  m[p] = mm;
  v[p] = vv;
  theta[p] = t0 - lr * (mm / bc1) / (sqrtf(vv / bc2) + eps);
}

// combine: refine where the predictor says so, otherwise keep the plain flag
// learned pre-flag: probability above 1/2 on a block that can still refine
__global__ void k_combine(const float *prob, const DevBlock *blk, signed char *flags, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n && prob[i] > 0.5f && blk[i].level < blk[i].lmax) flags[i] = 1;
}

}  // namespace

int mlp_n_params() { return NPAR; }
size_t mlp_partial_floats() { return (size_t)MLP_MAX_CTAS * PART; }

namespace {
template <typename real>
void features(const KParams &kp, const real *U, int slot0, int nslots, float *out, cudaStream_t s) {
  // three planes in at most 100 KB (two CTAs per SM): blocks of up to 36 x 36
  // columns; above, the kernel without shared planes
  const size_t smem = sizeof(double) * (9 * (size_t)(kp.nb[1] + 2) * (kp.nb[2] + 2) + (size_t)kp.nb[1] * kp.nb[2]);
  constexpr size_t most = 100 * 1024;
  if (smem > most) {
    k_features_large<real><<<nslots, 256, 0, s>>>(kp, U, slot0, out);
    return;
  }
  if constexpr (sizeof(real) == 4) {
    raise_smem_limit<k_features_pairs, most>();
    k_features_pairs<<<nslots, FEAT_NT, smem, s>>>(kp, U, slot0, out);
  } else {
    raise_smem_limit<k_features, most>();
    k_features<<<nslots, 256, smem, s>>>(kp, U, slot0, out);
  }
}
}  // namespace

void mlp_features_launch(const KParams &kp, const void *U, int precision, int slot0, int nslots, float *out,
                         cudaStream_t s) {
  if (nslots <= 0) return;
  if (precision)
    features(kp, (const float *)U, slot0, nslots, out, s);
  else
    features(kp, (const double *)U, slot0, nslots, out, s);
}

namespace {
// a launch whose first instructions may overlap the end of the kernel before it
template <typename... P, typename... A>
void launch_after(bool overlap, void (*kernel)(P...), int grid, int block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = overlap ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, (P)args...);
}

// one CTA per SM at most (the weights take 102 KB of shared memory each)
template <bool GRAD>
int mlp_launch(const float *theta, const float *X, const float *T, const int *idx, int B, float *y, float *part,
               bool overlap, cudaStream_t s) {
  raise_smem_limit<k_mlp<GRAD>, MLP_SMEM>();
  const int groups = (B + GS - 1) / GS, n = groups < MLP_MAX_CTAS ? groups : MLP_MAX_CTAS;
  launch_after(overlap, k_mlp<GRAD>, n, NT, MLP_SMEM, s, theta, X, T, idx, B, y, part);
  return n;
}
}  // namespace

void mlp_forward_launch(const float *theta, const float *X, const int *idx, int B, float *y, cudaStream_t s) {
  if (B > 0) mlp_launch<false>(theta, X, nullptr, idx, B, y, nullptr, false, s);
}

void mlp_grad_launch(const float *theta, const float *X, const float *T, const int *idx, int B, float *part, float *grad,
                     float *loss, cudaStream_t s) {
  if (B <= 0) return;
  const int n = mlp_launch<true>(theta, X, T, idx, B, nullptr, part, false, s);
  k_reduce<<<(PART + 63) / 64, 256, 0, s>>>(part, n, grad, loss, nullptr, nullptr, nullptr, 0.f, 0.f, 0.f, 0.f, 1.f, 1.f);
}

// In a run of batches (more: not the first) the two kernels of a step overlap
// their ends and beginnings: the gather of a batch, which no kernel writes,
// comes before the wait, all else behind it.  A training of 16 batches of 1024:
// 511 -> 424 us.
void mlp_step_launch(float *theta, float *m, float *v, const float *X, const float *T, const int *idx, int B, float *part,
                     float *loss, float lr, int step, bool more, cudaStream_t s) {
  if (B <= 0) return;
  const float b1 = 0.9f, b2 = 0.999f;
  const float bc1 = 1.f - powf(b1, (float)step), bc2 = 1.f - powf(b2, (float)step);
  const int n = mlp_launch<true>(theta, X, T, idx, B, nullptr, part, more, s);
  launch_after(true, k_reduce, (PART + 63) / 64, 256, 0, s, part, n, nullptr, loss, theta, m, v, lr, b1, b2, 1e-8f, bc1,
               bc2);
}

void mlp_combine_launch(const float *prob, const DevBlock *blk, signed char *flags, int n, cudaStream_t s) {
  if (n > 0) k_combine<<<(n + 255) / 256, 256, 0, s>>>(prob, blk, flags, n);
}
