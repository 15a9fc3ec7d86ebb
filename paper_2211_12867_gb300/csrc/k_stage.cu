// Stage operator of the midpoint predictor-corrector on every leaf block.
//
//   predictor  U*      = U^n + dt/2 L(U^n)
//   corrector  U^{n+1} = U^n + dt   L(U*) + cleaning(U*)
//
// L(U) = -(1/V) sum_faces A F_TVDLF + S_geometric + S_rotation (arXiv
// 2211.12867, Sect. 2.1: TVDLF with the Woodward limiter, second order in space
// and time, ideal MHD in the co-rotating frame, parabolic div B cleaning).
// Geometric sources come from the spherical divergence of the momentum and
// induction tensors with the pressure parts in face-area-difference form (a
// uniform state is preserved to round-off); rotation sources are the Coriolis
// and centrifugal forces with the centrifugal work.  Cleaning is the
// diffusive (parabolic) form dB = C_d h^2 grad(div B*), de = B*.dB, with
// central differences and h^-2 = sum_d dx_d^-2.
//
// GPU design: one CTA owns a (theta x phi) tile of one block and marches along
// r.  Primitives of five consecutive r-planes live in a shared-memory ring
// (each cell of the tile plus its 2-cell halo is loaded and converted once per
// CTA); the r-face flux is carried in registers from one plane to the next;
// theta and phi face fluxes are computed once per face into shared memory and
// read by the two cells that share the face; div B of the corrector lives in a
// 4-plane ring.  The corrector also accumulates the CFL time step of the new
// state (FP64 max of the inverse time step per member) and stores the
// area-weighted face fluxes of block faces that border a different level for
// the reflux.  The grid is persistent: CTAs stride over (block, tile,
// r-segment) work items of all levels and all ensemble members.
//
// What bounds it.  FP32: latency and the barrier between the phases of a
// plane, with 53 to 56 % of the issue slots used by 16 warps per SM at 128
// registers; DRAM is idle (16 % of its peak).  More CTAs at fewer
// registers, a single flux buffer with a second barrier, and the staging of
// U^n in shared memory were slower.  512 x 60 x 180 cells in 64 x 60 x 180
// blocks: predictor 400 -> 281 us, corrector 489 -> 374 us since cells are
// stored whole (16-byte copies, one sector per scattered cell), geometry
// factors are staged per plane and row and no constant is converted per cell.
// FP64: the FP64 pipe, 80 % busy (19 cycles of an SM for each instruction of a
// warp), so the arithmetic is arranged for few such instructions: comparisons,
// minima and signs by integers, reciprocals and roots of three and five
// instructions, and flux sides added by the multiply-adds that form them; 64 x
// 60 x 180 cells: both stages 6382 -> 2090 us.
#include <cstdio>

#include "mhd_device.cuh"

namespace {

// plane and row factors staged per work item (see the kernel)
constexpr int NPF = 8, NRF = 8;

template <typename real>
struct StageSmem {
  // tracer: a 5-plane ring of the CME tracer fraction X and the sources of the
  // threads' copies follow the rest
  static constexpr size_t bytes(int tj, int tk, bool tracer = false) {
    return sizeof(real) * (size_t)(5 * NVAR * (tj + 4) * (tk + 4) + 2 * NVAR * (tj + 1) * tk +
                                   2 * NVAR * tj * (tk + 1) + 4 * (tj + 2) * (tk + 2) + geo(tj, tk) +
                                   (tracer ? 5 * (tj + 4) * (tk + 4) : 0)) +
           (tracer ? sizeof(void *) * (size_t)((tj + 4) * (tk + 4) + (tj * tk + 31) / 32 * 32) : 0);
  }
  // factors of the planes (and two arrays of the divergence's), of the tile's rows, three row arrays of
  // the divergence, one column array; rounded up to 16 bytes
  static constexpr int geo(int tj, int tk) {
    return (NPF * (STAGE_SEG_MAX + 4) + NRF * tj + 2 * (STAGE_SEG_MAX + 4) + 3 * (tj + 4) + (tk + 4) + 3) / 4 * 4;
  }
};

// The inverse time step is accumulated in the working precision (a maximum is
// exact in any precision) and enters the FP64 reduction once per warp.
template <typename real>
__device__ __forceinline__ void flush_acc(const KParams &kp, real &acc, int member, int &hits) {
  // warp max of the inverse time step, one atomic per warp
  for (int o = 16; o > 0; o >>= 1) acc = RT<real>::max_(acc, __shfl_xor_sync(0xffffffffu, acc, o));
  int h = hits;
  for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
  if ((threadIdx.x & 31) == 0 && member >= 0) {
    if (acc > real(0)) atomic_max_pos(&kp.inv_max[member], (double)acc);
    if (h) atomicAdd(kp.floor_hits, (unsigned long long)h);
  }
  acc = real(0);
  hits = 0;
}

// Shared arrays of 8-variable cells (the primitive ring, the face fluxes) are
// stored as [NVAR / CH][cell][CH] with CH = 16 bytes / sizeof(real): a cell's
// variables come in NVAR / CH 16-byte loads and consecutive cells are
// consecutive vectors (no bank conflicts between neighbouring threads).
template <typename real> struct Vec16;
template <> struct Vec16<float> {
  using T = float4;
  static constexpr int CH = 4;
  static __device__ __forceinline__ void put(T x, float *w) { w[0] = x.x; w[1] = x.y; w[2] = x.z; w[3] = x.w; }
  static __device__ __forceinline__ T get(const float *w) { return make_float4(w[0], w[1], w[2], w[3]); }
};
template <> struct Vec16<double> {
  using T = double2;
  static constexpr int CH = 2;
  static __device__ __forceinline__ void put(T x, double *w) { w[0] = x.x; w[1] = x.y; }
  static __device__ __forceinline__ T get(const double *w) { return make_double2(w[0], w[1]); }
};
template <typename real, int N>
__device__ __forceinline__ void ld8(const real *a, int q, real *w) {
  using V = Vec16<real>;
#pragma unroll
  for (int c = 0; c < NVAR / V::CH; c++)
    V::put(*reinterpret_cast<const typename V::T *>(a + (c * N + q) * V::CH), w + c * V::CH);
}
template <typename real, int N>
__device__ __forceinline__ void st8(real *a, int q, const real *w) {
  using V = Vec16<real>;
#pragma unroll
  for (int c = 0; c < NVAR / V::CH; c++)
    *reinterpret_cast<typename V::T *>(a + (c * N + q) * V::CH) = V::get(w + c * V::CH);
}
// one variable of a cell in that layout
template <typename real, int N>
__device__ __forceinline__ real &el(real *a, int v, int q) {
  constexpr int CH = Vec16<real>::CH;
  return a[((v / CH) * N + q) * CH + v % CH];
}
template <typename real, int N>
__device__ __forceinline__ real el(const real *a, int v, int q) {
  constexpr int CH = Vec16<real>::CH;
  return a[((v / CH) * N + q) * CH + v % CH];
}

// threads per CTA: the tile's cells rounded up to whole warps (the extra
// threads own no cell but share the loads and the face fluxes)
constexpr int stage_threads(int tj, int tk) { return (tj * tk + 31) / 32 * 32; }
constexpr int cmin(int a, int b) { return a < b ? a : b; }
constexpr int cmax(int a, int b) { return a > b ? a : b; }
// resident CTAs per SM the register budget is sized for (FP32): as many as
// the shared memory of an SM (228 KB, 1 KB reserved per CTA) holds, and no
// more than leave 128 registers a thread; at least 2.  FP64: 1.
constexpr int stage_min_ctas(int real_bytes, int tj, int tk) {
  return real_bytes != 4 ? 1
                         : cmax(2, cmin(65536 / (stage_threads(tj, tk) * 128),
                                        (int)(233472 / (StageSmem<float>::bytes(tj, tk) + 1024))));
}

// The scheme's constants in the working precision.  Converted on the host:
// conversions from the double parameters in the kernel are FP64-pipe
// instructions, which the compiler repeats per cell to save registers (13 per
// cell and 38 % of that pipe's time in the FP32 corrector).
template <typename real>
struct StageConst {
  real gamma, igm1, p_floor, rho_floor, omega, cd;
  Isl isl;
  explicit StageConst(const KParams &kp)
      : gamma((real)kp.gamma), igm1(real(1) / (gamma - real(1))), p_floor((real)kp.p_floor),
        rho_floor((real)kp.rho_floor), omega((real)kp.omega), cd((real)kp.cd),
        isl{(float)kp.isl_pe, (float)kp.isl_beta} {}
};

template <typename real, int TJ, int TK, bool S2>
__global__ void __launch_bounds__(stage_threads(TJ, TK), stage_min_ctas(sizeof(real), TJ, TK))
    k_stage(const KParams kp, const StageLaunch sl, const StageConst<real> sc_) {
  constexpr int NT = stage_threads(TJ, TK), RJ = TJ + 4, RK = TK + 4, RP = RJ * RK;
  constexpr int DJ = TJ + 2, DK = TK + 2, DP = DJ * DK;
  constexpr int NTH = (TJ + 1) * TK, NPH = TJ * (TK + 1);   // theta / phi faces of a plane
  constexpr int CH = Vec16<real>::CH, NUN = (RP + NT - 1) / NT;
  constexpr int PL = NVAR * RP;                             // reals of a ring plane
  constexpr bool F32 = sizeof(real) == 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  real *ring = reinterpret_cast<real *>(smem_raw);
  real *fth = ring + 5 * PL;            // two buffers of theta-face fluxes
  real *fph = fth + 2 * NVAR * NTH;     // two buffers of phi-face fluxes
  real *fend = fph + 2 * NVAR * NPH;
  // Factors of the work item's planes (from plane ib-2): areas over volume of
  // the r faces (halved: the fluxes carry a factor 2), dr2/dr3, Omega^2 r_c,
  // 1 / two-cell spacing, 1/dr, 1/r_c, divergence factor.  Of the tile's rows:
  // areas over volume of the theta faces and of the phi faces (halved, to be
  // multiplied by dr2/dr3), sin, cos, 1 / two-cell spacing, 1/sin, 1/dtheta.
  // An update so needs neither a face area nor a volume of its own.
  constexpr int NRP = STAGE_SEG_MAX + 4, NJ = TJ + 4;
  // FP32 keeps the areas, the volume and their order of operations: past the
  // CME's cone the state runs through a near-vacuum where the pressure floor
  // decides on the last bit, and a run differs by 3e-4 twenty steps after one
  // rounding (it is as far from FP64), so a change of rounding could not be
  // told from an error.  Areas over volume would save 6 to 9 % of the step.
  enum { P_RP, P_RM, P_DR, P_CF, P_ID2, P_IDR, P_IRC, P_FR };        // FP64
  enum { Q_R2, Q_R2P, Q_DR2, Q_DR3, Q_ID2 = P_ID2, Q_IDR = P_IDR, Q_IRC = P_IRC, Q_RC };   // FP32
  enum { R_TP, R_TM, R_PW, R_ST, R_CT, R_ITC2, R_IST, R_IDTH };      // FP64
  enum { S_SF, S_SFP, S_DCOS, S_ST = R_ST, S_CT = R_CT, S_ITC2 = R_ITC2, S_DTH, S_IDTH = R_IDTH };   // FP32
  real *s_pl = fend, *s_row = s_pl + NPF * NRP;
  real *dring = s_row + NRF * TJ;
  // for the divergence: r_c^2 per plane; sin, 1 / (sin * two-cell spacing) and
  // 1/sin per row from row -2; 1 / two-cell spacing per column from column -2
  real *s_rc2 = dring + 4 * DP, *s_fr = s_rc2 + NRP, *s_st = s_fr + NRP, *s_tt = s_st + NJ, *s_ist = s_tt + NJ,
       *s_ipc2 = s_ist + NJ;
  real *xring = fend + StageSmem<real>::geo(TJ, TK) + 4 * DP;   // tracer X, 5 planes (if stored)
  const real **s_xsrc = reinterpret_cast<const real **>(xring + 5 * RP + (RP & 1));
  const bool trc = kp.nvs > NVAR;

  const int tid = threadIdx.x, jl = tid / TK, kl = tid % TK;
  const real gamma = sc_.gamma, pfl = sc_.p_floor, rfl = sc_.rho_floor;
  const int nb0 = kp.nb[0], nb1 = kp.nb[1], nb2 = kp.nb[2];
  const int P1 = kp.P[1], P2 = kp.P[2];
  const size_t plane = (size_t)P1 * P2, vstride = (size_t)kp.P[0] * plane, bstride = kp.nvs * vstride;
  const int per_block = sl.tiles_j * sl.tiles_k * sl.segs;
  const int nwork = sl.nlist * per_block;
  const bool spherical = kp.geometry == 0;
  const real Om = sc_.omega, Cd = sc_.cd, igm1 = sc_.igm1;
  const Isl isl = sc_.isl;
  // ring cell of the thread's own cell (a thread without one: cell (2, 2))
  const int o = tid < TJ * TK ? (jl + 2) * RK + kl + 2 : 2 * RK + 2;
  // extra faces of the tile's far edges: TK theta faces (row TJ), then TJ phi
  // faces (column TK), one per thread of the first warps, which convert fewer
  // cells
  static_assert(TK + TJ <= NT, "one extra face per thread");
  const bool x_th = tid < TK;
  const int xq = x_th ? tid : tid - TK;
  const int xo = x_th ? (TJ + 2) * RK + xq + 2 : (xq + 2) * RK + TK + 2;
  // exchanges the theta and phi components
  auto turn = [](real *x, bool on) {
    const real v = x[2], b = x[6];
    x[2] = on ? x[3] : v;
    x[3] = on ? v : x[3];
    x[6] = on ? x[7] : b;
    x[7] = on ? b : x[7];
  };

  // reflux face buffer layout (per slot): faces in order r-lo, r-hi, th-lo,
  // th-hi, ph-lo, ph-hi; each [v][t1][t2]
  const int fc0 = nb1 * nb2, fc1 = nb0 * nb2, fc2 = nb0 * nb1;
  const size_t fstride = (size_t)NVAR * 2 * (fc0 + fc1 + fc2);

  real inv_acc = real(0);
  int hits = 0;
  int cur_member = -1;

  for (int w = blockIdx.x; w < nwork; w += gridDim.x) {
    int li = w / per_block, rem = w - li * per_block;
    const int seg = rem % sl.segs;
    rem /= sl.segs;
    const int tk = rem % sl.tiles_k, tj = rem / sl.tiles_k;
    const int slot = sl.list[li];
    const DevBlock &B = kp.blk[slot];
    const int member = B.member;
    const double dtm = kp.dt_used[member];
    if (!(dtm > 0.0)) continue;  // member has reached its stop time (uniform)
    if (S2 && member != cur_member) {
      flush_acc(kp, inv_acc, cur_member, hits);
      cur_member = member;
    }
    const real dt = (real)(dtm * sl.dtfac);
    const LevelGeo<real> &G = GeoSel<real>::get(kp.geo, B.level);
    const int j0 = tj * TJ, k0 = tk * TK;
    const int nvj = min(TJ, nb1 - j0), nvk = min(TK, nb2 - k0);
    const int ib = seg * sl.seg_len, ie = min(nb0, ib + sl.seg_len);
    const int I0 = B.ix[0] * nb0, J0 = B.ix[1] * nb1 + j0, K0 = B.ix[2] * nb2 + k0;
    const real *Uin = reinterpret_cast<const real *>(sl.Uin) + (size_t)slot * bstride;
    const real *U0 = reinterpret_cast<const real *>(sl.U0) + (size_t)slot * bstride;
    real *Uout = reinterpret_cast<real *>(sl.Uout) + (size_t)slot * bstride;
    const bool own = tid < TJ * TK, valid = own && jl < nvj && kl < nvk;
    const int j = j0 + jl, k = k0 + kl;           // interior indices in the block
    const bool has_th = own && jl <= nvj && kl < nvk, has_ph = own && jl < nvj && kl <= nvk;
    const bool any_face = __any_sync(0xffffffffu, has_th || has_ph);
    const bool x_face = x_th ? nvj == TJ && xq < nvk : tid < TK + TJ && nvk == TK && xq < nvj;
    // block faces with a finer, and with a coarser or finer, neighbour; those
    // the thread's column touches
    unsigned fin = 0, cfb = 0, edge = 0;
    if (S2) {
#pragma unroll
      for (int f = 0; f < 6; f++) {
        const int q = B.nbr[f];
        fin |= (unsigned)(q == NB_FINER) << f;
        cfb |= (unsigned)(q == NB_FINER || q == NB_COARSER) << f;
      }
      edge = (unsigned)(j == 0) << 2 | (unsigned)(j == nb1 - 1) << 3 | (unsigned)(k == 0) << 4 |
             (unsigned)(k == nb2 - 1) << 5;
    }

    // Planes of U_in are copied asynchronously (cp.async, 16 bytes per copy)
    // straight into their ring slot and converted to primitives in place one
    // iteration later, by the thread that copied them (no barrier between
    // copy and conversion).  Cells go to the highest thread indices first,
    // which own no second div B position.  Cells of the plane outside the
    // block that a same-level leaf holds come straight from that leaf's
    // interior (sl.direct: the step's ghost fills leave such ghost copies
    // unfilled); the others from this block's ghost layer (coarser or finer
    // neighbours, physical boundaries).  A thread's sources change only where
    // the march enters or leaves the block's r range.
    const real *src[NUN];
    int src_side = 2;
    auto set_src = [&](int sr) {
      src_side = sr;
#pragma unroll
      for (int u = 0; u < NUN; u++) {
        const int q = NT - 1 - tid + u * NT, jj = q / RK, kk = q - (q / RK) * RK;
        const int pj = j0 + jj, pk = k0 + kk;
        src[u] = nullptr;
        if (q < RP && pj < P1 && pk < P2) {
          const real *blk = Uin;
          long long cell = (long long)NGH * (long long)plane + (long long)pj * P2 + pk;
          if (sl.direct) {
            const int sj = pj < NGH ? -1 : (pj >= NGH + nb1 ? 1 : 0);
            const int sk = pk < NGH ? -1 : (pk >= NGH + nb2 ? 1 : 0);
            if (sr | sj | sk) {
              const int n = kp.nb27[(size_t)slot * 27 + (sr + 1) * 9 + (sj + 1) * 3 + (sk + 1)];
              if (n >= 0) {
                blk = reinterpret_cast<const real *>(sl.Uin) + (size_t)n * bstride;
                cell -= (long long)sr * nb0 * (long long)plane + (long long)sj * nb1 * P2 + sk * nb2;
              }
            }
          }
          src[u] = blk + NVAR * cell;
          if (trc) s_xsrc[u * NT + tid] = blk + TRV * vstride + cell;
        }
      }
    };
    auto issue_plane = [&](int p, int at) {
      const int sr = p < 0 ? -1 : (p >= nb0 ? 1 : 0);
      if (sr != src_side) set_src(sr);
      const long long off = (long long)p * (long long)plane;
      real *dst = ring + at;
#pragma unroll
      for (int u = 0; u < NUN; u++)
        if (src[u]) {
          const int q = NT - 1 - tid + u * NT;
          const real *from = src[u] + NVAR * off;
#pragma unroll
          for (int v = 0; v < NVAR; v += CH) cp_async<16>(dst + ((v / CH) * RP + q) * CH, from + v);
          if (trc) cp_async<sizeof(real)>(xring + at / NVAR + q, s_xsrc[u * NT + tid] + off);
        }
      cp_async_commit();
    };
    auto convert_plane = [&](int at) {
      real *pl = ring + at;
#pragma unroll
      for (int u = 0; u < NUN; u++)
        if (src[u]) {
          const int q = NT - 1 - tid + u * NT;
          real uu[NVAR], wv[NVAR];
          ld8<real, RP>(pl, q, uu);
          cons2prim<real>(uu, wv, gamma, pfl, isl);
          st8<real, RP>(pl, q, wv);
          if (trc) xring[at / NVAR + q] *= RT<real>::rcp_(uu[0]);   // rho X -> X
        }
    };
    // U^n of the thread's own cell is read at the start of the update and used
    // behind the r flux, which hides an access to L2 (staging it one plane
    // ahead with the plane copies made the update wait for those as well); the
    // corrector, whose input is another array, brings it there one plane ahead
    const real *u0p = U0 + NVAR * ((size_t)(ib + NGH) * plane + (size_t)(j + NGH) * P2 + (k + NGH));
    // ring offset of the plane after the one at offset a
    auto next = [](int a) { return a == 4 * PL ? 0 : a + PL; };
    // half the limited radial slope of the thread's column at the middle of
    // the planes at offsets m, c, p
    // (FP64: the difference across the later face is kept for the next plane)
    real rdiff[F32 ? 1 : NVAR];
    auto rslope = [&](int m, int c, int p, real *out, bool carried) {
      if constexpr (F32) {
        real a[NVAR], b[NVAR], e[NVAR];
        ld8<real, RP>(ring + m, o, a);
        ld8<real, RP>(ring + c, o, b);
        ld8<real, RP>(ring + p, o, e);
        mc_half_slopes8<real>(a, b, e, out);
      } else {
        real b[NVAR], e[NVAR];
        ld8<real, RP>(ring + c, o, b);
        ld8<real, RP>(ring + p, o, e);
        if (!carried) {
          real a[NVAR];
          ld8<real, RP>(ring + m, o, a);
#pragma unroll
          for (int v = 0; v < NVAR; v++) rdiff[v] = b[v] - a[v];
        }
#pragma unroll
        for (int v = 0; v < NVAR; v++) {
          const real dp = e[v] - b[v];
          out[v] = mc_half_of(rdiff[v], dp);
          rdiff[v] = dp;
        }
      }
    };
    // radial face between the planes at offsets m and c from the slopes at both
    auto rflux = [&](int m, int c, const real *sm, const real *sp, real *F) {
      real b[NVAR], e[NVAR];
      ld8<real, RP>(ring + m, o, b);
      ld8<real, RP>(ring + c, o, e);
      if constexpr (sizeof(real) == 4) {
        tvdlf_pair<0>(b, e, sm, sp, gamma, igm1, F);
      } else {
        real WL[NVAR], WR[NVAR];
        axpy8<real>(b, real(1), sm, WL);
        axpy8<real>(e, real(-1), sp, WR);
        tvdlf_states<0>(WL, WR, b, e, gamma, igm1, F);
      }
    };
    // div B at plane p (offsets of planes p-1, p, p+1) on the (TJ+2) x (TK+2)
    // positions around the tile
    auto divb_plane = [&](int p, int m, int c, int e) {
      real *dst = dring + (p & 3) * DP;
      const real *pm = ring + m, *pc = ring + c, *pp = ring + e;
      const int pr = p - ib + 2;   // plane index in the staged arrays
      const real wm = s_rc2[pr - 1], wp = s_rc2[pr + 1], fr = F32 ? s_fr[pr] : s_pl[NPF * pr + P_FR];
      const real irc = s_pl[NPF * pr + P_IRC], rcc = s_pl[NPF * pr + Q_RC];
      for (int q = tid; q < DP; q += NT) {
        const int dj = q / DK, dk = q - (q / DK) * DK;   // row and column + 1
        if (dj > nvj + 1 || dk > nvk + 1) continue;
        const int at = (dj + 1) * RK + dk + 1;
        const real brm = el<real, RP>(pm, 5, at), brp = el<real, RP>(pp, 5, at);
        const real btm = el<real, RP>(pc, 6, at - RK), btp = el<real, RP>(pc, 6, at + RK);
        const real bpm = el<real, RP>(pc, 7, at - 1), bpp = el<real, RP>(pc, 7, at + 1);
        if constexpr (!F32) {
          dst[q] = (wp * brp - wm * brm) * fr + ((s_st[dj + 2] * btp - s_st[dj] * btm) * s_tt[dj + 1] +
                                                (bpp - bpm) * (s_ist[dj + 1] * s_ipc2[dk + 1])) * irc;
        } else {
          const real itc2 = s_tt[dj + 1], ipc2 = s_ipc2[dk + 1];
          real div;
          if (spherical) {
            const real stc = s_st[dj + 1];
            const real sm = s_st[dj], sp = s_st[dj + 2];
            const real irs = RT<real>::rcp_(rcc * stc);
            div = (wp * brp - wm * brm) * fr + (sp * btp - sm * btm) * irs * itc2 + (bpp - bpm) * irs * ipc2;
          } else {
            div = (brp - brm) * fr + (btp - btm) * itc2 + (bpp - bpm) * ipc2;
          }
          dst[q] = div;
        }
      }
    };

    // ---- prologue: planes ib-2 .. ib+2 converted, r flux at face ib ----
    // offsets of planes i-1 .. i+3 of the march (plane p sits at p + 2 - ib
    // planes past the first slot, modulo five)
    int om = PL, oc = 2 * PL, o1 = 3 * PL, o2 = 4 * PL, o3 = 0;
    for (int p = 0; p < 5; p++) {
      issue_plane(ib - 2 + p, p * PL);
    }
    if (S2 && valid) prefetch_cell(u0p);
    // ---- factors of the work item into shared memory (read after the
    // prologue's first barrier); rows / columns past the block's edge are
    // never read and not loaded ----
    const real dphi = G.dphi, idphi = RT<real>::rcp_(dphi);
    {
      const int npl = ie - ib + 4, ir0 = I0 + ib - 2 + NGH;
      for (int q = tid; q < npl; q += NT) {
        real *f = s_pl + NPF * q;
        const real rc = G.rc[ir0 + q], iv3 = RT<real>::rcp_(G.dr3[ir0 + q]);
        const real irc = spherical ? RT<real>::rcp_(rc) : real(1);
        f[P_IDR] = RT<real>::rcp_(G.dr[ir0 + q]);
        f[P_IRC] = irc;
        s_rc2[q] = spherical ? rc * rc : real(1);
        if (q >= 1 && q + 1 < npl) f[P_ID2] = RT<real>::rcp_(G.rc[ir0 + q + 1] - G.rc[ir0 + q - 1]);
        if constexpr (F32) {
          f[Q_R2] = G.r2f[ir0 + q];
          f[Q_R2P] = G.r2f[ir0 + q + 1];
          f[Q_DR2] = G.dr2[ir0 + q];
          f[Q_DR3] = G.dr3[ir0 + q];
          f[Q_RC] = rc;
          if (q >= 1 && q + 1 < npl)
            s_fr[q] = RT<real>::rcp_((spherical ? rc * rc : real(1)) * (G.rc[ir0 + q + 1] - G.rc[ir0 + q - 1]));
        } else {
          f[P_RP] = real(0.5) * G.r2f[ir0 + q + 1] * iv3;
          f[P_RM] = real(0.5) * G.r2f[ir0 + q] * iv3;
          f[P_DR] = G.dr2[ir0 + q] * iv3;
          f[P_CF] = Om * Om * rc;
          if (q >= 1 && q + 1 < npl) f[P_FR] = f[P_ID2] * irc * irc;
        }
      }
      const int jr0 = J0 - 2 + NGH;
      for (int q = tid; q < nvj + 4; q += NT) {
        const real st = G.sintc[jr0 + q], ist = RT<real>::rcp_(st);
        s_st[q] = st;
        s_ist[q] = ist;
        if (q >= 1 && q + 1 < nvj + 4) {
          const real itc2 = RT<real>::rcp_(G.tc[jr0 + q + 1] - G.tc[jr0 + q - 1]);
          s_tt[q] = F32 ? itc2 : ist * itc2;
          if (q >= 2 && q < nvj + 2) {
            real *f = s_row + NRF * (q - 2);
            f[R_ST] = st;
            f[R_CT] = G.costc[jr0 + q];
            f[R_ITC2] = itc2;
            f[R_IDTH] = RT<real>::rcp_(G.dth[jr0 + q]);
            if constexpr (F32) {
              f[S_SF] = G.sinf[jr0 + q];
              f[S_SFP] = G.sinf[jr0 + q + 1];
              f[S_DCOS] = G.dcos[jr0 + q];
              f[S_DTH] = G.dth[jr0 + q];
            } else {
              const real idc = RT<real>::rcp_(G.dcos[jr0 + q]);
              f[R_TP] = real(0.5) * G.sinf[jr0 + q + 1] * idc;
              f[R_TM] = real(0.5) * G.sinf[jr0 + q] * idc;
              f[R_PW] = real(0.5) * G.dth[jr0 + q] * idc * idphi;
              f[R_IST] = ist;
            }
          }
        }
      }
      const int kr0 = K0 - 2 + NGH;
      for (int q = 1 + tid; q + 1 < nvk + 4; q += NT) s_ipc2[q] = RT<real>::rcp_(G.pc[kr0 + q + 1] - G.pc[kr0 + q - 1]);
    }

    cp_async_wait_all();
    for (int p = 0; p < 5; p++) convert_plane(p * PL);
    __syncthreads();
    if (S2) {
      divb_plane(ib - 1, 0, om, oc);
      divb_plane(ib, om, oc, o1);
    }
    real Flo[NVAR], sc[NVAR];
    real xprev = real(0);   // tracer X of this column at the previous plane
    if (valid) {
      real s0[NVAR];
      rslope(0, om, oc, s0, false);
      rslope(om, oc, o1, sc, true);
      rflux(om, oc, s0, sc, Flo);
      if (trc) xprev = xring[RP + o];
    }
    __syncthreads();   // plane ib-2 is read no more: its slot takes plane ib+3
    if (ib + 3 <= ie + 1) issue_plane(ib + 3, o3);
    else cp_async_commit();

    // One barrier per plane.  Phase A (before it): theta and phi face fluxes
    // of plane i into face buffer i&1, div B of plane i+1, conversion of plane
    // i+3.  Phase B (after it): r flux at face i+1 and the update of the
    // thread's cell of plane i, then the copies of plane i+4 (into the slot of
    // plane i-1, which neither phase reads any more) and of U^n at plane i+1.
    // A thread in phase A of plane i+1 can overlap others still in phase B of
    // plane i: they use the other face buffer, another div B slot and
    // disjoint ring slots.
    for (int i = ib; i < ie; i++) {
      real *fthb = fth + (i & 1) * NVAR * NTH, *fphb = fph + (i & 1) * NVAR * NPH;
      {
        // The lower theta and phi face of the thread's cell, in one straight
        // run (a thread without one of the two computes on whatever its ring
        // cells hold and stores nothing), then the extra face.
        const real *pl = ring + oc;
        if (any_face) {
          real a[NVAR], b[NVAR], c[NVAR], e[NVAR], F[NVAR];
          ld8<real, RP>(pl, o - 2 * RK, a);
          ld8<real, RP>(pl, o - RK, b);
          ld8<real, RP>(pl, o, c);
          ld8<real, RP>(pl, o + RK, e);
          tvdlf_face<real, 1>(a, b, c, e, gamma, igm1, F);
          if (has_th) st8<real, NTH>(fthb, tid, F);
          ld8<real, RP>(pl, o - 2, a);
          ld8<real, RP>(pl, o - 1, b);
          ld8<real, RP>(pl, o + 1, e);
          tvdlf_face<real, 2>(a, b, c, e, gamma, igm1, F);
          if (has_ph) st8<real, NPH>(fphb, tid + jl, F);
        }
        if (x_face) {
          // theta and phi faces in the lanes of one warp: in FP64 a phi face is a
          // theta face with the theta and phi components exchanged, in FP32 (where
          // the order of a sum decides on its last bit) the direction is chosen
          // lane by lane
          real a[NVAR], b[NVAR], c[NVAR], e[NVAR], F[NVAR];
          const int d = x_th ? RK : 1;
          ld8<real, RP>(pl, xo - 2 * d, a);
          ld8<real, RP>(pl, xo - d, b);
          ld8<real, RP>(pl, xo, c);
          ld8<real, RP>(pl, xo + d, e);
          if constexpr (F32) {
            tvdlf_face<real, -1>(a, b, c, e, gamma, igm1, F, !x_th);
          } else {
            turn(a, !x_th);
            turn(b, !x_th);
            turn(c, !x_th);
            turn(e, !x_th);
            tvdlf_face<real, 1>(a, b, c, e, gamma, igm1, F);
            turn(F, !x_th);
          }
          if (x_th) st8<real, NTH>(fthb, TJ * TK + xq, F);
          else st8<real, NPH>(fphb, xq * (TK + 1) + TK, F);
        }
      }
      if (S2) divb_plane(i + 1, oc, o1, o2);
      if (i + 3 <= ie + 1) {
        cp_async_wait_group<0>();   // plane i+3 landed
        convert_plane(o3);
      }
      __syncthreads();
      if (valid) {
        real Fhi[NVAR], u0[NVAR];
        ld_cell(u0p, u0);
        u0p += NVAR * plane;
        if (S2 && i + 1 < ie) prefetch_cell(u0p);
        {
          real sn[NVAR];
          rslope(oc, o1, o2, sn, true);
          rflux(oc, o1, sc, sn, Fhi);
#pragma unroll
          for (int v = 0; v < NVAR; v++) sc[v] = sn[v];
        }
        const int pr = i - ib + 2;   // plane index in the staged arrays
        real pf[NPF], rf[NRF];
#pragma unroll
        for (int v = 0; v < NPF; v += CH) Vec16<real>::put(*reinterpret_cast<const typename Vec16<real>::T *>(s_pl + NPF * pr + v), pf + v);
#pragma unroll
        for (int v = 0; v < NRF; v += CH) Vec16<real>::put(*reinterpret_cast<const typename Vec16<real>::T *>(s_row + NRF * jl + v), rf + v);
        real w[NVAR];
        ld8<real, RP>(ring + oc, o, w);
        real un[NVAR];
        const size_t cidx = (size_t)(i + NGH) * plane + (size_t)(j + NGH) * P2 + (k + NGH);
        // FP64: areas over volume of the theta and phi faces.  FP32: half
        // areas and 1 / V
        real ctp, ctm, cpw, crp, crm, iV = real(1), Arm = real(0), Arp = real(0), Atm = real(0), Atp = real(0);
        if constexpr (F32) {
          const real dcos = rf[S_DCOS], dr2 = pf[Q_DR2];
          Arm = pf[Q_R2] * dcos * dphi;
          Arp = pf[Q_R2P] * dcos * dphi;
          Atm = rf[S_SF] * dr2 * dphi;
          Atp = rf[S_SFP] * dr2 * dphi;
          const real Ap = dr2 * rf[S_DTH];
          crm = real(0.5) * Arm;
          crp = real(0.5) * Arp;
          ctm = real(0.5) * Atm;
          ctp = real(0.5) * Atp;
          cpw = real(0.5) * Ap;
          const real V = pf[Q_DR3] * dcos * dphi;
          iV = RT<real>::rcp_(V);
        } else {
          crp = pf[P_RP];
          crm = pf[P_RM];
          ctp = pf[P_DR] * rf[R_TP];
          ctm = pf[P_DR] * rf[R_TM];
          cpw = pf[P_DR] * rf[R_PW];
        }
        {
          const int qp = tid + jl;
#pragma unroll
          for (int c = 0; c < NVAR / CH; c++) {
            real ftl[CH], fth_[CH], fpl[CH], fph_[CH];
            using V = Vec16<real>;
            V::put(*reinterpret_cast<const typename V::T *>(fthb + (c * NTH + tid) * CH), ftl);
            V::put(*reinterpret_cast<const typename V::T *>(fthb + (c * NTH + tid + TK) * CH), fth_);
            V::put(*reinterpret_cast<const typename V::T *>(fphb + (c * NPH + qp) * CH), fpl);
            V::put(*reinterpret_cast<const typename V::T *>(fphb + (c * NPH + qp + 1) * CH), fph_);
            if constexpr (F32)
              flux_balance32(Fhi + c * CH, Flo + c * CH, fth_, ftl, fph_, fpl, crp, crm, ctp, ctm, cpw, iV, un + c * CH);
            else
              flux_balance<real, CH>(Fhi + c * CH, Flo + c * CH, fth_, ftl, fph_, fpl, crp, crm, ctp, ctm, cpw,
                                     un + c * CH);
          }
        }
        if constexpr (F32) {
          if (spherical) {
            const real gr = (Arp - Arm) * iV, gt = (Atp - Atm) * iV, ir = real(0.5) * gr;
            const real rho = w[0], vr = w[1], vt = w[2], vp = w[3], Br = w[5], Bt = w[6], Bp = w[7];
            const real pt = w[4] + real(0.5) * (Br * Br + Bt * Bt + Bp * Bp);
            un[1] += (rho * (vt * vt + vp * vp) - (Bt * Bt + Bp * Bp)) * ir + pt * gr;
            un[2] += (-rho * vr * vt + Br * Bt) * ir + (rho * vp * vp - Bp * Bp) * gt + pt * gt;
            un[3] += (-rho * vr * vp + Br * Bp) * ir - (rho * vt * vp - Bt * Bp) * gt;
            un[6] += (vr * Bt - vt * Br) * ir;
            un[7] += (vr * Bp - vp * Br) * ir + (vt * Bp - vp * Bt) * gt;
            const real rc = pf[Q_RC], st = rf[S_ST], ct = rf[S_CT];
            const real vs = vr * st + vt * ct;
            un[1] += rho * (real(2) * Om * vp * st + Om * Om * rc * st * st);
            un[2] += rho * (real(2) * Om * vp * ct + Om * Om * rc * st * ct);
            un[3] += real(-2) * Om * rho * vs;
            un[4] += rho * Om * Om * rc * st * vs;
          }
        } else if (spherical) {
          // ir = (A_r+ - A_r-) / 2V, gt = (A_th+ - A_th-) / V
          const real ir = crp - crm, gt = real(2) * (ctp - ctm);
          const real rho = w[0], vr = w[1], vt = w[2], vp = w[3], Br = w[5], Bt = w[6], Bp = w[7];
          const real mt = rho * vt, mp = rho * vp, Bt2 = Bt * Bt, Bp2 = Bp * Bp;
          const real tpp = mp * vp - Bp2, ttt = mt * vt - Bt2;   // stress without pressure
          const real pt = w[4] + real(0.5) * (Br * Br + Bt2 + Bp2);
          un[1] += (tpp + ttt + real(2) * pt) * ir;
          un[2] += (Br * Bt - mt * vr) * ir + (tpp + pt) * gt;
          un[3] += (Br * Bp - mp * vr) * ir - (mt * vp - Bt * Bp) * gt;
          un[6] += (vr * Bt - vt * Br) * ir;
          un[7] += (vr * Bp - vp * Br) * ir + (vt * Bp - vp * Bt) * gt;
          // Coriolis and centrifugal forces, centrifugal work
          const real st = rf[R_ST], ct = rf[R_CT], cf = pf[P_CF] * st;
          const real c2 = real(2) * Om * mp + rho * cf;
          const real vs = vr * st + vt * ct, mvs = rho * vs;
          un[1] += c2 * st;
          un[2] += c2 * ct;
          un[3] -= real(2) * Om * mvs;
          un[4] += cf * mvs;
        }
        axpy8<real>(u0, dt, un, un);
        // reciprocal cell widths (FP64: the speeds of the corrector's CFL step, h
        // of the cleaning)
        const real irs = pf[P_IRC] * rf[R_IST];
        const real ix[3] = {pf[P_IDR], spherical ? pf[P_IRC] * rf[R_IDTH] : rf[R_IDTH], spherical ? irs * idphi : idphi};
        if (S2 && Cd > real(0)) {
          const real *dm = dring + ((i - 1) & 3) * DP, *dc = dring + (i & 3) * DP, *dp = dring + ((i + 1) & 3) * DP;
          const int q = (jl + 1) * DK + (kl + 1);
          const real ird2 = pf[P_ID2], itc2 = rf[R_ITC2], ipc2 = s_ipc2[kl + 2];
          real gr_, gt_, gp_, h2inv;
          if constexpr (F32) {
            const real idr = pf[Q_IDR], idth = rf[S_IDTH];
            if (spherical) {
              const real irc = pf[Q_IRC], irs32 = RT<real>::rcp_(pf[Q_RC] * rf[S_ST]);
              gr_ = (dp[q] - dm[q]) * ird2;
              gt_ = (dc[q + DK] - dc[q - DK]) * irc * itc2;
              gp_ = (dc[q + 1] - dc[q - 1]) * irs32 * ipc2;
              const real ixt = irc * idth, ixp = irs32 * idphi;
              h2inv = idr * idr + ixt * ixt + ixp * ixp;
            } else {
              gr_ = (dp[q] - dm[q]) * ird2;
              gt_ = (dc[q + DK] - dc[q - DK]) * itc2;
              gp_ = (dc[q + 1] - dc[q - 1]) * ipc2;
              h2inv = idr * idr + idth * idth + idphi * idphi;
            }
          } else {
            gr_ = (dp[q] - dm[q]) * ird2;
            gt_ = (dc[q + DK] - dc[q - DK]) * (pf[P_IRC] * itc2);
            gp_ = (dc[q + 1] - dc[q - 1]) * (irs * ipc2);
            h2inv = ix[0] * ix[0] + ix[1] * ix[1] + ix[2] * ix[2];
          }
          const real f = Cd * RT<real>::rcp_(h2inv);
          const real dB0 = f * gr_, dB1 = f * gt_, dB2 = f * gp_;
          un[5] += dB0;
          un[6] += dB1;
          un[7] += dB2;
          un[4] += w[5] * dB0 + w[6] * dB1 + w[7] * dB2;
        }
        if (trc) {
          // CME tracer (Sect. 3.1): rho X carried by each face's mass flux
          // with X from the face's upwind cell
          // X at plane i-1 of this column is carried from the previous plane:
          // that ring slot already receives the copy of plane i+4
          const real *xc = xring + oc / NVAR, *xp = xring + o1 / NVAR;
          const real X0 = xc[o];
          const real ftl0 = el<real, NTH>(fthb, 0, tid), fth0 = el<real, NTH>(fthb, 0, tid + TK);
          const real fpl0 = el<real, NPH>(fphb, 0, tid + jl), fph0 = el<real, NPH>(fphb, 0, tid + jl + 1);
          const real arm = crm * Flo[0] * (Flo[0] > real(0) ? xprev : X0);
          const real arp = crp * Fhi[0] * (Fhi[0] > real(0) ? X0 : xp[o]);
          const real atm = ctm * ftl0 * (ftl0 > real(0) ? xc[o - RK] : X0);
          const real atp = ctp * fth0 * (fth0 > real(0) ? X0 : xc[o + RK]);
          const real apm = cpw * fpl0 * (fpl0 > real(0) ? xc[o - 1] : X0);
          const real app = cpw * fph0 * (fph0 > real(0) ? X0 : xc[o + 1]);
          const real dT = -((arp - arm) + (atp - atm) + (app - apm)) * iV;
          Uout[TRV * vstride + cidx] = U0[TRV * vstride + cidx] + dt * dT;
          xprev = X0;
        }
        // Floors.  FP64: the pressure of the new state serves the CFL speed and
        // tells a cell that might be below a floor, which takes apply_floors
        real irn = real(0), pn = real(0);
        if constexpr (F32) {
          hits += apply_floors<real>(un, gamma, pfl, rfl, isl);
        } else {
          irn = RT<real>::rcp_(un[0]);
          pn = pressure_for_speed<real>(un, gamma);
          if (RT<real>::less_(un[0], rfl) || !RT<real>::less_(pfl, pn)) {
            hits += apply_floors<real>(un, gamma, pfl, rfl, isl);
            irn = RT<real>::rcp_(un[0]);
            pn = pressure_for_speed<real>(un, gamma);
            if (RT<real>::less_(pn, pfl)) pn = pfl;
          }
        }
        if (RT<real>::nan_(un[0]) || RT<real>::nan_(un[4])) atomicOr(kp.status, ST_NAN);
        st_cell(Uout + NVAR * cidx, un);
        if (S2) {
          const unsigned at = edge | (unsigned)(i == 0) | (unsigned)(i == nb0 - 1) << 1;
          // CFL contribution of the new state (cells next to a finer face are
          // left to the reflux, which changes them once more)
          if (!(at & fin)) {
            real s;
            if constexpr (F32) {
              real wn[NVAR];
              cons2prim_speed<real>(un, wn, gamma, pfl);
              real dx1 = rf[S_DTH], dx2 = dphi;
              if (spherical) {
                dx1 *= pf[Q_RC];
                dx2 *= pf[Q_RC] * rf[S_ST];
              }
              s = (RT<real>::abs_(wn[1]) + fast_speed<real, 0>(wn, gamma)) * pf[Q_IDR] +
                  (RT<real>::abs_(wn[2]) + fast_speed<real, 1>(wn, gamma)) * RT<real>::rcp_(dx1) +
                  (RT<real>::abs_(wn[3]) + fast_speed<real, 2>(wn, gamma)) * RT<real>::rcp_(dx2);
            } else {
              const real vn[3] = {un[1] * irn, un[2] * irn, un[3] * irn};
              s = cfl_rate(irn, vn, pn, un + 5, gamma, ix);
            }
            inv_acc = RT<real>::less_(inv_acc, s) ? s : inv_acc;
          }
          if (sl.flux && (at & cfb)) {
            // area-weighted fluxes of the block's coarse-fine faces
            real *fb = reinterpret_cast<real *>(sl.flux) + (size_t)slot * fstride;
            const unsigned hit = at & cfb;
            const int I = I0 + i + NGH, J = J0 + jl + NGH;
            const real dcos = G.dcos[J], dr2 = G.dr2[I];
            const size_t o2_ = (size_t)2 * NVAR * fc0, o4 = o2_ + (size_t)2 * NVAR * fc1;
            if (hit & 1u) {
              const real A = real(0.5) * (G.r2f[I] * dcos * dphi);
#pragma unroll
              for (int v = 0; v < NVAR; v++) fb[(size_t)v * fc0 + j * nb2 + k] = A * Flo[v];
            }
            if (hit & 2u) {
              const real A = real(0.5) * (G.r2f[I + 1] * dcos * dphi);
#pragma unroll
              for (int v = 0; v < NVAR; v++) fb[(size_t)NVAR * fc0 + (size_t)v * fc0 + j * nb2 + k] = A * Fhi[v];
            }
            if (hit & 4u) {
              const real A = real(0.5) * (G.sinf[J] * dr2 * dphi);
#pragma unroll
              for (int v = 0; v < NVAR; v++)
                fb[o2_ + (size_t)v * fc1 + i * nb2 + k] = A * el<real, NTH>(fthb, v, tid);
            }
            if (hit & 8u) {
              const real A = real(0.5) * (G.sinf[J + 1] * dr2 * dphi);
#pragma unroll
              for (int v = 0; v < NVAR; v++)
                fb[o2_ + (size_t)NVAR * fc1 + (size_t)v * fc1 + i * nb2 + k] = A * el<real, NTH>(fthb, v, tid + TK);
            }
            if (hit & 48u) {
              const real A = real(0.5) * (dr2 * G.dth[J]);
              if (hit & 16u)
#pragma unroll
                for (int v = 0; v < NVAR; v++)
                  fb[o4 + (size_t)v * fc2 + i * nb1 + j] = A * el<real, NPH>(fphb, v, tid + jl);
              if (hit & 32u)
#pragma unroll
                for (int v = 0; v < NVAR; v++)
                  fb[o4 + (size_t)NVAR * fc2 + (size_t)v * fc2 + i * nb1 + j] = A * el<real, NPH>(fphb, v, tid + jl + 1);
            }
          }
        }
#pragma unroll
        for (int v = 0; v < NVAR; v++) Flo[v] = Fhi[v];
      }
      if (i + 4 <= ie + 1) issue_plane(i + 4, om);
      else cp_async_commit();
      om = oc;
      oc = o1;
      o1 = o2;
      o2 = o3;
      o3 = next(o3);
    }
    cp_async_wait_all();
    __syncthreads();  // shared memory is reused by the next work item
  }
  if (S2) flush_acc(kp, inv_acc, cur_member, hits);
  else {
    int h = hits;
    for (int q = 16; q > 0; q >>= 1) h += __shfl_xor_sync(0xffffffffu, h, q);
    if ((threadIdx.x & 31) == 0 && h) atomicAdd(kp.floor_hits, (unsigned long long)h);
  }
}

template <typename real, int TJ, int TK>
int launch_t(const KParams &kp, const StageLaunch &sl, cudaStream_t s) {
  const size_t smem = StageSmem<real>::bytes(TJ, TK, kp.nvs > NVAR);
  // with the tracer's ring where that fits (227 KB a CTA)
  constexpr size_t full = StageSmem<real>::bytes(TJ, TK, true);
  constexpr size_t most = full <= 227 * 1024 ? full : StageSmem<real>::bytes(TJ, TK);
  if (sl.stage2) {
    raise_smem_limit<k_stage<real, TJ, TK, true>, most>();
    k_stage<real, TJ, TK, true><<<sl.grid, stage_threads(TJ, TK), smem, s>>>(kp, sl, StageConst<real>(kp));
  } else {
    raise_smem_limit<k_stage<real, TJ, TK, false>, most>();
    k_stage<real, TJ, TK, false><<<sl.grid, stage_threads(TJ, TK), smem, s>>>(kp, sl, StageConst<real>(kp));
  }
  return cudaPeekAtLastError() == cudaSuccess ? 0 : -1;
}

// the instantiated tiles
#define STAGE_TILES(X) \
  X(4, 32) X(6, 36) X(8, 8) X(8, 12) X(8, 16) X(8, 24) X(8, 32) X(10, 24) X(12, 12) X(12, 16) X(12, 20) X(16, 16)

template <typename real>
int dispatch(const KParams &kp, const StageLaunch &sl, cudaStream_t s) {
#define X(TJ, TK) \
  if (sl.tile_j == TJ && sl.tile_k == TK) return launch_t<real, TJ, TK>(kp, sl, s);
  STAGE_TILES(X)
#undef X
  return -2;
}

}  // namespace

// This file is compiled twice: k_stage_f64.cu defines STAGE_FP64 and holds the
// FP64 instances only, so that the two sets of kernels compile side by side.
#ifdef STAGE_FP64

int stage_launch_f64(const KParams &kp, const StageLaunch &sl, cudaStream_t s) { return dispatch<double>(kp, sl, s); }

#else

size_t stage_smem_bytes(int precision, int tj, int tk, int tracer) {
  return precision ? StageSmem<float>::bytes(tj, tk, tracer) : StageSmem<double>::bytes(tj, tk, tracer);
}

// an instantiated tile whose shared memory fits one CTA on this device
int stage_tile_supported(int precision, int tj, int tk, int tracer) {
  bool known = false;
#define X(TJ, TK) known = known || (tj == TJ && tk == TK);
  STAGE_TILES(X)
#undef X
  if (!known) return 0;
  int dev = 0, lim = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return 0;
  return stage_smem_bytes(precision, tj, tk, tracer) <= (size_t)lim;
}

int stage_tile(int n, int *tj, int *tk) {
  static const int tiles[][2] = {
#define X(TJ, TK) {TJ, TK},
      STAGE_TILES(X)
#undef X
  };
  if (n < 0 || n >= (int)(sizeof(tiles) / sizeof(tiles[0]))) return 0;
  *tj = tiles[n][0];
  *tk = tiles[n][1];
  return 1;
}

int stage_launch_f64(const KParams &kp, const StageLaunch &sl, cudaStream_t s);

// Resident CTAs of an instance from its shared memory and the registers its
// launch bounds grant (the kernels use close to all of them)
int stage_ctas(int precision, int tj, int tk, int tracer) {
  const int nt = stage_threads(tj, tk);
  const int by_smem = (int)(233472 / (stage_smem_bytes(precision, tj, tk, tracer) + 1024));
  const int regs = precision ? cmin(168, 65536 / (nt * stage_min_ctas(4, tj, tk)) / 8 * 8) : 256;
  return cmax(1, cmin(by_smem, 65536 / (nt * regs)));
}

int stage_launch(const KParams &kp, const StageLaunch &sl, int precision, cudaStream_t s) {
  if (sl.nlist <= 0) return 0;
  return precision ? dispatch<float>(kp, sl, s) : stage_launch_f64(kp, sl, s);
}

#endif
