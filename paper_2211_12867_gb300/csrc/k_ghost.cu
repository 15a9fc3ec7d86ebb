// Ghost-cell fill, reflux and time-step kernels.
//
// Two ghost layers per block (arXiv 2211.12867, Sect. 2.1).  All levels are
// filled at once, in an order in which no cell is read before it is written
// (first launch: copies, restrictions and physical cells; second:
// prolongations; third: the physical cells that come from ghost cells under
// another level).  By what holds a ghost cell:
//   * same-level leaf      -> copy of its interior cell
//   * coarser leaf          -> conservative prolongation: parent value plus
//                             monotonised-central slopes of the conserved
//                             variables times the offset of the child's
//                             volume-weighted centre (falls back to the parent
//                             value when a child's pressure or density would
//                             not be positive)
//   * finer leaves          -> volume-weighted restriction of the 8 children
//   * outside the domain    -> physical boundary: fixed inner boundary map
//                             with the cone CME overlay (Eqs. 1-4),
//                             zero-gradient copy, or reflection; applied per
//                             direction r, theta, phi in that order over the
//                             whole padded slab.
// Reflux: a coarse leaf face next to finer leaves takes the sum of the fine
// area-weighted fluxes of the corrector stage (exact conservation across
// levels on the stretched spherical grid).
#include <algorithm>

#include "mhd_device.cuh"

namespace {

__device__ __forceinline__ int wrap_dim(const KParams &kp, int L, int d, int G, bool &inside) {
  const int N = kp.n_base_cells[d] << (L - 1);
  if (kp.bc_lo[d] == 0) {  // periodic
    inside = true;
    G %= N;
    return G < 0 ? G + N : G;
  }
  inside = G >= 0 && G < N;
  return G;
}

// slot of the level-L leaf holding cell G (>=0), -1 coarser, -2 refined
__device__ __forceinline__ int lookup(const KParams &kp, int member, int L, const int *G) {
  const long long off = kp.lmap_off[member * (MAXLEV + 1) + L];
  const int s = L - 1;
  const int b0 = G[0] / kp.nb[0], b1 = G[1] / kp.nb[1], b2 = G[2] / kp.nb[2];
  const int n1 = kp.nbase[1] << s, n2 = kp.nbase[2] << s;
  return kp.lmap[off + ((long long)b0 * n1 + b1) * n2 + b2];
}

// Slot and padded cell that hold padded index (p0, p1, p2) of leaf `slot`: a
// cell of the ghost layer that a same-level leaf holds is located in that
// leaf's interior.
struct Place {
  size_t base;
  int cell;
};
__device__ __forceinline__ Place locate(const KParams &kp, int slot, int p0, int p1, int p2) {
  const int s0 = p0 < NGH ? -1 : (p0 >= NGH + kp.nb[0] ? 1 : 0);
  const int s1 = p1 < NGH ? -1 : (p1 >= NGH + kp.nb[1] ? 1 : 0);
  const int s2 = p2 < NGH ? -1 : (p2 >= NGH + kp.nb[2] ? 1 : 0);
  if (s0 | s1 | s2) {
    const int o = kp.nb27[(size_t)slot * 27 + (s0 + 1) * 9 + (s1 + 1) * 3 + (s2 + 1)];
    if (o >= 0)
      return {slot_base(kp, o), pad_cell(kp, p0 - s0 * kp.nb[0], p1 - s1 * kp.nb[1], p2 - s2 * kp.nb[2])};
  }
  return {slot_base(kp, slot), pad_cell(kp, p0, p1, p2)};
}

// the variables of a placed cell and, when stored, its tracer (u[TRV])
template <typename real>
__device__ __forceinline__ void fetch(const KParams &kp, const real *U, Place c, real *u) {
  ld_cell(U + c.base + (size_t)NVAR * c.cell, u);
  if (kp.nvs > NVAR) u[TRV] = U[c.base + (size_t)NVAR * kp.pcells + c.cell];
}
template <typename real>
__device__ __forceinline__ void store(const KParams &kp, real *U, Place c, const real *u) {
  st_cell(U + c.base + (size_t)NVAR * c.cell, u);
  if (kp.nvs > NVAR) U[c.base + (size_t)NVAR * kp.pcells + c.cell] = u[TRV];
}

// Conservative prolongation of coarse cell Ic (global at level Lc, held by
// leaf slot cs) into the 2 x 2 x 2 ghost cells of leaf `slot` starting at
// padded index p: child (i, j, k) = parent + MC slopes x offsets; if any
// child's density or pressure is not positive all eight take the parent
// value.  The seven stencil cells are located once (all their loads are
// independent); a first pass checks the eight children, a second writes them
// (one pass that wrote them and undid a failure, and two to eight lanes a
// group, were slower: 267 to 270-274 us the step of 808 leaves of three levels
// that takes two such launches).
template <typename real>
__device__ __forceinline__ void prolong_into(const KParams &kp, real *U, int cs, int Lc, const int *Ic, int slot, const int *p) {
  const DevBlock &C = kp.blk[cs];
  int pc[3];
#pragma unroll
  for (int d = 0; d < 3; d++) pc[d] = Ic[d] - C.ix[d] * kp.nb[d] + NGH;
  // the MHD variables and, when stored, the CME tracer (same slopes and
  // offsets; the positivity decision is the MHD variables')
  const int nv = kp.nvs;
  real up[NVAR + 1], s[3][NVAR + 1];
  fetch(kp, U, {slot_base(kp, cs), pad_cell(kp, pc[0], pc[1], pc[2])}, up);
  {
    real um[3][NVAR + 1], uq[3][NVAR + 1];
#pragma unroll
    for (int d = 0; d < 3; d++) {
      fetch(kp, U, locate(kp, cs, pc[0] - (d == 0), pc[1] - (d == 1), pc[2] - (d == 2)), um[d]);
      fetch(kp, U, locate(kp, cs, pc[0] + (d == 0), pc[1] + (d == 1), pc[2] + (d == 2)), uq[d]);
    }
#pragma unroll
    for (int d = 0; d < 3; d++)
#pragma unroll
      for (int v = 0; v < NVAR + 1; v++)
        if (v < nv) s[d][v] = mc_slope<real>(um[d][v], up[v], uq[d][v]);
  }
  const size_t wbase = slot_base(kp, slot);
  const int w0 = pad_cell(kp, p[0], p[1], p[2]), P1 = kp.P[1], P2 = kp.P[2];
  prolong_children<real>(kp, up, s, Lc, Ic, [&](int c, const real *u) {
    store(kp, U, {wbase, w0 + (((c >> 2) & 1) * P1 + ((c >> 1) & 1)) * P2 + (c & 1)}, u);
  });
}

// slot of the level-L leaf at block coordinates b (>= 0), -1 coarser, -2 refined
__device__ __forceinline__ int lookup_block(const KParams &kp, int member, int L, const int *b) {
  const long long off = kp.lmap_off[member * (MAXLEV + 1) + L];
  const int n1 = kp.nbase[1] << (L - 1), n2 = kp.nbase[2] << (L - 1);
  return kp.lmap[off + ((long long)b[0] * n1 + b[1]) * n2 + b[2]];
}

// volume-weighted mean of the 8 level-(L+1) cells under the level-L cell at
// padded index q of the level-L block b (global cell G); same arithmetic and
// order as the oracle's restriction.  Block sizes are even, so the eight
// children lie in one fine block: one lookup.
template <typename real>
__device__ __forceinline__ bool restrict_in_block(const KParams &kp, const real *U, int member, int L, const int *b, const int *q,
                                  const int *G, real *out) {
  const LevelGeo<real> &F = GeoSel<real>::get(kp.geo, L + 1);
  const int nv = kp.nvs;
  int fb[3], fq[3];
#pragma unroll
  for (int d = 0; d < 3; d++) {
    const int l = 2 * (q[d] - NGH);   // first child, 0 .. 2 nb - 2 within the two fine blocks
    const int hi = l >= kp.nb[d] ? 1 : 0;
    fb[d] = 2 * b[d] + hi;
    fq[d] = l - hi * kp.nb[d] + NGH;
  }
  const int fs = lookup_block(kp, member, L + 1, fb);
  if (fs < 0) return false;
  const size_t fbase = slot_base(kp, fs);
  const int f0 = pad_cell(kp, fq[0], fq[1], fq[2]);
  const int P1 = kp.P[1], P2 = kp.P[2];
  real sum[NVAR + 1];
#pragma unroll
  for (int v = 0; v < NVAR + 1; v++) sum[v] = real(0);
  real vsum = real(0);
  for (int c = 0; c < 8; c++) {
    const int c0 = (c >> 2) & 1, c1 = (c >> 1) & 1, c2 = c & 1;
    const real V = F.dr3[2 * G[0] + c0 + NGH] * F.dcos[2 * G[1] + c1 + NGH] * F.dphi;
    real u[NVAR + 1];
    fetch(kp, U, {fbase, f0 + (c0 * P1 + c1) * P2 + c2}, u);
#pragma unroll
    for (int v = 0; v < NVAR + 1; v++)
      if (v < nv) sum[v] += V * u[v];
    vsum += V;
  }
#pragma unroll
  for (int v = 0; v < NVAR + 1; v++) out[v] = sum[v] / vsum;
  return true;
}

// The ghost fill's work items cover the regions around a leaf (one of the 26,
// r = 9 (sx + 1) + 3 (sy + 1) + sz + 1) that a coarser leaf holds (one lane
// per 2 x 2 x 2 group, prolongation) or finer leaves hold (one lane per cell,
// restriction).  A work item is up to WIDTH such tasks of one region: item =
// (slot, r | finer << 8 | chunk << 9), tasks WIDTH chunk .. WIDTH chunk +
// WIDTH - 1 of the region-ordered shell list (group-first cells first) behind
// its table of (start, group-first cells, cells) per region.  Restrictions
// take a warp each (a face has 2 x 12 x 12 cells), prolongations 8 lanes: an
// edge has 6 groups and a corner one, and with a warp for each 7 of 32 lanes
// worked in the corrector's fill.  5981 leaves of 12^3 on three levels: 79 ->
// 42 us.
// Same-level halo cells the prolongation's stencil reaches are read from
// the neighbouring leaf (the step's fills leave those ghost copies unfilled,
// and the others fill them in the same launch).
struct Task {
  int member, L, slot;
  int p[3];   // padded index in the leaf
  int b[3];   // block across, at the leaf's level
  int q[3];   // padded index in that block
  int G[3];   // global cell
};
template <int WIDTH>
__device__ __forceinline__ bool region_task(const KParams &kp, const int2 e, const int *rshell, Task &t) {
  const int r = e.y & 255, n = (e.y >> 9) * WIDTH + (threadIdx.x & (WIDTH - 1));
  if (n >= rshell[3 * r + 1 + ((e.y >> 8) & 1)]) return false;
  const int code = rshell[81 + rshell[3 * r] + n];
  const DevBlock &B = kp.blk[e.x];
  const int side[3] = {r / 9 - 1, (r / 3) % 3 - 1, r % 3 - 1};
  t.member = B.member;
  t.L = B.level;
  t.slot = e.x;
  t.p[0] = code >> 20;
  t.p[1] = (code >> 10) & 1023;
  t.p[2] = code & 1023;
#pragma unroll
  for (int d = 0; d < 3; d++) {
    // items exist only for neighbours inside the domain or across a
    // periodic direction
    const int nbl = kp.nbase[d] << (t.L - 1);
    int bd = B.ix[d] + side[d];
    if (bd < 0) bd += nbl;
    else if (bd >= nbl) bd -= nbl;
    t.b[d] = bd;
    t.q[d] = t.p[d] - side[d] * kp.nb[d];
    t.G[d] = bd * kp.nb[d] + t.q[d] - NGH;
  }
  return true;
}

// Prolongation items of all levels: latency bound (a chain of five dependent
// loads ahead of the stencil's), so one launch of all levels instead of one a
// level.  A stencil reaches interiors, restricted
// ghost cells and physical ghost cells straight across a face of the coarse
// leaf, all of which the launch before has filled, and never a prolonged one:
// with 2:1 balance over faces, edges and corners a cell within two coarse
// cells of the fine leaf along an axis either touches it, so that its leaf is
// at most one level coarser than the fine one, or lies in the coarse leaf
// itself (blocks are four cells or more).
template <typename real>
__global__ void __launch_bounds__(128, sizeof(real) == 4 ? 5 : 3) k_ghost_prolong(const KParams kp, real *U, const int2 *items, int nitems, const int *rshell) {
  const int w = (blockIdx.x * 128 + threadIdx.x) / PROLONG_WIDTH;
  if (w >= nitems) return;
  Task t;
  if (!region_task<PROLONG_WIDTH>(kp, items[w], rshell, t)) return;
  int cb[3], Ic[3];
#pragma unroll
  for (int d = 0; d < 3; d++) {
    cb[d] = t.b[d] >> 1;
    Ic[d] = t.G[d] >> 1;
  }
  const int cs = lookup_block(kp, t.member, t.L - 1, cb);
  if (cs < 0) {
    atomicOr(kp.status, ST_TREE);
    return;
  }
  prolong_into<real>(kp, U, cs, t.L - 1, Ic, t.slot, t.p);
}

// Inner boundary state (FP64): map of the containing base cell, cone CME
// overlay; u[TRV] = rho X with the CME tracer X = 1 in the CME plasma, else 0.
// A cell is inside the cone where its angle from the axis is at most the
// opening angle acos(arg) of Eqs. 1-4, that is where the angle's cosine is at
// least arg: with the tables of the angles' sines and cosines no
// trigonometric function is left (sin, cos and two acos in FP64 took 19 of the
// pass's 22 us on the 512 x 60 x 180 wedge).
__device__ __forceinline__ void inner_state(const KParams &kp, int member, int L, int J, int K, double t, double *u) {
  double X = 0.0;
  const int n1 = kp.n_base_cells[1], n2 = kp.n_base_cells[2];
  const int jb = J >> (L - 1), kb = K >> (L - 1);
  const double *m = kp.bmap + (size_t)member * NVAR * n1 * n2;
  double w[NVAR];
#pragma unroll
  for (int v = 0; v < NVAR; v++) w[v] = m[((size_t)v * n1 + jb) * n2 + kb];
  const DevCme &c = kp.cme[member];
  if (c.active) {
    const double tau = t - c.t_start;
    if (tau >= 0.0 && tau <= c.t_max) {
      const LevelGeo<double> &G = kp.geo->d[L];
      const DevCone &e = kp.cone[member];
      const double R = G.rf[NGH];
      const double rh = R * e.sin_hw;
      const double Rc = tau * c.v + R - rh;
      const double arg = (Rc * Rc + R * R - rh * rh) / (2.0 * Rc * R);
      const double st = G.sintc[J + NGH];
      const double a = st * e.sin_colat * (G.cosp[K + NGH] * e.cos_lon + G.sinp[K + NGH] * e.sin_lon) +
                       G.costc[J + NGH] * e.cos_colat;
      if (arg >= -1.0 && arg <= 1.0 && fmin(a, 1.0) >= arg) {
        w[0] = c.rho;
        w[1] = c.v;
        w[2] = 0.0;
        w[3] = -kp.omega * R * st;
        w[4] = c.p;
        w[5] = w[6] = w[7] = 0.0;
        X = 1.0;
      }
    }
  }
  prim2cons<double>(w, u, 1.0 / (kp.gamma - 1.0));
  u[TRV] = w[0] * X;
}

// Physical boundaries of all directions; side = (slot, direction * 2 + side),
// idx a cell of its slab.  The boundaries apply in the order r, theta, phi
// over the whole padded slab, each reading what the earlier ones wrote; here a
// ghost cell belongs to its highest physical direction and composes the maps
// of that direction and of the lower ones down to the cell (or inner-boundary
// state) that its value comes from, so no pass waits for another.  faces: only
// the ghost cells inside the block in the two other directions.  The two
// layers of the inner boundary hold one state: a thread writes both.
// part: the cells whose value comes from an interior, a same-level leaf or the
// inner boundary (PHYS_READY) or from a ghost cell under a coarser or finer
// leaf (PHYS_REST).
enum { PHYS_READY = 1, PHYS_REST = 2 };
template <typename real>
__device__ __forceinline__ void physical_cell(const KParams &kp, real *U, const int2 sd, int idx, double tfac,
                                              int faces, int part) {
  const int slot = sd.x, dir = sd.y >> 1, side = sd.y & 1;
  const int da = dir == 0 ? 1 : 0, db = dir == 2 ? 1 : 2;
  const int Pa = faces ? kp.nb[da] : kp.P[da], Pb = faces ? kp.nb[db] : kp.P[db], off = faces ? NGH : 0;
  const bool inner = (side ? kp.bc_hi[dir] : kp.bc_lo[dir]) == 3;
  if (idx >= (inner ? 1 : NGH) * Pa * Pb) return;
  const int gl = idx / (Pa * Pb), r = idx - gl * (Pa * Pb), a = r / Pb + off, b = r - (r / Pb) * Pb + off;
  const DevBlock &B = kp.blk[slot];
  const int phys = B.phys, L = B.level;
  int q[3];
  q[dir] = side ? NGH + kp.nb[dir] + gl : NGH - 1 - gl;
  q[da] = a;
  q[db] = b;
  int s[3] = {q[0], q[1], q[2]};
  unsigned flip = 0;
  bool at_inner = false;
#pragma unroll
  for (int d = 2; d >= 0; d--) {
    const int nb = kp.nb[d];
    const int lo = s[d] < NGH && (phys >> (2 * d) & 1), hi = s[d] >= NGH + nb && (phys >> (2 * d + 1) & 1);
    if (!(lo | hi)) continue;
    if (d > dir) return;   // a higher direction's cell
    const int bc = hi ? kp.bc_hi[d] : kp.bc_lo[d];
    if (bc == 3) {
      at_inner = true;
    } else if (bc == 2) {
      s[d] = hi ? 2 * (NGH + nb) - 1 - s[d] : 2 * NGH - 1 - s[d];
      flip ^= 1u << d;
    } else {
      s[d] = hi ? NGH + nb - 1 : NGH;
    }
  }
  {
    bool ready = at_inner;
    if (!ready) {
      int r = 0;
#pragma unroll
      for (int d = 0; d < 3; d++) r = 3 * r + (s[d] < NGH ? 0 : (s[d] >= NGH + kp.nb[d] ? 2 : 1));
      ready = r == 13 || kp.nb27[(size_t)slot * 27 + r] >= 0;
    }
    if (ready != (part == PHYS_READY)) return;
  }
  real x[NVAR + 1];
  if (at_inner) {
    bool in;
    const int J = wrap_dim(kp, L, 1, B.ix[1] * kp.nb[1] + s[1] - NGH, in);
    const int K = wrap_dim(kp, L, 2, B.ix[2] * kp.nb[2] + s[2] - NGH, in);
    const double t = kp.t[B.member] + tfac * kp.dt_used[B.member];
    double u[NVAR + 1];
    inner_state(kp, B.member, L, J, K, t, u);
#pragma unroll
    for (int v = 0; v < NVAR + 1; v++) x[v] = (real)u[v];
  } else {
    fetch(kp, U, locate(kp, slot, s[0], s[1], s[2]), x);
  }
#pragma unroll
  for (int d = 0; d < 3; d++)
    if (flip >> d & 1) {
      x[1 + d] = -x[1 + d];
      x[5 + d] = -x[5 + d];
    }
  store(kp, U, {slot_base(kp, slot), pad_cell(kp, q[0], q[1], q[2])}, x);
  if (inner) store(kp, U, {slot_base(kp, slot), pad_cell(kp, 0, q[1], q[2])}, x);
}

// the physical cells left by k_ghost_first, after the prolongation
template <typename real>
__global__ void __launch_bounds__(128) k_ghost_physical(const KParams kp, real *U, const int2 *sides, double tfac,
                                                        int faces) {
  physical_cell(kp, U, sides[blockIdx.x], blockIdx.y * 128 + threadIdx.x, tfac, faces, PHYS_REST);
}

// First launch of a ghost fill, all levels: restriction items (the first
// rblocks CTAs), the physical ghost cells that come from interiors (nchunk
// CTAs a side), and, in the fills that cover them, copies from same-level
// leaves (ccopy CTAs a leaf; shell: the padded (p0, p1, p2) of a block's ghost
// cells packed as p0 << 20 | p1 << 10 | p2).  None reads what another writes.
template <typename real>
__global__ void __launch_bounds__(128) k_ghost_first(const KParams kp, real *U, const int2 *items, int nitems,
                                                     const int *rshell, int rblocks, const int2 *sides, int nsides,
                                                     int nchunk, double tfac, int faces, const int *shell, int nshell,
                                                     int ccopy) {
  int n = blockIdx.x;
  if (n < rblocks) {
    const int w = (n * 128 + threadIdx.x) / RESTRICT_WIDTH;
    if (w >= nitems) return;
    Task t;
    if (!region_task<RESTRICT_WIDTH>(kp, items[w], rshell, t)) return;
    real val[NVAR + 1];
    if (!restrict_in_block<real>(kp, U, t.member, t.L, t.b, t.q, t.G, val)) {
      atomicOr(kp.status, ST_TREE);
      return;
    }
    store(kp, U, {slot_base(kp, t.slot), pad_cell(kp, t.p[0], t.p[1], t.p[2])}, val);
    return;
  }
  n -= rblocks;
  if (n < nsides * nchunk) {
    const int s = n / nchunk;
    physical_cell(kp, U, sides[s], (n - s * nchunk) * 128 + threadIdx.x, tfac, faces, PHYS_READY);
    return;
  }
  n -= nsides * nchunk;
  const int slot = n / ccopy, c = (n - slot * ccopy) * 128 + threadIdx.x;
  if (c >= nshell) return;
  const int code = shell[c], p0 = code >> 20, p1 = (code >> 10) & 1023, p2 = code & 1023;
  const Place from = locate(kp, slot, p0, p1, p2), to = {slot_base(kp, slot), pad_cell(kp, p0, p1, p2)};
  if (from.base == to.base && from.cell == to.cell) return;   // not a same-level leaf's
  real val[NVAR + 1];
  fetch(kp, U, from, val);
  store(kp, U, to, val);
}

// sum over the directions of (|v_d| + c_f,d) / dx_d of a cell.  FP64: with the
// stage's reciprocals and roots (IEEE divisions and roots cost k_dt_full of 204
// leaves of 12^3 109 us, now 76)
__device__ __forceinline__ float speed_sum(const float *u, float gamma, float pfl, float dx0, float dx1, float dx2) {
  float w[NVAR];
  cons2prim_speed<float>(u, w, gamma, pfl);
  return (RT<float>::abs_(w[1]) + fast_speed<float, 0>(w, gamma)) / dx0 +
         (RT<float>::abs_(w[2]) + fast_speed<float, 1>(w, gamma)) / dx1 +
         (RT<float>::abs_(w[3]) + fast_speed<float, 2>(w, gamma)) / dx2;
}
__device__ __forceinline__ double speed_sum(const double *u, double gamma, double pfl, double dx0, double dx1, double dx2) {
  const double ir = RT<double>::rcp_(u[0]);
  double p = pressure_for_speed<double>(u, gamma);
  if (RT<double>::less_(p, pfl)) p = pfl;
  const double v[3] = {u[1] * ir, u[2] * ir, u[3] * ir};
  const double ix[3] = {RT<double>::rcp_(dx0), RT<double>::rcp_(dx1), RT<double>::rcp_(dx2)};
  return cfl_rate(ir, v, p, u + 5, gamma, ix);
}

// Reflux of the leaves with a finer face neighbour: one thread per cell of a
// face (blockIdx.y: chunks of 128 cells of the faces in order).  A cell on
// several finer faces belongs to the first one's thread, which corrects it
// face by face and then takes floors and CFL speed as often.  Latency bound
// (lookups, then 5 x 8 flux loads at once).  A CTA per leaf that went through
// its faces one after the other, with four lookups a coarse face instead of
// one, took 24 us between events on a tree of 1914 leaves of 12^3 (FP32) and 29
// on one of 204 (FP64); now 17 and 24.
template <typename real>
__global__ void __launch_bounds__(128) k_reflux(const KParams kp, real *U, const real *flux, const int *list) {
  const int slot = list[blockIdx.x];
  const DevBlock &B = kp.blk[slot];
  const int fc[3] = {kp.nb[1] * kp.nb[2], kp.nb[0] * kp.nb[2], kp.nb[0] * kp.nb[1]};
  int f = 0, chunk = blockIdx.y;
#pragma unroll
  for (int q = 0; q < 5; q++) {
    const int n = (fc[q / 2] + 127) / 128;
    if (f == q && chunk >= n) {
      chunk -= n;
      f = q + 1;
    }
  }
  const double dtm = kp.dt_used[B.member];
  if (B.nbr[f] != NB_FINER || !(dtm > 0.0)) return;
  const real dt = (real)dtm;
  const int L = B.level;
  const size_t fstride = (size_t)NVAR * 2 * (fc[0] + fc[1] + fc[2]);
  const LevelGeo<real> &G = GeoSel<real>::get(kp.geo, L);
  const real gamma = (real)kp.gamma, pfl = (real)kp.p_floor, rfl = (real)kp.rho_floor;
  double acc = 0.0;
  int hits = 0;
  int q[3];   // the cell inside the leaf
  const int t = chunk * 128 + threadIdx.x;
  {
    const int d = f / 2, d1 = d == 0 ? 1 : 0, d2 = d == 2 ? 1 : 2;
    q[d] = f % 2 ? kp.nb[d] - 1 : 0;
    q[d1] = t / kp.nb[d2];
    q[d2] = t - q[d1] * kp.nb[d2];
  }
  unsigned on = 0;   // finer faces the cell lies on
#pragma unroll
  for (int e = 0; e < 6; e++)
    if (B.nbr[e] == NB_FINER && q[e / 2] == (e % 2 ? kp.nb[e / 2] - 1 : 0)) on |= 1u << e;
  if (t < fc[f / 2] && !(on & ((1u << f) - 1))) {
    const int I = B.ix[0] * kp.nb[0] + q[0], J = B.ix[1] * kp.nb[1] + q[1];
    const real V = G.dr3[I + NGH] * G.dcos[J + NGH] * G.dphi;
    const size_t ci = cell_index(kp, slot, q[0] + NGH, q[1] + NGH, q[2] + NGH);
    real u[NVAR];
    ld_cell(U + ci, u);
    for (unsigned m = on; m; m &= m - 1) {
      const int e = __ffs(m) - 1, d = e / 2, hi = e & 1, d1 = d == 0 ? 1 : 0, d2 = d == 2 ? 1 : 2;
      size_t off = 0;   // of the face's fluxes in a slot; low and high face
      for (int p = 0; p < d; p++) off += (size_t)2 * NVAR * fc[p];
      const size_t face = (size_t)NVAR * fc[d];
      // the fine leaf across and its cell next to the coarse cell's corner
      // (blocks start at even indices: all four fine cells lie in it)
      int F[3];
#pragma unroll
      for (int p = 0; p < 3; p++) F[p] = 2 * (B.ix[p] * kp.nb[p] + q[p]);
      F[d] += hi ? 2 : -1;
      bool in;
#pragma unroll
      for (int p = 0; p < 3; p++) F[p] = wrap_dim(kp, L + 1, p, F[p], in);
      const int fsl = lookup(kp, B.member, L + 1, F);
      real fs[NVAR];
#pragma unroll
      for (int v = 0; v < NVAR; v++) fs[v] = real(0);
      if (fsl < 0) {
        atomicOr(kp.status, ST_TREE);
      } else {
        const DevBlock &FB = kp.blk[fsl];
        const int s1 = F[d1] - FB.ix[d1] * kp.nb[d1], s2 = F[d2] - FB.ix[d2] * kp.nb[d2];
        const real *src = flux + (size_t)fsl * fstride + off + (hi ? 0 : face) + s1 * kp.nb[d2] + s2;
#pragma unroll
        for (int a = 0; a < 2; a++)
#pragma unroll
          for (int c = 0; c < 2; c++)
#pragma unroll
            for (int v = 0; v < NVAR; v++) fs[v] += src[(size_t)v * fc[d] + a * kp.nb[d2] + c];
      }
      const real *own = flux + (size_t)slot * fstride + off + (hi ? face : 0) + q[d1] * kp.nb[d2] + q[d2];
      const real sg = hi ? real(-1) : real(1);
#pragma unroll
      for (int v = 0; v < NVAR; v++) u[v] += sg * dt / V * (fs[v] - own[(size_t)v * fc[d]]);
    }
    real dx0 = G.dr[I + NGH], dx1 = G.dth[J + NGH], dx2 = G.dphi;
    if (kp.geometry == 0) {
      dx1 *= G.rc[I + NGH];
      dx2 *= G.rc[I + NGH] * G.sintc[J + NGH];
    }
    for (unsigned m = on; m; m &= m - 1) {
      hits += apply_floors<real>(u, gamma, pfl, rfl, Isl{(float)kp.isl_pe, (float)kp.isl_beta});
      acc = fmax(acc, (double)speed_sum(u, gamma, pfl, dx0, dx1, dx2));
    }
    st_cell(U + ci, u);
  }
  for (int o = 16; o > 0; o >>= 1) {
    acc = fmax(acc, __shfl_xor_sync(0xffffffffu, acc, o));
    hits += __shfl_xor_sync(0xffffffffu, hits, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (acc > 0.0) atomic_max_pos(&kp.inv_max[B.member], acc);
    if (hits) atomicAdd(kp.floor_hits, (unsigned long long)hits);
  }
}

// the step a member takes next (none once it has reached its stop time)
__device__ __forceinline__ double next_dt(const KParams &kp, int m, const double *tstop) {
  const double dt = fmin(kp.dt_cfl[m], tstop[m] - kp.t[m]);
  return dt > 0.0 ? dt : 0.0;
}

__global__ void k_dt_begin(const KParams kp, const double *tstop) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= kp.n_members) return;
  kp.dt_used[m] = next_dt(kp, m, tstop);
}

// End of a step: times, CFL step of the new state, and the next step's dt (so
// that only the first step of a call has a launch for it)
__global__ void k_dt_finalize(const KParams kp, double cfl, const double *tstop) {
  const int m = threadIdx.x;
  if (m == 0) {
    // floor budget: the floors the step applied (both stages) against the
    // leaf cells it advanced
    const unsigned long long h = *kp.floor_hits, d = h - *kp.floor_prev;
    *kp.floor_prev = h;
    if (kp.floor_budget > 0.0 && d > 0) {
      double cells = 0.0;
      for (int q = 0; q < kp.n_members; q++)
        if (kp.dt_used[q] > 0.0) cells += kp.cells_m[q];
      if ((double)d > kp.floor_budget * cells) atomicOr(kp.status, ST_FLOOR);
    }
  }
  __syncthreads();   // the budget has read every member's step
  for (int q = m; q < kp.n_members; q += blockDim.x) {
    const double dt = kp.dt_used[q];
    if (dt > 0.0) {
      kp.t[q] += dt;
      kp.updates[q] += kp.cells_m[q];
      const double inv = __longlong_as_double((long long)kp.inv_max[q]);
      if (inv > 0.0) kp.dt_cfl[q] = cfl / inv;
    }
    kp.inv_max[q] = 0ull;
    kp.dt_used[q] = next_dt(kp, q, tstop);
  }
}

// CFL time step of the whole current state (after set_state / regrid / init)
template <typename real>
__global__ void k_dt_full(const KParams kp, const real *U) {
  const int slot = blockIdx.x;
  const DevBlock B = kp.blk[slot];
  const LevelGeo<real> &G = GeoSel<real>::get(kp.geo, B.level);
  const real gamma = (real)kp.gamma, pfl = (real)kp.p_floor;
  double acc = 0.0;
  for (int c = blockIdx.y * blockDim.x + threadIdx.x; c < kp.icells; c += gridDim.y * blockDim.x) {
    const int k = c % kp.nb[2], j = (c / kp.nb[2]) % kp.nb[1], i = c / (kp.nb[2] * kp.nb[1]);
    real u[NVAR];
    ld_cell(U + cell_index(kp, slot, i + NGH, j + NGH, k + NGH), u);
    const int I = B.ix[0] * kp.nb[0] + i + NGH, J = B.ix[1] * kp.nb[1] + j + NGH;
    real dx0 = G.dr[I], dx1 = G.dth[J], dx2 = G.dphi;
    if (kp.geometry == 0) {
      dx1 *= G.rc[I];
      dx2 *= G.rc[I] * G.sintc[J];
    }
    acc = fmax(acc, (double)speed_sum(u, gamma, pfl, dx0, dx1, dx2));
  }
  for (int o = 16; o > 0; o >>= 1) acc = fmax(acc, __shfl_xor_sync(0xffffffffu, acc, o));
  if ((threadIdx.x & 31) == 0 && acc > 0.0) atomic_max_pos(&kp.inv_max[B.member], acc);
}

__global__ void k_dt_from_max(const KParams kp, double cfl) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= kp.n_members) return;
  const double inv = __longlong_as_double((long long)kp.inv_max[m]);
  kp.dt_cfl[m] = inv > 0.0 ? cfl / inv : 0.0;
  kp.inv_max[m] = 0ull;
}

}  // namespace

namespace {
// chunks of 128 cells of the largest slab that can be physical
int physical_chunks(const KParams &kp, bool faces_only) {
  int n = 0;
  for (int d = 0; d < 3; d++) {
    if (kp.bc_lo[d] == 0) continue;
    const int da = d == 0 ? 1 : 0, db = d == 2 ? 1 : 2;
    const int c = NGH * (faces_only ? kp.nb[da] * kp.nb[db] : kp.P[da] * kp.P[db]);
    n = c > n ? c : n;
  }
  return (n + 127) / 128;
}
}  // namespace

void ghost_first_launch(const KParams &kp, void *U, int precision, const int2 *items, int nitems, const int *rshell,
                        const int2 *sides, int nsides, double tfac, bool faces_only, const int *shell, int nshell,
                        int nleaves, cudaStream_t s) {
  const int nchunk = physical_chunks(kp, faces_only), rblocks = (nitems * RESTRICT_WIDTH + 127) / 128;
  const int ccopy = (nshell + 127) / 128, grid = rblocks + nsides * nchunk + nleaves * ccopy;
  if (grid <= 0) return;
  if (precision)
    k_ghost_first<float><<<grid, 128, 0, s>>>(kp, (float *)U, items, nitems, rshell, rblocks, sides, nsides, nchunk, tfac,
        faces_only, shell, nshell, ccopy);
  else
    k_ghost_first<double><<<grid, 128, 0, s>>>(kp, (double *)U, items, nitems, rshell, rblocks, sides, nsides, nchunk, tfac,
        faces_only, shell, nshell, ccopy);
}

void ghost_prolong_launch(const KParams &kp, void *U, int precision, const int2 *items, int nitems, const int *rshell,
                          cudaStream_t s) {
  if (nitems <= 0) return;
  const int grid = (nitems * PROLONG_WIDTH + 127) / 128;
  if (precision)
    k_ghost_prolong<float><<<grid, 128, 0, s>>>(kp, (float *)U, items, nitems, rshell);
  else
    k_ghost_prolong<double><<<grid, 128, 0, s>>>(kp, (double *)U, items, nitems, rshell);
}

void ghost_physical_launch(const KParams &kp, void *U, int precision, const int2 *sides, int nsides, double tfac,
                           bool faces_only, cudaStream_t s) {
  if (nsides <= 0) return;
  dim3 grid(nsides, physical_chunks(kp, faces_only));
  if (precision)
    k_ghost_physical<float><<<grid, 128, 0, s>>>(kp, (float *)U, sides, tfac, faces_only);
  else
    k_ghost_physical<double><<<grid, 128, 0, s>>>(kp, (double *)U, sides, tfac, faces_only);
}

void reflux_launch(const KParams &kp, void *U, const void *flux, int precision, const int *list, int nlist,
                   cudaStream_t s) {
  if (nlist <= 0) return;
  const int *n = kp.nb;
  const int chunks = 2 * ((n[1] * n[2] + 127) / 128 + (n[0] * n[2] + 127) / 128 + (n[0] * n[1] + 127) / 128);
  const dim3 grid(nlist, chunks);
  if (precision)
    k_reflux<float><<<grid, 128, 0, s>>>(kp, (float *)U, (const float *)flux, list);
  else
    k_reflux<double><<<grid, 128, 0, s>>>(kp, (double *)U, (const double *)flux, list);
}

void dt_begin_launch(const KParams &kp, const double *tstop, cudaStream_t s) {
  k_dt_begin<<<(kp.n_members + 127) / 128, 128, 0, s>>>(kp, tstop);
}

void dt_finalize_launch(const KParams &kp, double cfl, const double *tstop, cudaStream_t s) {
  const int n = kp.n_members < 1024 ? (kp.n_members + 31) / 32 * 32 : 1024;
  k_dt_finalize<<<1, n, 0, s>>>(kp, cfl, tstop);
}

void dt_full_launch(const KParams &kp, const void *U, int precision, int nleaves, double cfl, cudaStream_t s) {
  if (nleaves > 0) {
    // cells a CTA: in FP32, where a cell is cheap against a CTA's start and
    // reduction, 4096 (2481 leaves of 12^3: 39 us; with 1024, 44); more in a
    // block that would take more CTAs than a grid has rows
    const int per = precision ? 4096 : 1024;
    const dim3 grid(nleaves, std::min((kp.icells + per - 1) / per, 65535));
    if (precision)
      k_dt_full<float><<<grid, 256, 0, s>>>(kp, (const float *)U);
    else
      k_dt_full<double><<<grid, 256, 0, s>>>(kp, (const double *)U);
  }
  k_dt_from_max<<<(kp.n_members + 127) / 128, 128, 0, s>>>(kp, cfl);
}
