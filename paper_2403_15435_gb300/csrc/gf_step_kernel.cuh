// The patch-step kernel, templated on the precision policy:
//   PrecF64 -- plain FP64 state (h, hu, hv) and bed b;
//   PrecF32 -- FP32 surface-deviation state (w = h + b - eta0, hu, hv) with
//              FP32 compensation terms for the update, bed b - eta0, exact
//              wet tests (FP32 with an FP64 tie-break) and FP64 volume sums.
//
// One CTA per patch, or per sub-tile of one.  The (M+4)^2 tile of the state
// and bed is staged in shared memory (whole patches by 1D TMA bulk copies);
// then, in barrier-separated phases:
// every x-edge's augmented Riemann solve (Sec. 3.3), the MC-limited f-wave
// corrections (Sec. 3.2, Eq. wpa_update_corrections), the per-cell x
// increments and their transverse split along y (2D extension, leveque2002
// cited in Sec. 3.2), the same for y, the unsplit update, Manning friction
// (Eq. manning), and the per-patch CFL rate (warp-shuffle max) and volume.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "gf_internal.h"
#include "gf_solver.cuh"

namespace gfs {

struct PrecF64 {
  using R = double;
  static constexpr bool DEV = false;
};
struct PrecF32 {
  using R = float;
  static constexpr bool DEV = true;
};

__device__ __forceinline__ unsigned smem_addr(const void* p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(count)
               : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile(
      "mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
          smem_addr(bar)),
      "r"(bytes)
      : "memory");
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src,
                                         unsigned bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes "
      "[%0], [%1], %2, [%3];" ::"r"(smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// Ask for `bytes` (a multiple of 16) at a 16-byte aligned address in L2.
__device__ __forceinline__ void bulk_prefetch(const void* src, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

// Bounded wait for the completion of the barrier's phase with the given
// parity; returns false on timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned limit,
                                          unsigned parity = 0u) {
  for (unsigned it = 0; it < limit; ++it) {
    unsigned done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], "
        "%2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// Phases of the two staging barriers of a CTA that stages one tile after
// another: the parity each barrier completes next.
struct TmaPhase {
  unsigned b0, b1;
  bool init;
};

// What a tile's chain of loads starts from, read by the kernel in as few
// round trips as possible.
struct TileHdr {
  GfPatch Pt;
  int cur, accepted;
  double dt;      // dt_use
  bool same_in;   // both buffers hold the same dry interior
  bool has_gauge;
  int* order;     // the next launch order (or null: another CTA enters the patch)
};

// Counters of a launch order that is being written (GfView::sched): [0] its
// head, [1] its tail.
__device__ __forceinline__ unsigned* order_ends(const GfView& V, const int* order) {
  return V.sched + (order == V.ord0 ? 3 : 1);
}

template <typename R>
__device__ __forceinline__ R warp_max(R v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const R w = __shfl_xor_sync(0xffffffffu, v, o);
    if constexpr (sizeof(R) == 8) v = gfk::dmax(v, w);
    else v = v > w ? v : w;
  }
  return v;
}

__device__ __forceinline__ double warp_sum_tree(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Patches that took no step in the previous launch share a CTA in groups of
// this many.  Valley of 10496 patches, 5480 of them dry: their CTAs, two to an
// SM because of the wet tiles' shared memory, were 43 of a launch's 358 us.
#define GF_STEP_GROUP 16

constexpr size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

// Writes that follow a new value (v0, v1, v2) of cell (gi, gj) of patch p
// (patch position (px, py); nxp x nyp patches on its level), other than the
// cell itself, into the next buffer: the ghost cells of the same-level
// neighbours (snb, one writer per ghost cell) that copy it, and the
// physical-boundary ghost cells of p or of those neighbours that mirror it
// (wall: reflected across the edge with the normal momentum negated;
// extrapolation: the edge cell copied into both ghost layers).  A boundary
// ghost whose mirror source is a neighbour's cell is written by that
// neighbour, so no ghost depends on another CTA's writes in the same launch.
template <typename R, int MP>
__device__ __forceinline__ void emit_edge(R* qnext, int p, int px, int py,
                                          int nxp, int nyp, const int* snb,
                                          const int* bc, bool push, int gi,
                                          int gj, R v0, R v1, R v2) {
  constexpr int TGW = MP + 2 * GF_NG, TG = TGW * TGW;
  if (gi >= GF_NG && gi < MP - GF_NG && gj >= GF_NG && gj < MP - GF_NG) return;
  auto target = [&](int q, int qx, int qy, int x, int y, bool self) {
    R* base = qnext + (size_t)q * 3 * TG;
    auto put = [&](int a, int b, R su, R sv) {
      R* d = base + (a + GF_NG) + (b + GF_NG) * TGW;
      d[0] = v0;
      d[TG] = su * v1;
      d[2 * TG] = sv * v2;
    };
    int xm[2], ym[2], nx = 0, ny = 0;
    R fx = R(1), fy = R(1);
    if (qx == 0 && (x == 0 || x == 1)) {
      if (bc[0] == 0) { xm[nx++] = -1 - x; fx = R(-1); }
      else if (x == 0) { xm[nx++] = -1; xm[nx++] = -2; }
    } else if (qx == nxp - 1 && (x == MP - 1 || x == MP - 2)) {
      if (bc[1] == 0) { xm[nx++] = 2 * MP - 1 - x; fx = R(-1); }
      else if (x == MP - 1) { xm[nx++] = MP; xm[nx++] = MP + 1; }
    }
    if (qy == 0 && (y == 0 || y == 1)) {
      if (bc[2] == 0) { ym[ny++] = -1 - y; fy = R(-1); }
      else if (y == 0) { ym[ny++] = -1; ym[ny++] = -2; }
    } else if (qy == nyp - 1 && (y == MP - 1 || y == MP - 2)) {
      if (bc[3] == 0) { ym[ny++] = 2 * MP - 1 - y; fy = R(-1); }
      else if (y == MP - 1) { ym[ny++] = MP; ym[ny++] = MP + 1; }
    }
    if (!self) put(x, y, R(1), R(1));
    for (int a = 0; a < nx; ++a) put(xm[a], y, fx, R(1));
    for (int b = 0; b < ny; ++b) put(x, ym[b], R(1), fy);
    for (int a = 0; a < nx; ++a)
      for (int b = 0; b < ny; ++b) put(xm[a], ym[b], fx, fy);
  };
  target(p, px, py, gi, gj, true);
  if (!push) return;
  const int dxs = gi < GF_NG ? -1 : (gi >= MP - GF_NG ? 1 : 0);
  const int dys = gj < GF_NG ? -1 : (gj >= MP - GF_NG ? 1 : 0);
  auto nb = [&](int r, int dx, int dy) {
    const int pn = snb[r];
    if (pn >= 0) target(pn, px + dx, py + dy, gi - dx * MP, gj - dy * MP, false);
  };
  if (dxs != 0) nb(dxs < 0 ? 0 : 1, dxs, 0);
  if (dys != 0) nb(dys < 0 ? 2 : 3, 0, dys);
  if (dxs != 0 && dys != 0) nb(4 + (dxs > 0 ? 1 : 0) + (dys > 0 ? 2 : 0), dxs, dys);
}

// Gauge samples of the state this launch starts from (the previous launch's
// accepted result, at time C->t), taken from the CTA's staged window: the
// window covers patch cells [ox - 2, ox + WM + 1]^2; a gauge whose stencil
// starts in sub-tile (ox, oy) is taken by that window's CTA.  mom = false:
// the momenta were not staged (a dry tile, where they are zero).
template <typename R, bool DEV, int MP, int WM>
__device__ __forceinline__ void sample_gauges(const GfView& V, int scen, const GfCtl* C,
                                              int p, int ox, int oy, const R* s0,
                                              const R* shu, const R* shv, const R* sb,
                                              bool mom) {
  constexpr int TGW = MP + 2 * GF_NG, WW = WM + 2 * GF_NG;
  const GfScenario& S = V.scen[scen];
  for (int g = threadIdx.x; g < S.ngauge; g += blockDim.x) {
    const GfGaugeRef r = S.gref[g];
    if (r.p != p) continue;
    const int i0 = r.c % TGW - GF_NG, j0 = r.c / TGW - GF_NG;
    const int ic = i0 < 0 ? 0 : i0, jc = j0 < 0 ? 0 : j0;
    if ((ic / WM) * WM != ox || (jc / WM) * WM != oy) continue;
    const int c = (i0 - ox + GF_NG) + (j0 - oy + GF_NG) * WW;
    const int cs[4] = {c, c + 1, c + WW, c + WW + 1};
    double a[4][4];  // h, hu, hv, h + b per stencil cell
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double b = (double)sb[cs[k]];
      const double h = DEV ? (double)s0[cs[k]] - b : (double)s0[cs[k]];
      a[k][0] = h;
      a[k][1] = mom ? (double)shu[cs[k]] : 0.0;
      a[k][2] = mom ? (double)shv[cs[k]] : 0.0;
      a[k][3] = h + b;
    }
    double v[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) v[f] = gf_bilinear(a[0][f], a[1][f], a[2][f], a[3][f], r.ax, r.ay);
    double* o = S.gout + 5 * g;
    const double t = C->t;
    o[0] = t;
    o[1] = v[0];
    o[2] = v[1];
    o[3] = v[2];
    o[4] = v[3] + (DEV ? S.eta0 : 0.0);
    if (S.garr[g] < 0.0 && v[0] > 0.01) S.garr[g] = t;
  }
}

// Shared-memory layout of one CTA.  DS = dimensional splitting: the x sweep
// covers every row of the window (two ghost rows each side) and there are no
// transverse-flux arrays.
template <class P, int M, bool DS = false>
struct Layout {
  using R = typename P::R;
  static constexpr int T = M + 2 * GF_NG;
  static constexpr int TT = T * T;
  // most lines in one sweep: one ghost line each side (unsplit) or two
  static constexpr int NR = DS ? M + 4 : M + 2;
  static constexpr int NE = M + 3;  // edges per line, a in [-1, M+1]
  // places of a wave plane.  FP32, unsplit: rows of pitch M + 4, so that
  // pairs of edges are 8-byte aligned
  static constexpr bool FAST = P::DEV && !DS;
  static constexpr int NEDGE = FAST ? (M + 3) * (M + 4) : NR * NE;
  static constexpr int NLIM = NR * (M + 1);   // edges a in [0, M] per line
  static constexpr int NCELL = M * NR;        // cells of the increments
  // FP64, unsplit: per-cell primitives beside the state (surface, two
  // velocities, celerity, root of the depth) and 11 wave planes
  static constexpr bool PRIM = !P::DEV && !DS;
  // FP32, unsplit: velocities and root of the depth beside the state, 10
  // wave planes, 6 planes of transverse parts
  static constexpr int NF = FAST ? 7 : (P::DEV ? 5 : (PRIM ? 9 : 4));  // tile fields
  static constexpr int NWP = FAST ? 10 : (PRIM ? 11 : 12);             // wave planes
  static constexpr size_t TRB =
      DS ? 0 : (FAST ? sizeof(R) * 3 * M * (M + 4) : sizeof(R) * 3 * M * (M + 1));
  // byte offsets in dynamic shared memory
  static constexpr size_t OFF_W = sizeof(R) * NF * TT;
  // FP64 8 x 8 sub-tiles: half the threads take the x sweep while the others
  // take the y sweep, each half with wave planes of its own
  static constexpr bool BOTH = PRIM && M == 8;
  static constexpr size_t OFF_F = OFF_W + sizeof(R) * NWP * NEDGE * (BOTH ? 2 : 1);
  static constexpr size_t OFF_G = OFF_F + TRB;
  static constexpr size_t OFF_RED = align16(OFF_G + TRB);
  static constexpr size_t OFF_NB = OFF_RED + sizeof(double) * 64;  // 8 ints
  static constexpr size_t OFF_WET = OFF_NB + 32;
  // FAST, whole 32 x 32 tiles: edges set aside: their number, then their places
  static constexpr int ASIDE = FAST && M == 32 ? 240 : 0;
  static constexpr size_t OFF_ASIDE = align16(OFF_WET + (P::DEV && DS ? TT : 16));
  static constexpr size_t OFF_BAR = align16(OFF_ASIDE + (FAST ? 4 + 2 * ASIDE : 0));
  static constexpr size_t BYTES = OFF_BAR + 16;
};

template <int M>
__device__ __forceinline__ int tix(int i, int j) {
  return (i + GF_NG) + (j + GF_NG) * (M + 2 * GF_NG);
}

// Increment cell of item k in a split sweep over NRL lines: items below M*M are
// interior cells in the fixed order (i = k % M, j = k / M) used by the final
// update, so each thread owns the same cells in both sweeps; then the ghost
// lines before the interior (from line L0 on) and those after it.  a is the
// position along the sweep, line the one across.
template <int M, int NRL, int L0>
__device__ __forceinline__ void cell_item(int k, int dir, int& a, int& line) {
  if (k < M * M) {
    const int i = k % M, j = k / M;
    a = dir == 0 ? i : j;
    line = dir == 0 ? j : i;
  } else {
    constexpr int HALF = (NRL - M) / 2;
    const int r = k - M * M, gl = r / M;
    a = r % M;
    line = gl < HALF ? L0 + gl : M + (gl - HALF);
  }
}

// M is the side of the sub-tile this CTA updates, MP the side of the patch:
// a patch of MP x MP cells is covered by (MP/M)^2 CTAs, each staging its
// (M+4)^2 window (interior + two ghost layers, taken from the patch tile,
// whose ghosts are filled) and writing its M x M cells.  Every cell's update
// depends only on its two-cell neighbourhood, so the result does not depend
// on M.
//
// FP64 (unsplit): the FP64 pipe (two operations per SM and clock) bounds the
// step, so the body computes a cell's velocities, celerity and root of the
// depth once (not once per edge side) and leaves only additions and products
// to that pipe (gf_fp64.cuh).  Both sweeps share one copy of the code and the
// quotients and roots are calls, since instruction fetch shows too; 8 x 8
// sub-tiles take both sweeps at once.  1024 x 1024 radial dam break, 36 % wet:
// 1770 -> 520 FP64-pipe operations per wet cell, 1060 -> 470 us per step (ncu:
// FP64 pipe 82 % busy before, 65 % after, the rest barrier waits between the
// phases); a 64 x 64 basin 270 -> 30 us per step.
//
// FP32 (unsplit): bound by issue slots and by the tile's chain of barriers
// (115 KB of shared memory allow two whole tiles per SM).  A thread takes two
// neighbouring edges or cells: packed instructions for their arithmetic, one
// index and one 8-byte shared-memory access for both; the cell's velocities
// and root of the depth are computed once per cell while its state is looked
// at; the six transverse parts of a cell are written once and read by its
// neighbours; the copies of the edge cells follow the update side by side.
// 4 km x 2 km valley, 10496 patches, 5012 of them with water: 269 M -> 191 M
// warp instructions, 393 -> 312 us per launch; 17 km x 9 km canyon of 19350 16
// x 16 patches, 1837 with water: 182 -> 75 us.  Results are those of one edge to
// a thread bit for bit, but for waves below 1e-19, which no longer switch their
// limiter off: equal on uniform grids, a rounding apart (1e-8 relative) in
// refined forests.
//
// Scheme variants (Sec. 3.2): G.first_order drops the limited corrections,
// G.no_transverse the transverse terms; DS (dimensional splitting) takes the
// x sweep on every row of the window, updates the interior columns of all
// rows in shared memory (negative depths reset, dry momenta zeroed), and
// takes the y sweep on that state, without transverse terms.
template <class P, int MP, int M, int NT, bool DS = false>
__device__ __forceinline__ int patch_body(const GfGeom& G, const GfView& V,
                                          unsigned char* smraw, const int p,
                                          const int sub, const TileHdr& H, TmaPhase* tp,
                                          bool* wrote) {
  using R = typename P::R;
  constexpr bool DEV = P::DEV;
  using Lo = Layout<P, M, DS>;
  constexpr int TT = Lo::TT, NE = Lo::NE, NEDGE = Lo::NEDGE;
  constexpr int TGW = MP + 2 * GF_NG, TG = TGW * TGW;  // patch tile
  constexpr int NS1 = MP / M, NSUB = NS1 * NS1;
  constexpr int RL = (Lo::NLIM + NT - 1) / NT;    // limiter items per thread
  // FAST: a thread's cells are pairs: columns 2 (tid % (M / 2)) and the next
  // of rows tid / (M / 2), + TLC, ..., in both sweeps and the update; rows M
  // and M + 1 stand for the ghost rows -1 and M, so that their pairs fill
  // warps of their own
  constexpr bool FAST = Lo::FAST;
  constexpr int M2 = M / 2, TLC = NT / M2;
  static_assert(!FAST || NT % M2 == 0, "whole rows of pairs per round");
  constexpr int RC = FAST ? (M + 2 + TLC - 1) / TLC : (M * M + NT - 1) / NT;  // cells per thread
  constexpr int RX = (Lo::NCELL + NT - 1) / NT;   // increment cells per thread

  const int unit = p * NSUB + sub;  // CTA work unit: volume slot, same[] flag
  const bool has_gauge = H.has_gauge;
  const int ox = (sub % NS1) * M, oy = (sub / NS1) * M;
  const GfPatch Pt = H.Pt;
  GfCtl* C = V.ctl + Pt.scen;
  // global tile index of local cell (i, j), and interior index in the patch
  auto gix = [&](int i, int j) { return (ox + i + GF_NG) + (oy + j + GF_NG) * TGW; };
  auto pix = [&](int i, int j) { return (ox + i) + (oy + j) * MP; };

  R* s0 = reinterpret_cast<R*>(smraw);  // h (FP64) or w (deviation form)
  R* shu = s0 + TT;
  R* shv = s0 + 2 * TT;
  R* sb = s0 + 3 * TT;
  R* sdep = DEV && DS ? s0 + 4 * TT : s0;  // depth
  constexpr bool PRIM = Lo::PRIM;
  // PRIM: surface, velocities, celerity and root of the depth of every cell
  R* seta = s0 + (PRIM ? 4 : 0) * TT;
  R* su = s0 + (PRIM ? 5 : (FAST ? 4 : 0)) * TT;
  R* sv = s0 + (PRIM ? 6 : (FAST ? 5 : 0)) * TT;
  R* sc = s0 + (PRIM ? 7 : 0) * TT;
  R* sq = s0 + (PRIM ? 8 : (FAST ? 6 : 0)) * TT;
  R* W = reinterpret_cast<R*>(smraw + Lo::OFF_W);
  R* Ftr = reinterpret_cast<R*>(smraw + Lo::OFF_F);  // [row j][edge 0..M][3]
  R* Gtr = reinterpret_cast<R*>(smraw + Lo::OFF_G);  // [column i][edge][3]
  double* red = reinterpret_cast<double*>(smraw + Lo::OFF_RED);
  unsigned char* swet = smraw + Lo::OFF_WET;
  int* snb = reinterpret_cast<int*>(smraw + Lo::OFF_NB);  // same-level neighbours
  uint64_t* bar = reinterpret_cast<uint64_t*>(smraw + Lo::OFF_BAR);
  // FAST: set by a thread whose bounded wait gave up
  volatile int* sflag = reinterpret_cast<volatile int*>(smraw + Lo::OFF_WET);
  unsigned* naside = reinterpret_cast<unsigned*>(smraw + Lo::OFF_ASIDE);
  unsigned short* aside = reinterpret_cast<unsigned short*>(naside + 1);

  const int tid = threadIdx.x;
  // level subcycling: this level's period in fine substeps, its buffer
  // (ceil(sub_k / per) steps taken in the macro step so far) and its time
  // step (the macro step's share for the level)
  const bool subc = G.subcycle != 0;
  const int per = subc ? 1 << (G.maxlevel - Pt.level) : 1;
  const int cur = subc ? H.cur ^ ((C->sub_k / per) & 1) : H.cur;
  const double dtp = subc ? (gfk::div_rn(H.dt, (double)G.sub_K)) * (double)per : H.dt;
  const R* qs;
  R* qd;
  const R* bs;
  if constexpr (DEV) {
    qs = V.qf[cur] + (size_t)p * 3 * TG;
    qd = V.qf[cur ^ 1] + (size_t)p * 3 * TG;
    bs = V.bf + (size_t)p * TG;
  } else {
    qs = V.q[cur] + (size_t)p * 3 * TG;
    qd = V.q[cur ^ 1] + (size_t)p * 3 * TG;
    bs = V.b + (size_t)p * TG;
  }

  // A tile whose interior is the same in both buffers (it was dry and copied)
  // needs only its surface and bed to find out whether it is still dry; its
  // momenta are fetched only if water has arrived.
  const bool same_in = H.same_in;
  bool mom_issued = false;
  // staging barrier phases (a CTA that stages several tiles keeps them in tp)
  const bool fresh = tp == nullptr || !tp->init;
  const unsigned ph0 = tp ? tp->b0 : 0u, ph1 = tp ? tp->b1 : 0u;
  if constexpr (M == MP) {
    // whole patch: its four contiguous fields arrive by 1D TMA bulk copies,
    // surface and bed on bar[0], the momenta on bar[1]
    if (tid == 0) {
      if (fresh) {
        mbar_init(bar, 1);
        mbar_init(bar + 1, 1);
      }
      if constexpr (FAST) *sflag = 0, *naside = 0u;
      mbar_expect_tx(bar, 2u * TT * sizeof(R));
      bulk_g2s(s0, qs, TT * sizeof(R), bar);
      bulk_g2s(sb, bs, TT * sizeof(R), bar);
      if (!same_in) {
        mbar_expect_tx(bar + 1, 2u * TT * sizeof(R));
        bulk_g2s(shu, qs + TT, TT * sizeof(R), bar + 1);
        bulk_g2s(shv, qs + 2 * TT, TT * sizeof(R), bar + 1);
        if constexpr (FAST)  // the update's compensation terms, towards L2
          bulk_prefetch(V.lof[cur] + (size_t)p * 3 * MP * MP, 3u * MP * MP * sizeof(float));
      }
    }
    mom_issued = !same_in;
    if (tp) tp->init = true;
    // every wait is bounded; the decision to give up is taken by the whole CTA
    // (FAST: the first wait comes after the scalars below)
    if constexpr (!FAST) {
      __syncthreads();
      if (!__syncthreads_and(mbar_wait(bar, GF_SPIN_LIMIT, ph0) ? 1 : 0)) {
        if (tid == 0) C->status = -7;  // GEOFLOOD_ERR_TIMEOUT
        mbar_wait(bar, GF_SPIN_LIMIT, ph0);
        if (mom_issued) mbar_wait(bar + 1, GF_SPIN_LIMIT, ph1);
        __syncthreads();
        return -1;
      }
      if (tp) tp->b0 ^= 1u;
    }
  } else {
    // sub-tile: the (M+4)^2 window of each field, row segments read with
    // consecutive threads on consecutive addresses
    if constexpr (FAST) {
      // 16-byte pieces (tile rows and sub-tile origins are multiples of 16 B)
      constexpr int Q = Lo::T / 4;
      for (int k = tid; k < Q * Lo::T; k += NT) {
        const int li = 4 * (k % Q), lj = k / Q;
        const int g = (ox + li) + (oy + lj) * TGW, c = li + lj * Lo::T;
        const float4 a0 = *reinterpret_cast<const float4*>(qs + g);
        const float4 a1 = *reinterpret_cast<const float4*>(qs + TG + g);
        const float4 a2 = *reinterpret_cast<const float4*>(qs + 2 * TG + g);
        const float4 a3 = *reinterpret_cast<const float4*>(bs + g);
        *reinterpret_cast<float4*>(s0 + c) = a0;
        *reinterpret_cast<float4*>(shu + c) = a1;
        *reinterpret_cast<float4*>(shv + c) = a2;
        *reinterpret_cast<float4*>(sb + c) = a3;
      }
      if (tid == 0) *sflag = 0, *naside = 0u;
    } else
    for (int k = tid; k < TT; k += NT) {
      const int li = k % Lo::T, lj = k / Lo::T;
      const int g = (ox + li) + (oy + lj) * TGW;
      s0[k] = qs[g];
      shu[k] = qs[TG + g];
      shv[k] = qs[2 * TG + g];
      sb[k] = bs[g];
    }
  }

  const bool push = V.push != 0 && V.nbr != nullptr;
  // FAST: what comes from global memory is asked for here and stored behind
  // the next barrier, which then waits for none of it
  [[maybe_unused]] int nbr = -1;
  [[maybe_unused]] float mann = 0.0f;
  constexpr int SCT = FAST ? 32 : 0;
  if constexpr (FAST) {
    if (push && tid < 8) nbr = V.nbr[(size_t)p * 8 + tid];
    if (tid == SCT) mann = V.scen[Pt.scen].manning_f;
  }
  // per-patch scalars: computed once by one thread (FP64 divisions are slow
  // on this part, so no thread repeats them; FAST: not by the one that asks
  // for the tile) and broadcast through shared memory
  double* scal = red + 48;  // dx, dy, nux, nuy, then the R-typed copies
  R* rscal = reinterpret_cast<R*>(red + 52);  // g, drytol, nux, nuy, n, dt
  float* fscal = reinterpret_cast<float*>(red + 60);  // drytol, margin
  if (tid == SCT) {
    if constexpr (DEV) {
      // FP32 from the host's per-level tables: one conversion per patch
      const float dtf32 = (float)dtp;
      rscal[0] = G.gf;
      rscal[1] = G.drytolf;
      rscal[2] = dtf32 * G.inv_dxf[Pt.level];
      rscal[3] = dtf32 * G.inv_dyf[Pt.level];
      if constexpr (!FAST) rscal[4] = V.scen[Pt.scen].manning_f;
      rscal[5] = dtf32;
      fscal[0] = G.drytolf;
      fscal[1] = G.marginf;
    } else {
      const double dx0 = G.dxl[Pt.level], dy0 = G.dyl[Pt.level];
      scal[0] = dx0;
      scal[1] = dy0;
      scal[2] = gfk::div_rn(dtp, dx0);
      scal[3] = gfk::div_rn(dtp, dy0);
      rscal[0] = (R)G.g;
      rscal[1] = (R)G.drytol;
      rscal[2] = (R)scal[2];
      rscal[3] = (R)scal[3];
      rscal[4] = (R)V.scen[Pt.scen].manning_n;
      rscal[5] = (R)dtp;
    }
  }
  if constexpr (!FAST) {
    if (push && tid < 8) snb[tid] = V.nbr[(size_t)p * 8 + tid];
  }
  const double drytol = G.drytol;
  R smx = R(0), smy = R(0);

  __syncthreads();
  const R g = rscal[0], rdry = rscal[1], nux = rscal[2], nuy = rscal[3];
  const R dtr = rscal[5];
  const float dtf = fscal[0], margin = fscal[1];

  // Per-cell depth and exact wet flag (deviation form), and whether the
  // tile holds any wet cell at all.  A tile whose interior is unchanged and
  // was dry (same_in) can only have taken water into its ghost cells, so the
  // interior is examined only if they hold some.
  constexpr int NRING = TT - M * M;
  auto ring_cell = [&](int k) {  // k-th ghost cell of the window
    const int band = 2 * Lo::T;
    if (k < band) return k;                                 // two bottom rows
    if (k < 2 * band) return (M + GF_NG) * Lo::T + (k - band);  // two top rows
    const int r = k - 2 * band, j = r / 4, c = r % 4;
    return (j + GF_NG) * Lo::T + (c < 2 ? c : M + c);       // side columns
  };
  auto examine = [&](int k) -> int {
    if constexpr (DEV) {
      const float w = s0[k], b = sb[k];
      const bool wt = gfk::wet_dev(w, b, drytol, dtf, margin);
      if constexpr (FAST) {
        sq[k] = wt ? sqrtf(w - b) : 0.0f;  // zero: dry
      } else {
        sdep[k] = w - b;
        swet[k] = wt ? 1 : 0;
      }
      return wt ? 1 : 0;
    } else {
      return gfk::above(s0[k], rdry) ? 1 : 0;
    }
  };
  int anywet = 0;
  // FAST: a quad of cells: wet tests, roots of the depths and velocities
  [[maybe_unused]] auto cells4 = [&](int k, bool velocities) {
    if constexpr (FAST) {
      const float4 w = *reinterpret_cast<const float4*>(s0 + k);
      const float4 b = *reinterpret_cast<const float4*>(sb + k);
      float4 q;
      auto one = [&](float wk, float bk) {
        const bool wt = gfk::wet_dev(wk, bk, drytol, dtf, margin);
        anywet |= wt ? 1 : 0;
        return wt ? sqrtf(wk - bk) : 0.0f;  // zero: dry
      };
      q.x = one(w.x, b.x);
      q.y = one(w.y, b.y);
      q.z = one(w.z, b.z);
      q.w = one(w.w, b.w);
      *reinterpret_cast<float4*>(sq + k) = q;
      if (!velocities) return;
      const float4 hu = *reinterpret_cast<const float4*>(shu + k);
      const float4 hv = *reinterpret_cast<const float4*>(shv + k);
      float4 u, v;
      auto vel = [](float qk, float h, float a, float c, float& x, float& y) {
        const float rh = gfk::rcpf(h);
        x = qk > 0.0f ? __fmul_rn(a, rh) : 0.0f;
        y = qk > 0.0f ? __fmul_rn(c, rh) : 0.0f;
      };
      vel(q.x, w.x - b.x, hu.x, hv.x, u.x, v.x);
      vel(q.y, w.y - b.y, hu.y, hv.y, u.y, v.y);
      vel(q.z, w.z - b.z, hu.z, hv.z, u.z, v.z);
      vel(q.w, w.w - b.w, hu.w, hv.w, u.w, v.w);
      *reinterpret_cast<float4*>(su + k) = u;
      *reinterpret_cast<float4*>(sv + k) = v;
    }
  };
  if constexpr (FAST) {
    if constexpr (M == MP) {
      bool ok = mbar_wait(bar, GF_SPIN_LIMIT, ph0);
      if (mom_issued) ok = mbar_wait(bar + 1, GF_SPIN_LIMIT, ph1) && ok;
      if (!ok) *sflag = 1;
      if (tp) {
        tp->b0 ^= 1u;
        if (mom_issued) tp->b1 ^= 1u;
      }
    }
    if (M == MP && same_in) {
      // an unchanged dry interior: only the ghost cells can have taken water
      for (int k = tid; k < NRING; k += NT) anywet |= examine(ring_cell(k));
    } else {
      for (int k = 4 * tid; k < TT; k += 4 * NT) cells4(k, true);
    }
    if (push && tid < 8) snb[tid] = nbr;
    if (tid == SCT) rscal[4] = mann;
    anywet = __syncthreads_or(anywet);
    if (*sflag) {
      // some wait gave up: wait (again with a limit) for the copies in
      // flight, then give the tile up
      if (tid == 0) C->status = -7;  // GEOFLOOD_ERR_TIMEOUT
      if constexpr (M == MP) {
        mbar_wait(bar, GF_SPIN_LIMIT, ph0);
        if (mom_issued) mbar_wait(bar + 1, GF_SPIN_LIMIT, ph1);
      }
      __syncthreads();
      return -1;
    }
  } else {
  if (same_in) {
    for (int k = tid; k < NRING; k += NT) anywet |= examine(ring_cell(k));
    anywet = __syncthreads_or(anywet);
    if (anywet) {
      for (int k = tid; k < M * M; k += NT)
        examine((k % M + GF_NG) + (k / M + GF_NG) * Lo::T);
      __syncthreads();  // the sweeps read every thread's depths and flags
    }
  } else {
    for (int k = tid; k < TT; k += NT) anywet |= examine(k);
    anywet = __syncthreads_or(anywet);
  }
  }
  if constexpr (M == MP) {
    // the momenta: requested now if water arrived at a copied dry tile, and
    // waited for whenever they were requested
    const bool late = anywet && !mom_issued;
    if (late) {
      if (tid == 0) {
        mbar_expect_tx(bar + 1, 2u * TT * sizeof(R));
        bulk_g2s(shu, qs + TT, TT * sizeof(R), bar + 1);
        bulk_g2s(shv, qs + 2 * TT, TT * sizeof(R), bar + 1);
      }
      mom_issued = true;
    }
    if ((FAST ? late : mom_issued) &&
        !__syncthreads_and(mbar_wait(bar + 1, GF_SPIN_LIMIT, ph1) ? 1 : 0)) {
      if (tid == 0) C->status = -7;  // GEOFLOOD_ERR_TIMEOUT
      mbar_wait(bar + 1, GF_SPIN_LIMIT, ph1);
      __syncthreads();
      return -1;
    }
    if ((FAST ? late : mom_issued) && tp) tp->b1 ^= 1u;
    if constexpr (FAST) {
      if (late) {
        for (int k = 4 * tid; k < TT; k += 4 * NT) cells4(k, true);
        __syncthreads();
      }
    }
  }
  // a dry tile whose interior is already the same in both buffers writes
  // nothing (its update is the identity on the surface, zero momenta)
  const bool skip_writes = same_in && !anywet;
  if (V.same != nullptr && tid == 0) V.same[unit] = anywet ? 0 : 1;
  if (has_gauge && H.accepted && (!subc || C->sub_k == 0))
    sample_gauges<R, DEV, MP, M>(V, Pt.scen, C, p, ox, oy, s0, shu, shv, sb,
                                 M != MP || mom_issued);
  if (skip_writes) {
    // nothing changes: no writes, no waves
    if (wrote) *wrote = false;
    return 0;
  }
  auto wetc = [&](int c) -> bool {
    if constexpr (FAST) return sq[c] > R(0);
    else if constexpr (DEV) return swet[c] != 0;
    else if constexpr (PRIM) return gfk::pos(sc[c]);  // zero celerity: dry
    else return s0[c] > rdry;
  };
  auto surf = [&](int c) -> R {
    if constexpr (DEV) return s0[c];
    else if constexpr (PRIM) return seta[c];
    else return s0[c] + sb[c];
  };
  if constexpr (PRIM) {
    if (anywet) {
      // what belongs to a cell, once per cell: an interior cell is a side of
      // four edges and is split twice
      for (int k = tid; k < TT; k += NT) {
        const double h = s0[k];
        const bool wt = gfk::above(h, rdry);
        seta[k] = h + sb[k];
        su[k] = wt ? gfk::div_rn(shu[k], h) : 0.0;
        sv[k] = wt ? gfk::div_rn(shv[k], h) : 0.0;
        sc[k] = wt ? gfk::sqrt_rn(g * h) : 0.0;
        sq[k] = wt ? gfk::sqrt_rn(h) : 0.0;
      }
      __syncthreads();
    }
  }

  R X[PRIM ? RC : 1][3];  // PRIM: nu dQ of owned interior cells
  R Y[DS ? RC : 1][3];    // split: nu_y * dQy
  // dimensional splitting, deviation form: compensation terms of the
  // intermediate state of owned interior cells
  float LO1[DS && DEV ? RC : 1][3];
  const float* los = nullptr;
  float* lod = nullptr;
  if constexpr (DEV) {
    los = V.lof[cur] + (size_t)p * 3 * MP * MP;
    lod = V.lof[cur ^ 1] + (size_t)p * 3 * MP * MP;
  }
  const bool corr = G.first_order == 0;              // limited corrections
  const bool trv = !DS && G.no_transverse == 0;      // transverse terms
  double clipd = 0.0;
  float clipf = 0.0f;  // deviation form: clipped depth, FP32 per thread
  unsigned nclip = 0, nwet = 0;

  // A tile without a wet cell (ghosts included) has only dry-dry edges: every
  // wave, correction and transverse term is zero and the update reduces to
  // zeroing the momenta of the (dry) cells, which the dry branch below does
  // without the sweeps; the results are identical.
  // one sweep; the direction is a compile-time constant so that the index
  // arithmetic of the two sweeps is resolved statically
  using gfk::f2;
  // FAST: of the pairs of owned cells, nu dQ summed over the sweeps and the
  // transverse fluxes' change
  [[maybe_unused]] f2 XP[FAST ? RC : 1][3], TP[FAST ? RC : 1][3];
  [[maybe_unused]] auto sweep32 = [&](auto dirc) {
    constexpr int dir = decltype(dirc)::value;
    if constexpr (FAST) {
    // Edge a in [-1, M + 1] of line l in [-1, M].  In both sweeps threads take
    // pairs of neighbours along a tile row: two edges of a row in the x
    // sweep, the edges of two columns (from column -2 on) in the y sweep.
    // Place of an edge in a wave plane: tile-like rows of pitch PW.
    constexpr int PW = M + 4;
    constexpr int SE = dir == 0 ? 1 : PW;        // place of the next edge of a line
    constexpr int CS = dir == 0 ? 1 : Lo::T;     // tile step along the sweep
    constexpr int CL = dir == 0 ? Lo::T : 1;     // and across it
    const R* sn = dir == 0 ? shu : shv;
    const R* un = dir == 0 ? su : sv;
    const R* ut = dir == 0 ? sv : su;
    const float nu = dir == 0 ? nux : nuy;
    const float sg = sqrtf(g);
    const f2 nz = gfk::pk1(G.negzero);
    float smax = dir == 0 ? smx : smy;
    // phase 1: Riemann solves.  x: row l, edges a = -1 + 2 m and the next;
    // y: edge row a, columns -2 + 2 m and the next
    constexpr int N1 = dir == 0 ? (M + 2) * PW / 2 : (M + 3) * PW / 2;
    // of pair k: tile cell left of (below) its first edge, and its cells
    auto cell_of = [&](int k) {
      const int m = k % (PW / 2), row = k / (PW / 2);  // row: l + 1, or a + 1
      return dir == 0 ? (row + 1) * Lo::T + 2 * m : row * Lo::T + 2 * m;
    };
    auto pair_r = [&](const R* p, int c, f2 l) {
      if constexpr (dir == 0) {
        float x, y;
        gfk::upk(l, x, y);
        return gfk::pk(y, p[c + 2]);
      } else {
        (void)l;
        return gfk::ld2(p + c + CS);
      }
    };
    // Edges between a wet and a dry cell: the blocks they add to a pair cost a
    // warp the same for one lane as for all.  With one pair to a thread they
    // are taken on the way; with several (whole 32 x 32 tiles, where a front
    // touches nearly every warp in every round) they are set aside and taken
    // together, one edge to a thread.  256 patches with a front: 22.2 us a
    // step on the way, 21.5 so.  What such a pair needs is found behind the
    // solver's own test for unusual edges, so that pairs of wet cells pay
    // nothing for it (valley of 6827 patches: 178.4 us a step with the
    // wetness of every pair found first, 175.8 so).
    constexpr bool LATER = Lo::ASIDE > 0 && N1 > NT;
#pragma unroll 1
    for (int k = tid; k < N1; k += NT) {
      const int m = k % (PW / 2), row = k / (PW / 2);
      const int c = cell_of(k), e = row * PW + 2 * m;
      R* w = W + e;
      const f2 ql = gfk::ld2(sq + c), qr = pair_r(sq, c, ql);
      if ((ql | qr) == 0ull) {  // dry cells
#pragma unroll
        for (int q = 0; q < 10; ++q) gfk::st2(w + q * NEDGE, 0ull);
        continue;
      }
      auto pair_l = [&](const R* p) { return gfk::ld2(p + c); };
      const gfk::Prim32x2 L{pair_l(s0), pair_l(sb), pair_l(sn), pair_l(un), pair_l(ut), ql};
      const gfk::Prim32x2 Rt{pair_r(s0, c, L.w), pair_r(sb, c, L.b), pair_r(sn, c, L.n),
                             pair_r(un, c, L.u), pair_r(ut, c, L.v), qr};
      f2 z[8], s1, s3;
      const bool usual = gfk::riemann32x2<!LATER>(L, Rt, g, sg, nz, z, s1, s3);
      if constexpr (LATER) {
        if (!usual) {
          // nothing (yet) where a cell is dry
          float a0, a1, b0, b1;
          gfk::upk(ql, a0, a1);
          gfk::upk(qr, b0, b1);
          const bool x0 = a0 > 0.0f, x1 = a1 > 0.0f, y0 = b0 > 0.0f, y1 = b1 > 0.0f;
#pragma unroll
          for (int q = 0; q < 8; ++q) z[q] = gfk::sel2(x0 && y0, x1 && y1, z[q], 0ull);
          s1 = gfk::sel2(x0 && y0, x1 && y1, s1, 0ull);
          s3 = gfk::sel2(x0 && y0, x1 && y1, s3, 0ull);
          const bool mix0 = x0 != y0, mix1 = x1 != y1;
          if (mix0 || mix1) {
            const unsigned at = atomicAdd(naside, (mix0 ? 1u : 0u) + (mix1 ? 1u : 0u));
            const unsigned at1 = at + (mix0 ? 1u : 0u);
            if (mix0 && at < (unsigned)Lo::ASIDE) aside[at] = (unsigned short)e;
            if (mix1 && at1 < (unsigned)Lo::ASIDE) aside[at1] = (unsigned short)(e + 1);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) gfk::st2(w + q * NEDGE, z[q]);
      gfk::st2(w + 8 * NEDGE, s1);
      gfk::st2(w + 9 * NEDGE, s3);
      // CFL rate: edges of interior lines that bound interior cells
      float s1a, s1b, s3a, s3b;
      gfk::upk(s1, s1a, s1b);
      gfk::upk(s3, s3a, s3b);
      const float ma = fmaxf(fabsf(s1a), fabsf(s3a)), mb = fmaxf(fabsf(s1b), fabsf(s3b));
      if constexpr (dir == 0) {
        if ((unsigned)(row - 1) < (unsigned)M) {  // a = 2 m - 1, 2 m
          if (m > 0 && m <= M2) smax = fmaxf(smax, ma);
          if (m <= M2) smax = fmaxf(smax, mb);
        }
      } else {
        if ((unsigned)(row - 1) <= (unsigned)M && m > 0 && m <= M2)
          smax = fmaxf(smax, fmaxf(ma, mb));
      }
    }
    if constexpr (LATER) {
      // the tile's rows are the planes', so the cell left of or below an edge
      // is at the same place, a row up in the x sweep
      static_assert(PW == Lo::T, "an edge's place gives its cells");
      __syncthreads();
      const unsigned na = *naside;
      const bool full = na > (unsigned)Lo::ASIDE;  // more than the list holds
#pragma unroll 1
      for (int x = tid; x < (full ? 2 * N1 : (int)na); x += NT) {
        const int e = full ? x : aside[x], c = dir == 0 ? e + Lo::T : e, row = e / PW, at = e % PW;
        if (full && (sq[c] > 0.0f) == (sq[c + CS] > 0.0f)) continue;
        const float l[6] = {s0[c], sb[c], sn[c], un[c], ut[c], sq[c]};
        const float r[6] = {s0[c + CS], sb[c + CS], sn[c + CS], un[c + CS], ut[c + CS], sq[c + CS]};
        float z[8], s1, s3;
        gfk::riemann32_front(l, r, g, sg, z, s1, s3);
#pragma unroll
        for (int q = 0; q < 8; ++q) W[q * NEDGE + e] = z[q];
        W[8 * NEDGE + e] = s1;
        W[9 * NEDGE + e] = s3;
        const bool counts =
            dir == 0 ? (unsigned)(row - 1) < (unsigned)M && (unsigned)(at - 1) <= (unsigned)M
                     : (unsigned)(row - 1) <= (unsigned)M && (unsigned)(at - 2) < (unsigned)M;
        if (counts) smax = fmaxf(smax, fmaxf(fabsf(s1), fabsf(s3)));
      }
    }
    if (dir == 0) smx = smax;
    else smy = smax;
    __syncthreads();
    // phase 2: limited fluxes of edges 0..M, kept until every wave was read.
    // x: pairs from a = -1 on; y: rows a = 0..M
    constexpr int N2 = dir == 0 ? (M + 2) * (M2 + 1) : (M + 1) * PW / 2;
    constexpr int RE = (N2 + NT - 1) / NT;
    f2 am[RE][3], ap[RE][3], ff[RE][3];
#pragma unroll
    for (int r = 0; r < RE; ++r) {
      const int k = tid + r * NT;
      if (k < N2) {
        const int m = dir == 0 ? k % (M2 + 1) : k % (PW / 2);
        const int row = dir == 0 ? k / (M2 + 1) : k / (PW / 2) + 1;  // l + 1, or a + 1
        const int e = row * PW + 2 * m;
        const int c = dir == 0 ? (row + 1) * Lo::T + 2 * m : row * Lo::T + 2 * m;
        float q0, q1, q2, q3;
        gfk::upk(gfk::ld2(sq + c), q0, q1);
        if constexpr (dir == 0) {
          q3 = sq[c + 2];
          q2 = q1;
        } else {
          gfk::upk(gfk::ld2(sq + c + CS), q2, q3);
        }
        gfk::edge32x2<NEDGE, SE>(W + e, nu, corr && fminf(q0, q2) > 0.0f,
                                 corr && fminf(q1, q3) > 0.0f, nz, am[r], ap[r], ff[r]);
      }
    }
    __syncthreads();
    if (LATER && tid == 0) *naside = 0u;
#pragma unroll
    for (int r = 0; r < RE; ++r) {
      const int k = tid + r * NT;
      if (k < N2) {
        const int m = dir == 0 ? k % (M2 + 1) : k % (PW / 2);
        const int row = dir == 0 ? k / (M2 + 1) : k / (PW / 2) + 1;
        R* w = W + row * PW + 2 * m;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          gfk::st2(w + q * NEDGE, am[r][q]);
          gfk::st2(w + (3 + q) * NEDGE, ap[r][q]);
          gfk::st2(w + (6 + q) * NEDGE, ff[r][q]);
        }
      }
    }
    __syncthreads();
    // phase 3: increments and their transverse split.  The x sweep covers
    // rows -1..M of the thread's columns; in the y sweep the threads of the
    // two ghost rows take the two ghost columns instead (two rows each).
    // Transverse parts (plus, minus; mass, hu, hv) in planes of pitch PT.
    // The last warp has no rows in the second round: its last thread enters
    // the patch in the next launch order meanwhile (at the tile's end the
    // round trip would be waited for)
    if (dir == 1 && tid == NT - 1 && H.order != nullptr)
      H.order[atomicAdd(order_ends(V, H.order), 1u)] = p;
    constexpr int PTP = M * (M + 4);          // one plane
    constexpr int PT = dir == 0 ? M : M + 4;  // its rows
    R* Tr = Ftr;
    auto tplace = [&](int i, int j) { return dir == 0 ? (j + 1) * M + i : j * PT + i + 2; };
    f2 opl[RC][3], omi[RC][3];
#pragma unroll
    for (int r = 0; r < RC; ++r) {
      const int lane = tid % M2, Lx = tid / M2 + r * TLC;
      const bool inner = Lx < M;
      const int Lr = inner ? Lx : (Lx == M ? -1 : M);
      if (!(Lx <= M + 1 && (inner || trv))) continue;
      const bool col = dir == 1 && !inner;  // a pair down a ghost column
      const int i = col ? Lr : 2 * lane, j = col ? 2 * lane : Lr;
      f2 d[3];  // mass, normal (sweep) momentum, transverse
      if constexpr (dir == 0) {
        const R* w = W + (j + 1) * PW + i + 1;  // edge a = i (odd place)
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const f2 apl = gfk::pk(w[(3 + q) * NEDGE], w[(3 + q) * NEDGE + 1]);
          const f2 fr = gfk::ld2(w + (6 + q) * NEDGE + 1);
          float f1, f2v;
          gfk::upk(fr, f1, f2v);
          const f2 fl = gfk::pk(w[(6 + q) * NEDGE], f1);
          d[q] = gfk::add2(gfk::add2(apl, gfk::ld2(w + q * NEDGE + 1)), gfk::sub2(fr, fl));
        }
      } else {
        const R* w = W + (j + 1) * PW + i + 2;  // edge a = j of column i
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const R *wa = w + q * NEDGE + PW, *wp = w + (3 + q) * NEDGE, *wf = w + (6 + q) * NEDGE;
          f2 amr, apl, fl, fr;
          if (col) {
            amr = gfk::pk(wa[0], wa[PW]);
            apl = gfk::pk(wp[0], wp[PW]);
            fl = gfk::pk(wf[0], wf[PW]);
            fr = gfk::pk(wf[PW], wf[2 * PW]);
          } else {
            amr = gfk::ld2(wa);
            apl = gfk::ld2(wp);
            fl = gfk::ld2(wf);
            fr = gfk::ld2(wf + PW);
          }
          d[q] = gfk::add2(gfk::add2(apl, amr), gfk::sub2(fr, fl));
        }
      }
      if (inner) {
        // (mass, hu, hv)
        const f2 n2 = gfk::pk1(nu);
        if constexpr (dir == 0) {
          XP[r][0] = gfk::mulr2(n2, d[0], nz);
          XP[r][1] = gfk::mulr2(n2, d[1], nz);
          XP[r][2] = gfk::mulr2(n2, d[2], nz);
        } else {
          XP[r][0] = gfk::add2(XP[r][0], gfk::mulr2(n2, d[0], nz));
          XP[r][1] = gfk::add2(XP[r][1], gfk::mulr2(n2, d[2], nz));
          XP[r][2] = gfk::add2(XP[r][2], gfk::mulr2(n2, d[1], nz));
        }
      }
      if (!trv) continue;
      const int c = tix<M>(i, j);
      const int c1 = col ? c + Lo::T : c + 1;  // the pair's second cell
      auto cells = [&](const R* p) {
        return col ? gfk::pk(p[c], p[c1]) : gfk::ld2(p + c);
      };
      const f2 w2 = cells(s0);
      float q0, q1;
      gfk::upk(cells(sq), q0, q1);
      f2 pl[3], mi[3];
      const f2 dd[3] = {d[0], d[2], d[1]};
      gfk::tsplit32x2(cells(ut), cells(un), gfk::sub2(w2, cells(sb)), g, nz, dd, pl, mi);
      // nothing from a dry cell, nor into a dry neighbour across the sweep
      // whose bed is above the cell's surface
      const float qp0 = sq[c + CL], qm0 = sq[c - CL], qp1 = sq[c1 + CL], qm1 = sq[c1 - CL];
      if (!(fminf(fminf(fminf(qp0, qm0), fminf(qp1, qm1)), fminf(q0, q1)) > 0.0f)) {
        float w0, w1;
        gfk::upk(w2, w0, w1);
        const bool p0 = q0 > 0.0f && (qp0 > 0.0f || !(sb[c + CL] > w0));
        const bool p1 = q1 > 0.0f && (qp1 > 0.0f || !(sb[c1 + CL] > w1));
        const bool m0 = q0 > 0.0f && (qm0 > 0.0f || !(sb[c - CL] > w0));
        const bool m1 = q1 > 0.0f && (qm1 > 0.0f || !(sb[c1 - CL] > w1));
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          pl[q] = gfk::sel2(p0, p1, pl[q], 0ull);
          mi[q] = gfk::sel2(m0, m1, mi[q], 0ull);
        }
      }
      // (mass, hu, hv): "along" is the transverse momentum
      const int hu = dir == 0 ? 2 : 1, hv = dir == 0 ? 1 : 2;
      const f2 po[3] = {pl[0], pl[hu], pl[hv]}, mo[3] = {mi[0], mi[hu], mi[hv]};
      R* o = Tr + tplace(i, j);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        if (col) {
          float x, y;
          gfk::upk(po[q], x, y);
          o[q * PTP] = x;
          o[q * PTP + PT] = y;
          gfk::upk(mo[q], x, y);
          o[(3 + q) * PTP] = x;
          o[(3 + q) * PTP + PT] = y;
        } else {
          gfk::st2(o + q * PTP, po[q]);
          gfk::st2(o + (3 + q) * PTP, mo[q]);
        }
        opl[r][q] = po[q];
        omi[r][q] = mo[q];
      }
    }
    __syncthreads();
    // transverse fluxes through the cell's two edges across the sweep:
    // -nu/2 of what enters each from both sides; their difference
    if (trv) {
      const f2 kt = gfk::pk1(-0.5f * nu), nx2 = gfk::pk1(nux);
#pragma unroll
      for (int r = 0; r < RC; ++r) {
        const int i = 2 * (tid % M2), j = tid / M2 + r * TLC;
        if ((unsigned)j >= (unsigned)M) continue;
        const R* o = Tr + tplace(i, j);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          f2 mn, pp;  // minus of the next line's cells, plus of the previous
          if constexpr (dir == 0) {
            mn = gfk::ld2(o + (3 + q) * PTP + PT);
            pp = gfk::ld2(o + q * PTP - PT);
          } else {
            float x, y;
            gfk::upk(omi[r][q], x, y);
            mn = gfk::pk(y, o[(3 + q) * PTP + 2]);
            gfk::upk(opl[r][q], x, y);
            pp = gfk::pk(o[q * PTP - 1], x);
          }
          const f2 hi = gfk::mulr2(kt, gfk::add2(opl[r][q], mn), nz);
          const f2 lo = gfk::mulr2(kt, gfk::add2(pp, omi[r][q]), nz);
          const f2 df = gfk::sub2(hi, lo);
          if constexpr (dir == 0) TP[r][q] = gfk::mul2(gfk::pk1(nuy), df);
          else TP[r][q] = gfk::fma2(nx2, df, TP[r][q]);
        }
      }
    } else {
#pragma unroll
      for (int r = 0; r < RC; ++r) TP[r][0] = TP[r][1] = TP[r][2] = 0ull;
    }
    }
  };
  // PRIM: one sweep, the direction a run-time value so that both sweeps share
  // one copy of the code (this kernel's instruction fetch shows in its time).
  // ht: the thread's number among the HN that take this sweep; Wd: their
  // wave planes.  Every thread of the CTA passes the same barriers.
  constexpr bool BOTH = Lo::BOTH;
  constexpr int HN = BOTH ? NT / 2 : NT;
  [[maybe_unused]] auto sweep64 = [&](const int dir, const int ht, R* const Wd) {
    if constexpr (PRIM) {
    constexpr int NRL = M + 2;
    constexpr int RL6 = (NRL * (M + 1) + HN - 1) / HN;
    constexpr int RX6 = (M * NRL + HN - 1) / HN;
    const bool xs = dir == 0;
    const int CS = xs ? 1 : Lo::T, CL = xs ? Lo::T : 1;  // tile steps along, across
    const R* sn = xs ? shu : shv;  // normal momentum
    const R* st = xs ? shv : shu;  // transverse momentum
    const R* un = xs ? su : sv;
    const R* ut = xs ? sv : su;
    const R nu = xs ? nux : nuy;
    // tile cell (position a along the sweep, line across it)
    auto at = [&](int a, int line) { return tix<M>(0, 0) + a * CS + line * CL; };
    // phase 1: Riemann solves on the lines -1..M, edges -1..M+1
    for (int k = ht; k < NRL * NE; k += HN) {
      const int line = (xs ? k / NE : k % NRL) - 1;
      const int a = (xs ? k % NE : k / NRL) - 1;
      const int cr = at(a, line), cl = cr - CS;
      R* w = Wd + ((line + 1) * NE + a + 1);
      double z[8], S[3];
      gfk::riemann_prim(gfk::Prim{s0[cl], sn[cl], st[cl], sb[cl], seta[cl], un[cl], ut[cl],
                                  sc[cl], sq[cl], wetc(cl)},
                        gfk::Prim{s0[cr], sn[cr], st[cr], sb[cr], seta[cr], un[cr], ut[cr],
                                  sc[cr], sq[cr], wetc(cr)},
                        g, z, S);
#pragma unroll
      for (int q = 0; q < 8; ++q) w[q * NEDGE] = z[q];
#pragma unroll
      for (int q = 0; q < 3; ++q) w[(8 + q) * NEDGE] = S[q];
    }
    __syncthreads();
    // phase 2: fluctuations and limited corrections on edges 0..M
    R AMr[RL6][3], APr[RL6][3], FFr[RL6][3];
    R smax = R(0);
#pragma unroll
    for (int r = 0; r < RL6; ++r) {
      const int k = ht + r * HN;
      if (k < NRL * (M + 1)) {
        const int line = k / (M + 1) - 1, a = k % (M + 1);
        const R* w = Wd + ((line + 1) * NE + a + 1);
        const int cr = at(a, line);
        const bool wet = corr && wetc(cr - CS) && wetc(cr);
        gfk::edge_fluxes_prim<NEDGE>(w, w - 1, w + 1, nu, wet, AMr[r], APr[r], FFr[r]);
        // |s| of the outer waves (the middle speed is their mean)
        if (line >= 0 && line < M)
          smax = gfk::dmax(smax, gfk::dmax(gfk::dabs(w[8 * NEDGE]), gfk::dabs(w[10 * NEDGE])));
      }
    }
    if (xs) smx = gfk::dmax(smx, smax);
    else smy = gfk::dmax(smy, smax);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RL6; ++r) {
      const int k = ht + r * HN;
      if (k < NRL * (M + 1)) {
        R* w = Wd + ((k / (M + 1)) * NE + k % (M + 1) + 1);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          w[q * NEDGE] = AMr[r][q];
          w[(3 + q) * NEDGE] = APr[r][q];
          w[(6 + q) * NEDGE] = FFr[r][q];
        }
      }
    }
    __syncthreads();
    // phase 3: per-cell increments and their transverse split
    R* Tr = xs ? Gtr : Ftr;
    R MIr[RX6][3];
    R Yb[BOTH ? RC : 1][3];
#pragma unroll
    for (int r = 0; r < RX6; ++r) {
      const int k = ht + r * HN;
      if (k < M * NRL) {
        // interior cells in the fixed order of the update, then ghost lines
        const int kk = k - M * M, i = k % M, j = k / M;
        const int line = k < M * M ? (xs ? j : i) : (kk < M ? -1 : M);
        const int a = k < M * M ? (xs ? i : j) : kk % M;
        const R* wl = Wd + ((line + 1) * NE + a + 1);  // edge a
        const R* wr = wl + 1;                           // edge a+1
        R d[3];  // frame: mass, normal (sweep) momentum, transverse
#pragma unroll
        for (int q = 0; q < 3; ++q)
          d[q] = (wl[(3 + q) * NEDGE] + wr[q * NEDGE]) +
                 (wr[(6 + q) * NEDGE] - wl[(6 + q) * NEDGE]);
        if (r < RC && k < M * M) {
          // nu * dQ in (h, hu, hv) order
          const R v1 = nu * d[1], v2 = nu * d[2];
          const R v[3] = {nu * d[0], xs ? v1 : v2, xs ? v2 : v1};
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            if constexpr (BOTH) {
              if (xs) X[r][q] = v[q];
              else Yb[r][q] = v[q];
            } else {
              X[r][q] = xs ? v[q] : X[r][q] + v[q];
            }
          }
        }
        if (trv) {
          const int ci = at(a, line), cm = ci - CL, cp = ci + CL;
          const R dd[3] = {d[0], d[2], d[1]};
          R pl[3], mi[3];
          gfk::tsplit_prim(ut[ci], un[ci], sc[ci], seta[ci], wetc(ci), wetc(cm), sb[cm], wetc(cp),
                           sb[cp], dd, pl, mi);
          // back to (h, hu, hv): "along" is the sweep's transverse momentum
          MIr[r][0] = mi[0];
          MIr[r][1] = xs ? mi[2] : mi[1];
          MIr[r][2] = xs ? mi[1] : mi[2];
          if (line + 1 <= M) {
            R* o = Tr + 3 * (a * (M + 1) + line + 1);
            o[0] = pl[0];
            o[1] = xs ? pl[2] : pl[1];
            o[2] = xs ? pl[1] : pl[2];
          }
        }
      }
    }
    __syncthreads();
    if (trv) {
      const R kt = R(-0.5) * nu;
#pragma unroll
      for (int r = 0; r < RX6; ++r) {
        const int k = ht + r * HN;
        if (k < M * NRL) {
          const int kk = k - M * M, i = k % M, j = k / M;
          const int line = k < M * M ? (xs ? j : i) : (kk < M ? -1 : M);
          const int a = k < M * M ? (xs ? i : j) : kk % M;
          if (line >= 0) {
            R* o = Tr + 3 * (a * (M + 1) + line);
#pragma unroll
            for (int q = 0; q < 3; ++q) o[q] = kt * (o[q] + MIr[r][q]);
          }
        }
      }
    }
    if constexpr (BOTH) {
      // the y half's increments, for the threads that own the cells
      if (!xs) {
#pragma unroll
        for (int r = 0; r < RC; ++r) {
          const int k = ht + r * HN;
          if (k < M * M) {
#pragma unroll
            for (int q = 0; q < 3; ++q) Wd[q * NEDGE + k] = Yb[r][q];
          }
        }
      }
    }
    __syncthreads();
    }
  };
  // dimensional splitting: one sweep
  [[maybe_unused]] auto sweep = [&](auto dirc) {
    constexpr int dir = decltype(dirc)::value;
    // lines swept: -2..M+1 (x), 0..M-1 (y)
    constexpr int NRL = dir == 0 ? M + 4 : M, L0 = dir == 0 ? -2 : 0;
    const R* sn = dir == 0 ? shu : shv;  // normal momentum
    const R* st = dir == 0 ? shv : shu;  // transverse momentum
    const R nu = dir == 0 ? nux : nuy;
    // phase 1: Riemann solves on the lines, edges -1..M+1.  Consecutive
    // threads take consecutive cells of a row: along the row in the x sweep,
    // across the lines in the y sweep (a column walk would make every tile
    // load a 4-way shared-memory bank conflict); each edge's wave planes
    // keep their place, so the work is the same whichever thread does it
    for (int k = tid; k < NRL * NE; k += NT) {
      const int line = (dir == 0 ? k / NE : k % NRL) + L0;
      const int a = (dir == 0 ? k % NE : k / NRL) - 1;
      const int cl = dir == 0 ? tix<M>(a - 1, line) : tix<M>(line, a - 1);
      const int cr = dir == 0 ? tix<M>(a, line) : tix<M>(line, a);
      // waves in planes: component q of edge e at W[q * NEDGE + e], e the
      // edge's place (line, a) in the sweep
      R* w = W + ((line - L0) * NE + a + 1);
      R Z[9], S[3];
      gfk::riemann<R, DEV>(
          gfk::Side<R>{sdep[cl], sn[cl], st[cl], sb[cl], s0[cl], wetc(cl)},
          gfk::Side<R>{sdep[cr], sn[cr], st[cr], sb[cr], s0[cr], wetc(cr)}, g,
          rdry, Z, S);
#pragma unroll
      for (int q = 0; q < 9; ++q)
        if (!(DEV && q == 3)) w[q * NEDGE] = Z[q];  // FP32: Z[3] is zero, not read
      w[9 * NEDGE] = S[0];
      w[10 * NEDGE] = S[1];
      w[11 * NEDGE] = S[2];
    }
    __syncthreads();
    // phase 2: fluctuations and limited corrections on edges 0..M
    R AMr[RL][3], APr[RL][3], FFr[RL][3];
#pragma unroll
    for (int r = 0; r < RL; ++r) {
      const int k = tid + r * NT;
      if (k < NRL * (M + 1)) {
        const int line = k / (M + 1) + L0, a = k % (M + 1);
        const int e = (line - L0) * NE + a + 1;
        const R* w = W + e;
        const int cl = dir == 0 ? tix<M>(a - 1, line) : tix<M>(line, a - 1);
        const int cr = dir == 0 ? tix<M>(a, line) : tix<M>(line, a);
        const bool wet = corr && wetc(cl) && wetc(cr);
        gfk::edge_fluxes<R, NEDGE, DEV>(w, w + 9 * NEDGE, w - 1, w + 1, nu, wet,
                                        AMr[r], APr[r], FFr[r]);
        if (line >= 0 && line < M) {
          R m = R(0);
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const R sq = w[(9 + q) * NEDGE];
            const R as = sq > R(0) ? sq : -sq;
            m = as > m ? as : m;
          }
          if (dir == 0) smx = m > smx ? m : smx;
          else smy = m > smy ? m : smy;
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RL; ++r) {
      const int k = tid + r * NT;
      if (k < NRL * (M + 1)) {
        const int line = k / (M + 1) + L0, a = k % (M + 1);
        R* w = W + ((line - L0) * NE + a + 1);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          w[q * NEDGE] = AMr[r][q];
          w[(3 + q) * NEDGE] = APr[r][q];
          w[(6 + q) * NEDGE] = FFr[r][q];
        }
      }
    }
    __syncthreads();
    // phase 3: per-cell increments, and the intermediate state of the x sweep
#pragma unroll
    for (int r = 0; r < RX; ++r) {
      const int k = tid + r * NT;
      if (k < M * NRL) {
        int a, line;  // a: position along the sweep, line: across
        cell_item<M, NRL, L0>(k, dir, a, line);
        const R* wl = W + ((line - L0) * NE + a + 1);  // edge a
        const R* wr = wl + 1;                           // edge a+1
        R d[3];  // frame: mass, normal (sweep) momentum, transverse
#pragma unroll
        for (int q = 0; q < 3; ++q)
          d[q] = (wl[(3 + q) * NEDGE] + wr[q * NEDGE]) +
                 (wr[(6 + q) * NEDGE] - wl[(6 + q) * NEDGE]);
        if (dir == 1 && r < RC) {  // nu * dQ in (h, hu, hv) order
          Y[r][0] = nu * d[0]; Y[r][1] = nu * d[2]; Y[r][2] = nu * d[1];
        }
        if constexpr (dir == 0) {
          // intermediate state of cell (a, line) in place: every read of
          // the window in this sweep is behind the barriers above
          const int c = tix<M>(a, line);
          const bool inner = k < M * M;
          const R xs[3] = {nu * d[0], nu * d[1], nu * d[2]};
          const R q[3] = {s0[c], shu[c], shv[c]};
          R o[3];
          if (inner) nwet += wetc(c) ? 1u : 0u;
          if constexpr (!DEV) {
#pragma unroll
            for (int f = 0; f < 3; ++f) o[f] = q[f] - xs[f];
            if (o[0] < R(0)) {
              if (inner) { clipd -= o[0]; ++nclip; }
              o[0] = R(0);
            }
            if (o[0] <= rdry) { o[1] = R(0); o[2] = R(0); }
          } else {
            const int kp = pix(a, line);
            float lo[3];
#pragma unroll
            for (int f = 0; f < 3; ++f) {
              const float x = (inner ? los[f * MP * MP + kp] : 0.0f) - xs[f];
              const float s = q[f] + x;
              const float bb = s - q[f];
              lo[f] = (q[f] - (s - bb)) + (x - bb);
              o[f] = s;
            }
            const float bc = sb[c];
            if (o[0] < bc) {
              if (inner) { clipf += bc - o[0]; ++nclip; }
              o[0] = bc;
              lo[0] = 0.0f;
            }
            const bool wnew = gfk::wet_dev(o[0], bc, drytol, dtf, margin);
            if (!wnew) { o[1] = 0.0f; o[2] = 0.0f; lo[1] = 0.0f; lo[2] = 0.0f; }
            sdep[c] = o[0] - bc;
            swet[c] = wnew ? 1 : 0;
            if (inner && r < RC) {
              LO1[r][0] = lo[0]; LO1[r][1] = lo[1]; LO1[r][2] = lo[2];
            }
          }
          s0[c] = o[0];
          shu[c] = o[1];
          shv[c] = o[2];
        }
      }
    }
    __syncthreads();
  };
  if (anywet) {
    if constexpr (FAST) {
      sweep32(std::integral_constant<int, 0>{});
      sweep32(std::integral_constant<int, 1>{});
    } else if constexpr (BOTH) {
      const int half = tid / HN;
      sweep64(half, tid % HN, W + half * Lo::NWP * NEDGE);
    } else if constexpr (PRIM) {
#pragma unroll 1
      for (int dir = 0; dir < 2; ++dir) sweep64(dir, tid, W);
    } else {
      sweep(std::integral_constant<int, 0>{});
      sweep(std::integral_constant<int, 1>{});
    }
  }
  // interior cell of round r (or -1): its index in the M x M tile
  auto owned = [&](int r) -> int {
    const int k = tid + r * NT;
    return k < M * M ? k : -1;
  };

  // New values of a cell near the patch edge also go to the ghost cells that
  // copy or mirror it (same-level neighbours, physical boundaries).
  R* qnext;
  if constexpr (DEV) qnext = V.qf[cur ^ 1];
  else qnext = V.q[cur ^ 1];
  const int nxp = G.mi << Pt.level, nyp = G.mj << Pt.level;
  auto push_edge = [&](int gi, int gj, R v0, R v1, R v2) {
    emit_edge<R, MP>(qnext, p, Pt.px, Pt.py, nxp, nyp, snb, G.bc, push, gi, gj, v0, v1, v2);
  };

  // ------------------------------------------------ update, friction, out
  const R mn = rscal[4];
  bool bad = false;
  // the compensation terms of every owned cell requested at once, so that
  // their global loads overlap instead of one wait per cell
  if constexpr (FAST) {
    if (anywet) {
      f2 lpre[RC][3];
#pragma unroll
      for (int r = 0; r < RC; ++r) {
        const int i = 2 * (tid % M2), j = tid / M2 + r * TLC;
        if ((unsigned)j >= (unsigned)M) continue;
#pragma unroll
        for (int f = 0; f < 3; ++f) lpre[r][f] = gfk::ld2(los + f * MP * MP + pix(i, j));
      }
      // new values of the tile for the edge cells' copies below; the wave
      // planes are free since the last barrier
      R* nv = W;
#pragma unroll
      for (int r = 0; r < RC; ++r) {
        const int i = 2 * (tid % M2), j = tid / M2 + r * TLC;
        if ((unsigned)j >= (unsigned)M) continue;
        const int c = tix<M>(i, j), cg = gix(i, j), kp = pix(i, j);
        // compensated update: (hi + lo) - change, hi rounded, lo the error
        f2 o2[3], l2[3];
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          const f2 q = gfk::ld2((f == 0 ? s0 : (f == 1 ? shu : shv)) + c);
          const f2 x = gfk::sub2(gfk::sub2(lpre[r][f], XP[r][f]), TP[r][f]);
          const f2 sum = gfk::add2(q, x), bb = gfk::sub2(sum, q);
          l2[f] = gfk::add2(gfk::sub2(q, gfk::sub2(sum, bb)), gfk::sub2(x, bb));
          o2[f] = sum;
        }
        float o[2][3], lo[2][3], bc[2], qc[2];
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          gfk::upk(o2[f], o[0][f], o[1][f]);
          gfk::upk(l2[f], lo[0][f], lo[1][f]);
        }
        gfk::upk(gfk::ld2(sb + c), bc[0], bc[1]);
        gfk::upk(gfk::ld2(sq + c), qc[0], qc[1]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          nwet += qc[h] > 0.0f ? 1u : 0u;
          if (o[h][0] < bc[h]) {  // negative depth: reset to a dry bed
            clipf += bc[h] - o[h][0];
            o[h][0] = bc[h];
            lo[h][0] = 0.0f;
            ++nclip;
          }
          const bool wnew = gfk::wet_dev(o[h][0], bc[h], drytol, dtf, margin);
          if (mn > 0.0f && wnew) {
            // approximate reciprocals and h^(-4/3) by the fast power
            // (relative error about 1e-6, far inside this path's tolerance)
            const float d = o[h][0] - bc[h];
            const float rh = gfk::rcpf(d);
            const float u = __fmul_rn(o[h][1], rh), v = __fmul_rn(o[h][2], rh);
            const float sp = sqrtf(fmaf(u, u, __fmul_rn(v, v)));
            const float D = g * mn * mn * sp * __powf(d, -4.0f / 3.0f);
            const float rden = gfk::rcpf(fmaf(dtr, D, 1.0f));
            o[h][1] = __fmul_rn(o[h][1], rden);
            o[h][2] = __fmul_rn(o[h][2], rden);
            lo[h][1] = __fmul_rn(lo[h][1], rden);
            lo[h][2] = __fmul_rn(lo[h][2], rden);
          }
          if (!wnew) { o[h][1] = 0.0f; o[h][2] = 0.0f; lo[h][1] = 0.0f; lo[h][2] = 0.0f; }
          bad |= !(isfinite(o[h][0]) && isfinite(o[h][1]) && isfinite(o[h][2]));
        }
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          const f2 v = gfk::pk(o[0][f], o[1][f]);
          gfk::st2(lod + f * MP * MP + kp, gfk::pk(lo[0][f], lo[1][f]));
          gfk::st2(qd + f * TG + cg, v);
          gfk::st2(nv + f * M * M + j * M + i, v);
        }
      }
      __syncthreads();
      // Copies of the cells within two of the tile's edge.
      if (M == MP) {
        // Every ghost cell that takes one of this patch's values, region by
        // region: bottom and top (2 M each, along x), left and right, then the
        // corners.  In the domain it is a cell of the neighbour there; beyond
        // its boundary a mirror cell of this patch or, at a corner beyond one
        // side only, of the neighbour along the other.
        const bool inland = Pt.px > 0 && Pt.px < nxp - 1 && Pt.py > 0 && Pt.py < nyp - 1;
        for (int k = tid; k < 8 * M + 16; k += NT) {
          int r, i, j;  // region, source cell
          if (k < 4 * M) {
            r = 2 + k / (2 * M);
            i = k % M;
            j = k / M + (r == 3 ? M - 4 : 0);
          } else if (k < 8 * M) {
            const int x = k - 4 * M;
            r = x / (2 * M);
            i = x % 2 + (r ? M - 2 : 0);
            j = x / 2 % M;
          } else {
            const int x = k - 8 * M;
            r = 4 + x / 4;
            i = x % 2 + (r & 1 ? M - 2 : 0);
            j = x / 2 % 2 + (r & 2 ? M - 2 : 0);
          }
          // its direction
          const int sx = r == 0 || r == 4 || r == 6 ? -1 : (r == 1 || r == 5 || r == 7 ? 1 : 0);
          const int sy = r == 2 || r == 4 || r == 5 ? -1 : (r == 3 || r == 6 || r == 7 ? 1 : 0);
          if (inland) {  // (most patches: no mirrors)
            const int pn = push ? snb[r] : -1;
            if (pn < 0) continue;
            const R* v = nv + j * M + i;
            R* d = qnext + (size_t)pn * 3 * TG + tix<M>(i - sx * M, j - sy * M);
            d[0] = v[0];
            d[TG] = v[M * M];
            d[2 * TG] = v[2 * M * M];
            continue;
          }
          const bool bx = sx != 0 && (unsigned)(Pt.px + sx) >= (unsigned)nxp;
          const bool by = sy != 0 && (unsigned)(Pt.py + sy) >= (unsigned)nyp;
          // the patch that holds it
          const int rr = r < 4 ? r : (bx ? (sy < 0 ? 2 : 3) : (by ? (sx < 0 ? 0 : 1) : r));
          const bool self = (bx || sx == 0) && (by || sy == 0);
          const int pn = self ? p : (push ? snb[rr] : -1);
          if (pn < 0) continue;
          // its cell there: beyond the opposite edge, or the mirror (wall: the
          // n-th ghost takes the n-th cell, extrapolation: the first)
          int gi = i - sx * M, gj = j - sy * M;
          R fx = R(1), fy = R(1);
          if (bx) {
            gi = sx < 0 ? -1 - i : 2 * M - 1 - i;
            if (G.bc[sx < 0 ? 0 : 1] == 0) fx = R(-1);
            else i = sx < 0 ? 0 : M - 1;
          }
          if (by) {
            gj = sy < 0 ? -1 - j : 2 * M - 1 - j;
            if (G.bc[sy < 0 ? 2 : 3] == 0) fy = R(-1);
            else j = sy < 0 ? 0 : M - 1;
          }
          const R* v = nv + j * M + i;
          R* d = qnext + (size_t)pn * 3 * TG + tix<M>(gi, gj);
          d[0] = v[0];
          d[TG] = fx * v[M * M];
          d[2 * TG] = fy * v[2 * M * M];
        }
      } else
      // otherwise cell by cell, side by side, so that a warp takes cells of
      // the same kind (updating and copying in one loop sent every warp
      // through the copies for its two outer columns)
      for (int k = tid; k < 8 * M - 16; k += NT) {
        int i, j;
        if (k < 4 * M) {
          i = k % M;
          j = k < 2 * M ? k / M : M - 4 + k / M;
        } else {
          const int r = k - 4 * M, x = r / (M - 4);
          j = 2 + r % (M - 4);
          i = x < 2 ? x : M - 4 + x;
        }
        const R* v = nv + j * M + i;
        push_edge(ox + i, oy + j, v[0], v[M * M], v[2 * M * M]);
      }
    } else if (!skip_writes) {
      for (int k = tid; k < M * M; k += NT) {
        const int i = k % M, j = k / M, cg = gix(i, j), kp = pix(i, j);
        const float w = s0[tix<M>(i, j)];
        qd[cg] = w;
        qd[TG + cg] = 0.0f;
        qd[2 * TG + cg] = 0.0f;
        push_edge(ox + i, oy + j, w, 0.0f, 0.0f);
        lod[kp] = los[kp];
        lod[MP * MP + kp] = 0.0f;
        lod[2 * MP * MP + kp] = 0.0f;
      }
    }
  }
#pragma unroll
  for (int r = 0; r < (FAST ? 0 : RC); ++r) {
    const int k = owned(r);
    if (k < 0) continue;
    const int i = k % M, j = k / M;
    const int c = tix<M>(i, j);
    const int cg = gix(i, j), kp = pix(i, j);
    if (!anywet) {
      if (!skip_writes) {
        qd[cg] = s0[c];
        qd[TG + cg] = R(0);
        qd[2 * TG + cg] = R(0);
        push_edge(ox + i, oy + j, s0[c], R(0), R(0));
        if constexpr (DEV) {
          lod[kp] = los[kp];
          lod[MP * MP + kp] = 0.0f;
          lod[2 * MP * MP + kp] = 0.0f;
        }
      }
      continue;
    }
    const R q[3] = {s0[c], shu[c], shv[c]};  // split: the intermediate state
    if (!DS) nwet += wetc(c) ? 1u : 0u;
    R o[3];
    if constexpr (!DEV) {
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        R fl;
        if constexpr (BOTH) fl = X[r][f] + W[(Lo::NWP + f) * NEDGE + k];
        else fl = DS ? Y[DS ? r : 0][f] : X[PRIM ? r : 0][f];
        const R* fa = Ftr + 3 * (j * (M + 1) + i);
        const R* ga = Gtr + 3 * (i * (M + 1) + j);
        const R tf = trv ? nux * (fa[3 + f] - fa[f]) + nuy * (ga[3 + f] - ga[f]) : R(0);
        o[f] = (q[f] - fl) - tf;
      }
      if (gfk::neg(o[0])) { gfk::rare(); clipd -= o[0]; o[0] = R(0); ++nclip; }
      const bool wnew = gfk::above(o[0], rdry);
      if (wnew && gfk::pos(mn)) {
        const R u = gfk::div_rn(o[1], o[0]), v = gfk::div_rn(o[2], o[0]);
        const R sp = gfk::sqrt_rn(u * u + v * v);
        const R D = gfk::div_rn(g * mn * mn * sp, o[0] * gfk::cbrt_pos(o[0]));
        const R den = R(1) + dtr * D;
        o[1] = gfk::div_rn(o[1], den);
        o[2] = gfk::div_rn(o[2], den);
      }
      if (!wnew) { o[1] = R(0); o[2] = R(0); }
    } else {
      // compensated update: (hi + lo) - fl - tf, hi rounded, lo the error
      float lo[3];
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        const float x = LO1[DS && DEV ? r : 0][f] - Y[DS ? r : 0][f];
        const float s = q[f] + x;
        const float bb = s - q[f];
        lo[f] = (q[f] - (s - bb)) + (x - bb);
        o[f] = s;
      }
      const float bc = sb[c];
      if (o[0] < bc) {  // negative depth: reset to a dry bed
        clipf += bc - o[0];
        o[0] = bc;
        lo[0] = 0.0f;
        ++nclip;
      }
      const bool wnew = gfk::wet_dev(o[0], bc, drytol, dtf, margin);
      if (mn > 0.0f && wnew) {
        // approximate reciprocals and h^(-4/3) by the fast power (relative
        // error about 1e-6, far inside the FP32 path's tolerance); products
        // rounded on their own, so every kernel variant rounds them alike
        const float h = o[0] - bc;
        const float rh = __fdividef(1.0f, h);
        const float u = __fmul_rn(o[1], rh), v = __fmul_rn(o[2], rh);
        const float sp = sqrtf(fmaf(u, u, __fmul_rn(v, v)));
        const float D = g * mn * mn * sp * __powf(h, -4.0f / 3.0f);
        const float rden = __fdividef(1.0f, fmaf(dtr, D, 1.0f));
        o[1] = __fmul_rn(o[1], rden);
        o[2] = __fmul_rn(o[2], rden);
        lo[1] = __fmul_rn(lo[1], rden);
        lo[2] = __fmul_rn(lo[2], rden);
      }
      if (!wnew) { o[1] = 0.0f; o[2] = 0.0f; lo[1] = 0.0f; lo[2] = 0.0f; }
#pragma unroll
      for (int f = 0; f < 3; ++f) lod[f * MP * MP + kp] = lo[f];
    }
    if constexpr (DEV) {
      bad |= !(isfinite(o[0]) && isfinite(o[1]) && isfinite(o[2]));
    } else {
#pragma unroll
      for (int f = 0; f < 3; ++f) bad |= (gfk::dbits(o[f]) & gfk::D_INF) == gfk::D_INF;
    }
    qd[cg] = o[0];
    qd[TG + cg] = o[1];
    qd[2 * TG + cg] = o[2];
    push_edge(ox + i, oy + j, o[0], o[1], o[2]);
  }
  // block reductions: CFL rate (max) and wet-cell count, one atomic of each
  // per CTA
  const int lane = tid & 31, wid = tid >> 5;
  constexpr int NW = NT / 32;
  static_assert(NW <= 32, "one warp reduces the per-warp partials");
  // the partials fit below the broadcast scalars at red + 48
  static_assert(DEV ? 3 * NW <= 96 : 3 * NW <= 48, "reduction area");
  // (speeds are not negative: their bits order as they do)
  if constexpr (DEV) {
    smx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(smx)));
    smy = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(smy)));
  } else {
    smx = warp_max(smx);
    smy = warp_max(smy);
  }
  nwet = __reduce_add_sync(0xffffffffu, nwet);
  if constexpr (DEV) {
    float* redf = reinterpret_cast<float*>(red);
    unsigned* redu = reinterpret_cast<unsigned*>(redf + 2 * NW);
    if (lane == 0) {
      redf[wid] = smx;
      redf[NW + wid] = smy;
      redu[wid] = nwet;
    }
    __syncthreads();
    if (wid == 0) {
      float mx = lane < NW ? redf[lane] : 0.0f;
      float my = lane < NW ? redf[NW + lane] : 0.0f;
      const unsigned nw = __reduce_add_sync(0xffffffffu, lane < NW ? redu[lane] : 0u);
      mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx)));
      my = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(my)));
      if (lane == 0) {
        const float cx = mx * G.inv_dxf[Pt.level], cy = my * G.inv_dyf[Pt.level];
        double cm = (double)(cx > cy ? cx : cy);
        if (subc) cm = cm * (double)per / (double)G.sub_K;  // cmax / n_L
        atomicMax(&C->cmax_bits, (unsigned long long)__double_as_longlong(cm));
        if (nw) atomicAdd(&C->wet_updates, (unsigned long long)nw);
      }
    }
    if (nclip) {
      atomicAdd(&C->step_nclip, (unsigned long long)nclip);
      atomicAdd(&C->step_clipvol, (double)clipf * G.areal[Pt.level]);
    }
  } else {
    const double dx = scal[0], dy = scal[1];
    unsigned* redu = reinterpret_cast<unsigned*>(red + 2 * NW);
    if (lane == 0) {
      red[wid] = (double)smx;
      red[NW + wid] = (double)smy;
      redu[wid] = nwet;
    }
    __syncthreads();
    if (tid == 0) {
      double mx = 0.0, my = 0.0;
      unsigned nw = 0u;
      for (int w = 0; w < NW; ++w) {
        mx = gfk::dmax(red[w], mx);
        my = gfk::dmax(red[NW + w], my);
        nw += redu[w];
      }
      double cm = gfk::dmax(gfk::div_rn(mx, dx), gfk::div_rn(my, dy));
      if (subc) cm = gfk::div_rn(cm * (double)per, (double)G.sub_K);  // cmax / n_L
      atomicMax(&C->cmax_bits, (unsigned long long)__double_as_longlong(cm));
      if (nw) atomicAdd(&C->wet_updates, (unsigned long long)nw);
    }
    if (nclip) {
      atomicAdd(&C->step_nclip, (unsigned long long)nclip);
      atomicAdd(&C->step_clipvol, clipd * (dx * dy));
    }
  }
  if (bad) C->nonfinite = 1;
  return anywet;
}

// Controller of a subcycled macro step (one thread of the last CTA of each
// substep launch per scenario).  The macro step of DT = dt_use runs as
// sub_K substeps; the rates cmax / n_L of the levels that stepped arrived in
// cmax_bits.  Substep 0 (every level steps) is checked against cfl_max: a
// violation rejects the macro step, whose remaining substeps then do
// nothing, and it is retaken with DT = cfl_desired / rate.  Later substeps
// are not checked; their rates bound the next DT.  After the last substep
// the time advances by DT and the next macro step is set up.
static __device__ void subcycle_finish(const GfGeom& G, const GfView& V, GfCtl* Cp,
                                       int s, int cells_per_patch) {
  // every field the rule needs, read from L2 at once
  const int K = G.sub_K;
  const int k = __ldcg(&Cp->sub_k), sub_rej = __ldcg(&Cp->sub_rej);
  const double rate = __longlong_as_double((long long)__ldcg(&Cp->cmax_bits));
  const double DT = __ldcg(&Cp->dt_use);
  const double t = __ldcg(&Cp->t), t_target = __ldcg(&Cp->t_target);
  const double dt_next0 = __ldcg(&Cp->dt_next);
  const double clipvol = __ldcg(&Cp->clipvol), step_clipvol = __ldcg(&Cp->step_clipvol);
  const unsigned long long step_nclip = __ldcg(&Cp->step_nclip);
  const unsigned long long cell_updates = __ldcg(&Cp->cell_updates);
  const unsigned long long rmax_bits = __ldcg(&Cp->rmax_bits);
  const long long steps = __ldcg(&Cp->steps), rejects = __ldcg(&Cp->rejects);
  const long long nclip = __ldcg(&Cp->nclip), taken = __ldcg(&Cp->taken);
  const long long max_steps = __ldcg(&Cp->max_steps);
  const int inrow = __ldcg(&Cp->inrow), lastf = __ldcg(&Cp->last);
  const int nonfinite = __ldcg(&Cp->nonfinite);
  if (!__ldcg(&Cp->active)) {
    Cp->accepted = 0;
    return;
  }
  Cp->cmax_bits = 0ull;
  const bool end = k == K - 1;
  double tn = t, dtn = dt_next0;
  long long tk = taken;
  if (nonfinite) {
    Cp->status = -5;  // GEOFLOOD_ERR_NAN
    Cp->active = 0;
    Cp->accepted = 0;
    return;
  }
  if (sub_rej) {
    Cp->accepted = 0;
  } else if (k == 0 && DT * rate > G.cfl_max) {
    dtn = gfk::div_rn(G.cfl_desired, rate);
    Cp->dt_next = dtn;
    Cp->rejects = rejects + 1;
    Cp->accepted = 0;
    Cp->step_nclip = 0ull;
    Cp->step_clipvol = 0.0;
    Cp->rmax_bits = 0ull;
    Cp->inrow = inrow + 1;
    Cp->sub_rej = 1;
    if (inrow + 1 > GF_MAXSTEP_REJECT) {
      Cp->status = -4;  // GEOFLOOD_ERR_CFL
      Cp->active = 0;
      return;
    }
  } else {
    // the substep stands: count the levels that stepped
    unsigned long long cells = 0ull;
    for (int L = G.minlevel; L <= G.maxlevel; ++L)
      if (k % (1 << (G.maxlevel - L)) == 0)
        cells += (unsigned long long)V.scen[s].lcount[L] * (unsigned long long)cells_per_patch;
    Cp->cell_updates = cell_updates + cells;
    unsigned long long rb = rmax_bits;
    if (rate > __longlong_as_double((long long)rmax_bits))
      rb = (unsigned long long)__double_as_longlong(rate);
    Cp->nclip = nclip + (long long)step_nclip;
    Cp->clipvol = clipvol + step_clipvol;
    Cp->step_nclip = 0ull;
    Cp->step_clipvol = 0.0;
    Cp->accepted = 1;
    if (end) {
      tn = lastf ? t_target : t + DT;
      tk = taken + 1;
      Cp->inrow = 0;
      Cp->t = tn;
      Cp->steps = steps + 1;
      Cp->taken = tk;
      const double r = __longlong_as_double((long long)rb);
      rb = 0ull;
      if (r > 0.0) {
        const double dn = gfk::div_rn(G.cfl_desired, r);
        dtn = dn < G.dt_max ? dn : G.dt_max;
        Cp->dt_next = dtn;
      }
    }
    Cp->rmax_bits = rb;
  }
  if (!end) {
    Cp->sub_k = k + 1;
    return;
  }
  Cp->sub_k = 0;
  Cp->sub_rej = 0;
  if (!(tn < t_target) || tk >= max_steps) {
    Cp->active = 0;
  } else {
    const double rem = t_target - tn;
    if (dtn < rem) { Cp->dt_use = dtn; Cp->last = 0; }
    else { Cp->dt_use = rem; Cp->last = 1; }
  }
}

// CFL rule of one scenario at the end of a step (Sec. 5.1 maximum CFL,
// Sec. 6.6), not subcycled: reject the step and set a smaller dt when
// dt*cmax exceeds cfl_max, else accept it (swap the state buffers, advance
// t) and pick the next dt = cfl_desired / cmax, clipped to land on t_target.
// One thread runs it: every field it needs is read from L2 at once
// (independent loads, one round trip instead of one per field), the
// decision is taken on the copies, and only the fields that change are
// written back.
static __device__ void ctl_finish(const GfGeom& G, GfCtl* Cp, unsigned long long cells) {
  const double cmax = __longlong_as_double((long long)__ldcg(&Cp->cmax_bits));
  const double dt = __ldcg(&Cp->dt_use);
  const double t = __ldcg(&Cp->t), t_target = __ldcg(&Cp->t_target);
  const double dt_next0 = __ldcg(&Cp->dt_next);
  const double clipvol = __ldcg(&Cp->clipvol), step_clipvol = __ldcg(&Cp->step_clipvol);
  const unsigned long long step_nclip = __ldcg(&Cp->step_nclip);
  const unsigned long long cell_updates = __ldcg(&Cp->cell_updates);
  const long long steps = __ldcg(&Cp->steps), rejects = __ldcg(&Cp->rejects);
  const long long nclip = __ldcg(&Cp->nclip), taken = __ldcg(&Cp->taken);
  const long long max_steps = __ldcg(&Cp->max_steps);
  const int cur = __ldcg(&Cp->cur), lastf = __ldcg(&Cp->last);
  const int inrow = __ldcg(&Cp->inrow), nonfinite = __ldcg(&Cp->nonfinite);
  if (!__ldcg(&Cp->active)) {
    Cp->accepted = 0;
    return;
  }
  Cp->cell_updates = cell_updates + cells;
  Cp->cmax_bits = 0ull;
  if (nonfinite) {
    Cp->status = -5;  // GEOFLOOD_ERR_NAN
    Cp->active = 0;
    Cp->accepted = 0;
    return;
  }
  double tn = t, dtn = dt_next0;
  long long tk = taken;
  if (dt * cmax > G.cfl_max) {
    dtn = gfk::div_rn(G.cfl_desired, cmax);
    Cp->dt_next = dtn;
    Cp->rejects = rejects + 1;
    Cp->accepted = 0;
    Cp->step_nclip = 0ull;
    Cp->step_clipvol = 0.0;
    Cp->inrow = inrow + 1;
    if (inrow + 1 > GF_MAXSTEP_REJECT) {
      Cp->status = -4;  // GEOFLOOD_ERR_CFL
      Cp->active = 0;
      return;
    }
  } else {
    tn = lastf ? t_target : t + dt;
    tk = taken + 1;
    Cp->inrow = 0;
    Cp->cur = cur ^ 1;
    Cp->t = tn;
    Cp->steps = steps + 1;
    Cp->taken = tk;
    Cp->nclip = nclip + (long long)step_nclip;
    Cp->clipvol = clipvol + step_clipvol;
    Cp->step_nclip = 0ull;
    Cp->step_clipvol = 0.0;
    Cp->accepted = 1;
    if (cmax > 0.0) {
      const double dn = gfk::div_rn(G.cfl_desired, cmax);
      dtn = dn < G.dt_max ? dn : G.dt_max;
      Cp->dt_next = dtn;
    }
  }
  if (!(tn < t_target) || tk >= max_steps) {
    Cp->active = 0;
  } else {
    const double rem = t_target - tn;
    if (dtn < rem) { Cp->dt_use = dtn; Cp->last = 0; }
    else { Cp->dt_use = rem; Cp->last = 1; }
  }
}

// End of a step: the last of the nctas working CTAs to finish applies the CFL rule to every active
// scenario, one thread per scenario (the scenarios' rules are independent).
// The volume of the state is not part of the step; geoflood_mass computes it
// on demand.
template <int NT>
__device__ void step_finish(const GfGeom& G, const GfView& V, int cells_per_patch, bool wrote,
                            unsigned nctas) {
  __shared__ int last;
  __syncthreads();
  if (threadIdx.x == 0) {
    // a CTA that updated the controller's counters (atomics) orders them
    // before it counts itself done; one that did not needs no fence
    if (wrote) __threadfence();
    const unsigned t = atomicAdd(V.done, 1u);
    last = t == nctas - 1u;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int s = threadIdx.x; s < G.nscen; s += NT) {
    GfCtl* Cp = V.ctl + s;
    if (G.subcycle)
      subcycle_finish(G, V, Cp, s, cells_per_patch);
    else
      ctl_finish(G, Cp, (unsigned long long)V.scen[s].pcount * (unsigned long long)cells_per_patch);
  }
  // the next launch reads the counters and the schedule after this kernel
  // has ended, which orders these writes before it (a thread without a
  // scenario, if there is one: its loads go beside the controller's)
  if (threadIdx.x == NT - 1 && V.sched) {
    const unsigned count = V.sched[0], par = count & 1u;
    // patches that took no step, at the tail of the next order
    // (in the word this launch does not read: CTAs beyond the working ones
    // may start after this and must still find themselves beyond).  CTAs that
    // did not fence may have entries on their way that this does not count;
    // those patches get CTAs of their own next time.
    unsigned tail;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];"
                 : "=r"(tail)
                 : "l"(V.sched + 2 + 2 * par)
                 : "memory");
    V.sched[0] = (count + 1u) % 6u;
    // After a write of the state nothing is known for two launches.
    if (V.inactive) {
      const unsigned none = (unsigned)V.npatch + 1u, idle = V.inactive[V.parity];
      V.inactive[V.parity ^ 1u] = idle < none ? tail : (idle == none ? 0u : none);
    }
    // the next launch's counters, which no CTA of this one touches: its own
    // may still be counted up
    V.sched[3 - 2 * par] = 0u;
    V.sched[4 - 2 * par] = 0u;
  }
  if (threadIdx.x == 0) *V.done = 0u;
}

// patch_body out of line, for the rare tiles that a CTA takes one after the
// other: inlined into a loop, everything that does not depend on the tile
// would be kept in registers across the tiles and spilled (1.6 KB a thread).
template <class P, int MP, int M, int NT, bool DS>
__device__ __noinline__ int patch_body_call(const GfGeom& G, const GfView& V, const int p,
                                            const int sub, const TileHdr& H, TmaPhase* tp,
                                            bool* wrote) {
  extern __shared__ __align__(16) unsigned char smraw[];
  return patch_body<P, MP, M, NT, DS>(G, V, smraw, p, sub, H, tp, wrote);
}

template <class P, int MP, int M, int NT, int MINB, bool DS = false>
__global__ void __launch_bounds__(NT, MINB)
    k_patch_step(const __grid_constant__ GfGeom G,
                 const __grid_constant__ GfView V) {
  extern __shared__ __align__(16) unsigned char smraw[];
  using Lo = Layout<P, M, DS>;
  constexpr int NSUB = (MP / M) * (MP / M);
  // (the FP64 tiles' own time hides their dry neighbours' CTAs)
  constexpr bool GROUPS = Lo::FAST;
  constexpr int GRP = GF_STEP_GROUP;
  const int slot = blockIdx.x / NSUB, sub = blockIdx.x % NSUB;
  // The launch order (see GfView::sched): first the patches that took the
  // step in the previous launch, one CTA each (or one per sub-tile), then
  // those that did not, GRP to a CTA, which usually finds that none of them
  // has to; the CTAs beyond return.  Among the first, short dry tiles stay
  // between the wet ones: with the wet ones strictly ahead the CTAs of an SM
  // run through their phases side by side and wait for the same unit
  // (1024 x 1024 grid: 47.6 us a step against 42.7, FP64 568 against 525).  A CTA is a chain of dependent loads, so
  // what the later ones need is read together: the counter, both orders'
  // entries and, when there is one scenario, its controller.
  const bool sched = V.sched != nullptr && V.done != nullptr;
  const bool use_flags = !DS && sched && V.runf != nullptr && !G.subcycle;
  const bool one = G.nscen == 1;
  unsigned count = 0u, idle = 0u;
  int e0 = slot, e1 = slot;
  if (sched) {
    count = V.sched[0];
    e0 = V.ord0[slot];
    e1 = V.ord1[slot];
    if (GROUPS && use_flags) idle = V.inactive[V.parity];
  }
  // Not known (the first two launches after a write): every patch runs and by
  // itself, and the order is kept, which the launches before the write made.
  // Entered as they end, the patches without water, which are done at once,
  // would come first and hold up the tiles with water, whose chain is the
  // launch's time; entered last, they would leave all wet tiles side by side
  // (see above) for as long as the state stands.  Six steps from a write of 400
  // patches of 32 x 32 with a front 162 us entered as they end, 151 kept; of 576
  // patches 223 and 199; 1024 patches, 64 steps 3.35, 3.55 (last) and 3.29 ms.
  const bool unknown = idle > (unsigned)V.npatch;
  const int inactive = unknown ? 0 : (int)idle;
  const int nact = V.npatch - inactive;
  const unsigned working =
      GROUPS ? (unsigned)(nact + (inactive + GRP - 1) / GRP) * NSUB : gridDim.x;
  if (GROUPS && blockIdx.x >= working) return;
  int act = 0, cur = 0, acc = 0;
  double dt = 0.0;
  if (one) {
    const GfCtl& C = V.ctl[0];
    act = C.active;
    cur = C.cur;
    acc = C.accepted;
    dt = C.dt_use;
  }
  const unsigned par = count & 1u, r3 = count % 3u;
  const int* ord = par ? V.ord1 : V.ord0;
  // run flags (GfView::runf): this launch's, the next one's, and the array
  // that is cleared for the one after
  auto flags = [&](unsigned k) { return V.runf + (size_t)((r3 + k) % 3u) * V.runf_stride; };
  int first = slot, n = 1;
  const bool group = GROUPS && slot >= nact;
  if (group) {
    first = nact + (slot - nact) * GRP;
    n = V.npatch - first < GRP ? V.npatch - first : GRP;
  }
  // lane l of every warp looks at patch l of the CTA: its run flag and
  // whether it may stand still (a dry, unchanged tile or sub-tile of an
  // unmarked patch without a gauge: the full path would find its ghost ring
  // dry and write nothing)
  const int lane = threadIdx.x & 31;
  int pl = -1;
  int4 rec = make_int4(0, 0, 0, 0);  // its patch record
  bool marked = false, same = false, gauge = false, skip = false;
  if (lane < n) {
    pl = group ? ord[first + lane] : (par ? e1 : e0);
    marked = use_flags && flags(0u)[pl] != 0;
    same = V.same != nullptr && V.same[pl * NSUB + sub] != 0;
    gauge = V.gflag != nullptr && V.gflag[pl] != 0;
    rec = *reinterpret_cast<const int4*>(V.patch + pl);
    skip = use_flags && !marked && same && !gauge;
    if (use_flags && sub == 0 && threadIdx.x < 32) {
      flags(2u)[pl] = 0;
      int* nxt = par ? V.ord0 : V.ord1;
      if (unknown)
        nxt[slot] = pl;
      else if (skip)
        nxt[V.npatch - 1 - (int)atomicAdd(order_ends(V, nxt) + 1, 1u)] = pl;
    }
  }
  unsigned todo = __ballot_sync(0xffffffffu, lane < n && !skip);
  bool wrote = false;
  // patch of lane l; body runs its tile
  auto take = [&](int l, auto body) -> int {
    const int p = __shfl_sync(0xffffffffu, pl, l);
    TileHdr H;
    H.Pt = GfPatch{__shfl_sync(0xffffffffu, rec.x, l), __shfl_sync(0xffffffffu, rec.y, l),
                   __shfl_sync(0xffffffffu, rec.z, l), __shfl_sync(0xffffffffu, rec.w, l)};
    H.same_in = __shfl_sync(0xffffffffu, same ? 1 : 0, l) != 0;
    H.has_gauge = __shfl_sync(0xffffffffu, gauge ? 1 : 0, l) != 0;
    if (!one) {
      const GfCtl& C = V.ctl[H.Pt.scen];
      act = C.active;
      cur = C.cur;
      acc = C.accepted;
      dt = C.dt_use;
    }
    H.cur = cur;
    H.accepted = acc;
    H.dt = dt;
    bool run = act != 0;
    if (run && G.subcycle) {
      // level subcycling: only the levels due at this substep step
      const GfCtl& C = V.ctl[H.Pt.scen];
      run = !C.sub_rej && C.sub_k % (1 << (G.maxlevel - H.Pt.level)) == 0;
    }
    int* nxt = sched && sub == 0 && !unknown ? (par ? V.ord0 : V.ord1) : nullptr;
    H.order = nxt;
    int wet = 0;
    if (run) {
      bool w = true;
      wet = body(p, H, &w);
      wrote |= w;
    }
    if (use_flags) {
      // a patch that did not run carries its mark forward
      if (threadIdx.x == 0 && !run) flags(1u)[p] = 1;
      if (wet && threadIdx.x < 9) {
        // water in this tile: it and its same-level neighbours run next
        // launch (their indices were staged in shared memory by patch_body)
        const int* snb = reinterpret_cast<const int*>(smraw + Lo::OFF_NB);
        const int q = threadIdx.x == 8 ? p : snb[threadIdx.x];
        if (q >= 0) flags(1u)[q] = 1;
      }
    }
    if (nxt != nullptr && threadIdx.x == 0 && !(Lo::FAST && wet > 0)) {
      unsigned* ends = order_ends(V, nxt);
      if (use_flags || wet) nxt[atomicAdd(ends, 1u)] = p;
      else nxt[V.npatch - 1 - (int)atomicAdd(ends + 1, 1u)] = p;
    }
    return wet;
  };
  if (!group) {
    if (todo)
      take(0, [&](int p, const TileHdr& H, bool* w) {
        return patch_body<P, MP, M, NT, DS>(G, V, smraw, p, sub, H, nullptr, w);
      });
  }
  if constexpr (GROUPS) {
  if (group && todo) {
    TmaPhase tp{0u, 0u, false};
    while (todo) {
      const int wet = take(__ffs(todo) - 1, [&](int p, const TileHdr& H, bool* w) {
        return patch_body_call<P, MP, M, NT, DS>(G, V, p, sub, H, &tp, w);
      });
      todo = wet < 0 ? 0u : todo & (todo - 1u);  // a wait gave up: the launch has failed
      // shared memory is reused, first by the next tile's bulk copies
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncthreads();
    }
  }
  }
  if (V.done)
    step_finish<NT>(G, V, MP * MP, wrote, working);
}

// Launch the patch step on every patch: MP x MP patches, M x M sub-tiles
// per CTA of NT threads (MINB CTAs per SM), DS = dimensional splitting.
template <class P, int MP, int M, int NT, int MINB, bool DS = false>
int launch_step(const GfGeom& g, const GfView& v, cudaStream_t st) {
  constexpr size_t bytes = Layout<P, M, DS>::BYTES;
  static bool attr = false;
  if (!attr) {
    if (cudaFuncSetAttribute(k_patch_step<P, MP, M, NT, MINB, DS>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)bytes) != cudaSuccess)
      return -2;
    attr = true;
  }
  constexpr int NSUB = (MP / M) * (MP / M);
  k_patch_step<P, MP, M, NT, MINB, DS><<<v.npatch * NSUB, NT, bytes, st>>>(g, v);
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

}  // namespace gfs
