// Persistent 2D stage kernel for float arithmetic (FP32 and MIXED) on sm_103a,
// for one instance or a batch of instances stacked in shared padded arrays.
//
// A launch is one stage, or several whole RK3 steps of one grid with a barrier
// of the CTAs between stages.  Each CTA walks the work list (tile = blockIdx.x
// + k * gridDim.x).  Thread 0 prepares the next tile -- decodes its instance, decides whether the instance
// still needs work, computes the instance's dt and flux alpha for this stage,
// and issues one TMA box per array (tile plus 3-node halo) into the other half
// of a double buffer on an mbarrier -- while all threads compute the current
// tile:
//   1. both sweeps in one pass, packed two lanes per value (f32x2): each
//      thread sweeps nodes 8w..8w+7 of row `lane` along x (warp w; it reads
//      its cells as 16-byte quads, which the box pitch keeps conflict-free) in
//      lane .x and 8 consecutive nodes of one column along y in lane .y
//      (consecutive lanes read consecutive columns), combining the two MIXED
//      parts (hi + lo, or hi + the previous stage's increment array, which
//      carries lo) as it goes; the sums and differences of the one-sided
//      derivatives go to shared memory;
//   2. each thread forms, for its 8 column nodes, the Lax-Friedrichs
//      Hamiltonian and the RK combination, and stores.
// A CTA keeps running maxima of |dH/dp|, |dH/dq| over consecutive tiles of
// one instance and folds them into the instance's slot (with the number of
// tiles done) when the instance changes; the CTA that completes an instance's
// last tile closes the instance's stage (dt, time, step count, buffer flip),
// so instances advance independently.
//
// What bounds it: instruction issue and the FMA pipe from about 2048^2 up, one tile's latency and the grid barrier
// below.  64 x 32 tiles with 8-node segments keep the work repeated at segment ends and the halo reads small with
// two CTAs (16 warps) per SM.  Measured (GB300, us per RK3 step of Example 3, MIXED; against a staged differences
// pass, the short-interval sweep and a launch per stage): 8192^2 1174 -> 988 alone, a pass of ten steps 13.31 ->
// 11.47 ms; 403 x 397 to t = 0.5/pi^2 2633 -> 1689 us; FP32 2048^2, forty steps 5314 -> 3074 us.  Slower than it was:
// FP32 with a trigonometric Hamiltonian on grids so fine that all segments sweep in full (Example 10, 4096^2 465 ->
// 489, 8192^2 1746 -> 1842): there the handover of the column sweep's results through shared memory gains nothing
// (the near-linear form tried in vain is below 1 % of it); and launches of single stages on grids of a few tiles
// with kinks, where a tile waits for the near-linear form and then for its list (a batch of 16 grids of 48^2-96^2, 410
// steps, 14.4 -> 16.1 ms).
#pragma once
#include <type_traits>

#include "alw_device.cuh"
#include "alw_params2d.h"
#include "alw_sweep32.cuh"
#include "alw_tma.cuh"

namespace alw {

// Hamiltonians of the 2D examples in float (compile-time kind), from the sums and differences of a node's
// one-sided derivatives, Sx = u^+ + u^-, Dx = u^+ - u^-, Sy = v^+ + v^-, Dy = v^+ - v^-: value is kUnit H at the mean
// derivatives (a power of two: the finish loop forms kUnit L and steps by dt / kUnit, both exactly, which saves
// Burgers the multiplication by 1/2 of every node), alpha the maximum of |H_p| and |H_q| over the four corners.  u^-+ = (Sx -+ Dx)/2, so the corner
// sums u + v are (Sx + Sy)/2 +- (Dx + Dy)/2 and +- (Dx - Dy)/2, and the largest and smallest |u| are
// (|Sx| +- |Dx|)/2 in magnitude.
template <int H> struct Ham2;
template <> struct Ham2<H_BURGERS2D> {
  static constexpr bool kSameAlpha = true;
  static constexpr float kUnit = 0.5f;
  __device__ __forceinline__ static float value(float su, float sv, float, float) {
    const float z = fmaf(0.25f, su + sv, 0.5f);   // half of p + q + 1
    return z * z;
  }
  // |H_p| = |H_q| = |u + v + 1|: at the largest or the smallest corner sum, (s +- e)/2
  __device__ __forceinline__ static void alpha(float sx, float dx, float sy, float dy, float, float, float &ax,
                                               float &ay) {
    const float s = sx + sy, e = fabsf(dx) + fabsf(dy);
    ax = ay = fmaxf(fmaf(0.5f, s + e, 1.0f), fmaf(0.5f, e - s, -1.0f));
  }
};
// largest |f| over the four corner sums c +- (dx + dy)/2, c +- (dx - dy)/2
template <class F>
__device__ __forceinline__ float corner_max(float c, float dx, float dy, F f) {
  const float p = dx + dy, m = dx - dy;
  return fmaxf(fmaxf(fabsf(f(fmaf(-0.5f, p, c))), fabsf(f(fmaf(-0.5f, m, c)))),
               fmaxf(fabsf(f(fmaf(0.5f, m, c))), fabsf(f(fmaf(0.5f, p, c)))));
}
template <> struct Ham2<H_NEGCOS2D> {
  static constexpr bool kSameAlpha = true;
  static constexpr float kUnit = 1.0f;
  __device__ __forceinline__ static float value(float su, float sv, float, float) {
    return -sfu_cos(fmaf(0.5f, su + sv, 1.0f));
  }
  __device__ __forceinline__ static void alpha(float sx, float dx, float sy, float dy, float, float, float &ax,
                                               float &ay) {
    ax = ay = corner_max(fmaf(0.5f, sx + sy, 1.0f), dx, dy, [](float z) { return sfu_sin(z); });
  }
};
template <> struct Ham2<H_SIN2D> {
  static constexpr bool kSameAlpha = true;
  static constexpr float kUnit = 1.0f;
  __device__ __forceinline__ static float value(float su, float sv, float, float) { return sfu_sin(0.5f * (su + sv)); }
  __device__ __forceinline__ static void alpha(float sx, float dx, float sy, float dy, float, float, float &ax,
                                               float &ay) {
    ax = ay = corner_max(0.5f * (sx + sy), dx, dy, [](float z) { return sfu_cos(z); });
  }
};
template <> struct Ham2<H_EIKONAL2D> {
  static constexpr bool kSameAlpha = false;
  static constexpr float kUnit = 1.0f;
  __device__ __forceinline__ static float value(float su, float sv, float, float) {
    const float p = 0.5f * su, q = 0.5f * sv, t = fmaf(p, p, fmaf(q, q, 1.0f));   // >= 1
    return t * sfu_rsqrt(t);
  }
  __device__ __forceinline__ static void alpha(float sx, float dx, float sy, float dy, float, float, float &ax,
                                               float &ay) {
    // |H_p| = |u| / sqrt(u^2 + v^2 + 1) grows with |u| and falls with |v|
    const float uh = 0.5f * (fabsf(sx) + fabsf(dx)), ul = 0.5f * (fabsf(sx) - fabsf(dx));
    const float vh = 0.5f * (fabsf(sy) + fabsf(dy)), vl = 0.5f * (fabsf(sy) - fabsf(dy));
    ax = uh * sfu_rsqrt(fmaf(uh, uh, fmaf(vl, vl, 1.0f)));
    ay = vh * sfu_rsqrt(fmaf(vh, vh, fmaf(ul, ul, 1.0f)));
  }
};

// Example 11 (optimal control): the only Hamiltonian that depends on the node position (x, y).
template <> struct Ham2<H_OPTCTRL2D> {
  static constexpr bool kSameAlpha = false;
  static constexpr float kUnit = 1.0f;
  __device__ __forceinline__ static float value(float su, float sv, float x, float y) {
    const float p = 0.5f * su, q = 0.5f * sv, sx = sfu_sin(x), cx = sfu_cos(x), sy = sfu_sin(y);
    // sin(y) p + (sin(x) + sign q) q - sin^2(y)/2 - (1 - cos x), with (sign q) q = |q|
    return fmaf(sy, p, fmaf(sx, q, fabsf(q))) - fmaf(0.5f * sy, sy, 1.0f - cx);
  }
  __device__ __forceinline__ static void alpha(float, float, float sv, float dv, float x, float y, float &ax,
                                               float &ay) {
    // H_p = sin y; H_q = sin x + sign q over [min v, max v] = (Sy -+ |Dy|)/2, both signs when it contains q = 0
    const float sx = sfu_sin(x), lo = sv - fabsf(dv), hi = sv + fabsf(dv);
    ax = fabsf(sfu_sin(y));
    ay = (lo <= 0.0f && hi >= 0.0f) ? fabsf(sx) + 1.0f : fabsf(sx + (lo > 0.0f ? 1.0f : -1.0f));
  }
};

// The Hamiltonian of a launch: a compile-time kind, or H_RUNTIME, for batches that run instances
// of several Hamiltonians in one launch: the kind of the tile's instance, dispatched per tile.
constexpr int H_RUNTIME = -1;
// Burgers with a grid-wide or fixed flux alpha: the finish loop does not need each node's alpha, only the
// grid maximum, so it tracks twice the largest and twice the negated smallest corner sum without their + 1 and
// forms max(hi + 1, -(lo + 1)) = max(|hi + 1|, |lo + 1|) once per fold (hi >= lo; the same bits as the largest
// node alpha, the last rounding being monotone)
constexpr int H_BURGERS2D_GRID = -2;
template <int H> struct HamSel {
  static constexpr bool kSameAlpha = Ham2<H>::kSameAlpha;
  static constexpr float kUnit = Ham2<H>::kUnit;
  static constexpr bool kGridFold = false;
  __device__ __forceinline__ float value(float su, float sv, float x, float y) const {
    return Ham2<H>::value(su, sv, x, y);
  }
  __device__ __forceinline__ void alpha(float sx, float dx, float sy, float dy, float x, float y, float &ax,
                                        float &ay) const {
    Ham2<H>::alpha(sx, dx, sy, dy, x, y, ax, ay);
  }
};
template <> struct HamSel<H_BURGERS2D_GRID> : HamSel<H_BURGERS2D> {
  static constexpr bool kGridFold = true;
};
// runtime kind (batches): the finish loop of a tile is that of its instance's kind, chosen once per tile
template <> struct HamSel<H_RUNTIME> {
  static constexpr bool kSameAlpha = false;
  static constexpr bool kGridFold = false;
};

// Segments of a warp (of 64) that are not near-linear from which the warp sweeps them in full itself; fewer are
// shared by the CTA node by node.  Example 10 on 1024^2: 24 segments 63.6 us per step, 40 55.4 us (a kink along a
// grid line fails the 32 segments of one direction).
constexpr int kWarpSegs = 40;
// Reads of the grid barrier's counter before a CTA gives up (about 0.5 us each).
constexpr int kBarrierSpins = 1 << 22;

// Tile geometry of the stage kernel for tiles TXv nodes wide and 32 high (64 or 32 wide): one thread
// per 8-node row segment and 8-node column segment, so TXv / 8 warps; the TMA box is the tile plus
// its halo (4 columns, 3 rows each side); 8 warps per SM per 32 columns of tile width.
template <int TXv>
struct Geo2D {
  static constexpr int TX = TXv, TY = kTile2DY, K = 8, NT = TX * TY / K;
  static constexpr int MINB = 512 / NT;                 // resident CTAs per SM the registers are sized for
  static constexpr int CG = TX / 32;                    // column groups of 32 in the y sweep
  // TMA box: halo 4 columns left, 8 right (3 are read: the row sweeps read their cells as 16-byte quads, and
  // with a pitch of 4 (odd number) floats the quads of a warp's rows fall into distinct banks), 3 rows each side
  static constexpr int SW = TX + 12, SH = TY + 6;
  static constexpr int ARR = ((SH * SW + 31) / 32) * 32; // floats per array slot (128-byte multiple)
  static constexpr int SUP = TX + 1;                    // x hand-off pitch in float2
  static constexpr int kListCap = 2 * NT;               // segments
  template <int NARR> static constexpr size_t smem_bytes() {
    return 128 + sizeof(float) * (size_t)(2 * NARR * ARR) + sizeof(float2) * (size_t)TY * (SUP + TX) +
           sizeof(unsigned short) * kListCap;
  }
};
static_assert(Geo2D<kTile2DX>::SW == kBox2DW && Geo2D<kTile2DX>::SH == kBox2DH, "TMA box must match the tile halo");
static_assert(Geo2D<kTile2DXNarrow>::SW == kBox2DWNarrow, "TMA box must match the tile halo");

// Everything a tile needs from its instance, gathered by thread 0 into shared memory when the
// tile is prepared (one tile ahead), so that the compute phase reads no instance data from
// global memory.
struct TileInfo {
  int inst, tx0, ty0, cur, skip, last;
  float dtf, fax, fay;
  double dt;
  int nx, ny, row_off, bc, ham, ntiles, tiles_x;
  float dx, dy, rdx, rdy, xlo, ylo;
  DevState *st;
};

struct SoloLocal {
  double t, tf, dt, a[2], ends[2][2];   // a: grid maxima of the last stage; ends: of stages 2, 3 of the last whole step
  int cur, last, err, steps;
};

template <int PREC, int W, int H, int TXv>
__global__ void __launch_bounds__(Geo2D<TXv>::NT, Geo2D<TXv>::MINB)
    stage2d_kernel(const __grid_constant__ Stage2DParams prm) {
  using G = Geo2D<TXv>;
  constexpr int TX = G::TX, TY = G::TY, K = G::K, NT = G::NT;
  constexpr int SW = G::SW, SH = G::SH, ARR = G::ARR;
  constexpr int SUP = G::SUP, CG = G::CG;
  constexpr int NARR = (PREC == P_MIXED) ? 3 : 2;
  const StageParams &p = prm.p;
  const bool batch = prm.insts != nullptr;
  // one stage, or (solo: a single grid, cooperative launch) prm.nsteps RK3 steps, stage run % 3 + 1 in run `run`.
  // The CTAs keep a copy of the grid's state each, advanced by the same arithmetic, and meet once per stage: the
  // maxima and the arrival count are the only global atomics between two stages.
  const bool solo = prm.nsteps > 0;
  const int runs = solo ? 3 * prm.nsteps : 1;
  int stage = p.stage, map_c = prm.map_c;
  if (!batch && !solo) {
    const DevState *st = prm.inst0.st;
    if (p.loop_mode == LOOP_STEP_TO && !(st->t < st->t_final)) return;
    if (st->err) return;
  }

  extern __shared__ __align__(128) unsigned char smem_dyn[];
  // TMA destinations are kept 128-byte aligned (the launch adds 128 bytes of slack)
  unsigned char *smem = smem_dyn + ((128u - (smem_u32(smem_dyn) & 127u)) & 127u);
  float *raw = reinterpret_cast<float *>(smem);            // [2][NARR][ARR]
  float2 *su = reinterpret_cast<float2 *>(raw + 2 * NARR * ARR);  // [TY][SUP] sums, differences along x
  float2 *sv = su + TY * SUP;                                     // [TY][TX] along y
  unsigned short *s_list = reinterpret_cast<unsigned short *>(sv + TY * TX);  // segments left to the full sweep
  __shared__ int s_nlist, s_stop, s_lost;
  __shared__ SoloLocal so;   // solo: the instance's state, advanced alike by thread 0 of every CTA
  __shared__ __align__(8) uint64_t bars[2];
  __shared__ TileInfo s_info[2];
  __shared__ TileInfo s_pinfo;  // thread 0's last prepared tile (per-instance scalars reused while it repeats)
  __shared__ float s_red[2][NT / 32];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ntiles = prm.ntiles;
  const bool local_alpha = (p.alpha_mode == A_LOCAL_LAGGED || p.alpha_mode == A_LOCAL_EXACT);
  const float eps = (float)p.eps;
  const uint32_t box_bytes = (uint32_t)(SH * SW * sizeof(float));

  auto desc = [&](int inst) -> const InstDesc & { return batch ? prm.insts[inst] : prm.inst0; };

  // thread 0: one TMA box per array of the tile (with halo) into buffer b
  auto issue_loads = [&](const TileInfo &info, int b) {
    const CUtensorMap *mA, *mB = nullptr, *mC = nullptr;
    if (PREC == P_MIXED) {
      mA = &prm.maps[prm.map_a + info.cur];
      mB = &prm.maps[prm.map_b + info.cur];
      if (map_c >= 0) mC = &prm.maps[map_c];
    } else {
      // the stage's input (of stage 0: that of the stage p.src_of) and phi^n
      mA = &prm.maps[stage == 0 ? prm.map_a : stage - 1];
      if (stage >= 2) mB = &prm.maps[0];
    }
    const int nm = 1 + (mB != nullptr) + (mC != nullptr);
    float *dst = raw + b * NARR * ARR;
    const int y = info.row_off + info.ty0;
    mbar_arrive_expect_tx(&bars[b], box_bytes * nm);
    tma_load_2d(dst, mA, info.tx0, y, &bars[b]);
    if (mB) tma_load_2d(dst + ARR, mB, info.tx0, y, &bars[b]);
    if (mC) tma_load_2d(dst + 2 * ARR, mC, info.tx0, y, &bars[b]);
  };

  // thread 0: decode work-list entry e (of list position t), gather its instance's fields and
  // stage scalars (reused while the instance repeats), issue its loads into buffer b
  auto prepare = [&](int t, int e, int b) {
    int inst = 0, tl = t;
    if (batch) {
      inst = e >> 16;
      tl = e & 0xffff;
    }
    if (inst == s_info[b].inst) {
      // the tile that last used this buffer belongs to the same instance (always so for a single
      // grid): only the tile origin changes
      TileInfo &bi = s_info[b];
      bi.tx0 = (tl % bi.tiles_x) * TX;
      bi.ty0 = (tl / bi.tiles_x) * TY;
      if (!bi.skip) issue_loads(bi, b);
      return;
    }
    TileInfo info;
    if (inst == s_pinfo.inst) {
      info = s_pinfo;
      info.tx0 = (tl % info.tiles_x) * TX;
      info.ty0 = (tl / info.tiles_x) * TY;
      s_info[b] = info;
      s_pinfo = info;
      if (!info.skip) issue_loads(info, b);
      return;
    }
    // the instance's descriptor and its state (contiguous states: no dependent load)
    const InstDesc &d = desc(inst);
    DevState *st = (batch && prm.states) ? prm.states + inst : d.st;
    info.inst = inst;
    info.nx = d.nx;
    info.ny = d.ny;
    info.row_off = d.row_off;
    info.bc = d.bc;
    info.ham = d.ham;
    info.ntiles = d.ntiles;
    info.tiles_x = d.tiles_x;
    info.dx = d.dx;
    info.dy = d.dy;
    info.rdx = d.rdx;
    info.rdy = d.rdy;
    info.xlo = d.xlo;
    info.ylo = d.ylo;
    info.st = st;
    const double lx = d.lx, ly = d.ly;
    const int s_cur = st->cur, s_err = st->err;
    const double s_t = st->t, s_tf = st->t_final, s_dt = st->dt;
    info.tx0 = (tl % info.tiles_x) * TX;
    info.ty0 = (tl / info.tiles_x) * TY;
    info.cur = (PREC == P_MIXED) ? s_cur : 0;
    info.skip = (s_err != 0) || (p.loop_mode == LOOP_STEP_TO && !(s_t < s_tf));
    double dt;
    int last = 0;
    if (stage == 1 && p.loop_mode != LOOP_STAGE) {
      double ax, ay;
      if (p.alpha_mode == A_FIXED) {
        ax = p.alpha_fixed[0];
        ay = p.alpha_fixed[1];
      } else {
        ax = bits_to_double(st->alpha_bits[p.dt_slot][0]);
        ay = bits_to_double(st->alpha_bits[p.dt_slot][1]);
      }
      const double den = ax / lx + ay / ly;
      dt = den > 0.0 ? p.cfl / den : (p.loop_mode == LOOP_ADVANCE ? 0.0 : INFINITY);
      if (p.loop_mode == LOOP_STEP_TO && s_t + dt >= s_tf) {
        dt = s_tf - s_t;
        last = 1;
      }
    } else if (p.loop_mode == LOOP_STAGE) {
      dt = p.dt_value;
    } else {
      dt = s_dt;
    }
    info.dt = dt;
    info.dtf = (float)dt;
    info.last = last;
    float fax = 0.0f, fay = 0.0f;
    if (p.alpha_mode == A_FIXED) {
      fax = (float)p.alpha_fixed[0];
      fay = (float)p.alpha_fixed[1];
    } else if (!local_alpha && p.read_slot >= 0) {
      fax = (float)bits_to_double(st->alpha_bits[p.read_slot][0]);
      fay = (float)bits_to_double(st->alpha_bits[p.read_slot][1]);
    }
    info.fax = fax;
    info.fay = fay;
    s_info[b] = info;
    s_pinfo = info;
    if (!info.skip) issue_loads(info, b);
  };

  if (tid == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&bars[1], 1);
    fence_mbar_init();
    s_nlist = 0;
  }
  __syncthreads();

  uint32_t phase = 0;  // bit b: parity of the next completion of bars[b]
  int k = 0;
  // running alpha maxima and tile count of the current run of same-instance tiles
  constexpr bool GF = HamSel<H>::kGridFold;
  constexpr float A0 = GF ? -INFINITY : 0.0f;  // identity of the running maxima
  float amx = A0, amy = A0;
  float nfin = 0.0f;  // NaN once a non-finite L was met (see the finish loop)
  int run_tiles = 0;
  int e_ahead = 0;  // thread 0: work-list entry of the tile after next, loaded one tile ahead of its use
  // thread 0, once every thread is past the previous tile's reads of buffer buf ^ 1 and of
  // s_info[buf ^ 1]: prepare the next tile into that buffer
  auto prepare_next = [&](int next, int buf) {
    if (tid == 0 && next < ntiles) {
      fence_proxy_async_smem();
      prepare(next, e_ahead, buf ^ 1);
      const int after = next + (int)gridDim.x;
      e_ahead = (batch && after < ntiles) ? prm.tiles[after] : 0;
    }
  };
  if (solo && tid == 0) {
    const DevState *st = prm.inst0.st;
    so.t = st->t;
    so.tf = st->t_final;
    so.dt = st->dt;
    so.last = st->last;
    so.cur = st->cur;
    so.err = st->err;
    so.steps = 0;
    for (int i = 0; i < 2; ++i) so.a[i] = bits_to_double(st->alpha_bits[2][i]);
  }
  // the stage's first tile: its loads are issued before the scalars are worked out
  auto prepare_solo = [&](int t, int b) {
    const InstDesc &d = prm.inst0;
    TileInfo info;
    info.inst = 0;
    info.tiles_x = d.tiles_x;
    info.tx0 = (t % d.tiles_x) * TX;
    info.ty0 = (t / d.tiles_x) * TY;
    info.row_off = d.row_off;
    info.cur = (PREC == P_MIXED) ? so.cur : 0;
    info.skip = 0;
    issue_loads(info, b);
    info.nx = d.nx;
    info.ny = d.ny;
    info.bc = d.bc;
    info.ham = d.ham;
    info.ntiles = d.ntiles;
    info.dx = d.dx;
    info.dy = d.dy;
    info.rdx = d.rdx;
    info.rdy = d.rdy;
    info.xlo = d.xlo;
    info.ylo = d.ylo;
    info.st = d.st;
    const bool fixed = p.alpha_mode == A_FIXED;
    if (stage == 1) {
      const double den = (fixed ? p.alpha_fixed[0] : so.a[0]) / d.lx + (fixed ? p.alpha_fixed[1] : so.a[1]) / d.ly;
      so.dt = den > 0.0 ? p.cfl / den : (p.loop_mode == LOOP_ADVANCE ? 0.0 : INFINITY);
      so.last = p.loop_mode == LOOP_STEP_TO && so.t + so.dt >= so.tf;
      if (so.last) so.dt = so.tf - so.t;
    }
    info.dt = so.dt;
    info.dtf = (float)so.dt;
    info.last = so.last;
    info.fax = fixed ? (float)p.alpha_fixed[0] : (local_alpha ? 0.0f : (float)so.a[0]);
    info.fay = fixed ? (float)p.alpha_fixed[1] : (local_alpha ? 0.0f : (float)so.a[1]);
    s_info[b] = info;
    s_pinfo = info;
  };
  for (int run = 0; run < runs; ++run) {
    if (solo) {
      stage = run % 3 + 1;
      map_c = stage == 1 ? -1 : stage + 2;
    }
    if (tid == 0) {
      s_pinfo.inst = s_info[0].inst = s_info[1].inst = -1;
      s_stop = solo && (so.err || (stage == 1 && p.loop_mode == LOOP_STEP_TO && !(so.t < so.tf)));
      if (!s_stop && (int)blockIdx.x < ntiles) {
        fence_proxy_async_smem();
        if (solo) prepare_solo(blockIdx.x, k & 1);
        else prepare(blockIdx.x, batch ? prm.tiles[blockIdx.x] : 0, k & 1);
        e_ahead = (batch && (int)(blockIdx.x + gridDim.x) < ntiles) ? prm.tiles[blockIdx.x + gridDim.x] : 0;
        // the next stage's maxima: last read in the stage before this one
        if (solo && blockIdx.x == 0) prm.solo->alpha[stage % 3][0] = prm.solo->alpha[stage % 3][1] = 0ull;
      }
    }
    __syncthreads();
    if (s_stop) break;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++k) {
      const int buf = k & 1;
      const int next = t + gridDim.x;
      const int i_inst = s_info[buf].inst, i_skip = s_info[buf].skip, i_cur = s_info[buf].cur;
      if (i_skip) {
        __syncthreads();
        prepare_next(next, buf);
        __syncthreads();
        continue;
      }
      const bool ok = mbar_wait_bounded(&bars[buf], (phase >> buf) & 1u);
      phase ^= 1u << buf;

      const TileInfo &d = s_info[buf];  // this tile's instance fields (shared memory)
      const int nx = d.nx, ny = d.ny, tx0 = d.tx0, ty0 = d.ty0;
      const size_t rbase = (size_t)d.row_off * p.pitch;   // element offset of the instance's rows
      const float dtf = s_info[buf].dtf, fax = s_info[buf].fax, fay = s_info[buf].fay;
      const float *A = raw + buf * NARR * ARR;
      const float *B = A + ARR;
      const float *C = A + 2 * ARR;
      // MIXED: the stage's input is A + X, the high part of phi^n plus X = its low part (stage 1) or the
      // increment array of the previous stage, which holds the low part as well (stages 2 and 3; see the
      // finish loop)
      const float *X = (PREC == P_MIXED && map_c >= 0) ? C : B;

      if (__syncthreads_or(!ok)) {
        // a tile load never completed: flag the instance and stop; the next tile's load is issued only
        // after this barrier, so no other load is in flight
        if (tid == 0) atomicOr(&s_info[buf].st->err, 2);
        __syncthreads();
        return;
      }
      // every thread has finished the previous tile (its finish loop read buffer buf ^ 1), so the next
      // tile's load can go there; the barrier after the sweeps publishes s_info[buf ^ 1]
      prepare_next(next, buf);

      const bool edge = (tx0 < 3) || (tx0 + TX > nx - 3) || (ty0 < 3) || (ty0 + TY > ny - 3);
      const int colY = (warp % CG) * 32 + lane, segY = warp / CG;

      // ---- 1. both sweeps in one pass: each thread's row segment (x, lane .x of the packed values)
      // and column segment (y, lane .y) run the same instruction stream; the sums and differences of the
      // one-sided derivatives go to shared memory
      {
        // first cell (node - 3) of the column segment, and the quad that ends with that of the row segment
        const int iy = (K * segY) * SW + colY + 4, ix = (lane + 3) * SW + K * warp;
        const float2 rd = make_float2(d.rdx, d.rdy);
        // v_at(m), called for m = 0, 1, 2, ... in order: (v, v) = first differences over dx, dy at position m;
        // the row's cells come as 16-byte quads (conflict-free, see Geo2D), the column's one by one
        // (consecutive lanes read consecutive columns)
        auto make_vat = [&]() {
          auto quad = [](const float *q, int i) { return *reinterpret_cast<const float4 *>(q + i); };
          float4 qa = quad(A, ix), qx = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          float2 pa = make_float2(qa.y, A[iy]), px = make_float2(0.0f, 0.0f);
          if (PREC == P_MIXED) {
            qx = quad(X, ix);
            px = make_float2(qx.y, X[iy]);
          }
          return [=](int m) mutable {
            const int k = (m + 2) & 3, i1 = iy + (m + 1) * SW;   // element of the row's quad
            if (k == 0) {
              qa = quad(A, ix + m + 2);
              if (PREC == P_MIXED) qx = quad(X, ix + m + 2);
            }
            auto pick = [&](const float4 &q) { return k == 0 ? q.x : k == 1 ? q.y : k == 2 ? q.z : q.w; };
            const float2 a1 = make_float2(pick(qa), A[i1]);
            float2 v = vsub(a1, pa);
            pa = a1;
            if (PREC == P_MIXED) {
              const float2 x1 = make_float2(pick(qx), X[i1]);
              v = vadd(v, vsub(x1, px));
              px = x1;
            }
            return vmul(v, rd);
          };
        };
        float2 *ox = su + lane * SUP + K * warp, *oy = sv + (K * segY) * TX + colY;
        auto emit = [&](int q, float2 S, float2 D) {
          ox[q] = make_float2(S.x, D.x);
          oy[q * TX] = make_float2(S.y, D.y);
        };
        // the sweeps that give the one-sided derivatives themselves
        auto emit_pm = [&](int q, float2 dm, float2 dp) { emit(q, vadd(dp, dm), vsub(dp, dm)); };
        // arc length: the near-linear form first; segments that do not qualify take the full form, swept again by
        // the warp where at least kWarpSegs fail (coarse grids, the rounding noise of FP32), else entered in a
        // list whose nodes all threads of the CTA share (a kink crosses few segments of a tile, and the CTA
        // would wait for their warps).  Both evaluate the same operations, so a node's derivatives depend only
        // on the data of its 8-node segment and its ghosts, whose position on the grid is the same for both tile
        // widths -- not on the order in which tiles or instances are processed, nor on history: a single solve, a
        // batch, a server round and a resumed checkpoint agree.
        if constexpr (W == W_ARCLEN) {
          // FP32 stores phi itself: its rounding over dx is what the derivatives carry anyway
          float2 size = make_float2(0.0f, 0.0f);
          if (PREC == P_F32) {
            size = make_float2(fmaxf(fabsf(A[ix + 4]), fabsf(A[ix + K + 3])) * d.rdx,
                               fmaxf(fabsf(A[iy + 3 * SW]), fabsf(A[iy + (K + 2) * SW])) * d.rdy);
          }
          // segments of rows or columns beyond the grid (ragged tiles) do not count; segments that cross the grid's
          // end are swept in full: beyond the three ghosts lies padding, which in the server's arena holds values
          // of earlier requests, and the near test takes all of a segment's cells
          // (only border tiles have any; in MIXED the test costs more than what it saves -- 8192^2, us per RK3 step of
          // Example 3 without / with it: FP32 1682 / 1652, MIXED 1013 / 1027)
          int out = 0, whole = 3;
          if (PREC == P_MIXED || edge) {
            const int endx = nx - tx0 - K * warp, endy = ny - ty0 - K * segY;   // nodes of the segment's line left
            const bool outx = ty0 + lane >= ny || endx <= 0, outy = tx0 + colY >= nx || endy <= 0;
            if (outx) size.x = INFINITY;
            if (outy) size.y = INFINITY;
            whole = (endx < K ? 0 : 1) | (endy < K ? 0 : 2);
            out = (outx ? 1 : 0) | (outy ? 2 : 0);
          }
          const int near = out | (whole & sweep_stream_near<K, float2>(make_vat(), rd,
              make_float2(fmaf(d.dx, d.dx, eps), fmaf(d.dy, d.dy, eps)), size, emit));
          if (__any_sync(0xffffffffu, near != 3)) {
            const bool fx = !(near & 1), fy = !(near & 2);
            if (__popc(__ballot_sync(0xffffffffu, fx)) + __popc(__ballot_sync(0xffffffffu, fy)) >= kWarpSegs) {
              SweepConsts<float2> sc;
              sc.eps4 = make_float2(4.0f * eps * d.rdx * d.rdx, 4.0f * eps * d.rdy * d.rdy);
              sc.h2 = make_float2(0.5f * d.dx, 0.5f * d.dy);
              sc.h3 = make_float2(d.dx * (1.0f / 3.0f), d.dy * (1.0f / 3.0f));
              sc.mh6 = make_float2(d.dx * (-1.0f / 6.0f), d.dy * (-1.0f / 6.0f));
              // -0, unknown to the assembler: it fuses a packed multiply (or one with a constant zero added) with
              // a packed add that is its only reader, as at the first and the last position, and the scalar
              // sweep of the list, where it does not, would differ in the last bit
              const float2 nz = vsplat(-(float)(p.stage >> 8), rd);
              auto v_at = make_vat();
              sweep_stream<K, float2>([&](int m) { return vfma(v_at(m), rd, nz); }, sc,
                                      [&](int q, float2 dm, float2 dp) {
                                        const float2 S = vadd(dp, dm), D = vsub(dp, dm);
                                        if (fx) ox[q] = make_float2(S.x, D.x);
                                        if (fy) oy[q * TX] = make_float2(S.y, D.y);
                                      });
            } else {
              // entry: line (row or column), segment along it, direction
              if (fx) s_list[atomicAdd(&s_nlist, 1)] = (unsigned short)((lane * 8 + warp) * 2);
              if (fy) s_list[atomicAdd(&s_nlist, 1)] = (unsigned short)((colY * 8 + segY) * 2 + 1);
            }
          }
        } else {
          sweep_stream_jp<K, float2>(make_vat(), make_float2(eps, eps), emit_pm);
        }
      }
      __syncthreads();
      if (W == W_ARCLEN && s_nlist > 0) {
        for (int i = tid; i < s_nlist * K; i += NT) {
          const int e = s_list[i / K], q = i % K, along_y = e & 1, line = e >> 4, at = ((e >> 1) & 7) * K + q;
          const int step = along_y ? SW : 1, i0 = along_y ? at * SW + line + 4 : (line + 3) * SW + at + 1;
          const float rdl = along_y ? d.rdy : d.rdx, dl = along_y ? d.dy : d.dx;
          SweepConsts<float> sc;
          sc.eps4 = 4.0f * eps * rdl * rdl;
          sc.h2 = 0.5f * dl;
          sc.h3 = dl * (1.0f / 3.0f);
          sc.mh6 = dl * (-1.0f / 6.0f);
          sweep_stream<1, float>(
              [&](int m) {
                const int j = i0 + m * step;
                float v = vsub(A[j + step], A[j]);
                if (PREC == P_MIXED) v = vadd(v, vsub(X[j + step], X[j]));
                return vmul(vmul(v, rdl), rdl);
              },
              sc, [&](int, float dm, float dp) {
                (along_y ? sv[at * TX + line] : su[line * SUP + at]) = make_float2(vadd(dp, dm), vsub(dp, dm));
              });
        }
        __syncthreads();
        if (tid == 0) s_nlist = 0;   // the next entries are made after the next tile's first barrier
      }

      // ---- 2. nodes (colY, K*segY + q): Lax-Friedrichs Hamiltonian, RK combination, store; one
      // unrolled loop per stage and per edge/interior tile, so that no node tests either
      float *out = reinterpret_cast<float *>(solo ? prm.outs[stage - 1] : p.out0);
      auto finish = [&](auto stage_c, auto edge_c, auto hsel) {
        using HS = decltype(hsel);
        constexpr int ST = decltype(stage_c)::value;
        constexpr bool EDGE = decltype(edge_c)::value;
        constexpr float U = HS::kUnit;
        const float dtu = (1.0f / U) * dtf, faxh = (0.5f * U) * fax, fayh = (0.5f * U) * fay;
#pragma unroll
        for (int q = 0; q < K; ++q) {
          const int y = K * segY + q;
          const float2 w = sv[y * TX + colY];    // (Sy, Dy)
          const float sy = w.x, dy = w.y;
          const int gi = tx0 + colY, gj = ty0 + y;
          const bool inside = !EDGE || (gi < nx && gj < ny);
          const float2 u = su[y * SUP + colY];   // (Sx, Dx)
          float L;   // U (-H + alpha_x/2 Dx + alpha_y/2 Dy)
          if constexpr (HS::kGridFold) {
            const float s = u.x + sy, e = fabsf(u.y) + fabsf(dy);
            L = fmaf(faxh, u.y, fmaf(fayh, dy, -hsel.value(u.x, sy, 0.0f, 0.0f)));
            if (inside) {
              nfin = fmaf(L, 0.0f, nfin);
              amx = fmaxf(amx, s + e);
              amy = fmaxf(amy, e - s);
            }
          } else {
            const float xn = fmaf((float)gi, d.dx, d.xlo), yn = fmaf((float)gj, d.dy, d.ylo);
            float ax, ay;
            hsel.alpha(u.x, u.y, sy, dy, xn, yn, ax, ay);
            const float aX = local_alpha ? ax * (0.5f * U) : faxh, aY = local_alpha ? ay * (0.5f * U) : fayh;
            L = fmaf(aX, u.y, fmaf(aY, dy, -hsel.value(u.x, sy, xn, yn)));
            if (inside) {
              // L depends on all four one-sided derivatives: L * 0 is NaN exactly when L is not finite
              nfin = fmaf(L, 0.0f, nfin);
              amx = fmaxf(amx, ax);
              // (with a runtime Hamiltonian the fold below does not copy amx, so amy is always kept)
              if (!HS::kSameAlpha || !HamSel<H>::kSameAlpha) amy = fmaxf(amy, ay);
            }
          }
          if (ST == 0 || !inside) continue;
          const int sidx = (y + 3) * SW + colY + 4;
          const size_t g = rbase + (size_t)(gj + GY) * p.pitch + gi + GX;
          if (PREC == P_MIXED) {
            // phi^n = hi + lo (A, B) and the stage states phi_1 = hi + e_1, phi_2 = hi + e_2, where the
            // increment arrays e_k = lo + (phi_k - phi^n) carry the low part (C = e_{k-1}):
            //   e_1 = lo + dt L,  e_2 = 3/4 lo + 1/4 (e_1 + dt L),  phi^{n+1} = hi + lo + 2/3 (e_2 + dt L - lo)
            // (Step 5's combinations with phi_k - phi^n = e_k - lo)
            if (ST == 3) {
              const float dd = (2.0f / 3.0f) * (fmaf(dtu, L, C[sidx]) - B[sidx]);
              float h, l;
              df_add(A[sidx], B[sidx], dd, h, l);
              float *oh = reinterpret_cast<float *>(p.mix_hi[i_cur ^ 1]);
              float *ol = reinterpret_cast<float *>(p.mix_lo[i_cur ^ 1]);
              if (EDGE) {
                store_node<float, 2>(oh + rbase, p.pitch, nx, ny, d.bc, gi, gj, h);
                store_node<float, 2>(ol + rbase, p.pitch, nx, ny, d.bc, gi, gj, l);
              } else {
                oh[g] = h;
                ol[g] = l;
              }
            } else {
              const float dd = (ST == 1) ? fmaf(dtu, L, B[sidx]) : fmaf(0.75f, B[sidx], 0.25f * fmaf(dtu, L, C[sidx]));
              float *o = out;
              if (EDGE) store_node<float, 2>(o + rbase, p.pitch, nx, ny, d.bc, gi, gj, dd);
              else o[g] = dd;
            }
          } else {
            const float src = A[sidx];
            float outv;
            if (ST == 1) {
              outv = fmaf(dtu, L, src);
            } else if (ST == 2) {
              outv = fmaf(0.75f, B[sidx], 0.25f * fmaf(dtu, L, src));
            } else {
              outv = fmaf(1.0f / 3.0f, B[sidx], (2.0f / 3.0f) * fmaf(dtu, L, src));
            }
            float *o = out;
            if (EDGE) store_node<float, 2>(o + rbase, p.pitch, nx, ny, d.bc, gi, gj, outv);
            else o[g] = outv;
          }
        }
      };
      // the Hamiltonian of the tile: the launch's, or with H_RUNTIME the instance's, chosen once per tile
      auto finish_h = [&](auto stage_c, auto edge_c) {
        if constexpr (H == H_RUNTIME) {
          switch (d.ham) {
            case H_BURGERS2D: finish(stage_c, edge_c, HamSel<H_BURGERS2D>{}); break;
            case H_NEGCOS2D: finish(stage_c, edge_c, HamSel<H_NEGCOS2D>{}); break;
            case H_SIN2D: finish(stage_c, edge_c, HamSel<H_SIN2D>{}); break;
            default: finish(stage_c, edge_c, HamSel<H_EIKONAL2D>{}); break;
          }
        } else {
          finish(stage_c, edge_c, HamSel<H>{});
        }
      };
      auto finish_stage = [&](auto stage_c) {
        if (edge) finish_h(stage_c, std::true_type{});
        else finish_h(stage_c, std::false_type{});
      };
      switch (stage) {
        case 0: finish_stage(std::integral_constant<int, 0>{}); break;
        case 1: finish_stage(std::integral_constant<int, 1>{}); break;
        case 2: finish_stage(std::integral_constant<int, 2>{}); break;
        default: finish_stage(std::integral_constant<int, 3>{}); break;
      }

      // ---- extrapolated boundary: the ghosts of the lines that end in this tile, from the two values just stored
      // at their ends (as separate launches after the stage, they took a third of a step at 1024^2: 57.9 us against
      // 37.1)
      if constexpr (TX == kTile2DX && H != H_RUNTIME) {
        if (prm.ghosts && edge) {
          __syncthreads();
          const int x0 = d.tx0, y0 = d.ty0, w = min(TX, d.nx - x0), h = min(TY, d.ny - y0);
          auto hi = reinterpret_cast<float *>(p.mix_hi[d.cur ^ 1]), lo = reinterpret_cast<float *>(p.mix_lo[d.cur ^ 1]);
          for (int c = warp; c < 12; c += NT / 32) {
            const int side = c / 3, m = c % 3 + 1;   // left, right, lower, upper; nodes beyond the end
            const bool ends = side == 0 ? x0 == 0 : side == 1 ? x0 + w == d.nx : side == 2 ? y0 == 0 : y0 + h == d.ny;
            if (!ends) continue;
            const int n = side < 2 ? h : w, dir = (side & 1) ? -1 : 1;   // inwards
            const int sstep = dir * (side < 2 ? 1 : SW);
            const long long gstep = dir * (side < 2 ? 1ll : (long long)p.pitch);
            for (int i = lane; i < n; i += 32) {
              const int x = side < 2 ? (side == 0 ? 0 : w - 1) : i, y = side < 2 ? i : (side == 2 ? 0 : h - 1);
              const int s = (y + 3) * SW + x + 4;
              const long long g = (long long)(d.row_off + y0 + y + GY) * p.pitch + x0 + x + GX;
              if (PREC != P_MIXED) {
                out[g - m * gstep] = extrapolate<float>(m, out[g], out[g + gstep]);
              } else if (stage == 3) {
                const double v = extrapolate<double>(m, (double)hi[g] + (double)lo[g],
                                                     (double)hi[g + gstep] + (double)lo[g + gstep]);
                const float vh = (float)v;
                hi[g - m * gstep] = vh;
                lo[g - m * gstep] = (float)(v - (double)vh);
              } else {
                // so that hi + increment is the extrapolated stage state (see ghosts_incr)
                const double v = extrapolate<double>(m, (double)A[s] + (double)out[g],
                                                     (double)A[s + sstep] + (double)out[g + gstep]);
                out[g - m * gstep] = (float)(v - (double)A[s - m * sstep]);
              }
            }
          }
        }
      }

      // ---- when the next tile of this CTA belongs to another instance (or there is none), fold the
      // run's maximum of alpha into the instance's slot and count its tiles; close the instance's stage
      ++run_tiles;
      const bool more = next < ntiles;
      if (more && !s_info[buf ^ 1].skip && s_info[buf ^ 1].inst == i_inst) {
        // no barrier: su, raw[buf] and s_info[buf] are rewritten only after the next tile's first
        // barrier, which every thread reaches after finishing this tile
        continue;
      }
      if constexpr (GF) {
        amx = fmaxf(fmaxf(fmaf(0.5f, amx, 1.0f), fmaf(0.5f, amy, -1.0f)), 0.0f);
        amy = amx;
      } else if (HamSel<H>::kSameAlpha) {
        amy = amx;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        amx = fmaxf(amx, __shfl_xor_sync(0xffffffffu, amx, o));
        amy = fmaxf(amy, __shfl_xor_sync(0xffffffffu, amy, o));
      }
      const int anybad = __syncthreads_or(nfin != nfin ? 1 : 0);
      if (lane == 0) {
        s_red[0][warp] = amx;
        s_red[1][warp] = amy;
      }
      __syncthreads();
      if (tid == 0) {
        for (int w = 1; w < NT / 32; ++w) {
          amx = fmaxf(amx, s_red[0][w]);
          amy = fmaxf(amy, s_red[1][w]);
        }
        DevState *st = d.st;
        if (solo) {
          // a NaN stands for a non-finite dH/dp anywhere (the largest bit pattern)
          atomicMax(&prm.solo->alpha[stage - 1][0], double_to_bits(anybad ? (double)NAN : (double)amx));
          atomicMax(&prm.solo->alpha[stage - 1][1], double_to_bits((double)amy));
        } else {
          if (anybad) atomicOr(&st->err, 1);
          if (p.write_slot >= 0) {
            atomicMax(&st->alpha_bits[p.write_slot][0], double_to_bits((double)amx));
            atomicMax(&st->alpha_bits[p.write_slot][1], double_to_bits((double)amy));
          }
          __threadfence();
          const unsigned int prev = atomicAdd(&st->counter, (unsigned int)run_tiles);
          if (prev + (unsigned int)run_tiles == (unsigned int)d.ntiles) {
            // every tile of this instance has finished this stage
            __threadfence();
            st->counter = 0;
            if (p.zero_slot >= 0) {
              st->alpha_bits[p.zero_slot][0] = 0ull;
              st->alpha_bits[p.zero_slot][1] = 0ull;
            }
            if (p.stage == 1 && p.loop_mode != LOOP_STAGE) {
              st->dt = s_info[buf].dt;
              st->last = s_info[buf].last;
            }
            if (p.stage == 3) {
              if (PREC == P_MIXED) st->cur = i_cur ^ 1;
              if (p.loop_mode != LOOP_STAGE) {
                const double tn = st->last ? st->t_final : st->t + st->dt;
                st->t = tn;
                st->steps += 1;
                if (p.loop_mode == LOOP_STEP_TO && !(tn < st->t_final) && prm.done_count) atomicAdd(prm.done_count, 1);
              }
            }
          }
        }
      }
      amx = amy = A0;
      nfin = 0.0f;
      run_tiles = 0;
      __syncthreads();  // raw[buf], su, s_info[buf] are free for the next tile
    }
    if (!solo) break;
    // ---- grid barrier: the stage's outputs (ordinary stores) before the next one's tile loads (async proxy)
    fence_proxy_async_global();
    __syncthreads();
    if (tid == 0) {
      volatile SoloState *sh = prm.solo;
      __threadfence();
      const unsigned long long target = (unsigned long long)(run + 1) * gridDim.x;
      unsigned long long seen = atomicAdd(&prm.solo->arrived, 1ull) + 1;
      for (int spin = 0; seen < target && spin < kBarrierSpins; ++spin) seen = sh->arrived;
      __threadfence();
      fence_proxy_async_global();
      s_lost = seen < target;
      // the maxima of the stage just closed; the step's end
      const double a0 = bits_to_double(sh->alpha[stage - 1][0]), a1 = bits_to_double(sh->alpha[stage - 1][1]);
      const bool bad = a0 != a0;
      if (stage == 3) {
        for (int i = 0; i < 2; ++i) so.ends[0][i] = so.a[i];
        so.ends[1][0] = bad ? 0.0 : a0;
        so.ends[1][1] = a1;
        so.t = so.last ? so.tf : so.t + so.dt;
        so.cur ^= 1;
        ++so.steps;
      }
      so.a[0] = a0;
      so.a[1] = a1;
      if (bad) so.err = 1;
    }
    __syncthreads();
    if (s_lost) {   // a CTA never arrived
      if (tid == 0) atomicOr(&prm.inst0.st->err, 2);
      return;
    }
  }
  if (solo && blockIdx.x == 0 && tid == 0) {
    // the state as launches of single stages would leave it
    DevState *st = prm.inst0.st;
    if (so.err) st->err |= so.err;
    st->dt = so.dt;
    st->last = so.last;
    if (so.steps > 0) {
      st->t = so.t;
      st->steps += so.steps;
      if (PREC == P_MIXED) st->cur = so.cur;
      st->alpha_bits[0][0] = st->alpha_bits[0][1] = 0ull;
      for (int i = 0; i < 2; ++i) {
        st->alpha_bits[1][i] = double_to_bits(so.ends[0][i]);
        st->alpha_bits[2][i] = double_to_bits(so.ends[1][i]);
      }
    }
  }
}

}  // namespace alw
