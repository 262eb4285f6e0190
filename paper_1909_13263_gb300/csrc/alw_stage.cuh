// The fused RK-stage kernel (see alw_device.cuh for the arithmetic).
#pragma once
#include <type_traits>

#include "alw_device.cuh"
#include "alw_sweep64.cuh"

namespace alw {

// Constants of the FP64 sweeps, formed on the host (nothing for the float variants).
template <int PREC> struct SweepArgs {};
template <> struct SweepArgs<P_F64> {
  Sweep64 x, y;
};
template <int PREC, int W>
static SweepArgs<PREC> sweep_args(const StageParams &p) {
  SweepArgs<PREC> a;
  if constexpr (PREC == P_F64) {
    a.x = make_sweep64<W>(p.dx, p.eps);
    a.y = p.dim == 2 ? make_sweep64<W>(p.dy, p.eps) : a.x;
  }
  return a;
}

// Largest of two non-negative doubles by their bit patterns (integer comparisons: FP64 ones run on the FP64
// pipe); a NaN counts as larger than everything, so it survives to the caller's check.
__device__ __forceinline__ double max_bits(double a, double b) {
  const unsigned long long x = double_to_bits(a), y = double_to_bits(b);
  return bits_to_double(x > y ? x : y);
}
__device__ __forceinline__ double min_bits(double a, double b) {
  const unsigned long long x = double_to_bits(a), y = double_to_bits(b);
  return bits_to_double(x < y ? x : y);
}

// H at the mean one-sided derivatives and the node alpha in double, sharing what they have in common.
// With c = (u^- + u^+ + v^- + v^+)/2 and e = (|u^+ - u^-| + |v^+ - v^-|)/2 the four corner sums u + v are
// c +- e and c +- |du - dv|/2.  `known` is a lower bound of the grid maximum the alphas are folded into:
// an alpha that cannot exceed it is returned as 0 (0 = evaluate always, for a flux that uses the node's own).
// The trigonometric kinds need sin and cos of c only: |cos(c +- d)| is at most |cos c| cos d + |sin c| sin d,
// attained by one of the two signs, with cos d and sin d by their series for small d.
__device__ __forceinline__ void ham_node64(int kind, double um, double up, double vm, double vp, double x, double y,
                                           double known, double &H, double &ax, double &ay) {
  const double su = up + um, du = up - um;
  switch (kind) {
    case H_BURGERS2D:
    case H_BURGERS1D: {
      const bool two = kind == H_BURGERS2D;
      const double c = fma(0.5, two ? su + (vp + vm) : su, 1.0);
      H = 0.5 * c * c;
      ax = fma(0.5, two ? fabs(du) + fabs(vp - vm) : fabs(du), fabs(c));
      ay = two ? ax : 0.0;
    } break;
    case H_NEGCOS2D:
    case H_NEGCOS1D:
    case H_SIN2D: {
      const bool two = kind != H_NEGCOS1D;
      const double s2 = two ? su + (vp + vm) : su;
      const double c = kind == H_SIN2D ? 0.5 * s2 : fma(0.5, s2, 1.0);
      double sn, cs;
      sincos(c, &sn, &cs);
      H = kind == H_SIN2D ? sn : -cs;
      const double a = fabs(kind == H_SIN2D ? cs : sn), b = fabs(kind == H_SIN2D ? sn : cs);
      const double dv = two ? vp - vm : 0.0;
      const double e = 0.5 * (fabs(du) + fabs(dv));
      ax = 0.0;
      if (!(fma(b, e, a) <= known)) {
        const double e2 = 0.5 * fabs(fabs(du) - fabs(dv));
        auto corner = [&](double d) {
          double sd, cd;
          if (d <= 0.015625) {
            const double q = d * d;
            cd = fma(q, fma(q, fma(q, -1.0 / 720.0, 1.0 / 24.0), -0.5), 1.0);
            sd = d * fma(q, fma(q, 1.0 / 120.0, -1.0 / 6.0), 1.0);
            return fma(a, cd, b * sd);
          }
          sincos(c + d, &sn, &cs);
          const double r1 = fabs(kind == H_SIN2D ? cs : sn);
          sincos(c - d, &sn, &cs);
          return max_bits(r1, fabs(kind == H_SIN2D ? cs : sn));
        };
        ax = corner(e);
        if (two) ax = max_bits(ax, corner(e2));
      }
      ay = two ? ax : 0.0;
    } break;
    case H_ADVECT1D: {
      H = 0.5 * su;
      ax = fabs(su) < INFINITY ? 1.0 : NAN;
      ay = 0.0;
    } break;
    case H_EIKONAL2D: {
      const double p = 0.5 * su, q = 0.5 * (vp + vm);
      H = sqrt(fma(p, p, fma(q, q, 1.0)));
      // |H_p| = |u| / sqrt(u^2 + v^2 + 1) grows with |u| and falls with |v|
      const double ul = min_bits(fabs(um), fabs(up)), uh = max_bits(fabs(um), fabs(up));
      const double vl = min_bits(fabs(vm), fabs(vp)), vh = max_bits(fabs(vm), fabs(vp));
      ax = uh * rsqrt(fma(uh, uh, fma(vl, vl, 1.0)));
      ay = vh * rsqrt(fma(vh, vh, fma(ul, ul, 1.0)));
    } break;
    default:
      H = ham_value<double>(kind, 0.5 * su, 0.5 * (vp + vm), x, y);
      node_alpha<double>(kind, um, up, vm, vp, x, y, ax, ay);
  }
}

template <int PREC> struct Types;
template <> struct Types<P_F64> { using S = double; using C = double; };
template <> struct Types<P_F32> { using S = float; using C = float; };
template <> struct Types<P_MIXED> { using S = float; using C = float; };

// SMALL (FP64 2D grids too small to fill the GPU with the default tiles): 16 x 16 tiles with 4-node
// sweep segments (SMALL = 1), or 2-node segments (SMALL = 2: twice the threads per tile, for grids
// whose 16 x 16 tiles are fewer than the SMs).
template <int PREC, int DIM, int SMALL = 0> struct Shape {
  static constexpr int TX = (DIM == 2) ? (SMALL ? 16 : Tile<PREC>::TX) : (PREC == P_F64 ? TX1D64 : TX1D);
  static constexpr int TY = (DIM == 2) ? (SMALL ? 16 : Tile<PREC>::TY) : 1;
  static constexpr int K = (DIM == 2) ? (SMALL == 2 ? 2 : SMALL == 1 ? 4 : Tile<PREC>::K) : (PREC == P_F64 ? 1 : K1D);
  static constexpr int NT = (TX / K) * TY;          // threads per CTA
  static constexpr int MINB = (PREC == P_F64 && DIM == 2) ? 512 / NT : 1;   // FP64: 16 warps per SM
  static constexpr int SW = TX + 8;                 // smem row: GX halo on each side
  static constexpr int SH = (DIM == 2) ? TY + 6 : 1;
  static constexpr int NARR = (PREC == P_MIXED) ? 3 : 1;
  static constexpr size_t smem_bytes() {
    return (size_t)NARR * SH * SW * sizeof(typename Types<PREC>::S) +
           (DIM == 2 ? (size_t)TY * TX * 2 * sizeof(typename Types<PREC>::C) : 0);
  }
};

// FP64: one-sided derivatives of K consecutive nodes from the cells a, a + step, ... (a = first node - 3) with
// the weights in float pairs; nv nodes of the segment count.  False when the segment does not qualify (and
// for the float variants).
template <int PREC, int K, int W, class S, class C>
__device__ __forceinline__ bool sweep_pairs(const S *a, int step, const SweepArgs<PREC> &sw, bool along_y, int nv,
                                            C (&dm)[K], C (&dp)[K]) {
  if constexpr (PREC == P_F64) {
    return sweep64<K, W>([&](int m) { return a[m * step]; }, along_y ? sw.y : sw.x, nv, [&](int q, double x, double y) {
      dm[q] = x;
      dp[q] = y;
    });
  } else {
    return false;
  }
}

template <int PREC, int DIM, int WEIGHTS, int SMALL>
__global__ void __launch_bounds__(Shape<PREC, DIM, SMALL>::NT, Shape<PREC, DIM, SMALL>::MINB)
    stage_kernel(const StageParams p, const SweepArgs<PREC> sw) {
  using S = typename Types<PREC>::S;
  using C = typename Types<PREC>::C;
  using Sh = Shape<PREC, DIM, SMALL>;
  constexpr int TX = Sh::TX, TY = Sh::TY, K = Sh::K, NT = Sh::NT, SW = Sh::SW, SH = Sh::SH;

  DevState *st = p.state;
  if (p.loop_mode == LOOP_STEP_TO && !(st->t < st->t_final)) return;
  if (st->err) return;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  S *s_a = reinterpret_cast<S *>(smem_raw);            // phi (or hi)
  S *s_b = s_a + SH * SW;                               // lo (MIXED)
  S *s_c = s_b + SH * SW;                               // previous stage's increment (MIXED)
  C *s_u = reinterpret_cast<C *>(smem_raw + (size_t)Sh::NARR * SH * SW * sizeof(S));
  __shared__ double s_red[2][NT / 32];
  __shared__ int s_last;

  const int tid = threadIdx.x;
  const int tx0 = blockIdx.x * TX, ty0 = blockIdx.y * TY;
  const int cur = (PREC == P_MIXED) ? st->cur : 0;

  // ---- time step of this stage
  double dt;
  int last = 0;
  if (p.stage == 1 && p.loop_mode != LOOP_STAGE) {
    double ax, ay;
    if (p.alpha_mode == A_FIXED) {
      ax = p.alpha_fixed[0];
      ay = p.alpha_fixed[1];
    } else {
      ax = bits_to_double(st->alpha_bits[p.dt_slot][0]);
      ay = bits_to_double(st->alpha_bits[p.dt_slot][1]);
    }
    double den = ax / p.lx;
    if (DIM == 2) den += ay / p.ly;
    dt = den > 0.0 ? p.cfl / den : (p.loop_mode == LOOP_ADVANCE ? 0.0 : INFINITY);
    if (p.loop_mode == LOOP_STEP_TO && st->t + dt >= st->t_final) {
      dt = st->t_final - st->t;
      last = 1;
    }
  } else if (p.loop_mode == LOOP_STAGE) {
    dt = p.dt_value;
  } else {
    dt = st->dt;
  }
  // ---- alpha of the flux when it is one value for the whole grid
  C fax = C(0), fay = C(0);
  const bool local_alpha = (p.alpha_mode == A_LOCAL_LAGGED || p.alpha_mode == A_LOCAL_EXACT);
  if (p.alpha_mode == A_FIXED) {
    fax = C(p.alpha_fixed[0]);
    fay = C(p.alpha_fixed[1]);
  } else if (!local_alpha && p.read_slot >= 0) {
    fax = C(bits_to_double(st->alpha_bits[p.read_slot][0]));
    fay = C(bits_to_double(st->alpha_bits[p.read_slot][1]));
  }

  // ---- load the tile and its halo (row 0 of smem = interior row ty0-3, col 0 = interior col tx0-4)
  const S *ga = reinterpret_cast<const S *>(PREC == P_MIXED ? p.mix_hi[cur] : p.src0);
  const S *gb = reinterpret_cast<const S *>(PREC == P_MIXED ? p.mix_lo[cur] : nullptr);
  const S *gc = reinterpret_cast<const S *>(p.src2);
  for (int idx = tid; idx < SH * SW; idx += NT) {
    const int r = idx / SW, c = idx - r * SW;
    const size_t g = (size_t)((DIM == 2) ? ty0 + r : 0) * p.pitch + tx0 + c;
    s_a[idx] = ga[g];
    if (PREC == P_MIXED) {
      s_b[idx] = gb[g];
      if (gc) s_c[idx] = gc[g];
    }
  }
  // MIXED: the stage's input is hi + X, X = the low part of phi^n (stage 1) or the increment array of the
  // previous stage, which holds the low part as well (stages 2 and 3; see finish_node)
  const S *s_x = gc ? s_c : s_b;
  __syncthreads();

  const C dx = C(p.dx), rdx = C(p.rdx), eps = C(p.eps);
  // Delta^+ phi between smem cells i0 and i1 (same row or column)
  auto diff = [&](int i0, int i1, C rd) -> C {
    if (PREC == P_MIXED) {
      return ((s_a[i1] - s_a[i0]) + (s_x[i1] - s_x[i0])) * rd;
    } else {
      return C(s_a[i1] - s_a[i0]) * rd;
    }
  };

  C amx = C(0), amy = C(0);
  bool bad = false;
  if constexpr (PREC == P_F64) {
    // what other CTAs have folded so far is a lower bound of the grid maximum
    if (!local_alpha && p.write_slot >= 0) {
      amx = bits_to_double(*(volatile unsigned long long *)&st->alpha_bits[p.write_slot][0]);
      amy = bits_to_double(*(volatile unsigned long long *)&st->alpha_bits[p.write_slot][1]);
    }
  }

  // RK combination, store, and alpha bookkeeping for node (lx, ly) of the tile
  auto finish_node = [&](int lxn, int lyn, C um, C up, C vm, C vp) {
    const int gi = tx0 + lxn, gj = ty0 + lyn;
    if (gi >= p.nx || gj >= p.ny) return;
    C ax, ay, H;
    const C xn = C(p.xlo + gi * p.dx), yn = C(p.ylo + gj * p.dy);
    if constexpr (PREC == P_F64) {
      ham_node64(p.ham, um, up, vm, vp, xn, yn, local_alpha ? -1.0 : (amx < amy ? amx : amy), H, ax, ay);
      amx = max_bits(amx, ax);
      amy = max_bits(amy, ay);
    } else {
      node_alpha<C>(p.ham, um, up, vm, vp, xn, yn, ax, ay);
      H = ham_value<C>(p.ham, C(0.5) * (up + um), C(0.5) * (vp + vm), xn, yn);
      if (!(isfinite(ax) && isfinite(ay))) bad = true;
      amx = fmax(amx, ax);
      amy = fmax(amy, ay);
    }
    if (p.stage == 0) return;
    const C aX = local_alpha ? ax : fax, aY = local_alpha ? ay : fay;
    const C L = -((H - aX * C(0.5) * (up - um)) - aY * C(0.5) * (vp - vm));
    const int sidx = ((DIM == 2) ? lyn + 3 : 0) * SW + lxn + 4;
    if (PREC == P_MIXED) {
      // phi^n = hi + lo and phi_k = hi + e_k with e_k = lo + (phi_k - phi^n):
      //   e_1 = lo + dt L,  e_2 = 3/4 lo + 1/4 (e_1 + dt L),  phi^{n+1} = hi + lo + 2/3 (e_2 + dt L - lo)
      const float dL = float(dt) * float(L);
      const float lo = float(s_b[sidx]);
      if (p.stage == 1) {
        store_node<float, DIM>(reinterpret_cast<float *>(p.out0), p.pitch, p.nx, p.ny, p.bc, gi, gj, lo + dL);
      } else if (p.stage == 2) {
        const float d = fmaf(0.75f, lo, 0.25f * (float(s_c[sidx]) + dL));
        store_node<float, DIM>(reinterpret_cast<float *>(p.out0), p.pitch, p.nx, p.ny, p.bc, gi, gj, d);
      } else {
        const float d = (2.0f / 3.0f) * ((float(s_c[sidx]) + dL) - lo);
        float h, l;
        df_add(float(s_a[sidx]), float(s_b[sidx]), d, h, l);
        store_node<float, DIM>(reinterpret_cast<float *>(p.mix_hi[cur ^ 1]), p.pitch, p.nx, p.ny, p.bc, gi, gj, h);
        store_node<float, DIM>(reinterpret_cast<float *>(p.mix_lo[cur ^ 1]), p.pitch, p.nx, p.ny, p.bc, gi, gj, l);
      }
    } else {
      const C src = C(s_a[sidx]);
      C outv;
      if (p.stage == 1) {
        outv = src + C(dt) * L;
      } else {
        const size_t g = (size_t)(gj + ((DIM == 2) ? GY : 0)) * p.pitch + gi + GX;
        const C base = C(reinterpret_cast<const S *>(p.base0)[g]);
        if (p.stage == 2) outv = C(0.75) * base + C(0.25) * (src + C(dt) * L);
        else if (PREC == P_F64) {
          // (phi^n + 2 (phi_2 + dt L)) / 3, the division as a product with its remainder folded back
          const C z = fma(C(2), fma(C(dt), L, src), base), third = C(1) / C(3), q = z * third;
          outv = fma(fma(C(-3), q, z), third, q);
        } else outv = base / C(3) + C(2) * (src + C(dt) * L) / C(3);
      }
      store_node<S, DIM>(reinterpret_cast<S *>(p.out0), p.pitch, p.nx, p.ny, p.bc, gi, gj, S(outv));
    }
  };

  // nodes of a K-node segment that lie inside the grid
  auto valid = [&](int left, bool inside) { return !inside || left <= 0 ? -9 : (left < K ? left : K); };

  // ---- phase X: each thread sweeps K consecutive nodes of one row
  {
    constexpr int SEGS = TX / K;
    const int r = tid / SEGS, seg = tid - r * SEGS;
    const int srow = (DIM == 2) ? r + 3 : 0;
    const int base_i = srow * SW + seg * K + 1;     // smem index of node x = seg*K - 3
    C dm[K], dp[K];
    const int nv = valid(p.nx - tx0 - seg * K, DIM == 1 || ty0 + r < p.ny);
    if (!sweep_pairs<PREC, K, WEIGHTS>(s_a + base_i, 1, sw, false, nv, dm, dp)) {
      C v[K + 5];
#pragma unroll
      for (int m = 0; m < K + 5; ++m) v[m] = diff(base_i + m, base_i + m + 1, rdx);
      weno_sweep<C, K, WEIGHTS>(v, rdx, dx, eps, dm, dp);
    }
    if (DIM == 2) {
#pragma unroll
      for (int q = 0; q < K; ++q) {
        s_u[2 * (r * TX + seg * K + q)] = dm[q];
        s_u[2 * (r * TX + seg * K + q) + 1] = dp[q];
      }
    } else {
#pragma unroll
      for (int q = 0; q < K; ++q) finish_node(seg * K + q, 0, dm[q], dp[q], C(0), C(0));
    }
  }
  if (DIM == 2) {
    __syncthreads();
    // ---- phase Y: each thread sweeps K consecutive nodes of one column
    const int x = tid % TX, seg = tid / TX;
    const int col = x + 4;
    const C dy = C(p.dy), rdy = C(p.rdy);
    C vm[K], vp[K];
    const int nv = valid(p.ny - ty0 - seg * K, tx0 + x < p.nx);
    if (!sweep_pairs<PREC, K, WEIGHTS>(s_a + seg * K * SW + col, SW, sw, true, nv, vm, vp)) {
      C v[K + 5];
#pragma unroll
      for (int m = 0; m < K + 5; ++m) v[m] = diff((seg * K + m) * SW + col, (seg * K + m + 1) * SW + col, rdy);
      weno_sweep<C, K, WEIGHTS>(v, rdy, dy, eps, vm, vp);
    }
#pragma unroll
    for (int q = 0; q < K; ++q) {
      const int y = seg * K + q;
      finish_node(x, y, s_u[2 * (y * TX + x)], s_u[2 * (y * TX + x) + 1], vm[q], vp[q]);
    }
  }

  // ---- grid maximum of alpha: warp shuffle, then one atomicMax per CTA
  double mx = double(amx), my = double(amy);
  if (PREC == P_F64) {
    // a NaN or an infinity in any alpha is the thread's maximum
    bad = !(mx < INFINITY) || !(my < INFINITY);
    if (bad) mx = my = 0.0;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mx = max_bits(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    my = max_bits(my, __shfl_xor_sync(0xffffffffu, my, o));
  }
  const int anybad = __syncthreads_or(bad ? 1 : 0);
  if ((tid & 31) == 0) {
    s_red[0][tid >> 5] = mx;
    s_red[1][tid >> 5] = my;
  }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < NT / 32; ++w) {
      mx = max_bits(mx, s_red[0][w]);
      my = max_bits(my, s_red[1][w]);
    }
    if (anybad) atomicOr(&st->err, 1);
    if (p.write_slot >= 0) {
      atomicMax(&st->alpha_bits[p.write_slot][0], double_to_bits(mx));
      atomicMax(&st->alpha_bits[p.write_slot][1], double_to_bits(my));
    }
    // last-CTA epilogue: every other CTA has finished reading the state
    __threadfence();
    const unsigned int total = gridDim.x * gridDim.y;
    const unsigned int prev = atomicAdd(&st->counter, 1u);
    s_last = (prev == total - 1);
  }
  __syncthreads();
  if (s_last && tid == 0) {
    __threadfence();
    st->counter = 0;
    if (p.zero_slot >= 0) {
      st->alpha_bits[p.zero_slot][0] = 0ull;
      st->alpha_bits[p.zero_slot][1] = 0ull;
    }
    if (p.stage == 1 && p.loop_mode != LOOP_STAGE) {
      st->dt = dt;
      st->last = last;
    }
    if (p.stage == 3) {
      if (PREC == P_MIXED) st->cur = cur ^ 1;
      if (p.loop_mode != LOOP_STAGE) {
        st->t = st->last ? st->t_final : st->t + st->dt;
        st->steps += 1;
      }
    }
  }
}

}  // namespace alw
