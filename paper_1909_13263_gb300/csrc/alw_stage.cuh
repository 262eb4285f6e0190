// The fused RK-stage kernel (see alw_device.cuh for the arithmetic).
#pragma once
#include <type_traits>

#include "alw_device.cuh"
#include "alw_node64.cuh"
#include "alw_sweep64.cuh"

namespace alw {

// Constants of the FP64 sweeps, formed on the host (nothing for the float variants).
template <int PREC> struct SweepArgs {};
template <> struct SweepArgs<P_F64> {
  Sweep64 c[2];
};
template <int PREC, int W>
static SweepArgs<PREC> sweep_args(const StageParams &p) {
  SweepArgs<PREC> a;
  if constexpr (PREC == P_F64) {
    a.c[0] = make_sweep64<W>(p.dx, p.eps, p.nx);
    a.c[1] = p.dim == 2 ? make_sweep64<W>(p.dy, p.eps, p.ny) : a.c[0];
  }
  return a;
}

template <int PREC> struct Types;
template <> struct Types<P_F64> { using S = double; using C = double; };
template <> struct Types<P_F32> { using S = float; using C = float; };
template <> struct Types<P_MIXED> { using S = float; using C = float; };

// SHAPE: tile shape of the FP64 2D grids.  In 2D half of the threads sweep rows and half columns.
template <int PREC, int DIM, int SHAPE = 0> struct Shape {
  static constexpr int TX = (DIM == 2) ? kShape64[SHAPE].tx : (PREC == P_F64 ? TX1D64 : TX1D);
  static constexpr int TY = (DIM == 2) ? kShape64[SHAPE].ty : 1;
  static constexpr int K = (DIM == 2) ? kShape64[SHAPE].k : (PREC == P_F64 ? 1 : K1D);
  static constexpr int NSEG = (TX / K) * TY;        // segments per direction
  static constexpr int NT = NSEG * DIM;             // threads per CTA
  static constexpr int MINB = (PREC == P_F64 && DIM == 2) ? kShape64[SHAPE].warps * 32 / NT : 1;
  static constexpr int SW = TX + 8;                 // smem row: GX halo on each side
  static constexpr int SH = (DIM == 2) ? TY + 6 : 1;
  // FP64 2D: sides that did not qualify from which a tile's threads sweep their own segments in double instead of
  // sharing a list of sides: a sixth of all.  The list costs twice the FP64 operations (nothing is shared between the
  // sides of a stencil) after a pair form in vain; a thread's sweep idles where few of its warp's segments have such
  // nodes.  Microseconds per RK3 step, always the list / from a half / from a sixth; with double indicators throughout:
  //   Example 3, noise on all nodes    2048^2 57290 / 16580 / 16580; 15040     512^2 3820 / 1155 / 1155; 1149
  //   noise on 3 % of them                    23250 / 19290 / 15840; 24740           2060 / 1410 / 1150; 1605
  //   noise on 1 %                            10760 / 10720 / 12240; 24970           1250 / 1110 / 1080; 1755
  //   shocks of a long run              256^2 666 / 364 / 242; 581    Example 10, 1024^2 1128 / 918 / 860; 8330
  //   Jiang-Peng, noise on all         2048^2 17210 / 5660 / 5660; 5000
  static constexpr int kDense = 2 * DIM * TX * TY / 6;
  static constexpr int NARR = (PREC == P_MIXED) ? 3 : 1;
  static constexpr size_t smem_bytes() {
    return (size_t)NARR * SH * SW * sizeof(typename Types<PREC>::S) +
           (PREC == P_F64 ? (size_t)DIM * TY * TX * 2 * (sizeof(double) + sizeof(short)) : 0);  // derivatives, list
  }
};

template <int PREC, int DIM, int WEIGHTS, int SHAPE>
__global__ void __launch_bounds__(Shape<PREC, DIM, SHAPE>::NT, Shape<PREC, DIM, SHAPE>::MINB)
    stage_kernel(const StageParams p, const SweepArgs<PREC> sw) {
  using S = typename Types<PREC>::S;
  using C = typename Types<PREC>::C;
  using Sh = Shape<PREC, DIM, SHAPE>;
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
  __shared__ int s_last, s_nrare;

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

  if (tid == 0) s_nrare = 0;
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
      const size_t g = (size_t)(gj + ((DIM == 2) ? GY : 0)) * p.pitch + gi + GX;
      const C base = p.stage == 1 ? C(0) : C(reinterpret_cast<const S *>(p.base0)[g]);
      C outv;
      if constexpr (PREC == P_F64) outv = rk_node64(p.stage, base, src, dt, L);
      else if (p.stage == 1) outv = src + C(dt) * L;
      else if (p.stage == 2) outv = C(0.75) * base + C(0.25) * (src + C(dt) * L);
      else outv = base / C(3) + C(2) * (src + C(dt) * L) / C(3);
      store_node<S, DIM>(reinterpret_cast<S *>(p.out0), p.pitch, p.nx, p.ny, p.bc, gi, gj, S(outv));
    }
  };

  if constexpr (PREC == P_F64) {
    // each thread sweeps K consecutive nodes of one row or one column, one code for both (see
    // alw_sweep64.cuh); the results go through shared memory, so that the sweep's loop holds nothing of what
    // finishing a node needs (registers)
    double2 *su = reinterpret_cast<double2 *>(s_u), *sv = su + (DIM - 1) * TY * TX;
    unsigned short *s_rare = reinterpret_cast<unsigned short *>(su + DIM * TY * TX);
    unsigned mine;   // the thread's segment: nodes that did not qualify
    auto segment = [&](auto use) {
      constexpr int SEGS = TX / K;
      const int dir = (DIM == 2 && tid >= Sh::NSEG) ? 1 : 0, seg = tid - dir * Sh::NSEG;
      const int x = dir == 0 ? (seg % SEGS) * K : seg % TX, y = dir == 0 ? seg / SEGS : (seg / TX) * K;
      const S *a = s_a + (DIM == 2 ? y + (dir == 0 ? 3 : 0) : 0) * SW + x + (dir == 0 ? 1 : 4);
      const int step = dir == 0 ? 1 : SW, ostep = dir == 0 ? 1 : TX, node0 = y * TX + x;
      // nodes of the segment that lie inside the grid
      const int left = dir == 0 ? p.nx - tx0 - x : p.ny - ty0 - y;
      const bool inside = dir == 0 ? (DIM == 1 || ty0 + y < p.ny) : tx0 + x < p.nx;
      use(a, step, dir, node0, ostep, !inside || left <= 0 ? -1 : (left < K ? left : K));
    };
    segment([&](const S *a, int step, int dir, int node0, int ostep, int nv) {
      double2 *o = (dir == 0 ? su : sv) + node0;
      mine = sweep64<WEIGHTS>(a, step, sw.c[dir], nv,
                              [&](int q, double dm, double dp) { o[q * ostep] = make_double2(dm, dp); });
      // nodes that did not qualify: both sides of each into the CTA's list
      for (unsigned rare = mine; rare; rare &= rare - 1) {
        const int q = __ffs(rare) - 1, at = atomicAdd(&s_nrare, 2);
        s_rare[at] = (unsigned short)(((dir * TY * TX + node0 + q * ostep) << 1));
        s_rare[at + 1] = (unsigned short)(s_rare[at] | 1);
      }
    });
    __syncthreads();
    if (DIM == 2 && s_nrare >= Sh::kDense) {
      // ... many (noise, data that the grid does not resolve): each thread its segment's, in double
      if (mine) {
        segment([&](const S *a, int step, int dir, int node0, int ostep, int) {
          sweep64_double<WEIGHTS>(a, step, sw.c[dir], mine, reinterpret_cast<double *>((dir == 0 ? su : sv) + node0),
                                  ostep);
        });
      }
      __syncthreads();
    } else if (s_nrare > 0) {
      // ... which all threads share: the kinks of a tile touch few threads' segments
      for (int i = tid; i < s_nrare; i += NT) {
        const int e = s_rare[i] >> 1, dir = e / (TY * TX), n = e % (TY * TX), x = n % TX, y = n / TX;
        const int step = dir == 0 ? 1 : SW;
        const S *a = s_a + (DIM == 2 ? y + (dir == 0 ? 3 : 0) : 0) * SW + x + (dir == 0 ? 1 : 4);
        double *o = reinterpret_cast<double *>((dir == 0 ? su : sv) + n);
        if (s_rare[i] & 1) o[1] = -minus64_rare<WEIGHTS>(a + 6 * step, -step, sw.c[dir]);
        else o[0] = minus64_rare<WEIGHTS>(a, step, sw.c[dir]);
      }
      __syncthreads();
    }
#pragma unroll 1
    for (int n = tid; n < TX * TY; n += NT) {
      const double2 u = su[n], v = DIM == 2 ? sv[n] : make_double2(0.0, 0.0);
      finish_node(n % TX, n / TX, u.x, u.y, v.x, v.y);
    }
  } else {
    static_assert(PREC == P_F64 || DIM == 1, "2D float stages run the persistent kernel");
    const int base_i = tid * K + 1;     // smem index of the segment's first node - 3
    C v[K + 5];
#pragma unroll
    for (int m = 0; m < K + 5; ++m) v[m] = diff(base_i + m, base_i + m + 1, rdx);
    C dm[K], dp[K];
    weno_sweep<C, K, WEIGHTS>(v, rdx, dx, eps, dm, dp);
#pragma unroll
    for (int q = 0; q < K; ++q) finish_node(tid * K + q, 0, dm[q], dp[q], C(0), C(0));
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
