// Whole RK3 steps of a 1D FP64 grid in one launch.
//
// A 1D grid of the paper's sizes (40 to 320 nodes) is a few warps of work; a launch per stage costs several
// times what the stage's arithmetic takes.  Here one thread-block cluster holds the whole grid in shared memory
// (phi^n and the two stage states, about 64 nodes per CTA, one thread per node) and runs step after step: the
// neighbours' edge values are read from their shared memory, the maxima of |dH/dp| are folded into every CTA's
// copy by remote atomics, and one cluster barrier closes a stage.  The device state (t, dt, steps, the alpha
// ring) is read at the start and written at the end as the per-stage kernels would leave it.
//
// Each thread forms one stencil -- both deviations it serves, the "-" side of its node and the "+" side of the
// node before, which is handed over in shared memory (alw_sweep64.cuh has the arithmetic).
//
// What bounds it: the latency of one stage's dependent operations.  Measured (GB300, RK3 steps of Example 6):
// N = 80 smooth 13 us per step (three stages), with kinks 20-68 us, against 72 us for the same arithmetic in one
// launch per stage (rare nodes included) and 570 us for the double-precision indicators; whole solves N = 80
// to t = 0.5/pi^2 8.1 -> 0.28 ms, N = 320 to 3.5/pi^2 195 -> 19.2 ms.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "alw_node64.cuh"
#include "alw_sweep64.cuh"

namespace alw {

namespace {

namespace cg = cooperative_groups;

constexpr int kLineNodes = 64;    // nodes per CTA aimed at
constexpr int kLineCluster = 8;   // CTAs of the largest (portable) cluster
constexpr int kLineCap = kLine64Max / kLineCluster;
constexpr int kLineThreads = kLineCap + 32;

// The cluster barrier in its unaligned form: a warp whose threads have not reconverged arrives thread by thread
// (the aligned form would count such a warp's arrival more than once).
__device__ __forceinline__ void cluster_barrier() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

struct LineParams {
  StageParams p;
  Sweep64 c;
  int nsteps;
};

template <int W>
__global__ void __launch_bounds__(kLineThreads) line64_kernel(const __grid_constant__ LineParams q) {
  const StageParams &p = q.p;
  const Sweep64 &c = q.c;
  DevState *st = p.state;
  if (st->err) return;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), ranks = (int)cl.num_blocks(), tid = threadIdx.x, lane = tid & 31;
  const int n = p.nx;
  // nodes [first, first + count) of this CTA, every CTA's share differing by one at most
  const int first = (int)((long long)n * rank / ranks), count = (int)((long long)n * (rank + 1) / ranks) - first;

  __shared__ double s_phi[3][kLineCap + 6];           // phi^n, stage 1, stage 2; cell k = node first + k - 3
  __shared__ float4 s_plus[kLineCap + 1];             // "+" deviation (pair) and |T_3| of each stencil
  __shared__ double2 s_u[kLineCap];                   // one-sided derivatives of nodes recomputed by others
  __shared__ unsigned short s_rare[2 * kLineCap];
  __shared__ int s_nrare[2];
  __shared__ double s_wmax[3][kLineThreads / 32];     // maximum of |dH/dp| per stage and warp
  __shared__ double s_alpha;                          // the grid's, of the last stage

  double t = st->t, dt = st->dt;
  const double t_final = st->t_final;
  double alpha = bits_to_double(st->alpha_bits[2][0]), alpha2 = bits_to_double(st->alpha_bits[1][0]);
  long long steps = 0;
  int last = st->last, err = 0;
  double *P = reinterpret_cast<double *>(p.out0);
  for (int k = tid; k < count + 6; k += blockDim.x) s_phi[0][k] = P[GX + first + k - 3];
  if (tid < 2) s_nrare[tid] = 0;
  const int warps = blockDim.x / 32;
  const bool local_alpha = p.alpha_mode == A_LOCAL_LAGGED || p.alpha_mode == A_LOCAL_EXACT;
  cluster_barrier();

  int par = 0;
  for (int step = 0; step < q.nsteps && !err; ++step) {
    if (p.loop_mode == LOOP_STEP_TO && !(t < t_final)) break;
    {
      const double den = (p.alpha_mode == A_FIXED ? p.alpha_fixed[0] : alpha) / p.lx;
      dt = den > 0.0 ? p.cfl / den : (p.loop_mode == LOOP_ADVANCE ? 0.0 : INFINITY);
      last = p.loop_mode == LOOP_STEP_TO && t + dt >= t_final;
      if (last) dt = t_final - t;
    }
#pragma unroll 1
    for (int stage = 1; stage <= 3; ++stage, par ^= 1) {
      const double *src = s_phi[stage - 1];
      double *dst = s_phi[stage == 3 ? 0 : stage];
      // ---- stencil tid: cells of node tid
      double v2 = 0.0, v3 = 0.0, v4 = 0.0, d1 = 0.0, d2 = 0.0, d3 = 0.0, s4 = 0.0;
      df minus = {0.0f, 0.0f};
      float tm = 0.0f;
      unsigned pb = 0;
      bool ok = true;
      if (tid <= count) {
        double x[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          x[k] = src[tid + k];
          const unsigned h = hi_(x[k]) & 0x7fffffffu;
          pb = h > pb ? h : pb;
        }
        const double v0 = x[1] - x[0], v1 = x[2] - x[1];
        v2 = x[3] - x[2];
        v3 = x[4] - x[3];
        v4 = x[5] - x[4];
        const double s1 = v1 - v0, s2 = v2 - v1, s3 = v3 - v2;
        s4 = v4 - v3;
        d1 = s2 - s1;
        d2 = s3 - s2;
        d3 = s4 - s3;
        const df D1 = mul_(split_(s1), c.scale), D2 = mul_(split_(s2), c.scale), D3 = mul_(split_(s3), c.scale);
        const df D4 = mul_(split_(s4), c.scale);
        const df w1 = sub_(D2, D1), w2 = sub_(D3, D2), w3 = sub_(D4, D3), T2 = sub_(w2, w1), T3 = sub_(w3, w2);
        df S = {0.0f, 0.0f}, q0, q1, q2, plus;
        if (W == W_ARCLEN) S = root_(D2);
        stencil_q<W>(D1, D2, D3, D4, w1, w2, w3, S, c, q0, q1, q2);
        ok = stencil_devs(q0, q1, q2, T2, T3, minus, plus);
        tm = fmaxf(fabsf(T2.h), fabsf(T3.h));
        s_plus[tid] = make_float4(plus.h, plus.l, fabsf(T3.h), ok ? 1.0f : 0.0f);
      }
      if (tid == 0) s_nrare[par ^ 1] = 0;
      __syncthreads();
      // ---- node tid
      double dm = 0.0, dp = 0.0;
      bool rare = false;
      if (tid < count) {
        const double x6 = src[tid + 6], s5 = (x6 - src[tid + 5]) - v4, d4 = s5 - s4;
        const float4 pl = s_plus[tid + 1];
        const double am = c.c0 * (v2 + v3);
        const double lm = fma(c.c2, d2, fma(c.c1, d1, fma(c.c3, d3, am)));
        const double lp = fma(c.c2, d3, fma(c.c1, d4, fma(c.c3, d2, am)));
        dm = fma(-c.cdev, widen_(minus.h) + widen_(minus.l), lm);
        dp = fma(c.cdev, widen_(pl.x) + widen_(pl.y), lp);
        rare = !(ok && pl.w != 0.0f && fmaxf(tm, pl.z) * c.t2phi <= phi_size(pb));
        if (rare) {
          const int at = atomicAdd(&s_nrare[par], 2);
          s_rare[at] = (unsigned short)(2 * tid);
          s_rare[at + 1] = (unsigned short)(2 * tid + 1);
        }
      }
      __syncthreads();
      const int nrare = s_nrare[par];
      if (nrare > 0) {
        for (int i = tid; i < nrare; i += blockDim.x) {
          const int e = s_rare[i], k = e >> 1;
          if (e & 1) s_u[k].y = -minus64_rare<W>(src + k + 6, -1, c);
          else s_u[k].x = minus64_rare<W>(src + k, 1, c);
        }
        __syncthreads();
        if (rare) {
          dm = s_u[tid].x;
          dp = s_u[tid].y;
        }
      }
      // ---- Hamiltonian, RK combination, maximum
      double ax = 0.0;
      if (tid < count) {
        double H, ay;
        const double xn = p.xlo + (first + tid) * p.dx;
        ham_node64(p.ham, dm, dp, 0.0, 0.0, xn, 0.0, -1.0, H, ax, ay);
        const double a = local_alpha ? ax : (p.alpha_mode == A_FIXED ? p.alpha_fixed[0] : alpha);
        const double L = -(H - a * 0.5 * (dp - dm));
        dst[tid + 3] = rk_node64(stage, s_phi[0][tid + 3], src[tid + 3], dt, L);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ax = max_bits(ax, __shfl_xor_sync(0xffffffffu, ax, o));
      if (lane == 0) s_wmax[stage - 1][tid >> 5] = ax;
      cluster_barrier();
      // ---- the first warp: the maximum over the cluster's warps
      if (tid < 32) {
        double a = 0.0;
        for (int k = lane; k < ranks * warps; k += 32)
          a = max_bits(a, cl.map_shared_rank(s_wmax[stage - 1], k / warps)[k % warps]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a = max_bits(a, __shfl_xor_sync(0xffffffffu, a, o));
        if (lane == 0) s_alpha = a;
      }
      // ---- ghost cells: from the neighbours (periodic images), or extrapolated at the grid's ends
      const int gt = tid - (blockDim.x - 32);   // by the last warp
      if (gt >= 0 && gt < 6) {
        const int g = gt < 3 ? first - 1 - gt : first + count + gt - 3;   // grid position
        const int cell = g - first + 3;
        if (p.bc == BC_PERIODIC || (g >= 0 && g < n)) {
          int w = g % n;
          if (w < 0) w += n;
          int r = (int)((long long)w * ranks / n);      // its owner: [n r / ranks, n (r + 1) / ranks)
          if (w >= (int)((long long)n * (r + 1) / ranks)) ++r;
          dst[cell] = cl.map_shared_rank(dst, r)[w - (int)((long long)n * r / ranks) + 3];
        } else if (g < 0) {
          const double m = (double)(-g);
          dst[cell] = (1.0 + m) * dst[3] - m * dst[4];
        } else {
          const double m = (double)(g - (n - 1));
          dst[cell] = (1.0 + m) * dst[count + 2] - m * dst[count + 1];
        }
      }
      __syncthreads();
      alpha2 = stage == 3 ? alpha : alpha2;
      alpha = s_alpha;
      if (!(alpha < INFINITY)) {   // the same value in every CTA
        err = 1;
        alpha = 0.0;
        if (stage < 3) break;
      }
      if (stage == 3) {
        t = last ? t_final : t + dt;
        ++steps;
      }
    }
  }
  // ---- back to global memory: phi^n with its ghosts and the device state
  if (tid < count) store_node<double, 1>(P, p.pitch, n, 1, p.bc, first + tid, 0, s_phi[0][tid + 3]);
  if (p.bc != BC_PERIODIC && tid < 3) {
    if (rank == 0) P[GX - 1 - tid] = s_phi[0][2 - tid];
    if (rank == ranks - 1) P[GX + n + tid] = s_phi[0][count + 3 + tid];
  }
  if (rank == 0 && tid == 0) {
    st->dt = dt;
    st->last = last;
    if (steps > 0) {
      st->t = t;
      st->steps += steps;
      st->alpha_bits[0][0] = st->alpha_bits[0][1] = 0ull;
      st->alpha_bits[1][0] = double_to_bits(alpha2);
      st->alpha_bits[2][0] = double_to_bits(alpha);
    }
    if (err) st->err |= 1;
  }
  cluster_barrier();  // no CTA leaves while another may still read its shared memory
}

template <int W>
int launch(const StageParams &p, int nsteps, cudaStream_t s) {
  LineParams q;
  q.p = p;
  q.c = make_sweep64<W>(p.dx, p.eps, p.nx);
  q.nsteps = nsteps;
  int ranks = 1;
  while (ranks < kLineCluster && p.nx > ranks * kLineNodes) ranks *= 2;
  const int count = (p.nx + ranks - 1) / ranks;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ranks);
  cfg.blockDim = dim3((count + 1 + 31) / 32 * 32);
  cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = ranks;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return (int)cudaLaunchKernelEx(&cfg, line64_kernel<W>, q);
}

}  // namespace

int launch_line64(const StageParams &p, int nsteps, void *stream) {
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  return p.weights == W_JP ? launch<W_JP>(p, nsteps, s) : launch<W_ARCLEN>(p, nsteps, s);
}

}  // namespace alw
