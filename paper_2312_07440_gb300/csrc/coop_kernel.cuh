// The fused reweighting kernel with one warp per event (qcd_coop.cuh), for
// g g -> t tbar g g: the arguments, results and reductions of k_reweight
// (kernels.cuh).  Warps take events grid-stride; a warp evaluates the launch's
// distinct kinematics two at a time (points that differ in the coupling only
// share one), then its lanes form r, W' and the cross sections of the points.
//
// Why: one thread (or one lane per helicity slice) per event repeats every
// current for each helicity it does not depend on and spills; its unrolled code
// overflows the instruction cache.  Here the sum takes about half the
// arithmetic, the code is compact loops over tasks, and 8 (FP64) or 16 (FP32, 8
// where the sums of 19 points or more take the room) warps fit an SM.  FP64 is
// bound by the FP64 pipe (92 % busy), FP32 by issue (71 %), shared-memory
// latency and addressing.  Per call with one point, against the
// per-thread kernels: FP64 131,072 events 118 -> 53.1 ms (57.5 before products
// of currents were shared between the three- and four-gluon currents), FP32
// 262,147 events 15.3 -> 3.31 ms, FP16-mixed 65,536 events 3.94 -> 1.13 ms.
//
// CM_STORE_*: instead of summing colours, the lanes write their amplitude
// vectors for the separate tensor-core pass (colour_tc.cuh), one evaluation
// per point.
#pragma once
#include "colour_tc.cuh"
#include "kernels.cuh"
#include "qcd_coop.cuh"

namespace rw {
namespace coop {

template <class T>
__device__ __forceinline__ T quad_sum(T v) {  // over the lanes of a group of four (particles 2..5)
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}
__device__ __forceinline__ df shfl_df(df v, int o) {
  return {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}
__device__ __forceinline__ df quad_sum(df v) {
  v = df_add(v, shfl_df(v, 1));
  return df_add(v, shfl_df(v, 2));
}

// shell_scale_near (qcd.cuh) over the lanes of a group, for the groups that are
// live: their FP32 root; x as it was for the others.  (Out of line as there;
// 262,147 events FP32: 3.332 ms in line, 3.316 out of line, as without it.)
__device__ __noinline__ float scale_near(float p2, float m2, float gap, float x, bool live) {
  const float m = sqrtf(m2);
  if (live) x = 1.0f;
#pragma unroll 1
  for (int it = 0; it < 40; ++it) {
    const float k = x * x * p2, r = rsqrtf(m2 + k);
    const float f = quad_sum(__fdividef(k, fmaf(m2 + k, r, m))) - gap, d = quad_sum(x * p2 * r);
    float step = __fdividef(f, d);
    if (x - step <= 0.0f) step = 0.5f * x;
    if (live) x -= step;
    live = live && fabsf(step) > 1e-6f * x;
    if (!__any_sync(0xffffffffu, live)) break;
  }
  return x;
}

// Momenta of up to two evaluations from the event's (W.u.p), moved onto the
// mass shell where the point's top mass differs: the common 3-momentum scale
// by Newton's method in FP32, then two FP64 or one double-float step (compare
// reshuffle_tops in qcd.cuh), particle 2 + (lane & 3) of evaluation
// (lane >> 2) & 1 in each lane.  Returns whether evaluation b's masses fit, in
// bit b.
template <class R>
__device__ __forceinline__ unsigned momenta(Warp<R>& W, int lane, const PointDev& pt0, const PointDev& pt1, int nb) {
  using mom = typename Warp<R>::mom;
  const int part = lane & 3, b = (lane >> 2) & 1;
  const double mt = b ? pt1.m_t : pt0.m_t;
  const bool moved = (b ? pt1.reshuffle : pt0.reshuffle) != 0;
  mom p[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) p[m] = W.u.p[4 * (2 + part) + m];
  mom scale, energy;
  bool fits = true;
  if (pt0.reshuffle || pt1.reshuffle) {
    mom p2, etot, mi2;
    float etf, pf, m2f, gap;
    if constexpr (sizeof(R) == 8) {
      p2 = p[1] * p[1] + p[2] * p[2] + p[3] * p[3];
      etot = quad_sum(p[0]);
      mi2 = part < 2 ? mt * mt : 0.0;
      fits = 2.0 * mt < etot;
      etf = float(etot);
      pf = float(p2);
      m2f = float(mi2);
      gap = float(etot - 2.0 * mt);
    } else {
      p2 = df_norm3(p);
      etot = quad_sum(p[0]);
      const df mtd = df_from_double(mt);
      mi2 = part < 2 ? df_mul(mtd, mtd) : df{0.0f, 0.0f};
      gap = df_sub(etot, df_scale(mtd, 2.0f)).hi;
      fits = gap > 0.0f;
      etf = etot.hi;
      pf = p2.hi;
      m2f = mi2.hi;
    }
    // a lane's group stops by itself, so an evaluation does not depend on its neighbour in the warp
    float xf = 1.0f, slope = 0.0f;
    bool live = fits && moved;
    for (int it = 0; it < 40; ++it) {
      const float r = rsqrtf(m2f + xf * xf * pf);
      const float f = quad_sum((m2f + xf * xf * pf) * r) - etf, d = quad_sum(xf * pf * r);
      float step = __fdividef(f, d);
      if (xf - step <= 0.0f) step = 0.5f * xf;
      if (live) {
        xf -= step;
        slope = d;
      }
      live = live && fabsf(step) > 1e-6f * xf;  // the next step would be below FP32's precision
      if (!__any_sync(0xffffffffu, live)) break;
    }
    // near the pair threshold in kinetic energies, as shell_scale (qcd.cuh)
    live = fits && moved && etf > 4.0f * slope * xf;
    if (__any_sync(0xffffffffu, live)) xf = scale_near(pf, m2f, gap, xf, live);
    if constexpr (sizeof(R) == 8) {
      double xi = xf, e = 0.0;
#pragma unroll
      for (int it = 0; it < 2; ++it) {
        e = sqrt(mi2 + xi * xi * p2);
        const double xp = xi * p2 / e;
        const double xn = xi - (quad_sum(e) - etot) / quad_sum(xp);
        if (it == 1) e += (xn - xi) * (xn + xi) * p2 / (2.0 * e);
        xi = xn;
      }
      scale = xi;
      energy = e;
    } else {
      const df a = df_mul(df_two_prod(xf, xf), p2);
      df e = df_sqrt(part < 2 ? df_add(mi2, a) : a);
      const df f = df_sub(quad_sum(e), etot);
      const float d = quad_sum(xf * pf / e.hi);
      const float corr = -f.hi / d;
      scale = df_fast_two_sum(xf, corr);
      energy = df_add_f(e, corr * (2.0f * xf + corr) * pf / (2.0f * e.hi));
    }
  }
  if (lane < 8 && b < nb) {
    mom* q = W.u.q[b] + 4 * (2 + part);
    q[0] = moved && fits ? energy : p[0];
#pragma unroll
    for (int m = 1; m < 4; ++m) {
      mom x;
      if constexpr (sizeof(R) == 8)
        x = scale * p[m];
      else
        x = df_mul(scale, p[m]);
      q[m] = moved && fits ? x : p[m];
    }
  } else if (lane >= 16 && ((lane >> 3) & 1) < nb) {  // the incoming momenta
    W.u.q[(lane >> 3) & 1][lane & 7] = W.u.p[lane & 7];
  }
  const unsigned v = __ballot_sync(0xffffffffu, fits || !moved);
  return (v & 1u) | ((v >> 3) & 2u);
}

template <class R, int CM>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 2 : 1) k_coop(const __grid_constant__ RwArgs a) {
  constexpr bool STORE = CM != CM_FMA;
  extern __shared__ __align__(16) unsigned char rw_dyn_bytes[];
  __shared__ unsigned words[N_WORDS];
  __shared__ double2 red[32];
  __shared__ int is_last;
  const int tid = threadIdx.x, nw = blockDim.x >> 5, warp = tid >> 5, lane = tid & 31;
  const int P = a.P, stride = P + 1;
  Warp<R>& W = reinterpret_cast<Warp<R>*>(rw_dyn_bytes)[warp];
  double2* sacc = reinterpret_cast<double2*>(rw_dyn_bytes + nw * sizeof(Warp<R>));
  double* sums = reinterpret_cast<double*>(sacc + nw * stride) + warp * stride;  // stripped sum of each class
  for (int i = tid; i < N_WORDS; i += blockDim.x) words[i] = TASK_WORDS[i];
  if constexpr (!STORE)
    for (int i = tid; i < nw * stride; i += blockDim.x) sacc[i] = make_double2(0.0, 0.0);
  __syncthreads();
  const int nk = a.me_only ? 1 : STORE ? P + 1 : a.nkin;
  const long long E = a.E, ldo = a.ldo ? a.ldo : a.E;
  const int lt = lane >> 4, lb = (lane >> 3) & 1, h1 = (lane >> 2) & 1, h2 = (lane >> 1) & 1, h3 = lane & 1;
  unsigned long long nbad = 0;
  for (long long base = (long long)blockIdx.x * nw; base < E; base += (long long)gridDim.x * nw) {
    const bool valid = base + warp < E;
    const long long ev = valid ? base + warp : E - 1;
#pragma unroll 1
    for (int k = 0; k < nk; k += NBATCH) {
      // FP32: the warps of a block start a batch together, so they stream
      // through the same instructions (its code is several times the
      // instruction cache next to the schedulers); left to themselves they
      // drift apart and a third of the issue slots wait for instructions
      // (262,147 events: 4.16 -> 3.36 ms; a barrier per phase: 3.57 ms)
      if constexpr (sizeof(R) == 4) __syncthreads();
      const int nb = min(NBATCH, nk - k);
      const int j0 = STORE || a.me_only ? k : a.kin_rep[k];
      const int j1 = nb < 2 ? j0 : STORE ? k + 1 : a.kin_rep[k + 1];
      // the previous batch's readers of the memory written below are done
      __syncwarp();
      if (lane < 24) load_mom(W.u.p[lane], __ldg(a.mom + (long long)lane * a.ld + ev));
      __syncwarp();
      const unsigned fits = momenta<R>(W, lane, a.pt[j0], a.pt[j1], nb);
      __syncwarp();
      const int eb = lane >> 4, el = lane & 15;
      const double m = eb ? a.pt[j1].m_t : a.pt[j0].m_t;
      if (eb < nb) W.externals(eb, el, m);
      __syncwarp();
      if (eb < nb) W.subsets(eb, el, m);
      __syncwarp();
#pragma unroll 1
      for (int t = lane; t < nb * N_J2; t += 32) {
        const int b = t >= N_J2;
        W.two_gluons(b, t - b * N_J2, words[TW_J2 + t - b * N_J2]);
      }
      __syncwarp();
#pragma unroll 1
      for (int t = lane; t < nb * N_DOT; t += 32) {
        const int b = t >= N_DOT, i = t - b * N_DOT;
        W.product(b, i, words[TW_DOT + i]);
      }
      __syncwarp();
#pragma unroll 1
      for (int t = lane; t < nb * N_J3; t += 32) {
        const int b = t >= N_J3, i = t - b * N_J3;
        W.three_gluons(b, i, words[TW_J3 + i], words[TW_J3B + i]);
      }
      __syncwarp();
#pragma unroll 1
      for (int t = lane; t < nb * N_J4; t += 32) {
        const int b = t >= N_J4, i = t - b * N_J4;
        W.four_gluons(b, i, words[TW_J4 + i], words[TW_J4B + i], words[TW_J4C + i], words[TW_J4D + i]);
      }
#pragma unroll 1
      for (int b = 0; b < nb; ++b) {
        cx<R> A[24];
        __syncwarp();
        if (lane < N_X1) W.one_gluon(b, lane, words[TW_X1 + lane]);
        W.start(b, lane, A);
        __syncwarp();
#pragma unroll 1
        for (int t = lane; t < 96; t += 32) W.work_r3(b, t, words[TW_R3 + t]);
        __syncwarp();
        add_r3_0<R>(W, lt, lb, h1, h2, h3, A);
        __syncwarp();
#pragma unroll 1
        for (int t = lane; t < N_R3 - 96; t += 32) W.work_r3(b, t, words[TW_R3 + 96 + t]);
        __syncwarp();
        add_r3_1<R>(W, lt, lb, h1, h2, h3, A);
        __syncwarp();
#pragma unroll 1
        for (int t = lane; t < 96; t += 32) W.work_y(b, t, words[TW_Y + t]);
        __syncwarp();
        add_y_0<R>(W, lt, lb, h1, h2, h3, A);
        __syncwarp();
#pragma unroll 1
        for (int t = lane; t < N_Y - 96; t += 32) W.work_y(b, t, words[TW_Y + 96 + t]);
        __syncwarp();
        add_y_1<R>(W, lt, lb, h1, h2, h3, A);
        __syncwarp();
#pragma unroll 1
        for (int t = lane; t < 96; t += 32) W.work_x2(b, t, words[TW_X2 + t]);
        __syncwarp();
        add_x2_0<R>(W, lt, lb, h1, h2, h3, A);
        __syncwarp();
#pragma unroll 1
        for (int t = lane; t < N_X2 - 96; t += 32) W.work_x2(b, t, words[TW_X2 + 96 + t]);
        __syncwarp();
        add_x2_1<R>(W, lt, lb, h1, h2, h3, A);
        const bool in = (fits >> b) & 1u;
        if constexpr (STORE) {
          constexpr int SLOTS = 32;
          const DeferLayout L(P + 1, a.defer_ld, 24, SLOTS);
          ColourSink<24, CM> sk{reinterpret_cast<uint4*>(a.defer + L.j16_off),
                                reinterpret_cast<short*>(a.defer + L.ex_off), L.ld, valid ? ev : -1, (k + b) * SLOTS + lane};
          sk.put(A);
          if (lane == 0 && valid) (a.defer + L.ins_off)[(long long)(k + b) * L.ld + ev] = in ? 1 : 0;
        } else {
          double s = 2.0 * (double)colour_sum<R>(A);  // x2: the helicity flip
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
          if (lane == 0) sums[k + b] = in ? s : 0.0;
        }
      }
    }
    if constexpr (!STORE) {
      __syncwarp();
      if (!valid) continue;
      const double me0 = sums[0] * a.pt[0].cscale;  // not moved, so never outside
      if (a.me_only) {
        if (lane == 0) a.me0[ev] = me0;
        continue;
      }
      const bool ok = isfinite(me0) && me0 != 0.0;
      const double w = __ldg(a.w + ev);
      if (lane == 0) {
        if (!ok) ++nbad;
        if (a.me0) a.me0[ev] = me0;
      }
      for (int j = lane; j <= P; j += 32) {
        double x = w;
        if (j < P) {
          const double me = with_coupling<true>(sums[a.kin_of[j + 1]], a.pt[j + 1].cscale);
          const double r = ok ? me / me0 : 0.0;
          x = ok ? r * w : 0.0;
          const long long o = (long long)j * ldo + ev;
          if (a.me_pts) a.me_pts[o] = me;
          if (a.ratio) a.ratio[o] = r;
          if (a.wnew) a.wnew[o] = x;
        }
        double2 v = sacc[warp * stride + j];  // slot j is always this lane's
        two_sum_acc(v.x, v.y, x, 0.0);
        sacc[warp * stride + j] = v;
      }
    }
  }
  if constexpr (!STORE)
    if (!a.me_only) reduce_sums(a, sacc, nbad, red, is_last);
}

}  // namespace coop
}  // namespace rw
