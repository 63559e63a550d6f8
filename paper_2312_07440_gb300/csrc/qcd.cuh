// Per-event set-up for g g -> t tbar + n g: external wavefunctions of both
// helicities (in the working precision R, cancellation-free formulas) and the
// propagator invariants, whose dot products are formed at ~double precision
// -- FP64 in FP64 mode, double-float (dfloat.cuh) in the FP32 modes -- so
// that FP32 mode never forms p^2 - m^2 by cancellation in single precision,
// before the reciprocals are taken in R.
#pragma once
#include "dfloat.cuh"
#include "helas.cuh"

namespace rw {

template <class R, int NG>
struct QcdExt {
  cv<R> eps[NG][2];  // gluon polarisations (conjugated for outgoing gluons)
  sp<R> ub[2];       // top: ubar(p3, lambda)
  sp<R> v[2];        // antitop: v(p4, lambda)
};

template <class R, int NG>
struct QcdKin {
  R P[1 << NG][4];   // summed incoming momentum of each gluon subset
  R cg[1 << NG];     // -1/K^2  (3-gluon vertex + gluon propagator)
  R c4[1 << NG];     // +1/K^2  (4-gluon vertex + gluon propagator)
  R qc[1 << NG][4];  // c (K - p4), c = -1/((K - p4)^2 - m^2)  (top propagator)
  R mc[1 << NG];     // c m
};

// Store for the gluon currents of three or more gluons (generated code puts
// each once and gets it at every use).  Registers: a plain array indexed by
// constants.  Shared memory (FP32): this thread's slice of the dynamic shared
// memory, [slot][half][thread] float4 so a warp's accesses are conflict-free;
// the accesses are volatile, so the compiler neither keeps a stored current
// in registers nor moves a read above the write of its slot.  The kernel
// places its own shared data after NS * 32 * blockDim.x bytes.
template <class R, int NS, bool SMEM>
struct JStore {
  cv<R> v[NS > 0 ? NS : 1];
  __device__ __forceinline__ void put(int s, const cv<R>& x) { v[s] = x; }
  __device__ __forceinline__ cv<R> get(int s) const { return v[s]; }
};

template <int NS>
struct JStore<float, NS, true> {
  unsigned base, stride;
  __device__ __forceinline__ JStore() {
    extern __shared__ float4 rw_dyn_smem[];
    base = (unsigned)__cvta_generic_to_shared(rw_dyn_smem + threadIdx.x);
    stride = 16u * blockDim.x;
  }
  __device__ __forceinline__ void put(int s, const cv<float>& x) const {
    const unsigned a = base + 2u * (unsigned)s * stride;
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(x.c[0].r), "f"(x.c[0].i), "f"(x.c[1].r),
                 "f"(x.c[1].i));
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a + stride), "f"(x.c[2].r), "f"(x.c[2].i),
                 "f"(x.c[3].r), "f"(x.c[3].i));
  }
  __device__ __forceinline__ cv<float> get(int s) const {
    const unsigned a = base + 2u * (unsigned)s * stride;
    cv<float> x;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(x.c[0].r), "=f"(x.c[0].i), "=f"(x.c[1].r), "=f"(x.c[1].i)
                 : "r"(a));
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(x.c[2].r), "=f"(x.c[2].i), "=f"(x.c[3].r), "=f"(x.c[3].i)
                 : "r"(a + stride));
    return x;
  }
};

// particle index of gluon g on the top line: 0, 1 incoming, then 4, 5, ...
__host__ __device__ constexpr int gluon_particle(int g) { return g < 2 ? g : g + 2; }

__device__ __forceinline__ double dot4(const double (&a)[4], const double (&b)[4]) {
  return a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3];
}

// Double-double arithmetic for the FP64 set-up's invariants of several
// gluons: Knuth's TwoSum, the FMA form of TwoProduct, one rounding at the end.
// A gluon propagator 1/K^2 of an incoming and an outgoing gluon near the beam
// axis has K^2 ~ 1e2-1e3 GeV^2 while k_i.k_j-style products are ~1e6 GeV^2,
// so K^2 formed in plain FP64 carries relative errors of ~1e-13, which the
// largest-|M|^2 events (near-collinear emission) pass on to |M|^2.
struct dd {
  double hi, lo;
};

__device__ __forceinline__ dd dd_two_sum(double a, double b) {
  const double s = a + b;
  const double bp = s - a;
  return {s, (a - (s - bp)) + (b - bp)};
}

__device__ __forceinline__ dd dd_add(dd x, double y) {
  const dd s = dd_two_sum(x.hi, y);
  const double lo = s.lo + x.lo;
  const double h = s.hi + lo;
  return {h, lo - (h - s.hi)};
}

__device__ __forceinline__ dd dd_add(dd x, dd y) {
  const dd s = dd_two_sum(x.hi, y.hi);
  const double lo = s.lo + (x.lo + y.lo);
  const double h = s.hi + lo;
  return {h, lo - (h - s.hi)};
}

// Minkowski product a.b carried to double-double: every product exact as
// p + e (FMA), the p added by TwoSum
__device__ __forceinline__ dd dd_dot4(const double (&a)[4], const double (&b)[4]) {
  dd acc = {0.0, 0.0};
  double small = 0.0;
#pragma unroll
  for (int m4 = 0; m4 < 4; ++m4) {
    const double x = m4 ? -a[m4] : a[m4];
    const double q = x * b[m4];
    small += fma(x, b[m4], -q);
    acc = dd_add(acc, q);
  }
  acc.lo += small;
  return acc;
}

// s + c += hi + lo with the rounding error of the leading sum kept in c
__device__ __forceinline__ void comp_add(double& s, double& c, double hi, double lo) {
  const dd t = dd_two_sum(s, hi);
  s = t.hi;
  c += t.lo + lo;
}
__device__ __forceinline__ void comp_add(float& s, float& c, float hi, float lo) {
  const df t = df_two_sum(s, hi);
  s = t.hi;
  c = __fadd_rn(c, __fadd_rn(t.lo, lo));
}

// K^2 and (K - p4)^2 - m^2 of every gluon subset K = sum_{i in S} k_i from the
// momenta themselves (no mass-shell assumption), each rounded once from a
// compensated sum of double-double products: K^2 = sum_i k_i.k_i +
// 2 sum_{i<j} k_i.k_j and (K - p4)^2 - m^2 = K^2 - 2 sum_i k_i.p4 +
// (p4.p4 - m^2), with the pairwise products formed once and each subset's sums
// continued from those of the subset without its first gluon.  Out of line:
// its temporaries stay out of the amplitude code's register allocation.
template <int NG>
__device__ __noinline__ void subset_invariants_dd(const double (&k)[NG][4], const double (&p4)[4], double m,
                                                  double (&K2)[1 << NG], double (&den)[1 << NG]) {
  dd kk[NG], kp[NG], d[NG][NG];
#pragma unroll
  for (int i = 0; i < NG; ++i) {
    kk[i] = dd_dot4(k[i], k[i]);
    kp[i] = dd_dot4(k[i], p4);
#pragma unroll
    for (int j = i + 1; j < NG; ++j) d[i][j] = dd_dot4(k[i], k[j]);
  }
  dd pm = dd_dot4(p4, p4);
  const double m2 = m * m;
  pm = dd_add(pm, dd{-m2, -fma(m, m, -m2)});
  constexpr int FULL = (1 << NG) - 1;
  dd sk[1 << NG], sq[1 << NG];  // K^2; -2 K.p4 + p4^2 - m^2
  sk[0] = {0.0, 0.0};
  sq[0] = pm;
#pragma unroll
  for (int msk = 1; msk <= FULL; ++msk) {
    const int rest = msk & (msk - 1);
    int i = 0;
#pragma unroll
    for (int g = NG - 1; g >= 0; --g)
      if ((msk >> g) & 1) i = g;
    dd s = kk[i];
    if (rest) {
      comp_add(s.hi, s.lo, sk[rest].hi, sk[rest].lo);
#pragma unroll
      for (int j = i + 1; j < NG; ++j)
        if ((msk >> j) & 1) comp_add(s.hi, s.lo, 2.0 * d[i][j].hi, 2.0 * d[i][j].lo);
    }
    sk[msk] = s;
    K2[msk] = s.hi + s.lo;
    if (msk != FULL) {
      dd q = sq[rest];
      comp_add(q.hi, q.lo, -2.0 * kp[i].hi, -2.0 * kp[i].lo);
      sq[msk] = q;
      comp_add(s.hi, s.lo, q.hi, q.lo);
      den[msk] = s.hi + s.lo;
    } else {
      den[msk] = 0.0;
    }
  }
}

template <class R, int NG, int NEXT>
__device__ __forceinline__ void qcd_setup(const double (&p)[NEXT][4], double m, QcdExt<R, NG>& X,
                                          QcdKin<R, NG>& Kn) {
  static_assert(NEXT == NG + 2, "t tbar + NG gluons");
  double k[NG][4];
  R kw[NG][4];  // incoming gluon momenta in the working precision
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    const int ip = gluon_particle(g);
    const double s = ip < 2 ? 1.0 : -1.0;
    R kr[4];
#pragma unroll
    for (int m4 = 0; m4 < 4; ++m4) {
      k[g][m4] = s * p[ip][m4];
      kr[m4] = R(p[ip][m4]);
      kw[g][m4] = ip < 2 ? kr[m4] : -kr[m4];
    }
    polvec<R>(kr, ip >= 2, X.eps[g]);
  }
  {
    R p3[4], p4[4];
#pragma unroll
    for (int m4 = 0; m4 < 4; ++m4) {
      p3[m4] = R(p[2][m4]);
      p4[m4] = R(p[3][m4]);
    }
    ubar_out<R>(p3, R(m), X.ub);
    v_out<R>(p4, R(m), X.v);
  }
  // Invariants: the dot products, where cancellation happens, in FP64 (two
  // or three gluons: double-double, see subset_invariants_dd); the
  // reciprocals in the working precision.
  [[maybe_unused]] double K2dd[1 << NG], dendd[1 << NG];
  if constexpr (NG >= 3) subset_invariants_dd<NG>(k, p[3], m, K2dd, dendd);
  double d[NG][NG];
#pragma unroll
  for (int i = 0; i < NG; ++i)
#pragma unroll
    for (int j = i + 1; j < NG; ++j) d[i][j] = dot4(k[i], k[j]);  // gluons are massless: k_i^2 = 0
  constexpr int FULL = (1 << NG) - 1;
#pragma unroll
  for (int msk = 1; msk <= FULL; ++msk) {
    double P[4] = {0.0, 0.0, 0.0, 0.0};
    double K2 = 0.0;
    int cnt = 0;
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      if (!((msk >> i) & 1)) continue;
      ++cnt;
#pragma unroll
      for (int m4 = 0; m4 < 4; ++m4) P[m4] += k[i][m4];
#pragma unroll
      for (int j = i + 1; j < NG; ++j)
        if ((msk >> j) & 1) K2 += 2.0 * d[i][j];
    }
    // vertex momenta: subset sums in the working precision
#pragma unroll
    for (int m4 = 0; m4 < 4; ++m4) {
      R v = R(0);
#pragma unroll
      for (int i = 0; i < NG; ++i)
        if ((msk >> i) & 1) v += kw[i][m4];
      Kn.P[msk][m4] = v;
    }
    if constexpr (NG >= 3) K2 = K2dd[msk];
    if (cnt >= 2) {
      const R inv = R(1) / R(K2);
      Kn.cg[msk] = -inv;
      Kn.c4[msk] = inv;
    } else {
      Kn.cg[msk] = R(0);
      Kn.c4[msk] = R(0);
    }
    if (msk != FULL) {
      // (K - p4)^2 - m^2 = K^2 - 2 K.p4  (p4^2 = m^2); several gluons: as above
      double den;
      if constexpr (NG >= 3)
        den = dendd[msk];
      else
        den = K2 - 2.0 * dot4(P, p[3]);
      const R c = R(-1) / R(den);
#pragma unroll
      for (int m4 = 0; m4 < 4; ++m4) Kn.qc[msk][m4] = c * R(P[m4] - p[3][m4]);
      Kn.mc[msk] = c * R(m);
    } else {
#pragma unroll
      for (int m4 = 0; m4 < 4; ++m4) Kn.qc[msk][m4] = R(0);
      Kn.mc[msk] = R(0);
    }
  }
}

// FP32 root of sum_i sqrt(m_i^2 + x^2 p_i^2) = E (m_i = m for the first two
// particles, else 0) by Newton's method from x = 1: the step that would move x
// by less than 1e-6 is the last, the next being below FP32's resolution.  One
// approximate reciprocal square root per particle.
//
// shell_scale takes the energies themselves, whose sum is rounded at E: x sees
// that as rounding E / (x dE/dx), and where it is more than a few 1e-7, near
// the pair threshold, shell_scale_near solves the same equation in kinetic
// energies x^2 p_i^2 / (e_i + m_i), whose sum is gap = E - 2 m.  Nothing
// cancels there, so its root is good to a few 1e-7 at any distance.  (For every
// event it costs g g -> t tbar g, 131,072 x 64 points, 6.63 -> 6.70 ms.)  The
// sum is convex: a step beyond x = 0 comes from rounding far above the root.
// (The second loop out of line, its array by value: interpolation of g g ->
// t tbar g, 262,144 events, 2.444 ms in line, 2.411 out of line.)
template <int N>
struct Squares {
  float p2[N];
};
template <int N>
__device__ __noinline__ float shell_scale_near(const Squares<N> s, float m, float gap) {
  const float(&p2)[N] = s.p2;
  const float m2 = m * m;
  float x = 1.0f;
#pragma unroll 1
  for (int it = 0; it < 40; ++it) {
    float f = -gap, df = 0.0f;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const float a = x * p2[i], k = x * a, e2 = i < 2 ? k + m2 : k, r = rsqrtf(e2);
      f += __fdividef(k, fmaf(e2, r, i < 2 ? m : 0.0f));
      df = fmaf(a, r, df);
    }
    float step = __fdividef(f, df);
    if (x - step <= 0.0f) step = 0.5f * x;
    x -= step;
    if (fabsf(step) <= 1e-6f * x) break;
  }
  return x;
}
template <int N>
__device__ __forceinline__ float shell_scale(const float (&p2)[N], float m, float m2, float etot, float gap) {
  float x = 1.0f, df = 0.0f;
  for (int it = 0; it < 40; ++it) {
    float f = -etot;
    df = 0.0f;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const float a = x * p2[i], e2 = fmaf(x, a, i < 2 ? m2 : 0.0f), r = rsqrtf(e2);
      f = fmaf(e2, r, f);
      df = fmaf(a, r, df);
    }
    float step = __fdividef(f, df);
    if (x - step <= 0.0f) step = 0.5f * x;
    x -= step;
    if (fabsf(step) <= 1e-6f * x) break;
  }
  if (etot > 4.0f * df * x) {
    Squares<N> s;
#pragma unroll
    for (int i = 0; i < N; ++i) s.p2[i] = p2[i];
    x = shell_scale_near(s, m, gap);
  }
  return x;
}

// The pair's closed form (reshuffle_tops below) in any frame: out of line, as
// the centre-of-mass frame needs the short one only (g g -> t tbar FP64,
// 1,048,576 events: 5.62 ms in line, 5.54 ms out of line).
template <class T>
struct Pair {
  T xi, e0, e1;  // common scale, the two energies
};
static __device__ __noinline__ Pair<double> pair_any_frame(double a, double b, double m, double E, double D) {
  const double s = a + b, h = (a - b) / E, mh = 2.0 * m * h;
  const double x = D / (s + sqrt(fma(4.0 * a, b, mh * mh))), c = 0.5 * x * h;
  // far from the centre-of-mass frame the smaller energy is not a difference
  return {sqrt(x), c < -0.25 * E ? sqrt(fma(x, a, m * m)) : fma(0.5, E, c),
          c > 0.25 * E ? sqrt(fma(x, b, m * m)) : fma(0.5, E, -c)};
}
static __device__ __noinline__ Pair<df> pair_any_frame(df a, df b, df m, df E, df D) {
  const df s = df_add(a, b), h = df_div(df_sub(a, b), E), r = df_scale(df_mul(m, df_div(h, s)), 2.0f);
  const df root = df_sqrt(df_add(df_scale(df_mul(df_div(a, s), df_div(b, s)), 4.0f), df_mul(r, r)));
  const df x = df_div(df_div(D, s), df_add_f(root, 1.0f)), c = df_scale(df_mul(x, h), 0.5f), half = df_scale(E, 0.5f);
  const df m2 = df_mul(m, m);
  return {df_sqrt(x), c.hi < -0.25f * E.hi ? df_sqrt(df_add(m2, df_mul(x, a))) : df_add(half, c),
          c.hi > 0.25f * E.hi ? df_sqrt(df_add(m2, df_mul(x, b))) : df_sub(half, c)};
}

// Move the outgoing particles (2..NEXT-1) onto the mass shells m_t (tops),
// 0 (gluons) at fixed partonic energy: p_i -> xi p_i (3-momenta) with
// sum_i sqrt(m_i^2 + xi^2 |p_i|^2) = sum_i E_i.
// Returns false when the new masses do not fit (sum m_i >= E).
//
// The pair alone has a closed form, to rounding at any distance from the
// threshold: with a, b the |p_i|^2, s = a + b, d = a - b and
// D = (E - 2 m)(E + 2 m), the energies are (E +- xi^2 d / E) / 2 and
// xi^2 = D / (s + sqrt(4 a b + (2 m d / E)^2)).  In the centre-of-mass frame d
// is rounding and the root is s.  (Against an FP32 root and one FP64 or
// double-float step, which lost the digits near the threshold and all of them
// within 1e-7 of it: 1,048,576 events FP64 5.60 -> 5.54 ms, FP32 339 -> 333 us.)
//
// With gluons: the FP32 root, then one step of third order in FP64
// (Chebyshev's), the energies expanded to second order around the root it
// starts from, so one square root per particle serves both.
template <int NEXT>
__device__ __forceinline__ bool reshuffle_tops(const double (&p)[NEXT][4], double mt, double (&q)[NEXT][4]) {
  constexpr int N = NEXT - 2;
  double etot = 0.0, p2[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const double (&v)[4] = p[i + 2];
    etot += v[0];
    p2[i] = v[1] * v[1] + v[2] * v[2] + v[3] * v[3];
  }
#pragma unroll
  for (int i = 0; i < NEXT; ++i)
#pragma unroll
    for (int m4 = 0; m4 < 4; ++m4) q[i][m4] = p[i][m4];
  if (!(2.0 * mt < etot)) return false;
  const double mt2 = mt * mt;
  if constexpr (N == 2) {
    const double lo = dd_two_sum(p[2][0], p[3][0]).lo;  // the energy's rounding counts in E - 2 m
    const double D = ((etot - 2.0 * mt) + lo) * (etot + 2.0 * mt);
    const double s = p2[0] + p2[1], d = p2[0] - p2[1];
    double xi;
    if ((__double2hiint(d) & 0x7FFFFFFF) + (30 << 20) < __double2hiint(s)) {  // |d| < 2^-30 s: d^2 vanishes in xi
      const double s2 = s + s, r = rsqrt(s2 * D);
      xi = D * r;
      xi = fma(0.5 * r, fma(-s2 * xi, xi, D), xi);
      const double c = 0.5 * double(__fdividef(float(xi * xi * d), float(etot)));
      q[2][0] = fma(0.5, etot, c);
      q[3][0] = fma(0.5, etot, -c);
    } else {
      const Pair<double> v = pair_any_frame(p2[0], p2[1], mt, etot, D);
      xi = v.xi;
      q[2][0] = v.e0;
      q[3][0] = v.e1;
    }
#pragma unroll
    for (int i = 2; i < NEXT; ++i)
#pragma unroll
      for (int m4 = 1; m4 < 4; ++m4) q[i][m4] = xi * p[i][m4];
  } else {
    float pf[N];
#pragma unroll
    for (int i = 0; i < N; ++i) pf[i] = float(p2[i]);
    const double xi = shell_scale(pf, float(mt), float(mt2), float(etot), float(etot - 2.0 * mt));
    double f = -etot, f1 = 0.0, f2 = 0.0, e[N], d1[N], d2[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const double a = xi * p2[i], x = fma(xi, a, i < 2 ? mt2 : 0.0), r = rsqrt(x);
      double s = x * r;
      s = fma(0.5 * r, fma(-s, s, x), s);  // the square root to rounding
      e[i] = s;
      d1[i] = a * r;                              // de/dxi
      d2[i] = i < 2 ? mt2 * p2[i] * (r * r * r) : 0.0;  // d2e/dxi2
      f += e[i];
      f1 += d1[i];
      f2 += d2[i];
    }
    const double i1 = 1.0 / f1, s0 = -f * i1;
    const double dx = s0 * fma(-0.5 * s0, f2 * i1, 1.0);
    const double xn = xi + dx;
#pragma unroll
    for (int i = 0; i < N; ++i) {
#pragma unroll
      for (int m4 = 1; m4 < 4; ++m4) q[i + 2][m4] = xn * p[i + 2][m4];
      q[i + 2][0] = fma(dx, fma(0.5 * dx, d2[i], d1[i]), e[i]);
    }
  }
  return true;
}

// FP32 modes: the same set-up from double-float momenta (the split of the
// FP64 inputs); invariants in double-float, everything else in float.  The
// set-up is a large part of the smaller processes' FP32 instructions: forming
// each subset's sums from a smaller subset's by one compensated addition per
// term, with one approximate root per particle and step in the reshuffle,
// took g g -> t tbar (1,048,576 events) from 490 to 375 us and g g -> t tbar g
// (131,072 x 64 points) from 9.28 to 8.19 ms.
template <class R, int NG, int NEXT>
__device__ __forceinline__ void qcd_setup(const df (&p)[NEXT][4], double m, QcdExt<R, NG>& X, QcdKin<R, NG>& Kn) {
  static_assert(NEXT == NG + 2, "t tbar + NG gluons");
  static_assert(sizeof(R) == 4, "double-float set-up feeds FP32 amplitudes");
  df k[NG][4];
  R kw[NG][4];
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    const int ip = gluon_particle(g);
    R kr[4];
#pragma unroll
    for (int m4 = 0; m4 < 4; ++m4) {
      k[g][m4] = ip < 2 ? p[ip][m4] : df_neg(p[ip][m4]);
      kr[m4] = p[ip][m4].hi;
      kw[g][m4] = ip < 2 ? kr[m4] : -kr[m4];
    }
    polvec<R>(kr, ip >= 2, X.eps[g]);
  }
  {
    R p3[4], p4[4];
#pragma unroll
    for (int m4 = 0; m4 < 4; ++m4) {
      p3[m4] = p[2][m4].hi;
      p4[m4] = p[3][m4].hi;
    }
    ubar_out<R>(p3, R(m), X.ub);
    v_out<R>(p4, R(m), X.v);
  }
  // products in double-float; each subset's sums compensated and continued
  // from those of the subset without its first gluon
  df d[NG][NG], kp[NG];
#pragma unroll
  for (int i = 0; i < NG; ++i) {
    kp[i] = df_scale(df_dot4(k[i], p[3]), -2.0f);  // -2 k_i.p4
#pragma unroll
    for (int j = i + 1; j < NG; ++j) d[i][j] = df_scale(df_dot4(k[i], k[j]), 2.0f);  // 2 k_i.k_j
  }
  constexpr int FULL = (1 << NG) - 1;
  df sk[1 << NG], sq[1 << NG], sp[1 << NG][4];  // K^2; -2 K.p4; K - p4
  sk[0] = sq[0] = {0.0f, 0.0f};
#pragma unroll
  for (int m4 = 0; m4 < 4; ++m4) sp[0][m4] = df_neg(p[3][m4]);
#pragma unroll
  for (int msk = 1; msk <= FULL; ++msk) {
    const int rest = msk & (msk - 1);
    int i = 0, cnt = 0;
#pragma unroll
    for (int g = NG - 1; g >= 0; --g)
      if ((msk >> g) & 1) {
        i = g;
        ++cnt;
      }
    df s = sk[rest];
#pragma unroll
    for (int j = i + 1; j < NG; ++j)
      if ((msk >> j) & 1) {
        if (cnt == 2)
          s = d[i][j];
        else
          comp_add(s.hi, s.lo, d[i][j].hi, d[i][j].lo);
      }
    sk[msk] = s;
#pragma unroll
    for (int m4 = 0; m4 < 4; ++m4) {
      R v = R(0);
#pragma unroll
      for (int g = 0; g < NG; ++g)
        if ((msk >> g) & 1) v += kw[g][m4];
      Kn.P[msk][m4] = v;
    }
    if (cnt >= 2) {
      const R inv = R(1) / (s.hi + s.lo);
      Kn.cg[msk] = -inv;
      Kn.c4[msk] = inv;
    } else {
      Kn.cg[msk] = R(0);
      Kn.c4[msk] = R(0);
    }
    if (msk != FULL) {
      // (K - p4)^2 - m^2 = K^2 - 2 K.p4  (p4^2 = m^2)
      df q = kp[i];
      if (cnt > 1) comp_add(q.hi, q.lo, sq[rest].hi, sq[rest].lo);
      sq[msk] = q;
      if (cnt > 1) comp_add(q.hi, q.lo, s.hi, s.lo);
      const R c = R(-1) / (q.hi + q.lo);
#pragma unroll
      for (int m4 = 0; m4 < 4; ++m4) {
        df x = sp[rest][m4];
        comp_add(x.hi, x.lo, k[i][m4].hi, k[i][m4].lo);
        sp[msk][m4] = x;
        Kn.qc[msk][m4] = c * (x.hi + x.lo);
      }
      Kn.mc[msk] = c * R(m);
    } else {
#pragma unroll
      for (int m4 = 0; m4 < 4; ++m4) Kn.qc[msk][m4] = R(0);
      Kn.mc[msk] = R(0);
    }
  }
}

// FP32 modes: the reshuffle on double-float momenta.  The pair alone in closed
// form as above.  With gluons the FP32 root, then one Newton step in
// double-float (from a few 1e-7 to the double-float precision), energies
// updated to first order, so that the moved momenta are on their mass shells
// to ~1e-14 relative.
template <int NEXT>
__device__ __forceinline__ bool reshuffle_tops(const df (&p)[NEXT][4], double mt, df (&q)[NEXT][4]) {
  df etot = {0.0f, 0.0f}, p2[NEXT];
#pragma unroll
  for (int i = 2; i < NEXT; ++i) {
    etot = i == 2 ? p[i][0] : df_add(etot, p[i][0]);
    p2[i] = df_norm3(p[i]);
  }
#pragma unroll
  for (int i = 0; i < NEXT; ++i)
#pragma unroll
    for (int m4 = 0; m4 < 4; ++m4) q[i][m4] = p[i][m4];
  const df mtd = df_from_double(mt), gap = df_sub(etot, df_scale(mtd, 2.0f));
  if (!(gap.hi > 0.0f)) return false;
  const df mt2 = df_mul(mtd, mtd);
  if constexpr (NEXT == 4) {
    const df D = df_mul(gap, df_add(etot, df_scale(mtd, 2.0f)));
    const df s = df_add(p2[2], p2[3]), d = df_sub(p2[2], p2[3]);
    const df half = df_scale(etot, 0.5f);
    df xi;
    if (fabsf(d.hi) < 3e-8f * s.hi) {  // d^2 vanishes in xi
      const df x = df_scale(df_div(D, s), 0.5f);
      xi = df_sqrt(x);
      const float c = 0.5f * __fdividef(x.hi * d.hi, etot.hi);
      q[2][0] = df_add_f(half, c);
      q[3][0] = df_add_f(half, -c);
    } else {
      const Pair<df> v = pair_any_frame(p2[2], p2[3], mtd, etot, D);
      xi = v.xi;
      q[2][0] = v.e0;
      q[3][0] = v.e1;
    }
#pragma unroll
    for (int i = 2; i < NEXT; ++i)
#pragma unroll
      for (int m4 = 1; m4 < 4; ++m4) q[i][m4] = df_mul(xi, p[i][m4]);
  } else {
    float pf[NEXT - 2];
#pragma unroll
    for (int i = 2; i < NEXT; ++i) pf[i - 2] = p2[i].hi;
    const float xf = shell_scale(pf, mtd.hi, mt2.hi, etot.hi, gap.hi);
    const df xi2 = df_two_prod(xf, xf);
    df e[NEXT];
    float ie[NEXT];
    df f = df_neg(etot);
    float dfx = 0.0f;
#pragma unroll
    for (int i = 2; i < NEXT; ++i) {
      const df a = df_mul(xi2, p2[i]);
      e[i] = df_sqrt(i < 4 ? df_add(mt2, a) : a);
      f = df_add(f, e[i]);
      ie[i] = __fdividef(1.0f, e[i].hi);
      dfx += xf * p2[i].hi * ie[i];
    }
    const float corr = -f.hi / dfx;
    const df xn = df_fast_two_sum(xf, corr);
#pragma unroll
    for (int i = 2; i < NEXT; ++i) {
      // e' = e + (xn^2 - xi^2) |p|^2 / (2 e), exact to O(corr^2)
      e[i] = df_add_f(e[i], corr * (2.0f * xf + corr) * p2[i].hi * (0.5f * ie[i]));
#pragma unroll
      for (int m4 = 1; m4 < 4; ++m4) q[i][m4] = df_mul(xn, p[i][m4]);
      q[i][0] = e[i];
    }
  }
  return true;
}

}  // namespace rw
