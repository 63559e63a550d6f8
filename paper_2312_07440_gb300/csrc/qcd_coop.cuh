// Warp-per-event amplitudes for g g -> t tbar g g (tables and formulas:
// gen/coop_gen.py, gen_coop_gg_ttgg.cuh).
//
// One warp evaluates one event, two evaluations (the original parameters and a
// point, or two points) at a time.  Every set-up constant, gluon current and
// one- or two-gluon spinor is formed once per helicity configuration it depends
// on, dealt out over the lanes as uniform tasks, and kept in shared memory;
// each lane then combines them into the 24 colour-ordered amplitudes of one of
// the 32 helicity configurations (gluon 0 fixed by the helicity flip) and sums
// colours in registers.
//
// The phases are methods of one lane; the kernel separates them by warp
// barriers.  Spinors of the top's side are kept with their chiral halves
// swapped, (u2, u3, u0, u1): a row spinor times a slash is then the column
// code with the vector's y component negated.
#pragma once
#include "dfloat.cuh"
#include "helas.cuh"
#include "qcd.cuh"

namespace rw {
namespace coop {

// (t2, t3, t0, t1) . (s0, s1, s2, s3) of a swapped row spinor and a spinor
template <class R>
__device__ __forceinline__ cx<R> ts_dot(const sp<R>& t, const sp<R>& s) {
  return cmac(t.c[3], s.c[1], cmac(t.c[2], s.c[0], cmac(t.c[1], s.c[3], cmul(t.c[0], s.c[2]))));
}
template <class R>
__device__ __forceinline__ cx<R> ts_mac(const sp<R>& t, const sp<R>& s, cx<R> a) {
  return cmac(t.c[3], s.c[1], cmac(t.c[2], s.c[0], cmac(t.c[1], s.c[3], cmac(t.c[0], s.c[2], a))));
}

}  // namespace coop
}  // namespace rw

#include "gen_coop_gg_ttgg.cuh"

namespace rw {
namespace coop {

// sign flips on the integer pipe: neg is 0 or 0x80000000
__device__ __forceinline__ float flip(float x, unsigned neg) { return __uint_as_float(__float_as_uint(x) ^ neg); }
__device__ __forceinline__ double flip(double x, unsigned neg) {
  return __hiloint2double(__double2hiint(x) ^ (int)neg, __double2loint(x));
}
template <class R>
__device__ __forceinline__ cv<R> flip(cv<R> v, unsigned neg) {
#pragma unroll
  for (int m = 0; m < 4; ++m) v.c[m] = {flip(v.c[m].r, neg), flip(v.c[m].i, neg)};
  return v;
}

template <class R>
struct Acc;  // value carried as (sum, compensation) in the set-up
template <>
struct Acc<double> {
  using mom = double;
  using two = dd;
};
template <>
struct Acc<float> {
  using mom = df;
  using two = df;
};

constexpr int NBATCH = 2;  // evaluations a warp carries at a time

// Objects (complex 4-vectors and spinors), indices within one evaluation ...
constexpr int O_E = 0;    // polarisations: gluon 0, then both of 1, 2, 3
constexpr int O_X0 = 7;   // v (2), ub (2)
constexpr int O_VC = 11;  // ub gamma v, index 2 lt + lb
constexpr int O_J2 = 15;
constexpr int O_J3 = O_J2 + N_J2;
constexpr int N_EV = O_J3 + N_J3;
// ... and shared by the two (the amplitudes of one evaluation at a time)
constexpr int O_X1 = NBATCH * N_EV;  // S(g) (14), T(g) (14)
constexpr int O_WK = O_X1 + N_X1;    // work spinors
constexpr int N_WK = 96;
constexpr int N_OBJ = O_WK + N_WK;

// One warp's shared memory.  An object's 16-byte chunks lie in planes of N_OBJ
// chunks, so lanes reading consecutive objects hit consecutive banks.
template <class R>
struct Warp {
  static constexpr int NCH = (int)(8 * sizeof(R) / 16);  // chunks per object
  using mom = typename Acc<R>::mom;
  using two = typename Acc<R>::two;
  struct Kin {
    R P[16][4];   // summed incoming momentum of each gluon subset
    R qc[16][4];  // c (K - p4), c = -1/((K - p4)^2 - m^2)
    R ik2[16];    // 1/K^2 (two or more gluons)
    R mc[16];     // c m
  };
  struct Setup {
    mom p[24];            // the event's momenta
    mom q[NBATCH][24];    // each evaluation's
    two d[NBATCH][16];    // products of k0..k3, p4 in pairs
  };
  unsigned char obj[NCH * N_OBJ * 16];
  union {
    Setup u;
    cx<R> wv[NBATCH][4][6][8];  // (ub gamma v).J(0 pi): [2 lt + lb][pi][h1 h2 h3]
  };
  Kin kin[NBATCH];

  template <class T>
  __device__ __forceinline__ T get(int i) const {
    T v;
    const unsigned char* a = obj + i * 16;
    if constexpr (sizeof(R) == 4) {
      const float4 x = *reinterpret_cast<const float4*>(a), y = *reinterpret_cast<const float4*>(a + N_OBJ * 16);
      v.c[0] = {x.x, x.y};
      v.c[1] = {x.z, x.w};
      v.c[2] = {y.x, y.y};
      v.c[3] = {y.z, y.w};
    } else {
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const double2 x = *reinterpret_cast<const double2*>(a + m * N_OBJ * 16);
        v.c[m] = {x.x, x.y};
      }
    }
    return v;
  }
  template <class T>
  __device__ __forceinline__ void put(int i, const T& v) {
    unsigned char* a = obj + i * 16;
    if constexpr (sizeof(R) == 4) {
      *reinterpret_cast<float4*>(a) = make_float4(v.c[0].r, v.c[0].i, v.c[1].r, v.c[1].i);
      *reinterpret_cast<float4*>(a + N_OBJ * 16) = make_float4(v.c[2].r, v.c[2].i, v.c[3].r, v.c[3].i);
    } else {
#pragma unroll
      for (int m = 0; m < 4; ++m) *reinterpret_cast<double2*>(a + m * N_OBJ * 16) = make_double2(v.c[m].r, v.c[m].i);
    }
  }
  // the products of currents (complex numbers): in the work spinors' first
  // chunks, which are free until the gluon currents are done
  __device__ __forceinline__ cx<R> prod(int b, int i) const {
    return *reinterpret_cast<const cx<R>*>(obj + (b * N_OBJ + O_WK + i) * 16);
  }
  __device__ __forceinline__ cx<R> prod(int b, int i, unsigned neg) const {
    const cx<R> v = prod(b, i);
    return {flip(v.r, neg), flip(v.i, neg)};
  }
  __device__ __forceinline__ cv<R> vec(int i) const { return get<cv<R>>(i); }
  __device__ __forceinline__ sp<R> spin(int i) const { return get<sp<R>>(i); }
  // the generated code's operands: work spinors, S(g), T(g)
  __device__ __forceinline__ sp<R> w(int i) const { return spin(O_WK + i); }
  __device__ __forceinline__ sp<R> s(int i) const { return spin(O_X1 + i); }
  __device__ __forceinline__ sp<R> t(int i) const { return spin(O_X1 + 14 + i); }

  // --- set-up ---------------------------------------------------------------
  // momentum of one of k0..k3 (incoming), p4 and its sign on the stored momenta
  __device__ __forceinline__ static int particle(int v) { return v < 2 ? v : v == 4 ? 3 : v + 2; }

  // lane 16 b + l of evaluation b: the pair products (l < 15) and the external
  // wavefunctions (l < 6), from u.q
  __device__ __forceinline__ void externals(int b, int l, double m) {
    const mom* q = u.q[b];
    if (l < 15) {
      const int i = l < 5 ? 0 : l < 9 ? 1 : l < 12 ? 2 : l < 14 ? 3 : 4;
      const int j = l - (i == 0 ? 0 : i == 1 ? 4 : i == 2 ? 7 : i == 3 ? 9 : 10);
      mom x[4], y[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        x[c] = q[4 * particle(i) + c];
        y[c] = q[4 * particle(j) + c];
      }
      const bool neg = (i == 2 || i == 3) != (j == 2 || j == 3);  // outgoing gluons enter with k = -p
      two d;
      if constexpr (sizeof(R) == 8) {
        d = dd_dot4(x, y);
        if (neg) d = {-d.hi, -d.lo};
        if (l == 14) {  // p4^2 - m^2
          const double m2 = m * m;
          d = dd_add(d, dd{-m2, -fma(m, m, -m2)});
        }
      } else {
        d = df_dot4(x, y);
        if (neg) d = df_neg(d);
      }
      u.d[b][l] = d;
    }
    const int ob = b * N_EV;
    if (l < 6) {
      const int ip = l < 4 ? particle(l) : l - 2;  // l = 4: top (2), 5: antitop (3)
      R p[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if constexpr (sizeof(R) == 8)
          p[c] = q[4 * ip + c];
        else
          p[c] = q[4 * ip + c].hi;
      }
      if (l < 4) {
        cv<R> e[2];
        polvec<R>(p, l >= 2, e);
        if (l == 0) {
          put(ob + O_E, e[0]);
        } else {
          put(ob + O_E + 2 * l - 1, e[0]);
          put(ob + O_E + 2 * l, e[1]);
        }
      } else {
        // the top's ub (swapped) and the antitop's v from the same pieces:
        // u(+) = (w- chi+, w+ chi+), u(-) = (w+ chi-, w- chi-), ub = (u_R*, u_L*)
        // and v(+) = (w+ chi-, -w- chi-), v(-) = (w- chi+, -w+ chi+)
        cx<R> cp[2], cm[2];
        const R pp = chi_pm(p, cp, cm);
        R wp, wm;
        omegas(p[0], pp, R(m), wp, wm);
        const bool top = l == 4;
        const R f[2] = {top ? wm : wp, top ? wp : wm}, g[2] = {top ? wp : -wm, top ? wm : -wp};
        const unsigned neg = top ? 0x80000000u : 0u;  // conjugated
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          sp<R> x;
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const cx<R> c = top == (h == 0) ? cp[i] : cm[i];
            x.c[i] = {f[h] * c.r, flip(f[h] * c.i, neg)};
            x.c[2 + i] = {g[h] * c.r, flip(g[h] * c.i, neg)};
          }
          put(ob + O_X0 + (top ? 2 : 0) + h, x);
        }
      }
    }
  }

  // lane 16 b + l: the constants of gluon subset l; ub gamma v (l < 4)
  __device__ __forceinline__ void subsets(int b, int l, double m) {
    Kin& K = kin[b];
    if (l > 0) {
      const two* d = u.d[b];
      const mom* q = u.q[b];
      constexpr int at[5] = {0, 5, 9, 12, 14};  // index of (i, i) among the pairs i <= j of five
      R s = R(0), c = R(0);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = i; j < 4; ++j) {
          if (i == j && sizeof(R) == 4) continue;  // FP32 modes: k_i^2 = 0 (and p4^2 = m^2 below)
          const bool in = ((l >> i) & 1) && ((l >> j) & 1);
          const R f = i == j ? R(1) : R(2);
          comp_add(s, c, in ? f * d[at[i] + j - i].hi : R(0), in ? f * d[at[i] + j - i].lo : R(0));
        }
      const R K2 = s + c;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const bool in = (l >> i) & 1;
        comp_add(s, c, in ? R(-2) * d[at[i] + 4 - i].hi : R(0), in ? R(-2) * d[at[i] + 4 - i].lo : R(0));
      }
      if constexpr (sizeof(R) == 8) comp_add(s, c, d[14].hi, d[14].lo);
      const R cc = R(-1) / (s + c);  // unused for the full set
      K.ik2[l] = R(1) / K2;          // unused for one gluon
      K.mc[l] = cc * R(m);
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        R P = R(0), hi = R(0), lo = R(0);
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          const mom y = q[4 * particle(g) + x];
          const bool in = (l >> g) & 1;
          if constexpr (sizeof(R) == 8) {
            const R k = g < 2 ? y : -y;
            P += in ? k : R(0);
          } else {
            const R kh = g < 2 ? y.hi : -y.hi, kl = g < 2 ? y.lo : -y.lo;
            P += in ? kh : R(0);
            comp_add(hi, lo, in ? kh : R(0), in ? kl : R(0));
          }
        }
        K.P[l][x] = P;
        const mom y = q[12 + x];
        if constexpr (sizeof(R) == 8) {
          K.qc[l][x] = cc * (P - y);
        } else {
          comp_add(hi, lo, -y.hi, -y.lo);
          K.qc[l][x] = cc * (hi + lo);
        }
      }
    }
    if (l < 4) {
      const sp<R> t = spin(b * N_EV + O_X0 + 2 + (l >> 1));
      put(b * N_EV + O_VC + l, fcur(sp<R>{{t.c[2], t.c[3], t.c[0], t.c[1]}}, spin(b * N_EV + O_X0 + (l & 1))));
    }
  }

  // --- gluon currents -------------------------------------------------------
  // 2 P.J for a subset's summed momentum (the other vertex momentum drops out:
  // every current is conserved, P_J.J = 0)
  __device__ __forceinline__ cx<R> p_dot(const Kin& K, int mask, const cv<R>& J) const {
    const R p[4] = {K.P[mask][0], K.P[mask][1], K.P[mask][2], K.P[mask][3]};
    const cx<R> s = dotr(p, J);
    return {s.r + s.r, s.i + s.i};
  }

  __device__ __forceinline__ void two_gluons(int b, int t, unsigned w) {
    const int ob = b * N_EV;
    const cv<R> A = vec(ob + O_E + (w & 7)), B = vec(ob + O_E + ((w >> 3) & 7));
    const int ma = 1 << ((w >> 6) & 3), mb = 1 << ((w >> 8) & 3);
    const Kin& K = kin[b];
    const R c = -K.ik2[ma | mb];
    const cx<R> ca = (-c) * p_dot(K, ma, B), cb = c * p_dot(K, mb, A), cp = c * dot(A, B);
    cv<R> o;
#pragma unroll
    for (int m = 0; m < 4; ++m)
      o.c[m] = cmac(A.c[m], ca, cmac(B.c[m], cb, (K.P[ma][m] - K.P[mb][m]) * cp));
    put(ob + O_J2 + t, o);
  }

  __device__ __forceinline__ void product(int b, int t, unsigned w) {
    const int ob = b * N_EV;
    const cv<R> A = vec(ob + O_E + (w & 7)), B = vec(ob + ((w >> 3) & 1 ? O_J2 : O_E) + ((w >> 4) & 31));
    *reinterpret_cast<cx<R>*>(obj + (b * N_OBJ + O_WK + t) * 16) = dot(A, B);
  }

  __device__ __forceinline__ void three_gluons(int b, int t, unsigned w, unsigned w2) {
    const int ob = b * N_EV;
    const cv<R> A = vec(ob + O_E + (w & 7)), B = vec(ob + O_E + ((w >> 3) & 7)), C = vec(ob + O_E + ((w >> 6) & 7));
    const cv<R> AB = flip(vec(ob + O_J2 + ((w >> 9) & 31)), (w >> 14) << 31);
    const cv<R> BC = flip(vec(ob + O_J2 + ((w >> 15) & 31)), (w >> 20) << 31);
    const int ma = 1 << ((w >> 21) & 3), mb = 1 << ((w >> 23) & 3), mc = 1 << ((w >> 25) & 3);
    const Kin& K = kin[b];
    const R c = -K.ik2[ma | mb | mc];
    const cx<R> ab = prod(b, w2 & 31), bc = prod(b, (w2 >> 5) & 31), ac = prod(b, (w2 >> 10) & 31);
    const cx<R> pa = prod(b, (w2 >> 15) & 127, (w >> 20) << 31), pc = prod(b, (w2 >> 22) & 127, (w >> 14) << 31);
    const cx<R> fa = c * (bc - p_dot(K, ma, BC)), fc = c * (ab + p_dot(K, mc, AB));
    const cx<R> fb = (R(-2) * c) * ac;
    const cx<R> fbc = c * p_dot(K, mb | mc, A), fab = (-c) * p_dot(K, ma | mb, C);
    const cx<R> ga = c * pa, gc = c * pc;
    cv<R> o;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      cx<R> x = (K.P[ma][m] - K.P[mb | mc][m]) * ga;
      x = rmac(K.P[ma | mb][m] - K.P[mc][m], gc, x);
      x = cmac(A.c[m], fa, x);
      x = cmac(B.c[m], fb, x);
      x = cmac(C.c[m], fc, x);
      x = cmac(AB.c[m], fab, x);
      o.c[m] = cmac(BC.c[m], fbc, x);
    }
    put(ob + O_J3 + t, o);
  }

  // (ub gamma v).J(0bcd) for the four spin states of the pair; the parts of the
  // current along its own momentum drop out (ub gamma v is conserved)
  __device__ __forceinline__ void four_gluons(int b, int t, unsigned w, unsigned w2, unsigned w3, unsigned w4) {
    const int ob = b * N_EV;
    const Kin& K = kin[b];
    const int gb = (w >> 26) & 3, gc = (w >> 28) & 3, gd = (w2 >> 12) & 3;
    const int mb = 1 << gb, mc = 1 << gc, md = 1 << gd;
    const unsigned nbc = (w >> 19) << 31, ncd = (w >> 25) << 31;
    const cv<R> A = vec(ob + O_E), B = vec(ob + O_E + (w & 7)), C = vec(ob + O_E + ((w >> 3) & 7)),
                D = vec(ob + O_E + ((w >> 6) & 7));
    cx<R> fa = prod(b, (w3 >> 15) & 127, nbc) + prod(b, w4 & 127, ncd);          // BC.D + B.CD
    cx<R> fd = prod(b, (w3 >> 22) & 127, nbc) + prod(b, (w4 >> 14) & 127);       // A.BC + AB.C
    const cx<R> ad = prod(b, (w3 >> 5) & 31), acd = prod(b, (w4 >> 7) & 127, ncd), abd = prod(b, (w4 >> 21) & 127);
    const cx<R> fbc = {R(-2) * ad.r, R(-2) * ad.i}, fb = {R(-2) * acd.r, R(-2) * acd.i},
                fc = {R(-2) * abd.r, R(-2) * abd.i};
    cx<R> fab, fcd, fabc, fbcd, ga, gab, gabc;
    {
      const cv<R> AB = vec(ob + O_J2 + ((w >> 9) & 31)), CD = flip(vec(ob + O_J2 + ((w >> 20) & 31)), ncd);
      const cx<R> z = dot(AB, CD);
      gab = z + z;
      fab = prod(b, (w3 >> 10) & 31) - p_dot(K, 1 | mb, CD);
      fcd = prod(b, w3 & 31) + p_dot(K, mc | md, AB);
    }
    {
      const cv<R> BCD = vec(ob + O_J3 + ((w2 >> 6) & 63));
      const cx<R> z = dot(A, BCD);
      ga = z + z;
      fa = fa - p_dot(K, 1, BCD);
      fbcd = p_dot(K, mb | mc | md, A);
    }
    {
      const cv<R> ABC = vec(ob + O_J3 + (w2 & 63));
      const cx<R> z = dot(ABC, D);
      gabc = z + z;
      fd = fd + p_dot(K, md, ABC);
      fabc = -p_dot(K, 1 | mb | mc, D);
    }
    cv<R> o;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      o.c[m] = K.P[1][m] * ga;
      o.c[m] = rmac(K.P[1 | mb][m], gab, o.c[m]);
      o.c[m] = rmac(K.P[1 | mb | mc][m], gabc, o.c[m]);
    }
    auto add = [&o](const cv<R>& J, const cx<R>& f) {
#pragma unroll
      for (int m = 0; m < 4; ++m) o.c[m] = cmac(J.c[m], f, o.c[m]);
    };
    add(A, fa);
    add(B, fb);
    add(C, fc);
    add(D, fd);
    add(vec(ob + O_J2 + ((w >> 9) & 31)), fab);
    add(flip(vec(ob + O_J2 + ((w >> 14) & 31)), nbc), fbc);
    add(flip(vec(ob + O_J2 + ((w >> 20) & 31)), ncd), fcd);
    add(vec(ob + O_J3 + (w2 & 63)), fabc);
    add(vec(ob + O_J3 + ((w2 >> 6) & 63)), fbcd);
    const R c = -K.ik2[15];
#pragma unroll
    for (int l = 0; l < 4; ++l) wv[b][l][t >> 3][t & 7] = c * dot(vec(ob + O_VC + l), o);
  }

  // --- spinors --------------------------------------------------------------
  // Jslash x, added to o when ACC; top: x a swapped row spinor
  template <bool ACC>
  __device__ __forceinline__ static void slash_side(sp<R>& o, cv<R> J, const sp<R>& x, bool top) {
    const unsigned neg = top ? 0x80000000u : 0u;
    J.c[2] = {flip(J.c[2].r, neg), flip(J.c[2].i, neg)};
    slash_body<R, ACC>(o, weyl_form(J), x);
  }
  __device__ __forceinline__ sp<R> propagate(const Kin& K, int mask, const sp<R>& x, bool top) const {
    const R q[4] = {K.qc[mask][0], K.qc[mask][1], flip(K.qc[mask][2], top ? 0x80000000u : 0u), K.qc[mask][3]};
    return fprop(q, K.mc[mask], x);
  }

  __device__ __forceinline__ void one_gluon(int b, int t, unsigned w) {
    const int ob = b * N_EV;
    const bool top = (w >> 4) & 1;
    sp<R> o;
    slash_side<false>(o, vec(ob + O_E + (w & 7)), spin(ob + O_X0 + ((w >> 3) & 3)), top);
    put(O_X1 + t, propagate(kin[b], (w >> 5) & 15, o, top));
  }
  __device__ __forceinline__ void work_r3(int b, int at, unsigned w) {
    const int ob = b * N_EV;
    sp<R> o;
    slash_side<false>(o, vec(ob + O_J3 + (w & 63)), spin(ob + O_X0 + ((w >> 6) & 3)), (w >> 7) & 1);
    put(O_WK + at, o);
  }
  __device__ __forceinline__ void work_y(int b, int at, unsigned w) {
    sp<R> o;
    slash_side<false>(o, vec(b * N_EV + O_J2 + (w & 31)), spin(O_X1 + ((w >> 5) & 15)), false);
    put(O_WK + at, o);
  }
  __device__ __forceinline__ void work_x2(int b, int at, unsigned w) {
    const int ob = b * N_EV;
    const bool top = (w >> 15) & 1;
    sp<R> o;
    slash_side<false>(o, vec(ob + O_E + (w & 7)), spin(O_X1 + ((w >> 3) & 31)), top);
    slash_side<true>(o, flip(vec(ob + O_J2 + ((w >> 8) & 31)), (w >> 13) << 31), spin(ob + O_X0 + ((w >> 14) & 3)), top);
    if (!top) o = propagate(kin[b], (w >> 16) & 15, o, false);
    put(O_WK + at, o);
  }

  // the six W of this lane, spread over the 24 orderings
  __device__ __forceinline__ void start(int b, int lane, cx<R> (&A)[24]) const {
    cx<R> W[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) W[i] = wv[b][lane >> 3][i][lane & 7];
    from_w<R>(W, A);
  }
};

}  // namespace coop
}  // namespace rw
