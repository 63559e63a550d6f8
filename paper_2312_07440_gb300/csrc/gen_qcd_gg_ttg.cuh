// ---- generated by gen/qcd_gen.py: gg_ttg (g g -> t tbar + 1 g), do not edit ----
// 16 Feynman diagrams, 6 colour orderings, 32 helicities.
// colour matrix C = Cint / 9
#pragma once
#include "colour_mma.cuh"
#include "qcd.cuh"

namespace rw { namespace gg_ttg {
constexpr int NG = 3;
constexpr int NEXT = 5;
constexpr int K = 6;
constexpr int NHEL = 32;
constexpr int NDIAG = 16;
constexpr int MAX_LB = 3;  // helicity levels that can be spread over lanes
constexpr int NJS = 0;  // currents of 3+ gluons, one JStore slot each
constexpr int CDEN = 9;
constexpr int IDENT = 1;  // identical outgoing gluons (1/IDENT!)
constexpr unsigned OUTGOING_GLUONS = 4u;  // bit g: gluon g outgoing
__host__ __device__ constexpr int cint(int i, int j) { constexpr int c[K * K] = {64, -8, -8, 1, 1, 10, -8, 64, 1, 10, -8, 1, -8, 1, 64, -8, 10, 1, 1, 10, -8, 64, 1, -8, 1, -8, 10, 1, 64, -8, 10, 1, 1, -8, -8, 64}; return c[i * K + j]; }
constexpr int ORDER[K][NG] = {{0, 1, 2}, {0, 2, 1}, {1, 0, 2}, {1, 2, 0}, {2, 0, 1}, {2, 1, 0}};
static __device__ const short CI[K * K] = {64, -8, -8, 1, 1, 10, -8, 64, 1, 10, -8, 1, -8, 1, 64, -8, 10, 1, 1, 10, -8, 64, 1, -8, 1, -8, 10, 1, 64, -8, 10, 1, 1, -8, -8, 64};  // row-major C_int for the tensor-core sum

// Sum over this lane's helicities of sum_{s,t} Cint_st Re(A_s^* A_t), g = 1;
// helicities with gluon 0 at +1 only, doubled (J^dagger C J(h) = J^dagger C J(-h)).
// CM: colour sum by FMA (CM_FMA, any R) or on the tensor cores (CM_FP16/CM_BF16, R = float);
// CM_STORE_FP16/CM_STORE_BF16: no colour sum here, each J vector goes to sink->put()
// for a later tensor-core pass (the return value is then 0).
template <class R, int LB, int CM = CM_FMA, bool JS = false, class Sink = NoSink>
__device__ __forceinline__ R hel_sum(const QcdExt<R, NG>& X, const QcdKin<R, NG>& Kn, int lane,
                                     [[maybe_unused]] Sink* sink = nullptr) {
  static_assert(CM == CM_FMA || sizeof(R) == 4, "tensor-core colour sum takes FP32 amplitudes");
  constexpr bool MMA = CM == CM_FP16 || CM == CM_BF16;
  const ColourMma<K, MMA ? CM : CM_FP16> cmma(MMA ? CI : nullptr, JS ? NJS * 32 : 0);
  JStore<R, NJS, JS> js;
  R acc = R(0);
  [[maybe_unused]] R cc0_0 = R(0), cc1_0 = R(0), cc2_0 = R(0), cc3_0 = R(0), cc0_1 = R(0), cc1_1 = R(0), cc2_1 = R(0), cc3_1 = R(0);  // per distinct c_ij and top helicity
  {
    const int h0 = 0;
    const cv<R> E0 = h0 ? X.eps[0][1] : X.eps[0][0];
    const ws<R> W0 = weyl_form(E0);
    const sp<R> T0_0 = row_prop(Kn.qc[6], Kn.mc[6], row_slash(W0, X.ub[0]));
    const sp<R> T0_1 = row_prop(Kn.qc[6], Kn.mc[6], row_slash(W0, X.ub[1]));
    // the quark line's currents and (below) the spinors of gluons 0 and 1 for both antitop
    // helicities at the level they depend on, in local memory, instead of once per inner trip
    // (200,003 events x 2 points FP64 15.03 -> 13.57 ms, 131,072 x 64 FP32 6.84 -> 6.59 ms)
    constexpr bool HV = LB < 3, H1 = LB < 2;
    cv<R> VC[HV ? 4 : 1];
    if constexpr (HV)
      for (int i = 0; i < 4; ++i) VC[i] = fcur(X.ub[i & 1], X.v[i >> 1]);
    [[maybe_unused]] sp<R> S_0v0, S_0v1;
    if constexpr (LB < 3) {
      S_0v0 = fprop(Kn.qc[1], Kn.mc[1], slash(W0, X.v[0]));
      S_0v1 = fprop(Kn.qc[1], Kn.mc[1], slash(W0, X.v[1]));
    }
    #pragma unroll 1
    for (int i1 = 0; i1 < (LB >= 1 ? 1 : 2); ++i1) {
      const int h1 = LB >= 1 ? ((lane >> (LB - 1)) & 1) : i1;
      const cv<R> E1 = h1 ? X.eps[1][1] : X.eps[1][0];
      const ws<R> W1 = weyl_form(E1);
      const sp<R> T1_0 = row_prop(Kn.qc[5], Kn.mc[5], row_slash(W1, X.ub[0]));
      const sp<R> T1_1 = row_prop(Kn.qc[5], Kn.mc[5], row_slash(W1, X.ub[1]));
      cv<R> J0_1 = current2(E0, Kn.P[1], E1, Kn.P[2], Kn.cg[3]);
      const cv<R> J1_0 = neg(J0_1);
      sp<R> S1v[H1 ? 2 : 1], X01v[H1 ? 2 : 1], X10v[H1 ? 2 : 1];
      if constexpr (H1) {
        const ws<R> WJ = weyl_form(J0_1);
        for (int i = 0; i < 2; ++i) {
          S1v[i] = fprop(Kn.qc[2], Kn.mc[2], slash(W1, X.v[i]));
          X01v[i] = slash(WJ, X.v[i]);
          X10v[i] = spneg(X01v[i]);
          slash_acc(X01v[i], W0, S1v[i]);
          slash_acc(X10v[i], W1, i ? S_0v1 : S_0v0);
        }
      }
      #pragma unroll 1
      for (int i2 = 0; i2 < (LB >= 2 ? 1 : 2); ++i2) {
        const int h2 = LB >= 2 ? ((lane >> (LB - 2)) & 1) : i2;
        const cv<R> E2 = h2 ? X.eps[2][1] : X.eps[2][0];
        const ws<R> W2 = weyl_form(E2);
        const sp<R> T2_0 = row_prop(Kn.qc[3], Kn.mc[3], row_slash(W2, X.ub[0]));
        const sp<R> T2_1 = row_prop(Kn.qc[3], Kn.mc[3], row_slash(W2, X.ub[1]));
        cv<R> J0_2 = current2(E0, Kn.P[1], E2, Kn.P[4], Kn.cg[5]);
        cv<R> J1_2 = current2(E1, Kn.P[2], E2, Kn.P[4], Kn.cg[6]);
        const cv<R> J2_0 = neg(J0_2);
        const cv<R> J2_1 = neg(J1_2);
        const cv<R> J0_1_2 = current3(E0, E1, E2, J0_1, J1_2, Kn.P[1], Kn.P[4], Kn.P[3], Kn.P[6], Kn.cg[7]);
        const cv<R> J0_2_1 = current3(E0, E2, E1, J0_2, J2_1, Kn.P[1], Kn.P[2], Kn.P[5], Kn.P[6], Kn.cg[7]);
        const cv<R> J1_2_0 = J0_2_1;
        const cv<R> J2_1_0 = J0_1_2;
        #pragma unroll 1
        for (int i3 = 0; i3 < (LB >= 3 ? 1 : 2); ++i3) {
          const int h3 = LB >= 3 ? ((lane >> (LB - 3)) & 1) : i3;
          const sp<R> S_E = h3 ? X.v[1] : X.v[0];
          sp<R> S_0;
          if constexpr (LB < 3) S_0 = h3 ? S_0v1 : S_0v0;
          else S_0 = fprop(Kn.qc[1], Kn.mc[1], slash(W0, S_E));
          sp<R> S_1;
          if constexpr (H1) S_1 = S1v[h3];
          else S_1 = fprop(Kn.qc[2], Kn.mc[2], slash(W1, S_E));
          const sp<R> S_2 = fprop(Kn.qc[4], Kn.mc[4], slash(W2, S_E));
          cx<R> A0_0, A0_1, A1_0, A1_1, A2_0, A2_1, A3_0, A3_1, A4_0, A4_1, A5_0, A5_1;
          {
            sp<R> x, y;  // J(01) v and J(10) v, then the single-gluon terms
            if constexpr (H1) {
              x = X01v[h3];
              y = X10v[h3];
            } else {
              x = slash(weyl_form(J0_1), S_E);
              y = spneg(x);
              slash_acc(x, W0, S_1);
              slash_acc(y, W1, S_0);
            }
            A4_0 = rowcol(T2_0, x);
            A5_0 = rowcol(T2_0, y);
            A4_1 = rowcol(T2_1, x);
            A5_1 = rowcol(T2_1, y);
          }
          {
            sp<R> x, y;  // J(02) v and J(20) v, then the single-gluon terms
            x = slash(weyl_form(J0_2), S_E);
            y = spneg(x);
            slash_acc(x, W0, S_2);
            slash_acc(y, W2, S_0);
            A2_0 = rowcol(T1_0, x);
            A3_0 = rowcol(T1_0, y);
            A2_1 = rowcol(T1_1, x);
            A3_1 = rowcol(T1_1, y);
          }
          {
            sp<R> x, y;  // J(12) v and J(21) v, then the single-gluon terms
            x = slash(weyl_form(J1_2), S_E);
            y = spneg(x);
            slash_acc(x, W1, S_2);
            slash_acc(y, W2, S_1);
            A0_0 = rowcol(T0_0, x);
            A1_0 = rowcol(T0_0, y);
            A0_1 = rowcol(T0_1, x);
            A1_1 = rowcol(T0_1, y);
          }
          {
            const sp<R> z = slash(J0_1, S_2);
            const cx<R> d0 = rowcol(X.ub[0], z);
            A0_0 = A0_0 + d0;
            A2_0 = A2_0 - d0;
            const cx<R> d1 = rowcol(X.ub[1], z);
            A0_1 = A0_1 + d1;
            A2_1 = A2_1 - d1;
          }
          {
            const sp<R> z = slash(J0_2, S_1);
            const cx<R> d0 = rowcol(X.ub[0], z);
            A1_0 = A1_0 + d0;
            A4_0 = A4_0 - d0;
            const cx<R> d1 = rowcol(X.ub[1], z);
            A1_1 = A1_1 + d1;
            A4_1 = A4_1 - d1;
          }
          {
            const sp<R> z = slash(J1_2, S_0);
            const cx<R> d0 = rowcol(X.ub[0], z);
            A3_0 = A3_0 + d0;
            A5_0 = A5_0 - d0;
            const cx<R> d1 = rowcol(X.ub[1], z);
            A3_1 = A3_1 + d1;
            A5_1 = A5_1 - d1;
          }
          {
            cv<R> V;
            if constexpr (HV) V = VC[2 * h3 + 0];
            else V = fcur(X.ub[0], S_E);
            const cx<R> u = dot(V, J0_1_2), t = dot(V, J0_2_1), m = u + t;
            A0_0 = A0_0 + u;
            A5_0 = A5_0 + u;
            A1_0 = A1_0 + t;
            A3_0 = A3_0 + t;
            A2_0 = A2_0 - m;
            A4_0 = A4_0 - m;
          }
          {
            cv<R> V;
            if constexpr (HV) V = VC[2 * h3 + 1];
            else V = fcur(X.ub[1], S_E);
            const cx<R> u = dot(V, J0_1_2), t = dot(V, J0_2_1), m = u + t;
            A0_1 = A0_1 + u;
            A5_1 = A5_1 + u;
            A1_1 = A1_1 + t;
            A3_1 = A3_1 + t;
            A2_1 = A2_1 - m;
            A4_1 = A4_1 - m;
          }
          if constexpr (CM != CM_FMA) {
            const cx<float> Aa0[K] = {A0_0, A1_0, A2_0, A3_0, A4_0, A5_0};
            const cx<float> Aa1[K] = {A0_1, A1_1, A2_1, A3_1, A4_1, A5_1};
            if constexpr (MMA) {
              acc += R(2) * (cmma.sum(Aa0) + cmma.sum(Aa1));  // x2 helicity flip
            } else {
              sink->put(Aa0);
              sink->put(Aa1);
            }
          } else {
            cc0_0 = fmadd(A0_0.r, A0_0.r, fmadd(A0_0.i, A0_0.i, cc0_0));
            cc1_0 = fmadd(A0_0.r, A1_0.r, fmadd(A0_0.i, A1_0.i, cc1_0));
            cc1_0 = fmadd(A0_0.r, A2_0.r, fmadd(A0_0.i, A2_0.i, cc1_0));
            cc2_0 = fmadd(A0_0.r, A3_0.r, fmadd(A0_0.i, A3_0.i, cc2_0));
            cc2_0 = fmadd(A0_0.r, A4_0.r, fmadd(A0_0.i, A4_0.i, cc2_0));
            cc3_0 = fmadd(A0_0.r, A5_0.r, fmadd(A0_0.i, A5_0.i, cc3_0));
            cc0_0 = fmadd(A1_0.r, A1_0.r, fmadd(A1_0.i, A1_0.i, cc0_0));
            cc2_0 = fmadd(A1_0.r, A2_0.r, fmadd(A1_0.i, A2_0.i, cc2_0));
            cc3_0 = fmadd(A1_0.r, A3_0.r, fmadd(A1_0.i, A3_0.i, cc3_0));
            cc1_0 = fmadd(A1_0.r, A4_0.r, fmadd(A1_0.i, A4_0.i, cc1_0));
            cc2_0 = fmadd(A1_0.r, A5_0.r, fmadd(A1_0.i, A5_0.i, cc2_0));
            cc0_0 = fmadd(A2_0.r, A2_0.r, fmadd(A2_0.i, A2_0.i, cc0_0));
            cc1_0 = fmadd(A2_0.r, A3_0.r, fmadd(A2_0.i, A3_0.i, cc1_0));
            cc3_0 = fmadd(A2_0.r, A4_0.r, fmadd(A2_0.i, A4_0.i, cc3_0));
            cc2_0 = fmadd(A2_0.r, A5_0.r, fmadd(A2_0.i, A5_0.i, cc2_0));
            cc0_0 = fmadd(A3_0.r, A3_0.r, fmadd(A3_0.i, A3_0.i, cc0_0));
            cc2_0 = fmadd(A3_0.r, A4_0.r, fmadd(A3_0.i, A4_0.i, cc2_0));
            cc1_0 = fmadd(A3_0.r, A5_0.r, fmadd(A3_0.i, A5_0.i, cc1_0));
            cc0_0 = fmadd(A4_0.r, A4_0.r, fmadd(A4_0.i, A4_0.i, cc0_0));
            cc1_0 = fmadd(A4_0.r, A5_0.r, fmadd(A4_0.i, A5_0.i, cc1_0));
            cc0_0 = fmadd(A5_0.r, A5_0.r, fmadd(A5_0.i, A5_0.i, cc0_0));
            cc0_1 = fmadd(A0_1.r, A0_1.r, fmadd(A0_1.i, A0_1.i, cc0_1));
            cc1_1 = fmadd(A0_1.r, A1_1.r, fmadd(A0_1.i, A1_1.i, cc1_1));
            cc1_1 = fmadd(A0_1.r, A2_1.r, fmadd(A0_1.i, A2_1.i, cc1_1));
            cc2_1 = fmadd(A0_1.r, A3_1.r, fmadd(A0_1.i, A3_1.i, cc2_1));
            cc2_1 = fmadd(A0_1.r, A4_1.r, fmadd(A0_1.i, A4_1.i, cc2_1));
            cc3_1 = fmadd(A0_1.r, A5_1.r, fmadd(A0_1.i, A5_1.i, cc3_1));
            cc0_1 = fmadd(A1_1.r, A1_1.r, fmadd(A1_1.i, A1_1.i, cc0_1));
            cc2_1 = fmadd(A1_1.r, A2_1.r, fmadd(A1_1.i, A2_1.i, cc2_1));
            cc3_1 = fmadd(A1_1.r, A3_1.r, fmadd(A1_1.i, A3_1.i, cc3_1));
            cc1_1 = fmadd(A1_1.r, A4_1.r, fmadd(A1_1.i, A4_1.i, cc1_1));
            cc2_1 = fmadd(A1_1.r, A5_1.r, fmadd(A1_1.i, A5_1.i, cc2_1));
            cc0_1 = fmadd(A2_1.r, A2_1.r, fmadd(A2_1.i, A2_1.i, cc0_1));
            cc1_1 = fmadd(A2_1.r, A3_1.r, fmadd(A2_1.i, A3_1.i, cc1_1));
            cc3_1 = fmadd(A2_1.r, A4_1.r, fmadd(A2_1.i, A4_1.i, cc3_1));
            cc2_1 = fmadd(A2_1.r, A5_1.r, fmadd(A2_1.i, A5_1.i, cc2_1));
            cc0_1 = fmadd(A3_1.r, A3_1.r, fmadd(A3_1.i, A3_1.i, cc0_1));
            cc2_1 = fmadd(A3_1.r, A4_1.r, fmadd(A3_1.i, A4_1.i, cc2_1));
            cc1_1 = fmadd(A3_1.r, A5_1.r, fmadd(A3_1.i, A5_1.i, cc1_1));
            cc0_1 = fmadd(A4_1.r, A4_1.r, fmadd(A4_1.i, A4_1.i, cc0_1));
            cc1_1 = fmadd(A4_1.r, A5_1.r, fmadd(A4_1.i, A5_1.i, cc1_1));
            cc0_1 = fmadd(A5_1.r, A5_1.r, fmadd(A5_1.i, A5_1.i, cc0_1));
          }
        }
      }
    }
  }
  if constexpr (CM == CM_FMA) acc = R(2) * (R(64) * (cc0_0 + cc0_1) + R(-16) * (cc1_0 + cc1_1) + R(2) * (cc2_0 + cc2_1) + R(20) * (cc3_0 + cc3_1));  // x2 helicity flip
  return acc;
}

// floating-point operations of one full helicity sum (all levels, all loop trips)
constexpr long FLOPS_HEL_SUM = 20969;
}}  // namespace
