// Process adapters for the fused kernel: |M|^2 / cscale of one event for one
// parameter point, helicity slices combined across the 2^LB lanes of a group.
#pragma once
#include <type_traits>

#include "colour_mma.cuh"
#include "helas.cuh"
#include "kernels.cuh"
#include "qcd.cuh"
#include "qed.cuh"

namespace rw {

// Tag::KSMEM (optional, default false): keep the per-event constants in
// shared memory in the FP32 modes
template <class T, class = void>
struct tag_ksmem : std::false_type {};
template <class T>
struct tag_ksmem<T, std::void_t<decltype(T::KSMEM)>> : std::integral_constant<bool, T::KSMEM> {};

// Tag::INLINE_ME (optional, default false): the FP32 amplitude code inlined
// into the kernel's single call site (small processes: no call-site saves)
template <class T, class = void>
struct tag_inline_me : std::false_type {};
template <class T>
struct tag_inline_me<T, std::void_t<decltype(T::INLINE_ME)>> : std::integral_constant<bool, T::INLINE_ME> {};

// g g -> t tbar + n g.  Tag provides NG, NEXT, MAX_LB and hel_sum<R, LB, CM>();
// CM selects the colour sum (FMA, or tensor cores in FP16/BF16).
template <class Tag, int CM = 0>
struct QcdProc {
  static constexpr int NG = Tag::NG;
  static constexpr int NEXT = Tag::NEXT;
  static constexpr bool MOVES = true;  // a new top mass moves the event, or does not fit it
  static constexpr int NCOL = Tag::NCOL;
  static constexpr bool kSymmetricHelicities = true;
  // per-event constants (external wavefunctions and propagator invariants):
  // one slot per event group in shared memory, written by the group's lanes
  // and read by them at every use, instead of a copy in every lane's
  // registers (FP32, at least 4 lanes per event)
  template <class R, int LB>
  static constexpr bool ksmem() {
    return tag_ksmem<Tag>::value && sizeof(R) == 4 && LB >= 2;
  }
  static constexpr int kSlot = (int)((sizeof(QcdExt<float, NG>) + sizeof(QcdKin<float, NG>) + 15) / 16 * 16);

  // Momenta: FP64 in FP64 mode, double-float in the FP32 modes (dfloat.cuh).
  template <class R>
  using mom_t = typename std::conditional<sizeof(R) == 8, double, df>::type;
  // dynamic shared memory per thread of the amplitude code: the current store,
  // then (tensor-core colour sum) the warp's colour staging, as a per-thread share
  template <class R>
  static constexpr int store_bytes() {
    return ((Tag::JSMEM && sizeof(R) == 4) ? Tag::NJS * 32 : 0) +
           ((CM == CM_FP16 || CM == CM_BF16) ? ColourStage<(Tag::NCOL + 15) / 16 * 16>::per_thread : 0);
  }
  template <class R, int LB = 0>
  static constexpr int jstore_bytes() {
    static_assert(kSlot % 16 == 0 && kSlot % (1 << Tag::MAX_LB) == 0, "the slots split evenly over the lanes");
    return store_bytes<R>() + (ksmem<R, LB>() ? kSlot >> LB : 0);
  }

  template <class R, int LB>
  __device__ __forceinline__ static double me_body(const mom_t<R> (&p)[NEXT][4], const PointDev& pt, int lane,
                                           unsigned gmask) {
    static_assert(LB <= Tag::MAX_LB, "more lane bits than helicity levels");
    double s;
    if constexpr (ksmem<R, LB>()) {
      extern __shared__ __align__(16) unsigned char rw_dyn_bytes[];
      unsigned char* slot =
          rw_dyn_bytes + (size_t)store_bytes<R>() * blockDim.x + (size_t)(threadIdx.x >> LB) * kSlot;
      QcdExt<R, NG>& X = *reinterpret_cast<QcdExt<R, NG>*>(slot);
      QcdKin<R, NG>& Kn = *reinterpret_cast<QcdKin<R, NG>*>(slot + sizeof(QcdExt<R, NG>));
      __syncwarp(gmask);  // the group's reads of the previous evaluation are done
      // every lane of the group writes the same values (same inputs, same code)
      qcd_setup<R, NG, NEXT>(p, pt.m_t, X, Kn);
      __syncwarp(gmask);
      s = double(Tag::template hel_sum<R, LB, CM>(X, Kn, lane));
    } else {
      QcdExt<R, NG> X;
      QcdKin<R, NG> Kn;
      qcd_setup<R, NG, NEXT>(p, pt.m_t, X, Kn);
      s = double(Tag::template hel_sum<R, LB, CM>(X, Kn, lane));
    }
#pragma unroll
    for (int o = 1; o < (1 << LB); o <<= 1) s += __shfl_xor_sync(gmask, s, o);
    return s;
  }  // Out of line by default: every evaluation runs the same instructions, so
  // identical inputs give bitwise identical |M|^2 (r == 1 exactly for
  // unchanged parameters).  Inlined (Tag::INLINE_ME, FP32) the kernel's one
  // call site, inside its loop over the points, keeps that property.
  template <class R>
  static constexpr bool inline_me() {
    return tag_inline_me<Tag>::value && sizeof(R) == 4;
  }
  template <class R, int LB>
  __device__ __noinline__ static double me(const mom_t<R> (&p)[NEXT][4], const PointDev& pt, int lane,
                                           unsigned gmask) {
    return me_body<R, LB>(p, pt, lane, gmask);
  }

  // The amplitudes of one event and point for a separate colour pass
  // (CM_STORE_*): the set-up as in me_body, then every J vector to sink.put();
  // false when the point's masses do not fit the event (its |M'|^2 is 0).
  template <class R, int LB, class Sink>
  __device__ __noinline__ static bool me_store(const mom_t<R> (&p)[NEXT][4], const PointDev& pt, int lane,
                                               unsigned gmask, Sink& sink) {
    static_assert(LB <= Tag::MAX_LB, "more lane bits than helicity levels");
    mom_t<R> q[NEXT][4];
    bool inside = true;
    if (pt.reshuffle) {
      inside = reshuffle<R>(p, pt.m_t, q);
    } else {
#pragma unroll
      for (int i = 0; i < NEXT; ++i)
#pragma unroll
        for (int m = 0; m < 4; ++m) q[i][m] = p[i][m];
    }
    if constexpr (ksmem<R, LB>()) {
      extern __shared__ __align__(16) unsigned char rw_dyn_bytes[];
      unsigned char* slot =
          rw_dyn_bytes + (size_t)store_bytes<R>() * blockDim.x + (size_t)(threadIdx.x >> LB) * kSlot;
      QcdExt<R, NG>& X = *reinterpret_cast<QcdExt<R, NG>*>(slot);
      QcdKin<R, NG>& Kn = *reinterpret_cast<QcdKin<R, NG>*>(slot + sizeof(QcdExt<R, NG>));
      __syncwarp(gmask);
      qcd_setup<R, NG, NEXT>(q, pt.m_t, X, Kn);
      __syncwarp(gmask);
      Tag::template hel_sum<R, LB, CM>(X, Kn, lane, &sink);
    } else {
      QcdExt<R, NG> X;
      QcdKin<R, NG> Kn;
      qcd_setup<R, NG, NEXT>(q, pt.m_t, X, Kn);
      Tag::template hel_sum<R, LB, CM>(X, Kn, lane, &sink);
    }
    return inside;
  }

  // FP64 mode refines the FP32 Newton solution with one third-order FP64 step,
  // the FP32 modes with one double-float step.
  template <class R>
  __device__ __forceinline__ static bool reshuffle(const mom_t<R> (&p)[NEXT][4], double mt, mom_t<R> (&q)[NEXT][4]) {
    if constexpr (sizeof(R) == 8)
      return reshuffle_tops<NEXT>(p, mt, q);
    else
      return reshuffle_tops<NEXT>(p, mt, q);
  }
};

// e-(p0) e+(p1) -> n photons (massless QED).  Tag provides NA, NEXT, MAX_LB
// and hel_sum<R, LB>() (generated by gen/qed_gen.py); |M|^2 = cscale * sum (the caller's product),
// cscale = e^(2n) / (4 n!).  Nothing moves with the parameters (no reshuffle).
template <class Tag>
struct QedProc {
  static constexpr int NA = Tag::NA;
  static constexpr int NEXT = Tag::NEXT;
  static constexpr bool MOVES = false;
  template <class R>
  using mom_t = typename std::conditional<sizeof(R) == 8, double, df>::type;
  template <class R, int LB = 0>
  static constexpr int jstore_bytes() {
    return 0;
  }
  template <class R>
  static constexpr bool inline_me() {
    return false;
  }

  template <class R, int LB>
  __device__ __noinline__ static double me(const mom_t<R> (&p)[NEXT][4], const PointDev& pt, int lane,
                                           unsigned gmask) {
    static_assert(LB <= Tag::MAX_LB, "more lane bits than helicity levels");
    QedExt<R, NA> X;
    QedKin<R, NA> Kn;
    qed_setup<R, NA, NEXT>(p, X, Kn);
    double s = double(Tag::template hel_sum<R, LB>(X, Kn, lane));
#pragma unroll
    for (int o = 1; o < (1 << LB); o <<= 1) s += __shfl_xor_sync(gmask, s, o);
    return s;
  }
  template <class R>
  __device__ __forceinline__ static bool reshuffle(const mom_t<R> (&p)[NEXT][4], double, mom_t<R> (&q)[NEXT][4]) {
#pragma unroll
    for (int i = 0; i < NEXT; ++i)
#pragma unroll
      for (int m = 0; m < 4; ++m) q[i][m] = p[i][m];
    return true;
  }
};

// e-(p0) e+(p1) -> mu-(p2) mu+(p3) through s-channel photon and Z (unitary
// gauge, fixed width), massless leptons:
//   M = e^2 (jo.ji)/s + [zo.zi - (k.zo)(k.zi)/MZ^2] / (s - MZ^2 + i MZ WZ)
// with ji = vbar(p1) gamma^mu u(p0), zi = vbar(p1) gamma^mu (gL PL + gR PR) u(p0)
// and jo, zo the same for ubar(p2) ... v(p3); |M|^2 averaged over the 4
// initial helicity states.  Massless: a helicity state has one chirality, so
// of the 16 helicity configurations the four of equal chirality along each
// line remain, and each current is one 2 x 2 block.
//
// The FP64 pipe (2 lanes per cycle and SM) bounds it even for a few thousand
// events, so with at least four lanes per event each lane forms the spinors of
// one particle, the group exchanges them, and each lane takes one of the four
// configurations (4,096 events, one point, whole call: 116 -> 54 us); the
// currents carry no parameter and are formed once per event (54 -> 45 us).
struct EeMumu {
  static constexpr int NEXT = 4;
  static constexpr bool MOVES = false;
  static constexpr int NHEL = 16;
  // FP64 momenta in every mode (a 4-particle process with no reshuffle: its
  // few FP64 invariants per event are not a bottleneck)
  template <class R>
  using mom_t = double;
  template <class R, int LB = 0>
  static constexpr int jstore_bytes() {
    return 0;
  }
  template <class R>
  static constexpr bool inline_me() {
    return false;
  }

  // sqrt(2E) chi_-(p) and sqrt(2E) chi_+(p): the chiral halves of the spinors
  template <class R>
  struct Weyl {
    cx<R> c[2][2];  // [L, R][component]
  };
  template <class R>
  __device__ __forceinline__ static Weyl<R> weyl(const R (&p)[4]) {
    cx<R> cp[2], cm[2];
    const R pp = chi_pm(p, cp, cm);
    R wp, wm;
    omegas(p[0], pp, R(0), wp, wm);
    return {{{wp * cm[0], wp * cm[1]}, {wp * cp[0], wp * cp[1]}}};
  }
  // row (conjugated) half a of one particle, gamma^mu, half b of another, both
  // of chirality ch (0: L, sigmabar; 1: R, sigma)
  template <class R>
  __device__ __forceinline__ static cv<R> current(const cx<R> (&a)[2], const cx<R> (&b)[2], int ch) {
    const cx<R> u0 = conjg(a[0]), u1 = conjg(a[1]);
    const cx<R> x = cmul(u0, b[0]), y = cmul(u1, b[1]), z = cmul(u0, b[1]), t = cmul(u1, b[0]);
    const R s = ch ? R(1) : R(-1);
    return {{x + y, s * (z + t), s * times_i(t - z), s * (x - y)}};
  }

  // What an event's evaluations have in common (the currents carry no
  // parameter): s and, per chirality configuration of this lane, jo.ji and
  // (k.jo)(k.ji).  With at least four lanes per event lane i < 4 has
  // configuration i, with fewer each lane has 4 >> LB of them.
  template <class R, int LB>
  struct Common {
    static constexpr int N = LB >= 2 ? 1 : 4 >> LB;
    double s;
    cx<R> jj[N], kk[N];
  };
  template <class R, int LB>
  __device__ __forceinline__ static void common(const double (&p)[NEXT][4], int lane, unsigned gmask, Common<R, LB>& c) {
    c.s = 2.0 * dot4(p[0], p[1]);
    R k[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) k[m] = R(p[0][m] + p[1][m]);
    Weyl<R> s[4];
    if constexpr (LB >= 2) {
      const int mine = lane & 3;
      R q[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) q[m] = R(mine == 0 ? p[0][m] : mine == 1 ? p[1][m] : mine == 2 ? p[2][m] : p[3][m]);
      const Weyl<R> own = weyl(q);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const cx<R> v = own.c[h >> 1][h & 1];
          s[i].c[h >> 1][h & 1] = {__shfl_sync(gmask, v.r, i, 4), __shfl_sync(gmask, v.i, i, 4)};
        }
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        R q[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) q[m] = R(p[i][m]);
        s[i] = weyl(q);
      }
    }
#pragma unroll
    for (int n = 0; n < Common<R, LB>::N; ++n) {
      const int h = config<LB>(lane, n), ci = h & 1, co = (h >> 1) & 1;
      const cv<R> ji = current(ci ? s[1].c[1] : s[1].c[0], ci ? s[0].c[1] : s[0].c[0], ci);
      const cv<R> jo = current(co ? s[2].c[1] : s[2].c[0], co ? s[3].c[1] : s[3].c[0], co);
      c.jj[n] = dot(jo, ji);
      c.kk[n] = dotr(k, jo) * dotr(k, ji);
    }
  }
  // chirality of the electron line (bit 0) and of the muon line (bit 1)
  template <int LB>
  __device__ __forceinline__ static int config(int lane, int n) {
    return LB >= 2 ? lane & 3 : lane * (4 >> LB) + n;
  }

  // |M|^2 of one parameter point
  template <class R, int LB>
  __device__ __noinline__ static double point(const Common<R, LB>& c, const PointDev& pt, int lane, unsigned gmask) {
    const R e2s = R(pt.e * pt.e / c.s);
    // 1/(s - MZ^2 + i MZ WZ)
    const double dr = c.s - pt.MZ * pt.MZ, di = pt.MZ * pt.WZ, dn = 1.0 / (dr * dr + di * di);
    const cx<R> dz = {R(dr * dn), R(-di * dn)};
    const R imz2 = R(1.0 / (pt.MZ * pt.MZ));
    R acc = R(0);
#pragma unroll
    for (int n = 0; n < Common<R, LB>::N; ++n) {
      const int h = config<LB>(lane, n);
      const R g = R(((h & 1) ? pt.gR : pt.gL) * ((h & 2) ? pt.gR : pt.gL));
      const cx<R> M = cmac(g * (c.jj[n] - imz2 * c.kk[n]), dz, e2s * c.jj[n]);
      acc += M.r * M.r + M.i * M.i;
    }
    double sum = LB < 3 || lane < 4 ? double(acc) : 0.0;
#pragma unroll
    for (int o = 1; o < (1 << LB); o <<= 1) sum += __shfl_xor_sync(gmask, sum, o);
    return 0.25 * sum;
  }

  template <class R, int LB>
  __device__ __noinline__ static double me(const double (&p)[NEXT][4], const PointDev& pt, int lane,
                                           unsigned gmask) {
    Common<R, LB> c;
    common<R, LB>(p, lane, gmask, c);
    return point<R, LB>(c, pt, lane, gmask);
  }
  template <class R>
  __device__ __forceinline__ static bool reshuffle(const double (&p)[NEXT][4], double, double (&q)[NEXT][4]) {
#pragma unroll
    for (int i = 0; i < NEXT; ++i)
#pragma unroll
      for (int m = 0; m < 4; ++m) q[i][m] = p[i][m];
    return true;
  }
};

}  // namespace rw
