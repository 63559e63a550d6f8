"""The mass-shell reshuffle of the device code (csrc/qcd.cuh, compiled for the host) against 40-digit roots, from the
middle of phase space to the pair threshold."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2312_07440_gb300 import events as ev

mpmath = pytest.importorskip("mpmath")

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2312_07440_gb300", "csrc")
WORKLOAD = {"gg_tt": "gg_tt_1m", "gg_ttg": "gg_ttg_4m", "gg_ttgg": "gg_ttgg_1m"}
SOURCE = """
#include "cuda_runtime.h"
#include "qcd.cuh"
using namespace rw;
template <int N> int f64(const double* p, double m, double* q) {
  double a[N][4], b[N][4];
  memcpy(a, p, sizeof a);
  const int ok = reshuffle_tops<N>(a, m, b);
  memcpy(q, b, sizeof b);
  return ok;
}
template <int N> int f32(const double* p, double m, double* q) {
  df a[N][4], b[N][4];
  for (int i = 0; i < 4 * N; ++i) a[i / 4][i % 4] = df_from_double(p[i]);
  const int ok = reshuffle_tops<N>(a, m, b);
  for (int i = 0; i < 4 * N; ++i) q[i] = (double)b[i / 4][i % 4].hi + b[i / 4][i % 4].lo;
  return ok;
}
extern "C" int reshuffle(int n, int fp32, const double* p, double m, double* q) {
  if (n == 4) return fp32 ? f32<4>(p, m, q) : f64<4>(p, m, q);
  if (n == 5) return fp32 ? f32<5>(p, m, q) : f64<5>(p, m, q);
  return fp32 ? f32<6>(p, m, q) : f64<6>(p, m, q);
}
// the momenta the FP32 modes start from
extern "C" double split(double x) {
  const df v = df_from_double(x);
  return (double)v.hi + v.lo;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("mass_shell")
    src, so = str(d / "shell.cpp"), str(d / "shell.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-w", "-shared", "-fPIC", "-I",
                    os.path.join(HERE, "host_shim"), "-I", CSRC, "-o", so, src], check=True)
    L = ctypes.CDLL(so)
    L.reshuffle.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_void_p, ctypes.c_double, ctypes.c_void_p]
    L.split.argtypes, L.split.restype = [ctypes.c_double], ctypes.c_double
    return L


def exact(p, m):
    """(xi, energies, d(sum of energies)/d xi) of outgoing momenta p [n][4], 40 digits; None: the masses do not fit."""
    mp = mpmath.mp
    E = mp.fsum(mp.mpf(float(v[0])) for v in p)
    p2 = [mp.fsum(mp.mpf(float(c)) ** 2 for c in v[1:]) for v in p]
    ms = [mp.mpf(float(m))] * 2 + [mp.mpf(0)] * (len(p) - 2)
    if sum(ms) >= E:
        return None
    x = mp.mpf(1)
    for _ in range(400):
        e = [mp.sqrt(a * a + x * x * b) for a, b in zip(ms, p2)]
        d = mp.fsum(x * b / c for b, c in zip(p2, e))
        step = (mp.fsum(e) - E) / d
        x = x - step if x > step else x / 2
        if abs(step) <= mp.mpf(10) ** -36 * x:
            break
    return x, [mp.sqrt(a * a + x * x * b) for a, b in zip(ms, p2)], d, E


@pytest.mark.parametrize("distance", [0.3, 1e-2, 1e-3, 1e-4, 1e-5, 1e-6, 1e-7, 6e-8, 1e-8])
@pytest.mark.parametrize("fp32", [0, 1])
@pytest.mark.parametrize("proc", ["gg_tt", "gg_ttg", "gg_ttgg"])
def test_reshuffle_from_phase_space_to_threshold(lib, proc, fp32, distance):
    """Top masses with 1 - 2 m / E = distance.  With u the unit roundoff of the arithmetic (2^-53; double-float: 2^-46, a
    few times 2^-48), every energy carries a few u of E, which xi sees as u E / (xi d sum/d xi); the pair's closed form
    has no such term.  The FP32 modes add the last step's neglected square, 2e-6 squared."""
    mpmath.mp.dps = 40
    n = ev.N_EXTERNAL[proc]
    mom, _ = ev.generate(ev.WORKLOADS[WORKLOAD[proc]], 60, start=int(1e4))
    u = 2.0 ** -46 if fp32 else 2.0 ** -53
    for e in range(mom.shape[-1]):
        p = np.ascontiguousarray(mom[:, :, e])
        if fp32:
            p = np.vectorize(lib.split)(p)
        m = 0.5 * (1.0 - distance) * p[2:, 0].sum()
        m = lib.split(m) if fp32 else m
        want = exact(p[2:], m)
        assert want is not None
        xi, en, d, E = want
        q = np.empty_like(p)
        assert lib.reshuffle(n, fp32, p.ctypes.data, m, q.ctypes.data) == 1
        assert np.all(np.isfinite(q))
        closed = n == 4
        noise = 0.0 if closed else float(E / (xi * d))
        tol = 16 * u * (1.0 + noise) + (4e-12 if fp32 and not closed else 0.0)
        got = np.linalg.norm(q[2:, 1:]) / np.linalg.norm(p[2:, 1:])
        assert abs(got / float(xi) - 1) <= tol, (e, got, float(xi))
        assert abs(mpmath.fsum(mpmath.mpf(float(x)) for x in q[2:, 0]) / E - 1) <= 16 * u + (4e-12 if fp32 and not closed else 0.0)
        for i in range(n - 2):
            assert abs(q[2 + i, 0] - float(en[i])) <= (32 * u + (4e-12 if fp32 and not closed else 0.0)) * float(E)


@pytest.mark.parametrize("ratio", [1.0 + 1e-12, 1.0 + 3e-9, 1.0 + 1e-7, 1.01, 3.0, 1e4])
@pytest.mark.parametrize("fp32", [0, 1])
def test_pair_with_unequal_momenta(lib, fp32, ratio):
    """The pair's closed form outside the centre-of-mass frame (|p2| = ratio |p3|), on both sides of its short form:
    xi and both energies to a few roundings each; in double-float the energies' sum is rounded, which E - 2 m sees as
    u E / (E - 2 m)."""
    mpmath.mp.dps = 40
    rng = np.random.default_rng(5)
    u = 2.0 ** -46 if fp32 else 2.0 ** -53
    for k in range(40):
        p = np.zeros((4, 4))
        for i, size in ((2, 300.0 * ratio), (3, 300.0)):
            v = rng.standard_normal(3)
            p[i, 1:] = size * v / np.linalg.norm(v)
            p[i, 0] = np.hypot(173.0, size)
        if fp32:
            p = np.vectorize(lib.split)(p)
        m = 0.5 * (1.0 - 10.0 ** rng.uniform(-6, -0.01)) * p[2:, 0].sum()
        m = lib.split(m) if fp32 else m
        xi, en, _, E = exact(p[2:], m)
        q = np.empty_like(p)
        assert lib.reshuffle(4, fp32, p.ctypes.data, m, q.ctypes.data) == 1
        got = np.linalg.norm(q[2:, 1:]) / np.linalg.norm(p[2:, 1:])
        tol = 16 * u * (1 + (float(E / (E - 2 * mpmath.mpf(m))) if fp32 else 0.0))
        assert abs(got / float(xi) - 1) <= tol, (k, got, float(xi))
        for i in (0, 1):
            assert abs(q[2 + i, 0] / float(en[i]) - 1) <= 16 * u
