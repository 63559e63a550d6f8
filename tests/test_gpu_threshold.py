"""Reweighting to top masses just below the pair threshold of an event: the mass-shell reshuffle's root is tiny there, and
for g g -> t tbar double."""
import numpy as np
import pytest

import oracle
from paper_2312_07440_gb300 import events as ev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_07440_gb300 import rwgt  # noqa: E402
from parity_helpers import TOL, rel  # noqa: E402

DEV = torch.device("cuda", 0)
WORKLOAD = {"gg_tt": "gg_tt_1m", "gg_ttg": "gg_ttg_4m", "gg_ttgg": "gg_ttgg_1m"}
N = {"gg_tt": 48, "gg_ttg": 24, "gg_ttgg": 12}  # events, each with a point of its own


def own_points(proc, distance):
    """Events and, for event j, point j with 1 - 2 m / E = distance."""
    mom, w = ev.generate(ev.WORKLOADS[WORKLOAD[proc]], N[proc], start=2000)
    E = mom[2:, 0].sum(axis=0)
    pts = np.stack([ev.param_vector(m_t=float(0.5 * (1.0 - distance) * x)) for x in E])
    return mom, w, pts


def run(proc, mode, mom, w, pts, lane_bits=-1):
    out = rwgt.reweight(proc, mode, torch.from_numpy(np.ascontiguousarray(mom)).to(DEV), torch.from_numpy(w).to(DEV),
                        ev.param_vector(), pts, lane_bits=lane_bits)
    torch.cuda.synchronize()
    return {k: v.cpu().numpy() if isinstance(v, torch.Tensor) else v for k, v in out.items()}


def own(x):
    return np.diagonal(x)


def oracle_own(proc, mom, w, pts, precision="extended"):
    """The oracle's results for each event at its own point."""
    o = [oracle.reweight(proc, ev.param_vector(), pts[j:j + 1], np.ascontiguousarray(mom[:, :, j:j + 1]), w[j:j + 1],
                         precision=precision) for j in range(len(w))]
    return {k: np.array([x[k][0, 0] for x in o]) for k in ("me", "ratio", "wnew")}


@pytest.mark.parametrize("mode", ["fp64", "fp32"])
@pytest.mark.parametrize("distance", [1e-2, 1e-3, 1e-4, 1e-5, 1e-6])
def test_pair_parity_up_to_threshold(mode, distance):
    mom, w, pts = own_points("gg_tt", distance)
    g = run("gg_tt", mode, mom, w, pts)
    o = oracle_own("gg_tt", mom, w, pts)
    for k in ("me", "ratio", "wnew"):
        assert rel(own(g[k]), o[k]).max() < TOL[mode], k


@pytest.mark.parametrize("mode", ["fp64", "fp32", "mixed_fp16"])
@pytest.mark.parametrize("proc,lane_bits", [("gg_tt", -1), ("gg_ttg", -1), ("gg_ttgg", 2), ("gg_ttgg", -1)])
@pytest.mark.parametrize("distance", [1e-7, 6e-8, 3e-8, 1e-8])
def test_weights_stay_finite_at_threshold(proc, lane_bits, mode, distance):
    """A wrong root there gave momenta, and so weights, of up to 1e90: all weights, and the cross sections, are finite, and
    the events' own points are those of the oracle to 1e-2 (soft gluons and 16-bit colour sums included; for the gluons
    the energies' FP32 rounding does not enter)."""
    mom, w, pts = own_points(proc, distance)
    g = run(proc, mode, mom, w, pts, lane_bits)
    o = oracle_own(proc, mom, w, pts, "fp64")
    assert np.all(np.isfinite(g["wnew"])) and np.all(np.isfinite(g["sigma"])) and g["n_bad"] == 0
    assert rel(own(g["me"]), o["me"]).max() < (0.1 if mode == "mixed_fp16" else 1e-2)


@pytest.mark.parametrize("proc,lane_bits", [("gg_ttg", -1), ("gg_ttgg", 1), ("gg_ttgg", -1)])
@pytest.mark.parametrize("distance", [1e-2, 1e-4])
def test_soft_gluon_parity_near_threshold(proc, lane_bits, distance):
    """FP64.  The gluons' common scale is (E - 2 m) / (their energies) there: the energies' roundings, a few 2^-53 of E,
    enter it divided by distance, and |M|^2 falls as its square per gluon."""
    mom, w, pts = own_points(proc, distance)
    g = run(proc, "fp64", mom, w, pts, lane_bits)
    o = oracle_own(proc, mom, w, pts)
    assert rel(own(g["me"]), o["me"]).max() < TOL["fp64"] + 32 * 2.0 ** -53 / distance
