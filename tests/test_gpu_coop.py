"""The warp-per-event g g -> t tbar g g kernel (32 lanes per event) against the oracle and the per-thread kernels."""
import math

import numpy as np
import pytest

import oracle
from paper_2312_07440_gb300 import events as ev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_07440_gb300 import rwgt  # noqa: E402
from parity_helpers import POINT_SETS, check_against_oracle, rel  # noqa: E402

DEV = torch.device("cuda", 0)
POINTS = POINT_SETS["multi"]()  # three distinct top masses (an odd number of evaluations), two coupling-only points


def run(mode, mom, w, pts, lane_bits=5, block=0):
    out = rwgt.reweight("gg_ttgg", mode, torch.from_numpy(np.ascontiguousarray(mom)).to(DEV),
                        torch.from_numpy(np.ascontiguousarray(w)).to(DEV), ev.param_vector(), pts, lane_bits=lane_bits,
                        block=block)
    torch.cuda.synchronize()
    return {k: v.cpu().numpy() if isinstance(v, torch.Tensor) else v for k, v in out.items()}


@pytest.mark.parametrize("mode", ["fp64", "fp32"])
@pytest.mark.parametrize("n,block", [(1, 0), (2, 256), (33, 32), (197, 0), (197, 64), (197, 256)])
def test_parity_ragged_batches_and_block_sizes(mode, n, block):
    mom, w = ev.generate(ev.WORKLOADS["gg_ttgg_1m"], n)
    o = oracle.reweight("gg_ttgg", ev.param_vector(), POINTS, mom, w)
    g = run(mode, mom, w, POINTS, block=block)
    check_against_oracle(g, o, mode, ("gg_ttgg", POINTS, mom, w), "gg_ttgg_197_multi")
    assert np.all(g["ratio"][-1] == 1.0) and np.all(g["wnew"][-1] == w)  # unchanged point, bitwise
    for j in range(len(POINTS)):
        exact = math.fsum(g["wnew"][j])
        assert abs(g["sigma"][j] - exact) <= 2 * np.spacing(exact)


@pytest.mark.parametrize("mode", ["fp64", "fp32"])
def test_an_evaluation_does_not_depend_on_its_place(mode):
    """The same point alone, beside another, or among many gives the same bits; so does eval_me."""
    mom, w = ev.generate(ev.WORKLOADS["gg_ttgg_1m"], 65, start=400)
    many = np.stack([ev.param_vector(m_t=m) for m in np.linspace(150.0, 200.0, 12)])
    g = run(mode, mom, w, many)
    for j in (0, 5, 11):
        one = run(mode, mom, w, many[j][None])
        assert np.array_equal(one["me"][0], g["me"][j]) and np.array_equal(one["me0"], g["me0"])
    with rwgt.Context(0, torch.cuda.current_stream(DEV).cuda_stream) as c:
        c.set_process("gg_ttgg", mode)
        c.set_params(ev.param_vector())
        c.set_reweight_points(many)
        nb = c.workspace_bytes(65)
        ws = torch.empty(nb, dtype=torch.uint8, device=DEV)
        c.load_events(torch.from_numpy(mom).to(DEV), torch.from_numpy(w).to(DEV), 65, ws, nb)
        me = torch.empty(65, dtype=torch.float64, device=DEV)
        c.eval_me(7, me)
        torch.cuda.synchronize()
    assert np.array_equal(me.cpu().numpy(), g["me"][7])


@pytest.mark.parametrize("mode,tol", [("fp64", 2e-12), ("fp32", 2e-5)])
def test_many_points_and_masses_that_do_not_fit(mode, tol):
    """256 points on 16 masses x 16 couplings, the heaviest masses above some events' energies: W' = 0 there, and the
    per-thread kernel's results (each within its mode's bound of the oracle) elsewhere."""
    pts = np.stack([ev.param_vector(m_t=m, alpha_s=a) for m in np.linspace(160.0, 460.0, 16)
                    for a in np.linspace(0.110, 0.126, 16)])
    mom, w = ev.generate(ev.WORKLOADS["gg_ttgg_1m"], 70, start=2000)
    g, t = run(mode, mom, w, pts, block=128), run(mode, mom, w, pts, lane_bits=2, block=64)
    assert np.array_equal(g["wnew"] == 0, t["wnew"] == 0) and (g["wnew"] == 0).any()
    assert rel(g["wnew"], t["wnew"]).max() < 2 * tol and rel(g["me0"], t["me0"]).max() < tol
    assert g["n_bad"] == t["n_bad"] == 0


@pytest.mark.parametrize("mode", ["fp64", "fp32"])
@pytest.mark.parametrize("P", [64, 70, 256])
def test_default_launch_fits_every_number_of_points(mode, P):
    """Enough events for the largest default block, and up to the most points: the sums of many points leave less room
    beside the warps' memory; the same results as a small block's."""
    n = 16 * torch.cuda.get_device_properties(DEV).multi_processor_count + 3
    mom, w = ev.generate(ev.WORKLOADS["gg_ttgg_1m"], n, start=100)
    pts = np.stack([ev.param_vector(m_t=175.0 if j % 3 else 173.0, alpha_s=0.1 + 1e-4 * j) for j in range(P)])
    g, t = run(mode, mom, w, pts, lane_bits=-1), run(mode, mom, w, pts, block=64)
    assert np.array_equal(g["wnew"], t["wnew"]) and np.array_equal(g["me"], t["me"])


@pytest.mark.parametrize("mode", ["mixed_fp16"])
def test_mixed_amplitude_pass(mode):
    """The amplitude pass of the separate colour sum in the warp-per-event form: the same rounding to 16 bits, so within
    twice the mode's bound of the 8-lane pass, three tiles with a ragged last one, r == 1 for unchanged parameters."""
    C, _ = oracle.colour_matrix(4)
    e = np.linalg.eigvalsh(C)
    b = 2 * (2.0 ** -11 if mode == "mixed_fp16" else 2.0 ** -8) * math.sqrt(e.max() / e.min()) + 1e-5
    mom, w = ev.generate(ev.WORKLOADS["gg_ttgg_1m"], 300, start=50)
    pts = np.stack([ev.param_vector(m_t=180.0), ev.param_vector()])
    o = oracle.reweight("gg_ttgg", ev.param_vector(), pts, mom, w)
    g, t = run(mode, mom, w, pts), run(mode, mom, w, pts, lane_bits=3, block=128)
    assert rel(g["me0"], o["me0"]).max() < b and rel(g["me"], o["me"]).max() < b
    assert rel(g["me"], t["me"]).max() < 2 * b
    assert np.all(g["ratio"][1] == 1.0)
