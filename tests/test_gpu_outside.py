"""Events outside a point's phase space have weight 0 whatever the point's coupling, also where its power overflows."""
import numpy as np
import pytest

from paper_2312_07440_gb300 import events as ev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_07440_gb300 import rwgt  # noqa: E402

DEV = torch.device("cuda", 0)
E = 70
HEAVY = np.stack([ev.param_vector(m_t=1e5, alpha_s=1e200), ev.param_vector(m_t=1e5), ev.param_vector(alpha_s=0.12)])


def inputs(wl):
    mom, w = ev.generate(ev.WORKLOADS[wl], E)
    return torch.from_numpy(mom).to(DEV), torch.from_numpy(w).to(DEV), w


def check(wnew, sigma, n_bad):
    assert np.all(wnew[:2] == 0.0) and np.all(np.asarray(sigma[:2]) == 0.0) and n_bad == 0
    assert np.all(wnew[2] != 0.0)


@pytest.mark.parametrize("mode", ["fp64", "fp32", "mixed_fp16", "mixed_bf16"])
@pytest.mark.parametrize("proc,wl,lane_bits", [("gg_tt", "gg_tt_1m", -1), ("gg_ttg", "gg_ttg_4m", -1),
                                               ("gg_ttgg", "gg_ttgg_1m", 1), ("gg_ttgg", "gg_ttgg_1m", -1)])
def test_reweight(proc, wl, lane_bits, mode):
    dm, dw, _ = inputs(wl)
    g = rwgt.reweight(proc, mode, dm, dw, ev.param_vector(), HEAVY, lane_bits=lane_bits)
    torch.cuda.synchronize()
    check(g["wnew"].cpu().numpy(), g["sigma"], g["n_bad"])


def test_one_launch_of_two_processes():
    keep, outs = [], []
    st = torch.cuda.current_stream(DEV).cuda_stream
    with rwgt.Multi(0, st) as m:
        for proc, wl in (("gg_tt", "gg_tt_1m"), ("gg_ttg", "gg_ttg_4m")):
            dm, dw, _ = inputs(wl)
            c = rwgt.Context(0, st)
            c.set_process(proc, "fp64")
            c.set_params(ev.param_vector())
            c.set_reweight_points(HEAVY)
            nb = c.workspace_bytes(E)
            ws = torch.empty(nb, dtype=torch.uint8, device=DEV)
            c.load_events(dm, dw, E, ws, nb)
            out = torch.empty((3, E), dtype=torch.float64, device=DEV)
            m.add(c, out)
            keep += [c, dm, dw, ws]
            outs.append((c, out))
        mb = m.workspace_bytes()
        mws = torch.empty(mb, dtype=torch.uint8, device=DEV)
        m.reweight_async(mws, mb)
        torch.cuda.synchronize()
        for c, out in outs:
            sig, _, nbad, _ = c.get_results(3)
            check(out.cpu().numpy(), sig, nbad)
