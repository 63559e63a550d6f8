"""Points that share an evaluation (they differ in the overall coupling only) give what each gives alone, bit for bit."""
import numpy as np
import pytest

from paper_2312_07440_gb300 import events as ev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_07440_gb300 import rwgt  # noqa: E402

DEV = torch.device("cuda", 0)
QCD = [dict(m_t=175.0), dict(alpha_s=0.12), dict(m_t=170.0, alpha_s=0.11), dict(), dict(m_t=175.0, alpha_s=0.13),
       dict(m_t=170.0)]
QED = [dict(alpha_em_inv=120.0), dict(), dict(alpha_em_inv=140.0), dict(m_t=175.0), dict(alpha_em_inv=120.0)]
EW = [dict(m_Z=92.0), dict(alpha_em_inv=130.0), dict(w_Z=2.6), dict(), dict(m_t=160.0), dict(m_Z=92.0)]


@pytest.mark.parametrize("proc,mode,wl,n,spec", [
    ("gg_tt", "fp64", "gg_tt_1m", 131, QCD), ("gg_tt", "fp32", "gg_tt_1m", 131, QCD), ("gg_tt", "fp32", "gg_tt_1m", 131, QCD[:3]),
    ("gg_ttg", "fp32", "gg_ttg_4m", 67, QCD), ("gg_ttg", "mixed_fp16", "gg_ttg_4m", 67, QCD[:5]),
    ("gg_ttgg", "fp64", "gg_ttgg_1m", 9, QCD), ("ee_5a", "fp32", "ee_5a_1m", 67, QED), ("ee_mumu", "fp64", "ee_mumu_4k", 99, EW)])
def test_points_together_and_alone(proc, mode, wl, n, spec):
    pts = np.stack([ev.param_vector(**d) for d in spec])
    mom, w = (torch.from_numpy(x).to(DEV) for x in ev.generate(ev.WORKLOADS[wl], n))
    g = rwgt.reweight(proc, mode, mom, w, ev.param_vector(), pts)
    for j, d in enumerate(spec):
        one = rwgt.reweight(proc, mode, mom, w, ev.param_vector(), pts[j][None])
        for k in ("wnew", "ratio", "me"):
            assert torch.equal(g[k][j], one[k][0]), (k, d)
        assert torch.equal(g["me0"], one["me0"])
        if not d:
            assert torch.all(g["ratio"][j] == 1.0)
