"""A launch shape chosen for the warp-per-event g g -> t tbar g g kernels (32 lanes, 256 threads), by hand, by the
autotuner, or by feeding rw_get_tuning's answer back, on the calls that run another kernel or carry more points."""
import ctypes

import numpy as np
import pytest

from paper_2312_07440_gb300 import events as ev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_07440_gb300 import rwgt  # noqa: E402

DEV = torch.device("cuda", 0)
E = 300
MOM, W = ev.generate(ev.WORKLOADS["gg_ttgg_1m"], E, start=5000)


def masses(n):
    return np.stack([ev.param_vector(m_t=m) for m in np.linspace(160.0, 190.0, n)])


def calls(mode, tune):
    """Every entry point's W' under a tuning (none: the defaults), from one context."""
    out = {}
    dm, dw = torch.from_numpy(MOM).to(DEV), torch.from_numpy(W).to(DEV)
    with rwgt.Context(0, torch.cuda.current_stream(DEV).cuda_stream) as c:
        c.set_process("gg_ttgg", mode)
        c.set_params(ev.param_vector())
        c.set_reweight_points(masses(2))
        nb = max(c.workspace_bytes(E), c.workspace_bytes_host(E))
        c.set_reweight_points(masses(256))
        nb = max(nb, c.workspace_bytes(E), c.workspace_bytes_host(E))
        ws = torch.empty(nb, dtype=torch.uint8, device=DEV)
        c.set_reweight_points(masses(2))
        c.load_events(dm, dw, E, ws, nb)
        tune(c)
        shape = c.get_tuning()
        for n in (2, 4, 65, 256):
            c.set_reweight_points(masses(n))
            wn = torch.empty((n, E), dtype=torch.float64, device=DEV)
            c.reweight_async(wn)
            torch.cuda.synchronize()
            out[f"device {n}"] = wn.cpu().numpy()
        me = torch.empty(E, dtype=torch.float64, device=DEV)
        c.eval_me(0, me)
        torch.cuda.synchronize()
        out["eval_me"] = me.cpu().numpy()
        if not mode.startswith("mixed"):
            c.set_reweight_points(masses(9))
            wn = torch.empty((9, E), dtype=torch.float64, device=DEV)
            fl = torch.empty(E, dtype=torch.uint8, device=DEV)
            rwgt.reweight_interp(c, 5, 1e-3, wn, fl)
            torch.cuda.synchronize()
            out["interpolation"] = wn.cpu().numpy()
        c.set_reweight_points(masses(2))
        sig = torch.zeros(3, dtype=torch.float64, device=DEV)
        nbad = torch.zeros(1, dtype=torch.int64, device=DEV)
        wn = torch.empty((2, E), dtype=torch.float64, device=DEV)
        fn = rwgt.load().rw_reweight_noalloc
        P = ctypes.c_void_p
        fn.argtypes, fn.restype = [P, P, P, ctypes.c_int64, P, P, P, P], ctypes.c_int
        assert fn(c.h, dm.data_ptr(), dw.data_ptr(), E, wn.data_ptr(), None, sig.data_ptr(), nbad.data_ptr()) == 0
        torch.cuda.synchronize()
        out["noalloc"] = wn.cpu().numpy()
        hm, hw = torch.from_numpy(MOM).pin_memory(), torch.from_numpy(W).pin_memory()
        for n in (2, 256):
            c.set_reweight_points(masses(n))
            ho = torch.empty((n, E), dtype=torch.float64).pin_memory()
            c.reweight_host(hm, hw, E, ho, n, ws, nb)
            out[f"host {n}"] = ho.numpy().copy()
        assert c.get_tuning() == shape
    return out


_REFERENCE = {}


def reference(mode):
    if mode not in _REFERENCE:
        _REFERENCE[mode] = calls(mode, lambda c: None)
    return _REFERENCE[mode]


def same(a, b, tol):
    assert a.keys() == b.keys()
    for k in a:
        # the interpolation's own bound is 1e-3 of the exact ratio
        t = max(tol, 2e-3) if tol and k == "interpolation" else tol
        assert np.all(np.abs(a[k] / b[k] - 1) <= t), k


@pytest.mark.parametrize("mode,lane_bits", [("fp64", 5), ("fp64", -1), ("fp32", 5), ("mixed_fp16", 5)])
def test_256_threads_chosen_for_the_warp_per_event_kernel(mode, lane_bits):
    """Every call runs, on the kernels of the defaults: the same bits (an evaluation does not depend on its place)."""
    same(calls(mode, lambda c: c.set_tuning(lane_bits, 256)), reference(mode), 0.0)


@pytest.mark.parametrize("mode", ["fp64", "fp32", "mixed_fp16"])
def test_the_shape_in_use_can_be_set(mode):
    same(calls(mode, lambda c: c.set_tuning(*c.get_tuning())), reference(mode), 0.0)


@pytest.mark.parametrize("mode,tol", [("fp64", 1e-11), ("fp32", 3e-5), ("mixed_fp16", 1e-2), ("mixed_bf16", 1e-1)])
def test_every_call_runs_after_the_autotuner(mode, tol):
    """Whatever it picks; other lanes are other kernels, within twice the mode's bound of each other per factor of r."""
    same(calls(mode, lambda c: c.autotune(max_events=E)), reference(mode), tol)


@pytest.mark.parametrize("mode", ["mixed_fp16", "mixed_bf16"])
def test_a_block_only_the_separate_colour_pass_takes(mode):
    """(3 bits, 256 threads) fits that pass's amplitude kernel and not the fused one."""
    same(calls(mode, lambda c: c.set_tuning(3, 256)), calls(mode, lambda c: c.set_tuning(3, 128)), 0.0)
