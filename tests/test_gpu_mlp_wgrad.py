"""The surrogate's tensor-core backward pass (2,048 rows and more) against the FP64 reference, element by element, and row
by row at the edges of its stages, slices and blocks."""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_07440_gb300 import rwgt  # noqa: E402
from test_gpu_surrogate import emulated_gpu_gradient, gpu_precision_params, gradient_error_scale  # noqa: E402

DEV = torch.device("cuda", 0)


def stream():
    return torch.cuda.current_stream(DEV).cuda_stream


@pytest.mark.parametrize("n_in,layers,B", [(40, 4, 2048), (40, 4, 2111), (40, 4, 16384), (8, 2, 2049), (136, 2, 2113)])
def test_gradient_elementwise(n_in, layers, B):
    """Two bounds per element, as for the small batches: the roundings on a product's path, and, in all but one element of
    a hundred, the FP32 accumulation of B terms with the kernels' rounding points reproduced."""
    rng = np.random.default_rng(B)
    x = rng.normal(size=(B, n_in)).astype(np.float32)
    y = (0.3 * np.sin(x[:, 0]) + 0.1 * x[:, 1] * x[:, 2]).astype(np.float32)
    with rwgt.Mlp(0, stream(), n_in, 256, layers, B, seed=6) as m:
        params = m.get_state()["params"]
        loss, g = m.gradient(torch.from_numpy(x).to(DEV), torch.from_numpy(y).to(DEV), tau=0.3, lam=0.1)
        m.status()
    g = g.astype(np.float64)
    q = gpu_precision_params(params, n_in, 256, layers)
    ref_loss, ref_g = omlp.loss_and_grad(q, x, y, 0.3, 0.1, n_in, 256, layers)
    bound = 2 * (layers + 1) * 2.0 ** -8 * gradient_error_scale(q, x, y, 0.3, 0.1, n_in, 256, layers) + 1e-12
    excess = np.abs(g - ref_g) / bound
    assert excess.max() <= 1.0, f"element {excess.argmax()}: {excess.max():.3f} x the bound"
    assert abs(loss / ref_loss - 1) < 1e-2
    ge, se = emulated_gpu_gradient(q, x, y, 0.3, 0.1, n_in, 256, layers)
    over = np.abs(g - ge) > 8 * B * 2.0 ** -24 * se + 1e-12
    assert over.mean() < 0.01, f"{over.mean():.4f} of the elements beyond the accumulation bound"


@pytest.mark.parametrize("n_in,layers,B", [(40, 4, 2111), (136, 2, 2113), (40, 4, 4097)])
def test_every_row_counts_once(n_in, layers, B):
    """One row at a time carries the gradient (the other rows' residuals are 0, its own is 1e4): a row left out or taken
    twice changes every block's norm by all of it, the roundings on a product's path by 2 (layers + 1) 2^-8."""
    rng = np.random.default_rng(B)
    x = rng.normal(size=(B, n_in)).astype(np.float32)
    dx = torch.from_numpy(x).to(DEV)
    out = torch.empty((B, 2), dtype=torch.float32, device=DEV)
    with rwgt.Mlp(0, stream(), n_in, 256, layers, B, seed=6) as m:
        q = gpu_precision_params(m.get_state()["params"], n_in, 256, layers)
        m.forward(dx, out)
        mu = out[:, 0].cpu().numpy()
        stage, slice_, head = 64, 128, 16
        rows = {0, stage - 1, stage, slice_ - 1, slice_, head - 1, head, 2047, 2048, B - stage, B - 2, B - 1}
        for r in sorted(rows):
            y = mu.copy()
            y[r] += 1e4
            _, g = m.gradient(dx, torch.from_numpy(y).to(DEV), tau=0.3, lam=0.1)
            m.status()
            ge, _ = emulated_gpu_gradient(q, x[r:r + 1], y[r:r + 1], 0.3, 0.1, n_in, 256, layers)
            ge, o = ge / B, 0  # the mean over the batch
            for k, n in omlp.layer_shapes(n_in, 256, layers):
                for size in (k * n, n):
                    a, b = g[o:o + size].astype(np.float64), ge[o:o + size]
                    o += size
                    assert np.linalg.norm(a - b) <= 2 * (layers + 1) * 2.0 ** -8 * np.linalg.norm(b), (r, k, n, size)
