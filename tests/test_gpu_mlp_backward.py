"""The surrogate network's tensor-core backward pass (weight gradients of all layers in one launch, output layer and loss
in one pass) and the row draw inside the input layer, at the edges of their tiles and slices."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_07440_gb300 import rwgt  # noqa: E402

DEV = torch.device("cuda", 0)


def stream():
    return torch.cuda.current_stream(DEV).cuda_stream


def rows(n, n_in, seed):
    g = torch.Generator().manual_seed(seed)
    x = torch.randn(n, n_in, generator=g)
    return x, torch.sin(x[:, 0]) + 0.2 * x[:, 1]


@pytest.mark.parametrize("n_in,layers,B", [(40, 4, 1), (40, 4, 2047), (40, 4, 2048), (8, 2, 2049), (40, 4, 2111), (64, 3, 3000),
                                           (72, 3, 2500), (136, 2, 2113), (40, 4, 4097)])
def test_gradient_matches_the_mma_sync_path(n_in, layers, B):
    """Per parameter block, 2-norms: both paths round the same quantities to BF16 (at most 2 (layers + 1) roundings on a
    product's path, unit 2^-8) and differ where an FP32 sum in another order turns a rounding."""
    x, y = rows(B, n_in, seed=B)
    out = {}
    with rwgt.Mlp(0, stream(), n_in, 256, layers, 4097, seed=6) as m:
        for kind in ("tcgen05", "mma_sync"):
            m.set_gemm(kind)
            out[kind] = m.gradient(x.to(DEV), y.to(DEV), tau=0.3, lam=0.1)
            m.status()
    (la, a), (lb, b) = out["tcgen05"], out["mma_sync"]
    assert abs(la / lb - 1) < 1e-2
    o, dims = 0, [n_in] + [256] * layers + [2]
    for k, n in zip(dims, dims[1:]):
        for size in (k * n, n):
            u, v = a[o:o + size].astype(np.float64), b[o:o + size].astype(np.float64)
            assert np.linalg.norm(u - v) <= 2 * (layers + 1) * 2.0 ** -8 * np.linalg.norm(v), (k, n, size)
            o += size


def splitmix_rows(seed, step, B, n):
    out, M = [], (1 << 64) - 1
    for b in range(B):
        z = (seed + 0x9E3779B97F4A7C15 * (step * 0x100000001 + b + 1)) & M
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M
        out.append(((z ^ (z >> 31)) % n))
    return np.array(out)


def test_training_step_draws_its_rows_and_is_repeatable():
    """One step equals Adam (float64) on the gradient of the rows the counter-based hash draws: the update's FP32
    arithmetic is within a few 2^-24 of the parameter plus 2^-20 of the step.  Two runs agree to the bit."""
    n, B, lr = 5000, 2100, 1e-3
    x, y = rows(n, 40, seed=3)
    dx, dy = x.to(DEV), y.to(DEV)
    got = []
    for _ in range(2):
        with rwgt.Mlp(0, stream(), 40, 256, 4, 4096, seed=2) as m:
            p0 = m.get_state()["params"]
            idx = torch.from_numpy(splitmix_rows(7, 0, B, n))
            _, g = m.gradient(x[idx].to(DEV), y[idx].to(DEV), 0.3, 0.1)
            m.train(dx, dy, B, 1, lr, 0.3, 0.1, seed=7)
            one = m.get_state()["params"]
            m.train(dx, dy, B, 4, lr, 0.3, 0.1, seed=7)
            got.append(m.get_state())
    g = g.astype(np.float64)
    want = p0 - lr * g / (np.abs(g) + 1e-8)  # the first step: both moments bias-corrected
    assert np.all(np.abs(one - want) <= 2.0 ** -22 * np.abs(p0) + 2.0 ** -12 * lr)
    assert np.array_equal(got[0]["params"], got[1]["params"]) and np.array_equal(got[0]["m2"], got[1]["m2"])


@pytest.mark.parametrize("n_in", [8, 24, 40])
@pytest.mark.parametrize("shift", [0, 1])
def test_inference_features_of_every_width_and_alignment(n_in, shift):
    """The split features are written in 16-byte chunks with the rest of the last k-block zero, from rows at any address:
    against the layer-by-layer path (FP32 input layer), which differs by the dropped 2^-16 product and where it turns a
    BF16 rounding of an activation."""
    n = 128 * 3 + 5
    x, _ = rows(n, n_in, seed=n_in)
    flat = torch.zeros(n * n_in + 4, device=DEV)
    flat[shift:shift + n * n_in] = x.reshape(-1).to(DEV)
    xs = flat[shift:shift + n * n_in].view(n, n_in)
    outs = []
    with rwgt.Mlp(0, stream(), n_in, 256, 2, 4096, seed=8) as m:
        for kind in ("tcgen05", "tcgen05_layers"):
            o = torch.empty(n, 2, device=DEV)
            m.set_gemm(kind)
            m.forward(xs if kind == "tcgen05" else x.to(DEV), o)
            m.status()
            outs.append(o.cpu().numpy().astype(np.float64))
    d = np.abs(outs[0] - outs[1]) / np.std(outs[1], axis=0)
    assert d.max() < 2e-2 and np.median(d) < 1e-4
