"""Performance cases: the work a user of the library has it do.

Reweighting calls of every process the library ships in its precision modes (device batches, a host-buffer
batch, the interpolation along a parameter axis), and the surrogate network's inference and training.  Event
samples, energies, cuts and parameter points are those of ``events.WORKLOADS`` and ``events.reweight_points``,
in sizes from a handful of events to about a million; inputs are drawn on the GPU from the seed alone.

Results of the FP64 mode are returned as they are.  The modes with 32-bit amplitudes write weights that carry
seven digits at most, which a program that chose them keeps in 32 bits: ``run`` ends with that conversion there.
"""
import itertools
import math

import numpy as np
import torch

from paper_2312_07440_gb300 import events as ev
from paper_2312_07440_gb300 import rwgt

DEV = "cuda"
SAMPLE = {"ee_mumu": "ee_mumu_4k", "gg_tt": "gg_tt_1m", "gg_ttg": "gg_ttg_4m", "gg_ttgg": "gg_ttgg_1m", "ee_5a": "ee_5a_1m"}
# floating-point operations one evaluation of the coupling-stripped helicity and colour sum cannot do without,
# by the recursions over off-shell currents, every current formed once per helicity it depends on
EVAL_FLOPS = {"ee_mumu": 3.0e3, "gg_tt": 2.2e3, "gg_ttg": 1.9e4, "gg_ttgg": 1.7e5, "ee_5a": 6.5e4}
MLP_IN, MLP_HIDDEN, MLP_LAYERS, MLP_BATCH = 40, 256, 4, 16384
TAU, LAM, LR = 0.5, 0.05, 1e-3


def listed():
    return [
        # a small sample reweighted on its own: launches and the host's share count
        dict(name="ee_mumu fp64 4k", kind="reweight", process="ee_mumu", mode="fp64", events=4096, points=1),
        # a production sample of the simplest QCD process, new top mass and coupling, in both precisions
        dict(name="gg_tt fp64 1M", kind="reweight", process="gg_tt", mode="fp64", events=1 << 20, points=1),
        dict(name="gg_tt fp32 1M", kind="reweight", process="gg_tt", mode="fp32", events=1 << 20, points=1),
        # a top-mass scan of 64 points over a real-emission sample
        dict(name="gg_ttg fp32 scan64", kind="reweight", process="gg_ttg", mode="fp32", events=131072, points=64),
        # a host program's buffers in and out (ragged size), double precision
        dict(name="gg_ttg fp64 host", kind="host", process="gg_ttg", mode="fp64", events=200003, points=2),
        # the costliest process: double precision, single precision (ragged), half-precision colour sum, and few events
        dict(name="gg_ttgg fp64 128k", kind="reweight", process="gg_ttgg", mode="fp64", events=131072, points=1),
        dict(name="gg_ttgg fp32 256k", kind="reweight", process="gg_ttgg", mode="fp32", events=262147, points=1),
        dict(name="gg_ttgg mixed_fp16 64k", kind="reweight", process="gg_ttgg", mode="mixed_fp16", events=65536, points=1),
        # electroweak coupling variations of a five-photon sample
        dict(name="ee_5a fp32 8pt", kind="reweight", process="ee_5a", mode="fp32", events=250000, points=8),
        # the same kind of scan as gg_ttg's, read off an interpolation along the mass axis
        dict(name="gg_ttg fp32 interp64", kind="interp", process="gg_ttg", mode="fp32", events=262144, points=64),
        # the surrogate network: prediction for many (event, point) rows, and a stretch of its training
        dict(name="mlp forward 2M", kind="forward", rows=2097152),
        dict(name="mlp train 16x16384", kind="train", rows=262144, batch=16384, steps=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["reweight"] * 7 + ["host", "interp", "forward", "train"])
    if kind == "forward":
        return dict(kind=kind, rows=_log(rng, 500, 2097152))
    if kind == "train":
        batch = rng.choice([1000, 4096, 8192, 16384])
        return dict(kind=kind, rows=_log(rng, 20000, 262144), batch=batch, steps=rng.randint(4, 16))
    if kind == "interp":
        return dict(kind=kind, process="gg_ttg", mode=rng.choice(["fp32", "fp32", "fp64"]), events=_log(rng, 300, 20000),
                    points=rng.randint(16, 64))
    if kind == "host":
        process, mode = rng.choice([("gg_tt", "fp64"), ("gg_tt", "fp32"), ("gg_ttg", "fp64"), ("gg_ttg", "fp32")])
        return dict(kind=kind, process=process, mode=mode, events=_log(rng, 1000, 200003), points=rng.randint(1, 2))
    process, mode, top = rng.choice([
        ("ee_mumu", "fp64", 1 << 20), ("gg_tt", "fp64", 1 << 20), ("gg_tt", "fp32", 1 << 20), ("gg_ttg", "fp64", 300000),
        ("gg_ttg", "fp32", 1 << 20), ("gg_ttgg", "fp64", 131072), ("gg_ttgg", "fp64", 131072), ("gg_ttgg", "fp32", 262147),
        ("gg_ttgg", "fp32", 262147), ("gg_ttgg", "mixed_fp16", 65536), ("gg_ttgg", "mixed_bf16", 65536), ("ee_5a", "fp32", 250000)])
    points = rng.randint(1, 3) if process != "gg_ttg" and process != "ee_5a" else rng.randint(1, 8)
    return dict(kind=kind, process=process, mode=mode, events=_log(rng, 200, top // max(1, points // 2)), points=points)


# --- inputs ---------------------------------------------------------------------------------------------------------
def _draw_events(wl, n, gen):
    """n phase-space points of the sample (flat RAMBO momenta, massless or on their mass shells) before cuts: [N][4][n]."""
    nf = ev.N_EXTERNAL[wl.process] - 2
    u = torch.rand((4, nf, n), generator=gen, device=DEV, dtype=torch.float64).clamp_min_(1e-300)
    rs = wl.sqrt_s[0] + (wl.sqrt_s[1] - wl.sqrt_s[0]) * torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)
    c, f, e = 2 * u[0] - 1, 2 * math.pi * u[1], -torch.log(u[2] * u[3])
    s = torch.sqrt((1 - c * c).clamp_min(0))
    q3 = torch.stack([e * s * torch.cos(f), e * s * torch.sin(f), e * c], 1)  # [nf][3][n]
    Q0, Q3 = e.sum(0), q3.sum(0)
    M = torch.sqrt(Q0 * Q0 - (Q3 * Q3).sum(0))
    b, x, g = -Q3 / M, rs / M, Q0 / M
    bq = (b[None] * q3).sum(1)
    p3 = x * (q3 + b[None] * (e + bq / (1 + g))[:, None])
    p3 = p3 - p3.mean(0, keepdim=True)
    p2 = (p3 * p3).sum(1)
    m2 = torch.tensor(wl.final_masses, device=DEV, dtype=torch.float64)[:, None] ** 2
    xi = torch.ones(n, device=DEV, dtype=torch.float64)
    for _ in range(60):  # the common momentum scale that puts the energies' sum at rs
        en = torch.sqrt(m2 + xi * xi * p2)
        step = (en.sum(0) - rs) / (xi * p2 / en).sum(0)
        xi = torch.where(step < xi, xi - step, 0.5 * xi)
    p = torch.zeros((nf + 2, 4, n), device=DEV, dtype=torch.float64)
    p[2:, 1:], p[2:, 0] = xi * p3, torch.sqrt(m2 + xi * xi * p2)
    p[0, 0] = p[1, 0] = p[0, 3] = 0.5 * rs
    p[1, 3] = -0.5 * rs
    return p


def _pass(wl, p):
    ok = torch.isfinite(p).all(0).all(0)
    if wl.pt_min > 0:
        q = p[(2 if wl.process == "ee_5a" else 4):]
        pt, phi = torch.hypot(q[:, 1], q[:, 2]), torch.atan2(q[:, 2], q[:, 1])
        eta = torch.asinh(q[:, 3] / pt)
        ok &= (pt > wl.pt_min).all(0)
        if wl.eta_max > 0:
            ok &= (eta.abs() < wl.eta_max).all(0)
        for a, b in itertools.combinations(range(q.shape[0]), 2):
            d = torch.remainder(phi[a] - phi[b] + math.pi, 2 * math.pi) - math.pi
            ok &= torch.hypot(eta[a] - eta[b], d) > wl.dr_min
    return ok


def _events(case, seed):
    wl, n = ev.WORKLOADS[SAMPLE[case["process"]]], case["events"]
    gen = torch.Generator(device=DEV).manual_seed(seed * 1000003 + n)
    got, have = [], 0
    while have < n:
        p = _draw_events(wl, max(4096, int(1.15 * (n - have) * (7 if wl.eta_max else 1.5 if wl.dr_min else 1))), gen)
        got.append(p[:, :, _pass(wl, p)])
        have += got[-1].shape[-1]
    w = torch.exp(torch.randn(n, generator=gen, device=DEV, dtype=torch.float64))
    return torch.cat(got, -1)[:, :, :n].contiguous(), w


def _points(case):
    """The modified parameter points: [P][8]."""
    process, P = case["process"], case["points"]
    k = [0.8 + 0.4 * (i + 0.5) / P for i in range(P)]  # the samples' range of relative top masses
    if process == "ee_mumu":
        return np.stack([ev.param_vector(m_Z=91.1876 + 0.8124 * (i + 1) / P, w_Z=2.6) for i in range(P)])
    if process == "ee_5a":
        return ev.coupling_points(P)
    if process == "gg_tt":
        return np.stack([ev.param_vector(m_t=173.0 + 2.0 * (i + 1), alpha_s=0.120) for i in range(P)])
    return np.stack([ev.param_vector(m_t=(k[i] if P > 1 else 1.2) * ev.M_TOP) for i in range(P)])


def _rows(n, seed):
    """Feature rows like the surrogate's (scaled momenta, a parameter, logarithms) and labels that depend on them."""
    gen = torch.Generator(device=DEV).manual_seed(seed * 1000003 + 7)
    x = torch.randn((n, MLP_IN), generator=gen, device=DEV) * 0.5
    x[:, 0] = torch.rand(n, generator=gen, device=DEV) * 2 - 1
    return x, torch.sin(x[:, 1] + x[:, 2] * x[:, 3]) + 0.3 * x[:, 4] - x[:, 5].abs()


def _network(seed):
    """Parameters and Adam moments as in the middle of a training run."""
    r = np.random.default_rng(seed)
    dims, p = [MLP_IN] + [MLP_HIDDEN] * MLP_LAYERS + [2], []
    for a, b in zip(dims, dims[1:]):
        p += [r.uniform(-1, 1, a * b) * math.sqrt(6 / a) * (0.2 if b == 2 else 0.7), r.uniform(-0.1, 0.1, b)]
    p = np.concatenate(p).astype(np.float32)
    m2 = (1e-4 * (0.5 + r.random(p.size))).astype(np.float32)
    return p, (1e-3 * r.standard_normal(p.size)).astype(np.float32), m2


def _stream():
    return torch.cuda.current_stream().cuda_stream


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] in ("forward", "train"):
        s["x"], s["y"] = _rows(case["rows"], seed)
        s["net"] = _network(seed)
        s["mlp"] = rwgt.Mlp(0, _stream(), n_in=MLP_IN, hidden=MLP_HIDDEN, n_layers=MLP_LAYERS, max_batch=MLP_BATCH)
        s["mlp"].set_state(*s["net"], step=1000)
        s["out"] = torch.empty((case["rows"], 2), device=DEV) if case["kind"] == "forward" else None
        return s
    E, P = case["events"], case["points"]
    mom, w = _events(case, seed)
    c = s["ctx"] = rwgt.Context(0, _stream())
    c.set_process(case["process"], case["mode"])
    c.set_params(ev.param_vector())
    c.set_reweight_points(_points(case))
    if case["kind"] == "host":
        s["mom"], s["w"] = mom.cpu().pin_memory(), w.cpu().pin_memory()
        s["wnew"] = torch.empty((P, E), dtype=torch.float64).pin_memory()
        s["bytes"] = c.workspace_bytes_host(E)
        s["ws"] = torch.empty(s["bytes"], dtype=torch.uint8, device=DEV)
        return s
    s["mom"], s["w"] = mom, w
    s["wnew"] = torch.empty((P, E), dtype=torch.float64, device=DEV)
    nb = c.workspace_bytes(E)
    s["ws"] = torch.empty(nb, dtype=torch.uint8, device=DEV)
    c.load_events(mom, w, E, s["ws"], nb)
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "forward":
        s["mlp"].forward(s["x"], s["out"])
        return {"out": s["out"]}
    if case["kind"] == "train":  # resumes from a checkpoint and leaves the next one
        p, m1, m2 = s["net"]
        s["mlp"].set_state(p, m1, m2, step=1000)
        s["mlp"].train(s["x"], s["y"], case["batch"], case["steps"], LR, TAU, LAM, seed=7)
        got = s["mlp"].get_state()
        return {"params": got["params"], "m1": got["m1"], "m2": got["m2"]}
    c, E, P = s["ctx"], case["events"], case["points"]
    if case["kind"] == "host":
        sig, so, _, _ = c.reweight_host(s["mom"], s["w"], E, s["wnew"], P, s["ws"], s["bytes"])
    elif case["kind"] == "interp":
        got = rwgt.reweight_interp(c, 9, 1e-3, s["wnew"])
        sig, so = got["sigma"], got["sigma_orig"]
    else:
        sig, so, _, _ = c.reweight(P, s["wnew"])
    if case["mode"] == "fp64":
        return {"wnew": s["wnew"], "sigma": sig, "sigma_orig": so}
    return {"wnew": s["wnew"].to(torch.float32), "sigma": sig.astype(np.float32), "sigma_orig": so}


def work(case):
    if case["kind"] in ("forward", "train"):
        dims = [MLP_IN] + [MLP_HIDDEN] * MLP_LAYERS + [2]
        n_par, row = sum(a * b + b for a, b in zip(dims, dims[1:])), 2 * sum(a * b for a, b in zip(dims, dims[1:]))
        if case["kind"] == "forward":
            return {"bytes": 4 * (case["rows"] * (MLP_IN + 2) + n_par), "flops": row * case["rows"]}
        n = case["batch"] * case["steps"]
        return {"bytes": 4 * (n * (MLP_IN + 1) + 6 * n_par), "flops": (3 * row - 2 * MLP_IN * MLP_HIDDEN) * n}
    E, P, N = case["events"], case["points"], ev.N_EXTERNAL[case["process"]]
    out = 8 if case["mode"] == "fp64" else 4
    # the couplings of QED photons factor out of the sum over helicities: one evaluation serves every point
    evals = 1 if case["process"] == "ee_5a" else 10 if case["kind"] == "interp" else P + 1
    return {"bytes": E * (8 * (4 * N + 1) + out * P), "flops": float(E) * evals * EVAL_FLOPS[case["process"]]}


# --- the same results in plain 64-bit torch -------------------------------------------------------------------------
def _shells(p, m):
    """The final state moved onto the mass shells (m, m, 0, ...) at fixed energy by a common momentum scale; whether it fits."""
    q, p2 = p.clone(), (p[2:, 1:] ** 2).sum(1)
    m2 = torch.zeros((p2.shape[0], 1), device=DEV, dtype=torch.float64)
    m2[:2] = m * m
    et = p[2:, 0].sum(0)
    inside, xi = 2 * m < et, torch.ones_like(et)
    for _ in range(60):
        e = torch.sqrt(m2 + xi * xi * p2)
        step = (e.sum(0) - et) / (xi * p2 / e).sum(0)
        xi = torch.where(step < xi, xi - step, 0.5 * xi)
    q[2:, 1:] *= xi
    q[2:, 0] = torch.sqrt(m2 + xi * xi * p2)
    return q, inside


_GAMMA = None


def _gamma():
    """Chiral-basis gamma matrices [4][4][4] (upper index first)."""
    global _GAMMA
    if _GAMMA is None:
        sg = np.array([[[1, 0], [0, 1]], [[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]])
        g = np.zeros((4, 4, 4), complex)
        for m in range(4):
            g[m, :2, 2:], g[m, 2:, :2] = sg[m], (sg[m] if m == 0 else -sg[m])
        _GAMMA = torch.tensor(g, device=DEV)
    return _GAMMA


def _dot(a, b):
    t = a * b
    return t[..., 0, :] - t[..., 1, :] - t[..., 2, :] - t[..., 3, :]


def _matvec(v, s):
    """vslash s for a real vector field v [..., 4, E] and spinors s [..., 4, E]."""
    v0, v1, v2, v3 = (v[..., i, :] for i in range(4))
    a, b = v0 - v3, v0 + v3
    bm, bp = torch.complex(v1, -v2), torch.complex(v1, v2)
    s0, s1, s2, s3 = (s[..., i, :] for i in range(4))
    return torch.stack(torch.broadcast_tensors(a * s2 - bm * s3, b * s3 - bp * s2, b * s0 + bm * s1, a * s1 + bp * s0), -2)


def _colour(n):
    """Tr of the two orderings' products of generators, summed over colours, lexicographic orderings."""
    l = np.zeros((8, 3, 3), complex)
    for k, (i, j) in enumerate([(0, 1), (0, 2), (1, 2)]):
        a = [0, 3, 5][k]
        l[a, i, j] = l[a, j, i] = 1
        l[a + 1, i, j], l[a + 1, j, i] = -1j, 1j
    l[2] = np.diag([1, -1, 0])
    l[7] = np.diag([1, 1, -2]) / math.sqrt(3)
    t, words = l / 2, []
    for o in itertools.permutations(range(n)):
        x = t
        for _ in range(n - 1):
            x = np.einsum("...ij,ajk->...aik", x, t)
        inv = [o.index(g) for g in range(n)]
        words.append(np.transpose(x, inv + [n, n + 1]).reshape(-1))
    return (np.stack(words).conj() @ np.stack(words).T).real


def _qcd_sum(p, m):
    """sum over polarisations and colours of the squared tree amplitude of g g -> t tbar + gluons, g = 1: [E]."""
    E, n = p.shape[-1], p.shape[0] - 2
    k = torch.cat([p[:2], -p[4:]], 0)
    pol = []
    for g in range(n):  # two real transverse polarisations
        v = p[g if g < 2 else g + 2][1:]
        u = v / torch.sqrt((v * v).sum(0))
        ax = torch.zeros_like(u)
        ax.scatter_(0, u.abs().argmin(0, keepdim=True), 1.0)
        e1 = torch.cross(u, ax, dim=0)
        e1 = e1 / torch.sqrt((e1 * e1).sum(0))
        e = torch.zeros((2, 4, E), device=DEV, dtype=torch.float64)
        e[0, 1:], e[1, 1:] = e1, torch.cross(u, e1, dim=0)
        pol.append(e.reshape([2 if i == g else 1 for i in range(n)] + [4, E]))
    P = lambda s: k[list(s)].sum(0)  # noqa: E731
    J = {(g,): pol[g] for g in range(n)}
    for L in range(2, n + 1):
        for s in itertools.permutations(range(n), L):
            if s[::-1] in J:
                J[s] = J[s[::-1]] * (-1) ** (L + 1)
                continue
            o = 0
            for c in range(1, L):
                a, b, Pa, Pb = J[s[:c]], J[s[c:]], P(s[:c]), P(s[c:])
                o = o - a * _dot(2 * Pa + Pb, b)[..., None, :] + b * _dot(2 * Pb + Pa, a)[..., None, :] + (Pa - Pb) * _dot(a, b)[..., None, :]
                for d in range(c + 1, L):
                    a, b, e = J[s[:c]], J[s[c:d]], J[s[d:]]
                    o = o - 2 * b * _dot(a, e)[..., None, :] + a * _dot(b, e)[..., None, :] + e * _dot(a, b)[..., None, :]
            K = P(s)
            J[s] = -o / _dot(K, K) if L < n else -o / (p[2] + p[3])[0].square().sub((p[2] + p[3])[1:].square().sum(0))
    g = _gamma()
    lead = [1] * n

    def mass_states(q, sign):  # spinors spanning (qslash + sign m): columns [2][1...][4][E]
        r = torch.sqrt(2 * (q[0] + m))
        slash = torch.einsum("mij,me->ije", g * torch.tensor([1, -1, -1, -1], device=DEV).reshape(4, 1, 1), q.to(torch.complex128))
        chi = torch.zeros((2, 4, 1), device=DEV, dtype=torch.complex128)
        for i in range(2):
            chi[i, i] = 1 / math.sqrt(2)
            chi[i, 2 + i] = sign / math.sqrt(2)
        out = torch.einsum("ije,hj->hie", slash, chi[..., 0]) + sign * m * chi
        return (out * math.sqrt(2) / r).reshape([2] + lead + [4, E])

    u, v = mass_states(p[2], 1.0), mass_states(p[3], -1.0)
    ub = torch.cat([u[..., 2:, :], u[..., :2, :]], -2).conj().unsqueeze(1)  # [2 top][1 antitop][pol...][4][E]
    S = {(): v.unsqueeze(0)}

    def node(s):
        return sum(_matvec(J[s[:c]], S[s[c:]]) for c in range(1, len(s) + 1))

    for L in range(1, n):
        for s in itertools.permutations(range(n), L):
            x, q = node(s), P(s) - p[3]
            den = _dot(P(s), P(s) - 2 * p[3])
            S[s] = -(_matvec(q, x) + m * x) / den
    A = torch.stack([(ub * node(s)).sum(-2) for s in itertools.permutations(range(n))]).reshape(math.factorial(n), -1, E)
    C = torch.tensor(_colour(n), device=DEV)
    AR, AI = A.real, A.imag
    f = lambda B: (B * torch.einsum("st,the->she", C, B)).sum((0, 1))  # noqa: E731
    return f(AR) + f(AI)


def _mumu(p, q):
    """Spin-averaged e+ e- -> mu+ mu- through photon and Z."""
    alpha, MZ = 1 / q["alpha_em_inv"], q["m_Z"]
    MW2 = 0.5 * MZ * MZ + math.sqrt(0.25 * MZ ** 4 - math.pi * alpha * MZ * MZ / (math.sqrt(2) * q["G_F"]))
    sw2, e2 = 1 - MW2 / MZ ** 2, 4 * math.pi * alpha
    gl, gr = (math.sqrt(e2) * x / math.sqrt(sw2 * (1 - sw2)) for x in (-0.5 + sw2, sw2))
    s, t, u = 2 * _dot(p[0], p[1]), -2 * _dot(p[0], p[2]), -2 * _dot(p[0], p[3])
    chi = 1 / torch.complex(s - MZ * MZ, torch.full_like(s, MZ * q["w_Z"]))
    f = lambda a, b: (e2 / s + a * b * chi).abs().square()  # noqa: E731
    return (f(gl, gl) + f(gr, gr)) * u * u + 2 * f(gl, gr) * t * t


def _reweighted(case, seed):
    mom, w = _events(case, seed)
    process, p0, pts = case["process"], ev.param_vector(), _points(case)
    named = [dict(zip(ev.PARAM_FIELDS, row)) for row in [p0, *pts]]
    wn = torch.empty((len(pts), w.numel()), dtype=torch.float64, device=DEV)
    if process == "ee_5a":
        for j, q in enumerate(named[1:]):
            wn[j] = w * (named[0]["alpha_em_inv"] / q["alpha_em_inv"]) ** 5
        return wn, w
    n = mom.shape[0] - 2
    step = {"gg_ttgg": 4096, "gg_ttg": 32768}.get(process, 1 << 20)
    for a in range(0, w.numel(), step):
        p, me = mom[:, :, a:a + step], []
        for j, q in enumerate(named):
            if process == "ee_mumu":
                me.append(_mumu(p, q))
                continue
            moved, inside = _shells(p, q["m_t"]) if q["m_t"] != named[0]["m_t"] else (p, True)
            v = _qcd_sum(moved, q["m_t"]) * q["alpha_s"] ** n
            me.append(v if inside is True else torch.where(inside, v, torch.zeros_like(v)))
        for j in range(len(pts)):
            wn[j, a:a + step] = w[a:a + step] * me[j + 1] / me[0]
    return wn, w


def _layers(p):
    dims, out, o = [MLP_IN] + [MLP_HIDDEN] * MLP_LAYERS + [2], [], 0
    for a, b in zip(dims, dims[1:]):
        out.append((p[o:o + a * b].reshape(a, b), p[o + a * b:o + a * b + b]))
        o += a * b + b
    return out


def _forward(p, x):
    h = x
    for i, (W, b) in enumerate(_layers(p)):
        h = h @ W + b
        h = torch.nn.functional.silu(h) if i < MLP_LAYERS else h
    return h


def _wrap(x):
    """x modulo 2^64 as the signed 64-bit integer with the same bits."""
    x &= (1 << 64) - 1
    return x - (1 << 64) if x >> 63 else x


def _batch(seed, step, n, rows):
    """The rows of a minibatch: splitmix64's output function of a counter, modulo the number of rows."""
    srl = lambda z, b: (z >> b) & ((1 << (64 - b)) - 1)  # noqa: E731
    z = _wrap(seed + 0x9E3779B97F4A7C15 * (step * 0x100000001 + 1)) + torch.arange(n, device=DEV) * _wrap(0x9E3779B97F4A7C15)
    z = (z ^ srl(z, 30)) * _wrap(0xBF58476D1CE4E5B9)
    z = (z ^ srl(z, 27)) * _wrap(0x94D049BB133111EB)
    z = z ^ srl(z, 31)
    return (((z >> 1) & ((1 << 63) - 1)) % rows * 2 + (z & 1)) % rows


def exact(case, seed):
    if case["kind"] == "forward":
        x, _ = _rows(case["rows"], seed)
        p = torch.tensor(_network(seed)[0], device=DEV, dtype=torch.float64)
        return {"out": torch.cat([_forward(p, c.double()) for c in x.split(131072)])}
    if case["kind"] == "train":
        x, y = _rows(case["rows"], seed)
        p, m1, m2 = (torch.tensor(v, device=DEV, dtype=torch.float64) for v in _network(seed))
        for it in range(case["steps"]):
            idx = _batch(7, 1000 + it, case["batch"], case["rows"])
            q = p.clone().requires_grad_(True)
            out = _forward(q, x[idx].double())
            r, s = y[idx].double() - out[:, 0], out[:, 1].clamp(-16.0, 4.0)
            (r * r / TAU ** 2 + LAM * (0.5 * r.detach() ** 2 * torch.exp(-2 * s) + s)).mean().backward()
            m1, m2 = 0.9 * m1 + 0.1 * q.grad, 0.999 * m2 + 0.001 * q.grad ** 2
            t = 1001 + it
            p = p - LR * (m1 / (1 - 0.9 ** t)) / (torch.sqrt(m2 / (1 - 0.999 ** t)) + 1e-8)
        return {"params": p, "m1": m1, "m2": m2}
    if case["process"] == "gg_ttg" and case["events"] * case["points"] > 10_000_000:
        return None  # too long in plain torch
    wn, w = _reweighted(case, seed)
    return {"wnew": wn, "sigma": wn.sum(1), "sigma_orig": float(w.sum())}
