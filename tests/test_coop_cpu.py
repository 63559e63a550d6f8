"""Generated tables of the warp-per-event g g -> t tbar g g code."""
import itertools
import os

import numpy as np

from paper_2312_07440_gb300.gen import coop_gen, qcd_gen


def test_committed_header_matches_the_generator():
    here = os.path.join(os.path.dirname(coop_gen.__file__), "..", "csrc", "gen_coop_gg_ttgg.cuh")
    assert open(here).read() == coop_gen.emit()


def test_colour_blocks_sum_to_the_colour_form():
    C, _ = qcd_gen.colour_matrix_int(4)
    rng = np.random.default_rng(1)
    A = rng.standard_normal(24) + 1j * rng.standard_normal(24)
    z = 0.0
    for rows, L, D in coop_gen.colour_blocks():
        b = [sum(s * A[k] for k, s in r.items()) for r in rows]
        for i in range(len(b)):
            y = b[i] + sum(float(L[i][j]) * b[j] for j in range(i + 1, len(b)))
            z += float(D[i]) * abs(y) ** 2
    want = np.real(np.conj(A) @ np.array(C, dtype=float) @ A)
    assert abs(z / want - 1) < 1e-13


def test_every_product_enters_every_ordering_as_the_cut_line_has_it():
    """Each ordering collects its eight ways of cutting the line into blocks: T(ab).S(cd), one J(bc), one ub J(abc),
    one J(bcd) v, and (three-term where gluon 0 is inside) J(abcd)."""
    count = {}
    for name, dots in coop_gen.steps():
        for _, _, targets in dots:
            for k, _ in targets:
                count[name, k] = count.get((name, k), 0) + 1
    for k, s in enumerate(coop_gen.ORDERS):
        assert count["X2", k] == 1 and count["Y", k] == 1
        # a three-gluon current with its lowest gluon in the middle is a sum of two basis orders
        mid = sum(t.index(min(t)) == 1 for t in (s[:3], s[1:]))
        assert count["R3", k] == 2 + mid
    assert all(len(v) == (1 if coop_gen.ORDERS[k].index(0) in (0, 3) else 3) for k, v in coop_gen.w_terms().items())


def test_colour_matrix_has_the_symmetries_the_blocks_use():
    C, _ = qcd_gen.colour_matrix_int(4)
    idx = {s: i for i, s in enumerate(coop_gen.ORDERS)}
    for f in (lambda s: tuple({0: 1, 1: 0}.get(g, g) for g in s), lambda s: tuple({2: 3, 3: 2}.get(g, g) for g in s),
              lambda s: s[::-1]):
        assert all(C[idx[f(a)]][idx[f(b)]] == C[idx[a]][idx[b]] for a, b in itertools.product(coop_gen.ORDERS, repeat=2))
