"""Build-time generator of the tables of the warp-per-event amplitude code for g g -> t tbar g g (csrc/qcd_coop.cuh).

One warp evaluates one event: every off-shell current is formed once per helicity configuration it depends on, as
a list of tasks dealt out to the lanes, and kept in shared memory.  With gluons 0..3, v the antitop spinor, ub the
top's row spinor and J(s) the gluon current of the ordered sequence s,

  S(b)  = prop J_b v,      S(cd) = prop (J_c S(d) + J(cd) v),
  T(a)  = (ub J_a) prop,   T(ab) = T(a) J_b + ub J(ab),
  A(abcd) = T(ab).S(cd) + T(a) J(bc) S(d) + (ub J(abc)).S(d) + T(a).(J(bcd) v) + (ub gamma v).J(abcd)

(the fermion line is cut between its second and third gluon, so no spinor with three gluons is ever formed).  The
gluon currents obey J(reversed) = (-1)^(L+1) J and vanish on shuffles, so of a set's L! orders only (L-1)! are
independent; the others are signed sums of at most three of them.

Colour: C_st depends only on s^-1 t, so it commutes with relabelling the gluons (0 1), (2 3) and with reversing the
orderings.  In the common characters of these three involutions the 24 x 24 form falls into four 4 x 4 and four
2 x 2 blocks, each then a sum of squares (L D L^T, exact rationals).

Run ``python -m paper_2312_07440_gb300.gen.coop_gen`` to regenerate ``csrc/gen_coop_gg_ttgg.cuh``.
"""
from __future__ import annotations

import itertools
import os
from fractions import Fraction

from . import qcd_gen

N = 4
ORDERS = qcd_gen.orderings(N)
PAIRS = [(0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3)]
SETS = [(0, 1, 2), (0, 1, 3), (0, 2, 3), (1, 2, 3)]
PERMS = list(itertools.permutations((1, 2, 3)))  # J4 is formed for (0,) + each


def bits(fields):
    """Pack (value, width) fields, lowest first."""
    o = at = 0
    for v, w in fields:
        assert 0 <= v < (1 << w), (v, w)
        o |= v << at
        at += w
    assert at <= 32
    return o


# --- object indices (h: helicity bits of gluons 0..3, h[0] = 0) -------------------------------------------------
def e_idx(g, h):
    return 0 if g == 0 else 1 + 2 * (g - 1) + h[g]


def j2_idx(a, b, h):
    """(index, negative) of J(ab)."""
    x, y = min(a, b), max(a, b)
    p = PAIRS.index((x, y))
    return (2 * p + h[y] if x == 0 else 6 + 4 * (p - 3) + 2 * h[x] + h[y]), int(a > b)


N_J2 = 18
# basis orders of three gluons: two per set with gluon 0, three for (1, 2, 3) (the third only feeds J4)
J3_ORDERS = [(t, o, s) for t, st in enumerate(SETS)
             for o, s in enumerate([st, (st[0], st[2], st[1])] + ([(2, 1, 3)] if t == 3 else []))]


def j3_idx(t, o, h):
    x, y, z = SETS[t]
    return t * 8 + o * 4 + 2 * h[y] + h[z] if x == 0 else 24 + o * 8 + 4 * h[1] + 2 * h[2] + h[3]


N_J3 = 48


def j3_of(seq, h):
    """Index of J(seq) for a sequence that is, up to reversal (sign +), a basis order."""
    for t, o, s in J3_ORDERS:
        if s in (seq, seq[::-1]):
            return j3_idx(t, o, h)
    raise KeyError(seq)


def ee_idx(a, b, h):
    """Index of E_a.E_b among the products."""
    return j2_idx(a, b, h)[0]


def ej_idx(i, j, k, h):
    """Index of E_i.J(jk) among the products, up to the sign of the order j, k (as j2_idx)."""
    st = tuple(sorted((i, j, k)))
    t, w = SETS.index(st), st.index(i)
    hh = 2 * h[st[1]] + h[st[2]] if t < 3 else 4 * h[1] + 2 * h[2] + h[3]
    return N_J2 + 12 * t + (4 if t < 3 else 8) * w + hh


def x1_idx(g, h, lam):
    """S(g) or T(g) within its 14 spinors."""
    return lam if g == 0 else 2 + (g - 1) * 4 + h[g] * 2 + lam


def hels(gs):
    """Helicity assignments of the gluons gs (gluon 0 fixed), last gluon fastest."""
    free = [g for g in gs if g]
    for v in itertools.product((0, 1), repeat=len(free)):
        h = [0, 0, 0, 0]
        for g, x in zip(free, v):
            h[g] = x
        yield h


def tasks():
    """Task words of every phase, in the order of the objects they write."""
    out = {}
    # J(ab): E_a, E_b, gluons a, b
    out["J2"] = [bits([(e_idx(a, h), 3), (e_idx(b, h), 3), (a, 2), (b, 2)]) for a, b in PAIRS for h in hels((a, b))]
    # products of currents that several three- and four-gluon currents need: E_a.E_b, then E_i.J(jk):
    # E, whether the other is a J, its index
    d = {}
    for a, b in PAIRS:
        for h in hels((a, b)):
            d[ee_idx(a, b, h)] = bits([(e_idx(a, h), 3), (0, 1), (e_idx(b, h), 5)])
    for st in SETS:
        for i in st:
            j, k = [g for g in st if g != i]
            for h in hels(st):
                d[ej_idx(i, j, k, h)] = bits([(e_idx(i, h), 3), (1, 1), (j2_idx(j, k, h)[0], 5)])
    assert sorted(d) == list(range(len(d)))
    out["DOT"] = [d[i] for i in range(len(d))]
    # J(abc), two words: E_a, E_b, E_c, J(ab), sign, J(bc), sign, gluons | products ab, bc, ac, a.bc, c.ab
    j3, j3b = {}, {}
    for t, o, (a, b, c) in J3_ORDERS:
        for h in hels(SETS[t]):
            (ab, sab), (bc, sbc) = j2_idx(a, b, h), j2_idx(b, c, h)
            j3[j3_idx(t, o, h)] = bits([(e_idx(a, h), 3), (e_idx(b, h), 3), (e_idx(c, h), 3), (ab, 5), (sab, 1), (bc, 5),
                                        (sbc, 1), (a, 2), (b, 2), (c, 2)])
            j3b[j3_idx(t, o, h)] = bits([(ee_idx(a, b, h), 5), (ee_idx(b, c, h), 5), (ee_idx(a, c, h), 5),
                                         (ej_idx(a, b, c, h), 7), (ej_idx(c, a, b, h), 7)])
    assert sorted(j3) == list(range(N_J3))
    out["J3"], out["J3B"] = [j3[i] for i in range(N_J3)], [j3b[i] for i in range(N_J3)]
    # J(0bcd), four words: E_b, E_c, E_d, J(0b), J(bc), sign, J(cd), sign, gluons b, c | J(0bc), J(bcd), gluon d |
    # products 0b, 0d, cd, d.bc, 0.bc | b.cd, 0.cd, c.0b, d.0b
    lo, hi, pc, pd = [], [], [], []
    for b, c, d in PERMS:
        for h in hels((1, 2, 3)):
            (ob, _), (bc, sbc), (cd, scd) = j2_idx(0, b, h), j2_idx(b, c, h), j2_idx(c, d, h)
            lo.append(bits([(e_idx(b, h), 3), (e_idx(c, h), 3), (e_idx(d, h), 3), (ob, 5), (bc, 5), (sbc, 1), (cd, 5),
                            (scd, 1), (b, 2), (c, 2)]))
            hi.append(bits([(j3_of((0, b, c), h), 6), (j3_of((b, c, d), h), 6), (d, 2)]))
            pc.append(bits([(ee_idx(0, b, h), 5), (ee_idx(0, d, h), 5), (ee_idx(c, d, h), 5), (ej_idx(d, b, c, h), 7),
                            (ej_idx(0, b, c, h), 7)]))
            pd.append(bits([(ej_idx(b, c, d, h), 7), (ej_idx(0, c, d, h), 7), (ej_idx(c, 0, b, h), 7),
                            (ej_idx(d, 0, b, h), 7)]))
    out["J4"], out["J4B"], out["J4C"], out["J4D"] = lo, hi, pc, pd
    # S(g), then T(g): E, spinor (0, 1 v; 2, 3 ub), propagator mask
    x1 = [None] * 28
    for side in (0, 1):
        for g in range(4):
            for h in hels((g,)):
                for lam in (0, 1):
                    m = (15 ^ (1 << g)) if side else 1 << g
                    x1[14 * side + x1_idx(g, h, lam)] = bits([(e_idx(g, h), 3), (2 * side + lam, 2), (m, 4)])
    out["X1"] = x1
    # (ub J(abc)) and (J(abc) v): J3, spinor; sets with gluon 0 (96), then (1, 2, 3) (64)
    r = []
    for t in range(4):
        for kind in (0, 1):  # 0: ub, 1: v
            for o in (0, 1):
                for lam in (0, 1):
                    for h in hels(SETS[t]):
                        r.append(bits([(j3_idx(t, o, h), 6), (lam + (2 if kind == 0 else 0), 2)]))
    out["R3"] = r
    # J(bc) S(d), grouped by the remaining gluon a = 0 (48), 1, 2, 3 (24 each): J2, S
    y = []
    for a in range(4):
        rest = [g for g in range(4) if g != a]
        for d in rest:
            b, c = [g for g in rest if g != d]
            for lam in (0, 1):
                for h in hels(rest):
                    y.append(bits([(j2_idx(b, c, h)[0], 5), (x1_idx(d, h, lam), 4)]))
    out["Y"] = y
    # T(ab) and S(cd): E of the outer gluon, one-gluon spinor (S 0..13, T 14..27), J2, sign, spinor, propagator mask
    x2 = []

    def side_tasks(pair, side):
        for o in (0, 1):
            s = pair if o == 0 else pair[::-1]
            outer, inner = (s[1], s[0]) if side else s
            for lam in (0, 1):
                for h in hels(pair):
                    j, neg = j2_idx(*s, h)
                    x2.append(bits([(e_idx(outer, h), 3), (14 * side + x1_idx(inner, h, lam), 5), (j, 5), (neg, 1),
                                    (2 * side + lam, 2), ((1 << s[0]) | (1 << s[1]), 4)]))

    for group in (PAIRS[:2], PAIRS[2:3]):  # {01|23, 02|13}, then {03|12}
        for side in (1, 0):
            for p in group:
                side_tasks(p, side)
            for p in group:
                side_tasks(tuple(g for g in range(4) if g not in p), side)
    out["X2"] = x2
    assert [len(out[k]) for k in ("J2", "J3", "J4", "X1", "R3", "Y", "X2")] == [18, 48, 48, 28, 160, 120, 144]
    return out


# --- the combination of a lane's amplitudes ---------------------------------------------------------------------
# lane = 16 lt + 8 lb + 4 h1 + 2 h2 + h3; every entry below is (work-object index as a C++ expression, ...)
def hx(gs):
    """C++ expression of the helicity index of the gluons gs (last fastest)."""
    free = [g for g in gs if g]
    return " + ".join(f"{1 << (len(free) - 1 - i)} * h{g}" if i < len(free) - 1 else f"h{g}" for i, g in enumerate(free)) or "0"


def x1_expr(g, lam):
    return lam if g == 0 else f"{2 + (g - 1) * 4} + 2 * h{g} + {lam}"


def steps():
    """[(phase, [(left spinor, right spinor, [(ordering, sign)])])]: a dot product left.right added to amplitudes;
    spinors are ("w", expr) work objects, ("s", expr) S(g), ("t", expr) T(g)."""
    def oi(s):
        return ORDERS.index(tuple(s))

    ph = []
    for part in (range(3), range(3, 4)):
        dots = []
        for t in part:
            x, y, z = SETS[t]
            d = 6 - x - y - z
            nh = 4 if t < 3 else 8
            base = 32 * t if t < 3 else 0
            for kind, lam in ((0, "lt"), (1, "lb")):
                for o in (0, 1):
                    w = ("w", f"{base + kind * 4 * nh + o * 2 * nh} + {nh} * {lam} + {hx(SETS[t])}")
                    plus = [(x, y, z), (z, y, x)] if o == 0 else [(x, z, y), (y, z, x)]
                    minus = [(y, x, z), (z, x, y)]
                    if kind == 0:  # ub J(abc) . S(d)
                        tg = [(oi(s + (d,)), 1) for s in plus] + [(oi(s + (d,)), -1) for s in minus]
                        dots.append((w, ("s", x1_expr(d, "lb")), tg))
                    else:
                        tg = [(oi((d,) + s), 1) for s in plus] + [(oi((d,) + s), -1) for s in minus]
                        dots.append((("t", x1_expr(d, "lt")), w, tg))
        ph.append(("R3", dots))
    for group in ((0, 1, 2), (3,)):
        dots, base = [], 0
        for a in group:
            rest = [g for g in range(4) if g != a]
            nh = 8 if a == 0 else 4
            for k, d in enumerate(rest):
                b, c = [g for g in rest if g != d]
                w = ("w", f"{base + k * 2 * nh} + {nh} * lb + {hx(rest)}")
                dots.append((("t", x1_expr(a, "lt")), w, [(oi((a, b, c, d)), 1), (oi((a, c, b, d)), -1)]))
            base += 6 * nh
        ph.append(("Y", dots))
    for group in (PAIRS[:2], PAIRS[2:3]):
        dots, at, base = [], {}, 0
        for side in (1, 0):
            for p in group:
                at[side, p] = (base, 2)
                base += 8
            for p in group:
                at[side, tuple(g for g in range(4) if g not in p)] = (base, 4)
                base += 16

        def ob(side, s):
            p = tuple(sorted(s))
            o, nh = at[side, p]
            return ("w", f"{o + (0 if s == p else 2 * nh)} + {nh} * {'lt' if side else 'lb'} + {hx(p)}")

        for p in group:
            q = tuple(g for g in range(4) if g not in p)
            for l, r in ((p, q), (q, p)):
                for s in (l, l[::-1]):
                    for u in (r, r[::-1]):
                        dots.append((ob(1, s), ob(0, u), [(oi(s + u), 1)]))
        ph.append(("X2", dots))
    return ph


def w_terms():
    """{ordering: [(PERMS index, sign)]} of (ub gamma v).J(abcd)."""
    out = {}
    pi = {p: i for i, p in enumerate(PERMS)}
    for k, s in enumerate(ORDERS):
        at = s.index(0)
        r = tuple(g for g in s if g)
        if at == 0:
            out[k] = [(pi[r], 1)]
        elif at == 3:
            out[k] = [(pi[r[::-1]], -1)]
        else:
            a, b, c = r if at == 1 else r[::-1]
            sg = -1 if at == 1 else 1
            out[k] = [(pi[x], sg) for x in ((a, b, c), (b, a, c), (b, c, a))]
    return out


def colour_blocks():
    """[(rows, L, D)]: a block's characters as {ordering: +-1} rows, and the block of C_int in them as L D L^T
    (z = sum over blocks and i of D_i |b_i + sum_{j > i} L_ij b_j|^2)."""
    C, _ = qcd_gen.colour_matrix_int(N)

    def act(gen, s):
        if gen == 2:
            return s[::-1]
        sw = {0: 1, 1: 0} if gen == 0 else {2: 3, 3: 2}
        return tuple(sw.get(g, g) for g in s)

    blocks = []
    for ch in itertools.product((1, -1), repeat=3):
        rows, seen = [], set()
        for s in ORDERS:
            if s in seen:
                continue
            row = {}
            for e in itertools.product((0, 1), repeat=3):
                x, c = s, 1
                for g in range(3):
                    if e[g]:
                        x, c = act(g, x), c * ch[g]
                seen.add(x)
                row[ORDERS.index(x)] = row.get(ORDERS.index(x), 0) + c
            if any(row.values()):
                m = max(abs(v) for v in row.values())
                rows.append({k: v // m for k, v in row.items()})
        # A = sum_rows b_row row / |row|^2 in this sector: the form in b
        n = len(rows)
        M = [[Fraction(sum(C[i][j] * vi * vj for i, vi in rows[p].items() for j, vj in rows[q].items()),
                       len(rows[p]) * len(rows[q])) for q in range(n)] for p in range(n)]
        L, D = [[Fraction(0)] * n for _ in range(n)], []
        for i in range(n):
            D.append(M[i][i])
            for j in range(i + 1, n):
                L[i][j] = M[i][j] / M[i][i]
            for p in range(i + 1, n):
                for q in range(i + 1, n):
                    M[p][q] -= D[i] * L[i][p] * L[i][q]
        blocks.append((rows, L, D))
    return blocks


def flops_per_evaluation():
    """Floating-point operations of one helicity and colour sum (FMA = 2; the set-up is not counted)."""
    F = qcd_gen.FLOPS
    t = {k: len(v) for k, v in tasks().items()}
    n = 4 * F["fcur"] + t["J2"] * F["current2"] + t["DOT"] * F["dot"]
    n += t["J3"] * (F["current3"] - 5 * F["dot"])
    # four gluons: three more products, six momentum products, nine currents and three momenta combined, four
    # products with the quark line's current
    n += t["J4"] * (3 * F["dot"] + 6 * 16 + 20 + 9 * 32 + 40 + 4 * (F["dot"] + 2))
    n += t["X1"] * (F["slash"] + F["fprop"]) + (t["R3"] + t["Y"]) * F["slash"]
    n += t["X2"] * (2 * F["slash"] + F["sp_add"]) + t["X2"] // 2 * F["fprop"]
    lane = sum(F["rowcol"] + 2 * len(tg) for _, dots in steps() for _, _, tg in dots)
    lane += sum(2 * (len(v) - 1) for v in w_terms().values())
    lane += 2 * 2 * (8 * 3 + 4 * 2)  # butterflies: two orbits of eight, two of four
    for rows, L, D in colour_blocks():
        lane += sum(4 for r in L for x in r if x) + 5 * len(D)
    return n + 32 * lane


def emit():
    lines = []
    w = lines.append
    w("// ---- generated by gen/coop_gen.py, do not edit ----")
    w("// Task words, amplitude combination and colour sum of the warp-per-event g g -> t tbar g g code (qcd_coop.cuh).")
    w("#pragma once")
    w('#include "helas.cuh"')
    w("")
    w("namespace rw { namespace coop {")
    T = tasks()
    at = 0
    words = []
    for k in ("J2", "DOT", "J3", "J3B", "J4", "J4B", "J4C", "J4D", "X1", "R3", "Y", "X2"):
        w(f"constexpr int TW_{k} = {at}, N_{k} = {len(T[k])};")
        words += T[k]
        at += len(T[k])
    w(f"constexpr int N_WORDS = {at};")
    w("static __device__ const unsigned TASK_WORDS[N_WORDS] = {")
    for i in range(0, at, 12):
        w("    " + ", ".join(f"{x:#x}u" for x in words[i:i + 12]) + ",")
    w("};")
    w("")
    w("// (ub gamma v).J(abcd) of every ordering from the six W = (ub gamma v).J(0 pi)")
    w("template <class R>")
    w("__device__ __forceinline__ void from_w(const cx<R> (&W)[6], cx<R> (&A)[24]) {")
    for k, terms in w_terms().items():
        e = ("-" if terms[0][1] < 0 else "") + f"W[{terms[0][0]}]"
        for i, sg in terms[1:]:
            e += f" {'+' if sg > 0 else '-'} W[{i}]"
        w(f"  A[{k}] = {e};  // {ORDERS[k]}")
    w("}")
    for i, (name, dots) in enumerate(steps()):
        part = i % 2
        w("")
        w(f"// phase {name}, part {part}: left.right products of the stored spinors added to the amplitudes")
        w("template <class R, class M>")
        w(f"__device__ __forceinline__ void add_{name.lower()}_{part}(const M& m, int lt, int lb, int h1, int h2, int h3, "
          "cx<R> (&A)[24]) {")
        for (lk, le), (rk, re), tg in dots:
            op = f"ts_dot<R>(m.{lk}({le}), m.{rk}({re}))"
            if len(tg) == 1:
                w(f"  A[{tg[0][0]}] = ts_mac<R>(m.{lk}({le}), m.{rk}({re}), A[{tg[0][0]}]);")
                continue
            w(f"  {{ const cx<R> d = {op};")
            w("    " + " ".join(f"A[{k}] = A[{k}] {'+' if sg > 0 else '-'} d;" for k, sg in tg) + " }")
        w("}")
    w("")
    w("// sum_st Cint_st Re(A_s^* A_t)")
    w("template <class R>")
    w("__device__ __forceinline__ R colour_sum(const cx<R> (&A)[24]) {")
    w("  R acc[4] = {R(0), R(0), R(0), R(0)};")
    # butterflies: the three involutions on every orbit
    blocks = colour_blocks()
    done = set()
    name = {}
    for s in ORDERS:
        if s in done:
            continue
        sw = [lambda x: tuple({0: 1, 1: 0}.get(g, g) for g in x), lambda x: tuple({2: 3, 3: 2}.get(g, g) for g in x),
              lambda x: x[::-1]]
        gens = [0, 1, 2] if sw[1](sw[0](s)) != s[::-1] else [0, 1]
        cur = {}
        for e in itertools.product((0, 1), repeat=len(gens)):
            x = s
            for g, k in zip(gens, e):
                if k:
                    x = sw[g](x)
            done.add(x)
            cur[e] = f"A[{ORDERS.index(x)}]"
        o = ORDERS.index(s)
        for st in range(len(gens)):
            nxt = {}
            for e in cur:
                if e[st] == 0:
                    e1 = e[:st] + (1,) + e[st + 1:]
                    n0, n1 = (f"b{o}_{st}_" + "".join(map(str, q)) for q in (e, e1))
                    w(f"  const cx<R> {n0} = {cur[e]} + {cur[e1]}, {n1} = {cur[e]} - {cur[e1]};")
                    nxt[e], nxt[e1] = n0, n1
            cur = nxt
        for e, nm in cur.items():  # character of generator g: -1 where e is 1
            ch = [(-1 if k else 1) for k in e]
            if len(gens) == 2:
                ch.append(ch[0] * ch[1])
            name[o, tuple(ch)] = nm
    for q, (ch, (rows, L, D)) in enumerate(zip(itertools.product((1, -1), repeat=3), blocks)):
        b = [name[min(r), ch] for r in rows]
        n = len(rows)
        w(f"  {{  // characters {ch}")
        for i in range(n):
            yr, yi = f"{b[i]}.r", f"{b[i]}.i"
            for j in range(i + 1, n):
                if L[i][j]:
                    c = f"R({L[i][j].numerator}.0 / {L[i][j].denominator}.0)"
                    yr, yi = f"fmadd({c}, {b[j]}.r, {yr})", f"fmadd({c}, {b[j]}.i, {yi})"
            w(f"    const R r{i} = {yr}, i{i} = {yi};")
            w(f"    acc[{q % 4}] = fmadd(R({D[i].numerator}.0 / {D[i].denominator}.0), fmadd(r{i}, r{i}, i{i} * i{i}), acc[{q % 4}]);")
        w("  }")
    w("  return (acc[0] + acc[1]) + (acc[2] + acc[3]);")
    w("}")
    w("}}  // namespace")
    return "\n".join(lines) + "\n"


def main():
    here = os.path.dirname(os.path.abspath(__file__))
    with open(os.path.join(os.path.dirname(here), "csrc", "gen_coop_gg_ttgg.cuh"), "w") as f:
        f.write(emit())


if __name__ == "__main__":
    main()
