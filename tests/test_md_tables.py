"""The generated tables of the Hermite engine, run on the CPU as the kernel decodes them (kc, bc,
z1, z2, coefficient polynomials), against the oracle's primitive integrals: every class, two bra
and three ket primitive pairs, so that every contraction step runs more than once."""
import importlib.util
import os

import numpy as np
import pytest

import oracle
from tests.test_schedule_emulation import CLASSES, expected, pair

_spec = importlib.util.spec_from_file_location(
    "gen_md_tables", os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                                  "paper_2009_03559_gb300", "csrc", "gen_md_tables.py"))
gen = importlib.util.module_from_spec(_spec)
_spec.loader.exec_module(gen)
MD = gen.classes()
HERM = [r for n in range(9) for r in gen.monos(n)]


def hermite(Lt, G, rho, PQ, dtype=np.float64):
    """S_r of all orders up to Lt by the kernel's recursion (z, then y, then x)."""
    S = {((0, 0, 0), m): dtype((2 * rho) ** m * G[m]) for m in range(Lt + 1)}
    X = [dtype(v) for v in PQ]
    for r in HERM[1:gen.n_herm(Lt)]:
        ax = 0 if r[0] else (1 if r[1] else 2)
        r1 = tuple(v - (i == ax) for i, v in enumerate(r))
        r2 = tuple(v - 2 * (i == ax) for i, v in enumerate(r))
        for m in range(Lt - sum(r) + 1):
            v = X[ax] * S[r1, m + 1]
            if r1[ax]:
                v = v - dtype(r1[ax]) * S[r2, m + 1]
            S[r, m] = v
    return np.array([S[r, 0] for r in HERM[:gen.n_herm(Lt)]], dtype=dtype)


def weights(p, ea, eb):
    """W_s of a primitive pair."""
    q = ea + eb
    return np.array([(eb / q) ** i * (ea / q) ** j * (0.5 / q) ** (k + h) for k, i, j, h in p.sets])


def coefs(p, AB, sign):
    mono = lambda m: AB[0] ** m[0] * AB[1] ** m[1] * AB[2] ** m[2]  # noqa: E731
    return np.array([sign * sum(v * mono(m) for m, v in d) for d in p.coefs])


def gather(g, T, src, n):
    out = np.zeros(n)
    for r, (off, nt) in enumerate(g.rounds):
        for lane in range(32):
            ws = g.words[off + lane:off + 32 * nt:32]
            v = sum(T[w & 0xFFFF] * src[w >> 16] for w in ws)
            d = g.dst[32 * r + lane]
            if d != 0xFFFF:
                out[d] = v
    return out


def run_tables(c, bra, ket, cen, omega, dtype=np.float64):
    """bra, ket: exponent pairs of the primitive pairs."""
    b, k = gen.PAIRS[c.hi], gen.PAIRS[c.lo]
    A = np.zeros(len(c.bc), dtype)
    for ea, eb in bra:
        p, P, Cab = pair(ea, eb, cen[0], cen[1])
        H = np.zeros(len(c.kc), dtype)
        for ec, ed in ket:
            q, Q, Ccd = pair(ec, ed, cen[2], cen[3])
            rho = p * q / (p + q)
            T = rho * float((P - Q) @ (P - Q))
            G = oracle.gboys(c.Lt, T, omega ** 2 / (omega ** 2 + rho)) if omega > 0 else oracle.boys(c.Lt, T)
            S = hermite(c.Lt, Cab * Ccd / np.sqrt(p + q) * G, rho, P - Q, dtype)
            W = weights(k, ec, ed).astype(dtype)
            H += np.array([W[s] * S[i] for i, s in c.kc], dtype)
        W = weights(b, ea, eb).astype(dtype)
        A += np.array([W[s] * H[h] for h, s in c.bc], dtype)
    A = A.astype(np.float64)
    Tk = coefs(k, cen[2] - cen[3], 1.0)
    Tb = coefs(b, -(cen[0] - cen[1]), (-1.0) ** b.L)
    Y = gather(c.z1, Tk, A, c.n_rows * c.ncd)
    return gather(c.z2, Tb, Y, c.nab * c.ncd)


@pytest.mark.parametrize("ci", range(21), ids=[c.name() for c in MD])
def test_tables_reproduce_oracle_integrals(ci):
    c, os_class = MD[ci], CLASSES[ci]
    rng = np.random.default_rng(500 + ci)
    cen = rng.uniform(-1.5, 1.5, (4, 3))
    omega = 0.11 if ci % 5 else 0.0
    bra, ket = rng.uniform(0.2, 3.0, (2, 2)), rng.uniform(0.2, 3.0, (3, 2))
    got = run_tables(c, bra, ket, cen, omega)
    ref = expected(os_class, [np.array([*e, *f]) for e in bra for f in ket], cen, omega)
    scale = np.abs(ref).max()
    assert np.allclose(got, ref.reshape(-1), rtol=1e-10, atol=1e-12 * scale), (c.name(), np.abs(got - ref.reshape(-1)).max())


@pytest.mark.parametrize("ci", range(21), ids=[c.name() for c in MD])
def test_digest_tasks_make_the_four_blocks(ci):
    """Every term of every sum once: A_ac += v P_bd, A_ad += v P_bc, A_bc += v P_ad, A_bd += v P_ac."""
    c = MD[ci]
    na, nb, nc, nd = c.dims
    rng = np.random.default_rng(ci)
    v = rng.standard_normal(c.dims)
    P = rng.standard_normal((4, 4, 5, 5))  # P[i, j]: block of shells i, j (a, b, c, d = 0 .. 3)
    got = {}
    for e in c.digest.words:
        isb, isd, x, y, u, w, n = e & 1, (e >> 1) & 1, (e >> 2) & 7, (e >> 5) & 7, (e >> 8) & 7, (e >> 11) & 7, e >> 14
        acc = 0.0
        for _ in range(n):
            a, b = (u, x) if isb else (x, u)
            cc, d = (w, y) if isd else (y, w)
            acc += v[a, b, cc, d] * P[0 if isb else 1, 2 if isd else 3][u, w]
            w += 1
            if w == (nc if isd else nd):
                u, w = u + 1, 0
        if n:
            got[isb, isd, x, y] = got.get((isb, isd, x, y), 0.0) + acc
    want = {(0, 0): np.einsum("abcd,bd->ac", v, P[1, 3][:nb, :nd]), (0, 1): np.einsum("abcd,bc->ad", v, P[1, 2][:nb, :nc]),
            (1, 0): np.einsum("abcd,ad->bc", v, P[0, 3][:na, :nd]), (1, 1): np.einsum("abcd,ac->bd", v, P[0, 2][:na, :nc])}
    assert len(got) == sum(w.size for w in want.values())
    for (isb, isd, x, y), val in got.items():
        assert abs(val - want[isb, isd][x, y]) <= 1e-13


def hermite_f32(Lt, G, rho, PQ):
    """S_r as the FP32 pass makes them: the recursion on S_r / lam^|r|, lam = sqrt(2 rho), times lam^|r|."""
    f = np.float32
    lam = f(np.sqrt(f(2 * rho)))
    S = {((0, 0, 0), m): f(G[m]) for m in range(Lt + 1)}
    X = [f(v) * lam for v in PQ]
    lp = [f(1)]
    for _ in range(Lt):
        lp.append(lp[-1] * lam)
    for r in HERM[1:gen.n_herm(Lt)]:
        ax = 0 if r[0] else (1 if r[1] else 2)
        r1 = tuple(v - (i == ax) for i, v in enumerate(r))
        r2 = tuple(v - 2 * (i == ax) for i, v in enumerate(r))
        for m in range(Lt - sum(r) + 1):
            v = X[ax] * S[r1, m + 1]
            if r1[ax]:
                v = v - f(r1[ax]) * S[r2, m + 1]
            S[r, m] = v
    return np.array([S[r, 0] * lp[sum(r)] for r in HERM[:gen.n_herm(Lt)]], dtype=f)


@pytest.mark.parametrize("ci", range(21), ids=[c.name() for c in MD])
def test_fp32_pass_error_by_class(ci, monkeypatch):
    """The tables run in FP32 as the FP32 pass does (recursion and both contractions; the transformations in
    FP64) on far-apart quartets, the kind that qualify: error relative to the quartet's largest integral.  A value
    passes 3 roundings of 2^-24 in each of L steps and 6 around them; 4 times that for sums whose terms
    cancel: 1.4e-6 at L = 0, 7.2e-6 at L = 8.  (Measured 5e-8 in (ss|ss), 2.6e-7 in (dd|dd): no class stands out, unlike
    the Obara-Saika schedules' in test_schedule_emulation.py, which no kernel runs.)"""
    c = MD[ci]
    rng = np.random.default_rng(900 + ci)
    worst = 0.0
    for _ in range(4):
        A = rng.uniform(-1, 1, 3)
        shift = rng.normal(size=3)
        shift *= rng.uniform(9, 12) / np.linalg.norm(shift)
        cen = np.array([A, A + rng.uniform(-2, 2, 3), shift + rng.uniform(-1, 1, 3), shift + rng.uniform(-2, 2, 3)])
        bra, ket = rng.uniform(0.1, 3.0, (2, 2)), rng.uniform(0.1, 3.0, (3, 2))
        ref = run_tables(c, bra, ket, cen, 0.11)
        with monkeypatch.context() as mk:
            mk.setitem(globals(), "hermite", lambda Lt, G, rho, PQ, dtype: hermite_f32(Lt, G, rho, PQ))
            got = run_tables(c, bra, ket, cen, 0.11, np.float32)
        worst = max(worst, np.abs(got - ref).max() / np.abs(ref).max())
    print(c.name(), worst)
    assert 0 < worst <= 4 * (3 * c.Lt + 6) * 2.0 ** -24
