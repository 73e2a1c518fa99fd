"""The work that users of this framework have it do, as measurable cases.

Every case goes through the public binding (``paper_2009_03559_gb300.hfx``).  Systems come
from the repository's own generators (``inputs``): jittered cubic clusters (s and p shells,
no cutoff, threshold 1e-10) and diamond-lattice pieces (s, s, p, p, d shells, 6-bohr orbital
cutoff, threshold 1e-8, density truncated beyond 10 bohr), three primitives per shell.

Kinds of a case:
  build     one exchange build for the density of an SCF iteration; the basis and the pair
            list are resident, as a program keeps them between iterations
  fresh     a new geometry: basis upload, pair list and the first exchange build
  batch     several systems in one batched build (captured graph)
  serve     requests of several resident systems through the request server
  periodic  lattice sums K^G of a crystal for a few cells
  nao       the fit of numerical radial functions by Gaussians
"""
import math

import numpy as np
import torch

from paper_2009_03559_gb300 import hfx, inputs

MIXED = {"fp64": hfx.HFX_FP64, "mixed": hfx.HFX_MIXED}


def listed():
    return [
        # the smallest workload of the benchmark set: 16 atoms, 64 functions; launches count
        {"name": "cluster16", "kind": "build", "system": "cluster", "atoms": 16, "precision": "fp64", "dens": 0.0},
        # the paper's SZ size: 128 shells, 256 functions, s and p only, no cutoff
        {"name": "cluster64", "kind": "build", "system": "cluster", "atoms": 64, "precision": "fp64", "dens": 0.0},
        # one conventional diamond cell with d shells: an ordinary small build
        {"name": "diamond8", "kind": "build", "system": "diamond", "atoms": 8, "precision": "fp64", "dens": 0.0},
        # an odd-sized piece of the solid, plain double precision: the largest build
        {"name": "diamond33", "kind": "build", "system": "diamond", "atoms": 33, "precision": "fp64", "dens": 0.0},
        # the same kind of solid in the mixed-precision option
        {"name": "diamond32-mixed", "kind": "build", "system": "diamond", "atoms": 32, "precision": "mixed", "dens": 0.0},
        # late SCF iterations: density-weighted screening switched on
        {"name": "diamond21-screened", "kind": "build", "system": "diamond", "atoms": 21, "precision": "fp64",
         "dens": 1e-8},
        # a step of a geometry run: new positions, everything from the basis on
        {"name": "fresh-cluster9", "kind": "fresh", "system": "cluster", "atoms": 9, "precision": "fp64", "dens": 0.0},
        # uneven small systems of both kinds in one batched launch
        {"name": "batch6", "kind": "batch", "systems": 6, "lo": 8, "hi": 24, "precision": "fp64"},
        # a handful of requests over resident systems, mixed precision as the server is run
        {"name": "serve8", "kind": "serve", "systems": 3, "requests": 8, "lo": 8, "hi": 20, "precision": "mixed"},
        # a crystal: one atom per cell with s, p and d shells, home cell and two neighbours
        {"name": "periodic-spd", "kind": "periodic", "shells": "spd", "a": 6.0, "rcut": 6.0, "cells": 3},
        # radial functions of two elements, 128 restarts each
        {"name": "nao10", "kind": "nao", "elements": 2, "restarts": 128, "n_r": 512},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["build", "build", "build", "build", "fresh", "batch", "serve", "periodic", "nao"])
    if kind in ("build", "fresh"):
        system = rng.choice(["cluster", "diamond", "diamond"])
        hi = {"build": {"cluster": 64, "diamond": 32}, "fresh": {"cluster": 40, "diamond": 16}}[kind][system]
        mixed = kind == "build" and rng.random() < 0.35
        dens = 10.0 ** rng.uniform(-10, -7) if kind == "build" and not mixed and rng.random() < 0.3 else 0.0
        return {"kind": kind, "system": system, "atoms": _log_int(rng, 2, hi),
                "precision": "mixed" if mixed else "fp64", "dens": dens}
    if kind == "batch":
        return {"kind": kind, "systems": rng.randint(2, 8), "lo": rng.randint(2, 8), "hi": rng.randint(9, 20),
                "precision": rng.choice(["fp64", "mixed"])}
    if kind == "serve":
        return {"kind": kind, "systems": rng.randint(2, 4), "requests": rng.randint(3, 10), "lo": rng.randint(4, 8),
                "hi": rng.randint(9, 20), "precision": rng.choice(["fp64", "mixed"])}
    if kind == "periodic":
        return {"kind": kind, "shells": rng.choice(["sp", "spd", "sd"]), "a": rng.uniform(5.0, 8.0),
                "rcut": rng.uniform(3.5, 6.0), "cells": rng.randint(1, 4)}
    return {"kind": kind, "elements": rng.randint(1, 3), "restarts": _log_int(rng, 16, 160),
            "n_r": rng.choice([256, 384, 500, 512])}


def _system(kind, atoms, seed):
    s = inputs.make_system(kind, atoms, seed)
    return s, inputs.density_matrix(s, truncate_bohr=inputs.truncation_for(kind))


def _mix(case, seed):
    """The systems of a batch or of a server's pool: sizes spread over [lo, hi], kinds in turn."""
    n = case["systems"]
    out = []
    for i in range(n):
        atoms = case["lo"] + (case["hi"] - case["lo"]) * i // max(1, n - 1)
        kind = "diamond" if i % 2 else "cluster"
        out.append((kind, atoms) + _system(kind, atoms, 1000 * seed + i))
    return out


def _context(s, case):
    return hfx.HFX(s, precision=MIXED[case["precision"]], density_tau=case.get("dens", 0.0))


def _cells(case):
    return [(0, 0, 0), (1, 0, 0), (0, 1, 1), (1, 1, 1)][: case["cells"]]


def _crystal(case, seed):
    return inputs.periodic_sc(a=case["a"], seed=seed, rcut=case["rcut"], tau=1e-9,
                              shells=tuple("spd".index(c) for c in case["shells"]))


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("build", "fresh"):
        s, P = _system(case["system"], case["atoms"], seed)
        st = {"case": case, "system": s, "P": torch.from_numpy(P).cuda()}
        if kind == "build":
            st["h"] = _context(s, case).build_pairs()
            st["K"] = torch.empty_like(st["P"])
        return st
    if kind == "batch":
        mix = _mix(case, seed)
        ctx = [_context(s, case).build_pairs() for _, _, s, _ in mix]
        Ps = [torch.from_numpy(P).cuda() for _, _, _, P in mix]
        return {"case": case, "batch": hfx.Batch(ctx), "ctx": ctx, "Ps": Ps, "Ks": [torch.empty_like(P) for P in Ps]}
    if kind == "serve":
        mix = _mix(case, seed)
        server = hfx.Server(precision=MIXED[case["precision"]])
        ids = [server.add_system(_context(s, case).build_pairs()) for _, _, s, _ in mix]
        which = [r % len(ids) for r in range(case["requests"])]
        Ps = [torch.from_numpy(inputs.density_matrix(mix[w][2], seed=100 * seed + r,
                                                     truncate_bohr=inputs.truncation_for(mix[w][0]))).cuda()
              for r, w in enumerate(which)]
        return {"case": case, "server": server, "ids": [ids[w] for w in which], "Ps": Ps,
                "Ks": [torch.empty_like(P) for P in Ps]}
    if kind == "periodic":
        ps = _crystal(case, seed)
        return {"case": case, "h": hfx.Periodic(ps).build_pairs(), "P": inputs.periodic_density(ps, 2, seed=seed + 1),
                "G": _cells(case)}
    rs = inputs.nao_set(case["elements"], seed=seed, n_r=case["n_r"])
    return {"case": case, "fit": hfx.NAOFit(rs.phi, rs.l, rs.h),
            "opt": hfx.nao_options(n_restarts=case["restarts"], seed=seed + 1)}


def run(state):
    kind = state["case"]["kind"]
    if kind == "build":  # an SCF iteration reads the exchange energy
        K = state["h"].build_K(state["P"], state["K"])
        return {"K": K, "E": state["h"].energy()}
    if kind == "fresh":
        h = _context(state["system"], state["case"]).build_pairs()
        K = h.build_K(state["P"])
        E = h.energy()
        h.close()
        return {"K": K, "E": E}
    if kind == "batch":
        state["batch"].run(state["Ps"], state["Ks"])
        return {"K": state["Ks"], "E": [c.energy() for c in state["ctx"]]}
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit(i, P, K) for i, P, K in zip(state["ids"], state["Ps"], state["Ks"])]
        done = [server.wait(t, release=True) for t in tickets]
        return {"K": state["Ks"], "E": [d["energy"] for d in done]}
    if kind == "periodic":
        K = state["h"].build_K(state["P"], state["G"])
        return {"K": [K[g] for g in state["G"]]}
    return state["fit"].fit(state["opt"])


# Per evaluated quartet: primitive quartets left of 3^4, and the flops of a primitive quartet
# (two Boys evaluations and the recurrences; with d shells the average over the classes).
_PRIMS, _FLOPS = 64, {"cluster": 400, "diamond": 900}


def _build_work(system, atoms, density_share=1.0):
    s = inputs.make_system(system, atoms, 0)
    d = np.linalg.norm(s.xyz[:, None] - s.xyz[None], axis=-1)
    near = (d < 2 * s.rcut) if s.rcut > 0 else np.ones_like(d, bool)
    per_atom = s.n_shells / atoms
    pairs = 0.5 * per_atom ** 2 * near.sum()
    quartets = 0.35 * density_share * pairs * pairs / 2
    return 2 * 8.0 * s.n_bf ** 2, float(quartets * _PRIMS * _FLOPS[system])


def work(case):
    kind = case["kind"]
    if kind in ("build", "fresh"):
        b, f = _build_work(case["system"], case["atoms"], 0.7 if case["dens"] > 0 else 1.0)
        return {"bytes": b, "flops": f}
    if kind in ("batch", "serve"):
        n = case["systems"]
        each = [_build_work("diamond" if i % 2 else "cluster", case["lo"] + (case["hi"] - case["lo"]) * i // max(1, n - 1))
                for i in range(n)]
        take = range(n) if kind == "batch" else [r % n for r in range(case["requests"])]
        return {"bytes": sum(each[i][0] for i in take), "flops": sum(each[i][1] for i in take)}
    if kind == "periodic":
        ns, nf = len(case["shells"]), sum(2 * "spd".index(c) + 1 for c in case["shells"])
        near = 4 / 3 * math.pi * (2 * case["rcut"] / case["a"]) ** 3
        pairs = ns * ns * near
        return {"bytes": 8.0 * nf * nf * (125 + case["cells"]), "flops": 0.3 * case["cells"] * pairs ** 2 * _PRIMS * 600}
    fits = 5 * case["elements"] * case["restarts"]
    points = case["n_r"] * 32 * 31  # population times generations (and the start)
    return {"bytes": 8.0 * 5 * case["elements"] * (case["n_r"] + 40 * case["restarts"]), "flops": fits * points * 40.0}


# ---------------------------------------------------------------------------------------
# Values in 64 bits: the definition of the exchange matrix, written with plain tensors.
# Hermite expansion of every shell pair, attenuated Boys values by Gauss-Legendre
# quadrature of int u^{2m} exp(-T u^2) du over [sqrt(kappa), 1], Hermite integrals by their
# recursion, and all two-electron integrals of the system as one four-index array.
# ---------------------------------------------------------------------------------------
_NODES, _WEIGHTS = np.polynomial.legendre.leggauss(48)
_D = [((1, 1, 0, 1.0),), ((0, 1, 1, 1.0),),
      ((0, 0, 2, 1 / math.sqrt(3)), (2, 0, 0, -0.5 / math.sqrt(3)), (0, 2, 0, -0.5 / math.sqrt(3))),
      ((1, 0, 1, 1.0),), ((2, 0, 0, 0.5), (0, 2, 0, -0.5))]
_SHAPES = {0: [((0, 0, 0, 1.0),)], 1: [((1, 0, 0, 1.0),), ((0, 1, 0, 1.0),), ((0, 0, 1, 1.0),)], 2: _D}


def _herm(n):
    return [(x, y, t - x - y) for t in range(n + 1) for x in range(t, -1, -1) for y in range(t - x, -1, -1)]


def _pair_tables(s, w, pairs, dev):
    """Hermite expansion of shell pairs (a, b) of one class: centres, exponents, and per
    primitive pair the coefficients E[pair, prim, function pair, Hermite index]."""
    la, lb = int(s.shell_l[pairs[0][0]]), int(s.shell_l[pairs[0][1]])
    off = np.concatenate([[0], np.cumsum(s.shell_nprim)])
    a, b = np.array(pairs).T
    pa = np.stack([s.alpha[off[a] + i] for i in range(3)], 1)[:, :, None]
    pb = np.stack([s.alpha[off[b] + i] for i in range(3)], 1)[:, None, :]
    wa = np.stack([w[off[a] + i] for i in range(3)], 1)[:, :, None]
    wb = np.stack([w[off[b] + i] for i in range(3)], 1)[:, None, :]
    A, B = s.xyz[s.shell_atom[a]], s.xyz[s.shell_atom[b]]
    t = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(dev)  # noqa: E731
    p = t((pa + pb).reshape(len(a), 9))
    ra, rb = t(np.broadcast_to(pa, (len(a), 3, 3)).reshape(len(a), 9)), t(np.broadcast_to(pb, (len(a), 3, 3)).reshape(len(a), 9))
    A, B = t(A)[:, None, :], t(B)[:, None, :]
    P = (ra[..., None] * A + rb[..., None] * B) / p[..., None]
    c = t((wa * wb).reshape(len(a), 9)) * torch.exp(-ra * rb / p * ((A - B) ** 2).sum(-1))
    e1 = {}  # (i, j) -> [pair, prim, axis, t]
    z = torch.zeros(P.shape + (la + lb + 1,), dtype=torch.float64, device=dev)
    z[..., 0] = 1.0

    def raised(e, X):  # multiplied by (x - X)
        out = (P - X)[..., None] * e
        out[..., 1:] += e[..., :-1] / (2 * p)[..., None, None]
        k = torch.arange(1, e.shape[-1], device=dev, dtype=torch.float64)
        out[..., :-1] += e[..., 1:] * k
        return out

    for i in range(la + 1):
        e1[i, 0] = z if i == 0 else raised(e1[i - 1, 0], A)
        for j in range(1, lb + 1):
            e1[i, j] = raised(e1[i, j - 1], B)
    H = _herm(la + lb)
    E = torch.zeros(len(a), 9, len(_SHAPES[la]) * len(_SHAPES[lb]), len(H), dtype=torch.float64, device=dev)
    f = 0
    for fa in _SHAPES[la]:
        for fb in _SHAPES[lb]:
            for xa in fa:
                for xb in fb:
                    for h, (u, v, x) in enumerate(H):
                        if u <= xa[0] + xb[0] and v <= xa[1] + xb[1] and x <= xa[2] + xb[2]:
                            E[:, :, f, h] += xa[3] * xb[3] * c * (e1[xa[0], xb[0]][:, :, 0, u] * e1[xa[1], xb[1]][:, :, 1, v]
                                                                 * e1[xa[2], xb[2]][:, :, 2, x])
            f += 1
    return {"p": p, "P": P, "E": E, "H": H, "L": la + lb, "n": len(a)}


def _block(x, y, omega):
    """(pairs of x | pairs of y): [pair, functions, pair, functions] in chunks over x's pairs."""
    dev, L = x["p"].device, x["L"] + y["L"]
    HR = _herm(L)
    at = {h: i for i, h in enumerate(HR)}
    pick = torch.tensor([[at[tuple(a + b for a, b in zip(h, g))] for g in y["H"]] for h in x["H"]], device=dev)
    sign = torch.tensor([(-1.0) ** sum(g) for g in y["H"]], dtype=torch.float64, device=dev)
    nodes, weights = (torch.from_numpy(v).to(dev) for v in (_NODES, _WEIGHTS))
    out = torch.empty(x["n"], x["E"].shape[2], y["n"], y["E"].shape[2], dtype=torch.float64, device=dev)
    q, Q = y["p"].reshape(-1), y["P"].reshape(-1, 3)
    step = max(1, int(2.5e8 // (9 * len(q) * (len(HR) + len(x["H"]) * len(y["H"])))))
    for i0 in range(0, x["n"], step):
        i1 = min(x["n"], i0 + step)
        p, P = x["p"][i0:i1].reshape(-1, 1), x["P"][i0:i1].reshape(-1, 1, 3)
        rho = p * q / (p + q)
        D = P - Q
        T = rho * (D * D).sum(-1)
        lo = torch.sqrt(omega * omega / (omega * omega + rho))
        hi = torch.minimum(torch.ones_like(T), torch.sqrt(lo * lo + 50.0 / T.clamp(min=1e-30)))
        G = [torch.zeros_like(T) for _ in range(L + 1)]
        for k in range(len(nodes)):
            u = 0.5 * (hi + lo) + 0.5 * (hi - lo) * nodes[k]
            u2 = u * u
            v = torch.exp(-T * u2).mul_(0.5 * weights[k] * (hi - lo))
            for m in range(L + 1):
                G[m] += v
                v = v * u2
        pre = 2 * math.pi ** 2.5 / (p * q * torch.sqrt(p + q))
        level = {}
        for m in range(L, -1, -1):  # R_{t}^{m} from the level m + 1
            now = {(0, 0, 0): pre * (-2 * rho) ** m * G[m]}
            for h in HR[1:]:
                if sum(h) > L - m:
                    break
                ax = next(i for i in range(3) if h[i])
                g = tuple(h[i] - (i == ax) for i in range(3))
                now[h] = D[..., ax] * level[g]
                if g[ax]:
                    now[h] = now[h] + g[ax] * level[tuple(g[i] - (i == ax) for i in range(3))]
            level = now
        R = torch.stack([level[h] for h in HR], -1)  # [prim x, prim y, Hermite]
        del level
        R = R[..., pick.reshape(-1)].reshape(i1 - i0, 9, y["n"], 9, len(x["H"]), len(y["H"])) * sign
        half = torch.einsum("aibjtu,bjgu->aitbg", R, y["E"])
        out[i0:i1] = torch.einsum("aitbg,aift->afbg", half, x["E"][i0:i1])
        del R, half
    return out


def _exact_build(s, P, dens):
    if s.n_bf > 110:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    off = np.concatenate([[0], np.cumsum(s.shell_nprim)])
    w = np.empty_like(s.alpha)
    for k in range(s.n_shells):  # unit self-overlap
        e, l = s.alpha[off[k]:off[k + 1]], int(s.shell_l[k])
        c = s.coef[off[k]:off[k + 1]] * e ** ((2 * l + 3) / 4)
        g = e[:, None] + e[None, :]
        w[off[k]:off[k + 1]] = c / math.sqrt((c[:, None] * c[None, :] * (math.pi / g) ** 1.5 * (2 * g) ** (-float(l))).sum())
    groups = {}
    for i in range(s.n_shells):
        for j in range(i + 1):
            d = np.linalg.norm(s.xyz[s.shell_atom[i]] - s.xyz[s.shell_atom[j]])
            if s.rcut <= 0 or s.shell_atom[i] == s.shell_atom[j] or d < 2 * s.rcut:
                a, b = (i, j) if s.shell_l[i] >= s.shell_l[j] else (j, i)
                groups.setdefault((int(s.shell_l[a]), int(s.shell_l[b])), []).append((a, b))
    tabs = {k: _pair_tables(s, w, v, dev) for k, v in groups.items()}
    Q = {}
    for k, x in tabs.items():
        each = [_block({**x, "p": x["p"][i:i + 1], "P": x["P"][i:i + 1], "E": x["E"][i:i + 1], "n": 1},
                       {**x, "p": x["p"][i:i + 1], "P": x["P"][i:i + 1], "E": x["E"][i:i + 1], "n": 1}, s.omega)[0, :, 0, :].diagonal().abs().max()
                for i in range(x["n"])]
        Q[k] = torch.stack(each).sqrt()
    qmax = max(float(q.max()) for q in Q.values())
    n, bf = s.n_bf, s.shell_offset
    Pt = torch.from_numpy(P).to(dev)
    shell_of = torch.from_numpy(np.repeat(np.arange(s.n_shells), s.shell_nbf)).to(dev)
    pm = torch.zeros(s.n_shells * s.n_shells, dtype=torch.float64, device=dev)
    pm.scatter_reduce_(0, (shell_of[:, None] * s.n_shells + shell_of[None, :]).reshape(-1), Pt.abs().reshape(-1), "amax")
    pm = pm.reshape(s.n_shells, s.n_shells)
    eri = torch.zeros(n, n, n, n, dtype=torch.float64, device=dev)
    index = {}
    for (la, lb), v in groups.items():
        na, nb = 2 * la + 1, 2 * lb + 1
        a = torch.tensor([[bf[i] + f // nb for f in range(na * nb)] for i, _ in v], device=dev)
        b = torch.tensor([[bf[j] + f % nb for f in range(na * nb)] for _, j in v], device=dev)
        index[la, lb] = a, b, torch.tensor(v, device=dev)
    for k, x in tabs.items():
        for g, y in tabs.items():
            if g > k:
                continue
            qq = Q[k][:, None] * Q[g][None, :]
            keep = (qq >= s.tau) & (Q[k] * qmax >= s.tau)[:, None] & (Q[g] * qmax >= s.tau)[None, :]
            if dens > 0:
                (a, b), (c, d) = index[k][2].T, index[g][2].T
                most = torch.stack([pm[b][:, d], pm[b][:, c], pm[a][:, d], pm[a][:, c]]).amax(0)
                keep &= qq * most >= dens
            V = _block(x, y, s.omega) * keep[:, None, :, None]
            V = V.reshape(x["n"] * V.shape[1], -1)
            a, b, c, d = (t.reshape(-1) for t in (*index[k][:2], *index[g][:2]))
            for i, j in ((a, b), (b, a)):
                for m, l in ((c, d), (d, c)):
                    eri[i[:, None], j[:, None], m[None, :], l[None, :]] = V
                    eri[m[:, None], l[:, None], i[None, :], j[None, :]] = V.T
    K = torch.einsum("ijkl,jl->ik", eri, Pt)
    return {"K": K, "E": float((Pt * K).sum())}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("build", "fresh"):
        return _exact_build(*_system(case["system"], case["atoms"], seed), case["dens"])
    if kind == "batch":
        got = [_exact_build(s, P, 0.0) or {"K": None, "E": None} for _, _, s, P in _mix(case, seed)]
        return {"K": [g["K"] for g in got], "E": [g["E"] for g in got]}
    return None
