#!/usr/bin/env python3
"""Generate the per-class tables of the Hermite engine (hfx_md.cuh).

A shell pair's function product is expanded in Hermite Gaussians (McMurchie-Davidson), and the
expansion is split into factors that depend on the primitive pair and factors that do not, so
that the contraction over primitives runs before any transformation (the order of the PRISM
methods of Gill, Head-Gordon and Pople).  For the pair (l_a, l_b) with centres A, B, exponents
a, b, p = a + b, u_a = a / p, u_b = b / p and AB = A - B, per axis
    (x - A)^m (x - B)^n e^{-p (x-P)^2} = sum over i, j of C(m,i) C(n,j) PA^i PB^j x_P^{m-i+n-j} e^{..},
    PA = -u_b AB,  PB = u_a AB,
    x_P^N e^{..} = sum_h N! / (2^h h! (N-2h)!) (1/2p)^{N-h} Lambda_{N-2h}.
Multiplied over the axes and with the spherical components of d shells taken, a function pair f is
    sum over sets s = (k, i, j, h) and Hermite indices t of order k of
        W_s T_f[s, t] Lambda_t,   W_s = u_b^i u_a^j (1/2p)^{k+h}   (the primitive pair's factor)
    with T_f[s, t] a polynomial in the components of AB (the pair's factor), i + j + k + 2h = l_a + l_b.
A spherical d has no trace, so only pairs of powers from the two different shells survive in h.

The integral of two function pairs is then (with the Hermite integrals S_r = (-1)^{|r|} R_r of
order up to L = l_a + l_b + l_c + l_d, S^(m)_0 = (2 rho)^m G_m and
    S^(m)_{r+1} = X S^(m+1)_r - r S^(m+1)_{r-1},  X = (P - Q) along the raised axis)
    (ab|cd) = sum T_ab[s',p] T_cd[s,q] (-1)^{|p|} sum over primitive pairs of W_s' W_s S_{p+q},
evaluated in this order, each step one table:
  kc  per bra primitive pair: H[s, r] = sum over ket primitive pairs of W_s S_r,
      r of order k .. k + l_a + l_b;
  bc  A[s', s, r] += W_s' H[s, r], r of order k' + k, once per bra primitive pair;
  z1  per quartet: Y[s', p; cd] = sum over (s, q) of T_cd[s, q] A[s', s, p + q];
  z2  (ab|cd) = sum over (s', p) of T_ab'[s', p] Y[s', p; cd], where T_ab' (the sign (-1)^{|p|}
      taken in) is (-1)^{l_a + l_b} times T_ab at -AB.
Run:  python gen_md_tables.py > md_tables.inc
"""
from __future__ import annotations

import math
import sys

PAIR_CLASSES = [(0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (2, 2)]
S3 = 1.0 / (2.0 * math.sqrt(3.0))
# function components: lists of (power of x, y, z, factor); d: xy, yz, (2zz-xx-yy)/(2 sqrt 3), xz, (xx-yy)/2
SHAPES = {
    0: [[(0, 0, 0, 1.0)]],
    1: [[(1, 0, 0, 1.0)], [(0, 1, 0, 1.0)], [(0, 0, 1, 1.0)]],
    2: [[(1, 1, 0, 1.0)], [(0, 1, 1, 1.0)], [(0, 0, 2, 2.0 * S3), (2, 0, 0, -S3), (0, 2, 0, -S3)], [(1, 0, 1, 1.0)],
        [(2, 0, 0, 0.5), (0, 2, 0, -0.5)]],
}


def monos(n):
    """Hermite indices (x, y, z) of order n."""
    return [(i, j, n - i - j) for i in range(n, -1, -1) for j in range(n - i, -1, -1)]


def herm_index(r):
    """Position of r in the list of all indices by order (x descending, then y)."""
    n, x = sum(r), r[0]
    return n * (n + 1) * (n + 2) // 6 + (n - x) * (n - x + 1) // 2 + (n - x - r[1])


def n_herm(n):
    return (n + 1) * (n + 2) * (n + 3) // 6


def axis_terms(m, n):
    """(x-A)^m (x-B)^n: {(t, i, j, h): factor}, the sign of PA = -u_b AB taken in."""
    out = {}
    for i in range(m + 1):
        for j in range(n + 1):
            N = m - i + n - j
            c = math.comb(m, i) * math.comb(n, j) * (-1) ** i
            for h in range(N // 2 + 1):
                f = math.factorial(N) // (2 ** h * math.factorial(h) * math.factorial(N - 2 * h))
                out[N - 2 * h, i, j, h] = out.get((N - 2 * h, i, j, h), 0) + c * f
    return out


class PairType:
    """Sets and transformation T of a pair (la, lb)."""

    def __init__(self, la, lb):
        self.la, self.lb, self.L = la, lb, la + lb
        T = []      # per function pair: {(set, t): {monomial of AB: factor}}
        for fa in SHAPES[la]:
            for fb in SHAPES[lb]:
                acc = {}
                for xa in fa:
                    for xb in fb:
                        ax = [axis_terms(xa[d], xb[d]) for d in range(3)]
                        for (t0, i0, j0, h0), c0 in ax[0].items():
                            for (t1, i1, j1, h1), c1 in ax[1].items():
                                for (t2, i2, j2, h2), c2 in ax[2].items():
                                    t = (t0, t1, t2)
                                    s = (sum(t), i0 + i1 + i2, j0 + j1 + j2, h0 + h1 + h2)
                                    mono = (i0 + j0, i1 + j1, i2 + j2)
                                    d = acc.setdefault((s, t), {})
                                    d[mono] = d.get(mono, 0.0) + xa[3] * xb[3] * c0 * c1 * c2
                out = {}
                for key, d in acc.items():
                    d = {m: c for m, c in d.items() if abs(c) > 1e-12}
                    if d:
                        out[key] = d
                T.append(out)
        self.sets = sorted({s for f in T for s, _ in f})
        pos = {s: n for n, s in enumerate(self.sets)}
        self.T = [{(pos[s], t): d for (s, t), d in f.items()} for f in T]
        self.k = [s[0] for s in self.sets]
        # rows: (set, Hermite index of its order)
        self.rows = [(s, t) for s in range(len(self.sets)) for t in monos(self.k[s])]
        self.row = {r: n for n, r in enumerate(self.rows)}
        # distinct coefficients: polynomials in AB, coefficient 0 = zero
        self.coefs = [()]
        self.coef_of = {}
        for f in self.T:
            for d in f.values():
                key = tuple(sorted((m, round(c, 14)) for m, c in d.items()))
                if key not in self.coef_of:
                    self.coef_of[key] = len(self.coefs)
                    self.coefs.append(tuple(sorted(d.items())))
        self.n_fun = len(self.T)

    def terms(self, f):
        """[(coefficient index, set, t)] of function pair f."""
        return [(self.coef_of[tuple(sorted((m, round(c, 14)) for m, c in d.items()))], s, t)
                for (s, t), d in sorted(self.T[f].items())]


PAIRS = [PairType(la, lb) for la, lb in PAIR_CLASSES]


class Gather:
    """A sparse pass out[dst] = sum of coef[c] in[i]: outputs sorted by their number of terms and
    dealt to 32 lanes a round, every lane of a round padded to the round's longest (with
    coefficient 0)."""

    def __init__(self, outs):
        order = sorted(range(len(outs)), key=lambda o: (-len(outs[o][1]), o))
        self.rounds, self.words, self.dst = [], [], []
        for r0 in range(0, len(order), 32):
            lanes = order[r0:r0 + 32]
            n = len(outs[lanes[0]][1])
            self.rounds.append((len(self.words), n))
            for t in range(n):
                for l in range(32):
                    ts = outs[lanes[l]][1] if l < len(lanes) else []
                    c, i = ts[t] if t < len(ts) else (0, 0)
                    self.words.append(c | (i << 16))
            self.dst += [outs[lanes[l]][0] if l < len(lanes) else 0xFFFF for l in range(32)]


class Digest:
    """The sums of the four blocks A_ac, A_ad, A_bc, A_bd over the final block (a, b, c, d), as lane
    tasks: (row of b instead of a, column of d instead of c, row, column, first u, first w, terms), u
    and w the two summed indices, w running fastest.  A sum is cut into tasks of at most `chunk`
    terms (each adds its part to the matrix), the tasks dealt to lanes by length: the chunk that
    costs the fewest instructions, a round counting its longest task and two more."""

    def __init__(self, dims):
        na, nb, nc, nd = dims
        best = None
        for chunk in range(1, 26):
            tasks = []
            for isb in (0, 1):
                for isd in (0, 1):
                    nw = nc if isd else nd
                    n = (na if isb else nb) * nw
                    parts = -(-n // chunk)
                    cuts = [n * i // parts for i in range(parts + 1)]
                    for x in range(nb if isb else na):
                        for y in range(nd if isd else nc):
                            tasks += [(isb, isd, x, y, c0 // nw, c0 % nw, c1 - c0) for c0, c1 in zip(cuts, cuts[1:])]
            tasks.sort(key=lambda s: -s[6])
            cost = sum(tasks[r][6] + 2 for r in range(0, len(tasks), 32))
            if best is None or (cost, len(tasks)) < best[:2]:
                best = (cost, len(tasks), tasks)
        self.cost, _, tasks = best
        tasks = tasks + [(0,) * 7] * (-len(tasks) % 32)
        self.words = [b | d << 1 | x << 2 | y << 5 | u << 8 | w << 11 | n << 14 for b, d, x, y, u, w, n in tasks]


class MdClass:
    def __init__(self, hi, lo):
        self.hi, self.lo = hi, lo
        b, k = PAIRS[hi], PAIRS[lo]
        self.Lt = b.L + k.L
        # H[s, r]: ket set s, r of order k_s + (0 .. bra orders present)
        self.kc, hidx = [], {}
        for s, ks in enumerate(k.k):
            for n in range(ks, ks + max(b.k) + 1):
                for r in monos(n):
                    hidx[s, r] = len(self.kc)
                    self.kc.append((herm_index(r), s))
        self.bc, aidx = [], {}
        for sb, kb in enumerate(b.k):
            for s, ks in enumerate(k.k):
                for r in monos(kb + ks):
                    aidx[sb, s, r] = len(self.bc)
                    self.bc.append((hidx[s, r], sb))
        add = lambda p, q: (p[0] + q[0], p[1] + q[1], p[2] + q[2])  # noqa: E731
        self.n_rows, self.ncd, self.nab = len(b.rows), k.n_fun, b.n_fun
        self.z1 = Gather([(row * self.ncd + f, [(c, aidx[sb, s, add(p, q)]) for c, s, q in k.terms(f)])
                          for row, (sb, p) in enumerate(b.rows) for f in range(self.ncd)])
        self.z2 = Gather([(ab * self.ncd + f, [(c, b.row[sb, p] * self.ncd + f) for c, sb, p in b.terms(ab)])
                          for ab in range(self.nab) for f in range(self.ncd)])

        self.dims = [2 * l + 1 for l in (*PAIR_CLASSES[hi], *PAIR_CLASSES[lo])]
        self.digest = Digest(self.dims)

    def name(self):
        L = "spd"
        return "(" + "|".join("".join(L[x] for x in PAIR_CLASSES[c]) for c in (self.hi, self.lo)) + ")"

    def flops(self):
        """Add/mul 1, fma 2: per primitive quartet (Hermite recursion, ket contraction), per run of a
        bra primitive pair (bra contraction), per quartet (transformations and digest, digest alone)."""
        r = 0
        for o in range(1, self.Lt + 1):
            for t in monos(o):
                n = t[0] or t[1] or t[2]
                r += (self.Lt - o + 1) * (1 if n == 1 else (3 if n - 1 in (3, 5, 6, 7) else 2))
        terms = self.n_rows * sum(len(PAIRS[self.lo].T[f]) for f in range(self.ncd))
        terms += self.ncd * sum(len(PAIRS[self.hi].T[f]) for f in range(self.nab))
        na, nb, nc, nd = self.dims
        dig = 8 * na * nb * nc * nd + (na + nb) * (nc + nd)
        return r + 2 * len(self.kc), 2 * len(self.bc), 2 * terms + dig, dig

    def r_ops(self):
        """FP64 instructions of the Hermite recursion, x last (2 S is an exponent increment)."""
        n = 0
        for o in range(1, self.Lt + 1):
            for r in monos(o):
                t = r[0] or r[1] or r[2]
                n += (self.Lt - o + 1) * (1 if t in (1, 2, 3, 5) else 2)
        return n


def classes():
    return [MdClass(hi, lo) for hi in range(6) for lo in range(hi + 1)]


# warps that work on one stream together (the kernel's choice and its reasons: hfx_md.cuh)
def team(Lt):
    return 1 if Lt <= 5 else (2 if Lt == 6 else 4)


def emit(w):
    cl = classes()
    kc, bc, zw, zd, zr, dg, rows = [], [], [], [], [], [], []
    for c in cl:
        r = dict(kc=len(kc), nkc=len(c.kc), bc=len(bc), nbc=len(c.bc))
        kc += [i | (s << 8) for i, s in c.kc]
        kc += [0] * (-len(kc) % 32)
        bc += [h | (s << 12) for h, s in c.bc]
        bc += [0] * (-len(bc) % 32)
        for nm in ("z1", "z2"):
            g = getattr(c, nm)
            r[nm] = (len(zr), len(g.rounds), len(zd))
            zr += [(len(zw) + o) | (n << 24) for o, n in g.rounds]
            zw += g.words
            zd += g.dst
        r["dig"] = (len(dg), len(c.digest.words) // 32)
        dg += c.digest.words
        rows.append((c, r))
    assert len(zw) < 1 << 24
    w("// Generated by gen_md_tables.py -- do not edit by hand.\n#pragma once\n\n")

    def arr(name, typ, v, hexa=True):
        w(f"HFX_TABLE_QUAL {typ} {name}[{len(v)}] = {{\n")
        for i in range(0, len(v), 16):
            w(" " + ",".join(f"{x:#x}" if hexa else repr(x) for x in v[i:i + 16]) + ",\n")
        w("};\n\n")
    w("// ket contraction: Hermite index | ket set << 8;  bra contraction: H index | bra set << 12\n")
    arr("kMdKc", "uint16_t", kc)
    arr("kMdBc", "uint16_t", bc)
    w("// transformation passes: coefficient | source << 16; outputs; rounds (first word | terms << 24)\n")
    arr("kMdZ", "uint32_t", zw)
    arr("kMdZDst", "uint16_t", zd)
    arr("kMdZRound", "uint32_t", zr)
    w("// digest: row b | column d << 1 | row << 2 | column << 5 | first u << 8 | first w << 11 | terms << 14\n")
    arr("kMdDigest", "uint32_t", dg)
    by_l = [[c for c in cl if c.Lt == l] for l in range(9)]
    rounds = lambda n, l: -(-(-(-n // 32)) // team(l))  # noqa: E731
    w("// by total angular momentum: warps of a team; the most rounds a warp of it has in a ket and in a\n"
      "// bra contraction; the most sets of a ket\n")
    for name, v in (("md_team", [team(l) for l in range(9)]),
                    ("md_kc_rounds", [max(rounds(len(c.kc), l) for c in by_l[l]) for l in range(9)]),
                    ("md_bc_rounds", [max(rounds(len(c.bc), l) for c in by_l[l]) for l in range(9)]),
                    ("md_ket_sets", [max(len(PAIRS[c.lo].sets) for c in by_l[l]) for l in range(9)])):
        w(f"__host__ __device__ constexpr int {name}(int Lt) {{\n  const int v[9] = {{{', '.join(map(str, v))}}};\n"
          "  return v[Lt];\n}\n")
    w("\n")
    # coefficients per pair type: polynomials over the 35 monomials of AB up to degree 4
    mono = {m: i for i, m in enumerate(m for n in range(5) for m in monos(n))}
    poly, cf, sign, info = [], [], [], []
    for p in PAIRS:
        info.append((len(cf), len(p.coefs), len(p.sets)))
        for d in p.coefs:
            cf.append(len(poly) | (len(d) << 16))
            sign.append((p.L + (sum(d[0][0]) if d else 0)) & 1)   # k and the degree add up to L, less 2h
            poly += [(mono[m], v) for m, v in d]
    w("// transformation coefficients: first term | terms << 16; terms: monomial of AB and factor\n")
    arr("kMdCoef", "uint32_t", cf)
    arr("kMdCoefSign", "unsigned char", sign)
    arr("kMdTermMono", "unsigned char", [m for m, _ in poly])
    arr("kMdTermVal", "double", [v for _, v in poly], hexa=False)
    w("// flops (add/mul 1, fma 2) per primitive quartet, per bra run, per quartet, of it in the digest\n")
    w("static const int kMdFlops[HFX_N_CLASSES][4] = {\n")
    for c in cl:
        w(f"  {{{', '.join(map(str, c.flops()))}}},\n")
    w("};\n\n")
    w("static const MdPairInfo kMdPair[6] = {\n")
    for (off, n, ns), p in zip(info, PAIRS):
        st = [(k + h) | (i << 4) | (j << 8) for k, i, j, h in p.sets] + [0] * (14 - len(p.sets))
        w(f"  {{{off}, {n}, {ns}, {{{', '.join(map(str, st))}}}}},\n")
    w("};\n\nstatic const MdClassInfo kMdClass[HFX_N_CLASSES] = {\n")
    for c, r in rows:
        z = (sum(n for _, n in c.z1.rounds), sum(n for _, n in c.z2.rounds))
        w(f"  // {c.name()}: Hermite recursion {c.r_ops()} instructions on every primitive quartet's lane, contraction "
          f"{-(-len(c.kc) // 32)} per primitive quartet, {-(-len(c.bc) // 32)} per bra pair, transformation {z[0]} + {z[1]}, digest {c.digest.cost}\n")
        b, k = info[c.hi], info[c.lo]
        w(f"  {{{c.Lt}, {r['kc']}, {r['nkc']}, {r['bc']}, {r['nbc']}, {c.n_rows}, {c.nab}, {c.ncd}, "
          f"{b[0]}, {b[1]}, {b[2]}, {k[1]}, {k[2]}, "
          f"{r['z1'][0]}, {r['z1'][1]}, {r['z1'][2]}, {r['z2'][0]}, {r['z2'][1]}, {r['z2'][2]}, {r['dig'][0]}, {r['dig'][1]}}},\n")
    w("};\n")


if __name__ == "__main__":
    if "--summary" in sys.argv:
        for c in classes():
            print(c.name(), "L", c.Lt, "R", c.r_ops(), "kc", len(c.kc), "bc", len(c.bc), "rows", c.n_rows,
                  "z1", sum(n for _, n in c.z1.rounds), "z2", sum(n for _, n in c.z2.rounds), "digest", c.digest.cost, len(c.digest.words) // 32, "coefs",
                  len(PAIRS[c.hi].coefs), len(PAIRS[c.lo].coefs), "Y", c.n_rows * c.ncd)
    else:
        emit(sys.stdout.write)
