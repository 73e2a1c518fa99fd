"""The Boys look-up of the FP64 kernels (csrc/boys.cuh), compiled for the host, against 40 digits.

Two errors are kept apart: that of the rows' leading entries (the series and the recursion that make
them, in FP64) and that of the evaluation, F_L(x_g + d) and exp(-x_g - d) from them.  The evaluation is
held to FP64: its last FMA rounds to half a unit (2^-53 relative), the ones before it count d <= 1/128
of that, and what runs in FP32 (from the fourth order in d on) adds at most its share of the value times
FP32's rounding: d^2 three times 2^-24, the mantissa or entry one, the polynomial one and a half, two products."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HALF, FP32 = 2.0 ** -53 * (1 + 1 / 64), 7.5 * 2.0 ** -24
LMAX = 8


@pytest.fixture(scope="module")
def boys(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("boys") / "boys.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-w", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2009_03559_gb300", "csrc"), "-o", so,
                    os.path.join(ROOT, "tests", "c", "boys_host.cpp")], check=True)
    lib = ctypes.CDLL(so)
    lib.boys_table_data.restype = ctypes.POINTER(ctypes.c_double)
    lib.boys_tables()
    s = (ctypes.c_int * 6)()
    lib.boys_sizes(s)
    lib.row_len, lib.per_unit, lib.rows, lib.table_len, lib.tail_bits, lib.n = list(s)
    lib.tab = np.ctypeslib.as_array(lib.boys_table_data(), (lib.n,))
    return lib


def at(lib, L, x, any_):
    F, e = ctypes.c_double(), ctypes.c_double()
    lib.boys_at(L, ctypes.c_double(x), any_, ctypes.byref(F), ctypes.byref(e))
    return F.value, e.value


def f32_down(x):
    """FP32 value of x by truncation: what the look-up rounds to a row."""
    f = np.float32(x)
    return float(f if float(f) <= x else np.nextafter(f, np.float32(0)))


def grid(lib, g):
    return float(np.float32(g) * (np.float32(1) / np.float32(lib.per_unit)))


def true_f(x, top):
    """F_0 .. F_top at an exact x."""
    F = [mp.mpf(0)] * (top + 1)
    F[top] = mp.exp(-x) * mp.hyp1f1(1, top + mp.mpf(3) / 2, x) / (2 * top + 1)
    for m in range(top, 0, -1):
        F[m - 1] = (2 * x * F[m] + mp.exp(-x)) / (2 * m - 1)
    return F


def test_evaluation_below_60(boys):
    mp.mp.dps = 40
    rng = np.random.default_rng(5)
    xs = np.concatenate([rng.uniform(0, 60, 150), rng.uniform(0, 2, 50),
                         (rng.integers(0, boys.rows - 1, 200) + 0.5 + 1e-4 * rng.standard_normal(200)) / boys.per_unit])
    worst = dict(F=0.0, e=0.0)
    for x in xs:
        g = int(np.rint(f32_down(x) * boys.per_unit))
        xg = mp.mpf(grid(boys, g))
        d = mp.mpf(float(x)) - xg
        T = true_f(xg, LMAX + 11)
        ex = boys.tab[boys.n - 2 * boys.rows + 2 * g]
        for L in range(LMAX + 1):
            row = boys.tab[L * boys.table_len + g * boys.row_len:][:3]
            want = sum(mp.mpf(float(row[k])) * d ** k for k in range(3))
            want += sum(T[L + k] * (-d) ** k / mp.factorial(k) for k in range(3, 12))
            want_e = mp.mpf(float(ex)) * mp.exp(-d)
            for any_ in (0, 1):
                F, e = at(boys, L, float(x), any_)
                rF, re = float(abs(F - want) / want), float(abs(e - want_e) / want_e)
                worst["F"], worst["e"] = max(worst["F"], rF), max(worst["e"], re)
                dm = 0.5 / boys.per_unit
                assert rF <= HALF + dm ** 4 / 24 * FP32, (L, x, rF)
                assert re <= HALF + dm ** 4 / 24 * FP32, (L, x, re)
    print("evaluation error", worst)


def test_evaluation_from_60_on(boys):
    mp.mp.dps = 40
    rng = np.random.default_rng(6)
    n = 1 << boys.tail_bits
    xs = np.concatenate([[60.0, 63.999, 64.0, 64.001, 255.99, 256.01, 1e6, 1e30], np.exp(rng.uniform(np.log(60), np.log(1e9), 150)),
                         64 * (1 + (rng.integers(0, n, 100) + 0.5 + 1e-4 * rng.standard_normal(100)) / n)])
    for x in map(float, xs):
        k = (int(np.floor(np.log2(x)))) // 2
        t = mp.mpf(x) / mp.mpf(4) ** k
        octave = 2 if t >= 2 else 1
        g = int(np.floor((f32_down(float(t)) / octave - 1) * n + 0.5))
        tg = (1 + mp.mpf(g) / n) * octave
        for L in range(LMAX + 1):
            F, e = at(boys, L, x, 1)
            assert e == 0.0
            row = boys.tab[L * boys.table_len + (boys.rows + (octave - 1) * n + g) * boys.row_len:][:3]
            d = t - tg
            a = mp.gamma(L + mp.mpf(1) / 2) / 2  # (2L-1)!!/2^{L+1} sqrt(pi)
            want = sum(mp.mpf(float(row[i])) * d ** i for i in range(3))
            want += sum(a * mp.binomial(-L - mp.mpf(1) / 2, i) * tg ** (-L - mp.mpf(1) / 2 - i) * d ** i for i in range(3, 12))
            want /= mp.mpf(4) ** (k * (L + mp.mpf(1) / 2))
            c4 = float(abs(mp.binomial(-L - mp.mpf(1) / 2, 4))) * (0.5 / n + 2.0 ** -22) ** 4
            assert abs(F - want) / want <= HALF + c4 * FP32, (L, x, float(abs(F - want) / want))


def test_entries(boys):
    """The leading entries, counting roundings of 2^-53: below 60 three for each of some 150 terms that make up
    the series, 250 sums of it, three for each of 15 steps down; the asymptote's constant (9), square root, L + 1
    divisions; of exp and of the sixth of it a unit each, two and three."""
    mp.mp.dps = 40
    rng = np.random.default_rng(7)
    u = 2.0 ** -53
    for g in [0, 1, *map(int, rng.integers(2, boys.rows - 1, 60)), boys.rows - 1]:
        x = mp.mpf(grid(boys, g))
        T = true_f(x, LMAX + 3)
        ex = boys.tab[boys.n - 2 * boys.rows + 2 * g:][:2]
        assert abs(ex[0] * mp.exp(x) - 1) <= 2 * u and abs(6 * ex[1] * mp.exp(x) - 1) <= 3 * u
        for L in range(LMAX + 1):
            for k in range(4):
                f = boys.tab[L * boys.table_len + g * boys.row_len + k]
                assert abs(f * mp.factorial(k) * (-1) ** k / T[L + k] - 1) <= 750 * u, (L, g, k)
    n = 1 << boys.tail_bits
    for g in [0, 1, n - 1, n, n + 1, 2 * n - 1, 2 * n, *map(int, rng.integers(2, 2 * n, 30))]:
        t = 1 + mp.mpf(g) / n if g < n else 2 + 2 * mp.mpf(g - n) / n
        for L in range(LMAX + 1):
            want = mp.gamma(L + mp.mpf(1) / 2) / 2 * t ** (-L - mp.mpf(1) / 2)
            assert abs(boys.tab[L * boys.table_len + (boys.rows + g) * boys.row_len] / want - 1) <= (11 + L) * u, (L, g)


def test_no_entry_close_below_a_power_of_two(boys):
    """The FP32 part is added to f_2 (and e_0 / 2) as an integer number of ulps: it may not reach the next
    power of two.  Largest parts: f_4 d^2 (1/12 of e_0 / 2, d^2), with a factor of 4 to spare."""
    n, dm = 1 << boys.tail_bits, 0.5 / boys.per_unit

    def room(v):
        m, _ = np.frexp(v)
        return (1 - m) / m

    for L in range(LMAX + 1):
        rows = boys.tab[L * boys.table_len:(L + 1) * boys.table_len].reshape(-1, boys.row_len)
        g = np.arange(len(rows)) - boys.rows
        d = np.where(g < 0, dm, np.where(g < n, 0.5 / n, 1.0 / n))
        part = rows[:, 4:].copy().view(np.float32)[:, 0] * 2.0 ** -44 * 2.0 ** (np.frexp(rows[:, 2])[1] - 1)
        assert np.all((part > 0) & (room(rows[:, 2]) > 4 * part * d ** 2 / rows[:, 2]))
    assert np.all(room(boys.tab[boys.n - 2 * boys.rows::2]) > 4 * dm ** 2 / 12)
