"""The Hermite engine where it can go wrong: arguments of the Boys tables at their seams, and
streams of quartets with very few and very many primitive quartets (queue, runs cut by batch
ends, teams of warps), against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2009_03559_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hfx_mod():
    from paper_2009_03559_gb300 import hfx
    return hfx


def check(hfx_mod, s, P, tol, **kw):
    Ko, eo = oracle.Screen(oracle.Basis(s)).build_K(P, "sym")
    h = hfx_mod.HFX(s, **kw).build_pairs()
    h.set_timing(True)
    K = h.build_K(torch.from_numpy(P).cuda()).cpu().numpy()
    assert np.abs(K - Ko).max() <= tol * np.abs(Ko).max(), np.abs(K - Ko).max()
    assert abs(h.energy() - eo) <= tol * np.abs(Ko).max() * s.n_bf
    return h


# exponents 1 on both atoms: rho = 1 for the quartets of two same-atom pairs, T = R^2.  60 is where
# the rows of the asymptote begin, powers of 4 where their scaling by 4^k changes, 1/512 off a grid
# point the largest distance from one.  Tolerance: 16 doubles' rounding in each of some 30 steps.
@pytest.mark.parametrize("T", [1e-6, 1.0 / 512, 17.0 + 1.0 / 512, 59.998, 60.0, 60.002, 63.999, 64.001, 255.99, 256.01,
                               4095.9, 4096.1, 1e6])
@pytest.mark.parametrize("omega", [0.0, 0.11])
def test_boys_seams(hfx_mod, T, omega):
    ls = [0, 1, 2]
    xyz = np.array([[0.0, 0.0, 0.0], [0.6, 0.48, 0.64]]) * np.sqrt(T)
    s = inputs.System("pair", xyz, np.repeat([0, 1], 3).astype(np.int32), np.array(ls * 2, np.int32),
                      np.ones(6, np.int32), np.ones(6), np.ones(6), omega=omega, tau=0.0)
    rng = np.random.default_rng(11)
    P = rng.standard_normal((s.n_bf, s.n_bf))
    check(hfx_mod, s, P + P.T, 16 * 30 * 1.2e-16)


@pytest.mark.parametrize("nprim,atoms", [(1, 5), (2, 3), (8, 1), (8, 2)])
@pytest.mark.parametrize("mixed", [False, True])
def test_streams_of_few_and_many_primitives(hfx_mod, nprim, atoms, mixed):
    s = inputs.diamond_system(atoms, seed=40 + nprim, nprim=nprim, tau=1e-12, alpha_range=(0.2, 4.0))
    P = inputs.density_matrix(s)
    kw = dict(precision=hfx_mod.HFX_MIXED, fp32_class_mask=hfx_mod.ALL_CLASS_MASK, fp32_tau=1e-3) if mixed else {}
    h = check(hfx_mod, s, P, 1e-6 if mixed else 1e-12, **kw)
    st = h.stats()
    assert sum(st["quartets_evaluated_class"]) > 0
    if mixed and atoms > 1:  # (the quartets of one atom are all large: its mixed build is the FP64 pass)
        assert sum(st["quartets_fp32_class"]) > 0


@pytest.mark.parametrize("alpha", [4e8, 3e10, 2e-10])
def test_mixed_build_at_the_ends_of_the_fp32_range(hfx_mod, alpha):
    """Powers of 2 rho and the prefactors leave FP32's range for such exponents: classes within it take
    the FP32 pass, the others the FP64 pass, all finite and right (a tiny density makes every quartet
    eligible)."""
    xyz = np.array([[0.0, 0.0, 0.0], [1.0, 0.8, -0.6]])
    s = inputs.System("pair", xyz, np.repeat([0, 1], 3).astype(np.int32), np.array([0, 1, 2] * 2, np.int32),
                      np.ones(6, np.int32), np.full(6, alpha) * np.array([1.0, 0.7, 0.9, 0.8, 1.0, 0.6]), np.ones(6),
                      omega=0.11, tau=0.0)
    P = 1e-14 * (np.ones((s.n_bf, s.n_bf)) + np.eye(s.n_bf))
    h = check(hfx_mod, s, P, 1e-6, precision=hfx_mod.HFX_MIXED, fp32_class_mask=hfx_mod.ALL_CLASS_MASK,
              prim_tau=0.0)  # (the oracle drops no primitive pairs)
    n32 = h.stats()["quartets_fp32_class"]
    assert n32[0] > 0 and n32[20] == 0  # (ss|ss) within, (dd|dd) beyond


# (2 rho)^L G leaves FP64's range beyond 4e24 and below 1e-25 in (dd|dd); 1e22 is where scaling begins.  The
# atoms lie an orbital's width apart.  The attenuated kernel cancels at 1e-30, so Coulomb there; no primitive
# pair is dropped by the oracle.
@pytest.mark.parametrize("alpha,omega", [(5e21, 0.11), (2e22, 0.11), (1e25, 0.11), (1e34, 0.11), (1e-30, 0.0)])
@pytest.mark.parametrize("mixed", [False, True])
def test_exponents_at_the_ends_of_the_fp64_range(hfx_mod, alpha, omega, mixed):
    xyz = np.array([[0.0, 0.0, 0.0], [0.4, 0.5, -0.3]]) / np.sqrt(alpha)
    s = inputs.System("pair", xyz, np.repeat([0, 1], 3).astype(np.int32), np.array([0, 1, 2] * 2, np.int32),
                      np.ones(6, np.int32), alpha * np.array([1.0, 0.7, 0.9, 0.8, 1.0, 0.6]), np.ones(6), omega=omega,
                      tau=0.0)
    P = np.ones((s.n_bf, s.n_bf)) + np.eye(s.n_bf)
    kw = dict(precision=hfx_mod.HFX_MIXED, fp32_class_mask=hfx_mod.ALL_CLASS_MASK) if mixed else {}
    h = check(hfx_mod, s, P, 1e-12, prim_tau=0.0, **kw)
    if not mixed:
        Ko, _ = oracle.Screen(oracle.Basis(s)).build_K(P, "sym")
        for cls in range(6):  # ss, ps and pp pairs in the thread kernel
            h.set_group_size(cls, 1)
        K1 = h.build_K(torch.from_numpy(P).cuda()).cpu().numpy()
        assert np.abs(K1 - Ko).max() <= 1e-12 * np.abs(Ko).max()
        # the same from a batch with an ordinary system beside it
        s2 = inputs.diamond_system(1, seed=7, tau=1e-12)
        h2 = hfx_mod.HFX(s2).build_pairs()
        P2 = torch.from_numpy(inputs.density_matrix(s2)).cuda()
        K = [torch.empty_like(P2), torch.empty(P.shape, dtype=torch.float64, device="cuda")]
        hfx_mod.Batch([h2, h]).run([P2, torch.from_numpy(P).cuda()], K)
        torch.cuda.synchronize()
        assert np.abs(K[1].cpu().numpy() - Ko).max() <= 1e-12 * np.abs(Ko).max()


def test_thread_kernel_takes_the_classes_that_fit(hfx_mod):
    """A thread's slots (at most 450 doubles: 64 threads in 227 KB) hold sixteen classes; their op lists are in
    the generated tables, the five others are refused."""
    s = inputs.diamond_system(3, seed=5, tau=1e-10)
    P = torch.from_numpy(inputs.density_matrix(s)).cuda()
    h = hfx_mod.HFX(s).build_pairs()
    K = h.build_K(P).clone()
    refused = []
    for cls in range(21):
        h.set_group_size(cls, 1)
        try:
            K1 = h.build_K(P)
        except hfx_mod.HFXError:
            refused.append(cls)
        else:
            assert torch.abs(K1 - K).max() <= 1e-12 * torch.abs(K).max(), cls
        h.set_group_size(cls, 0)
    assert refused == [14, 17, 18, 19, 20]


@pytest.mark.parametrize("kw", [{}, dict(schedule=0), dict(schedule=1), dict(density_tau=1e-8), dict(precision=1)])
def test_long_uncontracted_lists_take_the_thread_kernel(hfx_mod, kw):
    """48 atoms with s, p, d shells of one primitive: the long lists of the low classes go to the thread kernel
    (in FP64), the other classes stay; against whole warps everywhere."""
    s = inputs.diamond_system(48, seed=3, nprim=1)
    P = torch.from_numpy(inputs.density_matrix(s)).cuda()
    h = hfx_mod.HFX(s, **kw).build_pairs()
    K = h.build_K(P).clone()
    st = h.stats()
    gs = np.array(st["group_size_class"])
    nq = np.array(st["n_quartets_class"])
    low = np.isin(np.arange(21), [0, 1, 2, 3, 4, 6, 7, 10, 15])
    if kw.get("precision"):
        assert np.all(gs[:20] == 32)  # every class but (dd|dd) may take the FP32 pass
    else:
        assert np.all(gs[~low] == 32) and np.all(gs[nq < 1e5] == 32) and np.all(gs[low & (nq > 5e5)] == 1)
        assert (gs == 1).sum() >= 4
    for cls in range(21):
        h.set_group_size(cls, 32)
    K32 = h.build_K(P)
    assert torch.abs(K32 - K).max() <= 1e-12 * torch.abs(K).max()
    if kw.get("schedule") == 1:  # whole rows: no partitions
        return
    parts = torch.zeros_like(K)
    for cls in range(21):
        h.set_group_size(cls, 0)
    for i in range(3):  # (shorter lists)
        parts += h.build_K(P, part=i, n_parts=3)
    assert torch.abs(parts - K).max() <= 1e-12 * torch.abs(K).max()


@pytest.mark.parametrize("mixed", [False, True])
def test_build_inside_a_captured_graph(hfx_mod, mixed):
    """Overlapping class launches (a small system) as a captured graph, replayed for another density."""
    s, P0 = inputs.config1(3)
    h = hfx_mod.HFX(s, stream=torch.cuda.Stream(), precision=hfx_mod.HFX_MIXED if mixed else hfx_mod.HFX_FP64)
    h.build_pairs()
    P, K = torch.from_numpy(P0).cuda(), torch.empty(P0.shape, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=h.stream):
        h.build_K(P, K)
    for seed in (1, 2):
        P1 = inputs.density_matrix(s, seed=seed, truncate_bohr=10.0)
        P.copy_(torch.from_numpy(P1))
        graph.replay()
        torch.cuda.synchronize()
        Ko, _ = oracle.Screen(oracle.Basis(s)).build_K(P1, "sym")
        assert np.abs(K.cpu().numpy() - Ko).max() <= (1e-7 if mixed else 1e-12) * np.abs(Ko).max()


def test_device_memory_of_a_small_context(hfx_mod):
    """What a server's budget counts for a system of 15 shells (120 pairs): the Boys tables (2.5 MB), CUB's
    scratch (1 MB), two slabs of 128 KB, the primitive and Hermite pair data (less than 0.3 MB)."""
    s, _ = inputs.config1(3)
    h = hfx_mod.HFX(s)
    assert h.device_bytes() < 2.7e6
    assert h.build_pairs().device_bytes() < 4.1e6


def test_pair_records_of_few_and_many_pairs(hfx_mod):
    """Primitive-pair records are made by 16 lanes a pair for few pairs and by one for many: the same
    Schwarz factors, bit for bit, for the pairs two systems share (primitive pairs dropped among them)."""
    rng = np.random.default_rng(3)
    n, k = 200, 3  # 20100 and 4950 pairs
    xyz, al = rng.uniform(0, 40, (n, 3)), rng.uniform(0.2, 4.0, (n, k))

    def factors(m):
        s = inputs.System("s", xyz[:m], np.arange(m, dtype=np.int32), np.zeros(m, np.int32), np.full(m, k, np.int32),
                          al[:m].ravel(), np.ones(m * k), omega=0.11, tau=0.0)
        a, b, q = hfx_mod.HFX(s).build_pairs().pairs()
        out = np.zeros((n, n))
        out[a, b] = q
        return out

    many, few = factors(n), factors(99)
    assert (few > 0).sum() > 99 and np.array_equal(many[:99, :99], few[:99, :99])


def test_pair_records_on_both_sides_of_the_line(hfx_mod):
    """The same where 16 lanes a pair just fill the chip and where they just do not, for this chip's SMs."""
    line = torch.cuda.get_device_properties(0).multi_processor_count * 2048 // 16
    n = int((np.sqrt(8.0 * line + 1.0) - 1.0) / 2.0) + 1  # the first n with more than `line` pairs
    assert (n - 1) * n // 2 <= line < n * (n + 1) // 2
    rng = np.random.default_rng(4)
    k = 5  # 25 primitive pairs: two rounds of 16 lanes
    xyz, al = rng.uniform(0, 40, (n, 3)), rng.uniform(0.2, 4.0, (n, k))

    def factors(m):
        s = inputs.System("s", xyz[:m], np.arange(m, dtype=np.int32), np.zeros(m, np.int32), np.full(m, k, np.int32),
                          al[:m].ravel(), np.ones(m * k), omega=0.11, tau=0.0)
        a, b, q = hfx_mod.HFX(s).build_pairs().pairs()
        out = np.zeros((n, n))
        out[a, b] = q
        return out

    many, few = factors(n), factors(n - 1)
    assert (few > 0).sum() > n and np.array_equal(many[:n - 1, :n - 1], few[:n - 1, :n - 1])
