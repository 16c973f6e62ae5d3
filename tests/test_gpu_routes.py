"""The routes a call can take through the kernels, at the sizes where they part.

Sides: L <= 10 stays in shared memory (one link per thread), L = 12 .. 24 has its
x3 slabs there (pairs in a row where 4 divides L, pairs at x2 and x2 + L / 2
where not), L = 26 and 28 read them in place; L = 2 and 6 leave most of a warp
idle.  Batches: one, two, three or more lattices per CTA.  Every route against the FP64 oracle
(tolerances of tests/gpu_helpers.py) or bit for bit against another route."""
import numpy as np
import pytest

import oracle
from oracle import mlp as omlp
from oracle import recon
from paper_1509_08391_gb300 import llr, workloads
from tests import gpu_helpers as gh
from tests.test_gpu_mlp import _data, flat_to_list, list_to_flat
from tests.test_gpu_parity_fullsize import _check_or_pass

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1509_08391_gb300 import build
    build.build()
    oracle.build()


def _workload(L, n, dE=None, block=1, seed=11):
    dE = dE or max(4.0, 8.0 * (L / 8) ** 2)
    w = workloads._grid("routes", [L], n, 0.60, 0.66, [dE], 1, seed)
    w.block = block
    return w


def _ordered(L, n, seed=0):
    """Configurations in which a pass does not multiply rounding errors."""
    return np.random.default_rng([seed, L]).normal(0.0, 0.35, (n, 4 * L ** 4)).astype(np.float32)


@pytest.mark.parametrize("L,block,threads", [
    (2, 1, 512), (4, 2, 512), (6, 1, 512), (6, 32, 256), (6, 2, 128), (10, 1, 512),
    (10, 8, 256), (14, 1, 256), (14, 1, 512), (18, 1, 160)])
def test_class_updates_match_oracle(L, block, threads):
    """Every class of a heat-bath and an overrelaxation pass: groups of links
    that end a class in any place, every block size, every team."""
    n = 2 if L <= 10 else 1
    # a CTA takes more than one lattice where the batch has that many for every SM
    total = n if threads == 512 else 919
    w = _workload(L, total, block=block)
    if L == 2:   # 96 plaquettes: a window that any energy is in
        w.E_lo, w.dE = [-100.0] * n, [200.0] * n
    a = np.linspace(-1.02, -0.98, total)
    with llr.Batch.from_workload(w, max_approach=5000) as b:
        b.set_kernel_config(threads, True)
        b.sweep(a, 2)
        rep = gh.check_class_updates(b, w, range(n), a)
    assert rep["links"] == 2 * n * 4 * L ** 4
    assert gh.near_ties_are_rare(rep), rep


@pytest.mark.parametrize("L,n", [(2, 2), (6, 2), (10, 1), (12, 2), (14, 2), (16, 1), (18, 1),
                                 (20, 1), (22, 1), (24, 1), (26, 1), (28, 1)])
def test_overrelaxation_pass_matches_oracle(L, n):
    w = _workload(L, n)
    six_v = 6.0 * L ** 4
    w.E_lo, w.dE = [-1.1 * six_v] * n, [2.2 * six_v] * n
    rep = {}
    with llr.Batch.from_workload(w, max_approach=0) as b:
        for i, th in enumerate(_ordered(L, n)):
            b.set_links(i, th)
        _check_or_pass(b, w, np.full(n, -1.0), rep)
    assert rep["or_links"] == n * 4 * L ** 4


@pytest.mark.parametrize("L", [4, 6, 10, 12, 14, 20])
def test_chains_do_not_depend_on_lattices_per_cta(L):
    """1, 3, 4 and 6 lattices per CTA, with and without fast math, in windows."""
    w = _workload(L, 919)
    a = np.linspace(-1.02, -0.99, w.n_lattices)
    for fast in (True, False):
        outs = []
        for threads in (512, 256, 160, 128):
            with llr.Batch.from_workload(w, max_approach=0) as b:
                b.set_kernel_config(threads, fast)
                n_app = b.approach(3000)
                s = b.sweep(a, 2, measure=True)
                outs.append((n_app, s, b.tracked_energy(), b.get_links(w.n_lattices - 1),
                             b.stats()["hb_acc"]))
        for o in outs[1:]:
            assert all(np.array_equal(x, y) for x, y in zip(o, outs[0]))
        if L >= 12:
            break   # the accurate functions differ from fast math in the proposals only


def test_batch_sizes_that_choose_other_teams_give_the_same_chains():
    """310 and 240 lattices (three and two per CTA) against 5 (one)."""
    w = _workload(4, 310, dE=8.0)
    a = np.linspace(-1.02, -0.99, w.n_lattices)
    ref = None
    for n in (310, 240, 5):
        with llr.Batch.from_workload(workloads.subset(w, range(n)), max_approach=2000) as b:
            s, m = b.rm_step(a[:n], 1, 3, 2)
            got = (s[:5], m[:5], b.tracked_energy()[:5], b.get_links(4))
        if ref is None:
            ref = got
        assert all(np.array_equal(x, y) for x, y in zip(got, ref))


@pytest.mark.parametrize("n_int,jump,a0", [(1, 0.0, -1.0), (3, 0.5, -0.9), (400, 0.05, -1.0)])
def test_multicanonical_decisions_with_rough_tables(n_int, jump, a0):
    """One interval, slopes that jump, and intervals narrower than a move (more
    than one edge between the energies): the accept test's exact form decides
    where the float32 form is not sure."""
    w = workloads.subset(workloads.small_l4(), range(4))
    six_v = 6.0 * 4 ** 4
    e0, de = 0.5 * six_v, 0.25 * six_v / n_int
    a = -0.95 + jump * np.random.default_rng(5).uniform(-1, 1, n_int)
    weight = oracle.MucaWeight(e0, de, a)
    flips = 0
    with llr.Batch.from_workload(w, max_approach=1000) as b:
        b.sweep(np.full(w.n_lattices, -1.0), 1)
        b.set_muca_weight(e0, de, a, a0)
        for cls in (0, 3, 6):
            mirrors = {i: gh.oracle_mirror(b, w, i) for i in range(w.n_lattices)}
            S = {i: mirrors[i].staple_moduli() for i in mirrors}
            b.single_pass(2, None, class_mask=1 << cls)
            for i, o in mirrors.items():
                tr = oracle.muca_class_trace(o, weight, cls, a0)
                order = gh.class_links(w.L[i], cls)
                d = np.abs(gh.wrapped_diff(b.get_links(i).astype(np.float64), o.links()))[order]
                bad = np.nonzero(d > gh.link_tolerance(S[i])[order])[0]
                if bad.size:   # the first difference must be a decision at a near tie
                    k = int(bad[0])
                    assert abs(np.log(tr["u"][k]) - tr["x"][k]) < 1e-4, (cls, i, k)
                    flips += 1
    assert flips <= 2


@pytest.mark.parametrize("L", [2, 12, 26])
def test_fp64_energy_over_many_blocks(L):
    """One lattice spread over the GPU, and lattices of different sides."""
    w = workloads.Workload("e", [L, 4], [0.0, 0.0], [1.0, 1.0], [0, 1], [0, 0], 42)
    with llr.Batch.from_workload(w, max_approach=0) as b:
        th = _ordered(L, 1)[0]
        b.set_links(0, th)
        E = b.energy()
        g = oracle.Geom([L] * 4)
        o = oracle.Lattice(g, w.seed, 0, 0, 0.0, 1.0)
        o.set_links(th.astype(np.float64))
        assert abs(E[0] - o.energy()) <= 1e-12 * 6 * L ** 4
        assert abs(b.tracked_energy()[0] - o.energy()) <= 1e-12 * 6 * L ** 4 + 2.0 ** -32


@pytest.mark.parametrize("n,n_grid,tol", [(2, 2, 1.0), (40, 2, 1e-9), (300, 101, 1e-4),
                                          (513, 257, 1e-12), (64, 33, 1e-300)])
def test_cv_peak_search_depths(n, n_grid, tol):
    """No golden-section step, a few, many, and the limit of 200 (a tolerance no
    interval can reach)."""
    rng = np.random.default_rng(n)
    c = np.linspace(900.0, 1100.0, n)
    a = -1.0 + 0.002 * (c - 1000.0) + 1e-3 * rng.normal(size=n)
    bg, cg = llr.cv_peak(c, a, 0.5, 1.5, n_grid, tol)
    bo, co = recon.cv_peak(c, a, 0.5, 1.5, n_grid, max(tol, 1e-13))
    # the flat top of C_V leaves beta_c uncertain by its square root of the rounding
    assert abs(bg - bo) < max(1e-7, tol) and abs(cg - co) < 1e-8 * max(1.0, co)


@pytest.mark.parametrize("ns,n_beta", [(1, 1), (3, 4), (255, 5), (70001, 9)])
def test_reweighting_sizes(ns, n_beta):
    six_v = 6.0 * 10 ** 4
    e0, de = 0.59 * six_v, 0.1 * six_v / 64
    rng = np.random.default_rng(ns)
    a = -1.01 + 0.004 * np.sin(np.linspace(0, 3, 64))
    E = rng.uniform(e0 - 300.0, e0 + 64 * de + 300.0, ns)
    w = oracle.MucaWeight(e0, de, a)
    lr = np.array([w.lnrho(x) for x in E])
    betas = np.linspace(0.9, 1.1, n_beta)
    g1, g2 = llr.muca_reweight(E, e0, de, a, betas)
    for b, x1, x2 in zip(betas, g1, g2):
        o1, o2 = recon.muca_moments(E, lr, b)
        assert x1 == pytest.approx(o1, rel=1e-12) and x2 == pytest.approx(o2, rel=1e-12)


def test_reweighting_beyond_the_exponents_of_the_table_form():
    """Exponents above 2^39 take the general kernel: all the weight is on the
    largest sample."""
    E = np.array([0.0, 1.0, 2.0, 3.0]) * 1e12
    e1, e2 = llr.muca_reweight(E, 0.0, 1e12, np.zeros(4), [2.0, -2.0, 0.0])
    assert np.allclose(e1, [3e12, 0.0, 1.5e12], rtol=1e-14, atol=0)
    assert np.allclose(e2, [9e24, 0.0, 3.5e24], rtol=1e-14, atol=0)


@pytest.mark.parametrize("n", [1, 8, 9, 127, 129, 300])
def test_training_splits_of_the_samples(n):
    """Fewer samples than CTAs, ragged shares, tiles and chunks: five Adam steps
    within 1e-4 relative of the FP64 oracle's, as at 200 samples."""
    L, e, d, t = _data(n, 40 + n)
    raw = omlp.features(L, e, d)
    mean, std = raw.mean(axis=0), raw.std(axis=0)
    std = np.where(std > 0, std, 1.0)
    with llr.MLP(seed=5) as net:
        p = flat_to_list(net.get_params().astype(np.float64))
        net.set_params(list_to_flat(p))
        net.set_norm(mean, std)
        net.fit(L, e, d, t, epochs=2, lr=1e-3, standardise=False)
        net.fit(L, e, d, t, epochs=3, lr=1e-3, standardise=False)   # moments carry over
        x = (raw - mean) / std
        opt = omlp.Adam(p, lr=1e-3)
        for _ in range(5):
            p = opt.step(p, omlp.backward(p, x, t))
        for a, b in zip(flat_to_list(net.get_params().astype(np.float64)), p):
            assert np.max(np.abs(a - b)) <= 1e-4 * max(1.0, np.max(np.abs(b)))
