"""Calls whose inputs or settings lie off the usual range."""
import numpy as np
import pytest

import oracle
from paper_1509_08391_gb300 import llr, workloads
from tests import gpu_helpers as gh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1509_08391_gb300 import build
    build.build()
    oracle.build()


@pytest.mark.parametrize("L", [4, 10, 12, 14])
@pytest.mark.parametrize("poison", ["one", "pair", "all", "inf"])
def test_links_that_are_no_numbers_are_reported(L, poison):
    """A resync of such a lattice: status LLR_ERR_NUMERIC and no energy, however
    many plaquettes the links take with them; the others are as without it."""
    w = workloads._grid("nan", [L], 3, 0.60, 0.66, [40.0], 1, 7)
    th = np.random.default_rng(L).uniform(-3.0, 3.0, 4 * L ** 4).astype(np.float32)
    bad = th.copy()
    if poison == "all":
        bad[:] = np.nan
    elif poison == "inf":
        bad[L ** 4 + 5] = np.inf
    else:
        bad[[7] if poison == "one" else [7, 2 * L ** 4 + 1]] = np.nan
    with llr.Batch.from_workload(w, max_approach=0) as b:
        for i in range(3):
            b.set_links(i, bad if i == 1 else th)
        b.single_pass(3)   # the end of a composite sweep: a fresh energy
        E = b.tracked_energy()
        assert np.isnan(E[1])
        assert list(b.status()) == [0, llr.LLR_ERR_NUMERIC, 0]
        assert abs(E[0] - b.energy()[0]) < 1e-3 and E[0] == E[2]


def test_robbins_monro_step_reports_links_that_are_no_numbers():
    w = workloads.subset(workloads.small_l4(), [0, 1])
    with llr.Batch.from_workload(w, max_approach=1000) as b:
        th = b.get_links(1)
        th[3] = np.nan
        b.set_links(1, th)
        with pytest.raises(llr.LLRError) as e:
            b.rm_step(np.array([-1.0, -1.0]), 0, 1, 0)
        assert e.value.code == llr.LLR_ERR_NUMERIC
        assert list(b.status()) == [0, llr.LLR_ERR_NUMERIC]


@pytest.mark.parametrize("jump", [0.05, 2.0, 10.0])
def test_multicanonical_decisions_far_from_the_table_origin(jump):
    """A table that starts 1e9 below the energies, with a jump of the slope at
    them: float32 places the energy to no better than 32, so only the exact form
    of the accept test can decide."""
    w = workloads.subset(workloads.small_l4(), range(4))
    a0, de, n = -1.0, 1e8, 20
    a = np.where(np.arange(n) < 10, -1.0, -1.0 + jump)
    with llr.Batch.from_workload(w, max_approach=1000) as b:
        b.sweep(np.full(w.n_lattices, -1.0), 1)
        e0 = float(np.round(np.median(b.tracked_energy()))) - 10 * de   # edge 10: that energy
        weight = oracle.MucaWeight(e0, de, a)
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
                    assert abs(np.log(tr["u"][k]) - tr["x"][k]) < 1e-4 * (1 + jump), (cls, i, k)


def test_accurate_functions_keep_the_automatic_shape():
    """Asking for the default shape, to change the functions only, leaves the
    lattices per CTA to the batch, in a launch and in a captured step alike."""
    import torch
    w = workloads._grid("auto", [4], 200, 0.60, 0.66, [8.0], 1, 3)
    a = np.full(w.n_lattices, -1.0)
    ad = torch.full((w.n_lattices,), -1.0, dtype=torch.float64, device="cuda")
    grids = []
    with llr.Batch.from_workload(w, max_approach=0) as b:
        for setting in (None, lambda: b.set_kernel_shape(256, True, 4, -1),
                        lambda: b.set_kernel_config(256, False)):
            if setting:
                setting()
            b.sweep(a, 1)
            grids.append(b.last_launch()["grid"])
            b.rm_run(ad, 0, 1, 0, 1)
            torch.cuda.synchronize()
            grids.append(b.last_launch()["grid"])
    assert len(set(grids)) == 1, grids


def test_sides_that_alternate_give_the_chains_of_separate_batches():
    """Several lattices of different sides to a CTA, in and out of shared memory:
    every chain, history and energy is that of a batch of its side alone."""
    import torch
    for Ls in ([4, 8, 2], [4, 12, 6]):
        n = 170
        w = workloads._grid("mix", Ls, n, 0.60, 0.66, [16.0] * 3, 1, 9)
        idx = [(i % 3) * n + i // 3 for i in range(3 * n)]
        runs = {}
        for part in (idx, list(range(n)), list(range(n, 2 * n)), list(range(2 * n, 3 * n))):
            with llr.Batch.from_workload(workloads.subset(w, part), max_approach=0) as b:
                app = b.approach(1000) if 2 not in Ls else np.zeros(len(part), dtype=np.int32)
                a, mean = b.rm_step(np.full(len(part), -1.0), 1, 2, 3)
                ad = torch.tensor(a, device="cuda")
                hist = torch.zeros((2, len(part)), dtype=torch.float64, device="cuda")
                b.rm_run(ad, 0, 2, 4, 2, hist)
                E = b.tracked_energy()
                h = hist.cpu().numpy()
                for k, i in enumerate(part):
                    got = (app[k], a[k], mean[k], E[k], h[0, k], h[1, k],
                           hash(b.get_links(k).tobytes()))
                    assert runs.setdefault(i, got) == got, (Ls, i)
        assert len(runs) == 3 * n


@pytest.mark.parametrize("L,n,sweeps,grid", [(4, 160, 1, 80), (8, 200, 1, 100), (12, 200, 1, 100),
                                             (12, 200, 12, 152), (8, 152, 1, 152)])
def test_lattices_per_cta_follow_the_rounds_a_launch_takes(L, n, sweeps, grid):
    """Somewhat more lattices than SMs: two to a CTA for a sweep of which the GPU
    would otherwise take two rounds, one where the rounds of many sweeps fill it."""
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the sizes are those of 152 SMs")
    w = workloads._grid("rounds", [L], n, 0.60, 0.66, [8.0], 1, 3)
    with llr.Batch.from_workload(w, max_approach=0) as b:
        b.sweep(np.full(n, -1.0), sweeps)
        assert b.last_launch()["grid"] == grid


def test_a_coupling_does_not_depend_on_those_asked_for_with_it():
    """Bit for bit, for few and many couplings a launch, whole and ragged groups."""
    rng = np.random.default_rng(3)
    E = rng.normal(37000.0, 150.0, 200000)
    a = -1.0 + 1e-3 * rng.normal(size=64)
    betas = np.linspace(0.99, 1.01, 301)

    def f(b):
        return np.array(llr.muca_reweight(E, 36000.0, 2000 / 64, a, b))

    ref = f(betas)
    for k in (1, 3, 4, 5, 43):
        got = np.concatenate([f(betas[i:i + k]) for i in range(0, betas.size, k)], axis=1)
        assert np.array_equal(got, ref), k
