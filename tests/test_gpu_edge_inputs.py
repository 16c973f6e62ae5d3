"""Calls whose inputs or settings lie off the usual range."""
import numpy as np
import pytest

from paper_1509_08391_gb300 import llr, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1509_08391_gb300 import build
    build.build()


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
