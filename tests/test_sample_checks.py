"""The host pass over multicanonical samples: one non-finite sample at any place
is refused by its index, and finite ones of any size are not.  No GPU needed."""
import os

import numpy as np
import pytest

from paper_1509_08391_gb300 import llr

pytestmark = pytest.mark.skipif(not os.path.exists(llr.LIB_PATH), reason="library not built")


@pytest.mark.parametrize("ns", [1, 7, 8, 9, 17])
@pytest.mark.parametrize("bad", [np.nan, -np.nan, np.inf, -np.inf])
def test_every_place_is_checked(ns, bad):
    for i in range(ns):
        E = np.linspace(11.0, 12.0, ns)
        E[i] = bad
        with pytest.raises(llr.LLRError) as e:
            llr.muca_reweight(E, 10.0, 2.5, [-1.0, -1.1], [1.0])
        assert e.value.code == llr.LLR_ERR_ARG and "sample %d " % i in str(e.value)


def test_a_distance_beyond_the_largest_double_is_no_bad_sample():
    try:
        llr.muca_reweight([1.7e308, 1.0], -1.7e308, 1e300, [-1.0], [1.0])
    except llr.LLRError as e:   # without a GPU
        assert e.code == llr.LLR_ERR_CUDA
