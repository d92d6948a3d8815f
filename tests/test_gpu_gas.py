"""A gas: cells that are mostly empty, lists of a few entries or none.  The lists against the oracle's, exactly."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import assert_lists_equal, gpu_lists, margin_ok

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,lst", [("mixed", "full"), ("mixed", "half"), ("fp64", "full")])
@pytest.mark.parametrize("n,box", [(1500, (40.0, 44.0, 52.0)), (5000, (110.0, 70.0, 90.0))])
def test_lists_among_empty_cells(n, box, precision, lst):
    from paper_1009_4330_gb300 import System
    box = np.array(box)
    x = np.random.default_rng(n).random((n, 3)) * box
    assert margin_ok(x, box, 2.8)
    ref = oracle.neighbors(x, box, 2.8)
    with System.lj(x, np.zeros_like(x), box, cutoff=2.5, skin=0.3, dt=0.005, mass=1.0, precision=precision, list=lst,
                   tpa=1) as s:
        got = gpu_lists(*s.neighbors())
    if lst == "full":
        assert_lists_equal(got, ref)
    else:
        pairs = {(min(i, int(j)), max(i, int(j))) for i, r in enumerate(got) for j in r}
        assert sum(len(r) for r in got) == len(pairs) and pairs == {(i, int(j)) for i, r in enumerate(ref) for j in r if i < j}
