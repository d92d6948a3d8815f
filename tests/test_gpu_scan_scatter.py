"""The bin scan and the scatter of one system of at most 8,192 bins in one launch: numbers of bins at
the edges of its split (groups of four, 2,048 per pass, the largest and the first beyond it), atom counts about
its block of 512.  Exact: the lists are sets of integers."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_lists_equal, gpu_lists, margin_ok

pytestmark = pytest.mark.gpu

RL = 1.3  # cut-off + skin


@pytest.mark.parametrize("cells,n", [((2, 2, 2), 1), ((3, 3, 3), 64), ((2, 5, 7), 511), ((8, 16, 16), 512),
                                     ((3, 23, 31), 513), ((16, 16, 32), 1025), ((16, 32, 16), 6000),
                                     ((17, 16, 31), 1500)])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_lists_at_the_edges_of_the_scan(cells, n, precision):
    from paper_1009_4330_gb300 import System
    box = np.array(cells) * RL * 1.0001
    rng = np.random.default_rng(sum(cells) + n)
    sites = np.floor(box / 0.65).astype(int)
    pick = rng.choice(sites.prod(), n, replace=False)
    x = (np.stack(np.unravel_index(pick, sites), 1) + 0.5 + rng.uniform(-0.1, 0.1, (n, 3))) * (box / sites)
    assert margin_ok(x, box, RL)
    ref = oracle.neighbors(x, box, RL)
    with System.lj(x, np.zeros_like(x), box, cutoff=1.0, skin=0.3, dt=0.005, mass=1.0, precision=precision,
                   tpa=1) as s:
        assert_lists_equal(gpu_lists(*s.neighbors()), ref)
        s.set_state(x=np.roll(x, 1, axis=0))  # the same sites, other atoms on them: the bins are counted afresh
        got = gpu_lists(*s.neighbors())
    assert_lists_equal(got, oracle.neighbors(np.roll(x, 1, axis=0), box, RL))
