"""The list build's append buffer (entries written out four at a time, in
candidate order): every list layout holds the same entries in the same order,
full and half lists, lists shorter than four entries and longer than the
buffer, and a capacity that has to grow on the way.  Exact: integers only."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import assert_lists_equal, gpu_lists, margin_ok

pytestmark = pytest.mark.gpu


def _neighbors(s):
    c, nb = s.neighbors()
    c, nb = c.cpu().numpy(), nb.cpu().numpy()
    return [nb[i, :c[i]].copy() for i in range(c.size)]


@pytest.mark.parametrize("rho,rc", [(0.02, 2.5), (0.8442, 2.5), (0.8442, 4.4)])
def test_lists_do_not_depend_on_the_layout(rho, rc):
    from paper_1009_4330_gb300 import System
    n = 1237
    x, box = synth.fcc_subset(n, rho, 11)
    x = synth.displace(x, box, 0.05, 12)
    assert margin_ok(x, box, rc + 0.3)
    ref = oracle.neighbors(x, box, rc + 0.3)
    with System.lj(x, np.zeros_like(x), box, cutoff=rc, skin=0.3, dt=0.005, mass=1.0, precision="mixed", tpa=1) as s:
        first = _neighbors(s)
        assert_lists_equal([np.sort(r) for r in first], ref)
        for tpa in (1, 2, 4, 8, 16, 32):
            for vec in (1, 2, 4):
                s.set_kernel(tpa, "full", 128, vec)
                assert all(np.array_equal(a, b) for a, b in zip(_neighbors(s), first)), (tpa, vec)
        half = None
        for tpa, vec in ((1, 4), (4, 2), (32, 1)):
            s.set_kernel(tpa, "half", 128, vec)
            got = _neighbors(s)
            half = half or got
            assert all(np.array_equal(a, b) for a, b in zip(got, half)), (tpa, vec)
        assert sum(len(r) for r in half) * 2 == sum(len(r) for r in ref)


def test_capacity_grows_from_far_too_small():
    """A dense slab in a box of low mean density: the first capacity guess is far below the longest list."""
    from paper_1009_4330_gb300 import System
    x, _ = synth.fcc_subset(2000, 1.0, 21)
    x = synth.displace(x, np.full(3, 12.6), 0.03, 22)
    box = np.array([12.6, 12.6, 120.0])
    assert margin_ok(x, box, 4.3)
    ref = oracle.neighbors(x, box, 4.3)
    with System.lj(x, np.zeros_like(x), box, cutoff=4.0, skin=0.3, dt=0.005, mass=1.0, precision="mixed", tpa=2) as s:
        assert_lists_equal(gpu_lists(*s.neighbors()), ref)


@pytest.mark.parametrize("rc,copies", [(2.5, 60), (4.4, 130)])
def test_row_build_equals_the_cell_build(rc, copies):
    """A small system's lists are built by rows of cells, those of a batch with many cells by whole cells:
    the same entries in the same order (rc 4.4: rows of more candidates than are kept between the passes)."""
    from paper_1009_4330_gb300 import System, lj_params
    n = 1237
    x, box = synth.fcc_subset(n, 0.8442, 11)
    x = synth.displace(x, box, 0.05, 12)
    r = {"x": x, "v": np.zeros_like(x), "box": box}
    kw = dict(params=lj_params(1.0, 1.0, 1), cutoff=rc, skin=0.3, dt=0.005, mass=1.0, precision="mixed", tpa=1)
    for lst in ("full", "half"):
        with System(x, r["v"], None, box, list=lst, **kw) as s:
            solo = _neighbors(s)
        with System.batch([r] * copies, list=lst, **kw) as b:
            assert all(np.array_equal(a, c) for a, c in zip(_neighbors(b), solo))
