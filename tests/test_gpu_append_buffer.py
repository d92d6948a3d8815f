"""The list build by whole cells and its append buffer, in systems with more (cell, part) units than the build by rows
takes (six per SM): every list layout, full and half, lists longer than the buffer, and capacities that are
outgrown in that build.  Against the lists of one replica alone, which are built by rows, and the oracle's.  Exact."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import assert_lists_equal, margin_ok

pytestmark = pytest.mark.gpu

LAYOUTS = [(t, q) for t in (1, 2, 4, 8, 16, 32) for q in (1, 2, 4)]


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def _lists(s):
    c, nb = s.neighbors()
    c, nb = c.cpu().numpy(), nb.cpu().numpy()
    return [nb[i, :c[i]].copy() for i in range(c.size)]


def _kw(rc, lst="full", precision="mixed", tpa=1):
    from paper_1009_4330_gb300 import lj_params
    return dict(params=lj_params(1.0, 1.0, 1), cutoff=rc, skin=0.3, dt=0.005, mass=1.0, precision=precision, list=lst, tpa=tpa)


def _units(s, n):
    cells = int(np.prod(s.info()["bins"]))
    return cells * max(1, min(8, int(np.ceil(1.15 * n / cells / 32))))


@pytest.mark.parametrize("lst,precision", [("full", "mixed"), ("half", "mixed"), ("full", "fp64")])
@pytest.mark.parametrize("rc", [2.5, 4.4])
def test_every_layout(rc, lst, precision):
    from paper_1009_4330_gb300 import System
    n = 1237
    x, box = synth.fcc_subset(n, 0.8442, 11)
    x = synth.displace(x, box, 0.05, 12)
    assert margin_ok(x, box, rc + 0.3)
    r = {"x": x, "v": np.zeros_like(x), "box": box}
    with System(x, r["v"], None, box, **_kw(rc, lst, precision)) as s:
        units = _units(s, n)
        assert units <= 6 * _sms()  # by rows
        solo = _lists(s)
    if lst == "full":
        assert_lists_equal([np.sort(a) for a in solo], oracle.neighbors(x, box, rc + 0.3))
    copies = 8 * _sms() // units + 1  # by cells
    with System.batch([r] * copies, **_kw(rc, lst, precision)) as b:
        for tpa, vec in LAYOUTS:
            b.set_kernel(tpa, lst, 128, vec)
            got = _lists(b)
            for k in (0, copies - 1):
                assert all(np.array_equal(a, c) for a, c in zip(got[k * n:(k + 1) * n], solo)), (tpa, vec)


@pytest.mark.parametrize("tpa,vec", LAYOUTS)
def test_outgrown_capacity(tpa, vec):
    """Every replica's atoms fall from all over a tall box into a dense slab at its bottom, all but one of them."""
    from paper_1009_4330_gb300 import System
    n, box = 1000, np.array([8.7, 8.7, 150.0])
    y, _ = synth.fcc_subset(n, 1.3, 21)
    y = synth.displace(y[:, [0, 1, 2]] * (8.7 / (n / 1.3) ** (1 / 3)) * 0.999, np.full(3, 8.7), 0.02, 22)
    y[-1] = (4.0, 4.0, 80.0)
    assert margin_ok(y, box, 4.3)
    x = np.random.default_rng(1).random((n, 3)) * box
    ref = oracle.neighbors(y, box, 4.3)
    r = {"x": x, "v": np.zeros_like(x), "box": box}
    copies = 8 * _sms() // (2 * 2 * 34) + 1
    with System.batch([r] * copies, **_kw(4.0)) as b:
        assert _units(b, n) * copies > 6 * _sms()
        b.set_kernel(tpa, "full", 128, vec)
        before = b.info()["maxneigh"]
        b.set_state(x=np.concatenate([y] * copies))
        assert b.info()["maxneigh"] > before and max(map(len, ref)) > before
        got = _lists(b)
        for k in (0, copies // 2, copies - 1):
            assert_lists_equal([np.sort(a) for a in got[k * n:(k + 1) * n]], ref)
