"""Rebuilds of a batch inside md_step: by rows of cells where few (cell, part) units rebuild in a step, by whole cells where many do
(both builds are launched and one returns).  Whichever it is, every replica's trajectory is that of the replica
alone, bit for bit, with few and with all replicas rebuilding together, in batches on each side of the limits; a
list that overflows in such a step grows and the step is completed; and dense cells do not make it slow."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _replica(n, seed, temperature=1.44):
    x, box = synth.fcc_subset(n, 0.8442, seed)
    x = synth.displace(x, box, 0.03, seed + 1)
    return {"x": x, "v": synth.maxwell_boltzmann(n, temperature, 1.0, seed + 2), "box": box}


def _kw(rc, precision="mixed", lst="full", skin=0.3):
    from paper_1009_4330_gb300 import lj_params
    return dict(params=lj_params(1.0, 1.0, 1), cutoff=rc, skin=skin, dt=0.004, mass=1.0, precision=precision, list=lst,
                tpa=1)


@pytest.mark.parametrize("precision,lst", [("mixed", "full"), ("fp64", "full")])
@pytest.mark.parametrize("copies,n,rc", [(3, 700, 2.5),     # by rows only
                                         (40, 1237, 2.5),   # either
                                         (30, 1237, 4.4),   # either, cells of over a hundred atoms
                                         (200, 1237, 2.5)])  # by cells only
@pytest.mark.parametrize("together", [False, True])
def test_trajectories_are_the_replicas_alone(copies, n, rc, together, precision, lst):
    from paper_1009_4330_gb300 import System
    r = [_replica(n, 51 if together else 51 + 10 * k) for k in range(copies)]
    kw = _kw(rc, precision, lst)
    with System.batch(r, **kw) as b:
        b.step(25)
        x = b.state()[0].cpu().numpy().reshape(copies, n, 3)
        assert b.info()["rebuilds"] >= 2 * copies
    for k in (0, copies - 1):
        with System(r[k]["x"], r[k]["v"], None, r[k]["box"], potential="lj", **kw) as s:
            s.step(25)
            assert np.array_equal(s.state()[0].cpu().numpy(), x[k])


@pytest.mark.parametrize("copies", [3, 60])
def test_lists_grow_inside_a_step(copies):
    """Two slabs of liquid driven into each other (as in test_gpu_overflow): the lists outgrow their capacity in a call."""
    from paper_1009_4330_gb300 import System
    from test_gpu_overflow import colliding_slabs
    x, v, box = colliding_slabs()
    r = {"x": x, "v": v, "box": box}
    kw = dict(_kw(2.5), dt=0.0005)
    with System.batch([r] * copies, **kw) as b, System(x, v, None, box, potential="lj", **kw) as s:
        before = b.info()["maxneigh"]
        b.step(300)
        s.step(300)
        assert b.info()["maxneigh"] > before and b.info()["steps"] == 300
        xb = b.state()[0].cpu().numpy().reshape(copies, len(x), 3)
        assert np.array_equal(xb[0], xb[-1]) and np.array_equal(xb[0], s.state()[0].cpu().numpy())


def test_dense_cells_that_rebuild_together_are_not_slow():
    """A rebuild in every step (a tiny skin), inside md_step and by md_build_neighbors, which builds by cells: the same time as
    measured, 2.0 times it when such a batch was built by rows."""
    import torch
    from paper_1009_4330_gb300 import System
    r = _replica(8000, 51)
    with System.batch([r] * 40, **_kw(5.0, skin=0.002)) as b:
        def ms(fn):
            best = 1e9
            for _ in range(5):
                e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
                e[0].record()
                fn()
                e[1].record()
                torch.cuda.synchronize()
                best = min(best, e[0].elapsed_time(e[1]))
            return best

        b.step(3)
        one, built = ms(lambda: b.step(10)) / 10, ms(b.build_neighbors)
        assert one < 1.4 * built
