"""The FP64 list passes (eight lanes per atom, FP32 pre-test, one wave of
warps) at the sizes where their work split changes, against the oracle:

* fewer atoms than a warp's four groups, ragged ends, one atom more or less
  than a batch of 32, and both sides of the size (16 warps of 4 atoms per SM) at which
  one wave holds every atom;
* several atom types, full and half lists, every list layout (the result does
  not depend on it: bitwise for full lists).

Tolerances: TOL_FP64 (1e-12 relative max-norm), hundreds of roundings of a
sum of ~50 FP64 terms; half lists add their terms in any order.
"""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import TOL_FP64, rel_maxnorm

pytestmark = pytest.mark.gpu

EPS = np.array([[1.0, 1.5, 0.8], [1.5, 0.5, 1.1], [0.8, 1.1, 0.9]])
SIG = np.array([[1.0, 0.8, 0.9], [0.8, 0.88, 0.95], [0.9, 0.95, 1.05]])


def _case(n, nt, seed=5):
    x, box = synth.fcc_subset(max(n, 160), 0.8442, seed)  # the box of at least 160 atoms: 5.6 < edge
    x = synth.displace(x[:n], box, 0.03, seed + 1)
    t = np.random.default_rng(seed).integers(0, nt, n).astype(np.int32)
    return x, box, t


@pytest.mark.parametrize("nt,lst", [(1, "full"), (1, "half"), (3, "full"), (3, "half")])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 31, 33, 161, 601, 9727, 9761])
def test_forces_at_the_edges_of_the_split(n, nt, lst):
    from paper_1009_4330_gb300 import System
    x, box, t = _case(n, nt)
    e, s = EPS[:nt, :nt], SIG[:nt, :nt]
    fr, er, wr = oracle.lj(x, box, 2.5, eps=e, sig=s, types=t, n_types=nt)
    with System.lj(x, np.zeros_like(x), box, eps=e, sig=s, types=t, n_types=nt, cutoff=2.5, skin=0.3, dt=0.005,
                   mass=[1.0] * nt, precision="fp64", list=lst, tpa=1) as h:
        f = h.compute_forces().cpu().numpy()
        ev = h.energy_virial().cpu().numpy()[0]
    if n == 1:
        assert not f.any() and not ev.any()
        return
    assert np.abs(f - fr).max() <= TOL_FP64 * np.abs(fr).max()
    assert abs(ev[0] - er) <= 1e-11 * max(1.0, abs(er))


@pytest.mark.parametrize("tpa,vec", [(1, 1), (1, 2), (2, 4), (8, 4), (32, 1)])
def test_forces_do_not_depend_on_the_list_layout(tpa, vec):
    from paper_1009_4330_gb300 import System
    x, box, t = _case(601, 1)
    with System.lj(x, np.zeros_like(x), box, cutoff=2.5, skin=0.3, dt=0.005, mass=1.0, precision="fp64", tpa=1) as h:
        f0 = h.compute_forces().cpu().numpy()
        h.set_kernel(tpa, "full", 128, vec)
        assert np.array_equal(h.compute_forces().cpu().numpy(), f0)


@pytest.mark.parametrize("nt", [1, 2, 3])
@pytest.mark.parametrize("n", [161, 601, 9761])
def test_backward_at_the_edges_of_the_split(n, nt):
    from paper_1009_4330_gb300 import System
    x, box, t = _case(n, nt, seed=9)
    e, s = EPS[:nt, :nt], SIG[:nt, :nt]
    g = np.random.default_rng(3).standard_normal(x.shape)
    gxr, ger, gsr = oracle.lj_vjp(x, box, 2.5, g, e, s, types=t, n_types=nt)
    with System.lj(x, np.zeros_like(x), box, eps=e, sig=s, types=t, n_types=nt, cutoff=2.5, skin=0.3, dt=0.005,
                   mass=[1.0] * nt, precision="mixed", tpa=1) as h:
        gx, gp = h.backward(g)
    gp = gp.cpu().numpy()
    assert rel_maxnorm(gx.cpu().numpy(), gxr) < 1e-10
    for a in range(nt):
        for b in range(a, nt):
            for got, ref in ((gp[a * nt + b], ger[a, b]), (gp[nt * nt + b * nt + a], gsr[a, b])):
                assert abs(got - ref) <= 1e-10 * np.abs(gsr).max()


def test_a_nan_gradient_reaches_neighbours_only():
    """Lanes without a pair evaluate their own atom: one atom's NaN stays with it and its neighbours."""
    from paper_1009_4330_gb300 import System
    x, box, t = _case(601, 1)
    g = np.ones_like(x)
    g[300, 1] = np.nan
    d = x - x[300]
    near = ((d - box * np.round(d / box)) ** 2).sum(1) < 2.5 ** 2
    with System.lj(x, np.zeros_like(x), box, cutoff=2.5, skin=0.3, dt=0.005, mass=1.0, precision="fp64") as h:
        gx = h.backward(g)[0].cpu().numpy()
    assert np.array_equal(np.isnan(gx).any(1), near)


def test_coincident_atoms_give_nan_forces():
    from paper_1009_4330_gb300 import System
    x, box, t = _case(601, 1)
    x[7] = x[8]
    with System.lj(x, np.zeros_like(x), box, cutoff=2.5, skin=0.3, dt=0.005, mass=1.0, precision="fp64") as h:
        f = h.compute_forces().cpu().numpy()
    assert np.isnan(f[7]).all() and np.isnan(f[8]).all() and np.isfinite(np.delete(f, [7, 8], 0)).all()
