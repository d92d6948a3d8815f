"""Backward passes with a NaN or an infinity in dL/dF: it reaches the atoms whose gradient depends on it
and no others.  The lists reach beyond the cut-off and lanes without a pair go through the arithmetic of
their neighbours in the warp, so pairs just beyond rc, isolated atoms and the parameter gradients are looked
at.  Exact: which values are finite, and that the finite ones do not change by a bit."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

EPS = np.array([[1.0, 1.5], [1.5, 0.5]])
SIG = np.array([[1.0, 0.8], [0.8, 0.88]])


def _near(x, box, i, rc):
    d = x - x[i]
    d -= box * np.round(d / box)
    r = np.sqrt((d ** 2).sum(1))
    return (r < rc) & (np.arange(len(x)) != i), r


def _beyond(x, box, i, rc):
    """Move the atom nearest to the cut-off sphere of atom i to 1 + 2^-12 of its radius."""
    r = _near(x, box, i, rc)[1]
    j = int(np.argmin(np.abs(r - rc)))
    d = x[j] - x[i]
    d -= box * np.round(d / box)
    x[j] = np.mod(x[i] + d * (rc * (1 + 2.0 ** -12) / r[j]), box)
    return j


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("nt", [1, 2])
@pytest.mark.parametrize("n", [601, 12001])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_lj_reaches_neighbours_only(n, nt, precision, bad):
    from paper_1009_4330_gb300 import System
    x, box = synth.fcc_subset(n, 0.8442, 5)
    x = synth.displace(x, box, 0.03, 6)
    t = np.random.default_rng(7).integers(0, nt, n).astype(np.int32)
    far = _beyond(x, box, 300, 2.5)
    near, r = _near(x, box, 300, 2.5)
    assert not near[far] and r[far] < 2.5 * (1 + 2.0 ** -11)
    g = np.random.default_rng(8).standard_normal(x.shape)
    with System.lj(x, np.zeros_like(x), box, eps=EPS[:nt, :nt], sig=SIG[:nt, :nt], types=t, n_types=nt, cutoff=2.5,
                   skin=0.3, dt=0.005, mass=[1.0] * nt, precision=precision, tpa=1) as s:
        ref = s.backward(g)[0].cpu().numpy()
        g[300, 1] = bad
        gx = s.backward(g)[0].cpu().numpy()
    near[300] = True
    assert np.array_equal(~np.isfinite(gx).all(1), near)
    assert np.array_equal(gx[~near], ref[~near])


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_eam_reaches_neighbours_of_neighbours_only(precision, bad):
    from paper_1009_4330_gb300 import System
    rc = synth.EAM_PARAMS[0]
    x, box = synth.fcc_lattice(10, 10, 10, 3.615)
    x = synth.displace(x, box, 0.08, 9)
    _beyond(x, box, 777, rc)
    g = np.random.default_rng(8).standard_normal(x.shape)
    mu = _near(x, box, 777, rc)[0]  # atoms whose lambda takes in g[777]
    mu[777] = True
    hit = mu.copy()
    for i in np.flatnonzero(mu):
        hit |= _near(x, box, i, rc)[0]
    assert hit.sum() < len(x)
    with System.eam(x, np.zeros_like(x), box, eam_params=synth.EAM_PARAMS, skin=0.5, dt=1.0, mass=63.55,
                    ftm2v=synth.FTM2V_METAL, precision=precision, tpa=1) as s:
        ref = s.backward(g)[0].cpu().numpy()
        g[777, 2] = bad
        gx = s.backward(g)[0].cpu().numpy()
    assert np.array_equal(~np.isfinite(gx).all(1), hit)
    assert np.array_equal(gx[~hit], ref[~hit])


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("pot", ["lj", "lj2", "eam"])
def test_an_isolated_atom_changes_nothing(pot, bad):
    """Atoms alone in a large box, among a drop of liquid or metal: their gradients enter no sum.  (They come last in
    the sorted order, 502 atoms after its start: one warp has both.)"""
    from paper_1009_4330_gb300 import System
    if pot == "eam":
        x, b = synth.fcc_lattice(5, 5, 5, 3.615)  # 500 atoms, and two more at a corner
        box = np.full(3, 60.0)
    else:
        x, b = synth.fcc_subset(502, 0.8442, 11)
        box = np.full(3, 30.0)
    x = synth.displace(x, b, 0.03, 12) * 0.98
    if pot == "eam":
        x = np.concatenate([x, [b + [1.5, 0.2, 0.1], b + [0.2, 1.6, 0.0]]])
    lone = np.array([[0.9, 0.9, 0.9], [0.9, 0.6, 0.9], [0.6, 0.9, 0.9], [0.9, 0.9, 0.6], [0.6, 0.6, 0.9]]) * box
    x = np.concatenate([x, lone])
    g = np.random.default_rng(8).standard_normal(x.shape)
    nt = 2 if pot == "lj2" else 1
    t = (np.arange(len(x)) % nt).astype(np.int32)
    if pot == "eam":
        s = System.eam(x, np.zeros_like(x), box, eam_params=synth.EAM_PARAMS, skin=0.5, dt=1.0, mass=63.55,
                       ftm2v=synth.FTM2V_METAL, precision="fp64", tpa=1)
    else:
        s = System.lj(x, np.zeros_like(x), box, eps=EPS[:nt, :nt], sig=SIG[:nt, :nt], types=t, n_types=nt, cutoff=2.5,
                      skin=0.3, dt=0.005, mass=[1.0] * nt, precision="fp64", tpa=1)
    with s:
        ref = [a.cpu().numpy() for a in s.backward(g)]
        g[-5:] = bad
        got = [a.cpu().numpy() for a in s.backward(g)]
    assert not ref[0][-5:].any()
    for a, b in zip(ref, got):
        assert np.array_equal(a, b)
