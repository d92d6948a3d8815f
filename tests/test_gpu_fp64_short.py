"""FP64 forces of a gas, whose batches of short lists are walked one lane to an atom with one queue for the warp
(short_walk): clumps of one to ten atoms, so that lists of eight and nine entries and batches about the limit of
entries occur, against the oracle; and, bit for bit, the forces of atoms whose warp takes the one walk or the other
depending on which others are with them.

Tolerance: TOL_FP64 (1e-12 relative max-norm), hundreds of roundings of a sum of at most nine terms."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import TOL_FP64

pytestmark = pytest.mark.gpu

EPS = np.array([[1.0, 1.5], [1.5, 0.5]])
SIG = np.array([[1.0, 0.8], [0.8, 0.88]])


def _clump(m, rng, scale):
    """m atoms within 2 * scale of one another and not closer than 0.9 * scale."""
    g = np.array([[i, j, k] for i in (0, 1) for j in (0, 1) for k in (0, 1, 2)], float)
    return (g[rng.permutation(12)[:m]] * 0.97 + rng.uniform(-0.03, 0.03, (m, 3))) * scale


def _clumps(sizes, scale, cells):
    """One clump per site of a cubic grid, too far apart to see one another, each drawn for its site and size
    alone; the box and the site of each atom."""
    sites = np.stack(np.unravel_index(np.arange(cells ** 3), (cells,) * 3), 1) * (6.0 * scale) + 0.5
    x = [sites[k] + _clump(m, np.random.default_rng((k, m)), scale) for k, m in enumerate(sizes) if m]
    return np.concatenate(x), np.full(3, cells * 6.0 * scale), np.repeat(np.arange(len(sizes)), sizes)


def _system(pot, x, box, nt=1, lst="full", tpa=1):
    from paper_1009_4330_gb300 import System
    if pot == "eam":
        return System.eam(x, np.zeros_like(x), box, eam_params=synth.EAM_PARAMS, skin=0.5, dt=1.0, mass=63.55,
                          ftm2v=synth.FTM2V_METAL, precision="fp64", tpa=tpa)
    return System.lj(x, np.zeros_like(x), box, eps=EPS[:nt, :nt], sig=SIG[:nt, :nt], types=(np.arange(len(x)) % nt).astype(np.int32),
                     n_types=nt, cutoff=2.5, skin=0.3, dt=0.005, mass=[1.0] * nt, precision="fp64", list=lst, tpa=tpa)


@pytest.mark.parametrize("most", [1, 3, 9, 10])
@pytest.mark.parametrize("pot,nt,lst,tpa", [("lj", 1, "full", 1), ("lj", 2, "full", 4), ("lj", 1, "half", 1), ("lj", 2, "half", 2),
                                            ("eam", 1, "full", 1), ("eam", 1, "full", 16)])
def test_clumps_against_the_oracle(pot, nt, lst, tpa, most):
    rng = np.random.default_rng(most)
    x, box, _ = _clumps(rng.integers(0, most + 1, 343), 2.2 if pot == "eam" else 1.0, 7)
    t = (np.arange(len(x)) % nt).astype(np.int32)
    if pot == "eam":
        fr, er = oracle.eam(x, box, synth.EAM_PARAMS)[:2]
    else:
        fr, er = oracle.lj(x, box, 2.5, eps=EPS[:nt, :nt], sig=SIG[:nt, :nt], types=t, n_types=nt)[:2]
    with _system(pot, x, box, nt, lst, tpa) as s:
        f = s.compute_forces().cpu().numpy()
        ev = s.energy_virial().cpu().numpy()[0]
        again = s.state()[2].cpu().numpy()
    assert np.abs(f - fr).max() <= TOL_FP64 * np.abs(fr).max() and np.abs(again - fr).max() <= TOL_FP64 * np.abs(fr).max()
    assert abs(ev[0] - er) <= 1e-11 * max(1.0, abs(er))


@pytest.mark.parametrize("pot,nt", [("lj", 1), ("lj", 2), ("eam", 1)])
def test_same_bits_as_the_groups(pot, nt):
    """The clumps of up to four atoms with and without clumps of eleven between them: in the latter case the long lists send
    most batches to the groups of eight lanes.  (Even atom counts keep the types of the small clumps' atoms.)"""
    small = 2 * np.random.default_rng(2).integers(0, 3, 343)
    every = np.arange(343) % 5 == 0
    got = []
    for big in (0, 10):
        x, box, site = _clumps(np.where(every, big, small), 2.2 if pot == "eam" else 1.0, 7)
        with _system(pot, x, box, nt) as s:
            got.append(s.compute_forces().cpu().numpy()[~every[site]])
    assert got[0].shape == got[1].shape and got[0].any() and np.array_equal(got[0], got[1])
