"""Small mixed systems run whole steps in one launch (k_steps): the same
trajectory, step and rebuild counts bit for bit as the step's kernels launched
one by one (md_step_eager), for sizes on both sides of the limit, several types,
list layouts and call lengths; a non-finite state is reported."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _system(n, nt, tpa, vec, skin=0.3):
    from paper_1009_4330_gb300 import System
    x, box = synth.fcc_subset(n, 0.8442, 51)
    x = synth.displace(x, box, 0.03, 52)
    v = synth.maxwell_boltzmann(n, 1.44, 1.0, 53)
    t = np.random.default_rng(54).integers(0, nt, n).astype(np.int32)
    e = synth.pair_matrix(synth.KA_EPS) if nt == 2 else 1.0
    g = synth.pair_matrix(synth.KA_SIG) if nt == 2 else 1.0
    s = System.lj(x, v, box, eps=e, sig=g, types=t, n_types=nt, cutoff=2.5, skin=skin, dt=0.004, mass=[1.0, 1.5][:nt],
                  precision="mixed", tpa=1)
    s.set_kernel(tpa, "full", 128, vec)
    return s


@pytest.mark.parametrize("n,nt,tpa,vec", [(180, 1, 1, 4), (500, 1, 1, 4), (777, 2, 1, 4), (777, 1, 4, 1), (1999, 1, 2, 2),
                                          (192, 1, 16, 1), (4096, 1, 1, 4), (4097, 2, 1, 4)])
def test_same_bits_as_the_separate_launches(n, nt, tpa, vec):
    with _system(n, nt, tpa, vec) as a, _system(n, nt, tpa, vec) as b:
        for steps in (1, 2, 37, 1, 60):
            a.step(steps)
            b.step(steps, eager=True)
            ia, ib = a.info(), b.info()
            assert ia["steps"] == ib["steps"] and ia["rebuilds"] == ib["rebuilds"]
            for u, w in zip(a.state(), b.state()):
                assert np.array_equal(u.cpu().numpy(), w.cpu().numpy())
        assert a.info()["rebuilds"] > 5


@pytest.mark.parametrize("cells,tpa,vec", [(4, 1, 4), (6, 2, 1), (10, 1, 2)])
def test_eam_same_bits(cells, tpa, vec):
    from paper_1009_4330_gb300 import System
    x, box = synth.fcc_lattice(cells, cells, cells, 3.615)
    x = synth.displace(x, box, 0.1, 61)
    v = synth.maxwell_boltzmann(x.shape[0], 2000.0, 63.55, 62, kb=synth.KB_METAL, ftm2v=synth.FTM2V_METAL)
    got = []
    for eager in (False, True):
        with System.eam(x, v, box, eam_params=synth.EAM_PARAMS, skin=0.5, dt=2.0, mass=63.55, ftm2v=synth.FTM2V_METAL,
                        precision="mixed", tpa=1) as s:
            s.set_kernel(tpa, "full", 128, vec)
            for steps in (1, 40, 3):
                s.step(steps, eager=eager)
            got.append([u.cpu().numpy() for u in s.state()] + [s.info()["rebuilds"]])
    assert got[0][3] == got[1][3] >= 2
    assert all(np.array_equal(a, b) for a, b in zip(got[0][:3], got[1][:3]))


def test_a_rebuild_in_every_step():
    with _system(500, 1, 1, 4, skin=0.004) as a, _system(500, 1, 1, 4, skin=0.004) as b:
        a.step(12)
        b.step(12, eager=True)
        assert a.info()["rebuilds"] == b.info()["rebuilds"] == 13  # one at creation
        assert np.array_equal(a.state()[0].cpu().numpy(), b.state()[0].cpu().numpy())


def test_non_finite_state_is_reported():
    from paper_1009_4330_gb300 import MDError
    with _system(500, 1, 1, 4) as s:
        v = s.state()[1].cpu().numpy()
        v[17, 2] = np.inf
        s.set_state(v=v)
        with pytest.raises(MDError, match="NONFINITE"):
            s.step(5)
