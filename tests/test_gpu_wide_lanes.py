"""The lanes that stand in for a thread of the list layout in a small mixed system (k_lj_wide and its EAM
counterparts), at the numbers of lanes that its size and the rounds of its longest list allow: bit for bit the
forces, energies and virial of the same system in a batch large enough to be walked with one lane."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _results(s, n, tpa, vec):
    s.set_kernel(tpa, "full", 128, vec)
    return s.compute_forces()[:n].cpu().numpy(), s.energy_virial()[0].cpu().numpy()


def _same_bits(kw, r, copies, tpa, vec):
    from paper_1009_4330_gb300 import System
    n = len(r["x"])
    with System(r["x"], r["v"], r["types"], r["box"], **kw) as s:
        f, ev = _results(s, n, tpa, vec)
    with System.batch([r] * copies, **kw) as b:
        fb, evb = _results(b, n, tpa, vec)
    assert np.array_equal(f, fb) and np.array_equal(ev, evb)


def _lj(n, rho, rc, nt):
    from paper_1009_4330_gb300 import lj_params
    x, box = synth.fcc_subset(n, rho, 31)
    x = synth.displace(x, box, 0.04 if rho > 0.5 else 0.9, 32)
    r = {"x": x, "v": np.ones_like(x), "box": box, "types": (np.arange(n) % nt).astype(np.int32)}
    e, g = (synth.pair_matrix(synth.KA_EPS), synth.pair_matrix(synth.KA_SIG)) if nt == 2 else (1.0, 1.0)
    return r, dict(potential="lj", params=lj_params(e, g, nt), cutoff=rc, skin=0.3, dt=0.005, mass=[1.0] * nt, n_types=nt,
                   precision="mixed", tpa=1)


@pytest.mark.parametrize("tpa,vec", [(1, 4), (1, 1), (2, 4), (4, 2), (8, 1)])
@pytest.mark.parametrize("rho,rc", [(0.8442, 1.1225), (0.15, 2.5), (0.02, 2.5)])
def test_short_lists(rho, rc, tpa, vec):
    """Lists of no entry to a few dozen: fewer rounds than the size alone allows lanes."""
    r, kw = _lj(999, rho, rc, 1)
    _same_bits(kw, r, 160, tpa, vec)


def _atoms(per_sm):
    """Sizes follow the GPU's, as the rule for the lanes does (threads per SM)."""
    import torch
    return per_sm * torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("nt", [1, 2])
@pytest.mark.parametrize("tpa,vec,per_sm,copies", [(1, 4, 270, 2),   # two lanes
                                                   (1, 1, 160, 3),   # four
                                                   (1, 4, 80, 6),    # eight
                                                   (2, 2, 135, 2),   # two
                                                   (2, 4, 90, 3),    # four
                                                   (4, 4, 66, 2),    # two
                                                   (4, 1, 45, 3),    # four
                                                   (8, 4, 35, 2),    # two
                                                   (16, 1, 16, 3)])  # two
def test_lj_lanes(tpa, vec, per_sm, copies, nt):
    r, kw = _lj(_atoms(per_sm) + 3, 0.8442, 2.5, nt)
    _same_bits(kw, r, copies, tpa, vec)


def _eam(n):
    cells = int(round((n / 4) ** (1 / 3)))
    x, box = synth.fcc_lattice(cells, cells, cells, 3.615)
    x = synth.displace(x, box, 0.08, 41)
    return ({"x": x, "v": np.ones_like(x), "box": box, "types": np.zeros(len(x), np.int32)},
            dict(potential="eam", params=np.array(synth.EAM_PARAMS), cutoff=float(synth.EAM_PARAMS[0]), skin=0.5, dt=1.0,
                 mass=63.55, ftm2v=synth.FTM2V_METAL, precision="mixed", tpa=1))


@pytest.mark.parametrize("tpa,vec,per_sm,copies", [(1, 4, 270, 2), (1, 2, 160, 3), (2, 4, 135, 2), (4, 4, 66, 2), (8, 1, 35, 2)])
def test_eam_lanes(tpa, vec, per_sm, copies):
    r, kw = _eam(_atoms(per_sm))
    _same_bits(kw, r, copies, tpa, vec)


@pytest.mark.parametrize("vec", [1, 2, 4])
def test_eam_scalar_and_packed_density_pass(vec):
    """Sizes too large for several lanes take the scalar density pass up to 900 threads per SM, larger ones the packed one."""
    r, kw = _eam(_atoms(600))
    assert _atoms(330) < len(r["x"]) < _atoms(880)
    _same_bits(kw, r, 2, 1, vec)


def test_lists_that_get_longer():
    """A system made as a gas and then filled: the lanes follow its lists, in the passes and in the step's graph."""
    from paper_1009_4330_gb300 import System
    n = 1500
    y, _ = synth.fcc_subset(n, 0.8442, 31)
    y = synth.displace(y, np.full(3, (n / 0.8442) ** (1 / 3)), 0.04, 32)
    box = np.full(3, 60.0)
    x = np.random.default_rng(1).random((n, 3)) * box
    v = synth.maxwell_boltzmann(n, 1.44, 1.0, 33)
    kw = dict(_lj(64, 0.8442, 2.5, 1)[1], skin=0.3)
    with System(x, v, None, box, **kw) as a, System(y, v, None, box, **kw) as b:
        a.step(3)
        a.set_state(x=y, v=v)
        for s in (a, b):
            s.set_kernel(16, "full", 128, 1)  # (more turns than one cluster takes: separate launches)
        assert np.array_equal(a.compute_forces().cpu().numpy(), b.compute_forces().cpu().numpy())
        for s in (a, b):
            s.step(40)
        for u, w in zip(a.state(), b.state()):
            assert np.array_equal(u.cpu().numpy(), w.cpu().numpy())
