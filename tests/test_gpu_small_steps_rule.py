"""Which small mixed systems run their steps in one launch (k_steps): a system whose list layout has many threads per atom
must not be slowed down by it, and on both sides of the rule's lines a step is the separate launches' bit for bit."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _lj(n, tpa, vec):
    from paper_1009_4330_gb300 import System
    x, box = synth.fcc_subset(n, 0.8442, 51)
    x = synth.displace(x, box, 0.03, 52)
    s = System.lj(x, synth.maxwell_boltzmann(n, 1.44, 1.0, 53), box, cutoff=2.5, skin=0.3, dt=0.004, mass=1.0,
                  precision="mixed", tpa=1)
    s.set_kernel(tpa, "full", 128, vec)
    return s


def _eam(cells, tpa, vec):
    from paper_1009_4330_gb300 import System
    x, box = synth.fcc_lattice(*cells, 3.615)
    x = synth.displace(x, box, 0.1, 61)
    v = synth.maxwell_boltzmann(x.shape[0], 600.0, 63.55, 62, kb=synth.KB_METAL, ftm2v=synth.FTM2V_METAL)
    s = System.eam(x, v, box, eam_params=synth.EAM_PARAMS, skin=0.5, dt=1.0, mass=63.55, ftm2v=synth.FTM2V_METAL,
                   precision="mixed", tpa=1)
    s.set_kernel(tpa, "full", 128, vec)
    return s


def _ms(s, steps=200):
    import torch
    best = 1e9
    for _ in range(4):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        s.step(steps)
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]))
    return best


@pytest.mark.parametrize("make,size", [(_lj, 4096), (_eam, (10, 10, 10))])
def test_sixteen_threads_per_atom_are_not_far_slower_than_one(make, size):
    """Measured 1.2 times; 3 to 4 times when one cluster took four and eight turns through such a system."""
    with make(size, 1, 4) as a, make(size, 16, 1) as b:
        assert _ms(b) < 2.0 * _ms(a)


@pytest.mark.parametrize("make,size,tpa,vec", [(_lj, 1024, 8, 4), (_lj, 1025, 8, 4), (_lj, 4096, 2, 4), (_lj, 500, 16, 1),
                                               (_lj, 513, 16, 1), (_lj, 2048, 4, 2), (_lj, 2049, 4, 2),
                                               (_eam, (8, 8, 8), 1, 4), (_eam, (8, 8, 8), 4, 4), (_eam, (8, 8, 9), 1, 4),
                                               (_eam, (8, 8, 8), 8, 4)])
def test_same_bits_on_both_sides_of_the_lines(make, size, tpa, vec):
    with make(size, tpa, vec) as a, make(size, tpa, vec) as b:
        for steps in (1, 60):
            a.step(steps)
            b.step(steps, eager=True)
        assert a.info()["rebuilds"] == b.info()["rebuilds"]
        for u, w in zip(a.state(), b.state()):
            assert np.array_equal(u.cpu().numpy(), w.cpu().numpy())
