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
