"""Small systems walk their lists with several lanes per thread of the list
layout (k_lj_wide and its EAM counterparts): the same sums bit for bit as one
lane takes, held against the same system as one replica of a batch large
enough to be walked with one lane, at every lane count, list layout and
potential, with energies and virial."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import TOL_MIXED, rel_maxnorm

pytestmark = pytest.mark.gpu

KA_E, KA_S = synth.pair_matrix(synth.KA_EPS), synth.pair_matrix(synth.KA_SIG)


def _lj(n, nt):
    x, box = synth.fcc_subset(n, 0.8442, 31)
    x = synth.displace(x, box, 0.04, 32)
    return {"x": x, "v": synth.maxwell_boltzmann(n, 1.44, 1.0, 33), "box": box,
            "types": np.random.default_rng(34).integers(0, nt, n).astype(np.int32)}


def _results(s, n, tpa, vec):
    s.set_kernel(tpa, "full", 128, vec)
    f = s.compute_forces()[:n].cpu().numpy()
    ev = s.energy_virial()[0].cpu().numpy()
    return f, ev


@pytest.mark.parametrize("nt", [1, 2])
@pytest.mark.parametrize("tpa,vec", [(1, 4), (1, 1), (2, 2), (4, 4), (16, 1), (32, 4)])
@pytest.mark.parametrize("n,copies", [(777, 250), (6003, 30), (15001, 12)])
def test_lj_same_bits_as_one_lane(n, copies, tpa, vec, nt):
    from paper_1009_4330_gb300 import System, lj_params
    r = _lj(n, nt)
    e, g = (KA_E, KA_S) if nt == 2 else (1.0, 1.0)
    kw = dict(params=lj_params(e, g, nt), cutoff=2.5, skin=0.3, dt=0.005, mass=[1.0] * nt, n_types=nt,
              precision="mixed", tpa=1)
    with System(r["x"], r["v"], r["types"], r["box"], potential="lj", **kw) as s:
        f, ev = _results(s, n, tpa, vec)
    with System.batch([r] * copies, potential="lj", **kw) as b:
        fb, evb = _results(b, n, tpa, vec)
    assert np.array_equal(f, fb) and np.array_equal(ev, evb)
    fr = oracle.lj(r["x"], r["box"], 2.5, eps=np.broadcast_to(e, (nt, nt)), sig=np.broadcast_to(g, (nt, nt)),
                   types=r["types"], n_types=nt)[0]
    assert rel_maxnorm(f, fr) < TOL_MIXED


@pytest.mark.parametrize("tpa,vec", [(1, 4), (2, 1), (8, 2)])
def test_eam_same_bits_as_one_lane(tpa, vec):
    from paper_1009_4330_gb300 import System
    x, box = synth.fcc_lattice(6, 6, 6, 3.615)
    x = synth.displace(x, box, 0.08, 41)
    n = x.shape[0]
    P = np.array(synth.EAM_PARAMS)
    r = {"x": x, "v": np.zeros_like(x), "box": box}
    kw = dict(cutoff=float(P[0]), skin=0.5, dt=1.0, mass=63.55, ftm2v=synth.FTM2V_METAL, precision="mixed", tpa=1)
    with System.eam(x, r["v"], box, eam_params=P, **kw) as s:
        f, ev = _results(s, n, tpa, vec)
    with System.batch([r] * 220, potential="eam", params=P, **kw) as b:
        fb, evb = _results(b, n, tpa, vec)
    assert np.array_equal(f, fb) and np.array_equal(ev, evb)
