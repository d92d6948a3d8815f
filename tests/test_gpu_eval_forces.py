"""md_eval_forces: bit for bit the forces of md_set_params, md_set_state and
md_compute_forces in turn, with the same state behind it; a list that has to
grow on the way; the same refusals."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import TOL_MIXED, rel_maxnorm

pytestmark = pytest.mark.gpu


def _case(pot, n=601):
    x, box = synth.fcc_subset(n, 0.8442, 5) if pot == "lj" else synth.fcc_lattice(6, 6, 6, 3.615)
    x = synth.displace(x, box, 0.05, 6)
    v = np.random.default_rng(7).standard_normal(x.shape) * 0.1
    y = synth.displace(x, box, 0.2 if pot == "eam" else 0.03, 8)
    return x, v, box, y


def _make(pot, prec, lst, x, v, box):
    from paper_1009_4330_gb300 import System
    if pot == "eam":
        return System.eam(x, v, box, eam_params=synth.EAM_PARAMS, skin=0.5, dt=1.0, mass=63.55,
                          ftm2v=synth.FTM2V_METAL, precision=prec)
    return System.lj(x, v, box, cutoff=2.5, skin=0.3, dt=0.005, mass=1.0, precision=prec, list=lst)


@pytest.mark.parametrize("new", ["params", "x", "both", "neither"])
@pytest.mark.parametrize("pot,prec,lst", [("lj", "mixed", "full"), ("lj", "fp64", "full"), ("eam", "mixed", "full"),
                                          ("eam", "fp64", "full")])
def test_same_as_the_three_calls(pot, prec, lst, new):
    from paper_1009_4330_gb300 import lj_params
    x, v, box, y = _case(pot)
    p = np.array(synth.EAM_PARAMS) * [1, 1.1, 0.9, 1.05, 1.0] if pot == "eam" else lj_params(1.2, 0.97, 1)
    p = p if new in ("params", "both") else None
    y = y if new in ("x", "both") else None
    with _make(pot, prec, lst, x, v, box) as a, _make(pot, prec, lst, x, v, box) as b:
        if p is not None:
            a.set_params(p)
        if y is not None:
            a.set_state(x=y)
        fa = a.compute_forces()
        fb = b.eval_forces(p, y)
        assert np.array_equal(fa.cpu().numpy(), fb.cpu().numpy())
        for s in (a, b):
            s.step(5)
        for u, w in zip(a.state(), b.state()):
            assert np.array_equal(u.cpu().numpy(), w.cpu().numpy())


def test_list_grows_on_the_way():
    """New positions far denser than the ones the capacity was guessed from."""
    from paper_1009_4330_gb300 import System
    n, box = 2000, np.array([12.6, 12.6, 120.0])
    rng = np.random.default_rng(1)
    x = rng.random((n, 3)) * box
    y, _ = synth.fcc_subset(n, 1.0, 21)
    y = synth.displace(y, np.full(3, 12.6), 0.03, 22)
    with System.lj(x, np.zeros_like(x), box, cutoff=4.0, skin=0.3, dt=0.005, mass=1.0, precision="mixed") as s:
        cap = s.info()["maxneigh"]
        f = s.eval_forces(x=y).cpu().numpy()
        assert s.info()["maxneigh"] > cap
    assert rel_maxnorm(f, oracle.lj(y, box, 4.0)[0]) < TOL_MIXED


def test_refusals():
    from paper_1009_4330_gb300 import MDError
    x, v, box, y = _case("lj")
    with _make("lj", "mixed", "full", x, v, box) as s:
        with pytest.raises(MDError):
            y[3, 1] = np.nan
            s.eval_forces(x=y)
    with _make("eam", "mixed", "full", *_case("eam")[:3]) as s:
        f = s.compute_forces().cpu().numpy()
        with pytest.raises(MDError):
            s.eval_forces(params=np.array([4.0, 1, 0.5, -0.2, 0.02]))
        assert np.array_equal(s.compute_forces().cpu().numpy(), f)
