"""Arrays that are too small for the system are refused before their pointers reach the library, which would read or
write past their ends.  Runs without a GPU: the device copy is left out, and the library is a recorder that
must not be called."""
import numpy as np
import pytest
import torch

from paper_1009_4330_gb300 import MDError, system

N = 7


class Recorder:
    def __getattr__(self, name):
        raise AssertionError(f"{name} called with a bad argument")


@pytest.fixture
def sys_(monkeypatch):
    def dev(a, dtype, shape=None):
        t = torch.as_tensor(a, dtype=dtype)
        return (t.reshape(shape) if shape is not None else t).contiguous()

    monkeypatch.setattr(system, "_dev", dev)
    empty = torch.empty
    monkeypatch.setattr(torch, "empty", lambda *a, device=None, **k: empty(*a, **k))

    def make(potential="lj", n_types=1):
        s = system.System.__new__(system.System)
        s._h, s._lib, s._version = None, Recorder(), 0
        s.n, s.n_rep, s.n_types, s.potential, s.precision = N, 1, n_types, potential, "mixed"
        return s

    return make


SHORT = np.zeros((N - 1, 3))


@pytest.mark.parametrize("x", [SHORT, np.zeros((N + 1, 3)), np.zeros(3 * N - 3)])
def test_eval_forces_positions(sys_, x):
    s = sys_()
    with pytest.raises(MDError, match="INVALID"):
        s.eval_forces(x=x)
    assert s.version == 0


@pytest.mark.parametrize("potential,n_types,size", [("lj", 1, 1), ("lj", 1, 3), ("lj", 2, 7), ("lj", 2, 2), ("eam", 1, 4),
                                                    ("eam", 1, 6), ("lj", 1, 0)])
def test_eval_forces_parameters(sys_, potential, n_types, size):
    with pytest.raises(MDError, match="INVALID"):
        sys_(potential, n_types).eval_forces(params=np.ones(size))


@pytest.mark.parametrize("out", [torch.zeros(N, 3), torch.zeros(N, 3, dtype=torch.float64),  # on the host
                                 torch.zeros(3, N, dtype=torch.float64).T, torch.zeros(N - 1, 3, dtype=torch.float64)])
def test_outputs(sys_, out):
    s = sys_()
    for call in (s.eval_forces, s.compute_forces):
        with pytest.raises(MDError, match="INVALID"):
            call(out=out)


def test_the_other_entry_points(sys_):
    s = sys_("lj", 2)
    for call in (lambda: s.set_state(x=SHORT), lambda: s.set_state(v=SHORT), lambda: s.backward(SHORT),
                 lambda: s.reset(np.zeros((N, 3)), SHORT), lambda: s.set_params(np.ones(7))):
        with pytest.raises(MDError, match="INVALID"):
            call()
    assert s.version == 0
