"""LJForces takes one value per unordered type pair in a vector; other shapes are refused alike on the host and on the GPU."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("device", ["cpu", "cuda"])
@pytest.mark.parametrize("nt,shape", [(1, ()), (2, (1, 3)), (2, (2,))])
def test_other_shapes_are_refused(nt, shape, device):
    import torch
    from paper_1009_4330_gb300 import LJForces, System
    x, box = synth.fcc_subset(257, 0.8442, 5)
    t = (np.arange(257) % nt).astype(np.int32)
    one = np.ones((nt, nt))
    with System.lj(x, np.zeros_like(x), box, eps=one, sig=one, types=t, n_types=nt, cutoff=2.5, skin=0.3, dt=0.005,
                   mass=[1.0] * nt) as s:
        p = torch.ones(shape, dtype=torch.float64, device=device)
        with pytest.raises((IndexError, TypeError, ValueError)):
            LJForces.apply(s, None, p, p)
