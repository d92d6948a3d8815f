"""The EAM density pass with its x and y components packed two to an instruction (systems of many threads)
against the scalar one (few): periodic copies of a block have the block's forces.  The bins, and so the FP32
records' rounding, differ between the two systems, and each is held to 1e-5 (relative max-norm) of FP64."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vec", [1, 2, 4])
def test_packed_and_scalar_density_passes_agree(vec):
    from paper_1009_4330_gb300 import System
    a, cells, rep = 3.615, 9, 4
    basis = np.array([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]])
    grid = lambda m: np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 1, 3)
    x = ((grid(cells) + basis).reshape(-1, 3) + 0.25) * a
    x += np.random.default_rng(5).normal(0, 0.08, x.shape)
    big = (x[None] + grid(rep) * cells * a).reshape(-1, 3)
    e = synth.config2(cells=4)

    def forces(x, box):
        with System.eam(x, np.zeros_like(x), np.full(3, box), eam_params=e["eam"], skin=e["skin"], dt=e["dt"],
                        mass=e["mass"], ftm2v=e["ftm2v"], precision="mixed", tpa=1) as s:
            s.set_kernel(1, "full", 128, vec)
            return s.compute_forces().cpu().numpy()

    one, many = forces(x, cells * a), forces(big, rep * cells * a)
    assert len(x) < 152 * 900 < len(big)
    assert np.abs(many.reshape(rep ** 3, -1, 3) - one).max() <= 2e-5 * np.abs(one).max()
