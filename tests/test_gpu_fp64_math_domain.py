"""The library's FP64 reciprocal and reciprocal square root up to the ends of their stated domains: FLT_MIN to 2^126 and
to FLT_MAX.  The same bounds as in the middle of the range (test_gpu_fp64_math): one ulp from IEEE
division, three from CUDA's rsqrt; NaN below FLT_MIN."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _x(hi):
    rng = np.random.default_rng(7)
    lo = 2.0 ** -126
    ends = np.array([lo, np.nextafter(lo, 1), 1.5 * lo, hi, np.nextafter(hi, 0), 0.75 * hi])
    return np.concatenate([np.exp2(rng.uniform(-126, -100, 50000)), np.exp2(rng.uniform(100, np.log2(hi), 50000)), ends])


@pytest.mark.parametrize("op,hi,ulps", [("rcp", 2.0 ** 126, 1.0), ("rsqrt", float(np.finfo(np.float32).max) * 0.999999, 3.0)])
def test_ends_of_the_domain(op, hi, ulps):
    import torch
    from paper_1009_4330_gb300 import fp64_math
    x = torch.tensor(_x(hi), dtype=torch.float64, device="cuda")
    ref = (1.0 / x if op == "rcp" else torch.rsqrt(x)).cpu().numpy()
    y = fp64_math(op, x).cpu().numpy()
    assert (np.abs(y - ref) / np.spacing(np.abs(ref))).max() <= ulps
    below = torch.tensor([0.0, 1e-300, 2.0 ** -127], dtype=torch.float64, device="cuda")
    assert np.isnan(fp64_math(op, below).cpu().numpy()).all()
