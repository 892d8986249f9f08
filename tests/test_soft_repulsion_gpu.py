"""Soft steric forces where whole groups of pairs are skipped because their
exponential is zero: block and tile edges, ranges from below the spacing to
beyond the box, against the FP64 oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2510_02135_gb300 import lm  # noqa: E402


@pytest.mark.parametrize("n", [1, 2, 63, 65, 257, 1023])
@pytest.mark.parametrize("b,d_pair", [(1e-3, 2.0), (0.1, 2.0), (0.1, -3.0), (5.0, 2.0), (1e3, 0.0)])
@pytest.mark.parametrize("fp64", [False, True])
def test_forces_match_oracle(orc, n, b, d_pair, fp64):
    dt = np.float64 if fp64 else np.float32
    rng = np.random.default_rng(n)
    pos = (rng.uniform(0.0, 3.0 * n ** (1.0 / 3.0), (n, 3)) * 2.0).astype(dt)
    if n > 60:
        pos[n - 1] = pos[3]                      # a coincident pair gives no force
    s = lm.lm_create(1.0, 1.0, False, lm.LM_FP64 if fp64 else lm.LM_FP32C)
    x = torch.from_numpy(pos).cuda()
    lm.lm_set_positions(s, x)
    F = lm.lm_soft_repulsion(s, 4.0, b, d_pair, 1.0, like=x).double().cpu().numpy()
    ref = orc.soft_repulsion(pos, 4.0, b, d_pair, 1.0, wall=False)
    # rounding of r in the exponent, (d - r) / b of up to some 100 where it still counts, and of n terms of 4 / b
    eps = 2.0 ** -52 if fp64 else 2.0 ** -23
    scale = max(np.abs(ref).max(), 4.0 / b if n > 1 and np.abs(ref).max() > 0 else 0.0)
    side = 6.0 * n ** (1.0 / 3.0)
    assert np.abs(F - ref).max() <= eps * scale * (16.0 + 4.0 * side / b + n)
