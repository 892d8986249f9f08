"""Soft steric forces at the ends of their range: a pair whose exponential is
about to underflow still acts on each other, and one just beyond does not.
The two are the only near pair of their groups, so that nothing else keeps a
group from being skipped."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2510_02135_gb300 import lm  # noqa: E402

D, B = 2.0, 0.125   # exact, as r - D is


def forces(x, fp64, first, second):
    """Forces of two particles at r = D + x B among 68 that are far apart."""
    dt = np.float64 if fp64 else np.float32
    pos = np.zeros((68, 3), dt)
    pos[:, 1] = 2.0 ** 20 * np.arange(1, 69)
    pos[first] = 0.0
    pos[second] = [D + x * B, 0.0, 0.0]
    s = lm.lm_create(1.0, 1.0, False, lm.LM_FP64 if fp64 else lm.LM_FP32C)
    t = torch.from_numpy(pos).cuda()
    lm.lm_set_positions(s, t)
    return lm.lm_soft_repulsion(s, 2.0 ** 60 * B, B, D, 1.0, like=t).double().cpu().numpy()


@pytest.mark.parametrize("first,second", [(0, 64), (1, 67), (40, 0)])
@pytest.mark.parametrize("x,fp64", [(1, False), (80, False), (100, False), (1, True), (700, True), (740, True)])
def test_last_pairs_act(x, fp64, first, second):
    F = forces(x, fp64, first, second)
    want = np.exp(np.longdouble(-x)) * np.longdouble(2.0) ** 60
    assert F[first, 0] < 0.0 < F[second, 0] and F[first, 0] == -F[second, 0]
    # roundings of r (four) enter the exponent times r / B; the exponential of 100 (FP32) and 740 (FP64) is subnormal
    eps = 2.0 ** -53 if fp64 else 2.0 ** -24
    tol = 2.0 * eps * (4.0 * (D + x * B) / B + 16.0)
    if x in (100, 740):
        tol = 0.5
    assert abs(F[second, 0] - want) <= tol * want, float(F[second, 0] / want - 1.0)
    F[[first, second], 0] = 0.0
    assert not F.any()


@pytest.mark.parametrize("x,fp64", [(104, False), (109, False), (111, False), (746, True), (759, True), (765, True)])
def test_pairs_beyond_add_nothing(x, fp64):
    assert not forces(x, fp64, 0, 64).any()
