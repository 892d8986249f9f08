"""One FP64 pair at a time against extended precision: the far field's
reciprocal square root over the range of distances, at the ends of binades and
at arguments that differ in their last bits only."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2510_02135_gb300 import lm  # noqa: E402


def distances():
    rng = np.random.default_rng(9)
    d = [2.0, 1e6, 9e14]
    d += [2.0 + k * 2.0 ** -51 for k in (1, 2, 3, 5, 1000, 2 ** 20, 2 ** 31, 2 ** 32, 2 ** 33)]
    d += [2.0 ** e * (1.0 + s * 2.0 ** -52) for e in (2, 3, 7, 20, 33) for s in (-1, 0, 1)]
    d += [2.0 ** (e + 0.5) for e in range(1, 12)]
    d += list(2.0 * 10.0 ** rng.uniform(0.0, 14.0, 120))
    return np.array(d)


def test_far_pair_is_within_a_few_roundings():
    """u_0 of a force on particle 1 alone, along and across the separation.

    Roundings of 2^-53: three of the separation's square (the separation itself
    is exact), half of that and two for the root, three times as much and two
    for its cube, and less than eight for the sums and the final scaling: below
    32 for the terms, which do not cancel by more than half."""
    x_ = np.longdouble
    s = lm.lm_create(1.0, 1.0, False, lm.LM_FP64)
    F = torch.zeros((2, 3), dtype=torch.float64, device="cuda")
    F[1, 0], F[1, 1] = 1.0, 1.0
    for d in distances():
        lm.lm_set_positions(s, torch.tensor([[0.0, 0.0, 0.0], [d, 0.0, 0.0]], dtype=torch.float64, device="cuda"))
        u = lm.lm_mdot(s, F, None)[0].cpu().numpy()[0]
        r = x_(d)
        c8 = x_(1) / (x_(8) * x_("3.14159265358979323846264338327950288"))
        A = 1 / r + x_(2) / 3 / r ** 3
        B = (1 / r ** 3 - 2 / r ** 5) * r * r
        for got, want in ((u[0], c8 * (A + B)), (u[1], c8 * A)):
            assert abs(x_(got) - want) <= 32 * 2.0 ** -53 * abs(want), (d, float((got - want) / want))
