"""The one-launch Lanczos iteration at the sizes where its elements per CTA
change (64, 128, 256, 512, then the separate kernels) and at their remainders."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2510_02135_gb300 import inputs, lm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2510_02135_gb300 import _build

    _build.build()


# 152 CTAs x 64, 128, 256 and 512 elements: n = 9728, 19456, 38912, 77824
@pytest.mark.parametrize("n", [1, 2, 21, 22, 1000, 3242, 3243, 6486, 12971, 25941, 25942])
@pytest.mark.parametrize("twice", [0, 1])
def test_root_of_the_root(n, twice):
    """M^{1/2} (M^{1/2} W) = M W, with one and with two Gram-Schmidt passes; a
    second call with another n follows on the same solver."""
    tol = 1e-4
    s_ = inputs.cube_suspension(11, n, 0.1)
    s = lm.lm_create(1.0, 1.0, False, lm.LM_FP32C)
    lm.lm_set_reorthogonalization(s, twice)
    for pos in (s_.pos, s_.pos[: max(1, n // 2)]):
        m = len(pos)
        lm.lm_set_positions(s, torch.from_numpy(np.ascontiguousarray(pos)).cuda())
        W = torch.from_numpy(np.random.default_rng(n).standard_normal(3 * m)).cuda()
        y = lm.lm_sqrt_mdot(s, W, tol=tol, max_iter=150)[0]
        z = lm.lm_sqrt_mdot(s, y.double().reshape(-1), tol=tol, max_iter=150)[0]
        u, _ = lm.lm_mdot(s, W.float().reshape(m, 3).contiguous(), None)
        # each root is within 20 tol of the exact one; M^{1/2} at most doubles the first one's relative error here
        assert float((z - u).norm() / u.norm()) <= 60.0 * tol
        assert lm.lm_get_lanczos_stats(s)["converged"] == 1
