"""lm_get_product_form names the kernel that the products run."""
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


def solver(n, angular, fp64, wall):
    s = lm.lm_create(1.0, 1.0, angular, lm.LM_FP64 if fp64 else lm.LM_FP32C,
                     periodicity=("open", "open", "single_wall" if wall else "open"))
    pos = inputs.cube_suspension(3, n, 0.1, 1.0, angular=False, fp32=not fp64).pos
    lm.lm_set_positions(s, torch.from_numpy(pos).cuda())
    return s


@pytest.mark.parametrize("n,angular,fp64,wall,symmetric,flops", [
    (500, False, False, False, True, 25.5), (500, True, False, False, True, 72.0),
    (99999, True, False, False, True, 72.0), (100000, True, False, False, False, 86.0),
    (500, False, False, True, True, 85.0), (500, True, False, True, True, 222.0),
    (500, True, True, False, True, 72.0), (500, False, True, True, False, 131.0), (500, True, True, True, False, 299.0)])
def test_form_of_the_default(n, angular, fp64, wall, symmetric, flops):
    assert lm.lm_get_product_form(solver(n, angular, fp64, wall)) == {"symmetric": symmetric, "flops_per_pair": flops}


def test_form_follows_a_pinned_configuration():
    s = solver(500, False, False, False)
    lm.lm_set_pair_config(s, 128, 2, 0, 1)
    assert lm.lm_get_product_form(s) == {"symmetric": False, "flops_per_pair": 35.0}
    F = torch.from_numpy(np.ones((500, 3), np.float32)).cuda()
    lm.lm_profile_enable(s)
    lm.lm_mdot(s, F, None)
    assert lm.lm_profile_read(s)["pair_flops"] == 35.0 * 500 ** 2
