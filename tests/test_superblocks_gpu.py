"""The symmetric kernels where i-blocks are joined into superblocks (later
blocks add into slots that earlier ones wrote), in every form: against the
oracle on sampled rows, the one-sided kernels and themselves."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import test_symmetric_gpu as sym  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2510_02135_gb300 import _build

    _build.build()


# blocks per superblock: 2 from the sizes at which one slot per block would pass 128 (or 256 MiB) on, 4 from twice
# those; 60001 and 99999 in free space with all blocks: the largest symmetric products with one block each
@pytest.mark.parametrize("n,angular,fp64,wall", [
    (40001, False, True, False), (60001, False, True, False), (30001, True, True, False), (40001, True, True, False),
    (80001, False, False, True), (150001, False, False, True), (40001, True, False, True), (70001, True, False, True),
    (60001, True, False, False), (99999, True, False, False)])
def test_product(orc, n, angular, fp64, wall):
    sym.test_symmetric_product(orc, n, angular, fp64, wall)


@pytest.mark.parametrize("n,angular,fp64", [(30001, False, True), (40001, False, True), (25001, True, True),
                                            (35001, True, True), (70001, True, False), (140001, True, False)])
def test_adjoint(n, angular, fp64):
    sym.test_symmetric_adjoint(n, angular, fp64)
