"""Scratch memory of the product and of the adjoint: a product captured in a
CUDA graph, products and gradients on two streams, and a capture on a solver
that has no scratch yet."""
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


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def setup(n, angular, fp64):
    s_ = inputs.cube_suspension(21, n, 0.1, 1.0, angular=angular, fp32=not fp64)
    s = lm.lm_create(1.0, 1.0, angular, lm.LM_FP64 if fp64 else lm.LM_FP32C)
    x = dev(s_.pos)
    lm.lm_set_positions(s, x)
    F, G = dev(s_.F), dev(s_.G)
    T, H = (dev(s_.T), dev(s_.H)) if angular else (None, None)
    out = [torch.empty_like(F), torch.empty_like(F) if angular else None]
    return s, x, (F, T, G, H), out


FORMS = [(4096, False, False), (3000, True, False), (700, False, True), (500, True, True)]


@pytest.mark.parametrize("n,angular,fp64", FORMS)
def test_captured_product_outlives_a_gradient(n, angular, fp64):
    """The adjoint needs more partial sums than the product; the replay still
    finds the buffer that it was captured with."""
    s, x, (F, T, G, H), out = setup(n, angular, fp64)
    lm.lm_mdot(s, F, T, *out)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        lm.lm_mdot(s, F, T, *out)
    lm.lm_mdot_backward(s, F, T, G, H)
    F.mul_(-0.5)
    lm.lm_set_positions(s, x * 1.25)
    for o in out:
        if o is not None:
            o.zero_()
    g.replay()
    torch.cuda.synchronize()
    again = lm.lm_mdot(s, F, T)
    for a, b in zip(out, again):
        assert b is None or torch.equal(a, b)


@pytest.mark.parametrize("n,angular,fp64", FORMS)
def test_product_and_gradient_on_two_streams(n, angular, fp64):
    s, _, (F, T, G, H), out = setup(n, angular, fp64)
    want = lm.lm_mdot(s, F, T)
    want_g = lm.lm_mdot_backward(s, F, T, G, H)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(20):
        with torch.cuda.stream(a):
            lm.lm_mdot(s, F, T, *out)
        with torch.cuda.stream(b):
            got_g = lm.lm_mdot_backward(s, F, T, G, H)
    torch.cuda.synchronize()
    for p, q in zip([*out, *got_g], [*want, *want_g]):
        assert q is None or torch.equal(p, q)


@pytest.mark.parametrize("angular", [False, True])
@pytest.mark.parametrize("fp64", [False, True])
def test_capture_without_scratch(angular, fp64):
    """A system of one j-tile needs no scratch in the one-sided form, which
    serves while a capture forbids allocation."""
    n = 100
    s, _, (F, T, G, H), _ = setup(n, angular, fp64)
    want, want_g = lm.lm_mdot(s, F, T), lm.lm_mdot_backward(s, F, T, G, H)
    fresh, _, _, out = setup(n, angular, fp64)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        lm.lm_mdot(fresh, F, T, *out)
        back = lm.lm_mdot_backward(fresh, F, T, G, H)
    g.replay()
    torch.cuda.synchronize()
    tol = 1e-12 if fp64 else 1e-5   # the product's and the adjoint's bounds
    for p, q in zip([*out, *back], [*want, *want_g]):
        if q is not None:
            assert float((p.double() - q.double()).norm() / q.double().norm()) <= tol
