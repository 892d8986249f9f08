"""The symmetric product (every unordered pair once, both particles written)
against the FP64 oracle at the sizes where its blocks, tiles, item rows and
superblocks change, against the pinned one-sided kernel, and bitwise against
itself."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2510_02135_gb300 import lm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2510_02135_gb300 import _build

    _build.build()


def dev(x):
    return None if x is None else torch.from_numpy(np.ascontiguousarray(x)).cuda()


def rel(y, ref):
    y, ref = np.asarray(y, np.float64).ravel(), np.asarray(ref, np.float64).ravel()
    return np.linalg.norm(y - ref) / np.linalg.norm(ref)


def system(n, dt, wall):
    """Spheres at volume fraction about 0.1 with overlapping neighbours, a
    coincident pair whose members lie in different blocks, and above a wall
    some particles that touch or cross it."""
    rng = np.random.default_rng(n)
    side = (n * 42.0) ** (1.0 / 3.0) + 1.0
    pos = rng.uniform(-side / 2, side / 2, (n, 3))
    if wall:
        pos[:, 2] = rng.uniform(-0.3, side, n)
    if n > 2:
        pos[n - 1] = pos[0]
        pos[n // 2] = pos[1] + [0.9, 0.2, 0.3]
    F, T = rng.standard_normal((2, n, 3))
    return pos.astype(dt), F.astype(dt), T.astype(dt)


# FP64: i-blocks of 128, j-tiles of 8, 16 (from 801) and 32 (from 3001).  FP32: i-blocks of 256 and j-tiles of 32
# or 64 up to some thousand particles, then i-blocks of 512 (free space to
# 40000, wall) and 1024 with j-tiles of 128; from N = 131073 blocks are joined
# into superblocks so that the slots stay at 128.
CASES = ([(n, ang, True, False) for n in (1, 2, 33, 129, 800, 801, 3001) for ang in (False, True)]
         + [(n, ang, False, wall) for n in (1, 2, 33, 257, 3499) for ang in (False, True) for wall in (False, True)]
         + [(n, False, False, False) for n in (3500, 9999, 10001, 40001, 150001)] + [(n, True, False, False) for n in (10999, 11000, 30001)]
         + [(n, False, False, True) for n in (3500, 10001)] + [(n, True, False, True) for n in (5000, 5377)])


@pytest.mark.parametrize("n,angular,fp64,wall", CASES)
def test_symmetric_product(orc, n, angular, fp64, wall):
    pos, F, T = system(n, np.float64 if fp64 else np.float32, wall)
    T = T if angular else None
    out = []
    for pinned in (False, True):
        s = lm.lm_create(0.9, 1.0, angular, lm.LM_FP64 if fp64 else lm.LM_FP32C,
                         periodicity=("open", "open", "single_wall" if wall else "open"))
        lm.lm_set_positions(s, dev(pos))
        if pinned:
            c = lm.lm_get_pair_config(s)
            lm.lm_set_pair_config(s, c["threads"], c["ilp"], c["splits"], c["packed"])
        out.append([v for v in lm.lm_mdot(s, dev(F), dev(T)) if v is not None])
        if not pinned:
            again = [v for v in lm.lm_mdot(s, dev(F), dev(T)) if v is not None]
            assert all(torch.equal(a, b) for a, b in zip(out[0], again))
    rows = np.unique(np.concatenate([[0, 1, n // 2, n - 1], np.random.default_rng(1).integers(0, n, 200)]) % n)
    ref = [v for v in orc.mdot(pos, F, T, 1.0, 0.9, angular, rows=rows, wall=wall) if v is not None]
    # the product's bounds: 1e-12 (FP64), 1e-5 (FP32 compensated)
    tol = 1e-12 if fp64 else 1e-5
    for a, b, r in zip(*out, ref):
        a, b = a.cpu().numpy(), b.cpu().numpy()
        if not np.abs(r).max() > 0.0:   # a single particle below the wall
            assert not a.any()
            continue
        assert rel(a[rows], r) <= tol, (n, rel(a[rows], r))
        assert rel(a, b) <= tol, (n, rel(a, b))


@pytest.mark.parametrize("fp64,wall,n", [(False, False, 400), (False, True, 400), (False, False, 4100), (True, False, 300)])
def test_symmetric_product_in_the_square_root(fp64, wall, n):
    """FP64 Krylov vectors enter the symmetric product and FP64 sums leave it."""
    pos, _, _ = system(n, np.float64 if fp64 else np.float32, wall)
    pos = pos[1:n - 1]   # without the coincident pair (M stays positive definite)
    W = dev(np.random.default_rng(2).standard_normal(3 * len(pos)))
    ys = []
    for pinned in (False, True):
        s = lm.lm_create(1.0, 1.0, False, lm.LM_FP64 if fp64 else lm.LM_FP32C,
                         periodicity=("open", "open", "single_wall" if wall else "open"))
        lm.lm_set_positions(s, dev(pos))
        if pinned:
            c = lm.lm_get_pair_config(s)
            lm.lm_set_pair_config(s, c["threads"], c["ilp"], c["splits"], c["packed"])
        ys.append(lm.lm_sqrt_mdot(s, W, tol=1e-4, max_iter=150)[0].double().cpu().numpy())
    assert rel(ys[0], ys[1]) <= 20e-4   # each within 20 tol of the root


@pytest.mark.parametrize("n,angular,fp64", [(1, False, True), (2, True, True), (129, False, True), (300, True, True),
                                            (129, True, False), (1000, True, False), (10241, True, False),
                                            (3000, False, False), (10241, False, False), (66000, False, False)])
def test_symmetric_adjoint(n, angular, fp64):
    """The default adjoint against the one-sided kernel and bitwise against
    itself; 66000 particles join i-blocks into superblocks."""
    dt = np.float64 if fp64 else np.float32
    pos, F, T = system(n, dt, False)
    G, H = np.random.default_rng(3).standard_normal((2, n, 3)).astype(dt)
    s = lm.lm_create(0.9, 1.0, angular, lm.LM_FP64 if fp64 else lm.LM_FP32C)
    lm.lm_set_positions(s, dev(pos))
    args = [dev(v) for v in ((F, T, G, H) if angular else (F, None, G, None))]
    out = []
    assert lm.lm_get_adjoint_config(s)["packed"] >= 3
    for one_sided in (False, True):
        if one_sided:
            ilp = 1 if fp64 else (2 if angular else 4)
            lm.lm_set_adjoint_config(s, 128, ilp, 0, 0 if fp64 or angular else 1)
        out.append([v for v in lm.lm_mdot_backward(s, *args) if v is not None])
        again = [v for v in lm.lm_mdot_backward(s, *args) if v is not None]
        assert all(torch.equal(a, b) for a, b in zip(out[-1], again))
    for a, b in zip(*out):   # the adjoint's bounds: 1e-12 (FP64), 1e-5 (FP32)
        b = b.cpu().numpy()
        if np.abs(b).max() > 0.0:
            assert rel(a.cpu().numpy(), b) <= (1e-12 if fp64 else 1e-5), n
        else:
            assert not a.cpu().numpy().any()
