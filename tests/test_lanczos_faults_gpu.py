"""The one-launch Lanczos iteration when its launch is refused (the separate
kernels serve; LM_ERR_CUDA when that happens with an iteration in flight) and
when a wait among its CTAs runs out (LM_ERR_TIMEOUT), in the bounds-checked
build, which can be told to make each happen.  The solver stays usable."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = r'''
import os, sys
sys.path.insert(0, ".")
import numpy as np, torch
from paper_2510_02135_gb300 import inputs as I, lm
assert lm.lm_debug_bounds(), "not the bounds-checked library"
tol = 1e-5
for n, fp64 in ((1, False), (700, False), (700, True), (5000, False)):
    s_ = I.cube_suspension(5, n, 0.1, 1.0, angular=False, fp32=not fp64)
    s = lm.lm_create(1.0, 1.0, False, lm.LM_FP64 if fp64 else lm.LM_FP32C)
    lm.lm_set_positions(s, torch.from_numpy(s_.pos).cuda())
    W = torch.from_numpy(np.random.default_rng(1).standard_normal(3 * n)).cuda()
    root = lambda: lm.lm_sqrt_mdot(s, W, tol=tol, max_iter=100)[0].double().cpu()
    y = root()
    os.environ["LM_DEBUG_LANCZOS_STEP"] = "refuse"
    z = root()
    # each within 20 tol of the root
    assert float((y - z).norm() / y.norm()) <= 40 * tol, n
    for fault, status in (("refuse_later", lm.LM_ERR_CUDA), ("expire", lm.LM_ERR_TIMEOUT)):
        if n != 700:
            continue
        os.environ["LM_DEBUG_LANCZOS_STEP"] = fault
        try:
            root()
            raise SystemExit("no error from " + fault)
        except lm.LmError as e:
            assert e.status == status, e
        # the scalars' memory grows for more iterations, and the flag of the next positions lies in it
        del os.environ["LM_DEBUG_LANCZOS_STEP"]
        lm.lm_sqrt_mdot(s, W, tol=tol, max_iter=100 + 50 * status)
        lm.lm_set_positions(s, torch.from_numpy(s_.pos).cuda())
        os.environ["LM_DEBUG_LANCZOS_STEP"] = "none"
    del os.environ["LM_DEBUG_LANCZOS_STEP"]
    assert torch.equal(y, root()), n
lm.lm_debug_check()
print("ok")
'''


def test_refused_launch_and_expired_wait():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2510_02135_gb300 import _build

    _build.build(debug_bounds=True)
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=dict(os.environ, LM_DEBUG_BOUNDS="1"),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.strip().endswith("ok")
