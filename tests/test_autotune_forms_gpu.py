"""The autotuner and the symmetric product: its answer given back to the solver
pins nothing, and a record that a one-sided configuration was faster is used."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2510_02135_gb300 import inputs, lm  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2510_02135_gb300 import _build

    _build.build()


def test_answer_given_back_pins_nothing():
    n = 8192   # forces: the symmetric form takes two thirds of the one-sided one's time
    s_ = inputs.cube_suspension(8, n, 0.1, 1.0, angular=False, fp32=True)
    x, F = torch.from_numpy(s_.pos).cuda(), torch.from_numpy(s_.F).cuda()

    def solver():
        s = lm.lm_create(1.0, 1.0, False, lm.LM_FP32C)
        lm.lm_set_positions(s, x)
        return s

    want = lm.lm_mdot(solver(), F, None)[0]
    s = solver()
    c = lm.lm_autotune(s, reps=1)
    assert torch.equal(lm.lm_mdot(s, F, None)[0], want)
    lm.lm_set_pair_config(s, c["threads"], c["ilp"], c["splits"], c["packed"])
    assert lm.lm_get_pair_config(s) == c
    assert torch.equal(lm.lm_mdot(s, F, None)[0], want)
    # on another solver, and with another configuration on this one, it pins
    pinned = solver()
    lm.lm_set_pair_config(pinned, c["threads"], c["ilp"], c["splits"], c["packed"])
    assert not torch.equal(lm.lm_mdot(pinned, F, None)[0], want)
    lm.lm_set_pair_config(s, 128, 2, 3, 0)
    assert not torch.equal(lm.lm_mdot(s, F, None)[0], want)


CHILD = r'''
import sys
sys.path.insert(0, ".")
import numpy as np, torch
from paper_2510_02135_gb300 import inputs as I, lm
def run(n, pin=None):
    s_ = I.cube_suspension(6, n, 0.1, 1.0, angular=False, fp32=True)
    s = lm.lm_create(1.0, 1.0, False, lm.LM_FP32C)
    lm.lm_set_positions(s, torch.from_numpy(s_.pos).cuda())
    if pin:
        lm.lm_set_pair_config(s, *pin)
    return lm.lm_mdot(s, torch.from_numpy(s_.F).cuda(), None)[0]
if sys.argv[1] == "key":
    s_ = I.cube_suspension(6, 3000, 0.1, 1.0, angular=False, fp32=True)
    s = lm.lm_create(1.0, 1.0, False, lm.LM_FP32C)
    lm.lm_set_positions(s, torch.from_numpy(s_.pos).cuda())
    lm.lm_autotune(s, reps=1)
else:
    pin = tuple(int(v) for v in sys.argv[2].split(","))
    print(int(torch.equal(run(3000), run(3000, pin))), int(torch.equal(run(5000), run(5000, (128, 2, 0, 1)))))
'''


def _child(cache, *args):
    r = subprocess.run([sys.executable, "-c", CHILD, *args], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, LM_AUTOTUNE_CACHE=str(cache)))
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout


def test_recorded_one_sided_choice_is_used(tmp_path):
    """The record holds for its N bucket; another N keeps the symmetric form."""
    cache = tmp_path / "tune.jsonl"
    _child(cache, "key")
    entry = json.loads(cache.read_text())
    entry.pop("one_sided", None)
    for one_sided in (False, True):
        e = dict(entry, threads=128, ilp=2, splits=7, packed=1, **({"one_sided": 1} if one_sided else {}))
        cache.write_text(json.dumps(e) + "\n")
        assert _child(cache, "run", "128,2,7,1").split() == ["%d" % one_sided, "0"]
