"""A remembered choice of the autotuner for the shorter span runs passes of that
span: spans S and S/2 are timed as what they are.  (A process of its own: the file
of choices is read once.)"""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

CODE = """
import numpy as np
from paper_2203_10477_gb300 import inputs, rswr as R
nx, T = 9001, 150
r = inputs.rng(1)
fA, q0 = (r.standard_normal(n).astype(np.float32) for n in (T + 1, nx))
make = lambda ov: R.Plan(0.0, 1.0, 1.0, nx, 0.9 / (nx - 1), 4, ov, dtype=R.F32)
ref = make(64).run(fA, None, T, q0=q0)["u"].cpu().numpy()
for ov, S, halo in ((64, 16, 16), (32, 16, 32), (40, 10, 12)):
    plan = make(ov)
    assert plan.autotune(64) == 0
    info = plan.info()
    assert (info["span_steps"], info["halo"]) == (S, halo), info
    assert np.array_equal(plan.run(fA, None, T, q0=q0)["u"].cpu().numpy(), ref)
    plan.check()
print("as remembered")
"""


def test_a_remembered_shorter_span_is_what_runs(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_10477_gb300 import build

    build.build()
    # dtype : form : log2 of the points : batch : longest span, then variant, mode, span
    cache = tmp_path / "choices"
    cache.write_text("0:1:13:0:32 0 0 16\n0:1:13:0:16 0 0 16\n0:1:13:0:20 0 0 10\n")
    env = dict(os.environ, RSWR_AUTOTUNE_CACHE=str(cache))
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    p = subprocess.run([sys.executable, "-c", CODE], cwd=root, env=env, capture_output=True, text=True, timeout=300)
    assert p.returncode == 0 and "as remembered" in p.stdout, p.stdout + p.stderr
