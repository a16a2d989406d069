"""The bounds-check build on the gather kernels and on the scatter kernels: clean runs
report nothing, a planted node id (tested before the load it would feed) is reported on
either route, single and batched."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))


def test_both_routes():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    env = dict(os.environ, FEM_DEBUG_BOUNDS="1")
    r = subprocess.run([sys.executable, os.path.join(HERE, "debug_bounds_routes_run.py")], env=env,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert len(out["clean"]) == 8 and all(out["clean"].values()), out["clean"]
    assert len(out["planted"]) == 14 and set(out["planted"].values()) == {"FEM_ERR_INDEX"}, out["planted"]
    assert all(out["after"].values()), out["after"]
