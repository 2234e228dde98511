"""The bounds-checked build on the kernels that small shapes do not reach: large FP64 updates, adjoints,
batches (needs a GB300).  No check may fire."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_index_checks_hold_in_updates_adjoints_and_batches():
    from paper_2311_11943_gb300 import build
    build.build(debug_bounds=True)
    r = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "_debug_bounds_update_child.py")],
                       capture_output=True, text=True, timeout=900, cwd=ROOT,
                       env=dict(os.environ, CQR_LIBRARY="debug"))
    assert r.returncode == 0, r.stderr[-3000:]
    out = json.loads([ln for ln in r.stdout.splitlines() if ln.startswith("{")][-1])
    assert sorted(out) == ["adjoint f32", "adjoint f64", "batch", "f64 update"]
    for name, c in out.items():
        assert c["status"] == 0 and c["bounds"] == 0 and c["site"] == 0, (name, c)
        assert c.get("finite", True), name
    assert out["f64 update"]["ran"] > 0 and out["f64 update"]["err"] < out["f64 update"]["tol"]
