"""The index-checked build on the persistent passes (rows and columns of 8192
points) and the fixed-point passes, as tests/test_gpu_checked.py does for the
other kernels: every index check holds, and the results agree with the
ordinary library's to rounding (1e-5 in FP32, 1e-12 else)."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_checked_build_runs_clean_and_agrees(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1509_01450_gb300 import build, sg
    from tests import checked_cases_persistent as cases

    build.build()
    assert sg.lib().sg_checked_build() == 0
    path = str(tmp_path / "checked.npz")
    p = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "checked_cases_persistent.py"), path],
                       env=dict(os.environ, SG_LIBRARY_VARIANT="checked"), capture_output=True, text=True, timeout=1200)
    assert p.returncode == 0, p.stdout[-3000:] + p.stderr[-3000:]
    got, ref = np.load(path), cases.run_all()
    assert set(got.files) == set(ref)
    for k, a in ref.items():
        tol = 1e-5 if k.startswith("float32-") else 1e-12
        assert np.linalg.norm(got[k] - a) <= tol * np.linalg.norm(a), k
