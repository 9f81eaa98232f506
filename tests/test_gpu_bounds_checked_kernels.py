"""The tests of the four-step, FP64, reduction, table and initial-state kernels on the bounds-checked build
(TRTR_BOUNDS_CHECK=1), where a conftest fixture asserts after every test that nothing was recorded."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_10316_gb300 import trtr as T  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SUITES = ["tests/test_gpu_sweep.py", "tests/test_gpu_sums.py", "tests/test_gpu_f64.py", "tests/test_gpu_sweep_units.py",
          "tests/test_gpu_narrow.py", "tests/test_gpu_init.py", "tests/test_gpu_pulse_tables.py", "tests/test_gpu_batch_tables.py",
          "tests/test_gpu_batch_clock.py", "tests/test_gpu_capture.py", "tests/test_gpu_launch_steps.py"]


@pytest.mark.skipif(T.BOUNDS_CHECKED, reason="already running on the checked build")
def test_kernel_suites_on_the_bounds_checked_build():
    from paper_2312_10316_gb300.build import build_library

    build_library(checked=True)
    cmd = [sys.executable, "-m", "pytest", "-q", "-x", "-m", "gpu", "-p", "no:cacheprovider", *SUITES]
    r = subprocess.run(cmd, cwd=ROOT, env=dict(os.environ, TRTR_BOUNDS_CHECK="1"), capture_output=True, text=True, timeout=1200)
    tail = r.stdout[-4000:] + r.stderr[-2000:]
    assert r.returncode == 0, tail
    assert " passed" in r.stdout and " failed" not in r.stdout, tail
