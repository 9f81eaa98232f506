"""Grids where a strip of the four-step sweep is mostly empty columns, or its segments mostly ramp, keep to
two steps a launch; the others take four.  The same bits either way."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_10316_gb300 import trtr as T  # noqa: E402

from .test_gpu_step2 import _pulse_solver, _random_solver  # noqa: E402


# (sizes, storage, source, steps a launch): narrow and tall, wide and low; beside them wider and higher ones,
# one column past a strip, and a narrow one where the two-step kernel does not apply
@pytest.mark.parametrize("nx,ny,prec,kind,taken", [
    (16, 8000, "f32", "pulse", 2), (16, 8000, "f32", "none", 2), (20000, 32, "f32", "pulse", 2), (20000, 32, "f32", "none", 2),
    (20000, 32, "f16", "pulse", 2), (64, 8000, "f32", "pulse", 4), (121, 2000, "f32", "pulse", 4), (4000, 64, "f32", "none", 4),
    (16, 8000, "f16", "pulse", 4), (17, 8000, "bf16", "none", 4)])
def test_four_steps_a_launch_only_where_they_end_sooner(nx, ny, prec, kind, taken):
    make = _random_solver if kind == "none" else _pulse_solver
    out = {}
    for k in (1, 2):
        with make(nx, ny, T.TRTR_GRAD_PERIODIC, k, precision=T.PRECISIONS[prec]) as s:
            s.step(4)
            l0 = s.launches
            s.step(32)
            launches = s.launches - l0
            out[k] = s.get_populations(), launches
    assert np.array_equal(out[1][0], out[2][0], equal_nan=True)
    # the launches of 32 steps, and the ghost cells' or the packed fields'
    assert 32 // taken <= out[2][1] <= 32 // taken + 2
