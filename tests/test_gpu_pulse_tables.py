"""The FP32 pulse tables, filled in sums of two floats: the source that they give, against the FP64 path's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_10316_gb300 import trtr as T  # noqa: E402

# a factor of the tables takes at most six roundings (2^x counted as two), a source term two products of two
# factors and five more, a step's update about ten: 16 + 5 + 10 units of 2^-24 at the worst, a third of it in L2
TOL = 31 * 2.0**-24 / 3


@pytest.mark.parametrize("nx,ny,sigma0,xc,step", [
    (64, 64, 0.1, 0.3, 0), (20000, 32, 0.1, 0.3, 0), (33, 700, 0.1, -0.5, 0), (512, 512, 0.01, 0.7, 0), (512, 96, 0.3, 0.0, 500),
    (16, 32, 0.05, 0.9, 63)])
def test_source_of_the_tables_is_accurate_to_fp32(nx, ny, sigma0, xc, step):
    """phi from zero after three steps is the source's alone; steps from `step` on, in tables filled there."""
    h = 2.0 / max(nx, ny)
    dt = 0.2 * h
    out = {}
    for prec in (T.TRTR_F64, T.TRTR_F32):
        p = T.Params(nx=nx, ny=ny, dx=h, dt=dt, x0=-h * nx / 2, y0=-h * ny / 2, precision=prec, src_mode=T.TRTR_SRC_PULSE,
                     grad_mode=T.TRTR_GRAD_ONESIDED_EDGE)
        with T.Solver(p) as s:
            s.set_pulse(1.0, xc * h * nx / 2, 0.0, sigma0, 0.0922 * h * h / dt, 0.5)
            s.set_populations(np.zeros((9, ny, nx)), step=step)
            s.step(3)
            out[prec] = s.moments()
    assert np.linalg.norm(out[T.TRTR_F32] - out[T.TRTR_F64]) <= TOL * np.linalg.norm(out[T.TRTR_F64])
