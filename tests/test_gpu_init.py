"""The initial state depends on a node's place alone: grids of every block width of the pulse's kernel (128 to
16 columns, ragged and of one node) hold, bit for bit, the window of a larger grid."""
import functools

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_10316_gb300 import trtr as T  # noqa: E402

PREC = {"f64": T.TRTR_F64, "f32": T.TRTR_F32, "bf16": T.TRTR_BF16_OFS}


def _state(nx, ny, prec, given):
    p = T.Params(nx=nx, ny=ny, dx=0.01, dt=0.002, x0=-0.9, y0=-0.4, precision=PREC[prec], grad_mode=T.TRTR_GRAD_ONESIDED_EDGE)
    with T.Solver(p) as s:
        s.set_pulse(0.5, 0.2, -0.1, 0.3, 0.01, 0.5)
        s.init_equilibrium(given)
        return s.get_populations()


@functools.cache
def _large(shape, prec, pulse):
    phi0 = np.random.default_rng(3).uniform(0.5, 1.5, size=shape[::-1])
    return _state(*shape, prec, None if pulse else phi0), phi0


@pytest.mark.parametrize("nx,ny", [(1, 50), (50, 1), (16, 40), (17, 33), (40, 3000), (63, 9), (64, 20), (130, 70), (257, 3), (1900, 40)])
@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("pulse", [True, False])
def test_initial_state_is_the_window_of_a_larger_grids(nx, ny, prec, pulse):
    large, phi0 = _large((300, 3100) if nx < 300 else (2048, 128), prec, pulse)
    got = _state(nx, ny, prec, None if pulse else phi0[:ny, :nx])
    assert np.array_equal(got, large[:, :ny, :nx])
