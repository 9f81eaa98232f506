"""phi and the reductions of the FP32-computing storages, which sum floats without rounding errors
instead of converting each to FP64: against exact sums (math.fsum) of the populations that the
library gives out, and with infinities, NaN and values at the end of the float range."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_10316_gb300 import trtr as T  # noqa: E402

PREC = {"f64": T.TRTR_F64, "f32": T.TRTR_F32, "f16": T.TRTR_F16_OFS, "bf16": T.TRTR_BF16_OFS}
ULP = 2.0**-52


def _solver(nx, ny, prec, g, **kw):
    s = T.Solver(T.Params(nx=nx, ny=ny, dx=0.1, dt=0.02, precision=PREC[prec], grad_mode=T.TRTR_GRAD_PERIODIC, **kw))
    s.set_fields(np.zeros((ny, nx)), np.zeros((ny, nx)), np.full((ny, nx), 0.1))
    s.set_populations(g)
    return s


@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 3), (7, 5), (64, 9), (129, 33)])
@pytest.mark.parametrize("prec", ["f64", "f32", "f16", "bf16"])
def test_phi_and_sums_are_exact_to_fp64(nx, ny, prec):
    rng = np.random.default_rng(nx * 100 + ny)
    g = rng.uniform(-1, 1, size=(9, ny, nx)) * 10.0 ** rng.integers(-4, 3, size=(9, ny, nx))
    ref = rng.uniform(-1, 1, size=(ny, nx))
    with _solver(nx, ny, prec, g, phi_ref=0.25) as s:
        got = s.get_populations()
        phi = s.moments()
        mass = s.mass()
        rms, rel = s.error_vs(ref)
    exact = np.array([[math.fsum(got[:, j, i]) for i in range(nx)] for j in range(ny)])
    size = np.abs(got).sum(axis=0)
    # FP64 storage adds eight times in FP64; the others round a sum of three parts twice
    assert np.all(np.abs(phi - exact) <= 8 * ULP * size)
    assert abs(mass - math.fsum(exact.ravel())) <= 32 * ULP * size.sum()
    d2 = math.fsum(((exact - ref) ** 2).ravel())
    assert abs(rms - math.sqrt(d2 / (nx * ny))) <= 1e-13 * rms
    assert abs(rel - math.sqrt(d2 / math.fsum((ref**2).ravel()))) <= 1e-13 * rel


@pytest.mark.parametrize("nx", [8, 9])
def test_phi_of_values_beyond_the_float_range(nx):
    ny = 4
    g = np.ones((9, ny, nx))
    g[:, 0, 0] = 3e38  # a finite sum past FP32's range
    g[2, 1, 1] = np.inf
    g[3, 1, 2] = np.nan
    g[1, 2, 3], g[2, 2, 3] = np.inf, -np.inf
    g[5, 3, nx - 1] = -np.inf
    with _solver(nx, ny, "f32", g) as s:
        got = s.get_populations()
        phi = s.moments()
        mass = s.mass()
    with np.errstate(invalid="ignore"):
        want = got.sum(axis=0)
    assert np.array_equal(phi, want, equal_nan=True)
    assert math.isnan(mass)
    with _solver(nx, ny, "f32", np.full((9, ny, nx), 3e38)) as s:
        assert abs(s.mass() - 9 * ny * nx * float(np.float32(3e38))) <= 1e-14 * s.mass()
