"""Four steps per launch (strips swept by four time levels behind one another, tiles on small grids): the
bits of one launch per step, at the edges of strips (120 columns), tiles, row blocks and ghost frames."""
import dataclasses

import numpy as np
import pytest

from paper_2312_10316_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_10316_gb300 import trtr as T  # noqa: E402

from ._gpu_util import random_case  # noqa: E402
from .test_gpu_step2 import _pulse_solver, _random_solver  # noqa: E402

PREC = {"f32": T.TRTR_F32, "f16": T.TRTR_F16_OFS, "bf16": T.TRTR_BF16_OFS}
# the smallest, the two tile heights of small grids (32 x 4 and 32 x 8 nodes) and sweeps (from 450 x 450
# on), ragged in both directions; odd widths, where halo pairs fall between the rounding's pairs
GRIDS = [(16, 32), (17, 33), (37, 50), (122, 35), (250, 300), (263, 301), (481, 470), (600, 330), (1201, 133)]


@pytest.mark.parametrize("nx,ny", GRIDS)
@pytest.mark.parametrize("prec", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("kind", ["none", "pulse"])
@pytest.mark.parametrize("rounding", [T.TRTR_ROUND_STOCHASTIC, T.TRTR_ROUND_NEAREST])
def test_sweeps_equal_one_step_launches_bitwise(nx, ny, prec, kind, rounding):
    if prec == "f32" and rounding == T.TRTR_ROUND_NEAREST:
        pytest.skip("FP32 storage is not rounded")
    make = _random_solver if kind == "none" else _pulse_solver
    kw = dict(precision=PREC[prec], rounding=rounding)
    if kind == "none" and prec != "f32":
        kw["phi_ref"] = 0.75
    out = {}
    for k in (1, 2):
        with make(nx, ny, T.TRTR_GRAD_ONESIDED_EDGE, k, **kw) as s:
            l0 = s.launches
            s.step(16)  # sweeps only
            l1 = s.launches
            s.step(13)  # sweeps and a single step
            s.step(15)  # sweeps from the one-wide frame that it left, a pair and a single step
            s.step(66)  # past the levels of the pulse tables' first fill
            out[k] = (s.get_populations(), s.moments())
        if k == 2:  # field packing, (pulse tables at odd widths of 2-byte storage), ghost columns, four launches
            assert 1 + 4 <= l1 - l0 <= 2 + 4
    assert np.array_equal(out[1][0], out[2][0], equal_nan=True)
    assert np.array_equal(out[1][1], out[2][1], equal_nan=True)


@pytest.mark.parametrize("nx,ny", [(16, 32), (243, 64), (1300, 130)])
@pytest.mark.parametrize("prec", ["f32", "f16"])
def test_sweeps_with_a_source_field_equal_one_step_launches_bitwise(nx, ny, prec):
    """Sweeps run while the field stays the same; after each change one single step comes first."""
    case = random_case(31 + nx, nx, ny)
    out = {}
    for k in (1, 2):
        p = T.Params(nx=nx, ny=ny, dx=case["dx"], dt=case["dt"], precision=PREC[prec], src_mode=T.TRTR_SRC_FIELD,
                     grad_mode=T.TRTR_GRAD_PERIODIC)
        with T.Solver(p) as s:
            s.set_steps_per_launch(k)
            s.set_fields(case["ux"], case["uy"], case["D"], case["S1"])
            s.set_populations(case["g"])
            l0 = s.launches
            s.step(16)
            l1 = s.launches
            s.set_source(case["S2"])
            s.step(19)
            blob = s.save()
            s.set_source(case["S1"])
            s.step(14)
            s.load(blob)
            s.step(12)
            out[k] = s.get_populations()
        if k == 2:
            assert 2 + 4 <= l1 - l0 <= 3 + 4  # fields, source term, (ghost columns), four launches
    assert np.array_equal(out[1], out[2])


def test_sweeps_stop_at_the_stability_checks():
    res = {}
    for k in (1, 2):
        with _random_solver(130, 64, T.TRTR_GRAD_PERIODIC, k, check_every=7) as s:
            s.step(30)
            res[k] = s.get_populations()
    assert np.array_equal(res[1], res[2])


@pytest.mark.parametrize("prec", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("D_amp", [0.0, 0.5])
def test_batched_sweeps_equal_single_solves_bitwise(prec, D_amp):
    """Uneven instances (odd widths, more than one strip, several segments) through the batch's four-step
    launches, with steps left over for the two- and one-step ones."""
    pulses = [W.Pulse(n=n, D_amp=D_amp, courant=0.3, sigma0=0.1 + 0.01 * k) for k, n in enumerate((700, 33, 250, 123, 641))]
    if prec != "f32":
        pulses = [dataclasses.replace(p, n=p.n + k % 2) for k, p in enumerate(pulses)]
    with T.Batch([T.pulse_instance(p, PREC[prec]) for p in pulses]) as b:
        b.step(8)
        b.step(7)
        b.step(70)
        got = [b.instance(k).get_populations() for k in range(len(pulses))]
    for p, g in zip(pulses, got):
        with T.pulse_solver(p, precision=PREC[prec]) as s:
            s.set_steps_per_launch(1)
            s.step(85)
            assert np.array_equal(s.get_populations(), g), p.n
