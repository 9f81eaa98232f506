"""Sweeps whose CTAs take several units (strips' segments) one after the other, bit for bit against one-step
launches: a grid with more units than the GPU has SMs, and batches, which are asserted to run them."""
import numpy as np
import pytest

from paper_2312_10316_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_10316_gb300 import trtr as T  # noqa: E402

from ._gpu_util import random_case  # noqa: E402
from .test_gpu_step2 import _pulse_solver  # noqa: E402

ROUND = {"sr": T.TRTR_ROUND_STOCHASTIC, "rn": T.TRTR_ROUND_NEAREST}


# 23 strips of 13 segments on 152 SMs, ragged in both directions
@pytest.mark.parametrize("nx,ny,prec,rounding", [(2641, 2003, "f32", "sr"), (2642, 2003, "f16", "sr"), (2642, 2003, "bf16", "rn"),
                                                 (2641, 2003, "f16", "sr")])
@pytest.mark.parametrize("kind", ["none", "pulse", "field"])
def test_a_ctas_units_follow_one_another_bitwise(nx, ny, prec, rounding, kind):
    out = {}
    for k in (1, 2):
        if kind == "pulse":
            s = _pulse_solver(nx, ny, T.TRTR_GRAD_ONESIDED_EDGE, k, precision=T.PRECISIONS[prec], rounding=ROUND[rounding])
        else:
            case = random_case(77, nx, ny)
            s = T.Solver(T.Params(nx=nx, ny=ny, dx=case["dx"], dt=case["dt"], precision=T.PRECISIONS[prec], rounding=ROUND[rounding],
                                  src_mode=T.TRTR_SRC_FIELD if kind == "field" else T.TRTR_SRC_NONE))
            s.set_steps_per_launch(k)
            s.set_fields(case["ux"], case["uy"], case["D"], 0.1 * case["S1"] if kind == "field" else None)
            s.set_populations(case["g"])
        with s:
            assert s.launch_steps(12) == (4 if k == 2 else 1)
            s.step(12)
            out[k] = s.get_populations()
    assert np.isfinite(out[1]).all()
    assert np.array_equal(out[1], out[2])


@pytest.mark.parametrize("prec,rounding", [("f32", "sr"), ("f16", "sr"), ("f16", "rn"), ("bf16", "sr"), ("bf16", "rn")])
@pytest.mark.parametrize("sizes", [(700, 34, 250, 124, 642), (96,) * 60, (130, 500, 64, 1024, 38, 366)])
@pytest.mark.parametrize("D_amp", [0.0, 0.5])
def test_batched_sweeps_of_even_widths_equal_single_solves_bitwise(prec, rounding, sizes, D_amp):
    kw = dict(rounding=ROUND[rounding])
    ps = [W.Pulse(n=n, D_amp=D_amp, courant=0.3, sigma0=0.1 + 0.001 * k) for k, n in enumerate(sizes)]
    with T.Batch([T.pulse_instance(p, T.PRECISIONS[prec], **kw) for p in ps]) as b:
        assert b.launch_steps(16) == 4
        b.step(16)
        b.step(71)
        got = {k: b.instance(k).get_populations() for k in (0, 1, 2, len(ps) - 1)}
    for k, g in got.items():
        with T.pulse_solver(ps[k], precision=T.PRECISIONS[prec], **kw) as s:
            s.set_steps_per_launch(1)
            s.step(87)
            assert np.array_equal(s.get_populations(), g), ps[k].n
