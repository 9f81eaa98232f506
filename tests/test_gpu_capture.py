"""trtr_step captured into a CUDA graph on the context's stream: a replay takes the same steps on from the
state, fields and pulse tables' times that an eager call would, whatever ran in between."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_10316_gb300 import trtr as T  # noqa: E402
from paper_2312_10316_gb300 import workloads as W  # noqa: E402

from ._gpu_util import random_case  # noqa: E402


def _flow(nx, ny, prec, stream, src=T.TRTR_SRC_NONE):
    case = random_case(7 + nx, nx, ny)
    s = T.Solver(T.Params(nx=nx, ny=ny, dx=case["dx"], dt=case["dt"], precision=T.PRECISIONS[prec], src_mode=src,
                          grad_mode=T.TRTR_GRAD_PERIODIC, rounding=T.TRTR_ROUND_NEAREST), stream=stream)
    s.set_fields(case["ux"], case["uy"], case["D"], case["S1"] if src == T.TRTR_SRC_FIELD else None)
    s.set_populations(case["g"])
    return s, case


def _capture(s, st, n):
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=st):
        s.step(n)
    return g


def _replay(g, st, times=1):
    with torch.cuda.stream(st):
        for _ in range(times):
            g.replay()
    st.synchronize()


# calls of an even number of launches of one and two steps, so that a replay leaves the state where it found it
@pytest.mark.parametrize("nx,ny,prec,src,n", [
    (64, 48, "f32", "none", 12), (640, 480, "f32", "none", 20), (640, 480, "f16", "none", 4), (130, 64, "f32", "none", 15),
    (65, 48, "bf16", "none", 12), (130, 64, "f32", "field", 12), (48, 40, "f64", "none", 4)])
def test_replays_go_on_from_the_state(nx, ny, prec, src, n):
    st = torch.cuda.Stream()
    mode = T.TRTR_SRC_FIELD if src == "field" else T.TRTR_SRC_NONE
    s, _ = _flow(nx, ny, prec, st.cuda_stream, mode)
    ref, _ = _flow(nx, ny, prec, st.cuda_stream, mode)
    with s, ref:
        s.step(n)
        g = _capture(s, st, n)
        _replay(g, st, 3)
        ref.step(n + 3 * n)
        assert np.array_equal(s.get_populations(), ref.get_populations())
        # eager calls between the replays
        s.step(2 * n)
        _replay(g, st)
        s.step(n)
        ref.step(4 * n)
        assert np.array_equal(s.get_populations(), ref.get_populations())


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_a_replay_takes_fields_that_were_set_in_between(prec):
    st = torch.cuda.Stream()
    s, case = _flow(64, 48, prec, st.cuda_stream)
    ref, _ = _flow(64, 48, prec, st.cuda_stream)
    with s, ref:
        s.step(4)
        g = _capture(s, st, 4)
        _replay(g, st)
        for t in (s, ref):
            if t is ref:
                t.step(8)
            t.set_fields(case["uy"], case["ux"], 0.5 * case["D"])
        _replay(g, st)
        ref.step(4)
        assert np.array_equal(s.get_populations(), ref.get_populations())


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
def test_a_replay_takes_the_pulse_at_the_captured_times(prec):
    st = torch.cuda.Stream()
    pulse = W.Pulse(n=64, D_amp=0.5, courant=0.3)
    with T.pulse_solver(pulse, precision=T.PRECISIONS[prec], stream=st.cuda_stream) as s:
        s.step(12)
        want = s.get_populations()
        s.init_equilibrium(None)
        g = _capture(s, st, 12)
        s.init_equilibrium(None)
        s.step(64)  # past the levels that the captured call uses
        later = s.get_populations()
        s.init_equilibrium(None)
        _replay(g, st)
        assert np.array_equal(s.get_populations(), want)
        s.init_equilibrium(None)
        s.step(40)
        blob = s.save()
        s.init_equilibrium(None)
        _replay(g, st)  # leaves the tables at its own levels
        s.load(blob)
        s.step(24)
        assert np.array_equal(s.get_populations(), later)
