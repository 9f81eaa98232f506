"""Which launches a call takes: the query's answers, and the sweeps that a batch and a large grid run."""
import pytest

from paper_2312_10316_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_10316_gb300 import trtr as T  # noqa: E402

from .test_gpu_step2 import _random_solver  # noqa: E402


@pytest.mark.parametrize("nx,ny,prec,answers", [
    (64, 48, "f32", {1: 1, 2: 2, 11: 2, 12: 4}),      # small: four steps in calls of 12 steps or more
    (640, 480, "f32", {1: 1, 3: 2, 4: 4, 60: 4}),     # 2^18 nodes: of four or more
    (65, 48, "f16", {2: 1, 11: 1, 12: 4}),            # an odd width: no two-step launches
    (20, 16, "f32", {60: 2}),                         # too low for strips
    (64, 48, "f64", {60: 1})])
def test_steps_of_a_calls_first_launch(nx, ny, prec, answers):
    with _random_solver(nx, ny, T.TRTR_GRAD_PERIODIC, 2, precision=T.PRECISIONS[prec]) as s:
        for n, k in answers.items():
            assert s.launch_steps(n) == k, n
        s.set_steps_per_launch(1)
        assert s.launch_steps(60) == 1
        assert T.lib.trtr_get_launch_steps(s.ctx, 0, None) == T.TRTR_EINVAL
    with _random_solver(640, 480, T.TRTR_GRAD_PERIODIC, 2, check_every=6) as s:
        assert s.launch_steps(60) == 4
        s.step(4)
        assert s.launch_steps(60) == 2  # two steps to the stability check


# batches near the line of the choice: the sweep measured 1.3 to 4 times as fast as two-step launches
@pytest.mark.parametrize("sizes", [(700, 33, 250, 123, 641), (64,) * 30, (96,) * 60, (256,) * 30])
@pytest.mark.parametrize("prec", ["f32", "f16"])
@pytest.mark.parametrize("D_amp", [0.0, 0.5])
def test_batches_take_the_sweep_where_it_is_the_faster(sizes, prec, D_amp):
    ps = [W.Pulse(n=n, D_amp=D_amp, courant=0.3) for n in sizes]
    with T.Batch([T.pulse_instance(p, T.PRECISIONS[prec]) for p in ps]) as b:
        assert [b.launch_steps(n) for n in (1, 4, 60)] == [1, 4, 4]
        b.set_steps_per_launch(1)
        assert b.launch_steps(60) == 1


def test_a_batch_of_narrow_instances_keeps_to_two_steps():
    h = 1e-3
    inst = [T.trtr_instance(T.Params(nx=16, ny=5000, dx=h, dt=0.1 * h, precision=T.TRTR_F32, src_mode=T.TRTR_SRC_PULSE,
                                     grad_mode=T.TRTR_GRAD_ONESIDED_EDGE).to_c(), 0.1, 0.0, 2.0, 0.5, 1e-3, 0.5) for _ in range(8)]
    with T.Batch(inst) as b:
        assert b.launch_steps(60) == 2
