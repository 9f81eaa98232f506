"""A batch after a launch whose wait gave up: its step counts, and what follows takes the pulse source at the
times that the host's step says."""
import numpy as np
import pytest

from paper_2312_10316_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_10316_gb300 import trtr as T  # noqa: E402


@pytest.mark.parametrize("prec", ["f32", "f16"])
@pytest.mark.parametrize("steps_per_launch", [1, 2])
def test_a_batch_goes_on_after_a_timeout(prec, steps_per_launch):
    precision = T.PRECISIONS[prec]
    pulses = [W.Pulse(n=n, D_amp=0.5, courant=0.3) for n in (64, 48, 130)]
    with T.Batch([T.pulse_instance(p, precision) for p in pulses]) as b:
        b.set_steps_per_launch(steps_per_launch)
        b.step(6)
        b.sync()
        for _ in range(3):  # void steps, each reported once
            assert T.trtr_batch_check_timeout_path(b.b, 1000) == T.TRTR_ETIMEOUT
            T.trtr_batch_sync(b.b)
        assert T.trtr_batch_check_timeout_path(b.b, 0) == T.TRTR_EINVAL
        step = b.info()["step"]
        assert step == 9
        states = []
        for k, p in enumerate(pulses):
            g = W.random_populations(50 + k, p.ny, p.nx, base=1.0, amp=0.1)
            T.trtr_set_populations(T.trtr_batch_instance(b.b, k), g.size, g, step=step)
            states.append(g)
        b.step(70)  # past the levels of the tables' fill
        b.step(75)
        b.sync()
        got = [b.instance(k).get_populations() for k in range(len(pulses))]
    for p, g, out in zip(pulses, states, got):
        with T.pulse_solver(p, precision=precision) as s:
            s.set_steps_per_launch(1)
            s.set_populations(g, step=step)
            s.step(145)
            assert np.array_equal(s.get_populations(), out, equal_nan=True), p.n
