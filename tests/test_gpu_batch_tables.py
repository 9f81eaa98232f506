"""The pulse tables of a batch's instances, which the batch and an instance's own calls fill: whoever steps
takes the source at its own times."""
import numpy as np
import pytest

from paper_2312_10316_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_10316_gb300 import trtr as T  # noqa: E402

PULSES = [W.Pulse(n=n, D_amp=0.5, courant=0.3) for n in (64, 48, 130)]


def _populations(ctx, p):
    out = np.zeros((9, p.ny, p.nx))
    T.trtr_get_populations(ctx, out)
    return out


def _single(p, steps):
    with T.pulse_solver(p, precision=T.TRTR_F32) as s:
        s.set_steps_per_launch(1)
        s.step(steps)
        return s.get_populations()


@pytest.mark.parametrize("steps_per_launch", [1, 2])
@pytest.mark.parametrize("steps", [16, 1])
def test_an_instance_starts_over_after_the_batch(steps_per_launch, steps):
    """The batch has refilled the tables from a later level; the instance goes back to step 0."""
    with T.Batch([T.pulse_instance(p, T.TRTR_F32) for p in PULSES]) as b:
        b.set_steps_per_launch(steps_per_launch)
        b.step(70)
        ctx = T.trtr_batch_instance(b.b, 1)
        T.trtr_init_equilibrium(ctx, PULSES[1].nx * PULSES[1].ny, None)
        T.trtr_step(ctx, steps)
        got = _populations(ctx, PULSES[1])
    assert np.array_equal(got, _single(PULSES[1], steps))


@pytest.mark.parametrize("steps_per_launch", [1, 2])
def test_a_batch_goes_on_after_an_instance_was_stepped_and_put_back(steps_per_launch):
    """The instance's own steps refill its tables; its state, step and buffer are then the batch's again."""
    with T.Batch([T.pulse_instance(p, T.TRTR_F32) for p in PULSES]) as b:
        b.set_steps_per_launch(steps_per_launch)
        b.step(72)
        ctx = T.trtr_batch_instance(b.b, 2)
        blob = T.trtr_save(ctx)
        T.trtr_set_steps_per_launch(ctx, 1)
        T.trtr_step(ctx, 60)  # past the levels that the batch has filled; an even number of launches
        T.trtr_set_steps_per_launch(ctx, 2)
        T.trtr_load(ctx, blob)
        b.step(30)
        got = [b.instance(k).get_populations() for k in range(len(PULSES))]
    for p, g in zip(PULSES, got):
        assert np.array_equal(g, _single(p, 102)), p.n


def test_an_instance_takes_its_own_pulse_after_the_batch_has_filled_its_tables():
    """trtr_set_pulse on an instance's context: the batch fills its tables with the pulse that it was made with,
    the instance's own steps take the new one's source."""
    p = PULSES[0]
    other = dict(omega=p.omega, xc=-p.xc, yc=p.yc + 0.1, sigma0=p.sigma0, D0=p.D0, D_amp=0.25)
    args = (other["omega"], other["xc"], other["yc"], other["sigma0"], other["D0"], other["D_amp"])
    with T.Batch([T.pulse_instance(q, T.TRTR_F32) for q in PULSES]) as b:
        b.step(16)
        ctx = T.trtr_batch_instance(b.b, 0)
        T.trtr_set_pulse(ctx, *args)
        b.step(16)
        T.trtr_init_equilibrium(ctx, p.nx * p.ny, None)
        T.trtr_step(ctx, 16)
        got = _populations(ctx, p)
    with T.pulse_solver(p, precision=T.TRTR_F32) as s:
        s.set_steps_per_launch(1)
        s.set_pulse(*args)
        s.init_equilibrium(None)
        s.step(16)
        assert np.array_equal(s.get_populations(), got)
