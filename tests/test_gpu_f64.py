"""The FP64 step past the time levels of the pulse tables' first fill, in one call."""
import pytest

from paper_2312_10316_gb300 import workloads as W

from ._gpu_util import TOL_F64, oracle_for_pulse, rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2312_10316_gb300 import trtr as T  # noqa: E402


def test_f64_pulse_source_over_several_table_fills():
    pulse = W.Pulse(n=45, D_amp=0.5, courant=0.2, D0=2e-2)
    o = oracle_for_pulse(pulse)
    with T.pulse_solver(pulse, precision=T.TRTR_F64) as s:
        s.step(150)
        o.step(150)
        assert rel_l2(s.moments(), o.phi()) <= TOL_F64
        s.init_equilibrium(None)  # back to step 0: the tables are filled again
        s.step(3)
        o.init_equilibrium(W.phi_analytic(pulse, 0.0))
        o.step(3)
        assert rel_l2(s.get_populations(), o.get_g()) <= TOL_F64
