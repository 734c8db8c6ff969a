"""The work model of the current step kernels against the ncu counts it was made
from: thread instructions (FP32 form) or FP64-pipe thread instructions (FP64
plain, D2Q49) per node, with the counters of the same launches. CPU only."""
import pytest

from paper_2009_13426_gb300 import costmodel as C


def test_instructions_of_the_fp32_form():
    # 2048^2 shear layer, second launch: smsp__thread_inst_executed 6,737 per node
    st = {"node_updates": 1.0, "fp32_iterations": 0.2525, "newton_calls": 1.0317,
          "fp64_evaluations": 1.0327, "fp64_updates": 1.0713, "reconstructions": 0.0938}
    assert C.issue_instr(st) == pytest.approx(6737, rel=0.01)
    more = dict(st, reconstructions=st["reconstructions"] + 1)
    assert C.issue_instr(more) - C.issue_instr(st) == pytest.approx(2000)


def test_slots_of_fp64_plain():
    # 1024^2 shear layer, second launch: 2,134.7
    st = {"node_updates": 1.0, "newton_iterations": 5.4419, "fp32_iterations": 2.328,
          "newton_calls": 1.069, "fp64_evaluations": 4.1829, "reconstructions": 0.1875}
    assert C.plain_slots(st) == pytest.approx(2134.7, rel=0.001)


@pytest.mark.parametrize("iters,iters32,calls,rebuilt,ncu,rel", [
    (6.7602, 3.3682, 1.1777, 1.3125, 8577, 0.001),   # 512^2: the calibration
    (7.1949, 3.1485, 1.474, 3.5, 11233, 0.02),       # 192^2
])
def test_slots_of_d2q49(iters, iters32, calls, rebuilt, ncu, rel):
    st = {"newton_iterations": iters, "fp32_iterations": iters32, "newton_calls": calls,
          "reconstructions": rebuilt}
    assert C.q49_slots(st, 1.0) == pytest.approx(ncu, rel=rel)


def test_issue_peak():
    assert C.ISSUE_PEAK_TINSTR == pytest.approx(152 * 4 * 32 * 2.07e9 / 1e12)
