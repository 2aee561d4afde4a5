"""The grid barrier of the solver's own launches runs out of polls: the solve has
to report it, and the same solver has to work afterwards."""
import pytest

from test_gpu_parity import P  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def test_solve_reports_a_barrier_that_gave_up(P):
    gave_up, seconds = P.pdnqp_selftest_wait(2)
    assert gave_up
    assert seconds < 60.0
