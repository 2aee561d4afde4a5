"""Counters of the batched graph: of the last batch only."""
import pytest

from test_gpu_loop_forms import sized
from test_gpu_parity import P  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

NAMES = ("batch_graph_seconds", "batch_graph_launches", "batch_kernel_launches", "batch_size")


def test_counters_of_a_problem_that_left_the_graph(P):
    hs = [P.create_from_instance(sized(n, 100)) for n in (300, 700)]
    for h in hs:
        P.pdnqp_set_param(h, "iter_budget", 64)
        P.pdnqp_set_param(h, "persistent", 0)
    P.pdnqp_solve_batch(hs, 1e-6, 1e-6)
    assert all(P.pdnqp_get_param(h, k) > 0 for h in hs for k in NAMES)
    P.pdnqp_set_param(hs[0], "persistent", 1)  # one block of its own
    P.pdnqp_solve_batch(hs, 1e-6, 1e-6)
    assert [P.pdnqp_get_param(hs[0], k) for k in NAMES] == [0, 0, 0, 0]
    assert P.pdnqp_get_param(hs[1], "batch_size") == 1
    for h in hs:
        h.close()
