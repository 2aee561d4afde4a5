"""Where the checks of the batched graph lie: a problem whose check is due waits for
the next one, so a check period shorter than a launch has checks inside it."""
import numpy as np
import pytest

from test_gpu_loop_forms import sized
from test_gpu_parity import P  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def make(P, inst, k_chk, chunk, precision):
    h = P.create_from_instance(inst, precision=precision)
    for name, v in (("persistent", 0), ("iter_budget", 800), ("k_chk", k_chk), ("batch_chunk", chunk)):
        P.pdnqp_set_param(h, name, v)
    return h


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("k_chk,chunk", [(1, 16), (8, 64), (24, 16), (63, 16), (64, 256), (7, 5)])
def test_launches_and_bits(P, k_chk, chunk, precision):
    inst = sized(900, 300)
    alone = make(P, inst, k_chk, chunk, precision)
    P.pdnqp_solve(alone, 1e-6, 1e-6)
    h = make(P, inst, k_chk, chunk, precision)
    P.pdnqp_solve_batch([h], 1e-6, 1e-6)
    (x, y, r), (xa, ya, ra) = P.pdnqp_get(h), P.pdnqp_get(alone)
    assert np.array_equal(x, xa) and np.array_equal(y, ya)
    assert (r["outer_iters"], r["trials"], r["restarts"]) == (ra["outer_iters"], ra["trials"], ra["restarts"])
    # Each inner solve ends in a launch of its own.  With the checks at most one
    # in twelve slots of a period is idle where k_chk allows it (25 slots of 24, 64 of 63),
    # and a rejection (rare here) may cost the slots up to the next check.
    rejected = r["trials"] - r["inner_iters"]
    every = {(1, 16): 1, (8, 64): 8, (24, 16): 8, (63, 16): 16, (64, 256): 64, (7, 5): 1}[k_chk, chunk]
    slots = r["trials"] * (64.0 / 63.0) + rejected * every
    assert P.pdnqp_get_param(h, "batch_graph_launches") <= slots / chunk + r["outer_iters"] + 1
    h.close()
    alone.close()
