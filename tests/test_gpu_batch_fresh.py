"""Batches of handles that the graph meets before their own first solve has written
their device state: fresh ones in memory that held doubles of 1.0 (whose words read as
a running state with a buffer index of 0x3ff00000), and ones that a debug run left
running.  Each problem ends with the bits of its solo solve."""
import numpy as np
import pytest

from test_gpu_loop_forms import sized
from test_gpu_parity import P  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def recycle(torch):
    """Blocks of the sizes a handle allocates, full of 1.0, back to the driver."""
    ones = [torch.ones(k, dtype=torch.float64, device="cuda") for k in [64] * 64 + [4096] * 64 + [1 << 18] * 64]
    torch.cuda.synchronize()
    del ones
    torch.cuda.empty_cache()


@pytest.mark.parametrize("first", ["fresh", "debug"])
@pytest.mark.parametrize("precision", [64, 32])
def test_graph_waits_for_the_first_setup(P, precision, first):
    import torch
    insts = [sized(n, 100) for n in (300, 500, 700, 900, 1100, 1300, 20000, 30000)]

    def make(inst):
        h = P.create_from_instance(inst, precision=precision)
        P.pdnqp_set_param(h, "persistent", 0)
        P.pdnqp_set_param(h, "iter_budget", 130)
        if first == "debug":
            P.pdnqp_debug_inner(h, [5, 70])
        return h

    want = []
    for inst in insts:
        h = make(inst)
        P.pdnqp_solve(h, 1e-6, 1e-6)
        want.append(P.pdnqp_get(h)[:2])
        h.close()
    for _ in range(5):
        recycle(torch)
        hs = [make(inst) for inst in insts]
        P.pdnqp_solve_batch(hs, 1e-6, 1e-6)
        for h, (x, y) in zip(hs, want):
            got = P.pdnqp_get(h)
            assert np.array_equal(got[0], x) and np.array_equal(got[1], y)
            h.close()
