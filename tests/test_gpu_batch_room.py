"""Batches around the limits of the cluster form: problems that take it only in a
batch whose clusters all find room at once, and the same problems in a batch where
they do not."""
import numpy as np
import pytest

from paper_2609_19557_gb300 import instances as I
from test_gpu_loop_forms import rows_qp, sized
from test_gpu_parity import P  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

# Tiles of 32 columns: 512 are the limit alone, 1,024 in a batch with room.
BETWEEN = {
    "tiles_lo": lambda: sized(512 * 32 + 1, 4000),
    "tiles_hi": lambda: sized(1024 * 32, 4000),
    "dense_row": lambda: rows_qp(6, 17000, [4] * 900 + [1500, 3000], q=1.0),
    "long_columns": lambda: I.clique_qp(3, n=5000, p=0.01),
}


def solve(P, insts, precision, persistent=1, batch=True):
    hs = []
    for inst in insts:
        h = P.create_from_instance(inst, precision=precision)
        P.pdnqp_set_param(h, "iter_budget", 100)
        P.pdnqp_set_param(h, "persistent", persistent)
        hs.append(h)
    if batch:
        P.pdnqp_solve_batch(hs, 1e-6, 1e-6)
    else:
        for h in hs:
            P.pdnqp_solve(h, 1e-6, 1e-6)
    out = [(*P.pdnqp_get(h)[:2], P.pdnqp_get(h)[2]["loop_blocks"]) for h in hs]
    for h in hs:
        h.close()
    return out


def same(a, b):
    return np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("precision", [64, 32])
def test_cluster_form_between_the_limits(P, precision):
    insts = [f() for f in BETWEEN.values()]
    together = solve(P, insts, precision)
    for name, inst, got in zip(BETWEEN, insts, together):
        assert got[2] == 8, name  # one cluster
        assert same(got, solve(P, [inst], precision)[0]), name
        alone = solve(P, [inst], precision, batch=False)[0]
        assert alone[2] != 8, name  # the grid
        if precision == 64:  # 100 iterations in another order of the sums
            assert np.abs(got[0] - alone[0]).max() <= 1e-8 * max(1.0, np.abs(alone[0]).max()), name


@pytest.mark.parametrize("precision", [64, 32])
def test_between_the_limits_without_room(P, precision):
    """24 clusters of smaller problems beside it: more than 152 SMs hold at once."""
    crowd = [sized(600 + k, 100) for k in range(24)]
    inst = BETWEEN["tiles_lo"]()
    got = solve(P, crowd + [inst], precision)
    assert [g[2] for g in got] == [8] * 24 + [0]
    assert same(got[-1], solve(P, [inst], precision, persistent=0, batch=False)[0])
    for k in (0, 23):
        assert same(got[k], solve(P, [crowd[k]], precision, batch=False)[0])


def test_small_problems_need_no_room(P):
    """Problems of one block each leave the clusters their room."""
    crowd = [sized(300 + k, 100) for k in range(24)]
    inst = BETWEEN["tiles_lo"]()
    got = solve(P, crowd + [inst], 32)
    assert [g[2] for g in got] == [1] * 24 + [8]
