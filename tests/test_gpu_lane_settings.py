"""Lane settings 4 and 8 of the graph form are one form: the same launches and
the same bits, also mixed in a batch."""
import numpy as np
import pytest

from test_gpu_loop_forms import sized
from test_gpu_parity import P  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def test_batch_of_lane_settings_4_and_8(P):
    out = []
    for lanes in ((8, 8, 8), (4, 8, 4)):
        hs = [P.create_from_instance(sized(n, 100)) for n in (300, 700, 900)]
        for h, g in zip(hs, lanes):
            for name, v in (("persistent", 0), ("iter_budget", 64), ("g_rows", g), ("g_cols", g)):
                P.pdnqp_set_param(h, name, v)
        P.pdnqp_solve_batch(hs, 1e-6, 1e-6)
        n = {k: P.pdnqp_get_param(hs[0], "batch_" + k + "_launches") for k in ("graph", "kernel")}
        out.append((n["kernel"] / n["graph"], [P.pdnqp_get(h)[0] for h in hs]))
        for h in hs:
            h.close()
    assert all(np.array_equal(a, b) for a, b in zip(out[0][1], out[1][1]))
    assert abs(out[0][0] - out[1][0]) < 8.0  # kernels a graph launch: one launch a phase for all three (16 trials)
