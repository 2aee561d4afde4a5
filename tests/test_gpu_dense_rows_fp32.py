"""Dense coupling rows in the FP32-bulk form: the stated error of its iterates against
the FP64 oracle, in the persistent forms (one block or cluster, grid) and the graph.
The SVM's one multiplier is left out: its row is a sum of 3,000 terms +-x_i that nearly
cancel, and rounding x to FP32 alone moves it by some 1e-3 of the multiplier."""
import numpy as np
import pytest

from paper_2609_19557_gb300 import instances as I
from test_gpu_dense_rows import many_dense_rows
from test_gpu_loop_forms import rows_qp
from test_gpu_parity import P, rel_err  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

CK = [1, 2, 5, 20]
CASES = {
    "svm": lambda: I.svm_qp(101, n_target=3000),
    "softlabel": lambda: I.softlabel_qp(104, n_target=12000),
    "many": many_dense_rows,
    "grid": lambda: rows_qp(6, 17000, [4] * 900 + [1500, 3000], q=1.0),
}


@pytest.mark.parametrize("case", list(CASES))
def test_dense_rows_fp32_error(P, oracle, case):
    inst = CASES[case]()
    assert np.diff(inst["A"].indptr).max() > 1024  # the split is exercised
    ref, _ = oracle.debug_inner(inst, CK)
    for persistent in (1, 0):
        h = P.create_from_instance(inst, precision=P.PDNQP_FP32_BULK)
        P.pdnqp_set_param(h, "persistent", persistent)
        gpu = P.pdnqp_debug_inner(h, CK)
        h.close()
        assert len(gpu) == len(CK)
        for s, r in zip(gpu, ref):
            assert s["t_total"] == r["t_total"]
            keys = ("w", "wbar") if case == "svm" else ("w", "y", "wbar", "ybar")
            assert max(rel_err(s[k], r[k]) for k in keys) < 1e-4, (persistent, s["t_total"])
