"""External KKT test on device data where its warp tiles can go wrong: sizes
around a tile, matrices with long and dense rows, no constraint rows, empty
rows, infinite bounds; against the oracle's checker."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2609_19557_gb300 import instances as I
from test_gpu_parity import P  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _random(n, m, q_len, a_len, seed):
    """Random symmetric Q and A whose row lengths run from 0 to the given ones."""
    rng = np.random.default_rng([seed, n, m])

    def mat(rows, cols, longest):
        lens = np.minimum(rng.integers(0, longest + 1, size=rows), cols)
        lens[rows // 2:rows // 2 + 1] = min(longest, cols)
        ci = np.concatenate([np.sort(rng.choice(cols, size=k, replace=False)) for k in lens] + [np.zeros(0, int)])
        return sp.csr_matrix((rng.normal(size=ci.size), ci, np.concatenate([[0], np.cumsum(lens)])), shape=(rows, cols))

    U = sp.triu(mat(n, n, q_len)).tocsr()
    Q = (U + sp.triu(U, 1).T).tocsr()
    A = mat(m, n, a_len)
    lo, hi = rng.uniform(-1, 0, m), rng.uniform(0, 1, m)
    lo[::3], hi[1::3] = -np.inf, np.inf
    lx, ux = rng.uniform(-1, 0, n), rng.uniform(0, 1, n)
    lx[::4], ux[1::4] = -np.inf, np.inf
    return dict(Q=Q, c=rng.normal(size=n), A=A, l_c=lo, u_c=hi, l_x=lx, u_x=ux), rng


@pytest.mark.parametrize("n,m,q_len,a_len", [(1, 1, 1, 1), (31, 5, 4, 3), (32, 33, 9, 8), (33, 31, 32, 33), (257, 64, 64, 40),
                                             (1000, 3, 20, 1000), (1025, 2000, 40, 300), (400, 7, 400, 400)])
def test_kkt_tiles_match_oracle(P, oracle, n, m, q_len, a_len):
    import torch
    inst, rng = _random(n, m, q_len, a_len, 3)
    prob = P.DeviceProblem(inst)
    x, y = rng.normal(size=n), rng.normal(size=m)
    xd, yd = torch.as_tensor(x, device="cuda"), torch.as_tensor(y, device="cuda")
    ref = np.array(oracle.kkt_check(inst, x, y))
    for fn in (P.pdnqp_kkt_residuals, P.pdnqp_kkt_residuals_noalloc):
        out = torch.full((4,), float("nan"), device="cuda", dtype=torch.float64)
        fn(prob, xd, yd, out)
        torch.cuda.synchronize()
        # Sums of at most 1000 terms of size ~1: 1000 * 2^-53 * a few.
        assert np.allclose(out.cpu().numpy(), ref, rtol=1e-12, atol=1e-12), (out.cpu().numpy(), ref)


def test_kkt_without_rows(P, oracle):
    """m = 0 (A, At, l_c and u_c unused): the same as one empty free row."""
    import ctypes
    import torch
    inst, rng = _random(100, 1, 12, 0, 4)
    inst["l_c"][:], inst["u_c"][:] = -np.inf, np.inf
    prob = P.DeviceProblem(inst)
    x = rng.normal(size=100)
    xd = torch.as_tensor(x, device="cuda")
    ref = np.array(oracle.kkt_check(inst, x, np.zeros(1)))
    s = P.pdnqp_device_problem.from_buffer_copy(prob.s)
    s.A, s.At, s.l_c, s.u_c = P.pdnqp_device_csr(), P.pdnqp_device_csr(), None, None
    out = torch.full((4,), float("nan"), device="cuda", dtype=torch.float64)
    assert P.load().pdnqp_kkt_residuals(ctypes.byref(s), xd.data_ptr(), None, out.data_ptr(), None) == 0
    assert np.allclose(out.cpu().numpy(), ref, rtol=1e-12, atol=1e-12)


def test_kkt_calls_on_two_streams(P, oracle):
    """Calls that overlap on two streams do not disturb each other."""
    import torch
    inst = I.mid_qp(2, n=20000, m=10000, replica_n=1000)
    prob = P.DeviceProblem(inst)
    rng = np.random.default_rng(5)
    pts = [(torch.as_tensor(rng.normal(scale=0.5 + k, size=20000), device="cuda"),
            torch.as_tensor(rng.normal(size=10000), device="cuda")) for k in range(2)]
    ref = []
    for x, y in pts:
        o = torch.zeros(4, device="cuda", dtype=torch.float64)
        P.pdnqp_kkt_residuals(prob, x, y, o)
        ref.append(o.cpu().numpy())
    streams = [torch.cuda.Stream() for _ in pts]
    outs = [torch.zeros((50, 4), device="cuda", dtype=torch.float64) for _ in pts]
    torch.cuda.synchronize()
    for i in range(50):
        for k, (x, y) in enumerate(pts):
            P.pdnqp_kkt_residuals_noalloc(prob, x, y, outs[k][i], stream=streams[k].cuda_stream)
    torch.cuda.synchronize()
    for k in range(2):
        assert np.array_equal(outs[k].cpu().numpy(), np.tile(ref[k], (50, 1)))
