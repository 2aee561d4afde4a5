"""Forms of the Lanczos estimate behind gamma: one cooperative launch, a launch per
phase (the setup of an escalation inside a batch), and one run at a time where the
bases of both find no room.  The sums and their order are the same: the same bits."""
import threading

import numpy as np
import pytest

from paper_2609_19557_gb300 import instances as I
from test_gpu_parity import P  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def free(seed, n, m):
    inst = I.small_qp(seed, n=n, m=m, shift=0.92)
    inst["l_x"][:], inst["u_x"][:] = -np.inf, np.inf
    return inst


@pytest.mark.parametrize("persistent", [1, 0])
@pytest.mark.parametrize("fused", [1, 0])
def test_escalations_inside_a_batch(P, fused, persistent):
    """Several FP32 problems of one batch escalate at the same time: from multipliers of
    1e25 the first step of a free variable has a square that overflows FP32, not FP64."""
    insts = [free(k, n, m) for k, (n, m) in enumerate([(300, 120), (1500, 700), (2000, 900)])]
    insts.append(I.small_qp(3, n=700, m=300, shift=0.92))
    hs = []
    for inst in insts:
        h = P.create_from_instance(inst, precision=32)
        for name, v in (("batch_fused", fused), ("persistent", persistent), ("iter_budget", 64)):
            P.pdnqp_set_param(h, name, v)
        if len(hs) < 3:
            P.pdnqp_set_start(h, None, np.full(inst["A"].shape[0], 1e25))
        hs.append(h)
    P.pdnqp_solve_batch(hs, 1e-6, 1e-6, threads=4)
    for k, (h, inst) in enumerate(zip(hs, insts)):
        assert P.pdnqp_get_param(h, "escalated") == (1 if k < 3 else 0)
        h64 = P.create_from_instance(inst, precision=64)
        assert P.pdnqp_get(h)[2]["gamma"] == P.pdnqp_get_param(h64, "gamma")
        h.close()
        h64.close()


def test_handles_created_at_the_same_time(P):
    """Cooperative launches of several threads: each handle as when made alone."""
    insts = [I.large_qp(k, n=60000, m=30000, replica_n=1000) for k in range(6)]

    def gamma(inst):
        h = P.create_from_instance(inst)
        g = P.pdnqp_get_param(h, "gamma")
        h.close()
        return g

    alone, got = [gamma(i) for i in insts], [[] for _ in insts]
    threads = [threading.Thread(target=lambda k=k: got[k].extend(gamma(insts[k]) for _ in range(4))) for k in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert got == [[g] * 4 for g in alone]


def test_create_where_two_bases_find_no_room(P):
    """Free memory for one basis (8 (steps + 1) n bytes) beside the handle, not for two."""
    import torch
    n, steps = 1000000, 64
    inst = I.large_qp(1, n=n, m=n // 2, replica_n=1000)
    torch.zeros(1, device="cuda")
    torch.cuda.empty_cache()
    free0 = torch.cuda.mem_get_info()[0]
    h = P.create_from_instance(inst, precision=32)
    held, gamma = free0 - torch.cuda.mem_get_info()[0], P.pdnqp_get_param(h, "gamma")
    h.close()
    # The handle holds at least its FP32 vectors and matrices (23 n + 36 m floats, 13 M values) besides what
    # is there when the basis is taken, so two bases of 1,056 n bytes do not fit in this.
    room = held + 8 * (steps + 2) * n + (64 << 20)
    fill = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
    try:
        h = P.create_from_instance(inst, precision=32)
        assert P.pdnqp_get_param(h, "gamma") == gamma
        h.close()
    finally:
        del fill
        torch.cuda.empty_cache()
