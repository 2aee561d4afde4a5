"""Forms of the inner loop by size and row lengths: tiles of 32 short rows with
longer rows as items of their own, tiles of 8 long rows, one block, one cluster,
the grid with and without the first items kept in shared memory, and a batch
whose problems run in different forms.  FP64: per-step parity with the oracle;
FP32: the stated error of the bulk form."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2609_19557_gb300 import instances as I
from test_gpu_parity import P, compare_snaps, rel_err  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

# Either side of every boundary of the row sums: 8 entries a round of a tile, 32
# (an item of its own), 256 a round of a whole warp, 512 (a warp alone), 1024.
EDGES = [0, 1, 7, 8, 9, 31, 32, 33, 63, 64, 65, 255, 256, 257, 511, 512, 513, 1023, 1024]


def rows_qp(seed, n, lengths, diag=False, q=2.0):
    """small_qp's Q (diag: a diagonal with two eigenvalues) with rows of A of the given lengths."""
    rng = np.random.default_rng(seed)
    base = I.small_qp(seed, n=n, m=max(1, len(lengths)), a_per_row=min(n, 4), q_offdiag_per_row=q)
    Q = sp.diags(np.where(np.arange(n) % 3 == 0, -1.0, 2.0)).tocsr() if diag else base["Q"]
    cols = [np.sort(rng.choice(n, size=k, replace=False)) for k in lengths]
    ptr = np.concatenate([[0], np.cumsum(lengths)]).astype(int)
    val = np.concatenate([rng.standard_normal(k) / np.sqrt(max(k, 1)) for k in lengths])
    A = sp.csr_matrix((val, np.concatenate(cols), ptr), shape=(len(lengths), n))
    x0 = base["x0"]
    ax = A @ x0
    lo, hi = ax - rng.uniform(0.1, 1.0, len(lengths)), ax + rng.uniform(0.1, 1.0, len(lengths))
    eq = (rng.random(len(lengths)) < 0.2) & (np.asarray(lengths) > 0)
    hi[eq] = lo[eq] = ax[eq]
    return I._pack(Q, base["c"], A, lo, hi, base["l_x"], base["u_x"], x0, workload="rows")


def sized(n, m, q=1.0):
    return I.small_qp(7, n=n, m=m, q_offdiag_per_row=q)


CASES = {
    # Cluster: short rows with the edges among them; grid: tiles of 8 for rows and columns.
    "edges": lambda: rows_qp(1, 2000, [3] * 400 + EDGES),
    "long": lambda: rows_qp(2, 2000, (EDGES * 37)[:700]),
    "diag": lambda: rows_qp(3, 1025, [4] * 33, diag=True),
    "n2": lambda: rows_qp(4, 2, [1, 2]),
    "n33": lambda: rows_qp(5, 33, [2] * 31),
    # One block up to 16 tiles, then the cluster up to 512, then the grid.
    "block": lambda: sized(512, 200),
    "cluster_lo": lambda: sized(513, 200),
    "cluster_hi": lambda: sized(16384, 8192),
    "grid": lambda: sized(16385, 8192),
    # 2 x 152 x 16 items: the first items of the warps are kept, and one more.
    "kept": lambda: sized(155648, 5000),
    "not_kept": lambda: sized(155649, 5000),
}


@pytest.fixture(scope="module")
def refs(oracle):
    memo = {}

    def get(name, ck):
        if name not in memo:
            inst = CASES[name]()
            memo[name] = (inst, *oracle.debug_inner(inst, ck))
        return memo[name]
    return get


def steps(name):
    return [1, 2, 5, 20] if name in ("kept", "not_kept") else [1, 2, 5, 20, 64, 65, 128]


@pytest.mark.parametrize("name", list(CASES))
def test_forms_per_step_parity(P, refs, name):
    inst, ref, info = refs(name, steps(name))
    h = P.create_from_instance(inst)
    gpu = P.pdnqp_debug_inner(h, steps(name))
    assert abs(P.pdnqp_get_param(h, "gamma") - info["gamma"]) <= 1e-10 * info["gamma"]
    compare_snaps(gpu, ref)
    h.close()


@pytest.mark.parametrize("name", ["edges", "long", "cluster_hi", "grid", "kept", "not_kept"])
def test_forms_fp32(P, refs, name):
    inst, ref, _ = refs(name, steps(name))
    h = P.create_from_instance(inst, precision=P.PDNQP_FP32_BULK)
    gpu = P.pdnqp_debug_inner(h, steps(name)[:4])
    assert len(gpu) == 4
    for s, r in zip(gpu, ref):
        assert s["t_total"] == r["t_total"]
        assert max(rel_err(s[k], r[k]) for k in ("w", "y", "wbar", "ybar")) < 1e-4, s["t_total"]
    h.close()


@pytest.mark.parametrize("precision", [64, 32])
def test_batch_of_both_forms(P, precision):
    """Problems in the cluster form and in the shared graph of one batch: each ends
    with the bits of its own solo solve in that form."""
    insts = [sized(300, 100), sized(1500, 700), sized(33000, 8000), rows_qp(1, 2000, [3] * 400 + EDGES),
             sized(36000, 9000)]

    def make(inst, persistent):
        h = P.create_from_instance(inst, precision=precision)
        P.pdnqp_set_param(h, "k_out", 4)
        P.pdnqp_set_param(h, "persistent", persistent)
        return h

    def result(h):
        x, y, r = P.pdnqp_get(h)
        h.close()
        return x, y, r["outer_iters"], r["inner_iters"]

    seq = []
    for inst in insts:
        h = make(inst, 1 if inst["Q"].shape[0] <= 16384 else 0)
        P.pdnqp_solve(h, 1e-5, 1e-5)
        seq.append(result(h))
    hs = [make(inst, 1) for inst in insts]
    P.pdnqp_solve_batch(hs, 1e-5, 1e-5, threads=4)
    for h, want in zip(hs, seq):
        got = result(h)
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
        assert got[2:] == want[2:]
