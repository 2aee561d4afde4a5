"""Performance cases of the PDNQP solver: what a user of the library has it do.

Six kinds of call, all through the public binding of the C ABI:

    solve   pdnqp_solve + pdnqp_get on a handle that the program keeps, with a
            budget of accepted inner iterations (as the benchmark's step);
    batch   pdnqp_solve_batch over problems of uneven sizes, then pdnqp_get of each;
    create  the whole way from host CSR data: pdnqp_create, solve, get, destroy;
    kkt     the external KKT test on device data (allocating entry point);
    kkt_na  the same test without allocation, asynchronous on the stream;
    train   one full-batch training step of the controller network (forward,
            weighted squared error, backward, Adam).

Results of the FP32-bulk form are returned in float32, the type its iterates
are held in; those of the FP64 form in float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_19557_gb300 import instances as I
from paper_2609_19557_gb300 import mlp_data as D
from paper_2609_19557_gb300 import pdnqp as P

EPS = 1e-6  # tolerance of every solve (a Motzkin-Straus point of n = 10,000 has entries of 1e-4)
SHIFT = 0.92  # diagonal shift of the small generator: about 30 % negative eigenvalues at its density
BATCH_MEDIAN, BATCH_SIGMA = 4000.0, 0.8  # size distribution of the batched set
CLIQUE_P = 0.01
LR = 3e-3


def listed():
    return [
        # The smallest workload (n = 200), plain form: nothing but latency.
        dict(name="small_fp64", kind="solve", gen="small", n=200, m=100, precision=64, budget=512),
        # A few thousand entries, odd sizes, bulk form: one or two blocks per pass.
        dict(name="ragged_fp32", kind="solve", gen="small", n=1201, m=603, precision=32, budget=512),
        # The mid-size family (power-law rows, free variables, equality rows) in both forms.
        dict(name="mid_fp64", kind="solve", gen="mid", n=50000, m=25000, precision=64, budget=512),
        dict(name="mid_fp32", kind="solve", gen="mid", n=50000, m=25000, precision=32, budget=512),
        # The headline workload (1M variables) in both forms.
        dict(name="large_fp32", kind="solve", gen="large", n=1000000, m=500000, precision=32, budget=512),
        dict(name="large_fp64", kind="solve", gen="large", n=1000000, m=500000, precision=64, budget=256),
        # Motzkin-Straus problem: long rows of Q (about 100 entries), one dense constraint row.
        dict(name="clique_fp64", kind="solve", gen="clique", n=10007, m=1, precision=64, budget=128),
        # The batched form: 24 problems of uneven sizes, half of them Motzkin-Straus.
        dict(name="batch_fp32", kind="batch", count=24, precision=32, budget=192),
        # From host data to the result, as a program that solves each problem once.
        dict(name="create_fp32", kind="create", gen="large", n=300001, m=150007, precision=32, budget=128),
        # Checking a point of the headline workload and of the mid-size family on the GPU.
        dict(name="kkt_large", kind="kkt", gen="large", n=1000000, m=500000),
        dict(name="kkt_mid", kind="kkt_na", gen="mid", n=50000, m=25000),
        # One epoch of the controller's training on the transitions of 320 trajectories.
        dict(name="train", kind="train", batch=231184),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "batch", "create", "kkt", "kkt_na", "train"])
    if kind == "train":
        return dict(kind=kind, batch=_log(rng, 300, 231184))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(6, 24), precision=rng.choice([32, 32, 64]), budget=rng.randint(96, 192))
    gen = rng.choice(["small", "mid", "large", "clique"])
    lo, hi = {"small": (64, 20000), "mid": (2000, 100000), "large": (10000, 1000000), "clique": (200, 12000)}[gen]
    if kind == "create":
        hi = min(hi, 300001)
    n = _log(rng, lo, hi)
    m = 1 if gen == "clique" else int(n * rng.uniform(0.3, 0.5))
    c = dict(kind=kind, gen=gen, n=n, m=m)
    if kind in ("solve", "create"):
        # Motzkin-Straus alone in the plain form only (in the bulk form its one
        # multiplier holds three digits); the batches have them in both.
        c["precision"] = 64 if gen == "clique" else rng.choice([32, 64])
        big = c["precision"] == 64 and n > 500000
        c["budget"] = rng.randint(64, 128) if kind == "create" or gen == "clique" else rng.randint(128, 256 if big else 512)
    return c


def _instance(gen, n, m, seed):
    if gen == "small":
        return I.small_qp(seed, n=n, m=m, shift=SHIFT)
    if gen == "mid":
        return I.mid_qp(seed, n=n, m=m, replica_n=1000)
    if gen == "large":
        return I.large_qp(seed, n=n, m=m, replica_n=1000)
    return I.clique_qp(seed, n=n, p=CLIQUE_P)


def _batch_sizes(count):
    """Quantiles of the batched set's log-normal sizes (clipped below at 1000), in a mixed order."""
    z = torch.special.ndtri((torch.arange(count, dtype=torch.float64) + 0.5) / count).numpy()
    n = np.clip(np.exp(np.log(BATCH_MEDIAN) + BATCH_SIGMA * z), 1000, 100_000).astype(int)
    return [int(n[(7 * k) % count] if math.gcd(7, count) == 1 else n[k]) for k in range(count)]


def _point(inst, seed):
    """A point near the box, some entries slightly outside, and multipliers."""
    rng = np.random.default_rng([seed, 17])
    lx = np.where(np.isfinite(inst["l_x"]), inst["l_x"], -2.0)
    ux = np.where(np.isfinite(inst["u_x"]), inst["u_x"], 2.0)
    return rng.uniform(lx - 0.1, ux + 0.1), rng.normal(size=inst["A"].shape[0])


def _train_inputs(batch, seed):
    """Standardised features, targets, sample weights and an optimizer in mid-training."""
    rng = np.random.default_rng([seed, 23])
    w = D.init_weights(seed)
    w[-D.N_OUT:] = [0.1, -0.3]
    x = D.features(seed + 1, batch)
    t = rng.normal(0.0, 0.5, (batch, D.N_OUT)).astype(np.float32)
    wt = np.exp(np.clip(rng.normal(size=batch), -3.0, 3.0)).astype(np.float32)
    m = (1e-3 * rng.normal(size=w.size)).astype(np.float32)
    v = (1e-5 * rng.uniform(0.5, 2.0, w.size)).astype(np.float32)
    return w, x, t, wt, m, v


def _handle(case, inst):
    h = P.create_from_instance(inst, precision=case["precision"])
    P.pdnqp_set_param(h, "iter_budget", case["budget"])
    return h


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "train":
        w, x, t, wt, m, v = (torch.as_tensor(a).cuda() for a in _train_inputs(case["batch"], seed))
        B = case["batch"]
        s.update(w=w, x=x, t=t, wt=wt, m=m, v=v, wb=torch.zeros(w.numel(), dtype=torch.int16, device="cuda"),
                 y=torch.zeros((B, 2), device="cuda"), cache=torch.zeros((B, 128), device="cuda"),
                 dy=torch.zeros((B, 2), device="cuda"), loss=torch.zeros(1, device="cuda"), grad=torch.zeros_like(w),
                 scratch=torch.zeros(((B + 15) // 16) * w.numel(), device="cuda"), step=200)
        P.mlp_to_bf16(w, s["wb"])
    elif kind == "batch":
        s["handles"] = []
        for k, n in enumerate(_batch_sizes(case["count"])):
            gen = "small" if k % 2 == 0 else "clique"
            s["handles"].append(_handle(case, _instance(gen, n, n // 2, 1000 * seed + k)))
    elif kind in ("kkt", "kkt_na"):
        inst = _instance(case["gen"], case["n"], case["m"], seed)
        x, y = _point(inst, seed)
        s.update(prob=P.DeviceProblem(inst), x=torch.as_tensor(x).cuda(), y=torch.as_tensor(y).cuda(),
                 out=torch.zeros(4, dtype=torch.float64, device="cuda"))
    else:
        inst = _instance(case["gen"], case["n"], case["m"], seed)
        if kind == "create":
            s["inst"] = inst
        else:
            s["handle"] = _handle(case, inst)
    return s


def _result(case, h):
    """x, y and the reported residuals and objective, in the form's type."""
    dt = np.float64 if case["precision"] == 64 else np.float32
    x, y, r = P.pdnqp_get(h)
    return x.astype(dt), y.astype(dt), np.array([r[k] for k in ("r_p", "r_d", "s_p", "s_d", "obj")], dtype=dt)


def run(state):
    case, s = state["case"], state
    kind = case["kind"]
    if kind == "train":
        s["step"] += 1
        P.mlp_forward(s["wb"], s["x"], s["y"], s["cache"])
        P.mlp_wmse(s["y"], s["t"], s["wt"], s["dy"], s["loss"])
        P.mlp_backward(s["wb"], s["x"], s["cache"], s["dy"], s["grad"], s["scratch"])
        P.mlp_adam(s["w"], s["wb"], s["grad"], s["m"], s["v"], s["step"], lr=LR)
        return dict({k: s[k] for k in ("y", "cache", "dy", "loss", "grad", "w", "m", "v")},
                    wb=s["wb"].view(torch.bfloat16))
    if kind == "batch":
        status = P.pdnqp_solve_batch(s["handles"], EPS, EPS)
        got = [_result(case, h) for h in s["handles"]]
        return dict(status=np.array(status), x=np.concatenate([g[0] for g in got]),
                    y=np.concatenate([g[1] for g in got]), res=np.stack([g[2] for g in got]))
    if kind == "kkt":
        P.pdnqp_kkt_residuals(s["prob"], s["x"], s["y"], s["out"], torch.cuda.current_stream().cuda_stream)
        return s["out"]
    if kind == "kkt_na":
        P.pdnqp_kkt_residuals_noalloc(s["prob"], s["x"], s["y"], s["out"], torch.cuda.current_stream().cuda_stream)
        return s["out"]
    h = _handle(case, s["inst"]) if kind == "create" else s["handle"]
    status = P.pdnqp_solve(h, EPS, EPS)
    x, y, res = _result(case, h)
    out = dict(status=status, x=x, y=y, res=res)
    if kind == "create":
        out["gamma"] = np.array([P.pdnqp_get_param(h, "gamma")])
        h.close()
    return out


def _sizes(gen, n, m):
    """Expected (nnz of Q with its diagonal, nnz of A)."""
    if gen == "small":
        return 5 * n, 4 * m
    if gen == "mid":
        return 9 * n, 6 * m
    if gen == "large":
        return 5 * n, 8 * m
    return CLIQUE_P * n * (n - 1) + n, n


def _solve_work(gen, n, m, v, budget):
    """Per accepted inner iteration, every array once: the three matrices with
    their row pointers, 14 touches of an n-vector, 20 of an m-vector (its s,
    r, y, averages, products, steps and bounds)."""
    q, a = _sizes(gen, n, m)
    per = (v + 4) * (q + 2 * a) + 4 * (2 * n + m) + v * (14 * n + 20 * m)
    return budget * per, budget * (2 * (q + 2 * a) + 20 * n + 40 * m)


def work(case):
    kind = case["kind"]
    if kind == "train":
        B, p = case["batch"], D.N_PARAMS
        per = 4 * (D.N_IN + 2 + 1 + 2 + 2 + 2 * D.N_HID)
        mul = D.N_IN * D.N_HID + D.N_HID * D.N_HID + D.N_HID * D.N_OUT
        return {"bytes": B * per + 4 * 8 * p, "flops": B * 2.0 * (2 * mul + D.N_HID * D.N_HID + D.N_HID * D.N_OUT)}
    if kind in ("kkt", "kkt_na"):
        q, a = _sizes(case["gen"], case["n"], case["m"])
        n, m = case["n"], case["m"]
        return {"bytes": 12 * (q + 2 * a) + 4 * (2 * n + m) + 8 * (4 * n + 3 * m), "flops": 2 * (q + 2 * a) + 10 * n}
    v = case["precision"] // 8
    if kind == "batch":
        got = [_solve_work("small" if k % 2 == 0 else "clique", n, n // 2 if k % 2 == 0 else 1, v, case["budget"])
               for k, n in enumerate(_batch_sizes(case["count"]))]
        return {"bytes": sum(g[0] for g in got), "flops": sum(g[1] for g in got)}
    b, f = _solve_work(case["gen"], case["n"], case["m"], v, case["budget"])
    if kind == "create":  # plus the host data in
        q, a = _sizes(case["gen"], case["n"], case["m"])
        b += 12 * (q + a) + 4 * (case["n"] + case["m"]) + 8 * (3 * case["n"] + 2 * case["m"])
    return {"bytes": b, "flops": f}


def _csr_mul(M, v):
    row = np.repeat(np.arange(M.shape[0]), np.diff(M.indptr))
    return np.bincount(row, weights=M.data * v[M.indices], minlength=M.shape[0])


def exact(case, seed):
    """In 64 bits: the KKT residuals and the training step.  A solve is some
    hundred dependent iterations behind a Lanczos estimate and row and column
    equilibration, with restarts and penalties decided on the way; it has no
    value short of the whole method."""
    if case["kind"] in ("kkt", "kkt_na"):
        inst = _instance(case["gen"], case["n"], case["m"], seed)
        x, y = _point(inst, seed)
        Q, A = inst["Q"], inst["A"]
        qx, ax = _csr_mul(Q, x), _csr_mul(A, x)
        row = np.repeat(np.arange(A.shape[0]), np.diff(A.indptr))
        aty = np.bincount(A.indices, weights=A.data * y[row], minlength=A.shape[1])
        lc, uc, lx, ux, c = (inst[k] for k in ("l_c", "u_c", "l_x", "u_x", "c"))
        rp = max(np.maximum(np.maximum(lc - ax, ax - uc), 0.0).max(), np.maximum(np.maximum(lx - x, x - ux), 0.0).max())
        rd = np.abs(x - np.clip(x - (qx + c + aty), lx, ux)).max()
        fin = [np.abs(b[np.isfinite(b)]).max(initial=0.0) for b in (lc, uc)]
        sp_ = max(1.0, np.abs(ax).max(), *fin)
        sd = max(1.0, np.abs(qx).max(), np.abs(c).max(), np.abs(aty).max())
        return np.array([rp, rd, sp_, sd])
    if case["kind"] != "train":
        return None
    w, x, t, wt, m, v = (torch.as_tensor(a).cuda().double() for a in _train_inputs(case["batch"], seed))
    q = w.float().bfloat16().double()
    cut = np.cumsum([D.N_HID * D.N_IN, D.N_HID, D.N_HID * D.N_HID, D.N_HID, D.N_OUT * D.N_HID])
    W1, b1, W2, b2, W3, b3 = (p.requires_grad_() for p in torch.tensor_split(q, [int(k) for k in cut]))
    z1 = x @ W1.view(D.N_HID, D.N_IN).T + b1
    z2 = torch.nn.functional.gelu(z1) @ W2.view(D.N_HID, D.N_HID).T + b2
    y = torch.nn.functional.gelu(z2) @ W3.view(D.N_OUT, D.N_HID).T + b3
    y.retain_grad()
    loss = (wt[:, None] * (y - t) ** 2).sum() / wt.sum()
    loss.backward()
    g = torch.cat([p.grad for p in (W1, b1, W2, b2, W3, b3)])
    b1_, b2_, eps, step = 0.9, 0.999, 1e-8, 201
    m, v = b1_ * m + (1 - b1_) * g, b2_ * v + (1 - b2_) * g * g
    w = w - LR * (m / (1 - b1_ ** step)) / ((v / (1 - b2_ ** step)).sqrt() + eps)
    return dict(y=y.detach(), cache=torch.cat([z1, z2], 1).detach(), dy=y.grad, loss=loss.detach().view(1), grad=g, w=w,
                m=m, v=v, wb=w)
