"""The work that programs using this library have it do, as measurable cases.

Each case is one call (or one forward + backward) through the package's public
functions on synthetic data of a stated size.  Listed cases:

* ``direct``      -- Q and R of a tall matrix: the library's main call, from
  the smallest problems (launch latency) to the sizes of the benchmark
  configurations (8,000,000 x 25 binary64, 50,000,000 x 50 binary32), with the
  binding's default arithmetic ("native") and the benchmark's ("auto").
* ``direct_host`` -- the same from and to page-locked host memory, copies
  overlapped (a matrix that a data loader has produced).
* ``svd``         -- U, S, V of a tall matrix (dimension reduction;
  20,000,000 x 100 binary32).
* ``svd_values``  -- S and V without U; ``r``: R alone (least squares,
  preconditioners).
* ``grad``        -- QRFunction forward and backward, as inside a training step
  (4,000,000 x 64, both types).
* ``cholqr`` and ``indirect`` -- the two comparators with one step of
  refinement, as in a stability comparison.

``draw`` gives further cases of the same calls over the ranges in between.
"""
from __future__ import annotations

import math

import torch

import paper_1301_1071_gb300 as tsqr

DTYPES = {"f64": torch.float64, "f32": torch.float32}
OPS = {"direct": tsqr.OP_DIRECT, "svd": tsqr.OP_SVD, "r": tsqr.OP_R, "svd_values": tsqr.OP_SVD_VALUES,
       "cholqr": tsqr.OP_CHOLQR, "indirect": tsqr.OP_INDIRECT, "direct_host": tsqr.OP_DIRECT_HOST}


def _case(op, dtype, m, n, prec="native", data="gauss", block_rows=0, name=None):
    c = {"op": op, "dtype": dtype, "m": m, "n": n, "prec": prec, "data": data, "block_rows": block_rows}
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # a small regression fit or one layer's gradient check: latency of the whole launch chain
        _case("direct", "f64", 2_000, 8, name="direct_f64_2kx8"),
        # the small benchmark configuration: row blocks of 1,000 rows
        _case("direct", "f64", 100_000, 10, prec="auto", block_rows=1000, name="direct_f64_100kx10"),
        # an ordinary call with the binding's defaults, a ragged row count
        _case("direct", "f64", 1_000_003, 25, data="cond", name="direct_f64_1Mx25"),
        # the headline benchmark shape in the benchmark's arithmetic
        _case("direct", "f64", 8_000_000, 25, prec="auto", data="cond", name="direct_f64_8Mx25_auto"),
        # the mixed-precision configuration: badly scaled columns, 10 GB of binary32
        _case("direct", "f32", 50_000_000, 50, prec="auto", data="colscale", name="direct_f32_50Mx50_auto"),
        # host matrix in, host matrices out
        _case("direct_host", "f64", 8_000_000, 25, prec="auto", data="cond", name="host_f64_8Mx25_auto"),
        # dimension reduction of a wide-for-tall matrix
        _case("svd", "f32", 20_000_000, 100, prec="auto", data="spectrum", name="svd_f32_20Mx100_auto"),
        # singular values and right vectors alone
        _case("svd_values", "f64", 8_000_000, 25, data="spectrum", name="svdvals_f64_8Mx25"),
        # QR inside a differentiated program, both types
        _case("grad", "f64", 4_000_000, 64, name="grad_f64_4Mx64"),
        _case("grad", "f32", 4_000_000, 64, name="grad_f32_4Mx64"),
        # the comparators with one refinement step
        _case("cholqr", "f64", 8_000_000, 25, data="cond", name="cholqr_f64_8Mx25"),
        _case("indirect", "f64", 1_000_000, 50, data="cond", name="indirect_f64_1Mx50"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["direct", "direct", "direct", "svd", "r", "svd_values", "grad", "cholqr", "indirect",
                     "direct_host"])
    dtype = rng.choice(["f64", "f32"])
    n = _log_int(rng, 4, 100)
    # at most 2e8 (binary64) or 1e9 (binary32) entries and the work of the largest listed case of the type
    cap = min(2e8 / n, 1e10 / (n * n)) if dtype == "f64" else min(1e9 / n, 1e11 / (n * n))
    if op == "direct_host":
        cap = min(cap, 1e8 / n)
    m = _log_int(rng, 2_000, int(max(cap, 4_000)))
    prec = rng.choice(["native", "auto"]) if op in ("direct", "svd", "direct_host") else "native"
    data = "spectrum" if op in ("svd", "svd_values") else rng.choice(["gauss", "colscale", "cond"])
    if data == "cond" and dtype == "f32":
        data = "colscale"
    block_rows = 0
    if op == "direct" and rng.random() < 0.25:
        block_rows = max(n, rng.choice([1000, 1024, 4096]))
        block_rows = min(block_rows, m)
    return _case(op, dtype, m, n, prec, data, block_rows)


def _generator(seed, device="cuda"):
    return torch.Generator(device=device).manual_seed(int(seed))


def _matrix(case, seed):
    """The tall matrix of a case, on the GPU: N(0, 1) entries; the same with
    column factors log-spaced over 1 .. 1e-4; G diag(sigma) V^T with sigma
    log-spaced over 1 .. 1e-4 (condition number 1e4); or the same with sigma
    linear from 1 to 1/n (well separated singular values)."""
    m, n, dt = case["m"], case["n"], DTYPES[case["dtype"]]
    g = _generator(seed)
    A = torch.randn(m, n, dtype=dt, device="cuda", generator=g)
    if case["data"] == "gauss":
        return A
    if case["data"] == "colscale":
        A *= torch.logspace(0, -4, n, dtype=torch.float64, device="cuda").to(dt) if n > 1 else 1.0
        return A
    if case["data"] == "cond":
        sigma = torch.logspace(0, -4, n, dtype=torch.float64, device="cuda")
    else:
        sigma = torch.arange(n, 0, -1, dtype=torch.float64, device="cuda") / n
    V, _ = torch.linalg.qr(torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g))
    M = (sigma[:, None] * V.T / math.sqrt(m)).to(dt)
    for r0 in range(0, m, 1 << 22):
        A[r0:r0 + (1 << 22)] = A[r0:r0 + (1 << 22)] @ M
    return A


def _cotangents(case, seed):
    """Gradients of a loss with respect to Q and R (grad cases)."""
    m, n, dt = case["m"], case["n"], DTYPES[case["dtype"]]
    g = _generator(seed + 1_000_003)
    return (torch.randn(m, n, dtype=dt, device="cuda", generator=g),
            torch.randn(n, n, dtype=dt, device="cuda", generator=g))


def prepare(case, seed):
    m, n, dt, op = case["m"], case["n"], DTYPES[case["dtype"]], case["op"]
    st = {"case": case, "A": _matrix(case, seed)}
    if op == "grad":
        st["A"].requires_grad_()
        st["gQ"], st["gR"] = _cotangents(case, seed)
        return st
    # a program that calls repeatedly keeps its workspace and output buffers
    prec = case["prec"] if op in ("direct", "svd", "direct_host") else "native"
    need = tsqr.workspace_size(OPS[op], m, n, dt, case["block_rows"], prec=prec)
    st["work"] = torch.empty(need, dtype=torch.uint8, device="cuda")
    if op == "direct":
        st["out"] = (torch.empty_like(st["A"]), torch.empty(n, n, dtype=torch.float64, device="cuda"))
    if op == "direct_host":
        Ah = torch.empty(m, n, dtype=dt, pin_memory=True)
        Ah.copy_(st["A"])
        st["dbuf"] = st["A"]  # the device buffer of the call: overwritten by it
        st["A"] = Ah
        st["out"] = (torch.empty(m, n, dtype=dt, pin_memory=True),
                     torch.empty(n, n, dtype=torch.float64, pin_memory=True))
        st["copy_stream"] = torch.cuda.Stream()
    return st


def run(state):
    case, A = state["case"], state["A"]
    op = case["op"]
    if op == "grad":
        A.grad = None
        Q, R = tsqr.QRFunction.apply(A)
        torch.autograd.backward([Q, R], [state["gQ"], state["gR"]])
        return {"Q": Q.detach(), "R": R.detach(), "dA": A.grad}
    work = state["work"]
    if op == "direct":
        Q, R = tsqr.direct(A, block_rows=case["block_rows"], work=work, out=state["out"], check=False,
                           prec=case["prec"])
        return {"Q": Q, "R": R}
    if op == "direct_host":
        Q, R = tsqr.direct_host(A, out=state["out"], dbuf=state["dbuf"], work=work,
                                copy_stream=state["copy_stream"], check=False, prec=case["prec"])
        return {"Q": Q, "R": R}
    if op == "svd":
        U, S, V = tsqr.svd(A, work=work, check=False, prec=case["prec"])
        return {"U": U, "S": S, "V": V}
    if op == "svd_values":
        S, V = tsqr.svd_values(A, work=work, check=False)
        return {"S": S, "V": V}
    if op == "r":
        return {"R": tsqr.r(A, work=work, check=False)}
    if op == "cholqr":
        Q, R = tsqr.cholqr(A, refine=1, work=work, check=False)
    else:
        Q, R = tsqr.indirect_refine(A, refine=1, work=work, check=False)
    return {"Q": Q, "R": R}


def work(case):
    m, n, s = case["m"], case["n"], 8 if case["dtype"] == "f64" else 4
    tall, small, f = m * n * s, n * n * 8, m * n * n
    op = case["op"]
    if op in ("r", "svd_values"):  # A read; the reduction to R
        return {"bytes": tall + 2 * small, "flops": 2 * f}
    if op == "grad":  # A and dQ in, Q and dA out; QR, then the adjoint's Gram and two products
        return {"bytes": 4 * tall + 2 * small, "flops": 4 * f + 5 * f}
    if op == "cholqr":  # twice: symmetric Gram, product with a triangle
        return {"bytes": 2 * tall + small, "flops": 2 * (f + f)}
    if op == "indirect":  # twice: reduction to R, product with a triangle
        return {"bytes": 2 * tall + small, "flops": 2 * (2 * f + f)}
    return {"bytes": 2 * tall + 2 * small, "flops": 4 * f}  # A in, Q (or U) out


def _qr64(A):
    """Thin QR with diag(R) >= 0 in 64 bits: torch's QR of row chunks, of their
    stacked R factors, and the products."""
    m, n = A.shape
    rows = max(n, 1 << 20)
    parts, Rs = [], []
    for r0 in range(0, m, rows):
        r1 = m if m - r0 < rows + n else min(m, r0 + rows)
        q, r = torch.linalg.qr(A[r0:r1].to(torch.float64))
        parts.append(q)
        Rs.append(r)
        if r1 == m:
            break
    q2, R = torch.linalg.qr(torch.cat(Rs))
    sign = torch.where(torch.diagonal(R) < 0, -1.0, 1.0).to(torch.float64)
    R = R * sign[:, None]
    q2 = q2 * sign[None, :]
    Q = torch.empty(m, n, dtype=torch.float64, device=A.device)
    r0 = 0
    for i, q in enumerate(parts):
        Q[r0:r0 + q.shape[0]] = q @ q2[i * n:(i + 1) * n]
        r0 += q.shape[0]
        parts[i] = None
    return Q, R


def exact(case, seed):
    op = case["op"]
    A = _matrix(case, seed)
    Q, R = _qr64(A)
    if op == "r":
        return {"R": R}
    if op in ("svd", "svd_values"):
        Ur, S, Vh = torch.linalg.svd(R)
        V = Vh.T.contiguous()
        # each pair (u_j, v_j) signed so that the largest entry of v_j is positive
        top = V.gather(0, V.abs().argmax(0, keepdim=True))
        sign = torch.where(top < 0, -1.0, 1.0).to(torch.float64)
        V = V * sign
        return {"S": S, "V": V} if op == "svd_values" else {"U": Q @ (Ur * sign), "S": S, "V": V}
    if op == "grad":
        gQ, gR = _cotangents(case, seed)
        gQ, dR = gQ.to(torch.float64), torch.triu(gR.to(torch.float64))
        M = R @ dR.T - gQ.T @ Q
        C = torch.tril(M) + torch.tril(M, -1).T
        dA = torch.linalg.solve_triangular(R, (gQ + Q @ C).T, upper=True).T
        return {"Q": Q, "R": R, "dA": dA}
    if op == "direct_host":
        return {"Q": Q.cpu(), "R": R.cpu()}
    return {"Q": Q, "R": R}
