"""Workspaces: what the fastest plan wants (tsqr_workspace_size), the least a
call runs with (tsqr_workspace_min), and calls between the two -- the column
loop's taller tiles keep fewer T factors than the panels' 128-row tiles, and a
call that fits them is not refused for the panels' sake."""
import ctypes
import random

import numpy as np
import pytest

import oracle
import tsqr_inputs as ti

torch = pytest.importorskip("torch")

EPS64 = 2.0 ** -52
STATIC_BYTES = 16 * 1024 * 1024


def _T():
    import paper_1301_1071_gb300 as T
    return T


# The largest m whose call on the fixed scratch fits 16 MiB with the column
# loop's tiles and the tree of the largest fan-in, per n.
@pytest.mark.parametrize("n,m", [(7, 20_847_104), (8, 15_939_328), (10, 10_078_208), (16, 3_628_544), (24, 734_464),
                                 (25, 730_816), (32, 603_136), (48, 119_360), (64, 80_256), (100, 13_760)])
def test_reach_of_the_fixed_scratch(n, m):
    T = _T()
    assert T.workspace_min(T.OP_DIRECT, m, n, torch.float64) <= STATIC_BYTES
    assert T.workspace_min(T.OP_DIRECT, m // 3, n, torch.float64) <= STATIC_BYTES


# Bytes that the calls took with those tiles (and at most 304 partial Grams).
@pytest.mark.parametrize("op,m,n,was", [
    ("OP_DIRECT", 4_000_000, 64, 446_660_864), ("OP_DIRECT", 6_000_000, 32, 110_338_304),
    ("OP_DIRECT", 25_000_000, 16, 106_547_456), ("OP_DIRECT", 25_000_000, 8, 26_159_872),
    ("OP_SVD", 50_000_000, 50, 3_777_820_256), ("OP_INDIRECT", 4_000_000, 64, 446_660_864),
    ("OP_DIRECT_HOST", 8_000_000, 25, 159_155_280), ("OP_CHOLQR", 10_000, 25, 130_256),
    ("OP_BACKWARD", 10_000, 64, 1_736_960), ("OP_R", 2_000, 8, 9_984)])
def test_least_workspace(op, m, n, was):
    T = _T()
    assert T.workspace_min(getattr(T, op), m, n, torch.float64) <= was


def test_least_is_no_more_than_the_full_size():
    T = _T()
    rng = random.Random(7)
    for _ in range(2000):
        n = rng.randint(1, 100)
        m = max(n, int(10 ** rng.uniform(0, 9)))
        op, dt = rng.randint(0, 7), rng.choice([torch.float64, torch.float32])
        kw = dict(block_rows=rng.choice([0, 0, n, 4096]), fanout=rng.choice([0, 0, 2]))
        assert 0 < T.workspace_min(op, m, n, dt, **kw) <= T.workspace_size(op, m, n, dt, **kw)


def test_r_alone_keeps_no_t_factors():
    T = _T()
    for m, n in [(4_000_000, 64), (8_000_000, 25), (25_000_000, 16)]:
        blocks = T.plan_info(T.OP_INDIRECT, m, n, torch.float64)["blocks"]
        # the stacks of R factors (a geometric series over the levels) and small scratch
        assert T.workspace_size(T.OP_INDIRECT, m, n, torch.float64) <= (2 * blocks + 20) * n * n * 8 + 4096
        assert T.workspace_min(T.OP_R, m, n, torch.float64) <= T.workspace_size(T.OP_INDIRECT, m, n, torch.float64)


@pytest.mark.parametrize("m,n", [(88_439_502, 91), (60_999_768_310, 22)])
def test_block_heights_refused_by_either_form(m, n):
    """More tiles in a block than 2^20 of the taller kind: a shape error, also where
    the panels' tiles alone could be indexed."""
    T = _T()
    with pytest.raises(T.TSQRError) as e:
        T.workspace_size(T.OP_DIRECT, m, n, torch.float64, block_rows=2**31 - 1)
    assert e.value.status == 2


def test_binding_workspace(monkeypatch):
    """The binding keeps a buffer the call runs with, and takes the least one where
    the full size cannot be allocated (on the CPU allocator here)."""
    T = _T()
    m, n = 400_000, 64
    full, least = (f(T.OP_DIRECT, m, n, torch.float64) for f in (T.workspace_size, T.workspace_min))
    assert least < full

    def get(work=None, op=T.OP_DIRECT):
        return T._workspace(op, m, n, torch.float64, "cpu", 0, 0, work)

    assert get().numel() == full
    old = torch.empty(least, dtype=torch.uint8)
    assert get(old) is old
    assert get(torch.empty(least - 1, dtype=torch.uint8)).numel() == full
    assert get(op=T.OP_R).numel() == T.workspace_size(T.OP_INDIRECT, m, n, torch.float64) < full // 2
    empty = torch.empty

    def scarce(k, **kw):
        if k > least:
            raise torch.cuda.OutOfMemoryError("full")
        return empty(k, **kw)

    monkeypatch.setattr(T.torch, "empty", scarce)
    assert get().numel() == least


def _cuda(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


class _Bounded:
    """A workspace of `need` bytes with a guard behind it."""

    def __init__(self, need):
        self.need = need
        self.t = torch.full((need + 4096,), 0xAB, dtype=torch.uint8, device="cuda")

    def intact(self):
        return bool((self.t[self.need:] == 0xAB).all())


def _call(T, fn, *args, work, opts=None):
    st = torch.cuda.current_stream().cuda_stream
    p = [ctypes.c_void_p(a.data_ptr()) if isinstance(a, torch.Tensor) else a for a in args]
    return getattr(T.load(), fn)(*p, ctypes.c_void_p(work.t.data_ptr()), work.need, opts, ctypes.c_void_p(st))


def _check(A, Q, R):
    n = A.shape[1]
    Qo, Ro = oracle.householder_qr(A)
    tol = 10 * n * np.linalg.cond(A) * EPS64
    Q, R = Q.cpu().numpy(), R.cpu().numpy()
    assert np.linalg.norm(R - Ro) <= tol * np.linalg.norm(Ro) and np.max(np.abs(Q - Qo)) <= tol


@pytest.mark.gpu
@pytest.mark.parametrize("m,n", [(2000, 8), (20_000, 13), (30_000, 25), (9_001, 32), (20_000, 64), (5_000, 100)])
def test_calls_with_the_least_workspace(m, n):
    T = _T()
    A = ti.gaussian(m, n, 81)
    Ad = _cuda(A)
    Q, R = torch.empty_like(Ad), torch.empty(n, n, dtype=torch.float64, device="cuda")
    for op, fn, args in [
            (T.OP_DIRECT, "tsqr_direct", (Ad, m, n, n, 0, Q, n, R, n)),
            (T.OP_CHOLQR, "cholqr", (Ad, m, n, n, 0, Q, n, R, n, 1)),
            (T.OP_INDIRECT, "tsqr_indirect_refine", (Ad, m, n, n, 0, Q, n, R, n, 1))]:
        Q.zero_(), R.zero_()
        w = _Bounded(T.workspace_min(op, m, n, torch.float64))
        assert _call(T, fn, *args, work=w) == 0, fn
        assert T.load().tsqr_read_status(ctypes.c_void_p(w.t.data_ptr()), None) == 0 and w.intact(), fn
        _check(A, Q, R)
        w.need -= 16
        assert _call(T, fn, *args, work=w) == 4, fn  # TSQR_ERR_WORKSPACE, before any launch
    Ro = torch.tensor(oracle.householder_qr(A)[1])
    w = _Bounded(T.workspace_min(T.OP_R, m, n, torch.float64))
    assert _call(T, "tsqr_r", Ad, m, n, n, 0, R, n, work=w) == 0
    torch.cuda.synchronize()
    assert w.intact() and torch.linalg.norm(R.cpu() - Ro) <= 10 * n * np.linalg.cond(A) * EPS64 * torch.linalg.norm(Ro)
    # R alone in its fastest form: the size of TSQR_OP_INDIRECT, the bits of the full one
    w = _Bounded(T.workspace_size(T.OP_INDIRECT, m, n, torch.float64))
    assert _call(T, "tsqr_r", Ad, m, n, n, 0, R, n, work=w) == 0
    assert w.intact() and torch.equal(R, T.r(Ad, work=torch.empty(
        T.workspace_size(T.OP_R, m, n, torch.float64), dtype=torch.uint8, device="cuda")))


@pytest.mark.gpu
@pytest.mark.parametrize("m,n", [(3_000, 9), (20_000, 64)])
def test_backward_and_svd_with_the_least_workspace(m, n):
    T = _T()
    A = ti.gaussian(m, n, 82)
    Qo, Ro = oracle.householder_qr(A)
    dQ = ti.gaussian(m, n, 83)
    w = _Bounded(T.workspace_min(T.OP_BACKWARD, m, n, torch.float64))
    dA = torch.empty(m, n, dtype=torch.float64, device="cuda")
    assert _call(T, "tsqr_backward", _cuda(Qo), _cuda(Ro), _cuda(dQ), None, m, n, 0, dA, work=w) == 0
    torch.cuda.synchronize()
    want = oracle.qr_backward(Qo, Ro, dQ, np.zeros((n, n)))
    assert w.intact() and np.linalg.norm(dA.cpu().numpy() - want) <= 1e-12 * np.linalg.cond(Ro) * np.linalg.norm(want)
    S = torch.empty(n, dtype=torch.float64, device="cuda")
    for op, fn, args in [(T.OP_SVD, "tsqr_svd", (_cuda(A), m, n, n, 0, torch.empty_like(dA), n, S, torch.empty(
            n, n, dtype=torch.float64, device="cuda"), n)),
            (T.OP_SVD_VALUES, "tsqr_svd_values", (_cuda(A), m, n, n, 0, S, None, n))]:
        S.zero_()
        w = _Bounded(T.workspace_min(op, m, n, torch.float64))
        assert _call(T, fn, *args, work=w) == 0, fn
        torch.cuda.synchronize()
        assert w.intact() and np.max(np.abs(S.cpu().numpy() - np.linalg.svd(Ro)[1])) <= 10 * n * EPS64 * float(S[0])


@pytest.mark.gpu
def test_host_buffers_with_the_least_workspace():
    T = _T()
    m, n = 300_000, 64
    A = ti.gaussian(m, n, 84)
    least = T.workspace_min(T.OP_DIRECT_HOST, m, n, torch.float64)
    assert least < T.workspace_size(T.OP_DIRECT_HOST, m, n, torch.float64)
    Q, R = T.direct_host(torch.tensor(A).pin_memory(), work=torch.empty(least, dtype=torch.uint8, device="cuda"))
    torch.cuda.synchronize()
    _check(A, Q, R)


@pytest.mark.gpu
@pytest.mark.parametrize("m,n", [(300_000, 32), (70_001, 64)])
def test_fixed_scratch_beyond_the_panels_reach(m, n):
    T = _T()
    assert T.workspace_size(T.OP_DIRECT, m, n, torch.float64) > STATIC_BYTES
    A = ti.gaussian(m, n, 85)
    Q, R = T.direct_static(_cuda(A))
    _check(A, Q, R)
