"""The binary64 tall products as exact digit products (Gram, rows times an
n x n matrix, Step 3), at the edges of their fragments: n around multiples of
8 (column groups) and 16 (k steps), rows around 16 (row pieces), 64 (chunks)
and of several unaligned tiles, against the CPU oracle.

Tolerances: a product entry errs by at most a few units of 2^-53 of its row by
column scale, as a binary64 FMA chain does, so the bars are those of the
binary64 tests: 10 n kappa 2^-52 element-wise for Q and R, 1e-12 for dA.
"""
import ctypes

import numpy as np
import pytest

import oracle
import tsqr_inputs as ti

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS64 = 2.0 ** -52


def _T():
    import paper_1301_1071_gb300 as T
    return T


def _cuda(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("n", [1, 7, 8, 9, 16, 17, 25, 32, 33, 48, 49, 64, 65, 98])  # the adjoint's n x n step takes n <= 98
@pytest.mark.parametrize("m", [0, 15, 16, 1003])
def test_backward_edges(m, n):
    m = max(n, m) if m < 1003 else m + n
    A, dQ, dR = ti.gaussian(m, n, 1), ti.gaussian(m, n, 2), ti.gaussian(n, n, 3)
    Qo, Ro = oracle.householder_qr(A)
    want = oracle.qr_backward(Qo, Ro, dQ, np.triu(dR))
    got = _T().backward(_cuda(Qo), _cuda(Ro), _cuda(dQ), _cuda(dR)).cpu().numpy()
    kappa = np.linalg.cond(Ro)
    assert np.linalg.norm(got - want) <= 1e-12 * max(1.0, kappa) * np.linalg.norm(want)


def test_backward_scaled_columns():
    """Columns of dQ from 1 to 1e-10: each keeps its own relative accuracy
    (R diagonal, so that columns do not mix)."""
    m, n = 2003, 25
    Qo, _ = oracle.householder_qr(ti.gaussian(m, n, 1))
    R = np.diag(np.linspace(1.0, 2.0, n))
    scale = ti.log_spaced(n, 1.0, 1e-10)
    dQ = ti.gaussian(m, n, 2) * scale[None, :]
    dQ -= Qo @ (Qo.T @ dQ)  # no part along Q: dA = dQ R^-T up to rounding
    got = _T().backward(_cuda(Qo), _cuda(R), _cuda(dQ), None).cpu().numpy()
    want = oracle.qr_backward(Qo, R, dQ, np.zeros((n, n)))
    own = dQ / np.diag(R)[None, :]
    # a column's rounding is that of dQ R^-T (its own scale) and of Q C R^-T
    # with C = copyltu(-dQ^T Q), whose entries are rounding errors of dQ^T Q
    C = -np.tril(dQ.T @ Qo)
    extra = np.abs(Qo @ (C + np.tril(C, -1).T)).max(axis=0)
    err = np.linalg.norm(got - want, axis=0)
    assert np.all(err <= 40 * n * EPS64 * (np.linalg.norm(own, axis=0) + np.sqrt(m) * (extra + EPS64 * scale)))


def test_backward_in_place():
    """dA over dQ and over Q: each input is read before it is overwritten."""
    T = _T()
    m, n = 1003, 25
    Qo, Ro = oracle.householder_qr(ti.gaussian(m, n, 1))
    Q, R, dQ = _cuda(Qo), _cuda(Ro), _cuda(ti.gaussian(m, n, 2))
    want = T.backward(Q, R, dQ, None)
    lib = T.load()
    need = T.workspace_size(T.OP_BACKWARD, m, n, torch.float64)
    work = torch.empty(need, dtype=torch.uint8, device="cuda")
    for over in ("dQ", "Q"):
        q, d = Q.clone(), dQ.clone()
        out = d if over == "dQ" else q
        st = lib.tsqr_backward(ctypes.c_void_p(q.data_ptr()), ctypes.c_void_p(R.data_ptr()),
                               ctypes.c_void_p(d.data_ptr()), None, m, n, 0, ctypes.c_void_p(out.data_ptr()),
                               ctypes.c_void_p(work.data_ptr()), need, None,
                               ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert st == 0
        torch.cuda.synchronize()
        err = torch.linalg.norm(out - want) / torch.linalg.norm(want)
        assert err <= 1e-14, over


@pytest.mark.parametrize("n", [1, 8, 9, 16, 25, 33, 48, 49, 64, 65, 100])
def test_cholqr_column_scaled(n):
    """Columns from 1 to 1e-9 (the Gram's and R^-1's entries span 1e18)."""
    m = 4003
    A = ti.column_scaled(m, n, 1e-9, 4)
    Q, R = _T().cholqr(_cuda(A))
    Q, R = Q.cpu().numpy(), R.cpu().numpy()
    Qo, Ro = oracle.householder_qr(A)
    kappa = np.linalg.cond(A / np.linalg.norm(A, axis=0)[None, :])
    tol = 10 * n * kappa ** 2 * EPS64
    assert np.max(np.abs(Q - Qo)) <= tol
    assert np.max(np.linalg.norm(R - Ro, axis=0) / np.linalg.norm(Ro, axis=0)) <= tol


@pytest.mark.parametrize("n", [1, 7, 8, 9, 16, 17, 32, 33, 48, 49, 64, 65])
@pytest.mark.parametrize("m,b", [(331, 0), (5003, 1001), (5003, 2999)])
def test_direct_edges(m, n, b):
    A = ti.gaussian(m, n, 5)
    Q, R = _T().direct(_cuda(A), block_rows=b)
    Q, R = Q.cpu().numpy(), R.cpu().numpy()
    Qo, Ro = oracle.householder_qr(A)
    tol = 10 * n * np.linalg.cond(A) * EPS64
    assert np.linalg.norm(R - Ro) <= tol * np.linalg.norm(Ro)
    assert np.max(np.abs(Q - Qo)) <= tol
    assert oracle.orth_error(Q)[0] <= 1e-13


@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_non_finite_is_reported(value):
    T = _T()
    A = ti.gaussian(3000, 25, 6)
    Qo, Ro = oracle.householder_qr(A)
    dQ = ti.gaussian(3000, 25, 7)
    dQ[1234, 3] = value
    with pytest.raises(T.TSQRError) as e:
        T.backward(_cuda(Qo), _cuda(Ro), _cuda(dQ), None)
    assert e.value.status == 8
    A[77, 11] = value
    with pytest.raises(T.TSQRError):
        T.cholqr(_cuda(A))
    with pytest.raises(T.TSQRError) as e:
        T.direct(_cuda(A))
    assert e.value.status == 8


def _f32(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda")


# binary32: 8-column thread groups, k steps of 4, copies of 16, 8 or 4 bytes (n
# mod 4), 128-row tiles.  A product entry is a chain of at most 2 n binary32
# FMAs: 4 n 2^-24 of its row by column scale, and kappa of R for the adjoint.
@pytest.mark.parametrize("n", [7, 8, 9, 11, 12, 25, 32, 33, 50, 63, 64, 65, 66, 77, 98, 100])
@pytest.mark.parametrize("m,b", [(127, 0), (128, 0), (2003, 701)])
def test_binary32_direct_edges(m, n, b):
    A = ti.gaussian(m, n, 8).astype(np.float32)
    Q, R = _T().direct(_f32(A), block_rows=b, prec="native")
    Q, R = Q.double().cpu().numpy(), R.cpu().numpy()
    Qo, Ro = oracle.householder_qr(A.astype(np.float64))
    tol = 10 * n * np.linalg.cond(A) * 2.0 ** -24
    assert np.linalg.norm(R - Ro) <= tol * np.linalg.norm(Ro)
    assert np.max(np.abs(Q - Qo)) <= tol
    assert oracle.orth_error(Q)[0] <= 1e-5


@pytest.mark.parametrize("n", [7, 8, 9, 12, 25, 33, 50, 65, 98])
@pytest.mark.parametrize("m", [127, 1003])
def test_binary32_backward_edges(m, n):
    A, dQ, dR = ti.gaussian(m, n, 1), ti.gaussian(m, n, 2).astype(np.float32), ti.gaussian(n, n, 3)
    Qo, Ro = oracle.householder_qr(A)
    Q32 = Qo.astype(np.float32)
    got = _T().backward(_f32(Q32), _cuda(Ro), _f32(dQ), _cuda(dR)).double().cpu().numpy()
    want = oracle.qr_backward(Q32.astype(np.float64), Ro, dQ.astype(np.float64), np.triu(dR))
    tol = 4 * n * 2.0 ** -24 * np.linalg.cond(Ro)
    assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want)


def test_binary32_backward_in_place():
    T = _T()
    m, n = 1003, 25
    Qo, Ro = oracle.householder_qr(ti.gaussian(m, n, 1))
    Q, R, dQ = _f32(Qo), _cuda(Ro), _f32(ti.gaussian(m, n, 2))
    want = T.backward(Q, R, dQ, None)
    lib = T.load()
    need = T.workspace_size(T.OP_BACKWARD, m, n, torch.float32)
    work = torch.empty(need, dtype=torch.uint8, device="cuda")
    for over in ("dQ", "Q"):
        q, d = Q.clone(), dQ.clone()
        out = d if over == "dQ" else q
        st = lib.tsqr_backward(ctypes.c_void_p(q.data_ptr()), ctypes.c_void_p(R.data_ptr()),
                               ctypes.c_void_p(d.data_ptr()), None, m, n, 1, ctypes.c_void_p(out.data_ptr()),
                               ctypes.c_void_p(work.data_ptr()), need, None,
                               ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert st == 0
        torch.cuda.synchronize()
        assert torch.equal(out, want), over  # the same sums in the same order


@pytest.mark.parametrize("n", [7, 11, 12, 13, 25, 33, 50, 65, 100])
def test_binary32_cholqr(n):
    """The Gram of binary32 data is exact to binary64 rounding: R is the oracle's
    to kappa^2 2^-52, Q to its storage."""
    A = ti.column_scaled(4003, n, 1e-4, 4).astype(np.float32)
    Q, R = _T().cholqr(_f32(A))
    Qo, Ro = oracle.householder_qr(A.astype(np.float64))
    kappa = np.linalg.cond(A / np.linalg.norm(A, axis=0)[None, :])
    assert np.max(np.abs(Q.double().cpu().numpy() - Qo)) <= 10 * n * kappa ** 2 * 2.0 ** -24
    # the second pass factors the binary32 Q, so R carries its rounding
    assert np.max(np.linalg.norm(R.cpu().numpy() - Ro, axis=0) / np.linalg.norm(Ro, axis=0)) \
        <= 10 * n * kappa ** 2 * 2.0 ** -24
    A[77, 5] = np.inf
    with pytest.raises(_T().TSQRError):
        _T().cholqr(_f32(A))
