"""The binary64 products by digits entry by entry, against extended precision,
at the ends of the exponent range, and on rows of very different size -- and the
Householder scalars that go with them.

What the header promises of them is normwise: an entry of a product errs by a
few 2^-56 of its row's scale times its column's (column scales taken out first);
Step 1 holds a column in 62 bits against its norm.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
import tsqr_inputs as ti

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS64 = 2.0 ** -52
U = 2.0 ** -53
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _T():
    import paper_1301_1071_gb300 as T
    return T


def _cuda(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _backward(Q, R, dQ):
    return _T().backward(_cuda(Q), _cuda(R), _cuda(dQ), None).cpu().numpy()


@pytest.mark.parametrize("n", [7, 16, 25, 32, 33, 48, 64])
def test_rows_times_matrix(n):
    """dA = dQ R^-T (Q = 0) with R unit triangular of 0, 1, -1, whose inverse is of
    whole numbers: every entry within 2^-55 of row x column scale (4.5 times the
    root mean square of the digit diagonals left out, 2^-59.2 of the two powers of
    two above the scales) and its own half ulp."""
    rng = np.random.default_rng(90 + n)
    m = 517
    N = np.triu(rng.choice([0, 0, 0, 0, 0, 0, 0, 0, 0, 1, -1], (n, n)), 1)
    R = np.eye(n) + N
    M = np.rint(np.linalg.inv(R)).T
    assert np.array_equal(R @ M.T, np.eye(n)) and np.abs(M).max() < 2**40
    dQ = ti.gaussian(m, n, 91) * ti.log_spaced(n, 1.0, 1e-6)[None, :]
    got = _backward(np.zeros((m, n)), R, dQ)
    want = dQ.astype(np.longdouble) @ M.astype(np.longdouble)
    c = np.abs(dQ).max(axis=0)
    scale = (np.abs(dQ) / c).max(axis=1)[:, None] * (c[:, None] * np.abs(M)).max(axis=0)[None, :]
    assert np.all(np.abs(got - want) <= 2.0 ** -55 * scale + U * np.abs(want))


# tsqr::launch_gram_split, its C++ name
GRAM = "_ZN4tsqr17launch_gram_splitEPKdS1_liiPiPdS2_P11CUstream_st"


@pytest.mark.parametrize("n", [7, 16, 25, 33, 64, 65, 100])
@pytest.mark.parametrize("m", [1, 64, 1003])
@pytest.mark.parametrize("same", [False, True])
def test_gram(m, n, same):
    """The partial Grams X^T Y of the launcher itself, summed in extended precision.
    A chunk of 64 rows (32 for n > 64) errs by 2^-54 of the columns' scales at most,
    the sums over chunks by half an ulp each."""
    X, Y = ti.gaussian(m, n, 92), ti.gaussian(m, n, 93) * ti.log_spaced(n, 1.0, 1e-9)[None, :]
    if same:
        X = Y
    Xd = _cuda(X)
    Yd = Xd if same else _cuda(Y)
    most = 64
    part = torch.full((most * n * n,), float("nan"), dtype=torch.float64, device="cuda")
    got = ctypes.c_int(0)
    fn = getattr(_T().load(), GRAM)
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int64, ctypes.c_int, ctypes.c_int,
                   ctypes.POINTER(ctypes.c_int), ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]
    assert fn(Xd.data_ptr(), Yd.data_ptr(), m, n, most, ctypes.byref(got), part.data_ptr(), None, None) == 0
    torch.cuda.synchronize()
    chunks = -(-m // (64 if n <= 64 else 32))
    assert 1 <= got.value <= min(most, chunks)
    G = part[:got.value * n * n].cpu().numpy().reshape(got.value, n, n).astype(np.longdouble).sum(axis=0)
    want = X.T.astype(np.longdouble) @ Y.astype(np.longdouble)
    cx, cy = np.abs(X).max(axis=0), np.abs(Y).max(axis=0)
    tol = cx[:, None] * cy[None, :] * (2.0 ** -54 * np.sqrt(chunks) + U * chunks * 16) + 4 * U * np.abs(want)
    assert np.all(np.abs(G - want) <= tol)


@pytest.mark.parametrize("n", [9, 25, 48, 64])
@pytest.mark.parametrize("p", [-1000, -500, 500, 1000])
def test_products_scale_exactly(n, p):
    """A power of two through the digits changes exponents alone."""
    m = 333
    R, dQ = np.triu(ti.gaussian(n, n, 94)) + 4 * np.eye(n), ti.gaussian(m, n, 95)
    a, b = _backward(np.zeros((m, n)), R, dQ), _backward(np.zeros((m, n)), R, dQ * 2.0 ** p)
    assert np.array_equal(b, a * 2.0 ** p)


def test_products_of_subnormal_rows():
    m, n = 100, 25
    dQ = ti.gaussian(m, n, 96) * 2.0 ** -1060
    got = _backward(np.zeros((m, n)), np.eye(n), dQ)
    assert np.all(np.abs(got - dQ) <= 2.0 ** -1074)


@pytest.mark.parametrize("n", [8, 25, 32, 64])
@pytest.mark.parametrize("p", [-400, -60, 60, 400])
def test_direct_at_the_ends_of_the_range(n, p):
    """Norms beyond the fast Householder scalars' range (2^-56 .. 2^56) take the
    library's: the same accuracy.  Cholesky QR scales exactly."""
    T = _T()
    m = 2003
    A = ti.gaussian(m, n, 97)
    Qo, Ro = oracle.householder_qr(A)
    Q, R = T.direct(_cuda(A * 2.0 ** p))
    tol = 10 * n * np.linalg.cond(A) * EPS64
    assert np.max(np.abs(Q.cpu().numpy() - Qo)) <= tol
    assert np.linalg.norm(R.cpu().numpy() * 2.0 ** -p - Ro) <= tol * np.linalg.norm(Ro)
    Qc, Rc = T.cholqr(_cuda(A))
    Qs, Rs = T.cholqr(_cuda(A * 2.0 ** p))
    assert torch.equal(Qs, Qc) and torch.equal(Rs, Rc * 2.0 ** p)


@pytest.mark.parametrize("n", [8, 25, 32, 64, 72])
@pytest.mark.parametrize("order", ["falling", "rising", "mixed"])
def test_rows_of_very_different_size(n, order):
    """Rows from 1 to 1e-12.  Q within n kappa 2^-52 as a matrix; its rows within n
    kappa of 2^-52 of their own size plus 2^-60 (Step 1's fixed point, 62 bits against
    the column norm), but for the first n of a row block, which come out of a
    difference at the size of the block's coefficient (in any arithmetic).  In the
    adjoint every row has a scale of its own."""
    T = _T()
    m = 3000
    g = ti.log_spaced(m, 1.0, 1e-12)
    g = {"falling": g, "rising": g[::-1], "mixed": np.random.default_rng(98).permutation(g)}[order]
    A = ti.gaussian(m, n, 99) * g[:, None]
    Qe, Re = oracle.mgs_ld(A)
    kappa = np.linalg.cond(A)
    Q, _ = T.direct(_cuda(A))
    Q = Q.cpu().numpy()
    size = np.linalg.norm(Qe, axis=1)
    err = np.linalg.norm(Q - Qe, axis=1)
    assert np.linalg.norm(err) <= 10 * n * kappa * EPS64 * np.sqrt(n)
    below = np.arange(m) % T.plan_info(T.OP_DIRECT, m, n, torch.float64)["block_rows"] >= n
    assert np.all((err <= 10 * n * kappa * (EPS64 * size + 2.0 ** -60))[below])
    dQ = ti.gaussian(m, n, 100) * g[:, None]
    got = _T().backward(_cuda(Qe), _cuda(Re), _cuda(dQ), None).cpu().numpy()
    want = oracle.qr_backward(Qe, Re, dQ, np.zeros((n, n)))
    C = np.tril(dQ.T @ Qe)
    C = C + np.tril(C, -1).T
    size = (np.linalg.norm(dQ, axis=1) + size * np.linalg.norm(C)) * np.linalg.norm(np.linalg.inv(Re))
    assert np.all(np.linalg.norm(got - want, axis=1) <= 10 * n * EPS64 * size)


@pytest.mark.parametrize("n", [16, 25, 64])
@pytest.mark.parametrize("block_rows", [128, 4000])
def test_largest_reflector_coefficients(n, block_rows):
    """Columns equal or opposite to an earlier one of its panel take the largest
    coefficients there are, twice their norm (entries one ulp below a power of two:
    the least room above the column's scale)."""
    m = 4000
    A = ti.gaussian(m, n, 101)
    A[:, 0] = 2.0 - 2 * EPS64
    A[0, 0] = 0.0
    for c in range(8, n):
        A[:, c] = A[:, c % 8] * (1.0 if c & 1 else -1.0) + 1e-3 * A[:, c]
    Q, R = _T().direct(_cuda(A), block_rows=block_rows)
    Q, R = Q.cpu().numpy(), R.cpu().numpy()
    assert np.linalg.norm(A - Q @ R) <= 1e-14 * np.linalg.norm(A)
    assert oracle.orth_error(Q)[0] <= 1e-13


def test_householder_scalars(tmp_path):
    """make_reflector64 within its roundings of extended precision: the root 1 ulp,
    1 / beta 1, 1 / (alpha - beta) 2 (the sum's and the root's), tau 4 -- over and
    beyond its fast range -- and the library's zero column."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    so = str(tmp_path / "reflector.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O3", "--expt-relaxed-constexpr",
                    "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(ROOT, "paper_1301_1071_gb300", "csrc"), "-o", so,
                    os.path.join(ROOT, "tests", "host", "reflector.cu")], check=True, capture_output=True)
    rng = np.random.default_rng(102)
    k = 200_000
    s2 = (1 + rng.random(k)) * 2.0 ** rng.integers(-130, 130, k)
    s2[:4] = [2.0 ** -113, np.nextafter(2.0 ** 113, 0), 2.0 ** 113, np.nextafter(2.0 ** -113, 0)]
    alpha = np.sqrt(s2) * rng.choice([0.0, 1e-300, 1e-9, 0.3, 0.9, 1 - 2.0 ** -50, 1.0], k) * rng.choice([-1, 1], k)
    d = [_cuda(x) for x in (s2, alpha, np.zeros(4 * k))]
    lib = ctypes.CDLL(so)
    torch.cuda.synchronize()
    assert lib.reflector_scalars(*[ctypes.c_void_p(t.data_ptr()) for t in d[:2]], k, ctypes.c_void_p(d[2].data_ptr())) == 0
    beta, scal, ib, tau = d[2].cpu().numpy().reshape(k, 4).T
    L = np.longdouble
    root = np.sqrt(s2.astype(L))
    b = np.where(alpha >= 0, -root, root)
    b = np.where((alpha == 0) & np.signbit(alpha), root, b)
    for got, want, ulps in [(beta, b, 1), (ib, 1 / b, 1), (scal, 1 / (alpha - b), 2), (tau, (b - alpha) / b, 4)]:
        assert np.all(np.abs(got - want) <= ulps * EPS64 * np.abs(want))
    z = [_cuda(np.zeros(1)), _cuda(np.zeros(1)), _cuda(np.ones(4))]
    torch.cuda.synchronize()
    assert lib.reflector_scalars(*[ctypes.c_void_p(t.data_ptr()) for t in z[:2]], 1, ctypes.c_void_p(z[2].data_ptr())) == 0
    assert z[2].cpu().tolist() == [0.0, 0.0, 0.0, 0.0]
