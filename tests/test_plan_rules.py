"""Which form a size takes where two are at hand, and that the forms agree with the
oracle on both sides of a line: binary64 Step 1 by panels or by register tiles, one
or two tree levels, binary32 Step 3 by 128-row pieces or k_form_q."""
import numpy as np
import pytest

import oracle
import tsqr_inputs as ti

torch = pytest.importorskip("torch")

EPS = {torch.float64: 2.0 ** -52, torch.float32: 2.0 ** -23}


def _T():
    import paper_1301_1071_gb300 as T
    return T


@pytest.mark.parametrize("m,n,tiles", [
    (10_000, 11, 1), (10_000, 16, 1), (3_000, 92, 1), (130, 65, 1), (40_000, 50, 1),  # register tiles
    (10_000, 64, 2), (150_000, 48, 4), (400_000, 64, 11),                              # panels of 128 rows
])
def test_panels_or_tiles(m, n, tiles):
    T = _T()
    for op in (T.OP_DIRECT, T.OP_R, T.OP_SVD):  # the same plan, so that R is the same
        assert T.plan_info(op, m, n, torch.float64)["tiles_per_block"] == tiles


@pytest.mark.parametrize("m,n,dt,levels", [(40_000, 8, torch.float32, 1), (40_000, 3, torch.float64, 1),
                                           (40_000, 20, torch.float64, 2), (600_000, 8, torch.float64, 2)])
def test_one_level_of_narrow_triangles(m, n, dt, levels):
    T = _T()
    info = T.plan_info(T.OP_DIRECT, m, n, dt)
    assert info["tree_levels"] == levels and (levels > 1 or info["blocks"] == info["tree_fanout"])


@pytest.mark.gpu
@pytest.mark.parametrize("m,n,dt", [
    (10_000, 11, torch.float64), (3_000, 92, torch.float64), (130, 65, torch.float64), (40_000, 50, torch.float64),
    (10_000, 64, torch.float64), (40_000, 3, torch.float64), (40_000, 8, torch.float32), (700, 9, torch.float32),
    (60_000, 16, torch.float32), (300_000, 33, torch.float32), (20_000, 33, torch.float32), (40_000, 52, torch.float32)])
def test_both_sides_of_the_lines(m, n, dt):
    T = _T()
    A = ti.gaussian(m, n, 61).astype(np.float64 if dt == torch.float64 else np.float32)
    Ad = torch.tensor(A, device="cuda")
    Q, R = T.direct(Ad)
    Qo, Ro = oracle.householder_qr(A.astype(np.float64))
    tol = 10 * n * np.linalg.cond(A) * EPS[dt]
    assert np.linalg.norm(R.cpu().numpy() - Ro) <= tol * np.linalg.norm(Ro)
    assert np.max(np.abs(Q.double().cpu().numpy() - Qo)) <= tol
    assert torch.equal(T.r(Ad), R)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [65, 69, 80, 81])
def test_binary32_row_products_around_the_line(n):
    T = _T()
    m = 1003
    A = ti.gaussian(m, n, 62)
    Qo, Ro = oracle.householder_qr(A)
    Q32, dQ = Qo.astype(np.float32), ti.gaussian(m, n, 63).astype(np.float32)
    got = T.backward(torch.tensor(Q32, device="cuda"), torch.tensor(Ro, device="cuda"), torch.tensor(dQ, device="cuda"),
                     None).double().cpu().numpy()
    want = oracle.qr_backward(Q32.astype(np.float64), Ro, dQ.astype(np.float64), np.zeros((n, n)))
    assert np.linalg.norm(got - want) <= 4 * n * 2.0 ** -24 * np.linalg.cond(Ro) * np.linalg.norm(want)
