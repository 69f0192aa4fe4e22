"""Accuracy of the binary64 calls against long-double references, beyond the
bars of the parity tests."""
import numpy as np
import pytest

import oracle
import tsqr_inputs as ti

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -53  # half an ulp of 1


def _T():
    import paper_1301_1071_gb300 as T
    return T


def _cuda(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _q_error(A, **kw):
    """||Q - Q_exact||_F / ||Q_exact||_F of the direct call."""
    Q, _ = _T().direct(_cuda(A), **kw)
    Qe, _ = oracle.mgs_ld(A)
    return np.linalg.norm(Q.cpu().numpy() - Qe) / np.linalg.norm(Qe)


@pytest.mark.parametrize("n", [8, 16, 48, 64, 72, 100])
def test_many_tiles_in_a_block(n):
    """One row block of 64 tiles: what a tile adds is independent of the other
    tiles' and at most half an ulp of the running R and of the coefficient X
    (their one rounding a tile), so Q errs by at most sqrt(64) + 1 half ulps,
    the first tile's own included.  (With 2 - tau taken from the rounded tau, as
    the tiles' tau come close to 2, it was twice that.)"""
    tiles = 64
    errs = [_q_error(ti.gaussian(128 * tiles, n, 900 + s), block_rows=128 * tiles) for s in range(2)]
    assert max(errs) <= U * (np.sqrt(tiles) + 1), errs


@pytest.mark.parametrize("n", [25, 33, 48, 49, 64])
def test_small_entries_of_a_row(n):
    """dQ R^-T with R = I returns dQ (Q = 0 leaves the other terms out).  A row is
    held in 62-bit fixed point against its largest entry (columns relative to
    their own scale), so an entry 1e-8 of that keeps 2^-62 of it (doubled for
    the exponents' rounding up, twice) next to its own half ulp."""
    T = _T()
    m = 1003
    dQ = ti.gaussian(m, n, 31)
    dQ[::3, n - 1] *= 1e-8
    dQ[1::3, 0] *= 1e-6
    got = T.backward(_cuda(np.zeros((m, n))), _cuda(np.eye(n)), _cuda(dQ), None).cpu().numpy()
    col = np.abs(dQ).max(axis=0)
    row = (np.abs(dQ) / col).max(axis=1)
    assert np.all(np.abs(got - dQ) <= 2.0 ** -60 * row[:, None] * col + U * np.abs(dQ))


@pytest.mark.parametrize("m,block_rows,fanout,seeds,bar", [
    # 157 blocks of 128 rows in two levels of 13; the bar: 5 % above what 63
    # blocks of 320 rows under one level gave, 2.90e-16 +- 0.02
    (20_000, 0, 0, 24, 1.05 * 2.90e-16),
    # 128 blocks in seven levels of 2; the bar: what nodes factored with scaled
    # vectors and rounded roots and quotients gave, 4.80e-16 +- 0.05
    (16_384, 128, 2, 12, 4.80e-16),
])
def test_tree_levels(m, block_rows, fanout, seeds, bar):
    """The tree adds no more to Q's error (root mean square over the seeds) than
    fewer levels, or nodes in plain binary64 steps, did.  (With each level's top
    block C - W rounded at C's size and rows of R formed as r - tau (r + v^T a)
    the two were 3.30e-16 and 5.46e-16.)"""
    errs = [_q_error(ti.gaussian(m, 13, 950 + s), block_rows=block_rows, fanout=fanout) for s in range(seeds)]
    assert np.sqrt(np.mean(np.square(errs))) <= bar, errs
