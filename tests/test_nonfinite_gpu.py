"""A NaN or an infinity in A reaches what a caller may read without the status:
every entry of Q, and R from that column on (the columns left of it do not depend
on it).  One row block, where no tree spreads it."""
import numpy as np
import pytest

import tsqr_inputs as ti

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [7, 8, 25, 32, 64, 72])
@pytest.mark.parametrize("m", [120, 1000])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_one_block(m, n, value):
    import paper_1301_1071_gb300 as T
    A = ti.gaussian(m, n, 71)
    _, Rc = T.direct(torch.tensor(A, device="cuda"), block_rows=m)
    Rc = Rc.cpu().numpy()
    for col in sorted({0, 3, n // 2, n - 2, n - 1}):
        for row in (0, m // 2, m - 1):
            B = A.copy()
            B[row, col] = value
            Q, R = T.direct(torch.tensor(B, device="cuda"), block_rows=m, check=False)
            Q, R = Q.cpu().numpy(), R.cpu().numpy()
            assert not np.isfinite(Q).any(), (row, col)
            assert not np.isfinite(np.diag(R)[col:]).any(), (row, col)
            assert np.allclose(R[:, :col], Rc[:, :col], rtol=0, atol=1e-12 * np.linalg.norm(Rc)), (row, col)
