"""The FP64 product kernel over its row forms: one and two rows per CTA, an odd last row, one to four
column chunks, tables of one to four bytes of sites, against the one-spin matrices and the diagonal
multiplied out on the host."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_1307_7542_gb300 import workloads as W

from helpers import assert_entrywise

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def hub(cuda_ok):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1307_7542_gb300 import hub as H
    return H


def _reference(m, x, U, eps):
    """(H x, |H| |x|) as X H_up^T + H_dn X + diag o X."""
    X = x.reshape(m.count_dn, m.count_up)
    bits, A = [], []
    for spin, n in ((0, m.count_up), (1, m.count_dn)):
        rp, cols, vals = m.csr(spin)
        A.append(sp.csr_matrix((vals, cols, rp), shape=(n, n)))
        bits.append(((m.basis(spin).astype(np.int64)[:, None] >> np.arange(m.M)) & 1).astype(np.float64))
    diag = (bits[1] * U) @ bits[0].T
    if eps is not None:
        diag += (bits[0] @ eps)[None, :] + (bits[1] @ eps)[:, None]
    y = (A[0] @ X.T).T + A[1] @ X + diag * X
    a = np.abs(X)
    return y.ravel(), ((abs(A[0]) @ a.T).T + abs(A[1]) @ a + np.abs(diag) * a).ravel()


# sites, electrons: rows x columns
@pytest.mark.parametrize("M,nu,nd", [(4, 2, 1),       # 4 x 6
                                     (9, 3, 7),       # 36 x 84, two tables
                                     (11, 2, 3),      # 165 x 55: one row, narrow
                                     (13, 3, 3),      # 286 x 286: two would leave SMs idle
                                     (11, 5, 4),      # 330 x 462: two chunks
                                     (13, 5, 4),      # 715 x 1287: two rows, an odd last one, four chunks
                                     (17, 7, 1),      # 17 x 19448: long rows, three tables
                                     (25, 2, 2),      # 300 x 300, four tables
                                     (30, 1, 3)])     # 4060 x 30
@pytest.mark.parametrize("eps", [False, True])
def test_rows_and_tables(hub, M, nu, nd, eps):
    b = W.ring_bonds(M)
    U = W.uniform(2, M, -2.0, 8.0)
    e = W.uniform(3, M, -0.5, 0.5) if eps else None
    m = hub.Hubbard(M, nu, nd, b, W.uniform(1, len(b), -1.3, 1.3), U, e)
    x = W.normal(4, m.D)
    y = m.apply(torch.from_numpy(x).cuda()).cpu().numpy()
    ref, bound = _reference(m, x, U, e)
    m.close()
    # the site energies' terms can cancel in the diagonal: its rounding is relative to their sum
    assert_entrywise(y, ref, bound + (0.5 * (nu + nd) * np.abs(x) if eps else 0.0))
