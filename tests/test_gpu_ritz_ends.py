"""Ritz pairs whose tridiagonal part, eliminated from both ends, is one to four indices long after a
restart, and of every length in the first one, against LAPACK."""
import numpy as np
import pytest

from paper_2001_07428_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed_reorth"])
@pytest.mark.parametrize("m,left", [(8, 1), (9, 1), (8, 2), (9, 2), (12, 3), (17, 4), (30, 15), (31, 15)])
def test_short_tridiagonal_part(m, left, precision):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2001_07428_gb300.solver import JTRLan
    h = 40
    A11, A12 = inputs.dense_jsym(h, 11)
    A = np.block([[A11, A12], [A12.conj().T, A11.T]])
    s = JTRLan("dense", A11=A11, A12=A12, nev=3, m=m, mwin=m - left, tol=1e-9, precision=precision,
               max_restarts=1000, device="cuda:0")
    st = s.solve()
    ev, _, res = s.pairs()
    s.close()
    # a Hermitian matrix has an eigenvalue within ||A x - lambda x|| of lambda; J pairs each one
    want = np.linalg.eigvalsh(A)[::2][:3]
    assert np.abs(np.sort(ev) - want).max() <= 1e-9 + 1e-13 * np.abs(A).sum(1).max()
    assert st["n_ritz_fallbacks"] == 0
