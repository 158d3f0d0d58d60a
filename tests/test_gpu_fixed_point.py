"""The FP64 form's fixed-point basis and integer Gram-Schmidt at the sizes where its partition changes:
one tile of 32 row pairs, a ragged last tile, one thread-block cluster (up to 32 tiles) against a grid,
a basis beyond the 64 products a sum holds, and a start vector with one nonzero entry (every other
column entry lies far below the column's scale)."""
import numpy as np
import pytest
import torch

from paper_2001_07428_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2001_07428_gb300 import binding
    binding.load()


# h, m, start: 1 tile; 2 ragged; 8 full; 9; 22 of a cluster; 33 on a grid; m above 64 and 128
@pytest.mark.parametrize("h,nev,m,delta", [(20, 3, 12, False), (33, 4, 16, True), (256, 6, 70, False),
                                           (257, 6, 140, True), (700, 5, 40, False), (1030, 4, 65, False)])
def test_dense_pairs(h, nev, m, delta):
    from paper_2001_07428_gb300.solver import JTRLan
    A11, A12 = inputs.dense_jsym(h, 7 + h)
    v1 = None
    if delta:
        v1 = np.zeros(2 * h, dtype=np.complex128)
        v1[1] = 1.0
        v1[0] = -0.0
    s = JTRLan("dense", A11=A11, A12=A12, nev=nev, m=m, mwin=m // 2, tol=1e-9, v1=v1, device="cuda:0")
    s.solve()
    ev, X, res = s.pairs(with_partners=True)
    s.close()
    A = np.block([[A11, A12], [A12.conj().T, A11.T]])
    X = X.cpu().numpy()
    scale = np.abs(ev).max()
    exact = np.linalg.eigvalsh(A)[::2][:nev] if h <= 700 else None
    if exact is not None:
        assert np.abs(ev - exact).max() <= 1e-10 * scale
    Y = X[:, :nev]
    r = np.linalg.norm(A @ Y - Y * ev, axis=0)
    assert (r < 1e-9 + 1e-12 * scale).all() and (res < 1e-9).all()
    # [X, J X*] orthonormal: the integer dots hold V^H V = I and W^H V = 0 at FP64 level (about 1e-14)
    assert np.abs(X.conj().T @ X - np.eye(2 * nev)).max() < 1e-11
