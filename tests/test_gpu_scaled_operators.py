"""Operators whose norm lies beyond FP32's range, in plain FP64: a power of two changes no significand, so the
eigenvalues scale and the pairs stay as orthonormal as those of the operator itself."""
import numpy as np
import pytest

from paper_2001_07428_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TWO = 2.0 ** 200


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2001_07428_gb300 import binding
    binding.load()


def _check(ev, X, A11, A12, nev):
    A = np.block([[A11, A12], [A12.conj().T, A11.T]])
    exact = np.linalg.eigvalsh(A)[::2][:nev]
    # 1e-9 ||A|| of residual leaves 1e-18 ||A|| / gap in the eigenvalue; 4e-13 is the form's own error
    assert np.abs(ev / TWO - exact).max() <= 1e-12 * np.abs(exact).max()
    h = A11.shape[0]
    Z = np.concatenate([X, np.concatenate([-X[h:].conj(), X[:h].conj()])], axis=1)
    assert np.abs(Z.conj().T @ Z - np.eye(2 * nev)).max() < 1e-12


@pytest.mark.parametrize("gs_split", [False, True])
@pytest.mark.parametrize("h", [60, 400])       # one cluster of blocks; a grid
def test_single(h, gs_split):
    from paper_2001_07428_gb300.solver import JTRLan
    A11, A12 = inputs.dense_jsym(h, 3)
    s = JTRLan("dense", A11=A11 * TWO, A12=A12 * TWO, nev=6, m=24, mwin=12, tol=1e-9 * TWO, gs_split=gs_split,
               max_restarts=200, device="cuda:0")
    s.solve()
    ev, X, _ = s.pairs()
    s.close()
    _check(ev, X.cpu().numpy(), A11, A12, 6)


def test_batch():
    from paper_2001_07428_gb300.solver import JTRLanBatch
    blocks = [inputs.dense_jsym(h, 40 + h) for h in (33, 60, 130)]
    b = JTRLanBatch([a * TWO for a, _ in blocks], [k * TWO for _, k in blocks], nev=6, m=24, mwin=12, tol=1e-9 * TWO,
                    max_restarts=200, device="cuda:0")
    b.solve()
    ev, _, _ = b.results()
    for i, (a, k) in enumerate(blocks):
        _check(ev[i], b.vectors(i).cpu().numpy(), a, k, 6)
    b.close()
