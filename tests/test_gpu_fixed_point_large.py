"""The FP64 forms' integer sums beyond one chunk of 512: batched operators of more than 512 rows a half (more
than a block's threads too), separate Gram-Schmidt launches whose row blocks take several chunks, and a batched
operator whose rows differ by many orders."""
import numpy as np
import pytest

from paper_2001_07428_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2001_07428_gb300 import binding
    binding.load()


def _assemble(a, k):
    return np.block([[a, k], [k.conj().T, a.T]])


@pytest.mark.parametrize("threads", [256, 512])
def test_batch_beyond_one_chunk(threads):
    from paper_2001_07428_gb300.solver import JTRLanBatch
    blocks = [inputs.dense_jsym(h, 70 + h) for h in (513, 550, 512, 40)]
    b = JTRLanBatch([a for a, _ in blocks], [k for _, k in blocks], nev=4, m=24, mwin=12, tol=1e-9, device="cuda:0")
    b.set_shape(threads, 1)
    b.solve()
    ev, res, _ = b.results()
    for i, (a, k) in enumerate(blocks):
        A, h = _assemble(a, k), a.shape[0]
        lam = np.linalg.eigvalsh(A)
        X = b.vectors(i).cpu().numpy()
        scale = np.abs(lam).max()
        assert np.abs(ev[i] - lam[::2][:4]).max() <= 1e-12 * scale and res[i].max() < 1e-9
        assert np.linalg.norm(A @ X - X * ev[i], axis=0).max() < 1e-9 + 1e-13 * scale
        Z = np.concatenate([X, np.concatenate([-X[h:].conj(), X[:h].conj()])], axis=1)
        assert np.abs(Z.conj().T @ Z - np.eye(8)).max() < 1e-12
    b.close()


def test_batch_graded():
    """Rows and columns scaled from 1 down to 1e-6 (entries to 1e-12 of the largest).  The operator is rounded
    2^-57 below its largest entry, which moves eigenvalues and residuals by at most n 2^-57 max|a|; FP64 results
    are good to a few n u ||A||."""
    from paper_2001_07428_gb300.solver import JTRLanBatch
    h = 120
    a, k = inputs.dense_jsym(h, 9)
    d = 10.0 ** -np.linspace(0.0, 6.0, h)
    a, k = a * d[:, None] * d, k * d[:, None] * d
    A = _assemble(a, k)
    lam = np.linalg.eigvalsh(A)
    b = JTRLanBatch([a], [k], nev=4, m=24, mwin=12, tol=1e-10, device="cuda:0")
    b.solve()
    ev, res, _ = b.results()
    X = b.vectors(0).cpu().numpy()
    scale = np.abs(lam).max()
    assert np.abs(ev[0] - lam[::2][:4]).max() <= 2 * h * 2.0 ** -53 * scale
    true = np.linalg.norm(A @ X - X * ev[0], axis=0)
    assert np.abs(true - res[0]).max() <= 2 * h * 2.0 ** -53 * scale and res[0].max() < 1e-10
    b.close()


def test_split_steps_of_several_chunks():
    """20^4: 790 row pairs for each of the 608 blocks of the separate launches, 1600 for those of the single one."""
    from paper_2001_07428_gb300.solver import JTRLan
    dims, vol = (20, 20, 20, 20), 20 ** 4
    g = torch.Generator(device="cuda:0").manual_seed(3)
    U, W = (torch.randn((4, vol, 3, 3), dtype=torch.complex128, device="cuda:0", generator=g) * 0.4 for _ in range(2))
    out = []
    for split in (False, True):
        s = JTRLan("stencil", dims=dims, m0=8.5, kappa=0.3, U=U, W=W, nev=1, m=12, mwin=1, tol=1e-8, gs_split=split,
                   device="cuda:0")
        out.append(s.bounds(12))
        s.close()
    # the same exact sums, cut into other partials: a few ulp of ||A|| a step
    assert abs(out[0][0] - out[1][0]) <= 1e-13 * out[0][1] and abs(out[0][1] - out[1][1]) <= 1e-13 * out[0][1]
