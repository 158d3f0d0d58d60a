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


# volumes: below, at and beyond one 32-site block, beyond a block per SM; extents 1 and 2
@pytest.mark.parametrize("dims", [(2, 2, 2, 4), (1, 3, 4, 5), (3, 5, 2, 7), (7, 6, 9, 13), (8, 8, 8, 10)])
def test_stencil_product_in_a_solve(dims):
    """The integer stencil product of the FP64 form: two Lanczos steps' alpha and beta, through
    jtrlan_bounds (a 2 x 2 T), against the oracle's product."""
    from oracle import jsym
    from paper_2001_07428_gb300.solver import JTRLan
    U, W = inputs.stencil_links(dims, 3)
    n = 6 * inputs.lattice_volume(dims)
    s = JTRLan("stencil", dims=dims, m0=8.5, kappa=0.3, U=U, W=W, nev=1, m=2, mwin=1, tol=1e-8, device="cuda:0")
    lo, hi = s.bounds(2)
    s.close()
    # the library's start vector: splitmix64 on seed + 2 i and seed + 2 i + 1, to [-1, 1)
    z = (np.arange(2 * n, dtype=np.uint64) + np.uint64(0xb07d5)) + np.uint64(0x9E3779B97F4A7C15)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    z = z ^ (z >> np.uint64(31))
    r = (z >> np.uint64(11)).astype(np.float64) * (2.0 / 9007199254740992.0) - 1.0
    v = r[0::2] + 1j * r[1::2]
    V, T = [v / np.linalg.norm(v)], np.zeros((3, 3))
    for j in range(2):
        y = jsym.stencil_matvec(U, W, dims, 8.5, 0.3, V[j])
        T[j, j] = np.vdot(V[j], y).real
        for _ in range(2):
            for q in V:
                w = np.concatenate([-np.conj(q[n // 2:]), np.conj(q[:n // 2])])
                y = y - q * np.vdot(q, y)
                y = y - w * np.vdot(w, y)
        T[j + 1, j] = T[j, j + 1] = np.linalg.norm(y)
        V.append(y / T[j + 1, j])
    ev, Z = np.linalg.eigh(T[:2, :2])
    beta = T[2, 1]
    # products, dots and norms at a few ulp of ||A||, amplified by the 2 x 2 solve: 1e-12 ||A|| is 4,500 ulp
    assert abs(lo - (ev[0] - beta * abs(Z[1, 0]))) < 1e-12 * abs(hi)
    assert abs(hi - (ev[1] + beta)) < 1e-12 * abs(hi)
