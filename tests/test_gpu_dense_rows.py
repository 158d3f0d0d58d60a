"""The dense product at the edges of its splits: one row a block up to eight rows for every SM, the last
lane of a warp and of a block's columns, and the first size of the other kernel."""
import numpy as np
import pytest

from oracle import jsym
from paper_2001_07428_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("h", [7, 31, 32, 33, 127, 128, 129, 500, "last", "next"])
def test_dense_product(h, precision):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2001_07428_gb300.solver import JTRLan
    if not isinstance(h, int):
        h = 8 * torch.cuda.get_device_properties(0).multi_processor_count + (h == "next")
    A11, A12 = inputs.dense_jsym(h, 4)
    x = inputs.random_vector(2 * h, 6)
    s = JTRLan("dense", A11=A11, A12=A12, nev=1, m=6, mwin=2, tol=1e-4, precision=precision, device="cuda:0")
    y = s.apply(torch.from_numpy(x).to("cuda:0")).cpu().numpy()
    s.close()
    bound = np.abs(A11) @ np.abs(x[:h]) + np.abs(A12) @ np.abs(x[h:]), np.abs(A11) @ np.abs(x[h:]) + np.abs(A12) @ np.abs(x[:h])
    eps = 2.0 ** (-52 if precision == "fp64" else -23)
    # a complex sum of 2 h products: 8 h roundings at most on any path, and those of rounding the inputs
    assert (np.abs(y - jsym.dense_matvec(A11, A12, x)) <= (8 * h + 8) * eps * np.concatenate(bound)).all()


@pytest.mark.parametrize("h", [40, 129, 700])
def test_alpha_of_the_row_split(h):
    """Pairs of a solve, whose alphas are sums over the rows' partials, against the CPU product."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2001_07428_gb300.solver import JTRLan
    A11, A12 = inputs.dense_jsym(h, 4)
    v = inputs.random_vector(2 * h, 9)
    s = JTRLan("dense", A11=A11, A12=A12, nev=2, m=min(30, h - 2), mwin=6, tol=1e-10, device="cuda:0", v1=v)
    s.solve()
    ev, X, res = s.pairs()
    X = X.cpu().numpy()
    s.close()
    for i in range(2):
        r = jsym.dense_matvec(A11, A12, X[:, i]) - ev[i] * X[:, i]
        assert np.linalg.norm(r) <= 2e-10 + 1e-13 * np.abs(ev).max() * h
