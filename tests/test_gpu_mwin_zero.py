"""mwin = 0 (Algorithm 1 allows it): a restart in which nothing converged keeps no column but v_{m+1}."""
import ctypes

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


@pytest.mark.parametrize("precision", ["fp64", "mixed_reorth"])
@pytest.mark.parametrize("gs_split", [False, True])
def test_restart_without_a_kept_column(precision, gs_split):
    """Three restarts of 14 steps of a spectrum of 64 pairs to 1e-12: none converges, each takes m steps
    (Algorithm 1, k = min(icnv + mwin, m - 1) = 0)."""
    from paper_2001_07428_gb300 import binding as B
    from paper_2001_07428_gb300.solver import JTRLan
    A11, A12 = inputs.dense_jsym(64, 5)
    s = JTRLan("dense", A11=A11, A12=A12, nev=2, m=14, mwin=0, tol=1e-12, max_restarts=3, precision=precision,
               gs_split=gs_split, device="cuda:0")
    st = B.jtrlan_stats()
    assert B.load().jtrlan_solve(s.ctx, ctypes.byref(st)) == B.JTRLAN_ENOCONV
    assert (st.n_restarts, st.n_matvec, st.icnv) == (3, 42, 0)
    s.close()
