"""Kernels set up while their predecessor still runs must see all of its writes: results without any
synchronisation between launches equal, bit for bit, those with one after every launch."""
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


def _solver(kind, size, precision, **kw):
    from paper_2001_07428_gb300.solver import JTRLan
    par = dict(nev=4, m=20, mwin=8, tol=1e-8, precision=precision, device="cuda:0", **kw)
    if kind == "dense":
        A11, A12 = inputs.dense_jsym(size, 3)
        return JTRLan("dense", A11=A11, A12=A12, **par)
    U, W = inputs.stencil_links(size, seed=2)
    return JTRLan("stencil", dims=size, m0=8.5, kappa=0.3, U=U, W=W, **par)


@pytest.mark.parametrize("kind,size,precision", [
    ("dense", 25, "fp64"), ("dense", 100, "fp64"), ("stencil", (2, 2, 2, 2), "fp64"), ("stencil", (8, 8, 8, 8), "fp64"),
    ("stencil", (16, 16, 16, 16), "fp64"), ("stencil", (3, 5, 4, 7), "mixed"), ("stencil", (16, 16, 16, 16), "mixed")])
def test_chained_products(kind, size, precision):
    s = _solver(kind, size, precision)
    x0 = torch.from_numpy(inputs.random_vector(s.n, 5)).to("cuda:0")

    def chain(sync):
        x = x0
        for i in range(24):
            y = s.apply(x)
            if sync:
                torch.cuda.synchronize()
            x = y * (1.0 / 16) if i % 3 == 0 else y      # an elementwise kernel between some products
            if sync:
                torch.cuda.synchronize()
        return x.cpu().numpy().tobytes()

    want = chain(True)
    for _ in range(3):
        assert chain(False) == want
    s.close()


@pytest.mark.parametrize("kind,size,kw", [
    ("dense", 60, dict(precision="fp64")),
    ("stencil", (4, 4, 4, 4), dict(precision="fp64")),
    ("stencil", (8, 8, 8, 8), dict(precision="fp64")),
    ("stencil", (4, 4, 4, 4), dict(precision="mixed_reorth")),
    ("stencil", (8, 8, 4, 4), dict(precision="mixed_reorth", links_dtype="c64"))])
def test_steps_with_and_without_events_between(kind, size, kw):
    """The profile records an event around every launch, so nothing is set up early there."""
    out = []
    for profile in (True, False, False):
        s = _solver(kind, size, profile=profile, **kw)
        s.solve()
        ev, X, res = s.pairs()
        out.append((ev.tobytes(), X.cpu().numpy().tobytes(), res.tobytes()))
        s.close()
    assert out[1] == out[0] and out[2] == out[0]


@pytest.mark.parametrize("dims,links,degree", [
    ((2, 2, 2, 2), "c128", 1), ((3, 5, 4, 7), "c64", 9), ((8, 8, 8, 8), "c128", 16), ((16, 16, 16, 16), "c64", 17)])
def test_filter_chain(dims, links, degree):
    """The fused recurrence, whose vectors pass from launch to launch: repeated calls agree bit for bit,
    alone and with other products of the stream between them."""
    coeffs = np.linspace(1.0, 0.1, degree + 1)
    s = _solver("stencil", dims, "mixed_reorth", links_dtype=links, filter_final_coeffs=coeffs, filter_window=(2.0, 20.0))
    v = torch.from_numpy(inputs.random_vector(s.n, 7)).to("cuda:0")
    torch.cuda.synchronize()
    want = s.apply_filter(v).cpu().numpy().tobytes()
    for _ in range(3):
        a = s.apply_filter(v)
        b = s.apply_filter(a)
        c = s.apply_filter(v)
        assert a.cpu().numpy().tobytes() == want
        assert c.cpu().numpy().tobytes() == want
        assert bool(torch.isfinite(torch.view_as_real(b)).all())
    s.close()


@pytest.mark.parametrize("links", ["c64", "c128"])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (3, 3, 3, 3), (11, 9, 13, 7), (16, 16, 16, 5), (13, 13, 13, 13), (16, 16, 16, 8)])
def test_filter_splits_against_fp64(dims, links):
    """Each block split of the fused step against the FP64 filter.  A step's products are good to 2^-40 of
    the sum of their magnitudes, which is below 100 half-widths of the window here, and the recurrence
    carries a step's error on at most degree times."""
    degree = 9
    kw = dict(links_dtype=links, filter_final_coeffs=np.linspace(1.0, 0.1, degree + 1), filter_window=(1.3, 18.7))
    out = []
    for precision in ("fp64", "mixed_reorth"):
        s = _solver("stencil", dims, precision, **kw)
        v = torch.from_numpy(inputs.random_vector(s.n, 7)).to("cuda:0")
        out.append(s.apply_filter(v).cpu().numpy())
        s.close()
    assert np.abs(out[1] - out[0]).max() <= degree ** 2 * 100 * 2.0 ** -40 * np.abs(out[0]).max()
