"""The fixed-point copies of the links (plain FP64, stencil) are kept only where they are used, and give their
memory back to the context's own needs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2001_07428_gb300 import binding
    binding.load()


def _links(vol):
    g = torch.Generator(device="cuda:0").manual_seed(7)
    return [torch.randn((4, vol, 3, 3), dtype=torch.complex128, device="cuda:0", generator=g) * 0.3 for _ in range(2)]


def _solver(dims, links, **kw):
    from paper_2001_07428_gb300.solver import JTRLan
    return JTRLan("stencil", dims=dims, m0=8.5, kappa=0.3, U=links[0], W=links[1], nev=2, m=8, mwin=4, tol=1e-8,
                  device="cuda:0", **kw)


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_kept_where_used():
    dims, vol = (16, 16, 16, 16), 16 ** 4
    links = _links(vol)
    copies, vector = 2 * 36 * vol * 16, 6 * vol * 16
    filt = dict(filter_final_coeffs=np.linspace(1.0, 0.1, 5), filter_window=(1.0, 20.0))
    used = {}
    for name, kw in (("warm-up", {}), ("plain", {}), ("invert", dict(invert=True)), ("filtered", filt)):
        before = _free()
        s = _solver(dims, links, **kw)
        used[name] = before - _free()
        s.close()
    # CG keeps three vectors, a certifying filter four; everything else is the same but small arrays
    assert used["invert"] <= used["plain"] - copies + 3 * vector + 16 * MB
    assert used["filtered"] <= used["plain"] - copies + 4 * vector + 16 * MB


def test_memory_given_back():
    """With less room than a filter's four vectors (268 MB) left on the GPU, jtrlan_set_filter takes that of the
    copies (764 MB); the products of the Lanczos steps go on in FP64 multiply-adds."""
    from paper_2001_07428_gb300 import binding as B
    dims, vol = (24, 24, 24, 48), 24 ** 3 * 48
    links = _links(vol)
    s = _solver(dims, links)
    want = s.bounds(8)
    coeffs = np.linspace(1.0, 0.1, 5)
    del links
    torch.cuda.empty_cache()
    fill = torch.empty(_free() - 160 * MB, dtype=torch.uint8, device="cuda:0")
    try:
        B.jtrlan_set_filter(s.ctx, coeffs, (1.0, 20.0))
        got = s.bounds(8)
    finally:
        del fill
        torch.cuda.empty_cache()
        s.close()
    # the two products agree to a few ulp of ||A||; 1e-12 is what the eigenvalues of an 8 x 8 T leave of that
    assert abs(got[0] - want[0]) <= 1e-12 * abs(want[1]) and abs(got[1] - want[1]) <= 1e-12 * abs(want[1])
