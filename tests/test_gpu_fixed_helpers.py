"""The device helpers of csrc/fixed.cuh against exact Python integers, and one Gram-Schmidt step of
csrc/gsfx.cu on chosen columns (tests/cuda/fixed_probe.cu, compiled here)."""
import ctypes
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2001_07428_gb300 import build as B
    out = str(tmp_path_factory.mktemp("probe") / "fixed_probe.so")
    subprocess.run([B.nvcc(), *B.ARCH, "-O3", "-std=c++17", "-shared", "-cudart", "shared", "-Xcompiler", "-fPIC",
                    "-I", os.path.join(B.ROOT, "include"), "-o", out, os.path.join(HERE, "cuda", "fixed_probe.cu"),
                    os.path.join(B.CSRC, "launch.cu"), "-Xlinker", "-rpath," + B.cuda_lib_dir()], check=True)
    torch.cuda.init()
    return ctypes.CDLL(out)


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def _values(K):
    """Doubles below 2^(K - 1023): full, short and far smaller significands, zeros, subnormals."""
    rng = np.random.default_rng(K)
    e = K - 1023
    x = np.ldexp(rng.uniform(-1, 1, 400), e) * 2.0 ** -rng.integers(0, 64, 400).astype(float)
    x = np.concatenate([x, [0.0, -0.0, 5e-324, -5e-324, 2.0 ** -1023, -(2.0 ** -1022 - 2.0 ** -1074)],
                        np.ldexp([1.0 - 2.0 ** -53, -(1.0 - 2.0 ** -53), 0.5, -0.5, 2.0 ** -60, -(2.0 ** -60), 2.0 ** -61], e)])
    return x[np.abs(x) < math.ldexp(1.0, e)] if e > -1021 else np.array([0.0, -0.0, 5e-324, -(2.0 ** -1023)])


def _limbs(x, e):
    if abs(x) < 2.0 ** -1022:
        return 0, 0
    f = 2 * int(abs(Fraction(x)) * Fraction(2) ** (55 - e)) + 1
    f = -f if x < 0 else f
    return f >> 28, f & ((1 << 28) - 1)


@pytest.mark.parametrize("K", [1, 30, 1000, 1016, 1023, 1024, 1300])
def test_limbs_and_store(probe, K):
    x = _values(K)
    d, n, e = _dev(x), len(x), K - 1023
    lim = torch.empty((n, 2), dtype=torch.int32, device="cuda:0")
    assert probe.probe_limbs(_p(d), n, K, _p(lim)) == 0
    assert [tuple(r) for r in lim.cpu().tolist()] == [_limbs(v, e) for v in x]
    if K < 1000:
        return
    F = torch.empty(n, dtype=torch.int64, device="cuda:0")
    back = torch.empty(n, dtype=torch.float64, device="cuda:0")
    assert probe.probe_store(_p(d), n, K, _p(F), _p(lim), _p(back)) == 0
    for v, f, (h, l), b in zip(x, F.cpu().tolist(), lim.cpu().tolist(), back.cpu().tolist()):
        q = Fraction(v) * Fraction(2) ** (60 - e)
        want = math.floor(abs(q) + Fraction(1, 2)) * (-1 if q < 0 else 1) if abs(v) >= 2.0 ** -1022 else 0
        assert f == want and (h, l) == ((f + 8) >> 32, ((f + 8) & 0xffffffff) >> 4)
        assert b == float(Fraction(f) * Fraction(2) ** (e - 60))


@pytest.mark.parametrize("cnt", [1, 2, 32, 33, 700])
def test_warp_sums_of_zeros(probe, cnt):
    """Zeros and subnormals count as zero."""
    out = torch.empty(2, dtype=torch.float64, device="cuda:0")
    for x in (np.zeros(cnt), -np.zeros(cnt), np.full(cnt, 5e-324)):
        assert probe.probe_sum(_p(_dev(x)), cnt, _p(out)) == 0
        assert out.cpu().tolist() == [0.0, 0.0]


@pytest.mark.parametrize("cnt", [1, 2, 32, 33, 700])
def test_warp_sum_error(probe, cnt):
    """A term's limbs and a lane's dropped bit are each below 2^-56 of the scale, which is below twice the largest
    term: 2^-54 of that a term; the result is rounded once."""
    rng = np.random.default_rng(cnt)
    out = torch.empty(2, dtype=torch.float64, device="cuda:0")
    for x in (rng.standard_normal(cnt), rng.standard_normal(cnt) * 2.0 ** rng.integers(-80, 1, cnt).astype(float),
              np.full(cnt, 1.0 - 2.0 ** -53)):
        assert probe.probe_sum(_p(_dev(x)), cnt, _p(out)) == 0
        top = np.abs(x).max()
        for got, part in zip(out.cpu().tolist(), (x, x[:32])):
            want = sum(map(Fraction, part), Fraction(0))
            assert abs(Fraction(got) - want) <= len(part) * Fraction(2.0 ** -54) * Fraction(top) + abs(want) * Fraction(1, 2 ** 53)


def _pair(v):
    h = len(v) // 2
    return np.concatenate([-v[h:].conj(), v[:h].conj()])


def _step(probe, X, y, rpb):
    n, cols = X.shape
    d, w = _dev(X.T.copy()), _dev(y.copy())
    c = torch.zeros((cols, 4), dtype=torch.float64, device="cuda:0")
    assert probe.probe_step(_p(d), ctypes.c_longlong(n), cols, rpb, _p(w), _p(c)) == 0
    c = c.cpu().numpy()
    return w.cpu().numpy(), c[:, 0] + 1j * c[:, 1], c[:, 2] + 1j * c[:, 3]


def test_full_sums(probe):
    """512 row pairs of one block, every component just below its scale: 64 products a lane in each sum."""
    n = 1024
    t = 1.0 - 2.0 ** -53
    for sx in (1, -1):
        X = np.full((n, 1), t * (1 + 1j))
        y = np.full(n, sx * t * (1 + 1j))
        _, cv, cw = _step(probe, X, y, 512)
        assert abs(cv[0] - sx * 2 * n * t * t) <= 2.0 ** -53 * 4 * n and cw[0] == 0.0


@pytest.mark.parametrize("n,rpb", [(1 << 16, 4096), (1 << 18, 4096)])     # one cluster; a grid; eight chunks each
@pytest.mark.parametrize("spread", [False, True])
def test_update_error(probe, n, rpb, spread):
    """y - V c_v - W c_w for coefficients just below the line between a column's short and long form.  With
    `spread` one column has an entry near 1 and the others, like any vector of 2^18 entries, none above 2^-7."""
    cols = 4
    rng = np.random.default_rng(n + spread)
    X = rng.standard_normal((n, cols)) + 1j * rng.standard_normal((n, cols))
    if spread:
        X[5, 1] = 10.0 * math.sqrt(n)
    r = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    done = []
    for i in range(cols + 1):                     # orthonormal, with the partners
        v = X[:, i] if i < cols else r
        for _ in range(2):
            for u in done:
                v = v - u * np.vdot(u, v)
        v = v / np.linalg.norm(v)
        done += [v, _pair(v)]
        if i < cols:
            X[:, i] = v
        else:
            r = v
    line = 2.0 ** -30 / (cols * (cols + 3))
    y = r.copy()
    for i in range(cols):
        f = rng.uniform(0.5, 0.69, 4) * line      # components below the line
        y = y + X[:, i] * (f[0] + 1j * f[1]) + _pair(X[:, i]) * (f[2] - 1j * f[3])
    got, cv, cw = _step(probe, X, y, rpb)
    L = np.clongdouble
    want = y.astype(L)
    for i in range(cols):
        want = want - X[:, i].astype(L) * L(cv[i]) - _pair(X[:, i]).astype(L) * L(cw[i])
        assert max(abs(cv[i].real), abs(cv[i].imag), abs(cw[i].real), abs(cw[i].imag)) < line
    # the coefficients' short form 2^-50 / (j + 4), truncated V 2^-56 rho / (j + 4) (rho < 16: the peak of the
    # flattest column over its rms), and y rounded: 2^-53
    err = float(np.linalg.norm((got - want).astype(np.complex128)))
    assert err <= 2.0 ** -50 / (cols + 3) + 2.0 ** -52 / (cols + 3) + 2.0 ** -53, math.log2(err)
