"""The work that programs have this library do, as cases that can be timed and compared.

A program holds an operator (the lattice stencil's links, or the blocks of a dense matrix) and a context
or batch made from it, and calls the product A x, the polynomial filter p(A) x, the spectral bounds, the
whole solve or the batched solve; the restart rotation has an entry point of its own.  The listed cases
are those calls at the sizes of the library's own workloads (``paper_2001_07428_gb300.inputs.WORKLOADS``),
from the smallest lattice of the tests to the benchmark's; ``draw`` spreads over the same ranges.

Operators have the workloads' distributions -- Haar SU(3) links U, complex Gaussian W; dense blocks
A11 = (G + G^H)/2, A12 = (K - K^T)/2 with Gaussian G, K -- and are made on the GPU from the seed.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2001_07428_gb300 import binding as B
from paper_2001_07428_gb300 import inputs
from paper_2001_07428_gb300.solver import JTRLan, JTRLanBatch

DEV = "cuda"
C128, F64 = torch.complex128, torch.float64


def listed():
    return [
        # the product on the smallest lattice of the tests: a call that is all latency
        dict(name="apply_f64_4x4x4x4", kind="apply", lx=4, ly=4, lz=4, lt=4, precision="fp64", links="c128"),
        # the FP32 product of the mixed forms on the benchmark's lattice
        dict(name="apply_f32_24x24x24x48", kind="apply", lx=24, ly=24, lz=24, lt=48, precision="mixed_reorth",
             links="c64"),
        # p(A) x of the certifying phase on the benchmark's lattice: where most of its solve goes
        dict(name="filter_24x24x24x48", kind="filter", lx=24, ly=24, lz=24, lt=48, links="c64", degree=64),
        # the same on a lattice of odd extents with complex128 links, a lower degree
        dict(name="filter_9x11x13x15", kind="filter", lx=9, ly=11, lz=13, lt=15, links="c128", degree=33),
        # 200 Lanczos steps on the benchmark's lattice (m = 200): products and reorthogonalisation against
        # a basis that grows to its full size, in the compensated form
        dict(name="bounds_24x24x24x48", kind="bounds", lx=24, ly=24, lz=24, lt=48, precision="mixed_reorth",
             links="c64", steps=200),
        # the same in plain FP64 on the next smaller lattice of the workloads (m = 120)
        dict(name="bounds_f64_16x16x16x16", kind="bounds", lx=16, ly=16, lz=16, lt=16, precision="fp64",
             links="c128", steps=120),
        # the restart rotation at the benchmark's size
        dict(name="rotate_24x24x24x48", kind="rotate", n=3981312, m=200, kk=100),
        # whole solves: the dense workload, the 8^4 lattice in plain FP64, and 16^4 with the polynomial
        # filter in the compensated form (the benchmark's method, one lattice down)
        dict(name="solve_dense_n200", kind="solve_dense", h=100, nev=10, m=30, mwin=15, precision="fp64"),
        dict(name="solve_f64_8x8x8x8", kind="solve", lx=8, ly=8, lz=8, lt=8, nev=20, m=60, mwin=30,
             precision="fp64", links="c128", filtered=False),
        dict(name="solve_filtered_16x16x16x16", kind="solve", lx=16, ly=16, lz=16, lt=16, nev=50, m=120, mwin=60,
             precision="mixed_reorth", links="c64", filtered=True),
        # the batched workload, 512 dense operators of uneven order, in both forms
        dict(name="batch_f64_512", kind="batch", count=512, nlo=64, nhi=512, precision="fp64"),
        dict(name="batch_mixed_512", kind="batch", count=512, nlo=64, nhi=512, precision="mixed_reorth"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lattice(rng, lo, hi):
    """Four extents, each on its own, whose volume is spread over [lo, hi] on a logarithm."""
    vol = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    while True:
        w = [rng.uniform(0.8, 1.25) for _ in range(4)]
        scale = (vol / math.prod(w)) ** 0.25
        d = [max(2, int(round(scale * v))) for v in w]
        if math.prod(d) <= hi:
            return dict(lx=d[0], ly=d[1], lz=d[2], lt=d[3])


def draw(rng):
    kind = rng.choice(["apply", "filter", "bounds", "rotate", "solve_dense", "solve", "solve", "batch"])
    form = rng.choice(["fp64", "mixed_reorth"])
    links = rng.choice(["c64", "c128"])
    if kind == "apply":
        return dict(kind=kind, **_lattice(rng, 256, 663552), precision=form, links=links)
    if kind == "filter":
        return dict(kind=kind, **_lattice(rng, 1296, 663552), links=links, degree=rng.randint(8, 64))
    if kind == "bounds":
        if form == "fp64":   # plain FP64 is kept to the lattices it is used on
            return dict(kind=kind, **_lattice(rng, 1296, 65536), precision=form, links=links, steps=rng.randint(20, 120))
        return dict(kind=kind, **_lattice(rng, 1296, 400000), precision=form, links=links, steps=rng.randint(20, 200))
    if kind == "rotate":
        m = rng.randint(24, 220)
        return dict(kind=kind, n=2 * _log(rng, 12000, 1900000), m=m, kk=rng.randint(8, m // 2 + 4))
    if kind == "solve_dense":
        nev = rng.randint(4, 12)
        return dict(kind=kind, h=rng.randint(60, 256), nev=nev, m=3 * nev + rng.randint(0, 8), mwin=nev + rng.randint(2, 5),
                    precision=form)
    if kind == "solve":
        nev = rng.randint(8, 24)
        return dict(kind=kind, **_lattice(rng, 256, 5000), nev=nev, m=3 * nev + rng.randint(0, 9),
                    mwin=nev + rng.randint(5, 10), precision=form, links=links, filtered=False)
    lo = 2 * rng.randint(28, 60)
    return dict(kind="batch", count=rng.randint(100, 500), nlo=lo, nhi=2 * rng.randint(lo, 256), precision=form)


# ---------------------------------------------------------------- inputs
M0, KAPPA = 8.5, 0.3
# The filter's window [a, b] holds the spectrum of these operators (about 1.6 to 18.7 at every size:
# the hopping term's norm does not depend on the lattice), and its cut lies in the lower tail where the
# learned filter puts it for 50 pairs at 16^4.
WINDOW, CUT = (1.30, 18.75), -0.9735


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _gauss(g, shape):
    return torch.complex(torch.randn(shape, dtype=F64, device=DEV, generator=g),
                         torch.randn(shape, dtype=F64, device=DEV, generator=g))


def _dims(case):
    return case["lx"], case["ly"], case["lz"], case["lt"]


def _links(case, seed):
    """U: Haar SU(3) (rows of a Gaussian matrix orthonormalised, the last one completed to determinant
    1); W: complex Gaussian; shape (4, V, 3, 3)."""
    vol, g = math.prod(_dims(case)), _gen(seed)
    a, b = _gauss(g, (4 * vol, 3)), _gauss(g, (4 * vol, 3))
    a = a / torch.linalg.vector_norm(a, dim=1, keepdim=True)
    b = b - a * (a.conj() * b).sum(1, keepdim=True)
    b = b / torch.linalg.vector_norm(b, dim=1, keepdim=True)
    u = torch.stack([a, b, torch.linalg.cross(a, b).conj()], dim=1).reshape(4, vol, 3, 3).contiguous()
    w = _gauss(g, (4, vol, 3, 3))
    if case.get("links") == "c64":
        u, w = u.to(torch.complex64).to(C128), w.to(torch.complex64).to(C128)
    return u, w


def _damped_step(tau, degree):
    """Jackson-damped Chebyshev coefficients of the step [x <= tau] (FP64)."""
    n, k = degree + 1, np.arange(degree + 1)
    q = math.pi / (n + 1)
    jackson = ((n - k + 1) * np.cos(q * k) + np.sin(q * k) / math.tan(q)) / (n + 1)
    th = math.acos(tau)
    c = np.empty(n)
    c[0] = (math.pi - th) / math.pi
    c[1:] = -2.0 * np.sin(k[1:] * th) / (math.pi * k[1:])
    return jackson * c


def _vector(n, seed):
    return _gauss(_gen(seed + 7919), (n,))


def _filtered(case, seed):
    """A unit vector that has been through p(A) once, as the Lanczos vectors of a filtered solve have (on a
    vector without it p(A) x is what little p leaves, and its rounding)."""
    a = _Stencil(case, seed)
    y = a.poly(_vector(6 * a.vol, seed), _damped_step(CUT, case["degree"]))
    return y / torch.linalg.vector_norm(y)


def _dense(h, g):
    a, k = _gauss(g, (h, h)), _gauss(g, (h, h))
    return 0.5 * (a + a.conj().T), 0.5 * (k - k.T)


def _batch_blocks(case, seed):
    g = _gen(seed)
    return [_dense(int(n) // 2, g) for n in inputs.batched_dense_sizes(case["count"], case["nlo"], case["nhi"], 2)]


def _rotate_inputs(case, seed):
    """A basis as (hi, lo) FP32 pairs with entries of a unit vector's size, and orthonormal columns Z."""
    n, m, g = case["n"], case["m"], _gen(seed)
    v = torch.empty((m, n, 4), dtype=torch.float32, device=DEV)
    for j in range(m):
        hi = torch.randn((n, 2), device=DEV, generator=g) / math.sqrt(2 * n)
        v[j, :, :2] = hi
        v[j, :, 2:] = (torch.rand((n, 2), device=DEV, generator=g) - 0.5) * 2.0 ** -24 * hi
    z = torch.linalg.qr(torch.randn((m, m), dtype=F64, device=DEV, generator=g))[0][:, :case["kk"]]
    return v, z.T.contiguous()          # row c holds column c of Z


def prepare(case, seed):
    kind = case["kind"]
    if kind == "rotate":
        v, z = _rotate_inputs(case, seed)
        return dict(case=case, v=v, z=z, out=torch.empty((case["kk"], case["n"]), dtype=C128, device=DEV))
    if kind == "batch":
        blocks = _batch_blocks(case, seed)
        b = JTRLanBatch([a for a, _ in blocks], [k for _, k in blocks], nev=8, m=24, mwin=12, tol=1e-8,
                        precision=case["precision"])
        b.set_shape(512, 1)             # the shape and tiles that tune() settles on for this workload
        b.set_tiles(2, 0)
        return dict(case=case, b=b)
    if kind == "solve_dense":
        a11, a12 = _dense(case["h"], _gen(seed))
        return dict(case=case, s=JTRLan("dense", A11=a11, A12=a12, nev=case["nev"], m=case["m"], mwin=case["mwin"],
                                        tol=1e-8, precision=case["precision"]))
    u, w = _links(case, seed)
    kw = dict(dims=_dims(case), m0=M0, kappa=KAPPA, U=u, W=w, tol=1e-8, links_dtype=case["links"])
    if kind == "solve":
        if case["filtered"]:
            kw.update(filter_final_coeffs=_damped_step(CUT, 64), filter_window=WINDOW)
        return dict(case=case, s=JTRLan("stencil", nev=case["nev"], m=case["m"], mwin=case["mwin"],
                                        precision=case["precision"], **kw))
    if kind == "bounds":
        return dict(case=case, s=JTRLan("stencil", nev=1, m=case["steps"], mwin=1, precision=case["precision"], **kw))
    if kind == "filter":
        kw.update(filter_final_coeffs=_damped_step(CUT, case["degree"]), filter_window=WINDOW)
        s = JTRLan("stencil", nev=1, m=8, mwin=1, precision="mixed_reorth", **kw)
        return dict(case=case, s=s, x=_filtered(case, seed))
    s = JTRLan("stencil", nev=1, m=8, mwin=1, precision=case["precision"], **kw)
    x = _vector(s.n, seed)
    return dict(case=case, s=s, x=x if case["precision"] == "fp64" else x.to(torch.complex64))


def _signed(x):
    """Eigenvectors (columns) with a definite sign.  The start vector is (1, ..., 1)/sqrt(n) and T is
    real, so sum(x) is real and the solve leaves only the sign of each x open."""
    return x * torch.sign(x.real.sum(0))


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "apply":
        x, s = state["x"], state["s"]
        y = torch.empty_like(x)
        B.jtrlan_apply(s.ctx, x.data_ptr(), y.data_ptr())
        return y
    if kind == "filter":
        return state["s"].apply_filter(state["x"])
    if kind == "bounds":
        return list(state["s"].bounds(case["steps"]))
    if kind == "rotate":
        out = state["out"]
        B.jtrlan_rotate_df(state["v"].data_ptr(), case["n"], case["m"], state["z"].data_ptr(), case["kk"],
                           out.data_ptr(), 0, torch.cuda.current_stream().cuda_stream)
        return out
    # the residual norms of converged pairs are left out of what a solve returns: they are noise below
    # tol, the part of A x - lambda x that rounding decides
    if kind == "batch":
        b = state["b"]
        b.solve()
        count = len(b.ns)
        ev = np.zeros((count, b.nev))
        B.jtrlan_batch_results(b.b, ev.ctypes.data_as(ctypes.c_void_p), None, None)
        # the vectors of all instances stay on the device; a program fetches those that it looks at
        return [ev] + [_signed(b.vectors(i)) for i in range(0, count, max(1, -(-count // 32)))]
    s = state["s"]
    s.solve()
    ev, x, _ = s.pairs()
    return [ev, _signed(x)]


# ---------------------------------------------------------------- the least work of a pass
def _stencil_bytes(case, link, vec, vectors=2):
    vol = math.prod(_dims(case))
    return vol * (72 * link + 6 * vectors * vec)


def _lanczos_work(case, steps_from_to, products, link, vec):
    """Lanczos steps j0..j1 (products of A each): the operator read per product, the basis read twice per
    step (inner products, update)."""
    vol = math.prod(_dims(case))
    j0, j1 = steps_from_to
    cols = sum(j + 1 for j in range(j0, j1))
    n = 6 * vol
    by = (j1 - j0) * products * vol * (72 * link + 12 * vec) + 2 * cols * n * 16
    fl = (j1 - j0) * products * vol * 2304 + cols * n * 32
    return by, fl


def work(case):
    kind = case["kind"]
    if kind == "rotate":
        n, m, kk = case["n"], case["m"], case["kk"]
        return dict(bytes=n * m * 16 + n * kk * 16 + m * kk * 8, flops=4.0 * n * m * kk)
    if kind == "batch":
        h = (case["nlo"] + case["nhi"]) / 4
        h2 = (case["nlo"] ** 2 + case["nlo"] * case["nhi"] + case["nhi"] ** 2) / 12
        steps, cols = 80, 80 * 18        # Lanczos steps of an instance (about), columns over them
        return dict(bytes=case["count"] * (32 * h2 + 2 * h * 8 * 16), flops=case["count"] * (steps * 32 * h2 + cols * 64 * h))
    if kind == "solve_dense":
        h = case["h"]
        return dict(bytes=32 * h * h + 2 * h * case["nev"] * 16, flops=3 * case["m"] * (32 * h * h + 64 * h * case["m"] * 0.7))
    f64 = case.get("precision", "mixed_reorth") == "fp64"
    c64 = case["links"] == "c64"
    vol = math.prod(_dims(case))
    if kind == "apply":
        return dict(bytes=_stencil_bytes(case, 16 if f64 else 8, 16 if f64 else 8), flops=2304.0 * vol)
    if kind == "filter":
        d = case["degree"]                # links, t_k, t_{k-1} and the sum read, t_{k+1} and the sum written
        return dict(bytes=d * _stencil_bytes(case, 8 if c64 else 16, 16, 5), flops=2304.0 * vol * d)
    link = 16 if f64 or not c64 else 8
    if kind == "bounds":
        by, fl = _lanczos_work(case, (0, case["steps"]), 1, link, 16)
        return dict(bytes=by, flops=fl)
    # a solve: about 3 bases' worth of steps at 16^4 with the filter, 12 without
    k, m = case["mwin"], case["m"]
    by, fl = _lanczos_work(case, (k, m), 64 if case["filtered"] else 1, link, 16)
    rep = 3 if case["filtered"] else 12
    return dict(bytes=rep * by, flops=rep * fl)


# ---------------------------------------------------------------- the same in 64 bits, without the library
class _Stencil:
    """y = A x of the lattice operator in plain torch (complex128)."""

    def __init__(self, case, seed):
        self.u, self.w = _links(case, seed)
        lx, ly, lz, lt = _dims(case)
        self.grid, self.vol = (lt, lz, ly, lx), lx * ly * lz * lt

    def hop(self, p, mu, step):
        return torch.roll(p.view(*self.grid, 3), -step, dims=3 - mu).reshape(self.vol, 3)

    def back(self, link, mu):
        return torch.roll(link[mu].view(*self.grid, 3, 3), 1, dims=3 - mu).reshape(self.vol, 3, 3)

    def __call__(self, x):
        mul = lambda a, p: (a * p[:, None, :]).sum(2)   # noqa: E731
        x1, x2 = x.view(2, self.vol, 3)
        y1, y2 = M0 * x1, M0 * x2
        for mu in range(4):
            u, ub, w, wb = self.u[mu], self.back(self.u, mu), self.w[mu], self.back(self.w, mu)
            f1, f2, b1, b2 = self.hop(x1, mu, 1), self.hop(x2, mu, 1), self.hop(x1, mu, -1), self.hop(x2, mu, -1)
            ubt, wbt = ub.transpose(1, 2), wb.transpose(1, 2)
            y1 = y1 + mul(u, f1) + mul(ubt.conj(), b1) + KAPPA * (mul(w, f2) - mul(wbt, b2))
            y2 = y2 + mul(u.conj(), f2) + mul(ubt, b2) - KAPPA * (mul(w.conj(), f1) - mul(wbt.conj(), b1))
        return torch.cat([y1.reshape(-1), y2.reshape(-1)])

    def poly(self, x, g):
        """sum_k g_k T_k((A - c)/e) x on the window."""
        c, e = 0.5 * (WINDOW[0] + WINDOW[1]), 0.5 * (WINDOW[1] - WINDOW[0])
        t0, t1 = x, (self(x) - c * x) / e
        y = g[0] * t0 + g[1] * t1
        for k in range(2, len(g)):
            t0, t1 = t1, 2.0 / e * (self(t1) - c * t1) - t0
            y = y + g[k] * t1
        return y


def exact(case, seed):
    kind = case["kind"]
    if kind == "apply":
        x = _vector(6 * math.prod(_dims(case)), seed)
        if case["precision"] != "fp64":
            x = x.to(torch.complex64).to(C128)
        return _Stencil(case, seed)(x)
    if kind == "filter":
        return _Stencil(case, seed).poly(_filtered(case, seed), _damped_step(CUT, case["degree"]))
    if kind == "rotate":
        v, z = _rotate_inputs(case, seed)
        out = torch.empty((case["kk"], case["n"]), dtype=C128, device=DEV)
        for r in range(0, case["n"], 65536):
            b = v[:, r:r + 65536].to(F64)
            s = b[..., :2] + b[..., 2:]
            out[:, r:r + 65536] = torch.view_as_complex(torch.tensordot(z, s, dims=1).contiguous())
        return out
    if kind == "solve_dense":
        a11, a12 = _dense(case["h"], _gen(seed))
        ev = torch.linalg.eigvalsh(torch.cat([torch.cat([a11, a12], 1), torch.cat([a12.conj().T, a11.T], 1)]))
        return [ev[::2][:case["nev"]].cpu().numpy(), None]
    if kind == "batch":
        out = np.zeros((case["count"], 8))
        for i, (a11, a12) in enumerate(_batch_blocks(case, seed)):
            m = torch.cat([torch.cat([a11, a12], 1), torch.cat([a12.conj().T, a11.T], 1)])
            out[i] = torch.linalg.eigvalsh(m.cpu())[::2][:8].numpy()
        return [out]
    return None      # the spectrum of a lattice of some size takes minutes in a dense solver
