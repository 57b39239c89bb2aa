"""Work that users of the eigensolver have it do, as cases that can be timed.

Every case goes through a public entry point: the C ABI on device buffers for
the stand-alone kernels, ``Feast`` / ``SparseFeast`` / ``solve_batch`` /
``eig_sum_abs2`` for the solves.  Inputs are those of the package's own
workloads (``inputs.py``), drawn on the GPU: dense pencils A = P diag(lam) Q,
B = P Q with P, Q = I + 0.1 G / sqrt(n), whose eigenvalues and eigenvectors
are prescribed, and the convection-diffusion operator on an nx x nx grid,
whose spectrum has a closed form.

``kind`` of a case:

* ``shifted``: LU of q shifted matrices and their solves with r right-hand
  sides, FP64 (eq. 4.2 by hand: ``feast_zgetrf_batched``, ``feast_zgetrs_batched``);
* ``projected``: eigenpairs of b projected m x m pencils (``feast_zqz_batched``);
* ``gemm64``: the FP64-accurate tensor-core product (``feast_zgemm_oz``);
* ``gemm32``: the complex64 tensor-core product (``feast_cgemm_tc``);
* ``filter``: the subspace build alone, U = sum_j w_j (z_j B - A)^-1 B V, on
  a context set up beforehand (``Feast.filter``);
* ``dense``: a whole solve of a dense pencil, set-up to eigenpairs (``Feast``);
* ``band``: a whole solve of a banded or sparse pencil (``Feast``, ``SparseFeast``), run until every pair has converged;
* ``batch``: many small dense pencils at once (``solve_batch``);
* ``grad``: sum |lam|^2 over the inside eigenvalues and its gradients with
  respect to A and B, forward and backward (``eig_sum_abs2``).
"""
import math

import numpy as np
import torch

import paper_1404_1768_gb300 as fg

C128, C64 = torch.complex128, torch.complex64


def listed():
    return [
        # smallest calls: the 16 nodes of a contour around a few eigenvalues of a small pencil
        dict(name="shifted_n64", kind="shifted", n=64, q=16, r=16),
        # an ordinary FP64 subspace build by hand, at a size that is no multiple of any tile
        dict(name="shifted_n1000", kind="shifted", n=1000, q=8, r=150),
        # projected pencils of a batch of small problems (line 6, one pencil each)
        dict(name="projected_m24_b16", kind="projected", m=24, b=16),
        # the projected pencil of one ordinary solve
        dict(name="projected_m300", kind="projected", m=300, b=1),
        # operator product A U1 of the n = 2048 workload at FP64 accuracy
        dict(name="gemm64_2048x640", kind="gemm64", m=2048, n=640, k=2048, update=False),
        # trailing update of the complex64 LU, 8 nodes
        dict(name="gemm32_update_1792", kind="gemm32", m=1792, n=1792, k=256, b=8, update=True),
        # subspace build in the precision form, refined to full accuracy
        dict(name="filter_n1024", kind="filter", n=1024, m0=256, q=16, rule=0, prec=1),
        # the plain method in FP64 on the n = 200 workload, eigenvectors too (the defaults of Feast)
        dict(name="dense_n200_fp64", kind="dense", n=200, n_in=44, m0=64, q=16, rule=0, prec=0, eps=1e-12, vectors=True),
        # largest: the precision form on a dense pencil, eigenvalues to the host (its closest pairs are ~1e-3 apart, so
        # eigenvectors are only determined to ~1e-8 by residuals below eps)
        dict(name="dense_n2048_c64r", kind="dense", n=2048, n_in=512, m0=640, q=32, rule=0, prec=1, eps=1e-10, vectors=False),
        # the banded workload: convection-diffusion on the 128 x 128 grid, lowest 41 eigenvalues
        dict(name="band_nx128_c64r", kind="band", nx=128, n_in=41, m0=64, q=16, prec=1, sparse=False, eps=1e-10),
        # a ragged batch of independent pencils, each with its own circle
        dict(name="batch_12", kind="batch", b=12, n_lo=64, n_hi=512, q=16, prec=1, eps=1e-10),
        # forward and backward of the differentiation form
        dict(name="grad_n512", kind="grad", n=512, n_in=128, m0=192, q=24, prec=1, eps=1e-10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["shifted", "shifted", "projected", "projected", "gemm64", "gemm32", "filter", "dense", "dense",
                       "band", "batch", "grad"])
    if kind == "shifted":
        n = _log(rng, 32, 1400)
        return dict(kind=kind, n=n, q=rng.choice([4, 8, 16, 24]), r=max(1, min(n, _log(rng, 4, 400))))
    if kind == "projected":
        if rng.random() < 0.5:
            return dict(kind=kind, m=rng.randint(8, 64), b=_log(rng, 1, 64))
        return dict(kind=kind, m=_log(rng, 65, 480), b=1)
    if kind == "gemm64":
        return dict(kind=kind, m=_log(rng, 40, 3000), n=_log(rng, 16, 1000), k=_log(rng, 40, 3000),
                    update=rng.random() < 0.3)
    if kind == "gemm32":
        return dict(kind=kind, m=_log(rng, 64, 2048), n=_log(rng, 64, 2048), k=rng.choice([64, 200, 256, 512]),
                    b=_log(rng, 1, 8), update=rng.random() < 0.7)
    if kind == "filter":
        n = _log(rng, 150, 1400)
        return dict(kind=kind, n=n, m0=max(8, int(n * rng.uniform(0.1, 0.35))), q=rng.choice([8, 16, 24]),
                    rule=rng.choice([0, 1]), prec=rng.choice([0, 1, 1]) if n <= 800 else 1)
    if kind == "dense":
        prec = rng.choice([0, 1])
        n = _log(rng, 96, 640) if prec == 0 else _log(rng, 200, 1600)
        n_in = int(n * rng.uniform(0.15, 0.27))
        m0 = 8 * math.ceil((1.3 * n_in + 6) / 8)
        return dict(kind=kind, n=n, n_in=n_in, m0=m0, q=rng.choice([16, 24, 32]), rule=0, prec=prec,
                    eps=1e-12 if prec == 0 and m0 <= 64 else 1e-10, vectors=n <= 640)
    if kind == "band":
        nx, n_in = _log(rng, 28, 128), rng.randint(12, 41)
        prec = rng.choice([0, 1, 1]) if nx <= 80 else 1
        return dict(kind=kind, nx=nx, n_in=n_in, m0=8 * math.ceil(1.5 * n_in / 8), q=16, prec=prec,
                    sparse=rng.random() < 0.4, eps=1e-10)
    if kind == "batch":
        lo = rng.randint(64, 128)
        return dict(kind=kind, b=rng.randint(4, 12), n_lo=lo, n_hi=rng.randint(lo + 32, 512), q=16, prec=rng.choice([0, 1, 1]),
                    eps=1e-10)
    n = _log(rng, 128, 512)
    n_in = int(n * rng.uniform(0.15, 0.25))
    return dict(kind=kind, n=n, n_in=n_in, m0=8 * math.ceil((1.4 * n_in + 6) / 8), q=24, prec=rng.choice([0, 1]) if n <= 256 else 1,
                eps=1e-10)


# ------------------------------------------------------------------ inputs
class _Draws:
    """Random numbers on the GPU from a seed alone."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)
        self.h = np.random.default_rng(seed)

    def normal(self, *shape):
        return torch.randn(*shape, dtype=C128, device="cuda", generator=self.g)  # E|x|^2 = 1


def _factors(d, n):
    eye = torch.eye(n, dtype=C128, device="cuda")
    return eye + 0.1 / math.sqrt(n) * d.normal(n, n), eye + 0.1 / math.sqrt(n) * d.normal(n, n)


def _spectrum(d, n, n_in, center=0j, radius=1.0):
    """n eigenvalues uniform in the disk |z| < 2 given that n_in of them lie inside the circle; none within 0.2 % of it."""
    lam = []
    for inside, count in ((True, n_in), (False, n - n_in)):
        got = np.zeros(0, complex)
        while got.size < count:
            z = 2 * np.sqrt(d.h.random(8 * n)) * np.exp(2j * np.pi * d.h.random(8 * n))
            r = np.abs(z - center) / radius
            got = np.concatenate([got, z[r < 0.998] if inside else z[r > 1.002]])
        lam.append(got[:count])
    return d.h.permutation(np.concatenate(lam))


def _pencil(d, lam):
    P, Q = _factors(d, lam.size)
    return (P * torch.from_numpy(lam).cuda()) @ Q, P @ Q, P, Q


def _contour(case):
    return dict(contour_kind=0, rule=case.get("rule", 0), q=case["q"], center=0j, a=1.0)


def _grid(case, seed):
    """Convection-diffusion on the nx x nx grid (inputs.convection_diffusion with the seed's drift), the ellipse around
    its n_in lowest eigenvalues, and those eigenvalues in closed form."""
    d = _Draws(seed)
    nx, k = case["nx"], case["n_in"]
    beta = (float(d.h.uniform(18, 22)), float(d.h.uniform(9, 11)))
    h = 1.0 / (nx + 1)
    x = np.cos(np.arange(1, nx + 1) * np.pi * h)
    c = [math.sqrt(1 - (b * h / 2) ** 2) for b in beta]
    lam = np.sort((2 / h**2 * (2 - c[0] * x[:, None] - c[1] * x[None, :])).ravel())
    left, right = 0.7 * lam[0], 0.5 * (lam[k - 1] + lam[k])
    a = 0.5 * (right - left)
    return d, beta, h, lam[:k], dict(contour_kind=1, rule=1, q=case["q"], center=complex(left + a), a=a, b=a / 4)


def _stencil(nx, h, beta):
    """(offset i - j, value, mask over the columns j) of the five diagonals."""
    gx, gy = np.arange(nx * nx) % nx, np.arange(nx * nx) // nx
    s = 1.0 / (h * h)
    return [(0, 4 * s, gx >= 0), (1, (-1 - beta[0] * h / 2) * s, gx < nx - 1), (-1, (-1 + beta[0] * h / 2) * s, gx > 0),
            (nx, (-1 - beta[1] * h / 2) * s, gy < nx - 1), (-nx, (-1 + beta[1] * h / 2) * s, gy > 0)]


def _batch(case, seed):
    """Ragged pencils as inputs.ragged_batch makes them, the circle's inside count from the share of the disk it covers."""
    d, out = _Draws(seed), []
    shape = np.random.default_rng(1404)  # sizes and circles are the case's, matrices the seed's
    for _ in range(case["b"]):
        n = int(shape.integers(case["n_lo"], case["n_hi"] + 1))
        cr, ca = 0.9 * math.sqrt(shape.random()), 2 * math.pi * shape.random()
        center, radius = complex(cr * math.cos(ca), cr * math.sin(ca)), 0.5 + 0.5 * shape.random()
        n_in = max(2, round(n * radius**2 / 4))
        m0 = max(16, 8 * math.ceil(1.5 * n_in / 8))
        lam = _spectrum(d, n, n_in, center, radius)
        A, B, _, _ = _pencil(d, lam)
        out.append(dict(A=A, B=B, Y=d.normal(n, m0), center=center, a=radius, lam=lam))
    return out


def _projected(case, seed):
    """B upper triangular, A = B W X diag(lam) X^-1 W^H with W unitary: what an oblique projection of a dense pencil onto
    a random basis leaves.  Also the eigenvalues and W X."""
    d, m = _Draws(seed), case["m"]
    lams, As, Bs, Vs = [], [], [], []
    for _ in range(case["b"]):
        W = torch.linalg.qr(d.normal(m, m))[0]
        X = torch.eye(m, dtype=C128, device="cuda") + 0.1 / math.sqrt(m) * d.normal(m, m)
        lam = torch.from_numpy(_spectrum(d, m, max(1, (3 * m) // 4))).cuda()
        R = torch.triu(torch.linalg.qr(torch.eye(m, dtype=C128, device="cuda") + 0.2 / math.sqrt(m) * d.normal(m, m))[1])
        V = W @ X
        As.append(R @ torch.linalg.solve(V, V * lam, left=False))
        lams.append(lam)
        Bs.append(R)
        Vs.append(V)
    return torch.stack(lams), torch.stack(As), torch.stack(Bs), torch.stack(Vs)


def _shifted(case, seed):
    d, n, q = _Draws(seed), case["n"], case["q"]
    A, B, _, _ = _pencil(d, _spectrum(d, n, n // 4))
    z = torch.exp(2j * math.pi * (torch.arange(q, dtype=torch.float64, device="cuda") + 0.5) / q)
    return z[:, None, None] * B - A, B @ d.normal(n, case["r"])


def _gemm(case, seed, dtype):
    d, b = _Draws(seed), case.get("b", 1)
    A, X = d.normal(b, case["m"], case["k"]), d.normal(b, case["k"], case["n"])
    Cm = d.normal(b, case["m"], case["n"]) if case["update"] else torch.zeros(b, case["m"], case["n"], dtype=C128, device="cuda")
    return A.to(dtype), X.to(dtype), Cm.to(dtype)


def _cols(t):
    """(..., rows, cols) -> the same matrices with column-major storage."""
    return t.mT.contiguous()


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "shifted":
        M, R = _shifted(case, seed)
        n, q, r = case["n"], case["q"], case["r"]
        s.update(M=_cols(M), R=_cols(R), F=torch.empty(q, n, n, dtype=C128, device="cuda"),
                 X=torch.empty(q, r, n, dtype=C128, device="cuda"), piv=torch.zeros(q, n, dtype=torch.int32, device="cuda"),
                 info=torch.zeros(1, dtype=torch.int32, device="cuda"))
    elif kind == "projected":
        m, b = case["m"], case["b"]
        _, A, B, _ = _projected(case, seed)
        s.update(A0=_cols(A), B0=_cols(B))
        s.update(A=torch.empty_like(s["A0"]), B=torch.empty_like(s["B0"]), V=torch.empty_like(s["A0"]),
                 al=torch.empty(b, m, dtype=C128, device="cuda"), be=torch.empty(b, m, dtype=C128, device="cuda"),
                 work=torch.empty(int(fg.load().feast_zqz_work_bytes(m, b)), dtype=torch.uint8, device="cuda"),
                 st=torch.zeros(2, dtype=torch.int32, device="cuda"))
    elif kind in ("gemm64", "gemm32"):
        A, X, Cm = _gemm(case, seed, C128 if kind == "gemm64" else C64)
        s.update(A=_cols(A), X=_cols(X), C0=_cols(Cm), err=torch.zeros(1, dtype=torch.int32, device="cuda"))
        s["C"] = torch.empty_like(s["C0"])
        lib, m, n, k = fg.load(), case["m"], case["n"], case["k"]
        nb = lib.feast_zgemm_oz_work_bytes(m, n, k) if kind == "gemm64" else lib.feast_cgemm_tc_scratch_bytes(m, n, k, case["b"])
        s.update(work=torch.empty(int(nb), dtype=torch.uint8, device="cuda"), nb=int(nb))
    elif kind == "filter":
        d = _Draws(seed)
        A, B, _, _ = _pencil(d, _spectrum(d, case["n"], case["n"] // 4))
        s["V"] = d.normal(case["n"], case["m0"])
        s["handle"] = fg.Feast(A, B, s["V"], prec=case["prec"], **_contour(case))
    elif kind in ("dense", "grad"):
        d = _Draws(seed)
        A, B, _, _ = _pencil(d, _spectrum(d, case["n"], case["n_in"]))
        s.update(A=A, B=B, Y=d.normal(case["n"], case["m0"]))
        if kind == "grad":
            A.requires_grad_()
            B.requires_grad_()
    elif kind == "band":
        d, beta, h, _, s["contour"] = _grid(case, seed)
        nx = case["nx"]
        n = nx * nx
        s["Y"] = d.normal(n, case["m0"])
        if case["sparse"]:  # rows and columns in a random order, CSR on the host
            rows, cols, vals, p = [], [], [], d.h.permutation(n)
            for off, v, ok in _stencil(nx, h, beta):
                j = np.nonzero(ok)[0]
                rows.append(p[j + off]), cols.append(p[j]), vals.append(np.full(j.size, v, complex))
            rows, cols, vals = (np.concatenate(v) for v in (rows, cols, vals))
            o = np.lexsort((cols, rows))
            s["A"] = (np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))]), cols[o], vals[o])
        else:
            band = np.zeros((2 * nx + 1, n), complex)
            for off, v, ok in _stencil(nx, h, beta):
                band[nx + off, ok] = v
            s["A"] = torch.from_numpy(band).cuda()
    elif kind == "batch":
        s["problems"] = [dict(A=p["A"].cpu().numpy(), B=p["B"].cpu().numpy(), Y=p["Y"].cpu().numpy(), center=p["center"],
                              a=p["a"], q=case["q"], prec=case["prec"], eps=case["eps"]) for p in _batch(case, seed)]
    return s


# ------------------------------------------------------------------ passes
def _ok(status):
    if status != 0:
        raise RuntimeError(fg.load().feast_strerror(status).decode())


def _pairs(lam, V=None):
    """Eigenvalues in ascending order (real, then imaginary part), eigenvectors in that order with the largest entry of
    each real and positive."""
    lam = np.asarray(lam)
    o = np.lexsort((lam.imag, lam.real))
    if V is None:
        return lam[o]
    V = V[:, o]
    top = V[np.argmax(np.abs(V), axis=0), np.arange(V.shape[1])]
    return lam[o], V * (np.abs(top) / (top * np.linalg.norm(V, axis=0)))


def _pairs_on_gpu(lam, V):
    """The same for (b, m) eigenvalues and (b, m, m) matrices whose row i is eigenvector i."""
    o = torch.argsort(lam.real, dim=1)
    V = torch.gather(V, 1, o[:, :, None].expand_as(V))
    top = torch.gather(V, 2, V.abs().argmax(dim=2, keepdim=True))
    return torch.gather(lam, 1, o), V * (top.abs() / (top * torch.linalg.vector_norm(V, dim=2, keepdim=True)))


def run(s):
    case = s["case"]
    kind = case["kind"]
    lib, stream = fg.load(), torch.cuda.current_stream().cuda_stream
    if kind == "shifted":
        n, q, r = case["n"], case["q"], case["r"]
        s["F"].copy_(s["M"])
        s["X"].copy_(s["R"].expand(q, r, n))
        _ok(lib.feast_zgetrf_batched(n, q, s["F"].data_ptr(), n, n * n, s["piv"].data_ptr(), s["info"].data_ptr(), stream))
        _ok(lib.feast_zgetrs_batched(n, r, q, s["F"].data_ptr(), n, n * n, s["piv"].data_ptr(), s["X"].data_ptr(), n, n * r,
                                     stream))
        return dict(X=s["X"], F=s["F"], piv=s["piv"], info=s["info"])
    if kind == "projected":
        s["A"].copy_(s["A0"])
        s["B"].copy_(s["B0"])
        _ok(lib.feast_zqz_batched(case["m"], case["b"], s["A"].data_ptr(), s["B"].data_ptr(), s["al"].data_ptr(),
                                  s["be"].data_ptr(), s["V"].data_ptr(), s["work"].data_ptr(), s["st"].data_ptr(), stream))
        lam, V = _pairs_on_gpu(s["al"] / s["be"], s["V"])
        return dict(lam=lam, V=V, status=s["st"])
    if kind in ("gemm64", "gemm32"):
        m, n, k = case["m"], case["n"], case["k"]
        al, be = (-1.0, 1.0) if case["update"] else (1.0, 0.0)
        if case["update"]:
            s["C"].copy_(s["C0"])
        if kind == "gemm64":
            _ok(lib.feast_zgemm_oz(m, n, k, al, 0.0, s["A"].data_ptr(), m, s["X"].data_ptr(), k, be, 0.0, s["C"].data_ptr(), m,
                                   s["work"].data_ptr(), s["nb"], s["err"].data_ptr(), stream))
        else:
            _ok(lib.feast_cgemm_tc(m, n, k, al, 0.0, s["A"].data_ptr(), m, m * k, s["X"].data_ptr(), k, k * n, be, 0.0,
                                   s["C"].data_ptr(), m, m * n, case["b"], s["work"].data_ptr(), s["nb"], s["err"].data_ptr(),
                                   stream))
        return dict(C=s["C"], err=s["err"])
    if kind == "filter":
        return s["handle"].filter(s["V"])
    if kind == "dense":
        f = fg.Feast(s["A"], s["B"], s["Y"], eps=case["eps"], prec=case["prec"], **_contour(case))
        f.run()
        r = f.eigs(want_vectors=case["vectors"])
        f.close()
        if case["vectors"]:
            lam, X = _pairs(r["lam"], r["X"])
            return dict(lam=lam, X=X, flag=r["flag"])
        return dict(lam=_pairs(r["lam"]), flag=r["flag"])
    if kind == "band":
        kw = dict(eps=case["eps"], prec=case["prec"], converged_only=True, **s["contour"])
        nx = case["nx"]
        if case["sparse"]:
            f = fg.SparseFeast(nx * nx, s["A"], None, s["Y"], **kw)
        else:
            f = fg.Feast(s["A"], None, s["Y"], kind=fg.FEAST_BANDED, kl=nx, ku=nx, b_identity=True, **kw)
        f.run()
        r = f.eigs(want_vectors=False)
        f.close()
        return dict(lam=_pairs(r["lam"]), flag=r["flag"])
    if kind == "batch":
        got = fg.solve_batch(s["problems"])
        return dict(lam=np.concatenate([_pairs(g["lam"]) for g in got]), flag=[g["flag"] for g in got])
    L = fg.eig_sum_abs2(s["A"], s["B"], s["Y"], eps=case["eps"], prec=case["prec"], **_contour(case))
    gA, gB = torch.autograd.grad(L, (s["A"], s["B"]))
    return dict(L=L.detach(), gA=gA, gB=gB)


# ------------------------------------------------------------------ work and 64-bit results
def _passes(case, n_in, m0):
    """Passes until the filter of q nodes has shrunk the slowest inside pair from 1 to eps."""
    ratio = (m0 / n_in) ** (-0.5 * case["q"])
    return max(2, math.ceil(math.log(case["eps"]) / math.log(max(ratio, 1e-8))) + 1)


def _solve_work(n, m0, n_in, q, case):
    p = _passes(case, n_in, m0)
    return q * 8 / 3 * n**3 + p * (8 * q * n * n * m0 + 24 * n * n * m0 + 40 * n * m0 * m0 + 100 * m0**3)


def work(case):
    kind = case["kind"]
    if kind == "shifted":
        n, q, r = case["n"], case["q"], case["r"]
        return dict(bytes=32.0 * q * (n * n + n * r), flops=8.0 * q * (n**3 / 3 + n * n * r))
    if kind == "projected":
        m, b = case["m"], case["b"]
        return dict(bytes=16.0 * b * (3 * m * m + 2 * m), flops=100.0 * b * m**3)
    if kind in ("gemm64", "gemm32"):
        m, n, k, b = case["m"], case["n"], case["k"], case.get("b", 1)
        return dict(bytes=(16 if kind == "gemm64" else 8) * b * (m * k + k * n + m * n * (2 if case["update"] else 1)),
                    flops=8.0 * b * m * n * k)
    if kind == "filter":
        n, m0, q = case["n"], case["m0"], case["q"]
        return dict(bytes=q * n * n * (8.0 if case["prec"] else 16.0) + 32.0 * n * m0, flops=8.0 * n * n * m0 * (q + 1))
    if kind == "dense":
        n, m0, n_in = case["n"], case["m0"], case["n_in"]
        return dict(bytes=32.0 * n * n + 16.0 * n * (m0 + n_in), flops=_solve_work(n, m0, n_in, case["q"], case))
    if kind == "band":
        nx, m0, q = case["nx"], case["m0"], case["q"]
        n = nx * nx
        return dict(bytes=16.0 * n * (2 * nx + 1 + m0), flops=q * 8.0 * n * 2 * nx * nx + 5 * (q * 8.0 * n * 4 * nx * m0 + 40 * n * m0 * m0))
    if kind == "batch":
        n = 0.5 * (case["n_lo"] + case["n_hi"])
        return dict(bytes=case["b"] * 40.0 * n * n, flops=case["b"] * _solve_work(n, 0.22 * n, 0.15 * n, case["q"], case))
    n, m0, n_in = case["n"], case["m0"], case["n_in"]
    return dict(bytes=64.0 * n * n, flops=2 * _solve_work(n, m0, n_in, case["q"], case) + 16.0 * n * n * n_in)


def _weights(case):
    """Nodes and weights of the unit circle: trapezoid, or Gauss-Legendre in the angle (eq. 4.1)."""
    q = case["q"]
    t, w = np.polynomial.legendre.leggauss(q) if case["rule"] else ((2 * np.arange(q) + 1) / q - 1, np.full(q, 2 / q))
    z = np.exp(1j * np.pi * (1 + t))
    return z, 0.5 * w * z


def exact(case, seed):
    kind = case["kind"]
    if kind == "shifted":
        M, R = _shifted(case, seed)
        return dict(X=torch.linalg.solve(M, R.expand(case["q"], *R.shape)).mT.contiguous(), F=None, piv=None, info=None)
    if kind == "projected":
        lam, _, _, V = _projected(case, seed)
        lam, V = _pairs_on_gpu(lam, V.mT.contiguous())
        return dict(lam=lam, V=V, status=None)
    if kind in ("gemm64", "gemm32"):
        A, X, Cm = (t.to(C128) for t in _gemm(case, seed, C128 if kind == "gemm64" else C64))
        return dict(C=((Cm - A @ X) if case["update"] else A @ X).mT.contiguous(), err=None)
    if kind == "filter":
        d = _Draws(seed)
        lam = _spectrum(d, case["n"], case["n"] // 4)
        _, _, _, Q = _pencil(d, lam)
        z, w = _weights(case)
        f = torch.from_numpy((w[None, :] / (z[None, :] - lam[:, None])).sum(1)).cuda()
        return torch.linalg.solve(Q, f[:, None] * (Q @ d.normal(case["n"], case["m0"]))).cpu().numpy()
    if kind in ("dense", "grad"):
        d = _Draws(seed)
        lam = _spectrum(d, case["n"], case["n_in"])
        inside = np.abs(lam) < 1
        A, B, P, Q = _pencil(d, lam)
        if kind == "dense":
            if not case["vectors"]:
                return dict(lam=_pairs(lam[inside]), flag=None)
            ev, X = _pairs(lam[inside], np.linalg.inv(Q.cpu().numpy())[:, inside])
            return dict(lam=ev, X=X, flag=None)
        li = torch.from_numpy(np.where(inside, lam, 0)).cuda()
        Pih, Qih = torch.linalg.inv(P).mH, torch.linalg.inv(Q).mH
        L = torch.tensor(np.sum(np.abs(lam[inside]) ** 2))
        return dict(L=L, gA=2 * (Pih * li) @ Qih, gB=-2 * (Pih * (li.abs() ** 2)) @ Qih)
    if kind == "band":
        return dict(lam=_grid(case, seed)[3].astype(complex), flag=None)
    lam = []
    for p in _batch(case, seed):
        lam.append(_pairs(p["lam"][np.abs(p["lam"] - p["center"]) < p["a"]]))
    return dict(lam=np.concatenate(lam), flag=None)
