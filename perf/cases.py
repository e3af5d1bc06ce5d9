"""Workloads of the library as its users run them, through the Python binding.

Each case is one call (or one short job) on a gauge field, with the right-hand
sides in GPU memory, from the smallest lattices, where launches and latency
count, to the 24^3 x 64 production field. Lattices, hopping parameters, window
and eigenspace sizes are those of the repository's named workloads, or generic
odd extents. Solves run to a relative residual of 1e-12, two digits below the
workloads' 1e-10, so that a solution is defined to about 1e-11 whatever the
order of the sums. FP32 results (the FP32 operator, the oblique projection, the
inner-product matrix) are handed on as complex64, the precision they hold.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0911_2285_gb300.lqcd import Solver, field_dots

TOL = 1e-12


# ------------------------------------------------------------------- the cases
def _case(kind, dims, k, **more):
    c = dict(kind=kind, Lx=dims[0], Ly=dims[1], Lz=dims[2], Lt=dims[3], k=k)
    c.update(more)
    return c


def listed():
    mid, big = (16, 16, 16, 32), (24, 24, 24, 64)
    return [
        # one product with A^+ in FP64 on a small lattice: the smallest call a program makes
        dict(name="apply_fp64_8^4", **_case("apply", (8, 8, 8, 8), 1, precision="fp64", dagger=True, kappa=0.124,
                                            eps=0.3)),
        # the FP32 operator on four fields of the production lattice (smearing, three-point functions)
        dict(name="apply_mixed_24^3x64", **_case("apply", big, 4, precision="mixed", dagger=False, kappa=0.1245,
                                                 eps=0.3)),
        # one FP64 source on the smallest lattice: bound by launches and round trips
        dict(name="plain_fp64_4^4", **_case("solve", (4, 4, 4, 4), 1, precision="fp64", variant="bicg", kappa=0.12,
                                            eps=0.5)),
        # the Incremental eigBiCG job of the 8^4 workload: 4 sources by eigBiCG, 8 deflated
        dict(name="job_mixed_8^4", **_case("job", (8, 8, 8, 8), 12, precision="mixed", n1=4, nev=10, m=40,
                                           kappa=0.124, eps=0.3)),
        # extents that no tile divides, a batch that is not full
        dict(name="plain_mixed_10x6x14x9", **_case("solve", (10, 6, 14, 9), 3, precision="mixed", variant="bicg",
                                                   kappa=0.122, eps=0.3)),
        # the FP64 solver, one source (the reference solver the speed-ups are quoted against)
        dict(name="plain_fp64_16^3x32", **_case("solve", mid, 1, precision="fp64", variant="bicg", kappa=0.124,
                                                eps=0.3)),
        # phase 2 as the paper runs it: BiCGStab, a full batch
        dict(name="bicgstab_mixed_16^3x32", **_case("solve", mid, 8, precision="mixed", variant="bicgstab",
                                                    kappa=0.124, eps=0.3)),
        # the even-odd preconditioned system, a full batch
        dict(name="evenodd_mixed_16^3x32", **_case("solve", mid, 8, precision="mixed", variant="evenodd",
                                                   kappa=0.1245, eps=0.3)),
        # the Incremental eigBiCG job of the 16^3x32 workload: 4 sources by eigBiCG, 8 deflated
        dict(name="job_mixed_16^3x32", **_case("job", mid, 12, precision="mixed", n1=4, nev=10, m=60, kappa=0.124,
                                               eps=0.3)),
        # a full batch of plain mixed-precision solves on the production lattice
        dict(name="plain_mixed_24^3x64", **_case("solve", big, 8, precision="mixed", variant="bicg", kappa=0.1245,
                                                 eps=0.3)),
        # oblique deflation of a batch of initial guesses against 40 vector pairs
        dict(name="deflate_mixed_16^3x32", **_case("deflate", mid, 8, n=40, kappa=0.124, eps=0.3)),
        # Galerkin projections of a batch of residuals on the full eigenspace of the production lattice
        dict(name="dots_80x8_24^3x64", **_case("dots", big, 8, n=80)),
    ]


_KAPPA = (0.12, 0.122, 0.124, 0.1245)
_EXTENTS = (4, 5, 6, 7, 8, 9, 10, 12, 14, 16, 18, 20, 24)


def _dims(rng, lo, hi, step=1):
    """Extents of a lattice whose volume is about log-uniform in [lo, hi]."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    side = want ** 0.25
    ext = [e for e in _EXTENTS if e % step == 0 and 0.55 * side <= e <= 1.6 * side] or [4 if side < 4 else 24]
    d = [rng.choice(ext) for _ in range(3)]
    lt = int(round(want / (d[0] * d[1] * d[2]) / step)) * step
    return (*d, max(4, min(64, lt)))


def draw(rng):
    kind = rng.choice(("apply", "solve", "solve", "solve", "job", "deflate", "dots"))
    kappa = rng.choice(_KAPPA)
    if kind == "apply":
        return _case(kind, _dims(rng, 256, 500000), rng.randint(1, 5), precision=rng.choice(("fp64", "mixed")),
                     dagger=rng.random() < 0.5, kappa=kappa, eps=0.3)
    if kind == "solve":
        variant = rng.choice(("bicg", "bicg", "bicgstab", "evenodd"))
        precision = "fp64" if variant == "bicg" and rng.random() < 0.35 else "mixed"
        dims = _dims(rng, 256, 131072 if precision == "fp64" else 300000, 2 if variant == "evenodd" else 1)
        k = rng.randint(1, 2) if precision == "fp64" else rng.randint(1, 8)
        return _case(kind, dims, k, precision=precision, variant=variant, kappa=kappa, eps=0.3)
    if kind == "job":
        return _case(kind, _dims(rng, 2048, 131072), rng.randint(4, 12), precision="mixed", n1=rng.randint(1, 3),
                     nev=rng.choice((8, 10)), m=rng.choice((24, 40, 60)), kappa=kappa, eps=0.3)
    if kind == "deflate":
        return _case(kind, _dims(rng, 256, 100000), rng.randint(1, 8), n=rng.randint(8, 60), kappa=kappa, eps=0.3)
    dims = _dims(rng, 4096, 500000, 4)
    return _case(kind, dims, rng.randint(1, 20), n=rng.randint(8, 80))


def _volume(c):
    return c["Lx"] * c["Ly"] * c["Lz"] * c["Lt"]


def _extents(c):
    return (c["Lx"], c["Ly"], c["Lz"], c["Lt"])


# ------------------------------------------------------------------ the inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _gauge(c, g):
    """Random SU(3) links exp(i eps H), H Hermitian traceless Gaussian, [4][V][3][3]."""
    n = 4 * _volume(c)
    z = torch.randn(n, 3, 3, 2, dtype=torch.float64, device="cuda", generator=g)
    h = torch.view_as_complex(z) / math.sqrt(2.0)
    h = 0.5 * (h + h.mH)
    tr = h.diagonal(dim1=1, dim2=2).sum(1) / 3.0
    one = torch.eye(3, dtype=h.dtype, device="cuda")
    a = (0.125j * c["eps"]) * (h - tr[:, None, None] * one)   # exp(a)^8
    u = one.expand(n, 3, 3)
    for j in range(12, 0, -1):
        u = one + _mm(a, u) / j
    for _ in range(3):
        u = _mm(u, u)
    return u


def _mm(a, b):
    """Products of 3 x 3 (or 3 x 3 by 3 x n) matrices, element by element."""
    return sum(a[..., :, j, None] * b[..., j, None, :] for j in range(3))


def _z2(n, k, g):
    """k complex Z2 noise sources (+-1 +- i)/sqrt(2)."""
    s = torch.randint(0, 2, (k, n, 2), device="cuda", generator=g, dtype=torch.int8)
    return torch.view_as_complex((1.0 - 2.0 * s.double()) * math.sqrt(0.5))


def _gaussian(n, k, g, dtype=torch.float64):
    return torch.view_as_complex(torch.randn(k, n, 2, dtype=dtype, device="cuda", generator=g) * math.sqrt(0.5))


def _inputs(c, seed):
    """Links and fields of a case, on the GPU, from the seed alone."""
    g = _generator(seed)
    n = 12 * _volume(c)
    kind = c["kind"]
    if kind == "dots":
        return dict(X=_gaussian(n, c["n"], g, torch.float32), Y=_gaussian(n, c["k"], g, torch.float32))
    d = dict(links=_gauge(c, g))
    if kind == "apply":
        d["v"] = _gaussian(n, c["k"], g)
    elif kind == "deflate":
        # right and left vectors that are close to one another, as Ritz vectors are; FP32 values
        ur = _gaussian(n, c["n"], g, torch.float32) / math.sqrt(n)
        ul = ur + _gaussian(n, c["n"], g, torch.float32) * (0.3 / math.sqrt(n))
        d.update(ur=ur, ul=ul, b=_z2(n, c["k"], g), x0=0.1 * _gaussian(n, c["k"], g))
    else:
        d["b"] = _z2(n, c["k"], g)
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    if case["kind"] == "dots":
        return dict(kind="dots", X=d["X"], Y=d["Y"])
    links = d.pop("links").cpu().numpy()
    dims = _extents(case)
    kind = case["kind"]
    args = dict(nev=10, m=60, n1=4, tol=TOL, maxiter=5000, precision=case.get("precision", "mixed"),
                k_max=min(8, case["k"]))
    if kind == "apply":
        args.update(nev=2, m=8, n1=1, precision="mixed")   # both precisions of the operator from one context
    elif kind == "job":
        args.update(nev=case["nev"], m=case["m"], n1=case["n1"], k_max=8)
    elif kind == "deflate":
        args.update(n_def_max=case["n"])
    else:
        args.update(nev=2, m=8, n1=1, bicgstab=case["variant"] == "bicgstab", evenodd=case["variant"] == "evenodd")
    s = Solver(links, dims, case["kappa"], **args)
    if kind == "deflate":
        s.eigspace_set(d.pop("ur").cpu().numpy().astype(np.complex128), d.pop("ul").cpu().numpy().astype(np.complex128))
    return dict(kind=kind, case=case, solver=s, **d)


# ---------------------------------------------------------------- one pass each
def run(state):
    kind = state["kind"]
    if kind == "dots":
        c, _ = field_dots(state["X"], state["Y"])
        return c.astype(np.complex64)
    s = state["solver"]
    if kind == "apply":
        precision = state["case"]["precision"]
        y = s.apply(state["v"], dagger=state["case"]["dagger"], precision=precision)
        return y if precision == "fp64" else y.to(torch.complex64)
    if kind == "deflate":
        return s.deflate(state["b"], state["x0"]).to(torch.complex64)
    b = state["b"]
    if kind == "job":
        n1 = state["case"]["n1"]
        s.reset_eigenspace()
        x1, _, _ = s.solve(b[:n1], mode="eigbicg")
        x2, _, _ = s.solve(b[n1:], mode="deflated")
        return [*x1, *x2]
    x, _, _ = s.solve(b, mode="plain")
    return [*x]


# ------------------------------------------------------------ work of one pass
def _iterations(c):
    """About how many BiCG iterations (BiCGStab steps) a source of the case takes."""
    n = {0.12: 150, 0.122: 165, 0.124: 200, 0.1245: 215}.get(c["kappa"], 200)
    return n // 2 if c.get("variant") in ("evenodd", "bicgstab") else n


def work(case):
    v, k, kind = _volume(case), case["k"], case["kind"]
    links64 = 4 * 9 * 16 * v
    if kind == "dots":
        return dict(bytes=12 * v * 8 * (case["n"] + k) + 8 * case["n"] * k, flops=8 * 12 * v * case["n"] * k)
    if kind == "apply":
        links = links64 if case["precision"] == "fp64" else links64 // 3
        out = 16 if case["precision"] == "fp64" else 8
        return dict(bytes=links + k * 12 * v * (16 + out), flops=1368 * v * k)
    if kind == "deflate":
        n = case["n"]
        return dict(bytes=links64 // 3 + 2 * n * 12 * v * 8 + k * 12 * v * (16 + 16 + 8),
                    flops=1368 * v * k + 2 * 8 * 12 * v * n * k)
    # a solve: per iteration the links once, then the passes over a source's Krylov vectors that the two
    # inner products of a BiCG step (or the two of a BiCGStab step) force: 10 up to the first, 6 after it
    z = 16 if case["precision"] == "fp64" else 8
    links = links64 if z == 16 else links64 // 3
    field = 12 * v * z
    if case.get("variant") == "evenodd":
        field, links = field // 2, 2 * links
    it = _iterations(case)
    batches = -(-k // 8)
    nbytes = it * (batches * links + k * 16 * field) + k * 2 * 12 * v * 16
    flops = it * k * (2 * 1368 * v + 6 * 8 * 12 * v)
    if kind == "job":
        # window products of the restarts of n1 sources, both sides: m fields read, 2 nev written
        n1, m, r = case["n1"], case["m"], 2 * case["nev"]
        restarts = max(0, (it - m) // (m - r) + 1)
        nbytes += n1 * restarts * 2 * (m + r) * field
        flops += n1 * restarts * 2 * 8 * 12 * v * m * r
    return dict(bytes=nbytes, flops=flops)


# --------------------------------------------- the same results, in 64 bits
_SIGMA = np.array([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]])


def _gammas():
    g = np.zeros((4, 4, 4), dtype=np.complex128)
    for mu in range(4):
        m = -1j * _SIGMA[mu] if mu < 3 else np.eye(2)
        g[mu, :2, 2:], g[mu, 2:, :2] = m, m.conj().T
    return torch.from_numpy(g).cuda()


class _Wilson:
    """A = 1 - kappa D_hop on complex128 torch fields [k][Lt][Lz][Ly][Lx][4][3]."""

    def __init__(self, c, links):
        self.lat = (c["Lt"], c["Lz"], c["Ly"], c["Lx"])
        self.kappa = c["kappa"]
        self.u = links.reshape(4, *self.lat, 3, 3)
        self.gam = _gammas()
        self.one = torch.eye(4, dtype=torch.complex128, device="cuda")

    def _hop(self, psi, sign):
        out = torch.zeros_like(psi)
        for mu in range(4):
            ax = 4 - mu   # axis of direction mu behind the batch axis
            fwd, bwd = self.one - sign * self.gam[mu], self.one + sign * self.gam[mu]
            u = self.u[mu]
            h = torch.matmul(fwd, psi.roll(-1, ax))
            out += _mm(u, h.mT).mT
            h = torch.matmul(bwd, psi)
            out += _mm(u.mH, h.mT).mT.roll(1, ax)
        return out

    def __call__(self, v, dagger=False):
        k = v.shape[0]
        psi = v.reshape(k, *self.lat, 4, 3)
        return (psi - self.kappa * self._hop(psi, -1.0 if dagger else 1.0)).reshape(k, -1)


def _solve64(op, b):
    """BiCGStab in FP64 to about 1e-14, restarted from the true residual."""
    x = torch.zeros_like(b)
    bn = b.norm()
    for _ in range(8):
        r = b - op(x)
        if r.norm() <= 3e-14 * bn:
            break
        rh, p, rho = r.clone(), r.clone(), torch.vdot(r.flatten(), r.flatten())
        stop = max(1e-9 * float(r.norm()), 1e-14 * float(bn))
        for _ in range(400):
            v = op(p)
            alpha = rho / torch.vdot(rh.flatten(), v.flatten())
            s = r - alpha * v
            t = op(s)
            omega = torch.vdot(t.flatten(), s.flatten()) / torch.vdot(t.flatten(), t.flatten())
            x = x + alpha * p + omega * s
            r = s - omega * t
            if float(r.norm()) <= stop:
                break
            new = torch.vdot(rh.flatten(), r.flatten())
            p = r + (new / rho * alpha / omega) * (p - omega * v)
            rho = new
    return x


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "dots":
        x, y = d["X"], d["Y"]
        out = torch.zeros(case["n"], case["k"], dtype=torch.complex128, device="cuda")
        for e in range(0, x.shape[1], 1 << 18):
            out += x[:, e:e + (1 << 18)].to(torch.complex128).conj() @ y[:, e:e + (1 << 18)].to(torch.complex128).mT
        return out.cpu().numpy()
    op = _Wilson(case, d["links"])
    if kind == "apply":
        return torch.cat([op(d["v"][j:j + 1], case["dagger"]) for j in range(case["k"])])
    if kind == "deflate":
        ur, ul = d["ur"].to(torch.complex128), d["ul"].to(torch.complex128)
        aur = torch.cat([op(ur[j:j + 1]) for j in range(case["n"])])
        h = ul.conj() @ aur.mT
        r = d["b"] - torch.cat([op(d["x0"][j:j + 1]) for j in range(case["k"])])
        return d["x0"] + torch.linalg.solve(h, ul.conj() @ r.mT).mT @ ur
    # the first source of the batch, and for a job the first deflated one
    want = {0, case["n1"]} if kind == "job" else {0}
    return [_solve64(op, d["b"][j:j + 1])[0] if j in want else None for j in range(case["k"])]
