"""Cases for timing the framework through its public entry points.

Sizes come from the repository's own workloads: the 4 x 4 x 4 and 32 x 32 x 32
boxes of order 7, the orders 3..9 of the solve sweeps, the batched mix (E
log-uniform in [8, 4096], orders 3, 5, 7, 9), the served mix (E up to 8192,
orders 5 and 7), and odd-sided boxes of other orders.  Meshes are boxes of the
unit cube whose interior vertices are jittered by 5 % of the element size;
right-hand sides are assembled from normal nodal sources.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2606_12650_gb300 import Batch, Mesh, Server, sem

MAX_NODES = 32 ** 3 * 8 ** 3          # local nodes of the largest listed problem


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # one operator call on a problem of a few dozen elements: a coarse
        # level or a unit test of a user's own solver; latency
        dict(name="ax_small", kind="ax", nx=4, ny=4, nz=4, N=7),
        # the assembled operator inside a user's own Krylov loop, ordinary
        # size, odd sides and N + 1 = 6
        dict(name="axg_mid", kind="axg", nx=17, ny=13, nz=11, N=5),
        # the operator at the benchmark's size: throughput
        dict(name="ax_large", kind="ax", nx=32, ny=32, nz=32, N=7),
        # the FP32 operator of a user's own mixed solver, BF16 factors, full size
        dict(name="ax32_bf16_large", kind="ax32", nx=32, ny=32, nz=32, N=7, gprec=1),
        # the same with FP32 factors, odd sides, N + 1 = 7
        dict(name="ax32_f32_mid", kind="ax32", nx=19, ny=17, nz=15, N=6, gprec=0),
        # 100 CG iterations of a small problem (the solve sweeps' protocol): launch-bound
        dict(name="cg_small", kind="cg", nx=4, ny=4, nz=4, N=7, iters=100),
        # the same protocol between the two: neither launch- nor bandwidth-bound
        dict(name="cg_mid", kind="cg", nx=13, ny=12, nz=11, N=8, iters=100),
        # the same protocol at the benchmark's size
        dict(name="cg_large", kind="cg", nx=32, ny=32, nz=32, N=7, iters=100),
        # Jacobi-preconditioned CG, the original mini-app's method, order 9, odd sides
        dict(name="pcg_mid", kind="pcg", nx=15, ny=14, nz=11, N=9, iters=100),
        # a whole mixed-precision solve at the benchmark's size, to the accuracy
        # at which refinement replaces an FP64 solve (the iterates on the way
        # depend on FP32 rounding; at 1e-11 the solution no longer does)
        dict(name="mixed_large", kind="mixed", nx=32, ny=32, nz=32, N=7, gprec=1, tol=1e-11),
        # many independent uneven problems in one call, FP64
        dict(name="batch_f64", kind="batch", count=32, mix=11, e_lo=8, e_hi=4096, mode=0, tol=1e-10),
        # requests served with continuous batching, mixed precision, host in and out
        dict(name="serve_mixed", kind="serve", count=24, mix=23, e_lo=8, e_hi=8192, mode=1, tol=1e-11),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["ax", "axg", "ax32", "cg", "pcg", "mixed", "batch", "serve"])
    if kind == "batch":
        mode = rng.choice([0, 1, 2])
        return dict(kind=kind, count=rng.randint(8, 32), mix=rng.randrange(1 << 20), e_lo=8, e_hi=rng.choice([512, 2048, 4096]),
                    mode=mode, tol=1e-11 if mode else 1e-10)
    if kind == "serve":
        mode = rng.choice([0, 1])
        return dict(kind=kind, count=rng.randint(6, 24), mix=rng.randrange(1 << 20), e_lo=8, e_hi=rng.choice([512, 2048, 8192]),
                    mode=mode, tol=1e-11 if mode else 1e-10)
    N = rng.randint(3, 9)
    nq3 = (N + 1) ** 3
    E = _log_int(rng, 8, 0.9 * MAX_NODES / nq3)
    nx = max(1, int(round(E ** (1 / 3) * rng.uniform(0.8, 1.25))))
    ny = max(1, int(round(math.sqrt(E / nx) * rng.uniform(0.85, 1.15))))
    nz = max(1, min(E // (nx * ny), MAX_NODES // (nx * ny * nq3)))
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, N=N)
    if kind in ("ax32", "mixed"):
        c["gprec"] = rng.choice([0, 1, 1])
    if kind == "mixed":
        c["tol"] = 1e-11
    if kind in ("cg", "pcg"):
        c["iters"] = rng.choice([50, 100])
    return c


# ---------------------------------------------------------------- inputs
def _vertices(nx, ny, nz, seed):
    x, y, z = (np.linspace(0.0, 1.0, n + 1) for n in (nx, ny, nz))
    v = np.stack([a.ravel() for a in np.meshgrid(z, y, x, indexing="ij")][::-1], axis=1).reshape(nz + 1, ny + 1, nx + 1, 3).copy()
    move = np.random.default_rng(seed).uniform(-0.05, 0.05, size=v.shape) / np.array([nx, ny, nz])
    v[1:-1, 1:-1, 1:-1] += move[1:-1, 1:-1, 1:-1]
    return np.ascontiguousarray(v.reshape(-1, 3))


def _field(n, seed, dtype=torch.float64):
    return torch.randn(n, generator=torch.Generator("cuda").manual_seed(seed), device="cuda", dtype=torch.float64).to(dtype)


def _specs(case):
    """The boxes and orders of a batched or served mix (a property of the case, not of the seed)."""
    r = np.random.default_rng(case["mix"])
    orders = (3, 5, 7, 9) if case["kind"] == "batch" else (5, 7)
    out = []
    for _ in range(case["count"]):
        E = math.exp(r.uniform(math.log(case["e_lo"]), math.log(case["e_hi"])))
        N = int(orders[r.integers(len(orders))])
        nx = max(1, int(round(E ** (1 / 3))))
        ny = max(1, int(round(math.sqrt(E / nx))))
        out.append((nx, ny, max(1, int(round(E / (nx * ny)))), N))
    return out


_parked = []    # problems whose release the library put off: it holds them while any batch is open


def _release(meshes=()):
    _parked.extend(meshes)
    keep = []
    for m in _parked:
        try:
            m.free()
        except sem.SemError:
            keep.append(m)
    _parked[:] = keep


class _State:
    """Inputs, buffers and handles of one prepared case; the handles are given back with it."""

    def __init__(self, case):
        self.case, self.meshes, self.batch, self.server = case, [], None, None

    def __del__(self):
        torch.cuda.synchronize()
        if self.server is not None:
            self.server.close()
        if self.batch is not None:
            self.batch.free()
        _release(self.meshes)


def _start():
    if sem.stream() is None:
        sem.init(["--device=0"])
        torch.cuda.set_stream(sem.stream())   # the inputs are made on the library's stream


def _assembled(mesh, f):
    mesh.gs(f)
    mesh.mask(f)
    return f


def prepare(case, seed):
    _start()
    _release()
    s, kind = _State(case), case["kind"]
    if kind == "serve":
        s.server = Server(capacity=256, budget_gb=40.0, mode=case["mode"], tol=case["tol"])
        s.requests = []
        for k, (nx, ny, nz, N) in enumerate(_specs(case)):
            n = nx * ny * nz * (N + 1) ** 3
            f = np.random.default_rng([seed, k]).standard_normal(n)
            s.requests.append((nx, ny, nz, N, _vertices(nx, ny, nz, seed + k), f, np.empty(n)))
        return s
    if kind == "batch":
        parts = []
        for k, (nx, ny, nz, N) in enumerate(_specs(case)):
            s.meshes.append(Mesh(nx, ny, nz, N, _vertices(nx, ny, nz, seed + k)))
            parts.append(_assembled(s.meshes[-1], _field(s.meshes[-1].nL, seed + k)))
        s.batch = Batch(s.meshes)
        s.b, s.x = torch.cat(parts), torch.empty(s.batch.nL_total, dtype=torch.float64, device="cuda")
        return s
    nx, ny, nz, N = case["nx"], case["ny"], case["nz"], case["N"]
    m = Mesh(nx, ny, nz, N, _vertices(nx, ny, nz, seed))
    s.meshes.append(m)
    if kind in ("ax", "axg", "ax32"):
        s.x = _field(m.nL, seed, torch.float32 if kind == "ax32" else torch.float64)
        s.y = torch.empty_like(s.x)
    else:
        s.b = _assembled(m, _field(m.nL, seed))
        s.x = torch.empty_like(s.b)
        if kind in ("cg", "pcg"):
            s.hist = torch.empty(case["iters"] + 1, dtype=torch.float64, device="cuda")
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "serve":
        return _serve(s)
    if kind == "batch":
        s.batch.solve(s.b, s.x, tol=case["tol"], mode=case["mode"])
        return s.x
    m = s.meshes[0]
    if kind == "ax":
        m.ax(s.x, s.y)
        return s.y
    if kind == "axg":
        m.axg(s.x, s.y)
        return s.y
    if kind == "ax32":
        m.ax32(s.x, s.y, case["gprec"])
        return s.y
    if kind == "cg":
        m.cg_solve(s.b, s.x, 0.0, case["iters"], s.hist)
        return {"x": s.x, "hist": s.hist}
    if kind == "pcg":
        m.pcg_solve(s.b, s.x, 0.0, case["iters"], s.hist)
        return {"x": s.x, "hist": s.hist}
    m.cg_mixed(s.b, s.x, case["tol"], gprec=case["gprec"])
    return s.x


def _serve(s):
    """All requests arrive together; the client steps the server and fetches each result as it is done."""
    srv, where = s.server, {}
    for k, (nx, ny, nz, N, verts, f, _) in enumerate(s.requests):
        where[srv.submit(nx, ny, nz, N, verts, f, srv.now(), assemble=True)] = k
    left = len(where)
    while left:
        srv.step()
        for ticket in srv.drain():
            srv.result(ticket, s.requests[where[ticket]][-1])
            left -= 1
    return [r[-1] for r in s.requests]


# ---------------------------------------------------------------- work
def _op_flops(E, N):
    nq = N + 1
    return E * (12 * nq ** 4 + 15 * nq ** 3)


def _iterations(E, N, tol):
    """About the CG iterations of a solve to tol (the inner ones in mixed precision): they grow with the sides of the box and with N^1.25."""
    return 0.27 * math.log10(1 / tol) * E ** (1 / 3) * 1.25 * N ** 1.25 + 10


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        b = f = 0.0
        for nx, ny, nz, N in _specs(case):
            E = nx * ny * nz
            n, it = E * (N + 1) ** 3, _iterations(E, N, case["tol"])
            # factors, and three vectors read and written, per iteration
            per = 48 + 48 if case["mode"] == 0 else (12 if case["mode"] == 1 else 24) + 24
            b += n * per * it + 16 * n
            f += (_op_flops(E, N) + 12 * n) * it
        return {"bytes": b, "flops": f}
    E, N = case["nx"] * case["ny"] * case["nz"], case["N"]
    n = E * (N + 1) ** 3
    if kind in ("ax", "axg"):
        return {"bytes": n * (8 + 8 + 48), "flops": _op_flops(E, N)}
    g = {0: 24, 1: 12}.get(case.get("gprec"), 48)
    if kind == "ax32":
        return {"bytes": n * (4 + 4 + g), "flops": _op_flops(E, N)}
    if kind == "mixed":
        it = _iterations(E, N, case["tol"])
        return {"bytes": n * (24 + g) * it + 16 * n, "flops": (_op_flops(E, N) + 12 * n) * it}
    # per iteration: the factors (and the preconditioner), x, r and p read and written
    per = 48 + 48 + (8 if kind == "pcg" else 0)
    return {"bytes": n * per * case["iters"] + 16 * n, "flops": (_op_flops(E, N) + (14 if kind == "pcg" else 12) * n) * case["iters"]}


# ---------------------------------------------------------------- 64-bit values
class _Reference:
    """The assembled operator on one box in plain torch, 64 bits."""

    def __init__(self, nx, ny, nz, N, verts, gprec=None):
        dev, nq = "cuda", N + 1
        P = np.polynomial.legendre.Legendre.basis(N)
        xi = np.concatenate([[-1.0], np.sort(P.deriv().roots().real), [1.0]])
        xi = 0.5 * (xi - xi[::-1])
        w = 2.0 / (N * nq * P(xi) ** 2)
        diff = xi[:, None] - xi[None, :] + np.eye(nq)
        lam = 1.0 / diff.prod(axis=1)
        D = lam[None, :] / lam[:, None] / diff
        np.fill_diagonal(D, 0.0)
        np.fill_diagonal(D, -D.sum(axis=1))
        self.D, self.nq, self.E = torch.tensor(D, device=dev), nq, nx * ny * nz
        v = torch.tensor(verts, device=dev).reshape(nz + 1, ny + 1, nx + 1, 3)
        c = torch.stack([v[a:nz + a, b:ny + b, d:nx + d].reshape(-1, 3) for a in (0, 1) for b in (0, 1) for d in (0, 1)], 1)
        c = (c - c[:, :1]).reshape(self.E, 2, 2, 2, 3)          # corner (t, s, r) relative to the first
        h = torch.tensor(np.stack([0.5 * (1 - xi), 0.5 * (1 + xi)], 1), device=dev)
        dh = torch.tensor([-0.5, 0.5], device=dev, dtype=torch.float64).expand(nq, 2)
        J = [torch.einsum("ecbax,kc,jb,ia->ekjix", c, *(t if q != p else dh for q, t in enumerate((h, h, h)))) for p in (2, 1, 0)]
        cof = [torch.linalg.cross(J[1], J[2]), torch.linalg.cross(J[2], J[0]), torch.linalg.cross(J[0], J[1])]
        det = (J[0] * cof[0]).sum(-1)
        wt = torch.tensor(w[:, None, None] * w[None, :, None] * w[None, None, :], device=dev) / det
        self.G = {}
        for a in range(3):
            for b in range(a, 3):
                g = wt * (cof[a] * cof[b]).sum(-1)
                if gprec == 0:
                    g = g.float().double()
                elif gprec == 1:                                  # one rounding to 8 significant bits
                    m, e = torch.frexp(g)
                    g = torch.ldexp(torch.round(m * 256.0), e - 8)
                self.G[a, b] = self.G[b, a] = g
        ix = [(torch.arange(n, device=dev)[:, None] * N + torch.arange(nq, device=dev)[None, :]) for n in (nx, ny, nz)]
        size = (nx * N + 1, ny * N + 1, nz * N + 1)
        gid = (ix[2][:, None, None, :, None, None] * size[1] + ix[1][None, :, None, None, :, None]) * size[0] + ix[0][None, None, :, None, None, :]
        self.gid, self.nG = gid.reshape(-1), size[0] * size[1] * size[2]
        on = [((i > 0) & (i < n - 1)) for i, n in zip(ix, size)]
        self.free = (on[2][:, None, None, :, None, None] & on[1][None, :, None, None, :, None] & on[0][None, None, :, None, None, :]).reshape(-1)
        self.c = 1.0 / self.sum(torch.ones_like(self.gid, dtype=torch.float64))

    def _d(self, u, axis, t=False):
        D = self.D.T if t else self.D
        return torch.einsum(("ekjm,im->ekji", "ekmi,jm->ekji", "emji,km->ekji")[axis], u, D)

    def ax(self, x):
        u = x.double().reshape(self.E, self.nq, self.nq, self.nq)
        g = [self._d(u, a) for a in range(3)]
        y = 0.0
        for a in range(3):
            y = y + self._d(sum(self.G[a, b] * g[b] for b in range(3)), a, True)
        return y.reshape(-1)

    def diagonal(self):
        D2, d = self.D ** 2, torch.diagonal(self.D)
        G = self.G
        v = torch.einsum("ekjm,mi->ekji", G[0, 0], D2) + torch.einsum("ekmi,mj->ekji", G[1, 1], D2) + torch.einsum("emji,mk->ekji", G[2, 2], D2)
        i, j, k = d[None, None, None, :], d[None, None, :, None], d[None, :, None, None]
        return self.assemble((v + 2.0 * (i * j * G[0, 1] + i * k * G[0, 2] + j * k * G[1, 2])).reshape(-1))

    def sum(self, u):
        return torch.zeros(self.nG, dtype=torch.float64, device="cuda").index_add_(0, self.gid, u)[self.gid]

    def assemble(self, u):
        return self.sum(u) * self.free

    def dot(self, u, v):
        return (self.c * u * v).sum()

    def cg(self, b, iters, tol=0.0, dinv=None):
        """x and the residual norms after each iteration."""
        x, r, p = torch.zeros_like(b), b.clone(), torch.zeros_like(b)
        z = r if dinv is None else dinv * r
        rho, beta, hist = self.dot(r, z), 0.0, [self.dot(r, r).sqrt()]
        for k in range(iters):
            p = z + beta * p
            w = self.assemble(self.ax(p))
            alpha = rho / self.dot(p, w)
            x, r = x + alpha * p, r - alpha * w
            z = r if dinv is None else dinv * r
            new = self.dot(r, z)
            beta, rho = new / rho, new
            hist.append(self.dot(r, r).sqrt())
            if tol and k % 16 == 15 and hist[-1] <= tol * hist[0]:
                break
        return x, torch.stack(hist)


def exact(case, seed):
    _start()
    kind = case["kind"]
    if kind in ("batch", "serve"):
        specs = _specs(case)
        if sum(a * b * c * (N + 1) ** 3 for a, b, c, N in specs) > 6e6:   # about a millisecond an iteration and problem
            return None
        out = []
        for k, (nx, ny, nz, N) in enumerate(specs):
            R = _Reference(nx, ny, nz, N, _vertices(nx, ny, nz, seed + k))
            n = len(R.gid)
            f = _field(n, seed + k) if kind == "batch" else torch.from_numpy(np.random.default_rng([seed, k]).standard_normal(n)).cuda()
            out.append(R.cg(R.assemble(f), 4000, tol=1e-13)[0])
        return torch.cat(out) if kind == "batch" else [x.cpu().numpy() for x in out]
    nx, ny, nz, N = case["nx"], case["ny"], case["nz"], case["N"]
    if kind == "mixed" and nx * ny * nz * (N + 1) ** 3 > 2e6:             # thousands of iterations of tens of milliseconds
        return None
    R = _Reference(nx, ny, nz, N, _vertices(nx, ny, nz, seed), case.get("gprec") if kind == "ax32" else None)
    f = _field(len(R.gid), seed, torch.float32 if kind == "ax32" else torch.float64)
    if kind in ("ax", "ax32"):
        return R.ax(f)
    if kind == "axg":
        return R.assemble(R.ax(f))
    b = R.assemble(f)
    if kind == "mixed":
        return R.cg(b, 6000, tol=1e-13)[0]
    d = R.diagonal() if kind == "pcg" else None
    x, hist = R.cg(b, case["iters"], dinv=None if d is None else torch.where(d > 0, 1.0 / d, 0.0))
    return {"x": x, "hist": hist}
