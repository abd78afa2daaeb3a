"""The work that users of this library have it do, as timed cases.

Each case is one call sequence through the public entry points
(paper_2001_05798_gb300.gw and .adjoint) on seeded synthetic fields:

  solve      one right-hand side on a resident hierarchy (gw_pcg_solve), in the
             FP64, FP32-mixed, BF16- or FP16-stored form
  request    a whole flow problem from conductivities on the device:
             assembly, AMG setup, solve, Darcy face velocities
  host       gw.solve on host arrays, as a script calls it
  many       several right-hand sides on one hierarchy (gw_pcg_solve_many)
  adjoint    heads(lnK) and the gradient of a head misfit, setup included
  transient  two implicit steps on a cached hierarchy (gw_hierarchy_shift and solve)
  batch      several resident solves of different sizes in one gw_batch

Every solve runs to the paper's relative residual 1e-12, at which the heads do
not depend on the iteration at which the solve stopped.
"""
import math

import numpy as np
import torch

from paper_2001_05798_gb300 import adjoint, gw
from paper_2001_05798_gb300 import workload as wl

FORMS = {"fp64": gw.GW_PREC_FP64, "fp32": gw.GW_PREC_MIXED32, "fp16": gw.GW_PREC_MIXED16, "bf16": gw.GW_PREC_MIXEDBF16}
# heads of 1 and 0 on the x faces, or h = 0 on the top face with pumping wells below
BCS = {"x": ((1, 1, 0, 0, 0, 0), (1.0, 0.0, 0.0, 0.0, 0.0, 0.0)),
       "top": ((0, 0, 0, 0, 0, 1), (0.0, 0.0, 0.0, 0.0, 0.0, 0.0))}


def _case(kind, nx, ny, nz, **kw):
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, var=4.0, corr=8.0, kz=1.0, bc="x", wells=0, form="fp32", tol=1e-12, k=1,
             sides="")
    c.update(kw)
    return c


def listed():
    def named(name, c):
        return dict(c, name=name)

    return [
        # the small verification problem: 2D homogeneous flow, where launches and latency count
        named("solve_2d_128", _case("solve", 128, 128, 1, var=0.0)),
        # the benchmark: 128^3 heterogeneous field, hierarchy resident
        named("solve_128", _case("solve", 128, 128, 128)),
        # a serving-sized cube of odd side: no aligned row length anywhere
        named("solve_odd_117", _case("solve", 117, 117, 117, var=2.5)),
        # the reference precision, at the adjoint study's size
        named("solve_fp64_96", _case("solve", 96, 96, 96, var=2.0, corr=6.0, form="fp64")),
        # the largest configured grid: layered aquifer with wells, BF16-stored fine stencil
        named("solve_layered_bf16", _case("solve", 256, 256, 128, var=1.0, corr=32.0, kz=10.0, bc="top", wells=16,
                                          form="bf16")),
        # a small and a large request of the serving stream, from conductivities to velocities
        named("request_45", _case("request", 45, 45, 45, var=1.5, corr=6.0)),
        named("request_160", _case("request", 160, 160, 160, var=3.0, corr=12.0)),
        # a script's one call on host arrays: the 275,000-cell 2D grid
        named("host_2d_550x500", _case("host", 550, 500, 1, var=4.0, corr=10.0)),
        # eight well scenarios on one hierarchy
        named("many_128_k8", _case("many", 128, 128, 128, k=8)),
        # sensitivities of 64 observed heads with respect to every cell's ln K
        named("adjoint_96", _case("adjoint", 96, 96, 96, var=2.0, corr=6.0, k=64)),
        # implicit time stepping with the hierarchy kept
        named("transient_128", _case("transient", 128, 128, 128)),
        # a sweep's resident solves of mixed sizes advancing together
        named("batch_8", _case("batch", 0, 0, 0, var=2.0, corr=8.0, sides="33,40,45,52,57,64,71,96")),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "request", "request", "host", "many", "adjoint", "transient", "batch"])
    var, corr = round(rng.uniform(0.5, 4.0), 2), round(rng.uniform(4.0, 16.0), 1)
    if kind == "solve":
        form = rng.choice(["fp32", "fp32", "fp64", "bf16", "fp16"])
        if rng.random() < 0.25:
            return _case("solve", _log_int(rng, 100, 700), _log_int(rng, 100, 700), 1, var=var, corr=corr, form=form)
        side = _log_int(rng, 32, 150)
        nx, ny, nz = (max(24, int(side * rng.uniform(0.7, 1.3))) for _ in range(3))
        if rng.random() < 0.3:
            return _case("solve", nx, ny, nz, var=round(rng.uniform(0.5, 1.5), 2), corr=corr, kz=10.0, bc="top",
                         wells=rng.randint(4, 16), form=form)
        return _case("solve", nx, ny, nz, var=var, corr=corr, form=form)
    if kind == "request":
        s = _log_int(rng, 32, 160)
        return _case("request", s, s, s, var=var, corr=corr)
    if kind == "host":
        return _case("host", _log_int(rng, 100, 700), _log_int(rng, 100, 700), 1, var=var, corr=corr)
    if kind == "many":
        s = _log_int(rng, 32, 110)
        return _case("many", s, s, s, var=var, corr=corr, k=rng.randint(2, 11))
    if kind == "adjoint":
        s = _log_int(rng, 32, 110)
        return _case("adjoint", s, s, s, var=var, corr=corr, k=rng.randint(16, 128))
    if kind == "transient":
        s = _log_int(rng, 32, 128)
        return _case("transient", s, s, s, var=var, corr=corr)
    sides = ",".join(str(_log_int(rng, 32, 96)) for _ in range(rng.randint(2, 8)))
    return _case("batch", 0, 0, 0, var=var, corr=corr, sides=sides)


def _inputs(c, seed, nx, ny, nz):
    """Conductivities (device) and the source of one problem."""
    n = nx * ny * nz
    if c["var"] > 0.0:
        corr = (c["corr"], c["corr"], c["corr"] / 8.0) if c["bc"] == "top" else c["corr"]
        K = torch.exp(wl.lnk_field_device(nx, ny, nz, c["var"], corr, seed))
    else:
        K = torch.full((n,), 1.0 + 0.01 * (seed % 97), dtype=torch.float64, device="cuda")
    q = None
    if c["wells"]:
        q = torch.from_numpy(wl.wells(nx, ny, nz, c["wells"], seed, -1e-3)[0]).cuda()
    return K, (K if c["kz"] == 1.0 else K / c["kz"]), q


def _scenarios(c, seed, b):
    """b and k - 1 further right-hand sides, each with six random wells added."""
    rng = np.random.default_rng(seed)
    B = b.repeat(c["k"], 1)
    for r in range(1, c["k"]):
        idx = torch.from_numpy(rng.choice(b.numel(), 6, replace=False)).cuda()
        B[r, idx] += torch.from_numpy(rng.uniform(-1e-3, 1e-3, 6)).cuda()
    return B.contiguous()


def _observations(c, seed, n):
    rng = np.random.default_rng(seed + 1)
    return (torch.from_numpy(np.sort(rng.choice(n, c["k"], replace=False))).cuda(),
            torch.from_numpy(rng.uniform(0.2, 0.8, c["k"])).cuda())


def _storage(K, nx, ny, nz, seed):
    """Storage terms of two steps, 0.5 % of a cell's summed conductivity scale,
    10 % apart, and the heads before the first step."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    s = 0.005 * 2.0 * K.clamp(max=1.0) * (0.5 + 0.5 * torch.rand(K.numel(), generator=g, dtype=torch.float64, device="cuda"))
    # small against the row's own diagonal everywhere: bounded by the smallest neighbour
    f = K.reshape(nz, ny, nx)
    m = torch.nn.functional.max_pool3d(-f[None, None], 3, 1, 1)[0, 0].neg().reshape(-1)
    s = torch.minimum(s, 0.005 * m)
    h0 = torch.linspace(1.0, 0.0, nx, dtype=torch.float64, device="cuda").repeat(ny * nz)
    return s * 0.95, s * 1.05, h0


def _resident(c, seed, nx, ny, nz):
    K, Kz, q = _inputs(c, seed, nx, ny, nz)
    b = torch.empty_like(K)
    bct, bcv = BCS[c["bc"]]
    A, _ = gw.gw_assemble(nx, ny, nz, K, K, Kz, bct, bcv, q, b_out=b)
    return K, b, gw.Hierarchy(A, prec=FORMS[c["form"]])


def prepare(case, seed):
    c = case
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    s = dict(c=c)
    if c["kind"] == "batch":
        sides = [int(t) for t in c["sides"].split(",")]
        s["solves"] = [_resident(c, seed + r, m, m, m)[1:] for r, m in enumerate(sides)]
        s["batch"] = gw.Batch(len(sides))
        s["h"] = [torch.empty_like(b) for b, _ in s["solves"]]
        return s
    if c["kind"] in ("request", "host", "adjoint"):
        K, Kz, q = _inputs(c, seed, nx, ny, nz)
        if c["kind"] == "host":
            s["K"] = K.cpu().numpy()
        elif c["kind"] == "adjoint":
            s["lnK"] = torch.log(K).requires_grad_(True)
            s["obs"], s["hobs"] = _observations(c, seed, K.numel())
        else:
            s["K"], s["Kz"], s["q"] = K, Kz, q
        return s
    K, b, H = _resident(c, seed, nx, ny, nz)
    s["H"] = H
    if c["kind"] == "many":
        s["B"] = _scenarios(c, seed, b)
        s["X"] = torch.empty_like(s["B"])
    elif c["kind"] == "transient":
        s["b"] = b
        s["s1"], s["s2"], s["h0"] = _storage(K, nx, ny, nz, seed)
        H.shift(s["s1"])
        s["h1"], s["h2"] = torch.empty_like(b), torch.empty_like(b)
    else:
        s["b"], s["h"] = b, torch.empty_like(b)
    return s


def run(state):
    s, c = state, state["c"]
    kind, nx, ny, nz, tol = c["kind"], c["nx"], c["ny"], c["nz"], c["tol"]
    if kind == "solve":
        return s["H"].solve(s["b"], s["h"], tol=tol)[0]
    if kind == "request":
        bct, bcv = BCS[c["bc"]]
        K, Kz = s["K"], s["Kz"]
        b = torch.empty_like(K)
        A, _ = gw.gw_assemble(nx, ny, nz, K, K, Kz, bct, bcv, s["q"], b_out=b)
        h = gw.Hierarchy(A, prec=FORMS[c["form"]]).solve(b, tol=tol)[0]
        v = [torch.empty(m, dtype=torch.float64, device=K.device)
             for m in ((nx + 1) * ny * nz, nx * (ny + 1) * nz, nx * ny * (nz + 1))]
        gw.gw_darcy_flux(nx, ny, nz, K, h, v[0], v[1], v[2], Ky=K, Kz=Kz, bct=bct, bcv=bcv)
        return [h] + v
    if kind == "host":
        return gw.solve(nx, ny, nz, s["K"], tol=tol)[0]
    if kind == "many":
        return s["H"].solve_many(s["B"], s["X"], tol=tol)[0]
    if kind == "adjoint":
        h = adjoint.heads(s["lnK"], nx, ny, nz, tol=tol)
        J = ((h[s["obs"]] - s["hobs"]) ** 2).sum()
        return [h.detach(), torch.autograd.grad(J, s["lnK"])[0]]
    if kind == "transient":
        H, b = s["H"], s["b"]
        H.shift(s["s1"])
        H.solve(b + s["s1"] * s["h0"], s["h1"], tol=tol)
        H.shift(s["s2"])
        H.solve(b + s["s2"] * s["h1"], s["h2"], tol=tol)
        return [s["h1"], s["h2"]]
    B, left = s["batch"], {}
    for r, (b, H) in enumerate(s["solves"]):
        left[B.add(H, b, tol=tol)] = r
    while left:
        B.run(64)
        for slot in B.finished():
            B.take(slot, s["h"][left.pop(slot)])
    return s["h"]


def work(case):
    """Every input once, every output once; operations of one application of the operator."""
    c = case
    if c["kind"] == "batch":
        n = sum(int(t) ** 3 for t in c["sides"].split(","))
    else:
        n = c["nx"] * c["ny"] * c["nz"]
    # vectors of n doubles read or written; a resident operator is its 7-point stencil in FP64
    vectors = {"solve": 4 + 2, "request": 1 + 4, "host": 1 + 1, "many": 4 + 2 * c["k"], "adjoint": 1 + 2,
               "transient": 4 + 6, "batch": 4 + 2}[c["kind"]]
    solves = {"many": c["k"], "adjoint": 2, "transient": 2}.get(c["kind"], 1)
    return {"bytes": 8.0 * n * vectors, "flops": 13.0 * n * solves}


# ---------------------------------------------------- the same in plain torch, 64 bits --
class _Flow:
    """The 7-point operator of a conductivity field with its Dirichlet faces."""

    def __init__(self, nx, ny, nz, K, Kz, q, bc, shift=None):
        shape = (nz, ny, nx)
        self.K = [k.reshape(shape) for k in (K, K, Kz)]
        self.T = []
        for d, k in enumerate(self.K):
            a, b = k.narrow(2 - d, 0, shape[2 - d] - 1), k.narrow(2 - d, 1, shape[2 - d] - 1)
            self.T.append(2.0 * a * b / (a + b))
        self.bct, self.bcv = BCS[bc]
        diag, rhs = torch.zeros_like(self.K[0]), torch.zeros_like(self.K[0])
        for d, T in enumerate(self.T):
            m = shape[2 - d]
            diag.narrow(2 - d, 0, m - 1).add_(T)
            diag.narrow(2 - d, 1, m - 1).add_(T)
            for side in range(2):
                if self.bct[2 * d + side]:
                    at = 0 if side == 0 else m - 1
                    tb = 2.0 * self.K[d].narrow(2 - d, at, 1)
                    diag.narrow(2 - d, at, 1).add_(tb)
                    rhs.narrow(2 - d, at, 1).add_(tb * self.bcv[2 * d + side])
        if shift is not None:
            diag = diag + shift.reshape(shape)
        self.diag, self.shape = diag, shape
        self.b = rhs.reshape(-1) + (q if q is not None else 0.0)

    def apply(self, x):
        x = x.reshape(self.shape)
        y = self.diag * x
        for d, T in enumerate(self.T):
            m = self.shape[2 - d]
            if m < 2:
                continue
            lo, hi = x.narrow(2 - d, 0, m - 1), x.narrow(2 - d, 1, m - 1)
            y.narrow(2 - d, 0, m - 1).sub_(T * hi)
            y.narrow(2 - d, 1, m - 1).sub_(T * lo)
        return y.reshape(-1)

    def solve(self, b, tol=1e-13):
        """Jacobi-preconditioned CG, restarted from the true residual."""
        w = 1.0 / self.diag.reshape(-1)
        x = torch.zeros_like(b)
        bn = float(b.norm())
        for _ in range(6):
            r = b - self.apply(x)
            rn = float(r.norm())
            if bn == 0.0 or rn <= tol * bn:
                break
            stop, z = max(1e-8 * rn, 0.3 * tol * bn), w * r
            p, rz, y = z.clone(), torch.dot(r, z), torch.zeros_like(b)
            for it in range(20000):
                Ap = self.apply(p)
                a = rz / torch.dot(p, Ap)
                y += a * p
                r -= a * Ap
                if it % 64 == 63 and float(r.norm()) <= stop:
                    break
                z = w * r
                new = torch.dot(r, z)
                p = z + (new / rz) * p
                rz = new
            x = x + y
        return x

    def velocities(self, h):
        h = h.reshape(self.shape)
        out = []
        for d in range(3):
            m, ax = self.shape[2 - d], 2 - d
            size = list(self.shape)
            size[ax] = m + 1
            v = torch.zeros(size, dtype=h.dtype, device=h.device)
            if m > 1:
                v.narrow(ax, 1, m - 1).copy_(self.T[d] * (h.narrow(ax, 0, m - 1) - h.narrow(ax, 1, m - 1)))
            if self.bct[2 * d]:
                v.narrow(ax, 0, 1).copy_(2.0 * self.K[d].narrow(ax, 0, 1) * (self.bcv[2 * d] - h.narrow(ax, 0, 1)))
            if self.bct[2 * d + 1]:
                v.narrow(ax, m, 1).copy_(2.0 * self.K[d].narrow(ax, m - 1, 1)
                                         * (h.narrow(ax, m - 1, 1) - self.bcv[2 * d + 1]))
            out.append(v.reshape(-1))
        return out


def exact(case, seed):
    c = case
    nx, ny, nz, kind = c["nx"], c["ny"], c["nz"], c["kind"]
    if kind == "batch":
        out = []
        for r, m in enumerate(int(t) for t in c["sides"].split(",")):
            K, Kz, q = _inputs(c, seed + r, m, m, m)
            F = _Flow(m, m, m, K, Kz, q, c["bc"])
            out.append(F.solve(F.b))
        return out
    K, Kz, q = _inputs(c, seed, nx, ny, nz)
    if kind == "transient":
        s1, s2, h0 = _storage(K, nx, ny, nz, seed)
        h, out = h0, []
        for st in (s1, s2):
            F = _Flow(nx, ny, nz, K, Kz, q, c["bc"], shift=st)
            h = F.solve(F.b + st * h)
            out.append(h)
        return out
    if kind == "adjoint":
        K = Kz = torch.exp(torch.log(K))
    F = _Flow(nx, ny, nz, K, Kz, q, c["bc"])
    if kind == "many":
        return torch.stack([F.solve(r) for r in _scenarios(c, seed, F.b)])
    h = F.solve(F.b)
    if kind == "request":
        return [h] + F.velocities(h)
    if kind == "adjoint":
        obs, hobs = _observations(c, seed, K.numel())
        dJ = torch.zeros_like(h)
        dJ[obs] = 2.0 * (h[obs] - hobs)
        lam = F.solve(dJ)
        lnK = torch.log(K).requires_grad_(True)
        k = torch.exp(lnK)
        G = _Flow(nx, ny, nz, k, k, None, c["bc"])
        return [h, torch.autograd.grad(torch.dot(lam, G.b - G.apply(h)), lnK)[0]]
    return h.cpu().numpy() if kind == "host" else h
