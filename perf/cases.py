"""What a user of this library has it do, as cases that can be timed and checked.

A case names a grid (nx, ny, nz; nz = 1 is the 2D problem), a boundary condition per axis, the grid spacings, a
precision form and what is called:

  solve   one potential from one charge density, zero initial guess (Plan.solve)
  step    the next time step of a simulation: warm start from the previous potential (Plan.solve)
  batch   many grids, some right-hand sides each, in one call (tpcg_solve_batched, one plan and stream each)
  stream  a list of densities in pinned host memory, potentials back to host memory (Plan.solve_host_stream)
  precond one application of the pseudoinverse (Plan.precond)
  post    what follows a solve: the electric field and L ups (Plan.efield, Plan.laplacian)

The densities are Gaussian charged defects (+-1, sigma of a few cells) plus, for films, a little noise, scaled to
||eta|| = 1/N as in the benchmark; time steps move 1 % of the defects.
"""
import math

import numpy as np
import torch

from paper_2501_03377_gb300.binding import TPCG_OPT_SWEEP_GRAIN, TPCG_ZERO_GUESS, Plan, tpcg_solve_batched

BCS = ("P", "D", "N", "DN", "ND")
MAXIT = 60


def case(kind, nx, ny, nz, bc, prec, h="1,1,1", tol=1e-10, count=1, defects=200, sigma=1.5, noise=0.0, **name):
    return dict(name, kind=kind, nx=nx, ny=ny, nz=nz, bc=bc, prec=prec, h=h, tol=tol, count=count, defects=defects,
                sigma=sigma, noise=noise)


def listed():
    return [
        # the smallest call: a 2D plane, FP64 throughout; launches and latency are all of it
        case("solve", 64, 64, 1, "D,D,D", "fp64", tol=1e-12, defects=8, sigma=3.0, name="plane64_fp64"),
        # a thin film, FP64 throughout (the default precision form of a plan)
        case("solve", 128, 128, 64, "P,P,DN", "fp64", noise=1e-3, name="film128_fp64"),
        # the benchmark's cuboid in the FP64 form, the comparison arm of its headline: the largest work
        case("solve", 256, 256, 128, "P,P,N", "fp64", defects=2000, sigma=2.5, name="cuboid256_fp64"),
        # the same cuboid in the headline's form (split BF16) and in the other mixed form in use (scaled FP16)
        case("solve", 256, 256, 128, "P,P,N", "bf16x3", defects=2000, sigma=2.5, name="cuboid256_split"),
        case("solve", 256, 256, 128, "P,P,N", "fp16", defects=2000, sigma=2.5, name="cuboid256_fp16"),
        # odd extents and unequal spacings: every sweep's general form, ragged tiles, padded rows
        case("solve", 255, 201, 97, "ND,P,D", "bf16x3", h="1,0.5,2", defects=800, name="odd255_split"),
        # time steps of a small and of a large sample, as a server's sessions issue them
        case("step", 64, 64, 32, "P,D,N", "bf16x3", name="step64_split"),
        case("step", 224, 224, 192, "D,P,DN", "bf16x3", defects=600, name="step224_split"),
        # a sweep over samples: grids of mixed sizes and boundary conditions in one call, 1 to 3 densities each
        case("batch", 160, 160, 96, "mixed", "bf16x3", count=12, noise=1e-3, name="batch12_split"),
        # densities and potentials in pinned host memory, copies overlapped with the solves
        case("stream", 192, 192, 96, "P,P,N", "bf16x3", count=6, defects=600, name="stream192_split"),
        # one application of the FP64 preconditioner on extents that no tile divides
        case("precond", 150, 100, 75, "N,P,D", "fp64", name="precond150_fp64"),
        # after each solve: the field of the potential and its Laplacian
        case("post", 256, 256, 128, "P,P,N", "fp64", defects=2000, sigma=2.5, name="post256"),
    ]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("solve", "solve", "solve", "step", "step", "batch", "stream", "precond", "post"))
    flat = kind in ("solve", "precond") and rng.random() < 0.2
    nx, ny = _between(rng, 32, 256), _between(rng, 32, 256)
    nz = 1 if flat else _between(rng, 16, 192)
    if rng.random() < 0.5:  # simulations mostly take multiples of 16
        nx, ny = max(32, nx // 16 * 16), max(32, ny // 16 * 16)
        nz = nz if flat else max(16, nz // 16 * 16)
    prec = rng.choice(("fp64", "fp64", "bf16x3", "bf16x3", "bf16x3", "fp16", "tf32"))
    if kind in ("precond", "post"):
        prec = "fp64"
    if kind in ("batch", "stream") and prec == "fp64":
        prec = "bf16x3"
    if kind == "batch":  # the grids of a batch are drawn up to this one
        nx, ny, nz = rng.choice((96, 128, 160)), rng.choice((96, 128, 160)), rng.choice((64, 96))
    bc = "mixed" if kind == "batch" else ",".join(rng.choice(BCS) for _ in range(3))
    h = rng.choice(("1,1,1", "1,1,1", "1,1,1", "1,0.5,2", "0.8,0.8,1.1"))
    count = {"batch": rng.randint(6, 12), "stream": rng.randint(3, 6)}.get(kind, 1)
    if kind == "stream":
        nx, ny, nz = min(nx, 192), min(ny, 192), min(nz, 96)
    while nx * ny * nz * (nx + ny + nz) > 256 * 256 * 128 * 640:  # no larger than the largest listed case
        nz -= nz // 4
    defects = max(8, min(2000, nx * ny * nz // 5000))
    return case(kind, nx, ny, nz, bc, prec, h=h, count=count, defects=defects, sigma=rng.choice((1.5, 2.5, 3.0)))


# ----------------------------------------------------------------------------------------------- the inputs
def _grids(c):
    """(nx, ny, nz, bcs, h, right-hand sides) of every plan of a case."""
    h = tuple(float(v) for v in c["h"].split(","))
    if c["kind"] != "batch":
        return [(c["nx"], c["ny"], c["nz"], tuple(c["bc"].split(",")), h, c["count"] if c["kind"] == "stream" else 1)]
    r = np.random.default_rng(c["nx"] * 1000003 + c["ny"] * 1009 + c["nz"] * 31 + c["count"])
    out = []
    for s in range(c["count"]):
        nx, ny = (int(r.choice([v for v in (64, 96, 128, 160) if v <= c[a]])) for a in ("nx", "ny"))
        nz = int(r.choice([v for v in (32, 64, 96) if v <= c["nz"]]))
        out.append((nx, ny, nz, tuple(str(r.choice(BCS)) for _ in range(3)), h, int(r.integers(1, 4))))
    return out


def _density(nx, ny, nz, bcs, defects, sigma, noise, gen, moved=0.0):
    """Gaussian charged defects on a (nz, ny, nx) grid; with moved > 0 also the field after that share of the
    defects has moved: (before, after), scaled alike."""
    dims = (nx, ny, nz)
    pos = torch.rand(defects, 3, generator=gen, device="cuda", dtype=torch.float64)
    charge = torch.where(torch.rand(defects, generator=gen, device="cuda") < 0.5, -1.0, 1.0).double()
    to = torch.rand(max(1, int(defects * moved)), 3, generator=gen, device="cuda", dtype=torch.float64)

    def field(pos):
        g = []
        for m, n in enumerate(dims):
            i = torch.arange(n, device="cuda", dtype=torch.float64)
            d = (i[None, :] - pos[:, m : m + 1] * n).abs() if n > 1 else torch.zeros(defects, 1, device="cuda", dtype=torch.float64)
            if bcs[m] == "P":
                d = torch.minimum(d, n - d)
            w = torch.exp(-0.5 * (d / sigma) ** 2)
            g.append(w / w.sum(1, keepdim=True))
        out = torch.zeros(nz, ny * nx, device="cuda", dtype=torch.float64)
        for a in range(0, defects, 500):  # separable blobs, a few hundred at a time
            xy = ((charge[a : a + 500, None] * g[1][a : a + 500])[:, :, None] * g[0][a : a + 500][:, None, :]).reshape(-1, ny * nx)
            out += (g[2][a : a + 500].T.float() @ xy.float()).double()
        return out.reshape(nz, ny, nx)

    eta = field(pos)
    scale = 1.0 / (eta.numel() * eta.norm().item())
    if noise:
        eta = eta + noise * torch.randn(eta.shape, generator=gen, device="cuda", dtype=torch.float64)
        scale = 1.0 / (eta.numel() * eta.norm().item())
    if not moved:
        return eta * scale
    pos = pos.clone()
    pos[: to.shape[0]] = to
    return eta * scale, field(pos) * scale


def _lap1d(n, bc, h):
    """The 1D minus-Laplacian of an axis with its boundary rows, divided by h^2 (NumPy, FP64)."""
    L = 2.0 * np.eye(n) - np.eye(n, k=1) - np.eye(n, k=-1)
    if bc == "P":
        L[0, -1] -= 1.0
        L[-1, 0] -= 1.0
    if bc in ("N", "ND"):
        L[0, 0] = 1.0
    if bc in ("N", "DN"):
        L[-1, -1] = 1.0
    return L / (h * h)


def _axes(nx, ny, nz, bcs, h):
    out = []
    for n, bc, hh in zip((nx, ny, nz), bcs, h):
        L = _lap1d(n, bc, hh) if n > 1 else np.zeros((1, 1))
        lam, V = np.linalg.eigh(L)
        out.append((torch.from_numpy(L).cuda(), torch.from_numpy(lam).cuda(), torch.from_numpy(V).cuda()))
    return out


def _modes(t, mx, my, mz):
    """mz (x) my (x) mx applied to t[z, y, x]."""
    t = t @ mx.T
    t = my @ t
    return (mz @ t.reshape(t.shape[0], -1)).reshape(t.shape)


def _singular(nz, bcs):
    return all(b in ("P", "N") for b in bcs[: 3 if nz > 1 else 2])


def _pinv(eta, ax, singular):
    """The pseudoinverse of the Kronecker sum applied to eta, in 64 bits."""
    (_, lx, vx), (_, ly, vy), (_, lz, vz) = ax
    t = _modes(eta, vx.T, vy.T, vz.T)
    lam = lx[None, None, :] + ly[None, :, None] + lz[:, None, None]
    if singular:
        lam[0, 0, 0] = 1.0
    t = t / lam
    if singular:
        t[0, 0, 0] = 0.0
    return _modes(t, vx, vy, vz)


def _apply(u, ax):
    (Lx, _, _), (Ly, _, _), (Lz, _, _) = ax
    return u @ Lx.T + Ly @ u + (Lz @ u.reshape(u.shape[0], -1)).reshape(u.shape)


def _potential(eta, ax, singular):
    """The (minimum-norm) solution of L u = eta, refined once."""
    if singular:
        eta = eta - eta.mean()
    u = _pinv(eta, ax, singular)
    u = u + _pinv(eta - _apply(u, ax), ax, singular)
    return u - u.mean() if singular else u


def _inputs(c, seed):
    """Per plan: a list of (density, previous potential or None)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 17)
    out = []
    for nx, ny, nz, bcs, h, nrhs in _grids(c):
        ax = _axes(nx, ny, nz, bcs, h) if c["kind"] in ("step", "post") else None
        rhs = []
        for _ in range(nrhs):
            a = (nx, ny, nz, bcs, c["defects"], c["sigma"], c["noise"], gen)
            if c["kind"] == "step":
                before, eta = _density(*a, moved=0.01)
                rhs.append((eta, _potential(before, ax, _singular(nz, bcs))))
            elif c["kind"] == "post":
                rhs.append((None, _potential(_density(*a), ax, _singular(nz, bcs))))
            else:
                rhs.append((_density(*a), None))
        out.append(rhs)
    return out


# ----------------------------------------------------------------------------------------------- the calls
class State:
    pass


def prepare(c, seed):
    s = State()
    s.c, grids, inputs = c, _grids(c), _inputs(c, seed)
    s.streams = [torch.cuda.Stream() for _ in grids] if c["kind"] == "batch" else []
    s.plans = [Plan(nx, ny, nz, bcs, h=h, prec=c["prec"], stream=s.streams[i].cuda_stream if s.streams else None)
               for i, (nx, ny, nz, bcs, h, _) in enumerate(grids)]
    if c["kind"] == "batch":
        for p in s.plans:
            p.set_option(TPCG_OPT_SWEEP_GRAIN, 16)  # as the header advises for many small plans at once
        s.eta = [torch.stack([e for e, _ in rhs]) for rhs in inputs]
        s.ups = [torch.zeros_like(e) for e in s.eta]
    elif c["kind"] == "stream":
        s.eta = [e.cpu().pin_memory() for e, _ in inputs[0]]
        s.ups = [torch.zeros(e.shape, dtype=torch.float64).pin_memory() for e in s.eta]
    elif c["kind"] == "post":
        s.u = inputs[0][0][1]
        s.out = [torch.empty_like(s.u) for _ in range(4 if c["nz"] > 1 else 3)]
    else:
        s.eta, s.prev = inputs[0][0]
        s.ups = torch.zeros_like(s.eta)
    return s


def run(s):
    c, plan = s.c, s.plans[0]
    if c["kind"] == "solve":
        plan.solve(s.eta, s.ups, tol=c["tol"], maxit=MAXIT, zero_guess=True)
        return s.ups
    if c["kind"] == "step":
        s.ups.copy_(s.prev)
        plan.solve(s.eta, s.ups, tol=c["tol"], maxit=MAXIT)
        return s.ups
    if c["kind"] == "batch":
        tpcg_solve_batched([p.handle for p in s.plans], [e.shape[0] for e in s.eta], [e.data_ptr() for e in s.eta],
                           [u.data_ptr() for u in s.ups], [c["tol"]] * len(s.plans), MAXIT, TPCG_ZERO_GUESS)
        return s.ups
    if c["kind"] == "stream":
        plan.solve_host_stream(s.eta, s.ups, tol=c["tol"], maxit=MAXIT, zero_guess=True)
        return s.ups
    if c["kind"] == "precond":
        plan.precond(s.eta, s.ups)
        return s.ups
    plan.efield(s.u, s.out[1], s.out[2], s.out[3] if c["nz"] > 1 else None)
    plan.laplacian(s.u, s.out[0])
    return s.out


def work(c):
    """One application of the pseudoinverse per right-hand side (six mode products; the fewest a solve can do) and
    each input read and each output written once; post: the stencils' arithmetic."""
    b = f = 0.0
    for nx, ny, nz, _, _, nrhs in _grids(c):
        N = float(nx) * ny * nz
        if c["kind"] == "post":
            b += 8.0 * N * (5 if nz > 1 else 4)
            f += N * (13 if nz > 1 else 9)
        else:
            b += nrhs * 8.0 * N * (3 if c["kind"] == "step" else 2)
            f += nrhs * 4.0 * N * (nx + ny + (nz if nz > 1 else 0))
    return {"bytes": b, "flops": f}


def exact(c, seed):
    """The same in 64 bits by dense eigenbases of the assembled 1D operators (and, for the field, shifted copies)."""
    inputs = _inputs(c, seed)
    res = []
    for (nx, ny, nz, bcs, h, _), rhs in zip(_grids(c), inputs):
        ax, sing = _axes(nx, ny, nz, bcs, h), _singular(nz, bcs)
        if c["kind"] == "precond":
            return _pinv(rhs[0][0], ax, sing)
        if c["kind"] == "post":
            u = rhs[0][1]
            out = [_apply(u, ax)]
            for m in range(3 if nz > 1 else 2):
                d = 2 - m
                first, last = u.narrow(d, 0, 1), u.narrow(d, u.shape[d] - 1, 1)
                lo = last if bcs[m] == "P" else first if bcs[m] in ("N", "ND") else torch.zeros_like(first)
                hi = first if bcs[m] == "P" else last if bcs[m] in ("N", "DN") else torch.zeros_like(first)
                e = torch.cat([lo, u, hi], d)
                out.append((e.narrow(d, 0, u.shape[d]) - e.narrow(d, 2, u.shape[d])) * (0.5 / h[m]))
            return out
        res.append(torch.stack([_potential(e, ax, sing) for e, _ in rhs]))
    if c["kind"] == "batch":
        return res
    return [u for u in res[0]] if c["kind"] == "stream" else res[0][0]
