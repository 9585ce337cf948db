"""Measured workloads of the library: what a reservoir simulator has it do.

A simulator's Newton loop keeps one context per grid (the pattern never changes)
and, in every Newton iteration, uploads new Jacobian values, rebuilds the
preconditioner and solves (``newton``).  Around it: several right-hand sides on
one set-up context (``resolve``), the preconditioner or the operator inside a
caller's own Krylov loop (``precond``, ``spmv``, ``residual``), many small
systems solved in one launch (``batch``) and independent requests given to a
server (``serve``).

``listed`` returns the fixed cases, ``draw`` one more of the same ranges,
``prepare`` a case's inputs and contexts, ``run`` one pass, ``work`` the bytes
and operations that pass cannot do without and ``exact`` its outputs in FP64
PyTorch where those can be had quickly.

The matrices are seeded thermal-compositional Jacobians, 4x4 blocks on a
Cartesian grid or on a jittered point cloud joined to its nearest neighbours:
Darcy fluxes in the pressure column, upwind convection on the other unknowns,
conduction scaled to a Peclet number, a random accumulation block and one
well.  They are made on the GPU.
"""
from __future__ import annotations

import math
import time

import numpy as np
import torch

import paper_2308_11892_gb300 as P

DEV = "cuda"


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: a sector model of a few hundred cells, every launch and
        # synchronisation on the critical path
        dict(name="newton_500_fp64", kind="newton", grid="cartesian", nx=10, ny=10, nz=5, pe=1.0,
             precision="fp64", option="cptr"),
        # the ordinary mid-size grid of the configurations, at a balanced Peclet number ...
        dict(name="newton_131k_mixed", kind="newton", grid="cartesian", nx=64, ny=64, nz=32,
             pe=1.0, precision="mixed", option="cptr"),
        # ... and flow-dominated, where the coarse AMG rows grow long
        dict(name="newton_131k_pe100", kind="newton", grid="cartesian", nx=64, ny=64, nz=32,
             pe=100.0, precision="mixed", option="cptr"),
        # unstructured, odd sizes, conduction-dominated, everything in FP64
        dict(name="newton_110k_cloud_fp64", kind="newton", grid="cloud", nx=67, ny=53, nz=31,
             pe=0.5, precision="fp64", option="cptr"),
        # the pressure-only first stage (CPR) on a ragged flow-dominated grid
        dict(name="newton_323k_cpr", kind="newton", grid="cartesian", nx=101, ny=97, nz=33,
             pe=30.0, precision="mixed", option="cpr"),
        # the unstructured field model: one million points
        dict(name="newton_1m_cloud", kind="newton", grid="cloud", nx=200, ny=200, nz=25, pe=10.0,
             precision="mixed", option="cptr"),
        # the largest: four million cells, layered and anisotropic, longer restart
        dict(name="newton_4m_layered", kind="newton", grid="layered", nx=200, ny=200, nz=100,
             pe=1.0, precision="mixed", option="cptr"),
        # solves alone: three right-hand sides on one set-up context (sensitivities)
        dict(name="resolve_492k_mixed", kind="resolve", grid="cartesian", nx=128, ny=96, nz=40,
             pe=3.0, precision="mixed", option="cptr"),
        # one preconditioner application in a caller's own FP64 Krylov loop
        dict(name="precond_941k_fp64", kind="precond", grid="cartesian", nx=150, ny=110, nz=57,
             pe=1.0, precision="fp64", option="cptr"),
        # one operator application in a caller's own Krylov loop
        dict(name="spmv_1m_cloud", kind="spmv", grid="cloud", nx=200, ny=200, nz=25, pe=10.0,
             precision="mixed", option="cptr"),
        # many small systems of uneven size in one launch (ensemble of sector models)
        dict(name="batch_48", kind="batch", systems=48, small=2000, large=30000,
             precision="mixed"),
        # independent requests of uneven size through a server: create, set up, solve, destroy
        dict(name="serve_8", kind="serve", systems=8, small=8000, large=120000,
             precision="mixed"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["newton", "newton", "newton", "resolve", "precond", "spmv", "residual",
                       "batch", "serve"])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    if kind == "batch":
        return dict(kind=kind, systems=rng.randint(3, 64), small=rng.randint(500, 3000),
                    large=rng.randint(8000, 30000), precision=precision)
    if kind == "serve":
        return dict(kind=kind, systems=rng.randint(2, 10), small=rng.randint(4000, 9000),
                    large=rng.randint(20000, 150000), precision=precision)
    most = 260000 if kind == "residual" else 1000000
    cells = _log(rng, 400, most)
    nz = max(2, int((cells / 4.0) ** (1.0 / 3.0) * rng.uniform(0.7, 1.4)))
    nx = max(3, int(math.sqrt(cells / nz) * rng.uniform(0.8, 1.25)))
    ny = max(3, int(cells / (nz * nx)))
    if nx * ny * nz > most:
        ny = max(3, most // (nz * nx))
    grid = rng.choice(["cartesian", "layered", "cloud"])
    option = "cptr"
    if kind in ("newton", "resolve", "precond"):
        option = rng.choice(["cptr", "cptr", "cptr", "cpr", "cptr3", "agg2", "hgs"])
    # flow-dominated systems make dense coarse operators: those stay mid-size
    pe = _log(rng, 1.0, 100.0) if option == "cpr" else _log(rng, 0.01, 100.0)
    if nx * ny * nz > 200000:
        pe = min(pe, 10.0)
    if kind == "precond":  # a caller's own Krylov loop takes the FP64 preconditioner
        precision = "fp64"
    return dict(kind=kind, grid=grid, nx=nx, ny=ny, nz=nz, pe=round(pe, 4), precision=precision,
                option=option)


# ------------------------------------------------------------------ the matrices
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _lattice(nx, ny, nz):
    i = torch.arange(nx * ny * nz, device=DEV)
    return i % nx, (i // nx) % ny, i // (nx * ny)


def _cartesian_links(nx, ny, nz):
    """Per cell its 7-point row in column order: columns, validity, axis of the link."""
    ix, iy, iz = _lattice(nx, ny, nz)
    i = torch.arange(nx * ny * nz, device=DEV)
    cols = torch.stack([i - nx * ny, i - nx, i - 1, i, i + 1, i + nx, i + nx * ny], 1)
    ok = torch.stack([iz > 0, iy > 0, ix > 0, ix >= 0, ix < nx - 1, iy < ny - 1, iz < nz - 1], 1)
    return cols.clamp_(0, nx * ny * nz - 1), ok


def _morton(ix, iy, iz):
    m = torch.zeros_like(ix)
    for b in range(12):
        for a, v in enumerate((ix, iy, iz)):
            m |= ((v >> b) & 1) << (3 * b + a)
    return m


def _cloud_links(nx, ny, nz, g):
    """A jittered lattice, Morton-numbered, every point joined to its k ~ U{6..12} nearest
    (either way): columns sorted per row, validity, distances, positions."""
    n = nx * ny * nz
    ix, iy, iz = _lattice(nx, ny, nz)
    h = torch.tensor([0.05, 0.05, 0.08], device=DEV, dtype=torch.float64)
    lat = torch.stack([ix, iy, iz], 1)
    pos = (lat + 0.5 + 0.5 * _rand(g, n, 3) - 0.25) * h
    k = torch.randint(6, 13, (n,), generator=g, device=DEV)
    offs = [(a, b, c) for c in (-1, 0, 1) for b in (-2, -1, 0, 1, 2) for a in (-2, -1, 0, 1, 2)
            if (a, b, c) != (0, 0, 0)]
    nb, dist = [], []
    for a, b, c in offs:
        ok = ((ix + a >= 0) & (ix + a < nx) & (iy + b >= 0) & (iy + b < ny) & (iz + c >= 0)
              & (iz + c < nz))
        j = torch.where(ok, ix + a + nx * (iy + b + ny * (iz + c)), -1)
        d = (pos - pos[j.clamp(min=0)]).square().sum(1).sqrt()
        nb.append(j)
        dist.append(torch.where(ok, d, math.inf))
    nb, dist = torch.stack(nb, 1), torch.stack(dist, 1)
    near = dist.sort(1)[0].gather(1, (k - 1)[:, None])
    link = (dist <= near) & (nb >= 0)
    # the other end's choice: offset o seen from here is offset -o seen from there
    m = len(offs)
    back = torch.empty_like(link)
    for o in range(m):
        j = nb[:, o]
        back[:, o] = (j >= 0) & link[j.clamp(min=0), m - 1 - o]
    link |= back
    order = torch.argsort(_morton(ix, iy, iz))
    new = torch.empty_like(order)
    new[order] = torch.arange(n, device=DEV)
    nb = torch.where(link, new[nb.clamp(min=0)], n)[order]
    dist = dist[order]
    width = int(link.sum(1).max())
    nb, at = nb.sort(1)
    nb, dist = nb[:, :width], dist.gather(1, at)[:, :width]
    # the diagonal joins the row in column order
    nb = torch.cat([nb, torch.arange(n, device=DEV)[:, None]], 1)
    dist = torch.cat([dist, torch.ones(n, 1, device=DEV, dtype=torch.float64)], 1)
    nb, at = nb.sort(1)
    return nb.clamp(max=n - 1), nb < n, dist.gather(1, at), pos[order]


def system(grid, nx, ny, nz, pe, seed):
    """(n, rowptr, col, vals, rhs) of one seeded Jacobian, as device tensors."""
    g = _gen(seed)
    n = nx * ny * nz
    if grid == "cloud":
        cols, ok, dist, pos = _cloud_links(nx, ny, nz, g)
        geo = 1.0 / dist
        box = (0.05 * nx, 0.05 * ny, 0.08 * nz)
        inj = int((pos - torch.tensor([box[0] / 2, box[1] / 2, 0.0], device=DEV,
                                      dtype=torch.float64)).square().sum(1).argmin())
    else:
        cols, ok = _cartesian_links(nx, ny, nz)
        geo = torch.ones_like(cols, dtype=torch.float64)
        pos = torch.stack(_lattice(nx, ny, nz), 1).double() + 0.5
        box = (nx, ny, nz)
        inj = nx // 2 + nx * (ny // 2)
    if grid == "layered":
        lnk = (math.sqrt(3.0) * _randn(g, nz)).repeat_interleave(nx * ny) + _randn(g, n)
    else:
        lnk = _randn(g, n)
    k = lnk.exp()
    me = torch.arange(n, device=DEV)[:, None]
    off = ok & (cols != me)
    ki, kj = k[:, None], k[cols]
    if grid == "layered":  # ten times less permeable vertically
        vert = (cols - me).abs() == nx * ny
        ki, kj = torch.where(vert, 0.1 * ki, ki), torch.where(vert, 0.1 * kj, kj)
    zero = torch.zeros((), device=DEV, dtype=torch.float64)
    T = torch.where(off, geo * 2.0 * ki * kj / (ki + kj), zero)
    del ki, kj
    tau = 2.0 * math.pi
    phi = (pos[:, 0] + 0.3 * torch.sin(tau * pos[:, 1] / box[1]) * torch.cos(tau * pos[:, 2] / box[2])
           + 0.01 * _randn(g, n))
    F = T * (phi[:, None] - phi[cols])  # flux out of the row's cell
    aF, out = F.abs(), F > 0
    kappa = aF.sum() / (pe * torch.where(off, geo, zero).sum())
    cond = torch.where(off, kappa * geo, zero)
    u = 0.5 + _rand(g, n, 3)
    lam = torch.stack([torch.ones(n, device=DEV, dtype=torch.float64), 0.5 * u[:, 0],
                       0.5 * u[:, 1], 0.2 * u[:, 2]], 1)
    if grid == "layered":  # a 40 K cold plume around the well lowers the mobilities
        r2 = (pos[:, 0] - nx // 2 - 0.5) ** 2 + (pos[:, 1] - ny // 2 - 0.5) ** 2
        lam = lam * torch.exp(-0.8 * torch.exp(-r2 / 25.0))[:, None]
    sumT = T.sum(1)
    D = 0.1 * (2.0 * _rand(g, n, 16) - 1.0)
    D[:, [0, 5, 10, 15]] += 1.0 + _rand(g, n, 4)
    D *= 1e-2 * sumT.mean()
    vals = torch.zeros(*cols.shape, 16, device=DEV, dtype=torch.float64)
    for r in range(4):
        w = torch.where(out, lam[:, r:r + 1], lam[:, r][cols]) * T
        vals[:, :, 4 * r] = -w
        D[:, 4 * r] += w.sum(1)
        if r:
            vals[:, :, 5 * r] -= torch.where(out, zero, aF)
            D[:, 5 * r] += torch.where(out, aF, zero).sum(1)
    vals[:, :, 15] -= cond
    D[:, 15] += cond.sum(1)
    D[inj, [0, 15]] += 10.0 * sumT.max()
    vals = torch.where((cols == me)[:, :, None], D[:, None, :], vals)[ok]
    rowptr = torch.zeros(n + 1, device=DEV, dtype=torch.int32)
    rowptr[1:] = ok.sum(1).cumsum(0)
    rhs = _randn(g, 4 * n)
    rhs[4 * inj] += 100.0
    rhs[4 * inj + 3] -= 100.0
    return n, rowptr, cols[ok].to(torch.int32), vals.contiguous(), rhs


def _sizes(case):
    """Lattices of a batch's or a server's systems: from `small` to `large` cells, evenly in
    their logarithm, Cartesian and cloud in turn, Peclet numbers over the whole range."""
    m = case["systems"]
    for q in range(m):
        f = q / max(1, m - 1)
        cells = case["small"] * (case["large"] / case["small"]) ** f
        nz = max(2, int(round((cells / 4.0) ** (1.0 / 3.0))))
        nx = max(3, int(round(math.sqrt(cells / nz))))
        pe = 0.01 * 10.0 ** (4.0 * ((7 * q) % m) / max(1, m - 1))
        yield ("cartesian", "cloud")[q % 2], nx, nx + q % 3, nz, pe


# ------------------------------------------------------------------ the passes
def _params(case):
    kw = dict(precision=P.FP64 if case["precision"] == "fp64" else P.MIXED)
    opt = case.get("option", "cptr")
    if opt == "cpr":
        kw.update(e1=-1)
    elif opt == "cptr3":
        kw.update(precond=P.PREC_CPTR3)
    elif opt == "agg2":
        kw.update(agg=2)
    elif opt == "hgs":
        kw.update(smoother=P.SMOOTH_HYBRID_GS)
    if case.get("grid") == "layered":
        kw.update(restart=50)
    return kw


def _solver(n, rowptr, col, vals, stream, **kw):
    s = P.Solver(n, rowptr, col, vals, **kw)
    P.cptr_set_stream(s.h, stream.cuda_stream)
    return s


class _Server:
    def __init__(self, **kw):
        self.h = P.cptr_server_create(96 << 30, 4, P.params(**kw))

    def __del__(self):
        P.cptr_server_destroy(self.h)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":  # requests come from host memory
        systems = []
        for q, spec in enumerate(_sizes(case)):
            n, rp, ci, v, b = system(*spec, seed=1000 * seed + q)
            systems.append((n, rp.cpu().numpy(), ci.cpu().numpy(), v.cpu().numpy(),
                            b.cpu().numpy()))
        return dict(kind=kind, systems=systems, server=_Server(**_params(case)))
    stream = torch.cuda.Stream()
    if kind == "batch":
        systems = [system(*spec, seed=1000 * seed + q) for q, spec in enumerate(_sizes(case))]
        torch.cuda.synchronize()
        solvers = [_solver(*s[:4], stream, tri_tune=0, **_params(case)).setup() for s in systems]
        st = dict(kind=kind, stream=stream, solvers=solvers, rhs=[s[4] for s in systems],
                  x=[torch.zeros_like(s[4]) for s in systems])
        torch.cuda.synchronize()
        return st
    n, rp, ci, vals, rhs = system(case["grid"], case["nx"], case["ny"], case["nz"], case["pe"],
                                  seed)
    st = dict(kind=kind, n=n, stream=stream, vals=vals, rhs=rhs, x=torch.zeros_like(rhs))
    torch.cuda.synchronize()
    if kind == "residual":
        g = _gen(seed + 1)
        st.update(rp=rp, ci=ci, x=_randn(g, 4 * n), r=torch.empty_like(rhs),
                  norm=torch.zeros(1, device=DEV, dtype=torch.float64))
    else:
        st["solver"] = _solver(n, rp, ci, vals, stream, **_params(case))
        if kind in ("resolve", "precond"):
            st["solver"].setup()
        if kind == "resolve":
            g = _gen(seed + 1)
            st["rhs"] = [rhs, _randn(g, 4 * n), _randn(g, 4 * n)]
            st["x"] = [torch.zeros_like(rhs) for _ in range(3)]
        elif kind in ("precond", "spmv"):
            st.update(x=rhs, y=torch.empty_like(rhs))
    torch.cuda.synchronize()
    return st


def run(st):
    kind = st["kind"]
    if kind == "serve":
        srv = st["server"].h
        pending = {P.cptr_submit(srv, *s): k for k, s in enumerate(st["systems"])}
        xs = [np.empty(4 * s[0]) for s in st["systems"]]
        while pending:
            for rid, k in list(pending.items()):
                status, _ = P.cptr_poll(srv, rid, xs[k])
                if status in (P.OK, P.ERR_MAXIT):
                    del pending[rid]
                elif status != P._lib.PENDING:
                    raise RuntimeError(P.cptr_server_last_error(srv))
            time.sleep(0.0002)
        return xs
    with torch.cuda.stream(st["stream"]):
        if kind == "newton":
            s = st["solver"]
            st["x"].zero_()
            P.cptr_update_values(s.h, st["vals"])
            P.cptr_setup(s.h)
            P.cptr_solve(s.h, st["rhs"], st["x"])
            return st["x"]
        if kind == "resolve":
            for b, x in zip(st["rhs"], st["x"]):
                x.zero_()
                P.cptr_solve(st["solver"].h, b, x)
            return st["x"]
        if kind == "precond":
            P.cptr_apply(st["solver"].h, P.APPLY_PRECOND, st["x"], st["y"])
            return st["y"]
        if kind == "spmv":
            P.cptr_spmv(st["solver"].h, st["x"], st["y"])
            return st["y"]
        if kind == "residual":
            P.cptr_residual_noalloc(st["n"], st["rp"], st["ci"], st["vals"], st["x"], st["rhs"],
                                    st["r"], st["norm"], st["stream"].cuda_stream)
            return [st["r"], st["norm"]]
        for x in st["x"]:
            x.zero_()
        P.cptr_solve_batch([s.h for s in st["solvers"]], st["rhs"], st["x"])
        return st["x"]


# ------------------------------------------------------------------ floors and references
def _blocks(grid, nx, ny, nz):
    n = nx * ny * nz
    if grid == "cloud":
        return 11.4 * n  # mean row of the symmetrised neighbour graph
    return 7 * n - 2 * (nx * ny + ny * nz + nx * nz)


def work(case):
    """Bytes: the matrix, the right-hand sides and the results once.  Operations: 32 per
    block and product with A; with a setup also the products of the block ILU(0) (128 per
    updated block and per scaled lower block), and per solve the least that an iteration
    does (A, the factors and the first-stage correction) ten times over."""
    kind = case["kind"]
    specs = (list(_sizes(case)) if kind in ("batch", "serve")
             else [(case["grid"], case["nx"], case["ny"], case["nz"], 0.0)])
    nb = fl = 0.0
    for grid, nx, ny, nz, _ in specs:
        b, n = _blocks(grid, nx, ny, nz), nx * ny * nz
        iteration = 80.0 * b
        nb += 132.0 * b + 4 * n
        if kind in ("spmv", "residual"):
            nb += (64.0 if kind == "spmv" else 96.0) * n
            fl += 32.0 * b
        elif kind == "precond":
            nb += 64.0 * n
            fl += iteration
        elif kind == "resolve":
            nb += 3 * 64.0 * n
            fl += 30 * iteration
        else:
            nb += 64.0 * n
            fl += (0.0 if kind == "batch" else 128.0 * b) + 10 * iteration
    return {"bytes": nb, "flops": fl}


def _product(rp, ci, vals, x):
    n = rp.numel() - 1
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), (rp[1:] - rp[:-1]).long())
    prod = torch.bmm(vals.view(-1, 4, 4), x.view(-1, 4)[ci.long()][:, :, None])[:, :, 0]
    return torch.zeros(n, 4, device=DEV, dtype=torch.float64).index_add_(0, rows, prod).view(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("newton", "spmv", "residual"):
        return None
    if kind == "newton" and case["nx"] * case["ny"] * case["nz"] > 2000:
        return None
    n, rp, ci, vals, rhs = system(case["grid"], case["nx"], case["ny"], case["nz"], case["pe"],
                                  seed)
    if kind == "spmv":
        return _product(rp, ci, vals, rhs)
    if kind == "residual":
        r = rhs - _product(rp, ci, vals, _randn(_gen(seed + 1), 4 * n))
        return [r, r.norm()[None]]
    A = torch.zeros(n, n, 4, 4, device=DEV, dtype=torch.float64)
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), (rp[1:] - rp[:-1]).long())
    A[rows, ci.long()] = vals.view(-1, 4, 4)
    return torch.linalg.solve(A.permute(0, 2, 1, 3).reshape(4 * n, 4 * n), rhs)
