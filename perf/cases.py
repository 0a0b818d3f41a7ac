"""The work this library is used for, at sizes from one small system to a batch of hundreds.

Every case goes through the public Python API (`Hierarchy`, `Hierarchy.batched`, `autograd.solve`), which only
passes pointers to the C ABI. The matrix families, their coefficients and the solver options are those of
`workloads`, the benchmark and the tests; the matrices are assembled here with torch on the GPU, since the numpy
assembly of the large ones takes seconds. A seed draws the coefficients of the operator around those of its family
and the right-hand side.

`mode` says what a pass is:
  solve    a new system: set-up and solve, hierarchy released (device-resident inputs)
  host     the same with matrix, right-hand side and solution in pinned host memory
  adjoint  a differentiable solve: forward, adjoint solve, gradients with respect to b and A's nonzeros
  batch    many independent systems of drawn sizes: one set-up and solve of the whole batch
  step     time stepping: new values on the pattern of a kept hierarchy, then a solve
  rhs      a kept hierarchy and a new right-hand side
  apply    one V-cycle as the preconditioner of a caller's own iteration
"""
import math
import random

import numpy as np
import torch

from paper_1708_06065_gb300 import autograd, lair

DEV = "cuda"
# options of the benchmark workloads; "default" is what a user who sets nothing gets
OPTIONS = {
    "default": {},
    "classical": dict(distance=1, cf_mode=lair.CF_RS),
    "pmis": dict(distance=1, cf_mode=lair.CF_PMIS, interp=lair.P_ONEPOINT, lump_tol=0.05),
    "dg": dict(distance=2, interp=lair.P_ONEPOINT, strength_abs=1, block_size=6, cf_mode=lair.CF_PMIS),
}


def _case(name, mode, family, size, options, precision, outer, tol, **more):
    return dict(name=name, mode=mode, family=family, size=size, options=options, precision=precision, outer=outer,
                tol=tol, **more)


def listed():
    return [
        # the smallest system in earnest use: 4,096 unknowns, the exact classical first pass; latency throughout
        _case("fd2d_64", "solve", "fd2d", 64, "classical", "fp64", "stationary", 1e-10),
        # what a user gets without setting any option, at an odd size: blocked first pass, lAIP, FP64, FGMRES
        _case("fd2d_151_default", "solve", "fd2d", 151, "default", "fp64", "fgmres", 1e-8),
        # training through a solve: forward, adjoint, gradients
        _case("adjoint_fd2d_512", "adjoint", "fd2d", 512, "pmis", "mixed", "fgmres", 1e-8),
        # the DG transport system of the benchmark: block scaling, distance 2
        _case("dg_p2_256", "solve", "dg", 256, "dg", "mixed", "fgmres", 1e-8),
        # the largest single system: 7.1 million unknowns
        _case("fd3d_192", "solve", "fd3d", 192, "pmis", "mixed", "stationary", 1e-8),
        # a ragged 3D grid in plain FP64
        _case("fd3d_101_fp64", "solve", "fd3d", 101, "pmis", "fp64", "fgmres", 1e-8),
        # a 3D system that lives on the host
        _case("fd3d_96_host", "host", "fd3d", 96, "pmis", "mixed", "stationary", 1e-8),
        # hundreds of independent systems of mixed sizes and stiffness
        _case("batch_512", "batch", "fd2d", 512, "pmis", "mixed", "fgmres", 1e-8),
        # a small batch in FP64
        _case("batch_24_fp64", "batch", "fd2d", 24, "pmis", "fp64", "fgmres", 1e-8),
        # backward Euler time stepping with reuse of the hierarchy's structure
        _case("dg_p2_129_step", "step", "dg", 129, "dg", "mixed", "fgmres", 1e-8),
        # a new right-hand side on a kept hierarchy (default options)
        _case("fd2d_301_rhs", "rhs", "fd2d", 301, "default", "fp64", "fgmres", 1e-8),
        # the preconditioner alone
        _case("fd3d_128_apply", "apply", "fd3d", 128, "pmis", "mixed", "stationary", 1e-8),
    ]


def _between(rng, lo, hi):
    """An integer between lo and hi, spread over the logarithm; odd ones among them."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    mode = rng.choice(["solve", "solve", "solve", "host", "adjoint", "batch", "step", "rhs", "apply"])
    precision = rng.choice(["fp64", "mixed", "mixed"])
    if mode == "batch":
        return dict(mode=mode, family="fd2d", size=_between(rng, 8, 384), options="pmis", precision=precision,
                    outer="fgmres", tol=1e-8)
    family = "fd2d" if mode == "adjoint" else rng.choice(["fd2d", "fd2d", "fd3d", "dg"])
    if family == "dg":
        size, options, outer = _between(rng, 16, 256), "dg", "fgmres"
    elif family == "fd3d":
        size, options, outer = _between(rng, 16, 176), "pmis", rng.choice(["stationary", "fgmres"])
    else:
        options = "pmis" if mode == "adjoint" else rng.choice(["classical", "default", "pmis"])
        size = _between(rng, 32, 96 if options == "classical" else 512)
        outer = "stationary" if options == "classical" else "fgmres"
    return dict(mode=mode, family=family, size=size, options=options, precision=precision, outer=outer, tol=1e-8)


# ------------------------------------------------------------------------------------------------------------------
# matrices
# ------------------------------------------------------------------------------------------------------------------
def _fd(N, velocity, eps, c):
    """Upwind finite differences on (0,1)^dim, N interior points a side, x fastest (as workloads.fd_adr)."""
    dim, h = len(velocity), 1.0 / (N + 1)
    n, d = N ** dim, eps * (N + 1) ** 2
    i = torch.arange(n, device=DEV)
    sides = []
    for a, v in enumerate(velocity):
        at = (i // N ** a) % N
        sides.append((-N ** a, at > 0, -d - (v / h if v > 0 else 0.0)))
        sides.append((N ** a, at < N - 1, -d - (-v / h if v < 0 else 0.0)))
    diag = 2 * dim * d + sum(abs(v) for v in velocity) / h + c
    sides.append((0, torch.ones(n, dtype=torch.bool, device=DEV), diag))
    sides.sort(key=lambda s: s[0])
    keep = torch.stack([s[1] for s in sides], 1)
    col = (i[:, None] + torch.tensor([s[0] for s in sides], device=DEV)[None, :])[keep].to(torch.int32)
    val = torch.tensor([s[2] for s in sides], dtype=torch.float64, device=DEV)[None, :].expand(n, -1)[keep]
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(keep.sum(1), 0, out=rp[1:])
    return rp, col, val.contiguous()


def _p2(x, y):
    """Nodal P2 basis (vertices, then edge midpoints) and its reference gradients at points x, y."""
    l = [1.0 - x - y, x, y]
    g = ((-1.0, -1.0), (1.0, 0.0), (0.0, 1.0))
    edges = ((0, 1), (1, 2), (2, 0))
    phi = [l[k] * (2 * l[k] - 1) for k in range(3)] + [4 * l[p] * l[q] for p, q in edges]
    dphi = [torch.stack([(4 * l[k] - 1) * g[k][a] for a in (0, 1)]) for k in range(3)]
    dphi += [torch.stack([4 * (l[p] * g[q][a] + l[q] * g[p][a]) for a in (0, 1)]) for p, q in edges]
    return torch.stack(phi), torch.stack(dphi)


def _flow(x, y):
    return -torch.sin(math.pi * x) * torch.cos(math.pi * y), torch.cos(math.pi * x) * torch.sin(math.pi * y)


def _gauss(points):
    g, w = np.polynomial.legendre.leggauss(points)
    t = lambda v: torch.tensor(v, dtype=torch.float64, device=DEV)  # noqa: E731
    return t(0.5 * (g + 1.0)), t(0.5 * w)


def _inv2(J):
    (a, b), (c, d) = J.tolist()
    return torch.tensor([[d, -b], [-c, a]], dtype=torch.float64, device=DEV) / (a * d - b * c)


def _dg(M, dt):
    """Mass + dt * upwind advection, nodal P2 DG on M x M squares cut in two (as workloads.dg_p2_advection)."""
    h, sq = 1.0 / M, torch.arange(M * M, device=DEV)
    sx, sy = sq % M, sq // M
    g, w = _gauss(5)
    u, v = torch.meshgrid(g, g, indexing="ij")
    qx, qy, qw = u.reshape(-1), (v * (1 - u)).reshape(-1), (w[:, None] * w[None, :] * (1 - u)).reshape(-1)
    phi, dphi = _p2(qx, qy)
    corners = (((0, 0), (1, 0), (1, 1)), ((0, 0), (1, 1), (0, 1)))
    # neighbour across each local edge: (square offset, the other kind of triangle)
    across = (((0, -1), (1, 0), (0, 0)), ((0, 0), (0, 1), (-1, 0)))
    ref = ((0.0, 0.0), (1.0, 0.0), (0.0, 1.0))
    blocks = torch.zeros(M * M, 2, 4, 6, 6, dtype=torch.float64, device=DEV)
    other = torch.full((M * M, 2, 4), 2 ** 40, device=DEV)
    origin = torch.stack([sx, sy], 1).double() * h
    jac = [torch.tensor([[c[1][a] - c[0][a], c[2][a] - c[0][a]] for a in (0, 1)], dtype=torch.float64, device=DEV) * h
           for c in corners]
    for lu in (0, 1):
        c, J = corners[lu], jac[lu]
        Ji, area = _inv2(J), h * h
        first = origin + torch.tensor(c[0], dtype=torch.float64, device=DEV) * h
        X = first[:, None, :] + (J @ torch.stack([qx, qy])).T[None]
        bx, by = _flow(X[..., 0], X[..., 1])
        gp = torch.einsum("ba,kbq->kaq", Ji, dphi)
        adv = torch.einsum("iq,jq,eq->eij", phi * qw * area, gp[:, 0], bx)
        adv += torch.einsum("iq,jq,eq->eij", phi * qw * area, gp[:, 1], by)
        own = torch.einsum("iq,jq->ij", phi * qw * area, phi)[None] + dt * adv
        other[:, lu, 0] = 2 * sq + lu
        for e, (p, q) in enumerate(((0, 1), (1, 2), (2, 0))):
            t0, t1 = (torch.tensor(c[k], dtype=torch.float64, device=DEV) * h for k in (p, q))
            length = float((t1 - t0).norm())
            nx, ny = float(t1[1] - t0[1]) / length, -float(t1[0] - t0[0]) / length
            Xe = (origin + t0)[:, None, :] + (t1 - t0)[None, None, :] * g[None, :, None]
            ex, ey = _flow(Xe[..., 0], Xe[..., 1])
            flux = ex * nx + ey * ny
            into = flux.clamp(max=0.0) * w * length
            rx = ref[p][0] * (1 - g) + ref[q][0] * g
            ry = ref[p][1] * (1 - g) + ref[q][1] * g
            pe, _ = _p2(rx, ry)
            own -= dt * torch.einsum("ig,jg,eg->eij", pe, pe, into)
            (dx, dy), k = across[lu][e], 1 - lu
            there = (sx + dx >= 0) & (sx + dx < M) & (sy + dy >= 0) & (sy + dy < M) & (flux < 0).any(1)
            # the edge's points in the neighbour's reference triangle (the mesh is a translate of one square)
            shift = torch.tensor([dx, dy], dtype=torch.float64, device=DEV) * h
            at = t0 + (t1 - t0) * g[:, None] - shift - torch.tensor(corners[k][0], dtype=torch.float64, device=DEV) * h
            rn = at @ _inv2(jac[k]).T
            pn, _ = _p2(rn[:, 0], rn[:, 1])
            blocks[:, lu, e + 1] = dt * torch.einsum("ig,jg,eg->eij", pe, pn, into)
            other[:, lu, e + 1] = torch.where(there, 2 * ((sy + dy) * M + sx + dx) + k, 2 ** 40)
        blocks[:, lu, 0] = own
    other, order = other.reshape(-1, 4).sort(1)
    blocks = blocks.reshape(-1, 4, 6, 6).gather(1, order[:, :, None, None].expand(-1, -1, 6, 6))
    keep = (other < 2 ** 40)[:, None, :, None].expand(-1, 6, -1, 6)
    col = (6 * other[:, :, None] + torch.arange(6, device=DEV))[:, None].expand(-1, 6, -1, -1)[keep].to(torch.int32)
    val = blocks.transpose(1, 2)[keep]
    rp = torch.zeros(12 * M * M + 1, dtype=torch.int64, device=DEV)
    torch.cumsum((6 * (other < 2 ** 40).sum(1)).repeat_interleave(6), 0, out=rp[1:])
    return rp, col, val.contiguous()


def _coefficients(family, size, rng):
    """Operator coefficients around those of the family's benchmark system."""
    if family == "fd2d":
        a = 3 * math.pi / 16 + rng.uniform(-0.1, 0.1)
        return (math.cos(a), math.sin(a)), 1e-4 * 2.0 ** rng.uniform(-0.5, 0.5), 0.1 * rng.uniform(0.8, 1.25)
    if family == "fd3d":
        v = [x * rng.uniform(0.95, 1.05) for x in (1.0, 0.7, 0.4)]
        s = math.sqrt(sum(x * x for x in v))
        return tuple(x / s for x in v), 1e-5 * 2.0 ** rng.uniform(-0.5, 0.5), 0.05 * rng.uniform(0.8, 1.25)
    return (rng.uniform(0.8, 1.25) / size,)


def _matrix(family, size, rng):
    c = _coefficients(family, size, rng)
    return _dg(size, *c) if family == "dg" else _fd(size, *c)


def _sides(count):
    """The grid sides of a batch, 32 to 256 as in workloads.batched_fd: part of the case."""
    return [int(s) for s in np.random.default_rng(count).integers(32, 257, count)]


def _batch_draws(case, seed):
    """(side, velocity, eps, c) of each system, the coefficients drawn as in workloads.batched_fd."""
    rng, out = np.random.default_rng(seed), []
    for side in _sides(case["size"]):
        angle = float(rng.uniform(0.0, 2 * math.pi))
        out.append((side, (math.cos(angle), math.sin(angle)), float(10.0 ** rng.uniform(-6.0, 0.0)),
                    float(rng.uniform(0.0, 1.0))))
    return out


def _batch(case, seed):
    rps, cols, vals, offs, nnz = [torch.zeros(1, dtype=torch.int64, device=DEV)], [], [], [0], 0
    for side, v, eps, c in _batch_draws(case, seed):
        rp, col, val = _fd(side, v, eps, c)
        rps.append(rp[1:] + nnz)
        cols.append(col + offs[-1])
        vals.append(val)
        offs.append(offs[-1] + side * side)
        nnz += len(col)
    return torch.cat(rps), torch.cat(cols), torch.cat(vals), np.array(offs, np.int64)


def _uniform(n, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return 2 * torch.rand(n, dtype=torch.float64, device=DEV, generator=g) - 1


def _inputs(case, seed):
    """Matrix and right-hand side of a case, on the device; batches also give their offsets."""
    rng, offs = random.Random(seed), None
    if case["mode"] == "batch":
        rp, col, val, offs = _batch(case, seed)
    else:
        rp, col, val = _matrix(case["family"], case["size"], rng)
    return rp, col, val, _uniform(len(rp) - 1, seed), offs, rng


# ------------------------------------------------------------------------------------------------------------------
# passes
# ------------------------------------------------------------------------------------------------------------------
def prepare(case, seed):
    rp, col, val, b, offs, rng = _inputs(case, seed)
    opts = dict(OPTIONS[case["options"]], precision=lair.MIXED if case["precision"] == "mixed" else lair.FP64)
    s = dict(case=case, opts=opts, rp=rp, col=col, val=val, b=b, offs=offs,
             how=dict(tol=case["tol"], cycle=lair.FGMRES if case["outer"] == "fgmres" else lair.STATIONARY,
                      max_iter=500))
    mode = case["mode"]
    if mode == "host":
        for k in ("rp", "col", "val", "b"):
            s[k] = s[k].cpu().pin_memory()
        s["x"] = torch.zeros(len(b), dtype=torch.float64).pin_memory()
    elif mode == "adjoint":
        s["target"] = _uniform(len(b), seed + 1)
        s["val"].requires_grad_(True)
        s["b"].requires_grad_(True)
    elif mode in ("step", "rhs", "apply"):
        s["h"] = lair.Hierarchy(rp, col, val, **opts)
        if mode == "step":
            s["val"] = _matrix(case["family"], case["size"], rng)[2]  # the next step's values, same pattern
    return s


def run(s):
    mode, how = s["case"]["mode"], s["how"]
    if mode == "solve":
        h = lair.Hierarchy(s["rp"], s["col"], s["val"], **s["opts"])
        x, _ = h.solve(s["b"], raise_on_nc=True, **how)
        h.close()
        return x
    if mode == "host":
        s["x"].zero_()
        h = lair.Hierarchy(s["rp"], s["col"], s["val"], **s["opts"])
        x, _ = h.solve(s["b"], s["x"], raise_on_nc=True, **how)
        h.close()
        return x
    if mode == "adjoint":
        x = autograd.solve(s["rp"], s["col"], s["val"], s["b"], tol=how["tol"], max_iter=how["max_iter"], **s["opts"])
        loss = 0.5 * (x - s["target"]).square().sum()
        dval, db = torch.autograd.grad(loss, (s["val"], s["b"]))
        return {"x": x.detach(), "db": db, "dval": dval}
    if mode == "batch":
        h = lair.Hierarchy.batched(s["rp"], s["col"], s["val"], s["offs"], **s["opts"])
        x, _, _, _ = h.solve_batched(s["b"], raise_on_nc=True, **dict(how, max_iter=2000))
        h.close()
        return x
    if mode == "step":
        s["h"].refresh(s["val"])
        return s["h"].solve(s["b"], raise_on_nc=True, **how)[0]
    if mode == "rhs":
        return s["h"].solve(s["b"], raise_on_nc=True, **how)[0]
    return s["h"].precond(s["b"])


# ------------------------------------------------------------------------------------------------------------------
# what a pass cannot do without, and its result in 64 bits
# ------------------------------------------------------------------------------------------------------------------
def _sizes(case):
    """Unknowns and stored entries."""
    N = case["size"]
    if case["mode"] == "batch":
        return sum(k * k for k in _sides(N)), sum(5 * k * k - 4 * k for k in _sides(N))
    if case["family"] == "fd2d":
        return N * N, 5 * N * N - 4 * N
    if case["family"] == "fd3d":
        return N ** 3, 7 * N ** 3 - 6 * N * N
    return 12 * N * N, 36 * 2 * N * N * 2.5  # an element and on average one and a half inflow neighbours


def work(case):
    n, nnz = _sizes(case)
    vectors = 4 if case["mode"] == "adjoint" else 2  # right-hand side and solution; the gradient too
    matrix = 8 * nnz if case["mode"] == "step" else 12 * nnz + 8 * n  # a step brings values only
    if case["mode"] in ("rhs", "apply"):
        matrix = nnz * (8 if case["precision"] == "mixed" else 12)  # the kept operator is read once in its own form
    if case["mode"] == "adjoint":
        matrix += 8 * nnz  # the gradient of every entry
    return {"bytes": float(matrix + 8 * n * vectors), "flops": float(2 * nnz)}


def _jacobi(rp, col, val, b, block=1):
    """A x = b by (block) Jacobi iteration in 64 bits until the update is at rounding level; None if it does not get there."""
    n = len(b)
    A = torch.sparse_csr_tensor(rp, col.long(), val, (n, n), dtype=torch.float64, device=DEV)
    row = torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1])
    own = (row // block) == (col.long() // block)
    D = torch.zeros(n // block, block, block, dtype=torch.float64, device=DEV)
    D[row[own] // block, row[own] % block, col.long()[own] % block] = val[own]
    D = torch.linalg.inv(D) if block > 1 else 1.0 / D
    x = torch.zeros_like(b)
    for k in range(6000):
        e = torch.einsum("nij,nj->ni", D, (b - A @ x).reshape(-1, block)).reshape(-1)
        x += e
        if k % 50 == 49 and float(e.norm()) <= 1e-13 * float(x.norm()):
            return x
    return None


def _lines(side, velocity, eps, c, b):
    """One 2D system by block elimination over its grid lines, dense 64-bit blocks."""
    h, d = 1.0 / (side + 1), eps * (side + 1) ** 2
    vx, vy = velocity
    lx, ly = (-d - max(v, 0.0) / h for v in velocity)
    hx, hy = (-d - max(-v, 0.0) / h for v in velocity)
    one = lambda k, v: torch.diag(torch.full((side - abs(k),), v, dtype=torch.float64, device=DEV), k)  # noqa: E731
    T = one(0, 4 * d + (abs(vx) + abs(vy)) / h + c) + one(-1, lx) + one(1, hx)
    rhs, S, y = b.reshape(side, side), [], []
    for k in range(side):
        Tk = T if not k else T - ly * hy * S[-1]
        S.append(torch.linalg.inv(Tk))
        y.append(S[-1] @ (rhs[k] if not k else rhs[k] - ly * y[-1]))
    for k in range(side - 2, -1, -1):
        y[k] = y[k] - hy * (S[k] @ y[k + 1])
    return torch.stack(y).reshape(-1)


def _transposed(rp, col, val):
    n = len(rp) - 1
    row = torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1])
    order = torch.argsort(col.long() * n + row)
    trp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(col.long(), minlength=n), 0, out=trp[1:])
    return trp, row[order].to(torch.int32), val[order], row


def exact(case, seed):
    if case["mode"] == "apply":
        return None  # the cycle is this library's own operator: no value without its hierarchy
    rp, col, val, b, offs, rng = _inputs(case, seed)
    if case["mode"] == "batch":
        if case["size"] > 48:
            return None  # the line elimination of hundreds of systems takes minutes
        return torch.cat([_lines(*q, b[offs[k]:offs[k + 1]]) for k, q in enumerate(_batch_draws(case, seed))])
    if case["mode"] == "step":
        val = _matrix(case["family"], case["size"], rng)[2]
    block = 6 if case["family"] == "dg" else 1
    x = _jacobi(rp, col, val, b, block)
    if x is None or case["mode"] != "adjoint":
        return x
    trp, tcol, tval, row = _transposed(rp, col, val)
    lam = _jacobi(trp, tcol, tval, x - _uniform(len(b), seed + 1), block)
    return None if lam is None else {"x": x, "db": lam, "dval": -lam[row] * x[col.long()]}
