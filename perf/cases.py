"""The timed cases of this framework: what its users have it do, through its public entry points.

A user's program keeps a matrix handle and a preconditioner handle for one grid and one set of wells, and on every
Newton step gives it new values: assembly, preconditioner setup, Krylov solve.  The cases are those steps over the
range of grids, block sizes, precisions, Krylov methods and fill levels that the package offers, the adjoint step
with its gradients, and the single calls that a program with a solver of its own makes (products with A and A^T,
the residual, one application of the preconditioner, the gradient chain).

Inputs follow the synthetic generator of the package (lognormal or two-facies permeability, horizontal well pairs, a
dominant pressure column), drawn on the GPU.
"""
import math

import numpy as np
import torch

from paper_1812_03952_gb300 import autograd, synthetic, trs

SLOTS = ((0, 0, -1), (0, -1, 0), (-1, 0, 0), (0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1))
DENSE_MAX = 16_000   # unknowns up to which exact() solves densely


def _case(name, call, nx, ny, nz, b, pairs, **kw):
    c = dict(name=name, call=call, nx=nx, ny=ny, nz=nz, b=b, pairs=pairs, sigma=1.0, facies=False, shale=0.0,
             kvkh=1.0, precision="fp32", ilu=0, krylov="fgmres", restart=30, rtol=1e-6)
    c.update(kw)
    return c


def listed():
    return [
        # The smallest of the benchmark's grids: a box model or a sector of a field, thousands of steps in a row.
        _case("step_16x16x4_b4", "step", 16, 16, 4, 4, 1),
        # An odd, ragged grid of the tests with the package's default (all FP64) preconditioner and a tight tolerance.
        _case("step_33x17x9_b3_fp64", "step", 33, 17, 9, 3, 2, precision="fp64", rtol=1e-8, kvkh=0.5),
        # A sector model, the benchmark's 64x64x32.
        _case("step_64x64x32_b4", "step", 64, 64, 32, 4, 1),
        # The benchmark's headline: one Newton step of the million-cell model, anisotropic and heterogeneous.
        _case("step_128x128x64_b4", "step", 128, 128, 64, 4, 4, sigma=1.5, kvkh=0.1),
        # A large model with five unknowns per cell and channelised sand and shale, its grid not a power of two.
        _case("step_200x150x100_b5", "step", 200, 150, 100, 5, 12, facies=True),
        # A thin many-well grid (the size of the paper's SAGD example) with the paper's Krylov method.
        _case("bicgstab_100x100x6_b5", "step", 100, 100, 6, 5, 25, krylov="bicgstab", rtol=1e-8),
        # A later step of a high-contrast sequence: the aggregates are kept, the F stage is block ILU(1), FGMRES(60).
        _case("refresh_160x96x48_b4_ilu1", "refresh", 160, 96, 48, 4, 6, sigma=2.0, shale=0.1, ilu=1, restart=60),
        # One Newton step of the thermal model itself: Jacobian and residual from the physics, then the solve.
        _case("thermal_96x64x40_b4_ilu1", "thermal", 96, 64, 40, 4, 3, sigma=1.5, kvkh=0.1, ilu=1, restart=60,
              rtol=1e-8),
        # History matching: forward solve and gradients with respect to log-permeability and right-hand side.
        _case("adjoint_64x64x32_b4_fp64", "adjoint", 64, 64, 32, 4, 1, precision="fp64", rtol=1e-10),
        # A program with its own solver: A x, A^T x and the residual.
        _case("products_128x128x64_b4", "products", 128, 128, 64, 4, 4, sigma=1.5, kvkh=0.1),
        # ... and one application of the default preconditioner, and of the pressure V-cycle alone.
        _case("apply_96x96x48_b4_fp64", "apply", 96, 96, 48, 4, 2, precision="fp64", kvkh=0.1),
        # The gradient from a stored adjoint: dL/dA on the pattern and the chain to log-permeability.
        _case("chain_100x80x50_b3", "chain", 100, 80, 50, 3, 4),
    ]


def draw(rng):
    """A case of the same ranges.  Grids from about a thousand cells up, log-uniform, any extents."""
    call = rng.choice(["step", "step", "step", "refresh", "thermal", "adjoint", "products", "apply", "chain"])
    b = 4 if call == "thermal" else rng.choice([4, 4, 5, 3, 2, 1])
    top = {"step": 1.2e6, "refresh": 1.0e6, "thermal": 2.4e5, "adjoint": 1.3e5, "products": 1.5e6, "apply": 8.0e5,
           "chain": 1.0e6}[call]
    cells = math.exp(rng.uniform(math.log(1.0e3), math.log(top)))
    flat = math.exp(rng.uniform(math.log(0.08), math.log(0.8)))     # nz over the lateral extent
    nz = max(3, round((cells * flat * flat) ** (1.0 / 3.0)))
    nx = max(8, round(math.sqrt(cells / nz) * math.exp(rng.uniform(-0.4, 0.4))))
    ny = max(6, round(cells / nz / nx))
    pairs = rng.randint(1, max(1, ny // 8))
    c = _case("", call, nx, ny, nz, b, pairs, sigma=rng.choice([0.5, 1.0, 1.5]),
              kvkh=rng.choice([0.1, 0.3, 0.5, 1.0]), precision=rng.choice(["fp32", "fp32", "fp64"]))
    if call in ("step", "adjoint", "apply"):
        c["ilu"] = rng.choice([0, 0, 1])
    if call == "step":
        c["facies"] = rng.random() < 0.25
        c["krylov"] = rng.choice(["fgmres", "fgmres", "bicgstab"])
        c["rtol"] = 1e-8 if c["krylov"] == "bicgstab" else rng.choice([1e-6, 1e-6, 1e-8])
    elif call == "refresh":
        c.update(sigma=rng.choice([1.0, 1.5, 2.0]), shale=rng.choice([0.0, 0.1]), ilu=1, restart=60)
    elif call == "thermal":
        c.update(sigma=rng.choice([1.0, 1.5]), ilu=1, restart=60, kvkh=0.1, rtol=1e-8)
    elif call == "adjoint":
        c.update(precision="fp64", ilu=0, rtol=rng.choice([1e-8, 1e-10]))
    elif call == "apply":
        c["precision"] = "fp64"
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed, device="cuda"):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    return g


def _wells(c):
    """Horizontal pairs along x, as the package's generator places them: (n_wells, perf_well, perf_cell)."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    ys = [int(round(v)) for v in np.linspace(0, ny - 1, c["pairs"] + 2)[1:-1]]
    gap = min(5, max(1, nz // 4))     # layers between injector and producer
    zi = max(0, (nz - gap) // 2)
    zp = min(nz - 1, zi + gap)
    margin = max(1, nx // 9)
    pw, pc = [], []
    for p, y in enumerate(ys):
        for k, z in enumerate((zi, zp)):
            for x in range(margin, nx - margin):
                pw.append(2 * p + k)
                pc.append(x + nx * (y + ny * z))
    return 2 * len(ys), np.asarray(pw, np.int32), np.asarray(pc, np.int32)


def _perm(c, g):
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    n = nx * ny * nz
    if c["facies"]:
        # channels: noise constant over 8 x 2 cells of a layer, cut so that three tenths are shale
        noise = torch.randn((nz, -(-ny // 2), -(-nx // 8)), generator=g, device="cuda", dtype=torch.float64)
        noise = noise.repeat_interleave(2, 1)[:, :ny].repeat_interleave(8, 2)[:, :, :nx].reshape(-1)
        cut = torch.sort(noise).values[int(0.3 * n)]
        return torch.where(noise <= cut, 50.0, 2000.0).to(torch.float64).contiguous()
    mu = math.log(500.0) - 0.5 * c["sigma"] ** 2
    k = torch.exp(mu + c["sigma"] * torch.randn(n, generator=g, device="cuda", dtype=torch.float64))
    if c["shale"] > 0:
        # impermeable lenses of 16 x 8 cells in a layer
        m = torch.rand((nz, -(-ny // 8), -(-nx // 16)), generator=g, device="cuda") < c["shale"]
        m = m.repeat_interleave(8, 1)[:, :ny].repeat_interleave(16, 2)[:, :, :nx].reshape(-1)
        k = torch.where(m, torch.zeros_like(k), k)
    return k.contiguous()


def _inputs(c, seed):
    """The arrays a synthetic system is assembled from, on the GPU."""
    g = _gen(seed)
    n, b = c["nx"] * c["ny"] * c["nz"], c["b"]
    d = dict(device="cuda", dtype=torch.float64)
    k = _perm(c, g)
    s = synthetic.C_T * float(k.mean())
    M = torch.rand((n, 6, b, b), generator=g, **d).mul_(0.01)
    M[..., 0] = 1.0 + torch.rand((n, 6, b), generator=g, **d)
    acc = torch.rand((n, b, b), generator=g, **d).mul_(0.1).sub_(0.05)
    i = torch.arange(b, device="cuda")
    acc[:, i, i] = 0.5 + torch.rand((n, b), generator=g, **d)
    acc[:, 0, 0] *= 0.05
    acc *= s
    nw, pw, pc = _wells(c)
    wi = torch.full((len(pc),), 10.0 * s, **d)
    lam = 0.5 + torch.rand((len(pc), b), generator=g, **d)
    rhs = torch.randn((n + nw, b), generator=g, **d)
    rhs[n:, 1:] = 0.0
    return dict(n=n, nw=nw, pw=pw, pc=pc, k=k, M=M, acc=acc, wi=wi, lam=lam, rhs=rhs.reshape(-1).contiguous())


def _matrix(c, i):
    A = trs.Matrix.synthetic_pattern(c["nx"], c["ny"], c["nz"], c["b"], i["nw"], i["pw"], i["pc"])
    _assemble(c, i, A)
    return A


def _assemble(c, i, A, acc=None):
    A.assemble(i["k"], i["M"], i["acc"] if acc is None else acc, i["wi"], i["lam"], c["kvkh"], synthetic.C_T)


def _vector(i, b, g):
    """A vector of the system: values in every unknown, zero in the padding of the well blocks."""
    v = torch.randn((i["n"] + i["nw"], b), generator=g, device="cuda", dtype=torch.float64)
    v[i["n"]:, 1:] = 0.0
    return v.reshape(-1).contiguous()


def _system(c, i):
    """The package's SyntheticSystem of these inputs (host arrays), for the calls that take one."""
    h = lambda t: t.cpu().numpy()   # noqa: E731
    return synthetic.SyntheticSystem(
        nx=c["nx"], ny=c["ny"], nz=c["nz"], b=c["b"], k=h(i["k"]), kvkh=c["kvkh"], c_t=synthetic.C_T, M=h(i["M"]),
        acc=h(i["acc"]), n_wells=i["nw"], perf_well=i["pw"], perf_cell=i["pc"], wi=h(i["wi"]), lam=h(i["lam"]),
        rhs=h(i["rhs"]))


def prepare(case, seed):
    c = case
    if c["call"] == "thermal":
        g = _gen(seed)
        k = _perm(c, g).cpu().numpy()
        nw, pw, pc = _wells(c)
        none = np.zeros((0,))
        sysm = synthetic.SyntheticSystem(
            nx=c["nx"], ny=c["ny"], nz=c["nz"], b=4, k=k, kvkh=c["kvkh"], c_t=synthetic.C_T, M=none, acc=none,
            n_wells=nw, perf_well=pw, perf_cell=pc, wi=none, lam=none, rhs=none)
        ts = trs.ThermalSystem(sysm, synthetic.thermal_state(sysm, seed + 1), synthetic.SWT, synthetic.SLT)
        ts.assemble()
        return dict(c=c, ts=ts, M=trs.CPR(ts.A, precision=c["precision"], ilu_fill=c["ilu"]))
    i = _inputs(c, seed)
    g = _gen(seed + 7919)
    if c["call"] == "adjoint":
        sctx = autograd.SolveContext(_system(c, i), precision=c["precision"], rtol=c["rtol"], restart=c["restart"])
        theta = torch.log(i["k"]).requires_grad_(True)
        rhs = i["rhs"].clone().requires_grad_(True)
        grad = torch.zeros((i["n"] + i["nw"], c["b"]), device="cuda", dtype=torch.float64)
        grad[torch.from_numpy(i["pc"]).long().cuda(), 0] = 1.0    # the pressures of the perforated cells
        return dict(c=c, sctx=sctx, theta=theta, rhs=rhs, grad=grad.reshape(-1).contiguous())
    A = _matrix(c, i)
    st = dict(c=c, i=i, A=A)
    if c["call"] in ("step", "refresh", "apply"):
        st["M"] = trs.CPR(A, precision=c["precision"], ilu_fill=c["ilu"])
    if c["call"] == "refresh":
        # the next system of the sequence: the cells' accumulation rescaled by up to a fifth
        f = 0.8 + 0.4 * torch.rand((i["n"], 1, 1), generator=g, device="cuda", dtype=torch.float64)
        st["acc2"] = (i["acc"] * f).contiguous()
    if c["call"] in ("products", "chain"):
        st["x"] = _vector(i, c["b"], g)
        st["v"] = _vector(i, c["b"], g)
        st["r"] = torch.empty_like(st["x"])
    if c["call"] == "apply":
        st["v"] = i["rhs"]
        st["p"] = torch.randn(i["n"] + i["nw"], generator=g, device="cuda", dtype=torch.float64)
    return st


def _solve(c, A, M, rhs):
    x, _ = trs.krylov_solve(c["krylov"], A, M, rhs, rtol=c["rtol"], restart=c["restart"], maxit=300)
    return x


def run(state):
    c = state["c"]
    call = c["call"]
    if call == "thermal":
        ts, M = state["ts"], state["M"]
        R = ts.assemble()
        M.update(ts.A, reuse_amg=False)
        return {"residual": R, "x": _solve(c, ts.A, M, R)}
    if call == "adjoint":
        x = autograd.solve(state["theta"], state["rhs"], state["sctx"])
        dtheta, drhs = torch.autograd.grad(x, (state["theta"], state["rhs"]), state["grad"])
        return {"x": x.detach(), "dtheta": dtheta, "drhs": drhs}
    i, A = state["i"], state["A"]
    if call == "step":
        _assemble(c, i, A)
        state["M"].update(A, reuse_amg=False)
        return {"x": _solve(c, A, state["M"], i["rhs"])}
    if call == "refresh":
        _assemble(c, i, A, state["acc2"])
        state["M"].update(A, reuse_amg=True)
        return {"x": _solve(c, A, state["M"], i["rhs"])}
    if call == "products":
        y = A.spmv(state["x"])
        yt = A.spmv(state["v"], transpose=True)
        norm = trs.residual_norm_noalloc(A, state["x"], i["rhs"], state["r"])
        return {"y": y, "yt": yt, "r": state["r"], "norm": norm}
    if call == "apply":
        return {"z": state["M"].apply(state["v"]), "e": state["M"].vcycle(state["p"])}
    if call == "chain":
        return {"dA": trs.outer_product(A, state["v"], state["x"]),
                "dtheta": trs.chain_theta(A, i["k"], i["M"], state["v"], state["x"], c["kvkh"], synthetic.C_T)}
    raise ValueError(call)


# ------------------------------------------------------------------- work
def _nnzb(c):
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    faces = (nx - 1) * ny * nz + nx * (ny - 1) * nz + nx * ny * (nz - 1)
    nw, pw, _ = _wells(c)
    return nx * ny * nz + 2 * faces + 2 * len(pw) + nw


def work(case):
    """Each input read once, each output written once; a solve has to read its matrix at least once, too, and to
    multiply with it and with a preconditioner of its size a handful of times."""
    c = case
    b, n = c["b"], c["nx"] * c["ny"] * c["nz"]
    nw, pw, _ = _wells(c)
    nv = (n + nw) * b
    mat = _nnzb(c) * b * b
    inputs = n * (6 * b * b + b * b + 1) + len(pw) * (b + 1)
    spmv = 2 * mat
    call = c["call"]
    if call in ("step", "refresh"):
        return {"bytes": 8 * (inputs + mat + 2 * nv), "flops": 10 * 3 * spmv}
    if call == "thermal":
        return {"bytes": 8 * (2 * nv + n + mat + 2 * nv), "flops": 10 * 3 * spmv}
    if call == "adjoint":
        return {"bytes": 8 * (inputs + 2 * mat + 4 * nv + 2 * n), "flops": 2 * 10 * 3 * spmv}
    if call == "products":
        return {"bytes": 8 * (3 * mat + 7 * nv), "flops": 3 * spmv}
    if call == "apply":
        return {"bytes": 8 * (2 * mat + 2 * nv + mat // (b * b) + 2 * (n + nw)), "flops": 3 * spmv}
    return {"bytes": 8 * (mat + 2 * nv + 6 * n * b * b + 2 * n), "flops": spmv}


# ------------------------------------------------------------------ exact
def _faces(c, i):
    """Transmissibility of each directed face, [n, 6] in the order -z, -y, -x, +x, +y, +z, and its neighbour
    (-1: none)."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    n, k = i["n"], i["k"]
    a = torch.arange(n, device="cuda")
    x, y, z = a % nx, (a // nx) % ny, a // (nx * ny)
    T = torch.zeros((n, 6), device="cuda", dtype=torch.float64)
    J = torch.full((n, 6), -1, device="cuda", dtype=torch.long)
    for f, (dx, dy, dz) in enumerate(s for s in SLOTS if s != (0, 0, 0)):
        ok = (x + dx >= 0) & (x + dx < nx) & (y + dy >= 0) & (y + dy < ny) & (z + dz >= 0) & (z + dz < nz)
        j = torch.where(ok, a + dx + nx * (dy + ny * dz), a)
        h = c["kvkh"] if dz else 1.0
        ki, kj = k * h, k[j] * h
        s = ki + kj
        t = torch.where(s > 0, synthetic.C_T * 2.0 * ki * kj / torch.where(s > 0, s, torch.ones_like(s)),
                        torch.zeros_like(s))
        T[:, f] = torch.where(ok, t, torch.zeros_like(t))
        J[:, f] = torch.where(ok, j, torch.full_like(j, -1))
    return T, J


def _blocks(c, i, acc=None):
    """A as block triplets (row, column, b x b values) in 64 bits."""
    b, n, nw = c["b"], i["n"], i["nw"]
    T, J = _faces(c, i)
    TM = T[:, :, None, None] * i["M"]
    diag = (i["acc"] if acc is None else acc) + TM.sum(1)
    pw, pc = torch.from_numpy(i["pw"]).long().cuda(), torch.from_numpy(i["pc"]).long().cuda()
    q = i["wi"][:, None] * i["lam"]
    col = torch.zeros((len(pc), b, b), device="cuda", dtype=torch.float64)
    col[:, :, 0] = q
    diag = diag.index_add(0, pc, col)
    rows, cols, vals = [torch.arange(n, device="cuda")], [torch.arange(n, device="cuda")], [diag]
    for f in range(6):
        at = (J[:, f] >= 0).nonzero().flatten()
        rows.append(at)
        cols.append(J[at, f])
        vals.append(-TM[at, f])
    lam = i["lam"].sum(1) * i["wi"]
    one = torch.zeros((len(pc), b, b), device="cuda", dtype=torch.float64)
    one[:, 0, 0] = -lam
    wd = torch.eye(b, device="cuda", dtype=torch.float64).repeat(nw, 1, 1)
    wd[:, 0, 0] = torch.zeros(nw, device="cuda", dtype=torch.float64).index_add(0, pw, lam)
    rows += [pc, n + pw, n + torch.arange(nw, device="cuda")]
    cols += [n + pw, pc, n + torch.arange(nw, device="cuda")]
    vals += [-col, one, wd]
    return torch.cat(rows), torch.cat(cols), torch.cat(vals)


def _product(B, x, b, transpose=False):
    r, q, v = B
    if transpose:
        r, q, v = q, r, v.transpose(1, 2)
    return torch.zeros_like(x).view(-1, b).index_add(0, r, (v @ x.view(-1, b)[q][:, :, None])[:, :, 0]).reshape(-1)


def _dense(B, nv, b):
    r, q, v = B
    A = torch.zeros((nv, nv), device="cuda", dtype=torch.float64)
    e = torch.arange(b, device="cuda")
    A.index_put_(((r[:, None, None] * b + e[None, :, None]).expand_as(v), (q[:, None, None] * b + e).expand_as(v)), v,
                 accumulate=True)
    return A


def _chain(c, i, lam, x):
    """dL/dln k from dL/dA = -lambda x^T through the harmonic transmissibilities."""
    b, n, k = c["b"], i["n"], i["k"]
    T, J = _faces(c, i)
    X, L = x.view(-1, b), lam.view(-1, b)
    out = torch.zeros(n, device="cuda", dtype=torch.float64)
    for f in range(6):
        at = (J[:, f] >= 0).nonzero().flatten()
        j = J[at, f]
        d = X[j] - X[at]
        dT = (L[at] * (i["M"][at, f] @ d[:, :, None])[:, :, 0]).sum(1) \
            - (L[j] * (i["M"][j, 5 - f] @ d[:, :, None])[:, :, 0]).sum(1)
        s = k[at] + k[j]
        ok = s > 0
        out[at] += torch.where(ok, dT * T[at, f] * k[j] / torch.where(ok, s, torch.ones_like(s)), torch.zeros_like(s))
    return out


def exact(case, seed):
    c = case
    b = c["b"]
    if c["call"] in ("thermal", "apply"):
        return None     # properties and a preconditioner of the package's own: no plain 64-bit counterpart
    i = _inputs(c, seed)
    nv = (i["n"] + i["nw"]) * b
    g = _gen(seed + 7919)
    if c["call"] in ("step", "refresh", "adjoint"):
        if nv > DENSE_MAX:
            return None
        acc = None
        if c["call"] == "refresh":
            acc = i["acc"] * (0.8 + 0.4 * torch.rand((i["n"], 1, 1), generator=g, device="cuda", dtype=torch.float64))
        A = _dense(_blocks(c, i, acc), nv, b)
        x = torch.linalg.solve(A, i["rhs"])
        if c["call"] != "adjoint":
            return {"x": x}
        grad = torch.zeros((i["n"] + i["nw"], b), device="cuda", dtype=torch.float64)
        grad[torch.from_numpy(i["pc"]).long().cuda(), 0] = 1.0
        lam = torch.linalg.solve(A.T, grad.reshape(-1))
        return {"x": x, "dtheta": _chain(c, i, lam, x), "drhs": lam}
    x, v = _vector(i, b, g), _vector(i, b, g)
    if c["call"] == "products":
        B = _blocks(c, i)
        y = _product(B, x, b)
        r = i["rhs"] - y
        return {"y": y, "yt": _product(B, v, b, transpose=True), "r": r, "norm": torch.linalg.norm(r)}
    r, q, _ = _blocks(c, i)
    order = torch.argsort(r * (i["n"] + i["nw"]) + q)
    r, q = r[order], q[order]
    return {"dA": -(v.view(-1, b)[r][:, :, None] * x.view(-1, b)[q][:, None, :]).reshape(-1),
            "dtheta": _chain(c, i, v, x)}
