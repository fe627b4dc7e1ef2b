"""The work that is timed: what a program that steps the SEIRD model has this library do, each through an entry
point of ``paper_2208_01839_gb300.seird``.

Sizes and options are those of this repository's own workloads: the 33x33 square of the paper's Section 4.1, the
256x256 ensemble and adjoint, the 1024x1024 urban square (FP64 against mixed precision) and the 2.0M-node
Southern-Ontario-like mesh with 512 subdomains, plus sizes between them.  Densities, infection seeds and right-hand
sides are drawn from the seed; the mesh belongs to the size.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2208_01839_gb300 import inputs as I

OPTIONS_OF_A_LONG_RUN = dict(newton_rtol=1e-8, gmres_forcing=1, pc_lag=20, predictor=5)


def listed():
    return [
        # the smallest call: one residual of the paper's square, as a caller's own nonlinear solver asks for it
        dict(name="residual_33", kind="residual", mesh="square", nx=33, ny=33, rule=0, field=False),
        # the residual of a run-sized mesh with a per-node transmission field
        dict(name="residual_1m", kind="residual", mesh="square", nx=1024, ny=1024, rule=0, field=True),
        # the Jacobian assembled at a new state and applied once, irregular mesh
        dict(name="jacobian_200k", kind="jacobian", mesh="polygon", nodes=200000, rule=0, field=False, precision=0),
        # block SpMV on a caller's own matrix (no context): 5x5 blocks, ragged rows
        dict(name="spmv_300k", kind="spmv", rows=300007, f32=False),
        # what a new Jacobian costs before the first Krylov iteration: subdomain factors with fill, coarse inverse
        dict(name="precond_setup_500k", kind="precond_setup", mesh="square", nx=707, ny=709, sub=128, overlap=2,
             coarse=2, fill=1, precision=0),
        # one application of the two-grid preconditioner, the inner loop of every solve, at the 2.0M-node workload
        dict(name="precond_2m", kind="precond", mesh="polygon", nodes=2000000, sub=512, overlap=2, coarse=2, fill=1,
             precision=0),
        # the same with the mixed path's FP32 factors and basis on the 1024x1024 square
        dict(name="precond_1m_mixed", kind="precond", mesh="square", nx=1024, ny=1024, sub=512, overlap=2, coarse=2,
             fill=1, precision=1),
        # one whole step of the paper's Section 4.1 problem: hundreds of tiny launches, GMRES cycles as CUDA graphs
        dict(name="step_33", kind="step_square", side=33),
        # two steps of the 2.0M-node workload in FP64, one preconditioner for both
        dict(name="run_2m", kind="run", mesh="polygon", nodes=2000000, sub=512, overlap=2, coarse=2, fill=1,
             precision=0, steps=2, tune=True),
        # two mixed-precision steps on the 1024x1024 square with more fill, default launch shapes
        dict(name="run_1m_mixed", kind="run", mesh="square", nx=1024, ny=1024, sub=512, overlap=2, coarse=2, fill=2,
             precision=1, steps=2, tune=False),
        # one step of an ensemble of rate samples in one context
        dict(name="ensemble_16x256", kind="ensemble", nx=256, ny=256, samples=16, sub=16),
        # misfit and gradient of a short run: forward steps, recomputation, transposed solves
        dict(name="adjoint_256", kind="adjoint", nx=256, ny=256, sub=16, steps=4, every=2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any kind, sizes spread over the logarithm of the range, odd sides, every option in use."""
    kind = rng.choice(["residual", "jacobian", "spmv", "precond_setup", "precond", "precond", "step_square", "run",
                       "run", "ensemble", "adjoint"])
    if kind == "spmv":
        return dict(kind=kind, rows=_log(rng, 1000, 900000), f32=rng.random() < 0.4)
    if kind == "step_square":
        return dict(kind=kind, side=rng.choice([17, 21, 25, 27, 29, 31]))
    if kind == "ensemble":
        side = _log(rng, 48, 192)
        return dict(kind=kind, nx=side, ny=side + rng.randrange(1, 6), samples=rng.randrange(2, 17),
                    sub=max(2, side * side // 4000))
    if kind == "adjoint":
        side = _log(rng, 64, 200)
        return dict(kind=kind, nx=side, ny=side + rng.randrange(1, 6), sub=max(2, side * side // 4000),
                    steps=rng.randrange(2, 5), every=rng.randrange(1, 3))
    nodes = _log(rng, 2000, 800000)
    if rng.random() < 0.3:
        mesh = dict(mesh="polygon", nodes=nodes)
    else:
        nx = max(8, int(math.sqrt(nodes) * rng.uniform(0.7, 1.4)))
        mesh = dict(mesh="square", nx=nx, ny=max(8, nodes // nx))
    if kind == "residual":
        return dict(kind=kind, rule=rng.randrange(2), field=rng.random() < 0.5, **mesh)
    if kind == "jacobian":
        return dict(kind=kind, rule=rng.randrange(2), field=rng.random() < 0.5, precision=int(rng.random() < 0.3),
                    **mesh)
    ras = dict(sub=max(2, nodes // rng.randrange(1500, 6000)), overlap=rng.randrange(1, 4), fill=rng.randrange(0, 4),
               precision=int(rng.random() < 0.4), coarse=rng.choice([1, 2, 2, 3]), **mesh)
    if kind == "run":
        return dict(kind=kind, steps=rng.randrange(1, 5), tune=rng.random() < 0.5, **ras)
    return dict(kind=kind, **ras)


# ---- inputs ----------------------------------------------------------------------


@functools.lru_cache(maxsize=3)
def _polygon_mesh(nodes):
    return I.irregular_mesh(0, nodes)[:2]


@functools.lru_cache(maxsize=3)
def _square_mesh(nx, ny):
    return I.structured_mesh(nx, ny)


def _mesh(case):
    return _polygon_mesh(case["nodes"]) if case.get("mesh") == "polygon" else _square_mesh(case["nx"], case["ny"])


def _nodes(case):
    if case["kind"] == "spmv":
        return case["rows"]
    if case["kind"] == "step_square":
        return case["side"] ** 2
    n = case["nodes"] if case.get("mesh") == "polygon" else case["nx"] * case["ny"]
    return n * case.get("samples", 1)


def _urban(xy, seed):
    """Rural floor with 40 urban Gaussians, one to a cell of an 8x5 grid, and five infection seeds (the 1:1
    exposed:infected start of Section 4), on the GPU; returns the state [n, 5] and the rates that belong to its
    densest place."""
    g = torch.Generator().manual_seed(1000003 * seed + 17)
    cell = torch.randperm(40, generator=g)
    pos = torch.rand(40, 2, generator=g, dtype=torch.float64)
    pos[:, 0] = 0.15 + 0.7 * ((cell % 8) + 0.2 + 0.6 * pos[:, 0]) / 8
    pos[:, 1] = 0.15 + 0.7 * ((cell // 8) + 0.2 + 0.6 * pos[:, 1]) / 5
    amp = (10.0 * torch.exp(0.75 * torch.randn(40, generator=g, dtype=torch.float64))).clamp(3.0, 25.0)
    wid = torch.rand(40, generator=g, dtype=torch.float64) * 0.025 + 0.005
    p = torch.from_numpy(xy).cuda()
    N = torch.ones(len(xy), dtype=torch.float64, device="cuda")
    seeds = torch.zeros_like(N)
    for k in range(40):
        r2 = (p[:, 0] - float(pos[k, 0])) ** 2 + (p[:, 1] - float(pos[k, 1])) ** 2
        N += float(amp[k]) * torch.exp(-r2 / (2.0 * float(wid[k]) ** 2))
        if k < 5:
            seeds += torch.exp(-r2 / (2.0 * 0.01 ** 2))
    U = torch.zeros(len(xy), 5, dtype=torch.float64, device="cuda")
    U[:, 2] = 0.01 * N * seeds.clamp(max=1.0)
    U[:, 1] = U[:, 2]
    U[:, 0] = N - U[:, 1] - U[:, 2]
    return U, I.params_ontario(float(N.max()))


def _later(U, seed):
    """A state of the same density some days on, rough node by node: every compartment occupied."""
    g = torch.Generator(device="cuda").manual_seed(7 * seed + 3)
    r = torch.rand(U.shape, generator=g, dtype=torch.float64, device="cuda")
    N = U.sum(1, keepdim=True)
    share = torch.tensor([0.7, 0.08, 0.07, 0.14, 0.01], dtype=torch.float64, device="cuda")
    return N * share * (0.95 + 0.1 * r)


def _field(xy, seed):
    x = xy[:, 0] * (3.0 + seed % 5) + xy[:, 1] * (2.0 + seed % 3)
    return 1.0 + 0.4 * np.sin(x + 0.1 * (seed % 61))


def _vector(n, seed):
    g = torch.Generator(device="cuda").manual_seed(11 * seed + 5)
    return torch.randn(n, 5, generator=g, dtype=torch.float64, device="cuda")


def _matrix(case, seed):
    """BSR rows of four to nine blocks near the diagonal, as mesh rows have them."""
    n = case["rows"]
    g = torch.Generator(device="cuda").manual_seed(13 * seed + 1)
    cnt = torch.randint(4, 10, (n,), generator=g, device="cuda")
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = cnt.cumsum(0)
    nb = int(rp[-1])
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), cnt)
    side = max(2, int(math.sqrt(n)))
    k = torch.arange(nb, device="cuda") - rp[row]
    col = (row + (k % 3 - 1) + (k // 3 - 1) * side).clamp(0, n - 1)
    val = torch.randn(nb, 25, generator=g, dtype=torch.float64, device="cuda")
    return rp.int(), col.int(), (val.float() if case["f32"] else val), _vector(n, seed)


_stream = None


def _context(case, xy, tri, rates, U, field=None, **more):
    """A context on a stream of the caller's, which orders its calls with the tensors around them."""
    from paper_2208_01839_gb300 import seird as S
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    return S.Solver(xy, tri, rates, beta_field=field, stream=_stream, **more)


def _ras_options(case):
    return dict(n_subdomains=case["sub"], overlap=case["overlap"], coarse=case["coarse"], ilu_fill=case["fill"],
                precision=case["precision"], dt=0.5)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "spmv":
        rp, col, val, x = _matrix(case, seed)
        return dict(kind=kind, args=(rp, col, val, x), y=torch.empty_like(x))
    if kind == "step_square":
        wl = I.square_workload(case["side"])
        U = wl.U0 * (1.0 + 0.05 * (seed % 97) / 97.0)
        sv = _context(case, wl.xy, wl.tri, wl.params, U, owner=wl.owner, dt=wl.dt, overlap=wl.overlap,
                      newton_rtol=1e-10, gmres_maxit=400, graph=1)
        return dict(kind="run", sv=sv, U=torch.from_numpy(U).cuda(), steps=1, out=torch.empty(wl.n, 5, dtype=torch.float64, device="cuda"))
    xy, tri = _mesh(case)
    n = len(xy)
    U, rates = _urban(xy, seed)
    if kind == "ensemble":
        sets = I.rate_samples(rates, case["samples"], seed)
        sv = _context(case, xy, tri, sets, U, n_subdomains=case["sub"], overlap=2, coarse=2, dt=0.5, graph=1,
                      newton_rtol=1e-8, gmres_forcing=1, pc_lag=20)
        U = U.repeat(case["samples"], 1)
        return dict(kind="run", sv=sv, U=U, steps=1, out=torch.empty_like(U))
    if kind == "adjoint":
        sv = _context(case, xy, tri, rates, U, n_subdomains=case["sub"], overlap=2, coarse=1, dt=0.5,
                      newton_rtol=1e-10, gmres_forcing=1, pc_lag=20)
        rng = np.random.default_rng(seed)
        nodes = rng.choice(n, 50, replace=False).astype(np.int32)
        at = np.arange(1, case["steps"] + 1, dtype=np.int32)
        seen = U[torch.from_numpy(nodes).long().cuda()].cpu().numpy()
        Ih = np.tile(1.1 * seen[:, 2] + 1e-3, (len(at), 1))
        Dh = np.tile(0.01 * seen[:, 2] + 1e-4, (len(at), 1))
        return dict(kind=kind, sv=sv, U=U, spec=(case["steps"], nodes, at, Ih, Dh, case["every"], 1e-12))
    if kind in ("residual", "jacobian"):
        field = _field(xy, seed) if case["field"] else None
        sv = _context(case, xy, tri, rates, U, field, n_subdomains=max(1, n // 4096), overlap=0, dt=0.5,
                      gmres_restart=2, quadrature=case["rule"], precision=case.get("precision", 0))
        V = _later(U, seed)
        if kind == "residual":
            return dict(kind=kind, sv=sv, U=V, Un=U, out=torch.empty_like(U))
        return dict(kind=kind, sv=sv, U=V, x=_vector(n, seed), out=torch.empty_like(U))
    if kind == "run":
        sv = _context(case, xy, tri, rates, U, **_ras_options(case), autotune=int(case["tune"]),
                      pc_keep_steps=case["steps"] - 1, **OPTIONS_OF_A_LONG_RUN)
        return dict(kind=kind, sv=sv, U=U, steps=case["steps"], out=torch.empty_like(U))
    sv = _context(case, xy, tri, rates, U, **_ras_options(case), gmres_restart=2)
    sv.jacobian(_later(U, seed))
    st = dict(kind=kind, sv=sv, x=_vector(n, seed), out=torch.empty_like(U), single=case["precision"] == 1)
    if kind == "precond":
        sv.precond_setup()
    return st


def run(state):
    kind = state["kind"]
    if kind == "spmv":
        from paper_2208_01839_gb300 import seird as S
        rp, col, val, x = state["args"]
        S.bsr_spmv(rp, col, val, x, state["y"], stream=torch.cuda.current_stream())
        return state["y"]
    sv = state["sv"]
    with torch.cuda.stream(_stream):
        if kind == "residual":
            return sv.residual(state["U"], state["Un"], state["out"])
        if kind == "jacobian":
            sv.jacobian(state["U"])
            return sv.apply_jacobian(state["x"], state["out"])
        if kind in ("precond_setup", "precond"):
            if kind == "precond_setup":
                sv.precond_setup()
            z = sv.precond_apply(state["x"], state["out"])
            return z.float() if state["single"] else z  # FP32 values, widened by the call
        if kind == "adjoint":
            steps, nodes, at, Ih, Dh, every, rtol = state["spec"]
            sv.set_state(state["U"])
            return sv.adjoint(steps, nodes, at, Ih, Dh, checkpoint_every=every, lin_rtol=rtol)
        sv.set_state(state["U"])
        sv.run(state["steps"])
        return sv.get_state(state["out"])


# ---- work ------------------------------------------------------------------------


def work(case):
    """Bytes and flops of one pass: matrices, factors and vectors once per use.  Iteration counts of the solves are
    those that the workloads take; factor blocks per local row by level of fill are those of the meshes."""
    n = float(_nodes(case))
    m, nnzb, kind = 2.0 * n, 7.0 * n, case["kind"]
    mixed = case.get("precision", 0) == 1
    w = 4.0 if mixed else 8.0
    if kind == "spmv":
        nnzb = 6.5 * n
        return dict(bytes=nnzb * (25 * (4.0 if case["f32"] else 8.0) + 4) + 84 * n, flops=50 * nnzb)
    res = (136 * n + 12 * m, 400 * m)
    jac = (56 * n + 12 * m + 25 * w * nnzb, 700 * m)
    spmv = (nnzb * (25 * w + 4) + 84 * n, 50 * nnzb)
    if kind == "residual":
        return dict(bytes=res[0], flops=res[1])
    if kind == "jacobian":
        return dict(bytes=jac[0] + spmv[0], flops=jac[1] + spmv[1])
    per_row = {0: 7.0, 1: 9.1, 2: 13.0, 3: 17.0}[case.get("fill", 0)]
    sub = case.get("sub", 4) * case.get("samples", 1)
    ov = case.get("overlap", 2)
    rows = n * (1 + 2 * ov / max(1.0, math.sqrt(n / sub))) ** 2
    blocks = per_row * rows
    solve = (blocks * (25 * w + 4) + 72 * rows + 5 * n * w, 50 * blocks)
    setup = (nnzb * 25 * w + blocks * (25 * w + 4), 250 * blocks * per_row / 3)
    twice = 2 if case.get("coarse", 0) == 2 else 1
    pc = tuple(twice * solve[i] + (spmv[i] if twice == 2 else 0) for i in range(2))
    if kind == "precond":
        return dict(bytes=pc[0], flops=pc[1])
    if kind == "precond_setup":
        return dict(bytes=pc[0] + setup[0], flops=pc[1] + setup[1])
    # (Newton, GMRES, set-ups) of one pass
    if kind == "step_square":
        newton, gmres, setups = 4, 350, 4
    elif kind == "adjoint":
        newton, gmres, setups = 7 * case["steps"], 60 * case["steps"], 3 * case["steps"]
    elif kind == "ensemble":
        newton, gmres, setups = 3, 5, 1
    else:
        newton, gmres, setups = 3 * case["steps"], 12 * case["steps"], 1
    it = tuple(pc[i] + spmv[i] for i in range(2))
    return {name: newton * (res[i] + jac[i]) + gmres * (it[i] + (400 * n if name == "bytes" else 200 * n)) + setups * setup[i]
            for i, name in enumerate(("bytes", "flops"))}


# ---- the same results in 64 bits, plainly -----------------------------------------

_R15 = math.sqrt(15.0)


def _rule(rule):
    if rule == 1:
        return torch.eye(3, dtype=torch.float64), torch.full((3,), 1.0 / 3.0, dtype=torch.float64)
    pts, wts = [[1 / 3] * 3], [9 / 40]
    for s in (-1.0, 1.0):
        a, wt = (6 + s * _R15) / 21, (155 + s * _R15) / 1200
        for k in range(3):
            p = [a, a, a]
            p[k] = 1 - 2 * a
            pts.append(p)
            wts.append(wt)
    return torch.tensor(pts, dtype=torch.float64), torch.tensor(wts, dtype=torch.float64)


def _element(u, un, gx, gy, area, b, p, dt, rule):
    """Element vector [3, 5] of the backward-Euler weak form for one triangle (u, un: [3, 5])."""
    L, W = (t.to(u.device) for t in _rule(rule))
    M = (torch.ones(3, 3, dtype=u.dtype, device=u.device) + torch.eye(3, dtype=u.dtype, device=u.device)) * area / 12
    F = M @ (u - un)
    nu = torch.tensor(list(p.nu) + [0.0], dtype=u.dtype, device=u.device)
    cx, cy = gx @ u, gy @ u
    F = F + dt * area * u.sum(1).mean() * nu * (gx[:, None] * cx + gy[:, None] * cy)
    q = L @ u
    s, e, i, r = q[:, 0], q[:, 1], q[:, 2], q[:, 3]
    N = q.sum(1)
    tr = (1 - p.A / N) * s * (p.beta_i * i + p.beta_e * e) * (L @ b)
    R = torch.stack([p.alpha * N - tr - p.mu * s, tr - (p.sigma + p.gamma_e + p.mu) * e,
                     p.sigma * e - (p.gamma_r + p.gamma_d + p.mu) * i, p.gamma_e * e + p.gamma_r * i - p.mu * r,
                     p.gamma_d * i], 1)
    return F - dt * area * (L.T @ (W[:, None] * R))


def _elements(xy, tri):
    p = torch.from_numpy(np.ascontiguousarray(xy)).cuda()[torch.from_numpy(tri).long().cuda()]
    x, y = p[:, :, 0], p[:, :, 1]
    two = (x[:, 1] - x[:, 0]) * (y[:, 2] - y[:, 0]) - (x[:, 2] - x[:, 0]) * (y[:, 1] - y[:, 0])
    gx = torch.stack([y[:, 1] - y[:, 2], y[:, 2] - y[:, 0], y[:, 0] - y[:, 1]], 1) / two[:, None]
    gy = torch.stack([x[:, 2] - x[:, 1], x[:, 0] - x[:, 2], x[:, 1] - x[:, 0]], 1) / two[:, None]
    return gx, gy, 0.5 * two


def _by_elements(f, xy, tri, per_node, out, n):
    """out[node] += f(element data) over all triangles, in slices that fit."""
    gx, gy, area = _elements(xy, tri)
    t = torch.from_numpy(tri).long().cuda()
    for a in range(0, len(tri), 1 << 18):
        k = slice(a, a + (1 << 18))
        v = torch.func.vmap(f)(*(q[t[k]] for q in per_node), gx[k], gy[k], area[k])
        out.index_add_(0, t[k].reshape(-1), v.reshape(-1, 5))
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "spmv":
        rp, col, val, x = _matrix(case, seed)
        n = case["rows"]
        row = torch.repeat_interleave(torch.arange(n, device="cuda"), (rp[1:] - rp[:-1]).long())
        y = torch.zeros_like(x)
        for a in range(0, len(col), 1 << 20):
            k = slice(a, a + (1 << 20))
            y.index_add_(0, row[k], torch.einsum("bij,bj->bi", val[k].double().view(-1, 5, 5), x[col[k].long()]))
        return y
    if kind == "step_square":
        wl = I.square_workload(case["side"])
        Un = torch.from_numpy(wl.U0 * (1.0 + 0.05 * (seed % 97) / 97.0)).cuda()
        n, t = wl.n, torch.from_numpy(wl.tri).long().cuda()
        gx, gy, area = _elements(wl.xy, wl.tri)
        b = torch.ones(3, dtype=torch.float64, device="cuda")
        f = lambda u, un, x, y, a: _element(u, un, x, y, a, b, wl.params, wl.dt, 0)  # noqa: E731
        dof = (5 * t[:, :, None] + torch.arange(5, device="cuda")).reshape(-1, 15)
        U, first = Un.clone(), None
        for _ in range(30):
            F = torch.zeros(5 * n, dtype=torch.float64, device="cuda")
            F.index_add_(0, dof.reshape(-1), torch.func.vmap(f)(U[t], Un[t], gx, gy, area).reshape(-1))
            size = float(F.norm())
            first = first or size
            if size < 1e-14 * first:
                break
            J = torch.zeros(25 * n * n, dtype=torch.float64, device="cuda")
            E = torch.func.vmap(torch.func.jacfwd(f))(U[t], Un[t], gx, gy, area).reshape(-1, 15, 15)
            J.index_add_(0, (dof[:, :, None] * (5 * n) + dof[:, None, :]).reshape(-1), E.reshape(-1))
            U = U - torch.linalg.solve(J.view(5 * n, 5 * n), F).view(n, 5)
        return U
    if kind not in ("residual", "jacobian") or case.get("precision", 0) == 1:
        return None
    xy, tri = _mesh(case)
    U, rates = _urban(xy, seed)
    V = _later(U, seed)
    b = torch.from_numpy(_field(xy, seed)).cuda() if case["field"] else torch.ones(len(xy), dtype=torch.float64, device="cuda")
    lump = case["rule"]
    if kind == "residual":
        f = lambda u, un, bb, x, y, a: _element(u, un, x, y, a, bb, rates, 0.5, lump)  # noqa: E731
        return _by_elements(f, xy, tri, (V, U, b), torch.zeros_like(U), len(xy))

    def f(u, v, bb, x, y, a):
        return torch.func.jvp(lambda w: _element(w, torch.zeros_like(w), x, y, a, bb, rates, 0.5, lump), (u,), (v,))[1]
    return _by_elements(f, xy, tri, (V, _vector(len(xy), seed), b), torch.zeros_like(U), len(xy))
