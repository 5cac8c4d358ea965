"""The work that users of this solver have it do, as cases that can be timed.

A reservoir simulator calls the library in a few ways: it sets a solver up for a new grid,
hands it the Jacobian of every Newton step (same pattern, new values) and solves, with the
preconditioner kept (a large ``mu``) or regenerated for every solve (``mu = 0``, plain MSP);
it applies the preconditioner or the matrix by itself from a Krylov method of its own; it
solves many small systems as one block-diagonal stack; and it keeps a request loop over
several reservoirs whose matrices live on the host.  Each case is one such call on a grid of
the sizes that the repository's configurations, tests and benchmark use (2,048 cells with 3
unknowns up to 60x220x85 with 4).

The matrices follow the repository's synthetic recipe (``synthetic/jacobian.py``), drawn on
the GPU from the seed alone: 7-point stencil on a box, lognormal permeability (per layer
where ``layered``), harmonic transmissibilities, off-diagonal blocks -T (R + (b-1) I) with R
in U[0.1, 1], diagonal blocks = accumulation minus the row's couplings, and wells as extra
block rows that couple one column of cells each.
"""
import math

import numpy as np
import torch

import paper_2208_08594_gb300 as msp

DEV = "cuda"
MU_KEEP = 180  # keep the preconditioner while a solve takes at most this many iterations
TOL = 1e-6


def _case(name, op, nx, ny, nz, b, wells=0, layered=True, precision="fp64", colouring="alg41",
          count=1):
    return dict(name=name, op=op, nx=nx, ny=ny, nz=nz, b=b, wells=wells, layered=layered,
                precision=precision, colouring=colouring, count=count)


def listed():
    return [
        # one Newton step of the smallest grid: latency and launches are all there is
        _case("newton_small", "newton", 16, 16, 8, 3, layered=False),
        # y = A x alone, as a caller's own Krylov method or residual check uses it
        _case("spmv_mid", "spmv", 30, 110, 40, 4, wells=4),
        # one application of the preconditioner by a caller's own Krylov method: a ragged
        # grid with six unknowns, and the mid-size grid of the tests
        _case("apply_b6", "apply", 37, 41, 23, 6, wells=2),
        _case("apply_mid", "apply", 30, 110, 40, 4, wells=4),
        # a Newton step (new values, then a solve) with the preconditioner kept
        _case("newton_mid", "newton", 30, 110, 40, 4, wells=4),
        _case("newton_large", "newton", 60, 220, 85, 4, wells=4),
        # the same with the preconditioner stored in FP32, half the large grid
        _case("newton_fp32", "newton", 60, 220, 42, 4, wells=4, precision="fp32"),
        # a new grid: pattern and value SETUP, first use of the preconditioner, release
        _case("setup_new", "setup", 31, 35, 29, 4, wells=1),
        # plain MSP: the preconditioner regenerated for every Newton step
        _case("plain_msp", "plain", 30, 110, 40, 4, wells=4),
        # the same with the parallel colouring option, five unknowns, a ragged grid
        _case("plain_msp_jp", "plain", 61, 83, 37, 5, wells=3, colouring="jp"),
        # many small reservoirs of uneven size solved as one stack
        _case("batch", "batch", 24, 24, 12, 4, wells=1, count=24),
        # the request loop: Newton steps of several resident reservoirs, host buffers
        _case("serve", "serve", 28, 30, 20, 5, wells=1, count=4),
    ]


def _box(rng, lo, hi, nz_lo=5, nz_hi=40):
    """A box of log-uniform cell count, nz in the given range, an aspect of 1 to 4."""
    cells = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    nz = rng.randint(nz_lo, nz_hi)
    area = max(cells / nz, 16.0)
    nx = max(4, int(round(math.sqrt(area / rng.uniform(1.0, 4.0)))))
    return nx, max(4, int(round(area / nx))), nz


def draw(rng):
    op = rng.choice(["newton", "newton", "newton", "spmv", "apply", "apply", "setup", "plain",
                     "plain", "batch", "serve"])
    wells = rng.randint(0, 4)
    precision, colouring, count = "fp64", "alg41", 1
    if op == "newton":
        nx, ny, nz = _box(rng, 2e3, 4e5)
        b = rng.randint(3, 6)
        precision = rng.choice(["fp64", "fp64", "fp32"])
    elif op in ("spmv", "apply"):
        nx, ny, nz = _box(rng, 2e3, 4e5)
        b = rng.randint(2, 8) if nx * ny * nz < 2e5 else rng.randint(2, 5)
    elif op == "setup":
        nx, ny, nz = _box(rng, 2e3, 6e4)
        b = rng.randint(3, 6)
        colouring = rng.choice(["alg41", "jp"])
    elif op == "plain":
        nx, ny, nz = _box(rng, 1e4, 1.5e5)
        b = rng.randint(3, 6)
        colouring = rng.choice(["alg41", "jp"])
    elif op == "batch":
        nx, ny, nz = _box(rng, 2e3, 1e4)
        b, count = rng.choice([4, 6]), rng.randint(8, 24)
        wells = rng.randint(0, 2)
    else:
        nx, ny, nz = _box(rng, 1e4, 3e4)
        b, count = rng.randint(4, 6), rng.randint(2, 4)
    return dict(op=op, nx=nx, ny=ny, nz=nz, b=b, wells=wells, layered=True, precision=precision,
                colouring=colouring, count=count)


# ---------------------------------------------------------------- the matrices
class _Matrix:
    """A block system on the GPU: pattern, values of two Newton steps, right-hand side."""

    def __init__(self, nb, b, rp, ci, v0, v1, rhs):
        self.nb, self.b, self.rp, self.ci, self.v0, self.v1, self.rhs = nb, b, rp, ci, v0, v1, rhs


def _matrix(nx, ny, nz, b, wells, layered, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 1000003 + 17)
    f64 = dict(dtype=torch.float64, device=DEV)
    nc, nb = nx * ny * nz, nx * ny * nz + wells

    def rand(*shape):
        return torch.rand(*shape, generator=g, **f64)

    lnk = torch.randn(nz, ny, nx, generator=g, **f64)
    if layered:
        lnk = 2.0 * lnk + (6.0 * rand(nz) - 2.0)[:, None, None]
    k = torch.exp(lnk)
    eye = torch.eye(b, **f64)
    # the seven stencil slots of every cell in column order, then its well
    offs = (-nx * ny, -nx, -1, 0, 1, nx, nx * ny)
    T = torch.zeros(7, nz, ny, nx, **f64)

    def harmonic(p, q):
        return 2.0 * p * q / (p + q)

    fx, fy = harmonic(k[:, :, 1:], k[:, :, :-1]), harmonic(k[:, 1:], k[:, :-1])
    fz = (0.1 if layered else 1.0) * harmonic(k[1:], k[:-1])
    T[0, 1:], T[6, :-1] = fz, fz
    T[1, :, 1:], T[5, :, :-1] = fy, fy
    T[2, :, :, 1:], T[4, :, :, :-1] = fx, fx
    T = T.reshape(7, nc).t().contiguous()
    blocks = torch.zeros(nc, 8, b, b, **f64)
    for s in (0, 1, 2, 4, 5, 6):
        blocks[:, s] = -T[:, s, None, None] * (0.1 + 0.9 * rand(nc, b, b) + (b - 1) * eye)
    have = torch.zeros(nc, 8, dtype=torch.bool, device=DEV)
    have[:, :7] = T > 0
    have[:, 3] = True
    cols = torch.zeros(nc, 8, dtype=torch.int64, device=DEV)
    cells = torch.arange(nc, device=DEV)
    for s in range(7):
        cols[:, s] = cells + offs[s]
    wrows = torch.zeros(wells, nz + 1, b, b, **f64)
    wcols = torch.zeros(wells, nz + 1, dtype=torch.int64, device=DEV)
    place = torch.randperm(nx * ny, generator=torch.Generator().manual_seed(seed))[:wells]
    for w in range(wells):
        at = int(place[w]) + nx * ny * torch.arange(nz, device=DEV)
        wi = k.reshape(-1)[at]
        have[at, 7] = True
        cols[at, 7] = nc + w
        blocks[at, 7, :, 0] = -wi[:, None] * (0.1 + 0.9 * rand(nz, b))
        wrows[w, :nz, 0] = -wi[:, None] * (0.1 + 0.9 * rand(nz, b))
        wcols[w, :nz], wcols[w, nz] = at, nc + w
        wrows[w, nz] = eye
        wrows[w, nz, 0, 0] = 0.5 + 1.5 * float(rand(1))
    acc = (0.5 + 1.5 * rand(nc))[:, None, None] * eye + 0.1 * rand(nc, b, b)
    base_w = wrows[:, nz].clone()

    def close():
        """Diagonal blocks = accumulation minus the row's couplings; the flat values."""
        blocks[:, 3] = 0.0
        blocks[:, 3] = acc - blocks.sum(1)
        wrows[:, nz] = base_w
        wrows[:, nz, 0] -= wrows[:, :nz, 0].sum(1)
        return torch.cat([blocks[have].reshape(-1), wrows.reshape(-1)])

    v0 = close()
    # the next Newton step: every coupling times U[0.95, 1.05]
    for s in (0, 1, 2, 4, 5, 6, 7):
        blocks[:, s] *= 0.95 + 0.1 * rand(nc, b, b)
    wrows[:, :nz] *= 0.95 + 0.1 * rand(wells, nz, b, b)
    v1 = close()
    ci = torch.cat([cols[have], wcols.reshape(-1)]).to(torch.int32)
    counts = torch.cat([have.sum(1), torch.full((wells,), nz + 1, device=DEV)])
    rp = torch.zeros(nb + 1, dtype=torch.int32, device=DEV)
    rp[1:] = counts.cumsum(0).to(torch.int32)
    rhs = torch.randn(nb, b, generator=g, **f64)
    rhs[nc:, 1:] = 0.0
    return _Matrix(nb, b, rp, ci, v0, v1, rhs.reshape(-1).contiguous())


def _boxes(case):
    """The grids of a batch or of a request loop: uneven sizes around the case's box."""
    return [(max(4, case["nx"] - 3 * (i % 5)), max(4, case["ny"] - 2 * (i % 7)),
             max(4, case["nz"] - i % 3)) for i in range(case["count"])]


def _matrices(case, seed):
    wells, layered = case["wells"], case["layered"]
    if case["op"] in ("batch", "serve"):
        return [_matrix(nx, ny, nz, case["b"], wells, layered, seed * 64 + i)
                for i, (nx, ny, nz) in enumerate(_boxes(case))]
    return [_matrix(case["nx"], case["ny"], case["nz"], case["b"], wells, layered, seed)]


def _config(case, mu):
    return dict(mu=mu,
                precision=msp.MSP_PRECISION_FP32 if case["precision"] == "fp32" else msp.MSP_PRECISION_FP64,
                colouring=msp.MSP_COLOURING_JP if case["colouring"] == "jp" else msp.MSP_COLOURING_ALG41)


# ---------------------------------------------------------------- what a user has in hand
def prepare(case, seed):
    op = case["op"]
    ms = _matrices(case, seed)
    m = ms[0]
    n = m.nb * m.b
    if op == "setup":
        return dict(op=op, m=m, cfg=_config(case, MU_KEEP), w=torch.empty(n, dtype=torch.float64, device=DEV))
    if op == "serve":
        server = msp.Server(slots=4, hbm_budget=20 * 10**9, **_config(case, MU_KEEP))
        jobs = []
        for i, q in enumerate(ms):
            host = dict(values=q.v1.cpu().numpy(), rhs=q.rhs.cpu().numpy(), x=np.zeros(q.nb * q.b))
            first = server.submit(i, q.nb, q.b, host["rhs"], host["x"], values=q.v0.cpu().numpy(),
                                  row_ptr=q.rp.cpu().numpy(), col_idx=q.ci.cpu().numpy())
            jobs.append((i, q.nb, q.b, q.ci.numel(), host))
            server.wait(first)
        return dict(op=op, server=server, jobs=jobs)
    if op == "batch":
        nb = sum(q.nb for q in ms)
        off, rows, nz = [0], [torch.zeros(1, dtype=torch.int32, device=DEV)], 0
        for q in ms:
            rows.append(q.rp[1:] + nz)
            nz += q.ci.numel()
            off.append(off[-1] + q.nb)
        ci = torch.cat([q.ci + o for q, o in zip(ms, off)]).to(torch.int32)
        s = msp.BatchSolver(nb, m.b, torch.cat(rows), ci, torch.cat([q.v0 for q in ms]), off,
                            **_config(case, MU_KEEP))
        return dict(op=op, s=s, v1=torch.cat([q.v1 for q in ms]), rhs=torch.cat([q.rhs for q in ms]),
                    x=torch.empty(nb * m.b, dtype=torch.float64, device=DEV))
    s = msp.Solver(m.nb, m.b, m.rp, m.ci, m.v0, **_config(case, 0 if op == "plain" else MU_KEEP))
    x = torch.empty(n, dtype=torch.float64, device=DEV)
    if op == "plain":  # the first solve still uses the SETUP of the construction
        s.solve(m.rhs, x, TOL)
    return dict(op=op, s=s, v1=m.v1, rhs=m.rhs, x=x)


def run(state):
    op = state["op"]
    if op == "newton" or op == "plain":
        state["s"].update_values(state["v1"])
        state["s"].solve(state["rhs"], state["x"], TOL)
        return {"x": state["x"]}
    if op == "spmv":
        state["s"].spmv(state["rhs"], state["x"])
        return {"y": state["x"]}
    if op == "apply":
        state["s"].apply_precond(state["rhs"], state["x"])
        return {"w": state["x"]}
    if op == "setup":
        m = state["m"]
        s = msp.Solver(m.nb, m.b, m.rp, m.ci, m.v0, **state["cfg"])
        s.apply_precond(m.rhs, state["w"])
        colour = s.colour0()[0]
        sizes = [msp.msp_level_info(s.h, l) for l in range(s.num_levels)]
        s.close()
        return {"w": state["w"], "colour": colour, "levels": np.array(sizes)}
    if op == "batch":
        state["s"].update_values(state["v1"])
        state["s"].solve_batch(state["rhs"], state["x"], TOL)
        return {"x": state["x"]}
    server = state["server"]
    tickets = [server.submit(key, nb, b, h["rhs"], h["x"], values=h["values"], nnzb=nnzb, rel_tol=TOL)
               for key, nb, b, nnzb, h in state["jobs"]]
    for t in tickets:
        server.wait(t)
    return {"x%d" % key: h["x"] for key, _, _, _, h in state["jobs"]}


def exact(case, seed):
    """64-bit results of the products and, where a dense solve is small enough, of the solves."""
    op = case["op"]
    if op not in ("spmv", "newton"):
        return None
    m = _matrices(case, seed)[0]
    b, n = m.b, m.nb * m.b
    rows = torch.repeat_interleave(torch.arange(m.nb, device=DEV), m.rp.long().diff())
    if op == "spmv":  # the solver holds the first step's values
        p = (m.v0.view(-1, b, b) @ m.rhs.view(m.nb, b)[m.ci.long()].unsqueeze(-1)).squeeze(-1)
        y = torch.zeros(m.nb, b, dtype=torch.float64, device=DEV).index_add_(0, rows, p)
        return {"y": y.reshape(-1)}
    if n > 12000:
        return None
    a = torch.zeros(m.nb, b, m.nb, b, dtype=torch.float64, device=DEV)
    a[rows, :, m.ci.long(), :] = m.v1.view(-1, b, b)
    return {"x": torch.linalg.solve(a.view(n, n), m.rhs)}


# ---------------------------------------------------------------- what a pass cannot do without
def _sizes(nx, ny, nz, b, wells):
    nc = nx * ny * nz
    faces = (nx - 1) * ny * nz + nx * (ny - 1) * nz + nx * ny * (nz - 1)
    return nc + wells, nc + wells + 2 * faces + 2 * wells * nz


def _apply_work(nb, nnzb, b, e):
    """One application: six block Gauss-Seidel sweeps on the (b-1)^2 sub-blocks (the first
    from zero), the residual, the pressure column, the block ILU factors, a V-cycle on the
    pressure matrix and its coarser levels; each value once per use."""
    off = nnzb - nb
    values = 5.5 * off * (b - 1) ** 2 + nnzb * b * b * 2 + nnzb * b + nb * b * b
    amg = 3.0 * 1.75 * nnzb
    index = 4.0 * (5.5 * off + 3 * nnzb + amg)
    return e * (values + amg) + index + e * 20.0 * nb * b, 2.0 * (values + amg)


def work(case):
    grids = _boxes(case) if case["op"] in ("batch", "serve") else [(case["nx"], case["ny"], case["nz"])]
    b, op = case["b"], case["op"]
    bytes_, flops = 0.0, 0.0
    for nx, ny, nz in grids:
        nb, nnzb = _sizes(nx, ny, nz, b, case["wells"])
        n, vals = nb * b, nnzb * b * b
        once = 8.0 * vals + 4.0 * nnzb + 16.0 * n
        if op == "spmv":
            bytes_, flops = bytes_ + once, flops + 2.0 * vals
            continue
        ab, af = _apply_work(nb, nnzb, b, 4 if case["precision"] == "fp32" else 8)
        if op == "apply":
            bytes_, flops = bytes_ + ab, flops + af
            continue
        its = 1 if op == "setup" else 8 if nb < 4000 else 60
        # a step of FGMRES(30) reads about 15 basis vectors for the projections and again for
        # the update, and multiplies by the matrix
        bytes_ += once + its * (ab + once + 8.0 * 30 * n)
        flops += its * (af + 2.0 * vals + 4.0 * 30 * n)
        if op in ("setup", "plain"):  # the factors written once, the coarsest inverse
            nc = nb if nb <= 10000 else 5600
            bytes_ += 8.0 * (2 * vals + 8.0 * nc * nc)
            flops += 2.0 * nc ** 3 + 4.0 * vals * b
    return {"bytes": bytes_, "flops": flops}
