"""Workloads that the solver's speed is measured on: upwind advection problems
set up and solved through the public entry points of paper_2508_17517_gb300.

A case is a dict of plain values.  `kind` names the call a user makes:

  solve    one right-hand side on a hierarchy that is already set up
  rhs      many right-hand sides on one hierarchy, in one call
  grids    many separate grids of uneven size, one hierarchy each, in one call
  gradient forward and backward through AdvectionSolver.solve (adjoint solve)
  oneshot  a new operator: problem, setup, right-hand side and first solve

`theta` is the angle of the velocity (any quadrant), `options` one of the
settings below, `precision` that of the V-cycle (the outer iteration is FP64).
Operators are fixed by the case except for `oneshot`, whose direction, like
every inflow value, source and target, is drawn from the seed.
"""
import math

import numpy as np
import torch

import paper_2508_17517_gb300 as G

# The paper's command line; the coarse polynomial of order 30 with the tight
# truncation test that the benchmark runs; the order 10 of the rectangular
# domain; the order-4 smoother of the smallest problem.
OPTIONS = {"paper": {},
           "order30": {"coarse_poly_order": 30, "trunc_rtol": 1e-2},
           "order10": {"coarse_poly_order": 10},
           "small": {"poly_order": 4, "trunc_start_level": 4}}
PRECISION = {"fp64": G.AIRG_FP64, "fp32": G.AIRG_MIXED_FP32, "bf16r": G.AIRG_MIXED_FP32_BF16R}
OUTER = {"fgmres": G.AIRG_OUTER_FGMRES, "richardson": G.AIRG_OUTER_RICHARDSON}
SMOOTHER = {"polynomial": G.AIRG_SMOOTH_POLYNOMIAL, "assembled": G.AIRG_SMOOTH_ASSEMBLED}


def _case(kind, nx, ny, theta, options="order30", precision="fp64", rtol=1e-10, **more):
    return {"kind": kind, "nx": nx, "ny": ny, "theta": theta, "options": options, "precision": precision,
            "rtol": rtol, **more}


def listed():
    return [
        # the smallest problem of the tests: launches and latency count
        _case("solve", 64, 64, 3 * math.pi / 8, "small", name="solve 64x64 fp64"),
        # a mid-size grid whose hierarchy fits in L2
        _case("solve", 1024, 1024, 0.5713, name="solve 1024x1024 fp64"),
        # the benchmark's grid in both precisions of the V-cycle
        _case("solve", 4096, 4096, 0.9272, name="solve 4096x4096 fp64"),
        _case("solve", 4096, 4096, 0.9272, precision="fp32", name="solve 4096x4096 fp32"),
        # the paper's own settings and outer iteration, on odd sizes and a flow
        # out of another quadrant
        _case("solve", 1531, 977, 2.2345, "paper", outer="richardson", name="richardson 1531x977 fp64"),
        # the long rectangle, vectors in pinned host memory, and the assembled
        # smoother (the faster one per cycle)
        _case("solve", 500, 13000, math.pi / 4, "order10", "fp32", smoother="assembled", host=True,
              name="rectangle 500x13000 fp32 host"),
        # many inflow and source fields on one operator: a wide batch in mixed
        # precision, and a narrow odd one in FP64
        _case("rhs", 2048, 2048, 0.8123, precision="fp32", rtol=1e-8, k=32, name="32 rhs 2048x2048 fp32"),
        _case("rhs", 611, 403, 4.4231, rtol=1e-8, k=7, name="7 rhs 611x403 fp64"),
        # grids of uneven size solved together
        _case("grids", 128, 1024, 0.0, rtol=1e-8, count=8, draw=41, name="8 grids 128..1024 fp64"),
        # one step of fitting inflow and source to a target field
        _case("gradient", 1024, 1024, 0.6981, name="gradient 1024x1024 fp64"),
        # a direction that is solved for once: the setup counts in full
        _case("oneshot", 97, 80, 1.0345, name="oneshot 97x80 fp64"),
        _case("oneshot", 2048, 1536, 0.7432, precision="fp32", name="oneshot 2048x1536 fp32"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _sides(rng, least, most):
    """nx, ny with least^2 <= nx ny <= most^2, up to 1 : 16."""
    area = math.exp(rng.uniform(math.log(least * least), math.log(most * most)))
    aspect = math.exp(rng.uniform(-math.log(4), math.log(4)))
    a = max(32, int(math.sqrt(area) * aspect))
    b = max(32, int(math.sqrt(area) / aspect))
    return a, b


def _angle(rng):
    return rng.randrange(4) * math.pi / 2 + rng.uniform(math.pi / 12, 5 * math.pi / 12)


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "rhs", "grids", "gradient", "oneshot", "oneshot"])
    theta, precision = _angle(rng), rng.choice(["fp64", "fp64", "fp32", "fp32", "bf16r"])
    if kind == "solve":
        nx, ny = _sides(rng, 64, 4000)
        more = {}
        if rng.random() < 0.25:
            more["outer"] = "richardson"
        if rng.random() < 0.25:
            more["smoother"] = "assembled"
        if rng.random() < 0.25:
            more["host"] = True
        options = rng.choice(["order30", "order30", "order10", "paper"])
        if options == "paper" and nx * ny > 1500000:    # its truncation test takes 100 steps a level
            options = "order10"
        return _case(kind, nx, ny, theta, options, precision, **more)
    if kind == "rhs":
        nx, ny = _sides(rng, 64, 1800)
        k = _log_int(rng, 2, 64)
        while k > 2 and nx * ny * k > 100000000:
            k -= 1
        return _case(kind, nx, ny, theta, precision=precision, rtol=1e-8, k=k)
    if kind == "grids":
        lo = _log_int(rng, 48, 256)
        return _case(kind, lo, _log_int(rng, lo + 8, 1024), 0.0, precision=precision, rtol=1e-8,
                     count=rng.randrange(3, 9), draw=rng.randrange(1 << 20))
    if kind == "gradient":
        nx, ny = _sides(rng, 64, 1400)
        return _case(kind, nx, ny, theta, precision=precision)
    nx, ny = _sides(rng, 64, 1700)
    return _case(kind, nx, ny, theta, precision=precision)


# ------------------------------------------------------------------ inputs --
def _options(case):
    over = dict(OPTIONS[case["options"]], precision=PRECISION[case["precision"]],
                outer=OUTER[case.get("outer", "fgmres")], smoother=SMOOTHER[case.get("smoother", "polynomial")])
    return G.airg_options_default(**over)


def _grids(case):
    """The grids of a `grids` case: (n, theta) each, square."""
    r = np.random.default_rng(case["draw"])
    return [(int(r.integers(case["nx"], case["ny"] + 1)),
             float(r.uniform(math.pi / 12, 5 * math.pi / 12))) for _ in range(case["count"])]


def _theta(case, seed):
    if case["kind"] != "oneshot":
        return case["theta"]
    return case["theta"] + 0.02 * (float(np.random.default_rng(seed).random()) - 0.5)


def _n_inflow(nx, ny):
    return nx + ny - 1


def _generator(seed, device):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    return g


def _uniform(shape, gen):
    return torch.rand(shape, dtype=torch.float64, device=gen.device, generator=gen)


def _fields(case, seed, device):
    """What the case draws, in the order of the draws: inflow values ~ U[0,1],
    sources ~ N(0,1), the target ~ N(1, 0.1^2)."""
    gen = _generator(seed, device)
    if case["kind"] == "grids":
        return [{"g": _uniform(_n_inflow(n, n), gen)} for n, _ in _grids(case)]
    nx, ny = case["nx"], case["ny"]
    n, nin = nx * ny, _n_inflow(nx, ny)
    if case["kind"] == "rhs":
        return {"g": _uniform((case["k"], nin), gen),
                "s": torch.randn((case["k"], n), dtype=torch.float64, device=device, generator=gen)}
    f = {"g": _uniform(nin, gen)}
    if case["kind"] == "gradient":
        f["s"] = torch.randn(n, dtype=torch.float32, device=device, generator=gen)
        f["target"] = 1.0 + 0.1 * torch.randn(n, dtype=torch.float64, device=device, generator=gen)
    return f


def _problem(nx, ny, theta):
    return G.airg_problem_advection2d(nx, ny, math.cos(theta), math.sin(theta))


def prepare(case, seed):
    kind, f, opts = case["kind"], _fields(case, seed, "cuda"), _options(case)
    nx, ny = case["nx"], case["ny"]
    if kind == "oneshot":
        return {"case": case, "theta": _theta(case, seed), "g": f["g"], "options": opts}
    if kind == "gradient":
        th = case["theta"]
        solver = G.AdvectionSolver(nx, ny, math.cos(th), math.sin(th), opts=opts)
        # the adjoint hierarchy is built by the first adjoint call and kept in
        # the handle: a fitting loop has it from its second step on
        G.airg_solve_adjoint(solver.handle, f["target"], rtol=1e-2)
        return {"case": case, "solver": solver, "g": f["g"].requires_grad_(), "s": f["s"].requires_grad_(),
                "target": f["target"]}
    if kind == "grids":
        probs = [_problem(n, n, th) for n, th in _grids(case)]
        batch = G.airg_setup_batch([(p["rowptr"], p["col"], p["val"]) for p in probs], opts)
        bs = [G.airg_assemble_rhs_advection2d(p, q["g"]) for p, q in zip(probs, f)]
        return {"case": case, "batch": batch, "bs": bs}
    prob = _problem(nx, ny, case["theta"])
    handle = G.airg_setup(prob["rowptr"], prob["col"], prob["val"], opts)
    b = G.airg_assemble_rhs_advection2d(prob, f["g"], f.get("s"))
    st = {"case": case, "handle": handle, "b": b}
    if case.get("host"):
        st["b"] = b.cpu().pin_memory()
        st["x"] = torch.zeros_like(st["b"]).pin_memory()
    return st


def run(state):
    case = state["case"]
    kind, rtol = case["kind"], case["rtol"]
    if kind == "oneshot":
        prob = _problem(case["nx"], case["ny"], state["theta"])
        handle = G.airg_setup(prob["rowptr"], prob["col"], prob["val"], state["options"])
        b = G.airg_assemble_rhs_advection2d(prob, state["g"])
        x, _ = G.airg_solve(handle, b, rtol=rtol)
        return x
    if kind == "gradient":
        g, s = state["g"], state["s"]
        u = state["solver"].solve(g, s, rtol=rtol)
        loss = ((u - state["target"]) ** 2).sum()
        grad_g, grad_s = torch.autograd.grad(loss, (g, s))
        return {"u": u.detach(), "grad_g": grad_g, "grad_s": grad_s}
    if kind == "grids":
        xs, _ = G.airg_solve_batch(state["batch"], state["bs"], rtol=rtol)
        return xs
    if case.get("host"):
        state["x"].zero_()
        x, _ = G.airg_solve(state["handle"], state["b"], state["x"], rtol=rtol)
        return x
    x, _ = G.airg_solve(state["handle"], state["b"], rtol=rtol)
    return x


# -------------------------------------------------------------------- work --
def _operator_bytes(n):
    """CSR of the operator: at most three entries a row, 64-bit row pointers."""
    return 3 * n * 12 + 8 * (n + 1)


def work(case):
    """The operator and each vector once (right-hand side and initial guess in,
    solution out); one product with the operator per solve, which no check of
    the result can do without."""
    if case["kind"] == "grids":
        n = sum(m * m for m, _ in _grids(case))
        return {"bytes": _operator_bytes(n) + 24 * n, "flops": 6 * n}
    n, nin = case["nx"] * case["ny"], _n_inflow(case["nx"], case["ny"])
    if case["kind"] == "rhs":
        return {"bytes": _operator_bytes(n) + 24 * n * case["k"], "flops": 6 * n * case["k"]}
    if case["kind"] == "gradient":
        # forward: g, s in, u out; backward: target in, both gradients out
        return {"bytes": _operator_bytes(n) + 8 * nin + 4 * n + 8 * n + 8 * n + 8 * nin + 4 * n, "flops": 15 * n}
    if case["kind"] == "oneshot":
        return {"bytes": _operator_bytes(n) + 8 * nin + 8 * n, "flops": 6 * n}
    return {"bytes": _operator_bytes(n) + 24 * n, "flops": 6 * n}


# ------------------------------------------------------------------- exact --
def _inflow_mask(nx, ny, theta, device):
    """True on the inflow nodes, [ny, nx]."""
    m = torch.zeros((ny, nx), dtype=torch.bool, device=device)
    m[:, 0 if math.cos(theta) > 0 else nx - 1] = True
    m[0 if math.sin(theta) > 0 else ny - 1, :] = True
    return m


def _sweep(r, c1, c2, free):
    """u with u[k,a,b] = r[k,a,b] + c1 u[k,a,b-1] + c2 u[k,a-1,b] (terms off the
    grid absent), by anti-diagonals a + b in 64 bits; `free` = (give, take): the
    nodes that others take from, and the nodes that take."""
    if r.shape[1] > r.shape[2]:
        return _sweep(r.transpose(1, 2), c2, c1, tuple(m.t() for m in free)).transpose(1, 2)
    k, na, nb = r.shape
    d = na + nb - 1
    a = torch.arange(na, device=r.device)

    def skew(x):     # [.., a, b] -> [a + b, .., a], zero off the grid
        out = torch.zeros((d,) + tuple(x.shape[:-2]) + (na,), dtype=torch.float64, device=r.device)
        for i in range(na):
            out[i:i + nb, ..., i] = x[..., i, :].to(torch.float64).movedim(-1, 0)
        return out

    t, give, take = skew(r), skew(free[0]), skew(free[1])
    for q in range(1, d):
        v = t[q - 1] * give[q - 1]
        add = c1 * v
        add[:, 1:] += c2 * v[:, :-1]
        t[q] += take[q] * add
    out = torch.empty((k, na, nb), dtype=torch.float64, device=r.device)
    for i in range(na):
        out[:, i, :] = t[i:i + nb, :, i].movedim(0, -1)
    return out


def _flips(theta):
    return [d for d, v in ((2, math.cos(theta)), (1, math.sin(theta))) if v < 0]


def _forward(nx, ny, theta, g, s):
    """Exact solution of the upwind system, one row per right-hand side."""
    dev = g.device
    vx, vy = abs(math.cos(theta)), abs(math.sin(theta))
    diag, h = vx + vy, 1.0 / (nx - 1)
    g = g.reshape(-1, g.shape[-1])
    k = g.shape[0]
    mask = _inflow_mask(nx, ny, theta, dev)
    r = torch.zeros((k, ny, nx), dtype=torch.float64, device=dev)
    if s is not None:
        r += h / diag * s.reshape(k, ny, nx).double()
    r[:, mask] = g
    flips = _flips(theta)
    free = (~mask).unsqueeze(0).flip(flips)[0] if flips else ~mask
    r = r.flip(flips) if flips else r
    # an inflow node takes nothing from its neighbours; every node gives
    u = _sweep(r, vx / diag, vy / diag, (torch.ones_like(free), free))
    return (u.flip(flips) if flips else u).reshape(k, ny * nx)


def _adjoint(nx, ny, theta, w):
    """A^-T w for one vector w."""
    vx, vy = abs(math.cos(theta)), abs(math.sin(theta))
    diag = vx + vy
    free = ~_inflow_mask(nx, ny, theta, w.device)
    flips = [d for d in (1, 2) if d not in _flips(theta)]     # against the flow
    r = w.reshape(1, ny, nx) / diag
    fr = free.unsqueeze(0)
    if flips:
        r, fr = r.flip(flips), fr.flip(flips)
    # an inflow row has no upwind entries: its unknown gives nothing back
    lam = _sweep(r, vx / diag, vy / diag, (fr[0], torch.ones_like(fr[0])))
    return (lam.flip(flips) if flips else lam).reshape(-1)


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    f = _fields(case, seed, dev)
    if case["kind"] == "grids":
        return [_forward(n, n, th, q["g"], None)[0] for (n, th), q in zip(_grids(case), f)]
    nx, ny, th = case["nx"], case["ny"], _theta(case, seed)
    u = _forward(nx, ny, th, f["g"], f.get("s"))
    if case["kind"] == "rhs":
        return u
    u = u[0]
    if case["kind"] == "gradient":
        vx, vy = abs(math.cos(th)), abs(math.sin(th))
        lam = _adjoint(nx, ny, th, 2.0 * (u - f["target"]))
        inflow = _inflow_mask(nx, ny, th, dev).reshape(-1)
        grad_s = torch.where(inflow, torch.zeros_like(lam), lam / (nx - 1))
        return {"u": u, "grad_g": (vx + vy) * lam[inflow], "grad_s": grad_s}
    return u.cpu() if case.get("host") else u
