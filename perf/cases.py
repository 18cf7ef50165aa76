"""The workloads whose speed this repository is measured by.

A case is one call (or the few calls) a user of the solver makes again and
again on data already on the GPU: a whole solve, a batch of solves, the
point classification of a moving body, the right-hand side, the operator, the
preconditioner, and one layer of the learned part's network, forward and
backward.  Contexts, batches and buffers are made in ``prepare`` and kept, as
a program keeps them; fields, right-hand sides, body positions and layer
tensors come from the seed.

Solutions are polynomials in (x, y, z): the compact scheme and its modified
stencils reproduce degree 4 per variable, and degree 2 where a stencil had to
end early, so ``exact`` is the discrete solution itself.
"""
import math

import numpy as np
import torch

from paper_1901_08269_gb300 import cfp
from paper_1901_08269_gb300 import workloads as W

#: per geometry: tanh stretching per axis of [-1, 1] and the degree the
#: discretisation reproduces
GEOMETRIES = {
    "none": ((0.0, 0.0, 0.0), 4),      # the paper's Problem 1(i): uniform grid, no body
    "stretched": ((1.5, 1.5, 1.5), 4),  # no body, stretched grid
    "sphere": ((1.5, 1.5, 1.5), 4),    # one sphere, stretched towards it
    "bodies": ((2.0, 1.2, 1.2), 2),    # rotated ellipsoid and torus (some operators end early)
    "interior": ((0.8, 0.8, 0.8), 4),  # fluid inside a sphere
}


def listed():
    return [
        # the smallest whole solve, library defaults (FP64, eight red-black sweeps): latency and launches
        {"name": "solve-33-default", "op": "solve", "geometry": "none", "nx": 33, "ny": 33, "nz": 33,
         "precision": "fp64", "precond": "rbgs", "pre": 8, "post": 0, "inner_tol": 1e-5, "tol": 1e-12},
        # the paper's own configuration at the usual development size
        {"name": "solve-129-sphere-fp64", "op": "solve", "geometry": "sphere", "nx": 129, "ny": 129, "nz": 129,
         "precision": "fp64", "precond": "rbgs", "pre": 8, "post": 0, "inner_tol": 1e-5, "tol": 1e-14},
        # FP64 throughout with the multigrid preconditioner, uneven axes
        {"name": "solve-177x129x146-fp64-mg", "op": "solve", "geometry": "sphere", "nx": 177, "ny": 129, "nz": 146,
         "precision": "fp64", "precond": "mg", "pre": 2, "post": 0, "inner_tol": 1e-5, "tol": 1e-14},
        # an ordinary production solve: mixed precision, multigrid, library settings
        {"name": "solve-257-bodies-mixed", "op": "solve", "geometry": "bodies", "nx": 257, "ny": 257, "nz": 257,
         "precision": "mixed", "precond": "mg", "pre": 2, "post": 0, "inner_tol": 1e-5, "tol": 1e-14},
        # the largest: the benchmark's grid, bodies and solver settings
        {"name": "solve-513-bodies-mixed", "op": "solve", "geometry": "bodies", "nx": 513, "ny": 513, "nz": 513,
         "precision": "mixed", "precond": "mg", "pre": 5, "post": 3, "inner_tol": 3e-3, "tol": 1e-14},
        # many small uneven problems at once (33^3 to 129^3, random bodies), the graph kept between runs
        {"name": "batch-16-random", "op": "batch", "problems": 16, "first": 20261203, "largest": 129, "tol": 1e-12},
        # a body moves: points, IBI points and modified stencils anew on the benchmark's grid
        {"name": "classify-513-bodies", "op": "classify", "geometry": "bodies", "nx": 513, "ny": 513, "nz": 513},
        # a time step's new source and boundary data
        {"name": "rhs-321x257x289-stretched", "op": "rhs", "geometry": "stretched", "nx": 321, "ny": 257, "nz": 289},
        # the FP64 operator on a small uneven grid, as an outer iteration calls it
        {"name": "apply-f64-97x65x82-sphere", "op": "apply64", "geometry": "sphere", "nx": 97, "ny": 65, "nz": 82},
        # the FP32 operator of the mixed solve on a large uneven grid
        {"name": "apply-f32-449x385x321-stretched", "op": "apply32", "geometry": "stretched", "nx": 449, "ny": 385,
         "nz": 321},
        # the preconditioner alone in FP64 (an outer Krylov method of the user's own)
        {"name": "precond-rbgs-193x161x178", "op": "precond", "geometry": "stretched", "nx": 193, "ny": 161,
         "nz": 178, "pre": 8},
        # the network's finest level: a 16-channel layer, forward, input and weight gradients
        {"name": "layer-16-16-129x97x65", "op": "layer", "nx": 129, "ny": 97, "nz": 65, "cin": 16, "cout": 16},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["solve", "solve", "solve", "solve", "batch", "classify", "rhs", "apply64", "apply32", "precond",
                     "layer"])
    if op == "batch":
        return {"op": op, "problems": _log(rng, 2, 24), "first": rng.randrange(1, 10 ** 6),
                "largest": rng.choice([65, 97, 129]), "tol": 1e-12}
    if op == "layer":
        pairs = [(16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (64, 128), (128, 128)]
        cin, cout = rng.choice(pairs)
        hi = 129 * 16 // max(cin, 16)
        nx, ny, nz = (_log(rng, 9, max(hi, 17)) for _ in range(3))
        return {"op": op, "nx": nx, "ny": ny, "nz": nz, "cin": cin, "cout": cout}
    c = {"op": op, "geometry": rng.choice(["none", "stretched", "sphere", "sphere", "bodies", "interior"])}
    lo, hi = 33, 449
    if op == "classify":
        c["geometry"] = rng.choice(["sphere", "bodies", "interior"])
    if op == "solve":
        kind = rng.choice(["fp64-rbgs", "fp64-mg", "mixed-mg", "mixed-mg"])
        c["precision"], c["precond"] = kind.split("-")
        c["pre"], c["post"] = (8, 0) if c["precond"] == "rbgs" else rng.choice([(2, 0), (2, 0), (1, 1), (3, 2), (5, 3)])
        c["inner_tol"] = rng.choice([1e-5, 1e-3, 3e-3])
        c["tol"] = 1e-14
        hi = {"fp64-rbgs": 145, "fp64-mg": 193, "mixed-mg": 385}[kind]
    elif op == "precond":
        c["pre"] = rng.choice([1, 2, 4, 8, 8])
        hi = 257
    elif op == "apply64":
        hi = 321
    if c["geometry"] == "bodies":
        lo = 121  # the torus comes within a tenth of the box
    c["nx"], c["ny"], c["nz"] = (_log(rng, lo, hi) for _ in range(3))
    return c


# ------------------------------------------------------------------ inputs
def _grid(case):
    betas, _ = GEOMETRIES[case["geometry"]]
    return [W.tanh_grid(-1.0, 1.0, case[k], b) for k, b in zip(("nx", "ny", "nz"), betas)]


def _bodies(geometry, shift=(0.0, 0.0, 0.0)):
    if geometry == "sphere":
        b = [W.sphere((0.05, -0.03, 0.02), 0.3)]
    elif geometry == "bodies":
        b = W.config3_bodies()
    elif geometry == "interior":
        b = [W.sphere((0.02, -0.01, 0.03), 0.72)]
    else:
        b = []
    for one in b:
        one["c"] = tuple(x + s for x, s in zip(one["c"], shift))
    return b


def _poly(case, seed):
    """Coefficients p[a, b, c] of the solution sum p x^a y^b z^c."""
    d = GEOMETRIES[case["geometry"]][1] + 1
    g = np.random.default_rng(seed)
    deg = np.add.outer(np.add.outer(np.arange(d), np.arange(d)), np.arange(d))
    return g.standard_normal((d, d, d)) / (1.0 + deg)


def _laplace(p):
    """Coefficients of the Laplacian of the polynomial p."""
    q = np.zeros_like(p)
    m = np.arange(p.shape[0], dtype=np.float64)
    w = (m * (m - 1.0))[2:]
    q[:-2] += w[:, None, None] * p[2:]
    q[:, :-2] += w[None, :, None] * p[:, 2:]
    q[:, :, :-2] += w[None, None, :] * p[:, :, 2:]
    return q


def _powers(t, d):
    return torch.stack([t ** m for m in range(d)])


def _field(p, axes, device="cuda"):
    """The polynomial on every node, (nz, ny, nx)."""
    d = p.shape[0]
    x, y, z = (_powers(torch.as_tensor(a, dtype=torch.float64, device=device), d) for a in axes)
    t = torch.as_tensor(p, dtype=torch.float64, device=device)
    yx = torch.einsum("abc,ai,bj->cji", t, x, y)
    return torch.einsum("cji,ck->kji", yx, z).contiguous()


def _at(p, xyz):
    d = p.shape[0]
    x, y, z = (_powers(xyz[:, q], d) for q in range(3))
    t = torch.as_tensor(p, dtype=torch.float64, device=xyz.device)
    return torch.einsum("abc,an,bn,cn->n", t, x, y, z).contiguous()


def _noise(shape, seed, dtype=torch.float64):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype)


def _context(case, shift=(0.0, 0.0, 0.0), classify=True):
    x, y, z = _grid(case)
    ctx = cfp.Context(x, y, z, _bodies(case["geometry"], shift), fluid_inside=case["geometry"] == "interior")
    if classify:
        ctx.classify_points()
    return ctx


def _layer_tensors(case, seed):
    """Activations, weights and an incoming gradient of a layer, bfloat16,
    channels last, zero on the padding."""
    nx, ny, nz, cin, cout = (case[k] for k in ("nx", "ny", "nz", "cin", "cout"))

    def padded(c, s, relu):
        t = torch.zeros((nz + 2, ny + 2, nx + 2, c), dtype=torch.bfloat16, device="cuda")
        v = _noise((nz, ny, nx, c), s, torch.float32)
        t[1:-1, 1:-1, 1:-1] = (torch.relu(v) if relu else v).to(torch.bfloat16)
        return t

    inp = padded(cin, 4 * seed + 1, True)
    gout = padded(cout, 4 * seed + 2, False)
    w = (_noise((cout, 27, cin), 4 * seed + 3, torch.float32) * math.sqrt(2.0 / (27 * cin))).to(torch.bfloat16)
    bias = 0.1 * _noise((cout,), 4 * seed + 4, torch.float32)
    return inp, gout, w, bias


def _modes(k, amp, ph, X, Y, Z):
    s = torch.zeros_like(X)
    for m in range(8):
        s += amp[m] * torch.sin(k[m, 0] * X + k[m, 1] * Y + k[m, 2] * Z + ph[m])
    return s.reshape(-1).contiguous()


def prepare(case, seed):
    op = case["op"]
    if op == "layer":
        nx, ny, nz, cin, cout = (case[k] for k in ("nx", "ny", "nz", "cin", "cout"))
        axis = np.linspace(-1.0, 1.0, 9)
        inp, gout, w, bias = _layer_tensors(case, seed)
        return {"case": case, "ctx": cfp.Context(axis, axis, axis), "dims": (nx, ny, nz), "inp": inp, "gout": gout,
                "w": w, "bias": bias, "out": torch.empty_like(gout), "gin": torch.empty_like(inp),
                "dw": torch.zeros((cout, 27, cin), dtype=torch.float32, device="cuda"),
                "db": torch.zeros((cout,), dtype=torch.float32, device="cuda")}
    if op == "batch":
        # the generator's grids and bodies; eight Fourier modes as the source, zero Dirichlet data
        ctxs, fs, gs, gis, us = [], [], [], [], []
        g = np.random.default_rng(seed)
        for m in range(case["problems"]):
            w = W.random_problem(case["first"] + m, sizes=[n for n in (33, 49, 65, 97, 129) if n <= case["largest"]])
            ctx = cfp.Context(w.x, w.y, w.z, w.bodies, stream=torch.cuda.Stream())
            ctx.classify_points()
            X, Y, Z = w.mesh(torch, "cuda")
            k, amp, ph = g.integers(1, 7, (8, 3)), g.standard_normal(8), g.uniform(0.0, 2.0 * math.pi, 8)
            ctxs.append(ctx)
            fs.append(_modes(k, amp, ph, X, Y, Z))
            gs.append(torch.zeros(w.N, dtype=torch.float64, device="cuda"))
            gis.append(torch.zeros(ctx.n_ibi, dtype=torch.float64, device="cuda"))
            us.append(torch.zeros(w.N, dtype=torch.float64, device="cuda"))
        torch.cuda.synchronize()
        batch = cfp.Batch(ctxs, fs, gs, gis, us, tol=case["tol"], precision=cfp.PREC_MIXED, precond=cfp.PRECOND_MG)
        return {"case": case, "batch": batch, "us": us}
    if op == "classify":
        shift = 0.01 * (2.0 * np.random.default_rng(seed).random(3) - 1.0)
        ctx = _context(case, shift, classify=False)
        # room for the IBI points of every position the body may take
        most = 1024 + 5 * _context(case).n_ibi // 4
        return {"case": case, "ctx": ctx, "types": torch.empty(ctx.N, dtype=torch.uint8, device="cuda"),
                "ibi": torch.zeros((most, 3), dtype=torch.float64, device="cuda")}
    ctx = _context(case)
    n = ctx.N
    s = {"case": case, "ctx": ctx}
    if op in ("solve", "rhs"):
        p, axes = _poly(case, seed), _grid(case)
        s["f"] = _field(_laplace(p), axes).reshape(-1)
        s["g"] = _field(p, axes).reshape(-1)
        s["gi"] = _at(p, ctx.ibi_points()) if ctx.n_ibi else None
        s["out"] = torch.zeros(n, dtype=torch.float64, device="cuda")
    elif op == "apply32":
        s["x"] = _noise(n, seed, torch.float32)
        s["out"] = torch.empty(n, dtype=torch.float32, device="cuda")
    else:
        s["x"] = _noise(n, seed)
        s["out"] = torch.empty(n, dtype=torch.float64, device="cuda")
    if op == "solve":
        s["opts"] = cfp.default_opts(
            precision=cfp.PREC_MIXED if case["precision"] == "mixed" else cfp.PREC_FP64,
            precond=cfp.PRECOND_MG if case["precond"] == "mg" else cfp.PRECOND_RBGS, inner_tol=case["inner_tol"],
            **({"mg_smooth": case["pre"], "mg_post": case["post"]} if case["precond"] == "mg" else
               {"sweeps": case["pre"]}))
    return s


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "batch":
        for u in state["us"]:
            u.zero_()  # the batch solves from the iterate it finds
        torch.cuda.current_stream().synchronize()  # the contexts have streams of their own
        state["batch"].run()
        return state["us"]
    ctx = state["ctx"]
    if op == "solve":
        u = state["out"].zero_()
        ctx.solve(state["f"], state["g"], state["gi"], u, tol=case["tol"], opts=state["opts"])
        return u
    if op == "classify":
        ni, nb = ctx.classify_points(state["types"])
        return state["types"], ctx.ibi_points(state["ibi"]), ni, nb
    if op == "rhs":
        return ctx.assemble_rhs(state["f"], state["g"], state["gi"], state["out"])
    if op == "apply64":
        return ctx.apply(state["x"], state["out"])
    if op == "apply32":
        return ctx.apply_f32(state["x"], state["out"])
    if op == "precond":
        return ctx.precondition(state["x"], state["out"], sweeps=case["pre"])
    # a layer: forward with bias and ReLU, the input gradient through the
    # ReLU of the layer before, the weight and bias gradients
    dims, cin, cout = state["dims"], case["cin"], case["cout"]
    ctx.nn_conv3d(dims, cin, cout, state["inp"], state["w"], state["out"], bias=state["bias"], flags=cfp.NN_RELU)
    ctx.nn_conv3d(dims, cout, cin, state["gout"], state["w"], state["gin"], act=state["inp"],
                  flags=cfp.NN_DGRAD | cfp.NN_MASK)
    ctx.nn_wgrad(dims, cin, cout, state["inp"], state["gout"], state["dw"].zero_(), state["db"].zero_())
    return state["out"], state["gin"], state["dw"], state["db"]


# -------------------------------------------------------------------- work
def work(case):
    op = case["op"]
    if op == "batch":
        n = sum(W.random_problem(case["first"] + m, sizes=[q for q in (33, 49, 65, 97, 129) if q <= case["largest"]]).N
                for m in range(case["problems"]))
        # source and first iterate in, solution out; about 20 iterations of two V(2,2) cycles and two applies
        return {"bytes": 24.0 * n, "flops": 20.0 * 2.0 * (106 + 75) * n}
    n = float(case["nx"] * case["ny"] * case["nz"])
    if op == "layer":
        cin, cout = case["cin"], case["cout"]
        m = 27.0 * cin * cout
        return {"bytes": n * (2 * cin * 4 + 2 * cout * 3) + 8 * m, "flops": 3 * 2 * n * m}
    if op == "solve":
        # the paper's count per outer iteration (its table of operations): 106 + 20 per node for the two operator
        # products and the vector updates, 13 per node and sweep of each preconditioner solve (a V-cycle costs 8/7 of
        # its fine sweeps); the iterations are the usual ones of each preconditioner
        if case["precond"] == "mg":
            sweeps, its = 8.0 / 7.0 * (case["pre"] + (case["post"] or case["pre"])), 20.0
        else:
            sweeps, its = case["pre"], 0.7 * max(case["nx"], case["ny"], case["nz"])
        return {"bytes": 24.0 * n, "flops": its * (126.0 + 2 * 13.0 * sweeps) * n}
    if op == "classify":
        return {"bytes": n, "flops": 20.0 * n}
    if op == "rhs":
        return {"bytes": 16.0 * n, "flops": 30.0 * n}
    if op == "precond":
        return {"bytes": 16.0 * n, "flops": 13.0 * case["pre"] * n}
    return {"bytes": (16.0 if op == "apply64" else 8.0) * n, "flops": 40.0 * n}


# ------------------------------------------------------------------- exact
def _compact(a):
    """(L, R) of the compact fourth-order scheme L u'' = R u on the axis a, as
    (n, 3) tensors of the weights of i - 1, i, i + 1 (zero at the ends)."""
    x = torch.as_tensor(a, dtype=torch.float64, device="cuda")
    f, b = x[2:] - x[1:-1], x[1:-1] - x[:-2]
    D = f ** 3 + 4 * f * f * b + 4 * f * b * b + b ** 3
    one = torch.ones_like(f)
    L = torch.stack([f * (b * b + b * f - f * f) / D, one, b * (f * f + b * f - b * b) / D], 1)
    R = torch.stack([12 * f / D, -12 / (f * f + 3 * f * b + b * b), 12 * b / D], 1)
    pad = (0, 0, 1, 1)
    return torch.nn.functional.pad(L, pad), torch.nn.functional.pad(R, pad)


def _along(t, w, dim):
    """The three-point operator w along axis dim of t (zero at the ends)."""
    n = t.shape[dim]
    out = torch.zeros_like(t)
    shape = [1, 1, 1]
    shape[dim] = n - 2
    out.narrow(dim, 1, n - 2).copy_(sum(w[1:-1, q].reshape(shape) * t.narrow(dim, q, n - 2) for q in range(3)))
    return out


def _interior(t):
    out = torch.zeros_like(t)
    out[1:-1, 1:-1, 1:-1] = t[1:-1, 1:-1, 1:-1]
    return out


def _operator(axes, u):
    (Lx, Rx), (Ly, Ry), (Lz, Rz) = (_compact(a) for a in axes)
    ly = _along(_along(u, Lx, 2), Ly, 1)
    s = _along(ly, Rz, 0)
    s += _along(_along(_along(u, Rx, 2), Ly, 1) + _along(_along(u, Lx, 2), Ry, 1), Lz, 0)
    return _interior(s)


def _source(axes, f):
    (Lx, _), (Ly, _), (Lz, _) = (_compact(a) for a in axes)
    return _interior(_along(_along(_along(f, Lx, 2), Ly, 1), Lz, 0))


def _red_black(axes, rho, sweeps):
    k = []
    for dim, a in ((2, axes[0]), (1, axes[1]), (0, axes[2])):
        x = torch.as_tensor(a, dtype=torch.float64, device="cuda")
        f, b = x[2:] - x[1:-1], x[1:-1] - x[:-2]
        shape = [1, 1, 1]
        shape[dim] = -1
        k.append([t.reshape(shape) for t in (2 / (b * (f + b)), -2 / (b * f), 2 / (f * (f + b)))])
    (xl, xc, xh), (yl, yc, yh), (zl, zc, zh) = k
    inner = (slice(1, -1),) * 3
    r, diag = rho[inner], xc + yc + zc
    colour = torch.arange(r.shape[0], device="cuda")[:, None, None] + torch.arange(r.shape[1], device="cuda")[:, None]
    colour = (colour + torch.arange(r.shape[2], device="cuda") + 1) % 2  # node (1, 1, 1) has i + j + k odd
    phi = torch.zeros_like(rho)
    for q in range(2 * sweeps):
        off = (xl * phi[1:-1, 1:-1, :-2] + xh * phi[1:-1, 1:-1, 2:] + yl * phi[1:-1, :-2, 1:-1] +
               yh * phi[1:-1, 2:, 1:-1] + zl * phi[:-2, 1:-1, 1:-1] + zh * phi[2:, 1:-1, 1:-1])
        phi[inner] = torch.where(colour == q % 2, (r - off) / diag, phi[inner])
    return phi


def _solid(case, axes):
    X, Y, Z = (torch.as_tensor(a, dtype=torch.float64, device="cuda") for a in axes)
    Z, Y, X = torch.meshgrid(Z, Y, X, indexing="ij")
    inside = torch.zeros(X.shape, dtype=torch.bool, device="cuda")
    for b in _bodies(case["geometry"]):
        R, c, p = np.asarray(b["R"]), b["c"], b["p"]
        d = (X - c[0], Y - c[1], Z - c[2])
        q = [R[0, m] * d[0] + R[1, m] * d[1] + R[2, m] * d[2] for m in range(3)]
        if b["kind"] == "sphere":
            inside |= q[0] ** 2 + q[1] ** 2 + q[2] ** 2 <= p[0] ** 2
        elif b["kind"] == "ellipsoid":
            inside |= (q[0] / p[0]) ** 2 + (q[1] / p[1]) ** 2 + (q[2] / p[2]) ** 2 <= 1.0
        else:
            inside |= (torch.sqrt(q[0] ** 2 + q[1] ** 2) - p[0]) ** 2 + q[2] ** 2 <= p[1] ** 2
    solid = torch.zeros_like(inside)
    solid[1:-1, 1:-1, 1:-1] = (~inside if case["geometry"] == "interior" else inside)[1:-1, 1:-1, 1:-1]
    return solid


def _layer_exact(case, seed):
    nx, ny, nz, cin, cout = (case[k] for k in ("nx", "ny", "nz", "cin", "cout"))
    inp, gout, w, bias = (t.to(torch.float64) for t in _layer_tensors(case, seed))
    out, gin, dw = torch.zeros_like(gout), torch.zeros_like(inp), torch.zeros_like(w)
    inner = (slice(1, -1),) * 3
    g = gout[inner].reshape(-1, cout)
    for t in range(27):
        at = tuple(slice(o, o + n) for o, n in zip((t // 9, (t // 3) % 3, t % 3), (nz, ny, nx)))
        back = tuple(slice(2 - o, 2 - o + n) for o, n in zip((t // 9, (t // 3) % 3, t % 3), (nz, ny, nx)))
        a = inp[at].reshape(-1, cin)
        out[inner] += (a @ w[:, t].T).reshape(nz, ny, nx, cout)
        gin[inner] += (gout[back].reshape(-1, cout) @ w[:, t]).reshape(nz, ny, nx, cin)
        dw[:, t] = g.T @ a
    out[inner] = torch.relu(out[inner] + bias)
    return out, gin * (inp > 0), dw, g.sum(0)


def exact(case, seed):
    op = case["op"]
    if op == "layer":
        if 6.0 * 27 * case["nx"] * case["ny"] * case["nz"] * case["cin"] * case["cout"] > 5e12:
            return None  # too slow in 64 bits
        return _layer_exact(case, seed)
    if op in ("batch", "classify"):
        return None  # no closed form without a whole solver; the points themselves
    axes = _grid(case)
    shape = (case["nz"], case["ny"], case["nx"])
    if op == "solve":
        u = _field(_poly(case, seed), axes)
        return u.masked_fill_(_solid(case, axes), 0.0).reshape(-1)
    if _bodies(case["geometry"]):
        return None  # the modified rows have no short plain form
    if op == "rhs":
        p = _poly(case, seed)
        g = _field(p, axes)
        g[1:-1, 1:-1, 1:-1] = 0.0
        return (_source(axes, _field(_laplace(p), axes)) - _operator(axes, g)).reshape(-1)
    n = shape[0] * shape[1] * shape[2]
    if op == "precond":
        return _red_black(axes, _noise(n, seed).reshape(shape), case["pre"]).reshape(-1)
    x = _noise(n, seed, torch.float32 if op == "apply32" else torch.float64).to(torch.float64)
    return _operator(axes, x.reshape(shape)).reshape(-1)
