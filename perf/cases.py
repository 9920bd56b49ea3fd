"""What a program that uses this solver has it do, as timed cases.

A radiation-hydrodynamics code holds the coupled (G+2)x(G+2)-block system of
one time step in CSR arrays.  It sets up the preconditioner and solves (a
`step`), solves further right-hand sides with the setup it has (a `solve`),
uses the preconditioner inside a Krylov method of its own (an `apply`), does
the step from host arrays (a `host` step), checks a residual where it may not
allocate (a `relres`), or differentiates a solve (an `adjoint`: forward,
transposed solve and the gradient of the matrix values).

The systems are those of `paper_2002_04958_gb300.inputs`: cell-centred
two-point-flux stencils in 2-D or 3-D with log-uniform coefficients, groups
coupled to E and E to I cell by cell.  They are drawn here on the GPU, from the
seed alone, because the numpy generator takes tens of seconds at the largest
size.  Sizes are the configurations' (`inputs.PRESETS`), coarser grids of the
same systems, and grids whose extents are odd.
"""
import math

import numpy as np
import torch

from paper_2002_04958_gb300 import mgdamg

TOL = 1e-8  # relative residual that every solve asks for


def _case(name, op, G, dims, kind, law="multi", inclusion=False, interp=0, precision=0, smoother=0, graph=True):
    """One case: `law` is the diffusion law ("one" for the one-group system, "multi" for the multigroup one),
    `graph` the batched launches replayed from a CUDA graph (the framework's form for production runs)."""
    c = {"op": op, "G": G, "nx": dims[0], "ny": dims[1], "nz": dims[2] if len(dims) > 2 else 1, "kind": kind,
         "law": law, "inclusion": inclusion, "interp": interp, "precision": precision, "smoother": smoother,
         "graph": graph}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest call: a solve of the one-group 3-temperature system on a
        # coarse grid with the default options, as in a first test of a coupled code
        _case("solve-3t-32x32-amg", "solve", 1, (32, 32), "amg", law="one", graph=False),
        # the same preconditioner family on a box whose extents are no multiples of
        # anything, four groups in 3-D: a local refinement patch
        _case("solve-g4-37x29x23-schur1", "solve", 4, (37, 29, 23), "schur1"),
        # a residual check in a loop that may not allocate, just under the size
        # limit of that call
        _case("relres-g4-297x293", "relres", 4, (297, 293), "bd"),
        # the two-level scheme as the preconditioner of the caller's own Krylov method
        _case("apply-g4-45x41x43-pctl", "apply", 4, (45, 41, 43), "pctl"),
        # sensitivity of a solution to the coefficients: forward and transposed
        # solve and the value gradient, through autograd
        _case("adjoint-g4-64x64-amg", "adjoint", 4, (64, 64), "amg"),
        # the paper's smoother: monolithic AMG with C/F Gauss-Seidel, 20 groups in 2-D
        _case("solve-g20-256x256-amg-gs", "solve", 20, (256, 256), "amg", smoother=1),
        # a time step of the 20-group 2-D system, block-diagonal preconditioner, FP32 V-cycles
        _case("step-g20-256x256-bd-fp32", "step", 20, (256, 256), "bd", precision=1),
        # a time step from a host code's arrays, the one-group system with an inclusion
        _case("host-3t-500x500-schur1", "host", 1, (500, 500), "schur1", law="one", inclusion=True, interp=1),
        # the one-group system with an inclusion at its full size, further right-hand sides
        _case("solve-3t-1024x1024-schur1", "solve", 1, (1024, 1024), "schur1", law="one", inclusion=True, interp=1),
        # 20 groups in 3-D on a medium grid, FP32 V-cycles inside the FP64 Krylov method
        _case("solve-g20-64x64x64-schur2-fp32", "solve", 20, (64, 64, 64), "schur2", precision=1),
        # one preconditioner application on the largest system
        _case("apply-g20-96x96x96-schur2", "apply", 20, (96, 96, 96), "schur2"),
        # the largest: a time step of 20 groups in 3-D, 19.5 million unknowns
        _case("step-g20-96x96x96-schur2", "step", 20, (96, 96, 96), "schur2"),
    ]


# unknowns of a drawn case, per operation: an adjoint and a monolithic
# l1-Jacobi solve take hundreds of iterations, so their range ends earlier
_RANGE = {"solve": (3e3, 6e6), "step": (1e4, 1.2e7), "apply": (1e4, 1.9e7), "host": (1e4, 3e6),
          "relres": (2e3, 5.2e5), "adjoint": (3e3, 2.5e4)}


def draw(rng):
    op = rng.choice(["solve", "solve", "step", "step", "apply", "host", "relres", "adjoint"])
    lo, hi = _RANGE[op]
    G = rng.choice([1, 2, 3, 4, 7, 12, 20])
    law = "one" if G == 1 else "multi"
    smoother, interp = 0, 0
    if op == "adjoint":
        kind, G, law = "amg", rng.choice([2, 3, 4]), "multi"
    elif op == "relres":
        kind = "bd"
    else:
        kind = rng.choice(["schur1", "schur2", "bd", "pctl", "amg"])
    if kind == "amg" and op in ("solve", "step", "host"):
        smoother = 1
        hi = min(hi, 1.5e6)
    if law == "one":
        interp = 1 if kind != "amg" else 0
        if op != "relres" and kind not in ("amg", "schur1"):
            kind = "schur1"
    cells = math.exp(rng.uniform(math.log(lo), math.log(hi))) / (G + 2)
    nd = rng.choice([2, 3])
    side = cells ** (1.0 / nd)
    ext = [max(3, int(side * math.exp(rng.uniform(-0.35, 0.35)))) for _ in range(nd - 1)]
    ext.append(max(3, int(cells / math.prod(ext))))
    precision = 1 if op in ("solve", "step") and kind != "amg" and rng.random() < 0.4 else 0
    return _case("", op, G, ext, kind, law, False, interp, precision, smoother, rng.random() < 0.8)


# ------------------------------------------------------------------ the systems
def _dims(case):
    return [case["nx"], case["ny"]] + ([case["nz"]] if case["nz"] > 1 else [])


def _coefficients(case, seed):
    """Cell coefficients of the system: face transmissibilities per axis [nc, (nz,) ny, nx] (towards the upper
    neighbour, 0 on the last plane), couplings c_gE, c_Eg [G, N] and c_EI [N], the diagonal [nc, N], and b [n]."""
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev).manual_seed(int(seed) % (1 << 62))
    G, dims = case["G"], _dims(case)
    N, nc = math.prod(dims), case["G"] + 2
    shape = list(reversed(dims))

    def log_uniform(lo, hi, *size):
        u = torch.rand(*size, generator=gen, device=dev, dtype=torch.float64)
        return 10.0 ** (lo + (hi - lo) * u)

    k = torch.zeros(nc, N, dtype=torch.float64, device=dev)  # E does not diffuse
    for a in range(nc):
        if a < G and case["law"] == "multi":
            k[a] = log_uniform(-4.0, 2.0, N) * 10.0 ** (-(a + 1) / 5.0)
        elif a != G:
            k[a] = log_uniform(-3.0, 3.0, N)
    if case["inclusion"]:  # a disc with stronger diffusion
        u = torch.rand(3, generator=gen, device=dev, dtype=torch.float64).tolist()
        L = float(dims[0])
        ix = torch.arange(dims[0], device=dev, dtype=torch.float64) + 0.5
        iy = torch.arange(dims[1], device=dev, dtype=torch.float64) + 0.5
        inside = (ix[None, :] - u[0] * L) ** 2 + (iy[:, None] - u[1] * L) ** 2 <= ((0.1 + 0.15 * u[2]) * L) ** 2
        k *= torch.where(inside.expand(shape).reshape(-1), 1e4, 1.0)
    k = k.view(nc, *shape)
    cge, ceg, cei = log_uniform(-2.0, 2.0, G, N), log_uniform(-2.0, 2.0, G, N), log_uniform(-2.0, 2.0, N)
    diag = torch.ones_like(k)
    faces = []
    for ax in range(len(shape), 0, -1):  # x first
        n = shape[ax - 1]
        lo, hi = k.narrow(ax, 0, n - 1), k.narrow(ax, 1, n - 1)
        t = 2.0 * lo * hi / (lo + hi).clamp_min(1e-300)
        up = torch.zeros_like(k)
        up.narrow(ax, 0, n - 1).copy_(t)
        diag += up
        diag.narrow(ax, 1, n - 1).add_(t)
        for e in (0, n - 1):  # homogeneous Dirichlet faces
            diag.narrow(ax, e, 1).add_(2.0 * k.narrow(ax, e, 1))
        faces.append(up.view(nc, N))
    diag = diag.view(nc, N)
    diag[:G] += cge
    diag[G] += ceg.sum(0) + cei
    diag[G + 1] += cei
    b = torch.rand(nc * N, generator=gen, device=dev, dtype=torch.float64)
    return {"dims": dims, "G": G, "N": N, "nc": nc, "faces": faces, "cge": cge, "ceg": ceg, "cei": cei, "diag": diag,
            "b": b}


def _csr(s):
    """The block-major CSR arrays (int32 row pointers and columns, increasing in a row; float64 values)."""
    G, N, nc = s["G"], s["N"], s["nc"]
    dev = s["b"].device
    cell = torch.arange(N, device=dev, dtype=torch.int64)
    stride, lower, upper = 1, [], []
    for ax, d in enumerate(s["dims"]):
        pos = (cell // stride) % d
        lower.insert(0, (ax, stride, pos > 0))
        upper.append((ax, stride, pos < d - 1))
        stride *= d
    every = torch.ones(N, dtype=torch.bool, device=dev)
    counts, cols, vals = [], [], []
    for a in range(nc):
        link = [(G, s["cge"][a])] if a < G else [(G, s["cei"])] if a > G else \
            [(g, s["ceg"][g]) for g in range(G)] + [(G + 1, s["cei"])]
        C, V, M = [], [], []
        for beta, c in link:
            if beta < a:
                C.append(beta * N + cell), V.append(-c), M.append(every)
        if a != G:
            for ax, st, ok in lower:
                t = torch.zeros(N, dtype=torch.float64, device=dev)
                t[st:] = s["faces"][ax][a][:N - st]
                C.append(a * N + cell - st), V.append(-t), M.append(ok)
        C.append(a * N + cell), V.append(s["diag"][a]), M.append(every)
        if a != G:
            for ax, st, ok in upper:
                C.append(a * N + cell + st), V.append(-s["faces"][ax][a]), M.append(ok)
        for beta, c in link:
            if beta > a:
                C.append(beta * N + cell), V.append(-c), M.append(every)
        M = torch.stack(M, 1)
        counts.append(M.sum(1))
        cols.append(torch.stack(C, 1)[M].to(torch.int32))
        vals.append(torch.stack(V, 1)[M])
    rowptr = torch.zeros(nc * N + 1, dtype=torch.int64, device=dev)
    torch.cumsum(torch.cat(counts), 0, out=rowptr[1:])
    return rowptr.to(torch.int32), torch.cat(cols), torch.cat(vals)


# ------------------------------------------------------------------ the calls
def prepare(case, seed):
    s = _coefficients(case, seed)
    rowptr, col, val = _csr(s)
    b = s["b"]
    st = {"op": case["op"], "G": s["G"], "N": s["N"], "kind": case["kind"], "b": b}
    if case["op"] == "relres":
        # an iterate as a solver leaves it half way: the diagonal solution
        st.update(csr=(rowptr, col, val), x=b / s["diag"].reshape(-1),
                  out=torch.zeros(3, dtype=torch.float64, device=b.device))
        return st
    fast = 1 if case["graph"] else 0
    solver = mgdamg.Solver(precision=case["precision"], interp_type=case["interp"], smoother=case["smoother"],
                           batched=fast, use_graph=fast, keep_transpose=1 if case["op"] == "adjoint" else 0,
                           max_it=3000)
    st["solver"] = solver
    if case["op"] == "host":  # page-locked, as a code sets up its staging buffers once
        st["csr"] = tuple(t.cpu().pin_memory() for t in (rowptr, col, val))
        st["b"] = b.cpu().numpy()
        solver.setup_host(s["G"], s["N"], *st["csr"], case["kind"])
        return st
    solver.setup(s["G"], s["N"], rowptr, col, val, case["kind"])
    if case["op"] in ("step", "adjoint"):
        st["csr"] = (rowptr, col, val)
    if case["op"] == "adjoint":
        st["weight"] = torch.linspace(0.5, 1.5, b.numel(), dtype=torch.float64, device=b.device)
    return st


def run(st):
    op, solver = st["op"], st.get("solver")
    if op == "apply":
        return solver.precond_apply(st["b"])
    if op == "relres":
        mgdamg.relres_noalloc(*st["csr"], st["b"], st["x"], st["out"])
        return st["out"]
    if op == "step":
        solver.setup(st["G"], st["N"], *st["csr"], st["kind"])
    if op in ("step", "solve"):
        x, iterations, _, _ = solver.solve(st["b"], tol=TOL)
        return {"x": x, "iterations": iterations}
    if op == "host":
        solver.setup_host(st["G"], st["N"], *st["csr"], st["kind"])
        x, iterations, _ = solver.solve_host(st["b"], tol=TOL)
        return {"x": x, "iterations": iterations}
    val = st["csr"][2].detach().requires_grad_(True)
    b = st["b"].detach().requires_grad_(True)
    x = mgdamg.mgd_solve(val, b, solver, TOL)
    x.backward(st["weight"])
    return {"x": x.detach(), "dval": val.grad, "db": b.grad}


def work(case):
    """Inputs read once, outputs written once: the matrix (12 bytes an entry) and the vectors; one multiply-add per
    entry (an adjoint: two systems and the gradient)."""
    G, dims = case["G"], _dims(case)
    N, nc = math.prod(dims), case["G"] + 2
    nnz = nc * N + 2 * (G + 1) * N + (nc - 1) * sum(2 * (N - N // d) for d in dims)
    n = nc * N
    bytes_ = 12.0 * nnz + 4.0 * n + 16.0 * n
    flops = 2.0 * nnz
    if case["op"] == "adjoint":
        bytes_, flops = bytes_ + 8.0 * nnz + 16.0 * n, 2.0 * flops + nnz
    return {"bytes": bytes_, "flops": flops}


# ------------------------------------------------------------------ 64-bit results
def _matvec(s, x, transposed=False):
    """A x (or A^T x) from the coefficients; the stencils are symmetric, the couplings are not."""
    G, N = s["G"], s["N"]
    x = x.view(s["nc"], N)
    cge, ceg = (s["ceg"], s["cge"]) if transposed else (s["cge"], s["ceg"])
    y = s["diag"] * x
    stride = 1
    for t, d in zip(s["faces"], s["dims"]):
        y[:, :N - stride] -= t[:, :N - stride] * x[:, stride:]
        y[:, stride:] -= t[:, :N - stride] * x[:, :N - stride]
        stride *= d
    y[:G] -= cge * x[G]
    y[G] -= (ceg * x[:G]).sum(0) + s["cei"] * x[G + 1]
    y[G + 1] -= s["cei"] * x[G]
    return y.view(-1)


def _solve(s, b, transposed=False, tol=1e-14, most=4000):
    """A x = b by BiCGStab with the diagonal as its preconditioner, started again from the true residual until that
    stands at 64-bit rounding; None if `most` iterations do not get there."""
    dinv = 1.0 / s["diag"].reshape(-1)
    x = torch.zeros_like(b)
    bn, best, done, since = float(b.norm()), math.inf, 0, 0
    while True:
        r = b - _matvec(s, x, transposed)
        rn = float(r.norm()) / bn
        since = since + 1 if rn > 0.5 * best else 0
        best = min(best, rn)
        if rn <= tol or (best <= 1e-13 and since >= 2):
            return x
        if done >= most:
            return x if best <= 1e-12 else None
        goal = max(1e-9 * rn, 0.3 * tol) * bn
        r0, p, rho = r.clone(), r.clone(), r.dot(r)
        for it in range(1000):
            done += 1
            ph = dinv * p
            v = _matvec(s, ph, transposed)
            alpha = rho / r0.dot(v)
            q = r - alpha * v
            qh = dinv * q
            t = _matvec(s, qh, transposed)
            omega = t.dot(q) / t.dot(t)
            x = x + alpha * ph + omega * qh
            r = q - omega * t
            new = r0.dot(r)
            p = r + (new / rho * alpha / omega) * (p - omega * v)
            rho = new
            if it % 10 == 9 and not goal < float(r.norm()) < 1e3 * bn:
                break
        if not bool(torch.isfinite(x).all()):
            return None


def exact(case, seed):
    op = case["op"]
    if op == "apply":
        # a V-cycle's 64-bit value would need the whole hierarchy (coarsening, interpolation, Galerkin products) from
        # code that is not this repository's: far over the time allowed for plain torch
        return None
    if case["inclusion"]:
        return None  # coefficients up to 1e7 beside the unit mass term: no plain iteration gets to 64-bit rounding in time
    s = _coefficients(case, seed)
    b = s["b"]
    if op == "relres":
        r = float((b - _matvec(s, b / s["diag"].reshape(-1))).norm())
        return torch.tensor([r, float(b.norm()), r / float(b.norm())], dtype=torch.float64)
    x = _solve(s, b)
    if op == "adjoint":
        w = torch.linspace(0.5, 1.5, b.numel(), dtype=torch.float64, device=b.device)
        lam = _solve(s, w, transposed=True)
        if x is None or lam is None:
            return None
        rowptr, col, _ = _csr(s)
        row = torch.repeat_interleave(torch.arange(b.numel(), device=b.device), (rowptr[1:] - rowptr[:-1]).long())
        return {"x": x, "dval": -lam[row] * x[col.long()], "db": lam}
    if x is None:
        return None
    return {"x": x.cpu().numpy() if op == "host" else x, "iterations": None}
