"""The work a user has this library do, as timed cases.

Each case goes through the public entry points of ``paper_2311_08946_gb300``:

* ``spmv``     -- ``spmv_csr`` on the CSR matrix of an interfacial system, C x or C^T x;
* ``krylov``   -- ``solve_csr`` / ``solve_csr_noalloc`` on such a matrix, C u = b or C^T u = b;
* ``gemm``     -- ``gemm_tf32x3``, the batched split-TF32 product of the disk factorisations;
* ``cover``    -- ``Cover``: circles, knots, row owners and the CSR pattern;
* ``system``   -- ``System`` (every floating disk and Monte Carlo row) and ``System.solve``;
* ``gradient`` -- one ``MisfitSolve`` training step: forward solve and adjoint gradients.

The geometries, grids, path counts and step sizes are those of the workloads the tests and the
benchmark use, and smaller and larger domains of the same kinds.  A seed moves the domain, draws
the coefficient parameters and seeds the Monte Carlo streams, so another seed is another problem.
"""
import math

import numpy as np
import torch

import paper_2311_08946_gb300 as pdd

KNOTS = {"lattice": 16, "hex": 32, "poisson46": 44}


# ---------------------------------------------------------------------------
# problem descriptions
# ---------------------------------------------------------------------------
def _rbf(rng, n, sigma, box, negative):
    w = rng.standard_normal(n)
    return {"x": rng.uniform(box[0], box[2], n), "y": rng.uniform(box[1], box[3], n),
            "w": -np.abs(w) if negative else w, "sigma": sigma}


def _boundary_fourier(box, n_cos=16, n_sin=16, samples=2048):
    """Fourier coefficients along the square's arclength that fit e^x sin y there."""
    x0, y0, x1, y1 = box
    w, h = x1 - x0, y1 - y0
    per = 2 * (w + h)
    s = (np.arange(samples) + 0.5) * per / samples
    x = np.where(s < w, x0 + s, np.where(s < w + h, x1, np.where(s < 2 * w + h, x1 - (s - w - h), x0)))
    y = np.where(s < w, y0, np.where(s < w + h, y0 + (s - w), np.where(s < 2 * w + h, y1, y1 - (s - 2 * w - h))))
    t = 2 * np.pi * s / per
    cols = [np.cos(k * t) for k in range(n_cos)] + [np.sin(k * t) for k in range(1, n_sin + 1)]
    return np.linalg.lstsq(np.stack(cols, 1), np.exp(x) * np.sin(y), rcond=None)[0]


def _config(case, seed):
    """The workload description of a case's geometry for one seed."""
    rng = np.random.default_rng(seed)
    mc = {"paths": case.get("paths", 1000), "h": case.get("h", 1e-4), "seed": int(rng.integers(1 << 31))}
    geo, m = case["geometry"], case["size"]
    ox, oy = rng.uniform(-0.25, 0.25, 2)
    rows = case.get("rows", "farthest")
    if geo == "lattice":                     # harmonic data on an m x m square lattice, radius 0.8 spacings
        s = case["spacing"]
        box = [ox, oy, ox + m * s, oy + m * s]
        return {"name": geo, "domain": {"kind": "square", "p": box},
                "cover": {"kind": "square_lattice", "nx": m, "ny": m, "x_origin": ox + 0.5 * s,
                          "y_origin": oy + 0.5 * s, "spacing": s, "radius": 0.8 * s, "rows": rows},
                "n_knots": 16, "n_r": case["n_r"], "n_theta": case["n_theta"],
                "op": {"b": "zero", "c": "zero", "f": "zero", "g": "exp_sin"}, "mc": mc, "imq_c2": 1.5}
    if geo == "hex":                         # variable drift, killing and source; m circles along an edge
        s = 0.07
        side = (m + 4.0 / 7.0) * s           # m = 28: side 2 (on a multiple of s two circles meet the edge in one knot)
        return {"name": geo, "domain": {"kind": "square", "p": [ox, oy, ox + side, oy + side]},
                "cover": {"kind": "hex_lattice", "nx": m + 2, "ny": math.ceil(side / (s * math.sqrt(3) / 2)) + 2,
                          "x_origin": ox, "y_origin": oy, "spacing": s, "radius": 0.05, "rows": rows},
                "n_knots": 32, "n_r": 32, "n_theta": 32,
                "op": {"b": "sinx_cosy", "c": "quadratic", "f": "manufactured", "g": "sin_cos"}, "mc": mc,
                "imq_c2": 1.5}
    if geo == "poisson46":                   # the paper's Poisson test on [-5m, 5m]^2, moved a little
        mc |= {"boundary_shift": True, "cv_degree": 4}
        ox, oy = 4 * ox, 4 * oy
        return {"name": geo, "domain": {"kind": "square", "p": [ox - 5 * m, oy - 5 * m, ox + 5 * m, oy + 5 * m]},
                "cover": {"kind": "square_lattice", "nx": m, "ny": m, "x_origin": ox - 5 * m + 5,
                          "y_origin": oy - 5 * m + 5, "spacing": 10.0, "radius": 9.0, "rows": rows},
                "n_knots": 44, "n_r": 22, "n_theta": 44,
                "op": {"b": "zero", "c": "zero", "f": "eq46", "g": "eq46"}, "mc": mc, "imq_c2": 1.5}
    # "disk": uneven circles on the disk of radius m / 16, 16 macro cells along a unit-disk edge, c from
    # Gaussians; grids 16^2 .. 64^2 by radius and adaptive path counts
    cells, cw = 16, 0.125
    cx, cy, rr = [], [], []
    shape = np.random.default_rng(0)         # one cover for every seed: its size is the case's
    for j in range(cells):
        for i in range(cells):
            r = float(np.clip(shape.lognormal(math.log(0.025), 0.5), 0.02, 0.1))
            k = math.ceil(cw / (0.9 * r))
            g = (np.arange(k) + 0.5) * cw / k
            x, y = np.meshgrid(-1.0 + i * cw + g, -1.0 + j * cw + g)
            cx.append(x.ravel())
            cy.append(y.ravel())
            rr.append(np.full(k * k, r))
    cx, cy, rr = np.concatenate(cx), np.concatenate(cy), np.concatenate(rr)
    n = np.clip(16 + 8 * np.rint(6.0 * (rr - 0.02) / 0.08).astype(np.int64), 16, 64).astype(np.int32)
    mc |= {"paths_max": case["paths_max"], "se_target": case["se_target"]}
    return {"name": geo, "domain": {"kind": "disk", "p": [ox, oy, m / 16.0, 0.0]},
            "cover": {"kind": "explicit", "cx": cx + ox, "cy": cy + oy, "r": rr, "n_knots": n, "n_r": n,
                      "n_theta": n, "rows": rows},
            "n_knots": 0, "n_r": 0, "n_theta": 0,
            "op": {"b": "zero", "c": "rbf", "f": "zero", "g": "exp_sin",
                   "rbf": _rbf(rng, 64, 0.2, [ox - 0.8, oy - 0.8, ox + 0.8, oy + 0.8], False)},
            "mc": mc, "imq_c2": 1.5}


def _interfacial_csr(m, n, seed, transpose):
    """C and b of the Laplacian on an m x m lattice of circles with n knots each (radius 0.8 spacings).

    A knot inside the square takes its row from the other circle whose centre is nearest: minus the
    Fourier cardinals of the disk's Poisson kernel.  A knot outside is a Dirichlet row.  Columns ascend.
    b holds boundary data in the Dirichlet rows, or a misfit's derivative in every row for the adjoint.
    """
    d = torch.device("cuda")
    f = dict(dtype=torch.float64, device=d)
    i = torch.arange(m * m, device=d)
    cx, cy = (i % m).to(torch.float64) + 0.5, torch.div(i, m, rounding_mode="floor").to(torch.float64) + 0.5
    t = 2 * math.pi * torch.arange(n, **f) / n
    x = (cx[:, None] + 0.8 * torch.cos(t)).reshape(-1)
    y = (cy[:, None] + 0.8 * torch.sin(t)).reshape(-1)
    own = i.repeat_interleave(n)
    best, to = torch.full_like(x, 9.0), torch.zeros_like(own)
    for a in (-1, 0, 1):
        for b in (-1, 0, 1):
            if a == 0 and b == 0:
                continue
            px, py = own % m + a, torch.div(own, m, rounding_mode="floor") + b
            dist = torch.hypot(x - px.to(x.dtype) - 0.5, y - py.to(y.dtype) - 0.5)
            dist = torch.where((px < 0) | (px >= m) | (py < 0) | (py >= m), torch.full_like(dist, 9.0), dist)
            near = dist < best - 1e-9
            best, to = torch.where(near, dist, best), torch.where(near, py * m + px, to)
    inner = (x > 0) & (x < m) & (y > 0) & (y < m) & (best < 0.8)
    N = m * m * n
    row = torch.arange(N, device=d)
    dx, dy = x - cx[to], y - cy[to]
    rho, ang = torch.hypot(dx, dy) / 0.8, torch.atan2(dy, dx)
    ph = ang[:, None] - t
    w = torch.ones(N, n, **f)
    for j in range(1, n // 2):
        w += 2 * (rho ** j)[:, None] * torch.cos(j * ph)
    w += (rho ** (n // 2))[:, None] * torch.cos((n // 2) * ph)
    r = row[inner]
    rows = torch.cat([row, r.repeat_interleave(n)])
    cols = torch.cat([row, (to[inner, None] * n + torch.arange(n, device=d)).reshape(-1)])
    vals = torch.cat([torch.ones(N, **f), (-w[inner] / n).reshape(-1)])
    order = torch.argsort(rows * N + cols)
    rowptr = torch.zeros(N + 1, dtype=torch.int32, device=d)
    rowptr[1:] = torch.cumsum(torch.bincount(rows, minlength=N), 0).to(torch.int32)
    g = torch.Generator().manual_seed(seed)
    a = torch.rand(6, generator=g, dtype=torch.float64).tolist()
    if transpose:
        b = torch.randn(N, generator=g, dtype=torch.float64).to(d)
        return rowptr, cols[order].to(torch.int32), vals[order].contiguous(), b
    b = torch.where(inner, torch.zeros_like(x), a[0] + torch.sin((1 + a[1]) * 4 * x / m + 6 * a[2])
                    * torch.cos((1 + a[3]) * 4 * y / m + 6 * a[4]))
    return rowptr, cols[order].to(torch.int32), vals[order].contiguous(), b.contiguous()


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # one product with C: what a caller's own iteration does with the system of 3,844 circles
        {"name": "spmv", "kind": "spmv", "m": 62, "n": 16, "transpose": False},
        # the smallest solve, 4 x 4 circles: nothing but latency
        {"name": "solve_small", "kind": "krylov", "m": 4, "n": 16, "call": "solve_csr", "transpose": False},
        # the adjoint's solve with C^T, at about the size of the variable-coefficient cover
        {"name": "solve_transposed", "kind": "krylov", "m": 32, "n": 32, "call": "solve_csr", "transpose": True},
        # a Schur update of the 48 x 64 disk grid's factorisation, for 16 disks
        {"name": "gemm", "kind": "gemm", "batch": 16, "M": 1536, "N": 1536, "K": 1536},
        # the uneven cover of the unit disk: 7,108 circles, 127 thousand knots
        {"name": "cover", "kind": "cover", "geometry": "disk", "size": 16, "paths_max": 0, "se_target": 0.0},
        # the smallest whole call: 4 x 4 circles in the default all-FP64 form
        {"name": "tiny_fp64", "kind": "system", "geometry": "lattice", "size": 4, "spacing": 0.25, "n_r": 16,
         "n_theta": 16, "paths": 1000, "h": 1e-4, "precision": "fp64", "precond": "none"},
        # variable coefficients, 1,003 circles, in the mixed form, the solve preconditioned by RAS
        {"name": "varcoef_mixed", "kind": "system", "geometry": "hex", "size": 28, "paths": 10000, "h": 1e-5,
         "precision": "mixed", "precond": "ras"},
        # the same problem on a smaller domain in the all-FP64 form
        {"name": "varcoef_fp64", "kind": "system", "geometry": "hex", "size": 10, "paths": 10000, "h": 1e-5,
         "precision": "fp64", "precond": "ras"},
        # the benchmark's workload: 3,844 circles, 3,600 floating disks of 48 x 64 nodes
        {"name": "scaled_mixed", "kind": "system", "geometry": "lattice", "size": 62, "spacing": 4.0 / 62.0,
         "n_r": 48, "n_theta": 64, "paths": 1000, "h": 1e-5, "precision": "mixed", "precond": "ras"},
        # the paper's Poisson test on [-50, 50]^2: control variate and boundary shift
        {"name": "poisson46_mixed", "kind": "system", "geometry": "poisson46", "size": 10, "paths": 5000,
         "h": 0.015, "precision": "mixed", "precond": "ras"},
        # uneven circles, killing rate from 64 Gaussians, path counts by standard error
        {"name": "adaptive_mixed", "kind": "system", "geometry": "disk", "size": 11, "paths": 1000, "h": 1e-5,
         "paths_max": 20000, "se_target": 4e-3, "precision": "mixed", "precond": "none"},
        # a training step: u at the parameters, and the gradients of 64 + 16 + 32 of them
        {"name": "gradient", "kind": "gradient", "geometry": "lattice", "size": 4, "spacing": 0.25, "n_r": 16,
         "n_theta": 16, "paths": 1000, "h": 1e-4, "precision": "fp64"},
    ]


def _log(rng, a, b):
    """An integer in [a, b], even over its logarithm."""
    return min(b, max(a, int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))))


def draw(rng):
    kind = rng.choice(["spmv", "krylov", "gemm", "cover", "system", "system", "system", "system", "gradient"])
    if kind == "spmv":
        return {"kind": kind, "m": _log(rng, 4, 60), "n": rng.choice([16, 32, 44]), "transpose": rng.random() < 0.5}
    if kind == "krylov":
        call = rng.choice(["solve_csr", "solve_csr", "solve_csr_noalloc"])
        return {"kind": kind, "m": _log(rng, 5, 50), "n": rng.choice([16, 32]), "call": call,
                "transpose": call == "solve_csr" and rng.random() < 0.4}
    if kind == "gemm":
        return {"kind": kind, "batch": _log(rng, 1, 16), "M": _log(rng, 20, 1536), "N": _log(rng, 20, 1536),
                "K": _log(rng, 16, 1536)}
    if kind == "cover":
        if rng.random() < 0.5:
            return {"kind": kind, "geometry": "disk", "size": rng.randint(5, 16), "paths_max": 0, "se_target": 0.0}
        return {"kind": kind, "geometry": "hex", "size": _log(rng, 6, 100), "rows": rng.choice(["farthest", "averaged"])}
    if kind == "gradient":
        return {"kind": kind, "geometry": "lattice", "size": 4, "spacing": 0.25, "n_r": rng.randint(10, 16),
                "n_theta": 2 * rng.randint(8, 10), "paths": _log(rng, 200, 1000), "h": 1e-4,
                "precision": rng.choice(["fp64", "mixed"])}
    geometry = rng.choice(["lattice", "hex", "hex", "poisson46", "disk"])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    case = {"kind": kind, "geometry": geometry, "precision": precision, "precond": rng.choice(["none", "ras"])}
    if geometry == "lattice":
        if precision == "mixed":
            return case | {"size": _log(rng, 4, 40), "spacing": 4.0 / 62.0, "n_r": rng.randint(16, 48),
                           "n_theta": 2 * rng.randint(8, 32), "paths": _log(rng, 300, 1500), "h": 1e-5}
        return case | {"size": _log(rng, 4, 12), "spacing": 0.25, "n_r": rng.randint(10, 24),
                       "n_theta": 2 * rng.randint(8, 16), "paths": _log(rng, 300, 1500), "h": 1e-4}
    if geometry == "hex":
        rows = rng.choice(["farthest", "averaged"])
        return case | {"size": _log(rng, 6, 28 if precision == "mixed" else 9), "paths": _log(rng, 500, 10000),
                       "h": 1e-5, "rows": rows} | ({"precond": "none"} if rows == "averaged" else {})
    if geometry == "poisson46":
        if precision == "fp64":
            return case | {"size": rng.randint(3, 4), "paths": _log(rng, 100, 300), "h": 0.05}
        return case | {"size": rng.randint(3, 12), "paths": _log(rng, 500, 5000), "h": 0.015}
    # (larger disks cut circles into arcs whose interpolation matrices are singular in working precision:
    # those rows of C, and the path counts set by their standard errors, are rounding noise)
    return case | {"size": rng.randint(5, 11), "paths": 1000, "h": 1e-5, "paths_max": _log(rng, 3000, 20000),
                   "se_target": 4e-3, "precision": "mixed", "precond": "none"}


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("spmv", "krylov"):
        rowptr, col, val, b = _interfacial_csr(case["m"], case["n"], seed, case["transpose"])
        return {"case": case, "csr": (rowptr, col, val), "b": b, "u": torch.empty_like(b)}
    if kind == "gemm":
        g = torch.Generator(device="cuda").manual_seed(seed)
        # rows of a row-equilibrated matrix: entries within 1, most of them small
        A, B = (torch.randn(case["batch"], r, c, generator=g, device="cuda").clamp_(-4, 4).mul_(0.25)
                for r, c in ((case["M"], case["K"]), (case["K"], case["N"])))
        return {"case": case, "A": A, "B": B, "C": torch.empty(case["batch"], case["M"], case["N"], device="cuda")}
    cfg = _config(case, seed)
    if kind == "cover":
        return {"case": case, "cfg": cfg}
    if kind == "system":
        return {"case": case, "cfg": cfg, "cover": pdd.Cover(cfg)}
    rng = np.random.default_rng([seed, 1])
    box = cfg["domain"]["p"]
    cfg["op"] = {"b": "zero", "c": "rbf", "f": "rbf", "g": "boundary_fourier", "rbf": _rbf(rng, 64, 0.2, box, True),
                 "frbf": _rbf(rng, 16, 0.25, box, False), "g_coef": _boundary_fourier(box)}
    a = pdd.Cover(cfg).arrays()
    noise = torch.as_tensor(rng.normal(0.0, 1e-2, a["kx"].numel()), device="cuda")
    par = [torch.as_tensor(p, dtype=torch.float64, device="cuda")
           for p in (cfg["op"]["rbf"]["w"], cfg["op"]["g_coef"], 0.5 * cfg["op"]["frbf"]["w"])]
    return {"case": case, "cfg": cfg, "par": par, "obs": torch.exp(a["kx"]) * torch.sin(a["ky"]) + noise}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "spmv":
        return pdd.spmv_csr(*state["csr"], state["b"], transpose=case["transpose"])
    if kind == "krylov":
        if case["call"] == "solve_csr_noalloc":
            pdd.solve_csr_noalloc(*state["csr"], state["b"], state["u"])
            return state["u"]
        return pdd.solve_csr(*state["csr"], state["b"], transpose=case["transpose"])[0]
    if kind == "gemm":
        return pdd.gemm_tf32x3(state["C"], state["A"], state["B"], subtract=False)
    if kind == "cover":
        return pdd.Cover(state["cfg"]).arrays()
    if kind == "system":
        s = pdd.System(state["cover"], state["cfg"], case["precision"])
        u = s.solve(precond=case["precond"])
        return {"u": u, **s.csr()}
    w, a, v = (p.detach().requires_grad_() for p in state["par"])
    u = pdd.MisfitSolve.apply(w, a, state["cfg"], case["precision"], v)
    ((u - state["obs"]) ** 2).sum().backward()
    return {"u": u.detach(), "w": w.grad, "a": a.grad, "v": v.grad}


# ---------------------------------------------------------------------------
# what a pass cannot do without, and what it computes in 64 bits
# ---------------------------------------------------------------------------
def _geometry_work(case):
    """(disks, unknowns and right-hand sides of a disk, Monte Carlo rows, steps of a path, rows, stencil)."""
    geo, m = case["geometry"], case["size"]
    k = KNOTS.get(geo, 24)
    if geo == "lattice":
        r, c, per, n = 0.8 * case["spacing"], m * m, 4 * m - 4, case["n_r"] * case["n_theta"]
    elif geo == "hex":
        r, c, per, n = 0.05, int(1.155 * (m + 1) ** 2), int(4.9 * m), 1024
    elif geo == "poisson46":
        r, c, per, n = 9.0, m * m, 4 * m - 4, 968
    else:
        r, c, per, n = 0.03, int(7108 * (m / 16.0) ** 2), int(967 * m / 16.0), 600
    floating = max(0, c - per)
    steps = 0.25 * r * r / case.get("h", 1e-4)
    rows = c * k
    return floating, n, k + 1, int(0.7 * per * k), steps, rows, k


def work(case):
    kind = case["kind"]
    if kind in ("spmv", "krylov"):
        N = case["m"] ** 2 * case["n"]
        nnz = N * (case["n"] + 1)
        products = 1 if kind == "spmv" else 2 * case["m"] + 10       # iterations grow with the lattice
        return {"bytes": products * (12 * nnz + 20 * N), "flops": products * 2 * nnz}
    if kind == "gemm":
        b, M, N, K = case["batch"], case["M"], case["N"], case["K"]
        return {"bytes": 4 * b * (M * K + K * N + M * N), "flops": 2 * b * M * N * K}
    disks, n, nrhs, mc, steps, rows, k = _geometry_work(case)
    if kind == "cover":
        return {"bytes": rows * (4 * (k + 1) + 45), "flops": rows * 100}
    paths = mc * case["paths"] * steps
    if case["geometry"] == "disk":
        paths *= 15                                                  # reruns to the error target
        per_step = 150 + 64 * 8
    elif kind == "gradient":
        per_step = 150 + 2 * 80 * 25
    else:
        per_step = 150
    flops = disks * (2.0 / 3.0 * n ** 3 + 4.0 * n * n * nrhs) + paths * per_step
    bytes_ = rows * (k + 1) * 20 + rows * 40 + disks * n * 8.0 * nrhs
    return {"bytes": bytes_, "flops": flops}


def exact(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        s = prepare(case, seed)
        return torch.matmul(s["A"].double(), s["B"].double())
    if kind not in ("spmv", "krylov"):
        return None                      # Monte Carlo estimates and what follows from them
    N = case["m"] ** 2 * case["n"]
    rowptr, col, val, b = _interfacial_csr(case["m"], case["n"], seed, case["transpose"])
    C = torch.sparse_csr_tensor(rowptr.long(), col.long(), val, (N, N))
    if kind == "spmv":
        if not case["transpose"]:
            return torch.mv(C, b)
        row = torch.repeat_interleave(torch.arange(N, device="cuda"), torch.diff(rowptr).long())
        return torch.zeros_like(b).index_add_(0, col.long(), val * b[row])
    if N > 41000:
        return None
    # float32 factors of the dense matrix, refined with float64 residuals until they stop shrinking
    At = C.t() if case["transpose"] else C
    lu, piv = torch.linalg.lu_factor(C.to(torch.float32).to_dense().T if case["transpose"]
                                     else C.to(torch.float32).to_dense())
    x = torch.zeros_like(b)
    for _ in range(8):
        r = (b - torch.sparse.mm(At, x[:, None])[:, 0])
        x = x + torch.linalg.lu_solve(lu, piv, r.to(torch.float32)[:, None])[:, 0].double()
    return x
