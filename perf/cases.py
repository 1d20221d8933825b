"""What the library is measured on: filter applications and eigensolves as a user's program
calls them, over the meshes and options of this repository's workloads.

Every matrix is a P1 finite-element pencil S v = omega^2 M v on a voxel domain split into Kuhn
simplices (7 couplings per row in 2D, 15 in 3D), numbered lexicographically, with the mass
lumped and Dirichlet nodes eliminated, like the meshes of the workloads. The medium is
anisotropic and its stiffness and density vary from cell to cell with the seed, so that no
coupling vanishes and no two rows need be alike. Start vectors are N(0,1). The time step is 0.9
of the stable one by Gershgorin's bound.
"""
import itertools
import math

import numpy as np
import torch

import paper_2402_08515_gb300 as K

# cells of the boxes of a batch, h = 1/64 (30 thousand .. 857 thousand dofs)
BATCH = [(32, 32, 32), (40, 40, 40), (48, 40, 32), (48, 48, 48), (56, 48, 40), (64, 48, 48),
         (64, 64, 64), (72, 64, 56), (80, 64, 64), (80, 80, 80), (88, 80, 72), (96, 96, 96)]


def listed():
    return [
        # the smallest workload: a 2D square, 3,969 dofs, one filter application; every step is a few
        # microseconds of work at most, so launches and latency decide
        dict(name="filter_square64_fp64", do="filter", domain="box", nx=64, ny=64, nz=0, h=1 / 64, prec="fp64",
             b=1, F=1, L=300, wmin=20.0, wmax=30.0),
        # a small anisotropic box with odd edges (22 thousand dofs) in the FP32 form
        dict(name="filter_box37x29x23_fp32", do="filter", domain="box", nx=37, ny=29, nz=23, h=1 / 32, prec="fp32",
             b=1, F=1, L=600, wmin=10.0, wmax=14.0),
        # a mid-size cube (250 thousand dofs) with the fourth-order stepper; its matrix stays in L2
        dict(name="filter_cube64_fp64_leapfrog4", do="filter", domain="box", nx=64, ny=64, nz=64, h=1 / 64,
             prec="fp64", b=1, F=1, L=300, wmin=10.0, wmax=14.0, stepper="leapfrog4"),
        # the headline: the unit cube of 128^3 cells (2,048,383 dofs), plain FP64
        dict(name="filter_cube128_fp64", do="filter", domain="box", nx=128, ny=128, nz=128, h=1 / 128, prec="fp64",
             b=1, F=1, L=600, wmin=40.0, wmax=45.0),
        # the same cube in the FP32 form
        dict(name="filter_cube128_fp32", do="filter", domain="box", nx=128, ny=128, nz=128, h=1 / 128, prec="fp32",
             b=1, F=1, L=600, wmin=40.0, wmax=45.0),
        # blocks of 8 start vectors in FP64, as the block solver filters them
        dict(name="filter_box96_fp64_b8", do="filter", domain="box", nx=96, ny=96, nz=96, h=1 / 64, prec="fp64",
             b=8, F=1, L=150, wmin=20.0, wmax=24.0),
        # 12 uneven boxes in one context (3.1 million dofs), 8 columns: 4 intervals of 2 columns each
        dict(name="columns_batch12_fp32_b8", do="columns", domain="batch", first=0, count=12, prec="fp32", b=8, F=4,
             L=300, wmin=10.0, wmax=22.0),
        # a flared tube, the shape of the horn workload: ragged lines of nodes, Neumann walls, column
        # distances past 16 bits, blocks of 8 in the FP32 form
        dict(name="filter_tube_fp32_b8", do="filter", domain="tube", h=2.8e-3, prec="fp32", b=8, F=1, L=100,
             wmin=20.0, wmax=26.0),
        # whole eigensolves: the 2D square (latency of everything between the filters too),
        dict(name="solve_square64_fp64", do="solve", domain="box", nx=64, ny=64, nz=0, h=1 / 64, prec="fp64", b=1,
             F=1, L=300, wmin=20.0, wmax=30.0, kmax=40, tol=1e-8, sweeps=0),
        # a 3D cube of 250 thousand dofs with every accepted vector returned,
        dict(name="solve_cube64_fp64", do="solve", domain="box", nx=64, ny=64, nz=64, h=1 / 64, prec="fp64", b=1,
             F=1, L=600, wmin=10.0, wmax=14.0, kmax=60, tol=1e-8, sweeps=0),
        # and a batch of meshes in the FP32 block form, two intervals each, refined in FP32 pairs to 1e-8
        dict(name="solve_batch3_fp32_b8", do="solve", domain="batch", first=0, count=3, prec="fp32", b=8, F=2, L=600,
             wmin=10.0, wmax=14.0, kmax=48, tol=1e-8, sweeps=1),
        # the entry point for programs that allocate nothing after start-up, on their own CSR arrays
        dict(name="noalloc_cube48_fp64", do="noalloc", domain="box", nx=48, ny=48, nz=48, h=1 / 48, prec="fp64", b=1,
             F=1, L=300, wmin=10.0, wmax=14.0),
    ]


def draw(rng):
    """One more case: boxes, squares, tubes and batches of 500 to 2 million dofs, every width,
    precision and stepper, L from 30 to 600."""
    kind = rng.choice(["filter"] * 6 + ["columns"] * 2 + ["noalloc", "solve"])
    prec = rng.choice(["fp64", "fp32"])
    case = dict(do=kind, prec=prec)
    top = {"filter": 2.0e6, "columns": 1.0e6, "noalloc": 5.0e5, "solve": 1.0e5}[kind]
    n = math.exp(rng.uniform(math.log(500.0), math.log(top)))
    shape = rng.choice(["box"] * 5 + ["square", "tube"] + (["batch"] if kind != "noalloc" else []))
    if shape == "square" and n < 4.0e5:
        nx = max(8, int(math.sqrt(n) * math.exp(rng.uniform(-0.4, 0.4))))
        case.update(domain="box", nx=nx, ny=max(8, int(n / nx)), nz=0, h=1.0 / nx)
    elif shape == "tube" and n > 2.0e4:
        case.update(domain="tube", h=4.4e-3 * (1.0e6 / n) ** (1 / 3))
    elif shape == "batch" and n > 2.0e5:
        first = rng.randrange(0, 6)
        case.update(domain="batch", first=first, count=rng.randrange(2, 4))
    else:
        e = n ** (1 / 3)
        nx = max(7, int(e * math.exp(rng.uniform(-0.4, 0.4))))
        ny = max(6, int(e * math.exp(rng.uniform(-0.4, 0.4))))
        case.update(domain="box", nx=nx, ny=ny, nz=max(5, int(n / (nx * ny))), h=1.0 / nx)
    w0 = rng.uniform(5.0, 30.0)
    case.update(wmin=w0, wmax=w0 + rng.uniform(2.0, 8.0), b=1, F=1, L=rng.randrange(30, 601))
    if kind == "filter":
        case["b"] = rng.choice([1, 1, 1, 2, 3, 4, 5, 8])
        case["F"] = rng.choice([1, 1, 1, 2, 4])
        case["stepper"] = rng.choice(["leapfrog"] * 4 + ["leapfrog4"])
        case["sigma"] = rng.choice([1, 1, 1, 256])
    elif kind == "columns":
        case["F"], case["b"] = rng.choice([(1, 2), (2, 4), (2, 8), (4, 8), (3, 6)])
    elif kind == "noalloc":
        case["prec"] = "fp64"
    else:
        case["b"] = rng.choice([1, 1, 2, 8]) if case["domain"] != "batch" else 4
        case.update(kmax=rng.randrange(16, 49), tol=1e-8 if prec == "fp64" else 1e-4, sweeps=0)
    case["L"] = max(30, min(case["L"], int(1.2e9 / (n * case["b"] * max(1, case.get("kmax", 1) // case["b"])))))
    return case


# ------------------------------------------------------------------ the pencil

def _cell(dim, h):
    """Stiffness (2^d x 2^d, anisotropic medium), lumped mass and coupling pattern of one cell."""
    metric = np.array([[1.0, 0.25, 0.1], [0.25, 1.0, 0.15], [0.1, 0.15, 1.0]])[:dim, :dim]
    nc = 1 << dim
    S, m, pat = np.zeros((nc, nc)), np.zeros(nc), np.zeros((nc, nc), dtype=bool)
    for perm in itertools.permutations(range(dim)):
        at, corners = 0, [0]
        for axis in perm:
            at |= 1 << axis
            corners.append(at)
        x = np.array([[(c >> a) & 1 for a in range(dim)] for c in corners]) * h
        edges = (x[1:] - x[0]).T
        vol = abs(np.linalg.det(edges)) / math.factorial(dim)
        inv = np.linalg.inv(edges)
        grad = np.vstack([-inv.sum(axis=0), inv])
        loc = vol * grad @ metric @ grad.T
        for i, ci in enumerate(corners):
            m[ci] += vol / (dim + 1)
            for j, cj in enumerate(corners):
                S[ci, cj] += loc[i, j]
                pat[ci, cj] = True
    return S, m, pat


def _mesh(cells, h, present, dirichlet, seed):
    """CSR of S and the diagonal of M (host arrays) of a voxel domain; arrays are (z, y, x)."""
    dev = torch.device("cuda")
    dim = len(cells)
    gen = torch.Generator(device=dev).manual_seed(seed)
    stiff = torch.exp(0.3 * torch.randn(cells, generator=gen, device=dev, dtype=torch.float64))
    dens = torch.exp(0.2 * torch.randn(cells, generator=gen, device=dev, dtype=torch.float64))
    if present is not None:
        stiff, dens = stiff * present, dens * present
    S, mass, pat = _cell(dim, h)
    nodes = tuple(c + 1 for c in cells)
    bits = [[(c >> a) & 1 for a in reversed(range(dim))] for c in range(1 << dim)]  # corner -> array offsets
    m = torch.zeros(nodes, device=dev, dtype=torch.float64)
    used = torch.zeros(nodes, device=dev, dtype=torch.bool)
    window = lambda o: tuple(slice(o[a], o[a] + cells[a]) for a in range(dim))  # noqa: E731
    for c, o in enumerate(bits):
        m[window(o)] += mass[c] * dens
        used[window(o)] |= True if present is None else present
    free = used & ~dirichlet
    number = (torch.cumsum(free.reshape(-1).to(torch.int64), 0) - 1).reshape(nodes)
    n = int(free.sum())
    stride = [1] * dim
    for a in reversed(range(dim - 1)):
        stride[a] = stride[a + 1] * nodes[a + 1]
    offs = sorted({tuple(bits[j][a] - bits[i][a] for a in range(dim)) for i in range(1 << dim)
                   for j in range(1 << dim) if pat[i, j]}, key=lambda o: sum(o[a] * stride[a] for a in range(dim)))
    at = free.reshape(-1).nonzero().reshape(-1)
    val = torch.empty(n, len(offs), device=dev, dtype=torch.float64)
    has = torch.empty(n, len(offs), device=dev, dtype=torch.bool)
    col = torch.empty(n, len(offs), device=dev, dtype=torch.int32)
    for q, o in enumerate(offs):
        v = torch.zeros(nodes, device=dev, dtype=torch.float64)
        there = torch.zeros(nodes, device=dev, dtype=torch.bool)
        for i, bi in enumerate(bits):
            bj = tuple(bi[a] + o[a] for a in range(dim))
            if bj not in map(tuple, bits) or not pat[i, bits.index(list(bj))]:
                continue
            v[window(bi)] += S[i, bits.index(list(bj))] * stiff
            there[window(bi)] |= True if present is None else present
        far = (at + sum(o[a] * stride[a] for a in range(dim))).clamp_(0, free.numel() - 1)
        val[:, q] = v.reshape(-1)[at]
        has[:, q] = there.reshape(-1)[at] & free.reshape(-1)[far]
        col[:, q] = number.reshape(-1)[far].to(torch.int32)
    m = m.reshape(-1)[at]
    top = ((val.abs() * has).sum(dim=1) / m).max()
    row_ptr = torch.zeros(n + 1, device=dev, dtype=torch.int64)
    row_ptr[1:] = torch.cumsum(has.sum(dim=1), 0)
    return Pencil(n, row_ptr.cpu().numpy(), col[has].cpu().numpy(), val[has].cpu().numpy(), m.cpu().numpy(),
                  math.sqrt(float(top)))


class Pencil:
    def __init__(self, n, row_ptr, col, val, m, omega_bound):
        self.n, self.row_ptr, self.col, self.val, self.m, self.omega_bound = n, row_ptr, col, val, m, omega_bound


def _box(cells, h, seed):
    shape = tuple(c for c in reversed(cells) if c > 0)
    wall = torch.ones(tuple(c + 1 for c in shape), device="cuda", dtype=torch.bool)
    wall[tuple(slice(1, -1) for _ in shape)] = False
    return _mesh(shape, h, None, wall, seed)


def _tube(h, seed):
    """Radius 0.02 exp(3 x) over x in [0, 1]: Dirichlet at x = 0, natural condition elsewhere."""
    nx, ny = int(round(1.0 / h)), int(math.ceil(0.04 * math.exp(3.0) / h))
    x = (torch.arange(nx, device="cuda", dtype=torch.float64) + 0.5) * h
    y = (torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5) * h - ny * h / 2
    present = y[:, None, None] ** 2 + y[None, :, None] ** 2 <= (0.02 * torch.exp(3.0 * x)[None, None, :]) ** 2
    mouth = torch.zeros((ny + 1, ny + 1, nx + 1), device="cuda", dtype=torch.bool)
    mouth[:, :, 0] = True
    return _mesh((ny, ny, nx), h, present, mouth, seed)


def _meshes(case, seed):
    if case["domain"] == "batch":
        return [_box(c, 1 / 64, 100 * seed + j) for j, c in
                enumerate(BATCH[case["first"]:case["first"] + case["count"]])]
    if case["domain"] == "tube":
        return [_tube(case["h"], seed)]
    return [_box((case["nx"], case["ny"], case["nz"]), case["h"], seed)]


def _bands(case):
    """F neighbouring intervals that cover [wmin, wmax]."""
    edge = [case["wmin"] + (case["wmax"] - case["wmin"]) * f / case["F"] for f in range(case["F"] + 1)]
    return edge[:-1], edge[1:]


def _tau(case, p):
    return 0.9 * (2 * math.sqrt(3.0) if case.get("stepper") == "leapfrog4" else 2.0) / p.omega_bound


def _start(case, seed, n):
    gen = torch.Generator(device="cuda").manual_seed(7919 + seed)
    return torch.randn(case["b"], n, generator=gen, device="cuda", dtype=torch.float64)


# ------------------------------------------------------------------ a pass

def _stream():
    """The one stream that the program gives its contexts: its passes run one after the other."""
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


_streams = []


def prepare(case, seed):
    torch.cuda.set_device(0)
    meshes = _meshes(case, seed)
    n = sum(p.n for p in meshes)
    r = _start(case, seed, n)
    s = dict(case=case, r=r)
    if case["do"] == "noalloc":
        p, tau = meshes[0], _tau(case, meshes[0])
        s.update(n=n, row_ptr=torch.from_numpy(p.row_ptr).cuda(), col=torch.from_numpy(p.col).cuda(),
                 val=torch.from_numpy(p.val).cuda(), tau2m=torch.from_numpy(tau * tau / p.m).cuda(),
                 alpha=torch.from_numpy(K.kes_alpha_table(case["wmin"], case["wmax"], tau, case["L"])).cuda(),
                 out=torch.empty(n, device="cuda", dtype=torch.float64))
        return s
    torch.cuda.current_stream().synchronize()  # r is read on the library's stream
    ctx = K.Context(meshes if case["domain"] == "batch" else meshes[0], precision=case["prec"], block_b=case["b"],
                    stepper=case.get("stepper", "leapfrog"), sell_sigma=case.get("sigma", 1), stream=_stream())
    lo, hi = _bands(case)
    K.kes_set_filters_batch(ctx.handle, [lo] * len(meshes), [hi] * len(meshes), [_tau(case, p) for p in meshes],
                            case["L"])
    s["ctx"] = ctx
    if case["do"] == "filter":
        s["out"] = torch.empty(case["F"], case["b"], n, device="cuda", dtype=torch.float64)
    elif case["do"] == "columns":
        s["out"] = torch.empty(case["b"], n, device="cuda", dtype=torch.float64)
    else:
        o = K.kes_solve_opts_default()
        o.kmax, o.tol, o.check_every, o.want_vectors = case["kmax"], case["tol"], 16, 1
        o.refine_sweeps = case["sweeps"]
        o.refine_precision = K.KES_REFINE_F32X2 if case["sweeps"] else K.KES_REFINE_FP64
        # the program's own arrays of results, for as many pairs as the bases could hold
        most = case["kmax"] * case["F"]
        s["opts"], s["pairs"] = o, [{**{k: np.full(most, np.nan) for k in ("omega2", "rel_res", "interval")},
                                     "vectors": np.zeros((most, p.n))} for p in meshes]
    return s


def run(s):
    do, case = s["case"]["do"], s["case"]
    if do == "filter":
        K.kes_filter_apply(s["ctx"].handle, s["r"], s["out"], case["b"])
        return s["out"]
    if do == "columns":
        K.kes_filter_apply_columns(s["ctx"].handle, s["r"], s["out"], case["b"])
        return s["out"]
    if do == "noalloc":
        K.kes_filter_apply_noalloc(s["n"], s["row_ptr"], s["col"], s["val"], s["tau2m"], s["alpha"], case["L"],
                                   s["r"][0], s["out"])
        return s["out"]
    if case["b"] == 1 and case["F"] == 1 and case["domain"] != "batch":
        found = [K.kes_krylov_solve(s["ctx"].handle, s["r"], s["opts"])]
    else:
        found = K.kes_block_krylov_solve(s["ctx"].handle, s["r"], case["b"], s["opts"])
    for own, f in zip(s["pairs"], found):
        for k, a in own.items():
            if f["n_pairs"]:
                a[:f["n_pairs"]] = f[k]
    return [{**own, "ritz_omega2": f["ritz_omega2"], "ritz_rel_res": f["ritz_rel_res"]}
            for own, f in zip(s["pairs"], found)]


# ------------------------------------------------------------------ what a pass needs

def _rows(case):
    """Rows and stored entries, from the sizes alone (tubes: from the volume)."""
    if case["domain"] == "batch":
        boxes = BATCH[case["first"]:case["first"] + case["count"]]
    elif case["domain"] == "tube":
        n = 0.0843 / case["h"] ** 3
        return n, 15 * n
    else:
        boxes = [(case["nx"], case["ny"], case["nz"])]
    n = sum(math.prod(c - 1 for c in b if c > 0) for b in boxes)
    return n, n * (7 if boxes[0][2] == 0 else 15)


def work(case):
    """One step reads each value of the matrix (8 or 4 bytes; a column can be had for less than the
    value's size, so none is counted) and u_n and u_(n-1), and writes u_(n+1); its 2 FLOP per entry
    and column, 2 for the recurrence, and 2 per weighted term. A fourth-order step has two products. A
    solve filters kmax - b / F times a block and orthogonalises twice against the basis."""
    n, nnz = _rows(case)
    size = 8 if case["prec"] == "fp64" else 4
    b, F, products = case["b"], case["F"], 2 if case.get("stepper") == "leapfrog4" else 1
    terms = F if case["do"] == "filter" else 1
    bytes_, flops = size * (products * nnz + 3 * n * b), b * (products * 2 * nnz + 2 * n + 2 * n * terms)
    steps, g = case["L"], b // F if case["do"] == "solve" else 1
    if case["do"] != "solve":
        outs = b * F if case["do"] == "filter" else b
        return dict(bytes=steps * bytes_ + 8 * n * (b + outs), flops=steps * flops)
    blocks, k = -(-(case["kmax"] - g) // g), case["kmax"]
    return dict(bytes=blocks * steps * bytes_ + 4 * 8 * n * F * k * k / 2,
                flops=blocks * steps * flops + 4 * 2 * n * F * k * k / 2)


def _weights(wmin, wmax, tau, L):
    """alpha_n = tau (4 / (pi t)) sin(t (wmax - wmin) / 2) cos(t (wmax + wmin) / 2), t = n tau."""
    t = tau * np.arange(1, L + 1)
    first = tau * 2.0 * (wmax - wmin) / math.pi
    return np.concatenate([[first], tau * 4.0 / (math.pi * t) * np.sin(0.5 * t * (wmax - wmin))
                           * np.cos(0.5 * t * (wmax + wmin))])


def exact(case, seed):
    """The filter sum in 64 bits with torch's own sparse product; None for the solves, whose
    unconverged Ritz values have no value that rounding leaves alone."""
    if case["do"] == "solve":
        return None
    meshes = _meshes(case, seed)
    r = _start(case, seed, sum(p.n for p in meshes))
    lo, hi = _bands(case)
    parts, at = [], 0
    for p in meshes:
        tau = _tau(case, p)
        alpha = np.stack([_weights(a, c, tau, case["L"]) for a, c in zip(lo, hi)])  # F x (L + 1)
        S = torch.sparse_csr_tensor(torch.from_numpy(p.row_ptr).cuda(), torch.from_numpy(p.col).cuda().long(),
                                    torch.from_numpy(p.val).cuda(), size=(p.n, p.n))
        t2m = torch.from_numpy(tau * tau / p.m).cuda()[:, None]
        u = r[:, at:at + p.n].t().contiguous()
        at += p.n
        if case["do"] == "columns":  # column j has the weights of interval j // (b / F)
            own = torch.from_numpy(alpha[[j // (case["b"] // case["F"]) for j in range(case["b"])]]).cuda()
            weigh = lambda k, v: own[None, :, k] * v  # noqa: E731
        else:
            own = torch.from_numpy(alpha).cuda()
            weigh = lambda k, v: own[:, k, None, None] * v  # noqa: E731
        prev, acc = u, weigh(0, u)
        for k in range(1, case["L"] + 1):
            step = t2m * (S @ u)
            if case.get("stepper") == "leapfrog4":
                step = step - t2m * (S @ step) / 12.0
            prev, u = u, 2.0 * u - prev - step
            acc = acc + weigh(k, u)
        parts.append(acc.transpose(-1, -2))
    out = torch.cat(parts, dim=-1)
    return out[0, 0] if case["do"] == "noalloc" else out.contiguous()
