"""Workloads for timing the library through its public Python calls.

A case is a plain dict: `op` names the call sequence, the other entries its
sizes and options.  The operators are built here on the GPU from a seed:

* fd   7-point finite differences on the unit cube, homogeneous Dirichlet
       data, A = -Lap_h - k^2 (1 + 0.05i) I (the small boxes and the
       frequency sweep of the workloads package);
* fe   linear elements on a jittered tetrahedral mesh of a bar with
       impedance ends, 15 entries per row: real away from the ends without
       damping, complex with it (the cylinder operators);
* hex  trilinear hexahedra with a material that varies by cell, damping and
       impedance walls, 27 entries per row, every value complex (the
       car-cabin operators).

The wavenumber of a solve is a few wavelengths per domain, where the
preconditioner-free methods converge in a number of iterations that hardly
moves with rounding.
"""

import math

import torch

import paper_2112_06465_gb300 as hz

C128 = torch.complex128


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


# ------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest calls: BLAS-1 on a short vector, where launches count
        {"name": "blas1_1e3", "op": "blas1", "n": 1000},
        # BLAS-1 near the top of the length sweep of the benchmark
        {"name": "blas1_3e7", "op": "blas1", "n": 31622777},
        # one product with a finite-element operator of the benchmark's size,
        # real except at its impedance ends
        {"name": "spmv_fe_real", "op": "spmv", "grid": "fe", "nx": 59, "ny": 60, "nz": 168, "damping": 0.0},
        # one product with a hexahedral operator of the car cabin's size
        {"name": "spmv_hex", "op": "spmv", "grid": "hex", "nx": 70, "ny": 51, "nz": 181, "damping": 0.05},
        # the complex64 product, the inner operator of the mixed solver
        {"name": "cspmv_fe", "op": "cspmv", "grid": "fe", "nx": 59, "ny": 60, "nz": 168, "damping": 0.05},
        # the smallest solve in use: a 16^3 box
        {"name": "solve_box16", "op": "solve", "grid": "fd", "nx": 16, "k": 5.0, "mode": "fp64", "method": "bicgstab"},
        # an ordinary solve: the largest box of the frequency sweep
        {"name": "solve_box64", "op": "solve", "grid": "fd", "nx": 64, "k": 5.0, "mode": "fp64", "method": "bicgstab"},
        # a large finite-element solve, with the method that solves most of
        # the finite-element systems of the frequency sweep
        {"name": "solve_fe", "op": "solve", "grid": "fe", "nx": 84, "ny": 83, "nz": 85, "damping": 0.05, "k": 2.0,
         "mode": "fp64", "method": "tfqmr"},
        # the mixed-precision solver on a middle-sized box
        {"name": "mixed_box48", "op": "solve", "grid": "fd", "nx": 48, "k": 5.0, "mode": "mixed",
         "method": "bicgstab"},
        # one optimisation step of the inverse problem: the forward and the
        # adjoint solve with the gradients of the parameters and the source
        {"name": "adjoint_32", "op": "adjoint", "nx": 32, "k": 8.0},
        # a frequency sweep in one persistent launch, systems of uneven size
        {"name": "sweep_batched", "op": "sweep", "nx": 24, "systems": 12, "mode": "fp64"},
        # new parameters written into an operator and the gradient of its
        # stored values and of the parameters, without the solves
        {"name": "gradient_64", "op": "gradient", "nx": 64},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _bar(rng, lo, hi, aspect=3.0):
    """Cells of a bar about aspect times as long as wide, lo..hi nodes, uneven sides."""
    n = _log(rng, lo, hi)
    w = max(4, int(round((n / aspect) ** (1.0 / 3.0))))
    nx, ny = w + rng.randrange(-1, 2), w + rng.randrange(-1, 2)
    return nx, ny, max(4, n // ((nx + 1) * (ny + 1)) - 1)


def draw(rng):
    op = rng.choice(["blas1", "spmv", "spmv", "cspmv", "solve", "solve", "mixed", "adjoint", "sweep", "gradient"])
    if op == "blas1":
        return {"op": op, "n": _log(rng, 1000, 30000000)}
    if op in ("spmv", "cspmv"):
        grid = rng.choice(["fd", "fe", "fe", "hex"])
        c = {"op": op, "grid": grid, "damping": rng.choice([0.0, 0.05])}
        if grid == "fd":
            c["nx"] = _log(rng, 8, 80)
        else:
            c["nx"], c["ny"], c["nz"] = _bar(rng, 2000, 500000 if grid == "hex" else 600000)
        return c
    if op in ("solve", "mixed"):
        # BiCGStab on the finite-element operators takes a number of
        # iterations that moves with rounding by a tenth: TFQMR there
        c = {"op": "solve", "grid": "fd" if op == "mixed" else rng.choice(["fd", "fd", "fe"]),
             "k": round(rng.uniform(2.0, 5.0), 3), "mode": "mixed" if op == "mixed" else "fp64", "method": "bicgstab"}
        if c["grid"] == "fd":
            c["nx"] = _log(rng, 8, 64)
            if op == "solve":
                c["method"] = rng.choice(["bicgstab", "bicgstab", "tfqmr", "bicgstabl"])
        else:
            c["nx"], c["ny"], c["nz"] = _bar(rng, 2000, 400000, 1.0)
            c["damping"] = 0.05
            c["k"] = round(0.5 * c["k"], 3)
            c["method"] = "tfqmr"
        return c
    if op == "adjoint":
        return {"op": op, "nx": _log(rng, 8, 32), "k": round(rng.uniform(3.0, 8.0), 3)}
    if op == "sweep":
        return {"op": op, "nx": _log(rng, 10, 24), "systems": rng.randrange(3, 13),
                "mode": rng.choice(["fp64", "mixed"])}
    return {"op": "gradient", "nx": _log(rng, 8, 64)}


# --------------------------------------------------------------- operators
def _gen(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed) * 7919 + 13)
    return g


def _cnormal(g, n, dtype=C128):
    v = torch.randn(2, n, generator=g, device=_device(), dtype=torch.float64) * math.sqrt(0.5)
    return torch.complex(v[0], v[1]).to(dtype).contiguous()


def _csr(shape, offsets, val):
    """CSR arrays of a stencil: shape = nodes per direction (slowest first),
    val[s] = the entries towards offsets[s]; neighbours outside are dropped."""
    d0, d1, d2 = shape
    dev = val.device
    i, j, k = (torch.arange(d, device=dev) for d in shape)
    keep, col = [], []
    node = (i[:, None, None] * d1 + j[None, :, None]) * d2 + k[None, None, :]
    for a, b, c in offsets:
        ok = (((i + a >= 0) & (i + a < d0))[:, None, None] & ((j + b >= 0) & (j + b < d1))[None, :, None]
              & ((k + c >= 0) & (k + c < d2))[None, None, :])
        keep.append(ok.reshape(-1))
        col.append((node + ((a * d1 + b) * d2 + c)).reshape(-1))
    keep = torch.stack(keep, 1)
    col = torch.stack(col, 1)[keep].to(torch.int32).contiguous()
    rowptr = torch.zeros(d0 * d1 * d2 + 1, dtype=torch.int64, device=dev)
    rowptr[1:] = torch.cumsum(keep.sum(1), 0)
    vals = val.reshape(len(offsets), -1).t()[keep].contiguous()
    return rowptr.to(torch.int32), col, vals


def _sorted_offsets(offsets):
    return sorted(offsets)


_FD_OFFSETS = [(-1, 0, 0), (0, -1, 0), (0, 0, -1), (0, 0, 0), (0, 0, 1), (0, 1, 0), (1, 0, 0)]


def _fd(m, diag):
    """-Lap_h on the m^3 interior grid of the unit cube plus diag on the diagonal."""
    h2 = float(m + 1) ** 2
    val = torch.full((7, m * m * m), -h2, dtype=C128, device=diag.device)
    val[3] = 6.0 * h2 + diag
    return _csr((m, m, m), _FD_OFFSETS, val)


# the six tetrahedra of a cube along the axis permutations, and the edges of
# the mesh they make (15 offsets)
_PERMS = [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]


def _tet(perm):
    v = [[0, 0, 0]]
    for d in perm:
        v.append(list(v[-1]))
        v[-1][d] = 1
    return [tuple(q) for q in v]


_FE_OFFSETS = _sorted_offsets({tuple(q - p for p, q in zip(a, b)) for t in map(_tet, _PERMS) for a in t for b in t})


def _at(o, cells):
    return tuple(slice(p, p + c) for p, c in zip(o, cells))


def _fe(nx, ny, nz, k, damping, g):
    """Linear tetrahedra on a jittered nx x ny x nz bar (cross-section 1 x ny/nx,
    impedance condition on the two end faces): real and imaginary parts of
    K - k^2 (1 + i damping) M - i k B, one array per neighbour."""
    dev = _device()
    cells, nodes = (nz, ny, nx), (nz + 1, ny + 1, nx + 1)
    h = 1.0 / nx
    axes = [torch.arange(d, device=dev, dtype=torch.float64) * h for d in nodes]
    xyz = torch.stack(torch.meshgrid(*axes, indexing="ij"))
    u = (torch.rand(xyz.shape, generator=g, device=dev, dtype=torch.float64) - 0.5) * (0.4 * h)
    u[:, 0], u[:, -1] = 0.0, 0.0
    u[:, :, 0], u[:, :, -1], u[:, :, :, 0], u[:, :, :, -1] = 0.0, 0.0, 0.0, 0.0
    xyz = xyz + u
    at = {o: n for n, o in enumerate(_FE_OFFSETS)}
    K = torch.zeros((15,) + nodes, dtype=torch.float64, device=dev)
    M, B = torch.zeros_like(K), torch.zeros_like(K)
    for perm in _PERMS:
        o = _tet(perm)
        p = [xyz[(slice(None),) + _at(q, cells)] for q in o]
        e = [p[q] - p[0] for q in (1, 2, 3)]
        cr = [torch.linalg.cross(e[1], e[2], dim=0), torch.linalg.cross(e[2], e[0], dim=0),
              torch.linalg.cross(e[0], e[1], dim=0)]
        det = (e[0] * cr[0]).sum(0)
        grad = [c / det for c in cr]
        grad.insert(0, -(grad[0] + grad[1] + grad[2]))
        vol = det.abs() / 6.0
        for a in range(4):
            for b in range(4):
                s = at[tuple(q - r for r, q in zip(o[a], o[b]))]
                rows = (s,) + _at(o[a], cells)
                K[rows] += vol * (grad[a] * grad[b]).sum(0)
                M[rows] += vol * ((2.0 if a == b else 1.0) / 20.0)
    for z in (0, nz):
        for tri in ([(0, 0), (1, 0), (1, 1)], [(0, 0), (0, 1), (1, 1)]):
            for a in tri:
                for b in tri:
                    s = at[(0, b[0] - a[0], b[1] - a[1])]
                    B[s, z, a[0]:a[0] + ny, a[1]:a[1] + nx] += h * h / 2.0 * ((2.0 if a == b else 1.0) / 12.0)
    val = torch.complex(K - (k * k) * M, -(k * k * damping) * M - k * B)
    return nodes, _FE_OFFSETS, val


_M1 = ((1.0 / 3.0, 1.0 / 6.0), (1.0 / 6.0, 1.0 / 3.0))
_K1 = ((1.0, -1.0), (-1.0, 1.0))
_HEX_OFFSETS = [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)]


def _hex(nx, ny, nz, k, damping, g):
    """Trilinear cubes with a material factor in [0.8, 1.2] per cube,
    impedance on the two end faces: K - k^2 (1 + i damping) M - i k B."""
    dev = _device()
    cells, nodes = (nz, ny, nx), (nz + 1, ny + 1, nx + 1)
    h = 1.0 / nx
    rho = 0.8 + 0.4 * torch.rand(cells, generator=g, device=dev, dtype=torch.float64)
    re = torch.zeros((27,) + nodes, dtype=torch.float64, device=dev)
    im = torch.zeros_like(re)
    corner = [(a, b, c) for a in (0, 1) for b in (0, 1) for c in (0, 1)]
    for p in corner:
        for q in corner:
            m = [_M1[p[d]][q[d]] for d in range(3)]
            s = [_K1[p[d]][q[d]] for d in range(3)]
            ke = h * (s[0] * m[1] * m[2] + m[0] * s[1] * m[2] + m[0] * m[1] * s[2])
            me = h ** 3 * m[0] * m[1] * m[2]
            rows = (_HEX_OFFSETS.index(tuple(b - a for a, b in zip(p, q))),) + _at(p, cells)
            re[rows] += ke - (k * k * me) * rho
            im[rows] -= (k * k * damping * me) * rho
    for z in (0, nz):
        for a in [(b, c) for b in (0, 1) for c in (0, 1)]:
            for b in [(b, c) for b in (0, 1) for c in (0, 1)]:
                s = _HEX_OFFSETS.index((0, b[0] - a[0], b[1] - a[1]))
                im[s, z, a[0]:a[0] + ny, a[1]:a[1] + nx] -= k * h * h * _M1[a[0]][b[0]] * _M1[a[1]][b[1]]
    return nodes, _HEX_OFFSETS, torch.complex(re, im)


def _operator(c, g):
    """CSR arrays (int32, int32, complex128) of a case's operator."""
    k, damping = c.get("k", 20.0), c.get("damping", 0.05)
    if c["grid"] == "fd":
        m = c["nx"]
        shift = torch.full((m ** 3,), complex(-k * k, -k * k * damping), dtype=C128, device=_device())
        return _fd(m, shift)
    return _csr(*(_fe if c["grid"] == "fe" else _hex)(c["nx"], c["ny"], c["nz"], k, damping, g))


def _theta(m, g):
    """Smooth complex field 1 + 0.2 f on the m^3 grid, |f| <= 1, from a few low modes."""
    dev = _device()
    t = torch.arange(1, m + 1, device=dev, dtype=torch.float64) / (m + 1)
    f = torch.zeros(m, m, m, dtype=C128, device=dev)
    a = _cnormal(g, 27).reshape(3, 3, 3)
    w = [torch.cos(math.pi * q * t) for q in range(3)]
    for i in range(3):
        for j in range(3):
            for l in range(3):
                f = f + a[i, j, l] * (w[i][:, None, None] * w[j][None, :, None] * w[l][None, None, :])
    f = f.reshape(-1)
    return (1.0 + 0.2 * f / f.abs().max()).contiguous()


def _sweep_sizes(c):
    """(grid points per side, wavenumber) of the systems of a sweep: sizes from
    half of nx to nx, wavenumbers from 2 to 5."""
    ns, nx = c["systems"], c["nx"]
    return [(nx - (nx // 2) * (s % 4) // 4, 2.0 + 3.0 * s / max(1, ns - 1)) for s in range(ns)]


# -------------------------------------------------------------- one case
# the adjoint's tolerance, for TFQMR, whose stopping test bounds the residual;
# the other methods stop at it, and their solutions settle a little below
TOL_TFQMR, TOL = 1e-12, 2e-13


def prepare(case, seed):
    c, g = case, _gen(seed)
    st = {"case": c}
    if c["op"] == "blas1":
        n = c["n"]
        st["x"], st["y"] = _cnormal(g, n), _cnormal(g, n)
        st["a"], st["b"] = _cnormal(g, 1), _cnormal(g, 1)
        st["w"] = torch.empty_like(st["x"])
        return st
    if c["op"] in ("spmv", "cspmv", "solve"):
        rowptr, col, val = _operator(c, g)
        st["A"] = hz.Matrix(rowptr, col, val, c64=c["op"] == "cspmv" or c.get("mode") == "mixed")
        st["x"] = _cnormal(g, rowptr.numel() - 1, torch.complex64 if c["op"] == "cspmv" else C128)
        return st
    if c["op"] == "sweep":
        st["A"], st["b"] = [], []
        for m, k in _sweep_sizes(c):
            r = _operator({"grid": "fd", "nx": m, "k": k}, g)
            st["A"].append(hz.Matrix(*r, c64=c["mode"] == "mixed"))
            st["b"].append(_cnormal(g, m ** 3))
        return st
    # adjoint, gradient: A(theta) = -Lap_h - kappa^2 diag(theta)
    m = c["nx"]
    k = c.get("k", 0.5 * (m + 1))
    st["theta"] = _theta(m, g)
    st["base"] = torch.full((m ** 3,), 6.0 * (m + 1) ** 2, dtype=C128, device=_device())
    st["scale"] = -k * k
    st["A"] = hz.Matrix(*_fd(m, -k * k * st["theta"]))
    st["b"], st["g"] = _cnormal(g, m ** 3), _cnormal(g, m ** 3)
    if c["op"] == "adjoint":
        st["theta"].requires_grad_(True)
        st["b"].requires_grad_(True)
    else:
        # a parameter update small enough to be one of many
        st["theta2"] = (st["theta"] + 1e-3 * _cnormal(g, m ** 3)).contiguous()
    return st


def run(st):
    c = st["case"]
    if c["op"] == "blas1":
        # one vector update of a Krylov method, call by call
        w = hz.zcopy(st["y"], st["w"])
        hz.zaxpy(st["a"], st["x"], w)
        hz.zscal(st["b"], w)
        return [w, hz.zdotc(st["x"], w), hz.dznrm2(w)]
    if c["op"] == "spmv":
        return hz.zspmv(st["A"], st["x"])
    if c["op"] == "cspmv":
        return hz.cspmv(st["A"], st["x"])
    if c["op"] == "solve":
        tol = TOL_TFQMR if c["method"] == "tfqmr" else TOL
        x, info = hz.zsolve(st["A"], st["x"], tol=tol, maxit=4000, mode=c["mode"], method=c["method"])
        return x
    if c["op"] == "sweep":
        xs, infos = hz.zsolve_batched(st["A"], st["b"], tol=TOL, maxit=4000, mode=c["mode"])
        return xs
    if c["op"] == "adjoint":
        x = hz.solve_diag_param(st["theta"], st["b"], st["A"], st["base"], st["scale"], tol=TOL_TFQMR,
                                maxit=4000, method="tfqmr")
        gt, gb = torch.autograd.grad(x, (st["theta"], st["b"]), grad_outputs=st["g"])
        return [x.detach(), gt, gb]
    A = st["A"]
    hz.mat_set_diag(A, st["base"], st["scale"], st["theta2"])
    y = hz.zspmv(A, st["b"])
    gv = hz.outer_on_pattern(A, st["g"], y)
    return [y, gv, hz.diag_grad(A, st["g"], y, st["scale"])]


# ------------------------------------------------------------------- work
def _nodes(c):
    return c["nx"] ** 3 if c["grid"] == "fd" else (c["nx"] + 1) * (c["ny"] + 1) * (c["nz"] + 1)


def _row(c):
    return {"fd": 7, "fe": 15, "hex": 27}[c["grid"]]


def _iterations(m, fe=False):
    """Roughly the iterations that a grid of m points along its longest side
    takes to the tolerances below at these wavenumbers (two products each)."""
    return (11.0 if fe else 4.2) * m + 10


def work(case):
    """Bytes and operations a pass cannot do without.  A solve reads its
    operator once per product as long as it does not fit on the chip; here
    each input is counted once, and the operations of all iterations."""
    c = case
    if c["op"] == "blas1":   # five calls, each with its own operands
        return {"bytes": (32 + 48 + 32 + 32 + 16) * c["n"], "flops": (8 + 6 + 8 + 4) * c["n"]}
    if c["op"] in ("spmv", "cspmv"):
        n, half = _nodes(c), 2 if c["op"] == "cspmv" else 1
        real = c["op"] == "spmv" and c["grid"] != "hex" and not c["damping"]
        nnz = n * _row(c)
        return {"bytes": nnz * (4 + 16 // half) + n * (4 + 32 // half), "flops": nnz * (4 if real else 8)}
    if c["op"] == "solve":
        n = _nodes(c)
        it = _iterations(c["nx"], c["grid"] == "fe")
        return {"bytes": n * (_row(c) * 20 + 36), "flops": it * n * (2 * 8 * _row(c) + 84)}
    if c["op"] == "sweep":
        return {"bytes": sum(m ** 3 * (7 * 20 + 36) for m, _ in _sweep_sizes(c)),
                "flops": sum(_iterations(m) * m ** 3 * (2 * 8 * 7 + 84) for m, _ in _sweep_sizes(c))}
    n = c["nx"] ** 3
    if c["op"] == "adjoint":
        return {"bytes": n * (7 * 20 + 7 * 16), "flops": 2 * _iterations(c["nx"]) * n * (2 * 8 * 7 + 100)}
    return {"bytes": n * (7 * 20 + 7 * 16 + 7 * 16 + 6 * 16), "flops": n * (7 * 8 + 7 * 6 + 30)}


# ------------------------------------------------------------------ exact
def _dense_rows(rowptr, col, val):
    """The operator with every row padded to the longest one."""
    n = rowptr.numel() - 1
    rp = rowptr.to(torch.int64)
    length = rp[1:] - rp[:-1]
    w = int(length.max())
    pos = rp[:-1, None] + torch.arange(w, device=col.device)[None]
    ok = torch.arange(w, device=col.device)[None] < length[:, None]
    pos = torch.where(ok, pos, torch.zeros_like(pos))
    v = torch.where(ok, val[pos], torch.zeros((), dtype=val.dtype, device=val.device))
    return torch.where(ok, col[pos].to(torch.int64), torch.zeros_like(pos)).t().contiguous(), v.t().contiguous()


def _apply(E, x):
    c, v = E
    y = v[0] * x[c[0]]
    for s in range(1, c.shape[0]):
        y = y + v[s] * x[c[s]]
    return y


def _solve(E, b, tol=1e-13):
    """Plain BiCGStab with refinement steps until the residual stands at tol."""
    x, nb = torch.zeros_like(b), torch.linalg.vector_norm(b)
    for _ in range(6):
        r = b - _apply(E, x)
        if float(torch.linalg.vector_norm(r) / nb) <= tol:
            break
        rh, d = r.clone(), torch.zeros_like(b)
        p, v = torch.zeros_like(b), torch.zeros_like(b)
        rho = alpha = omega = torch.ones((), dtype=b.dtype, device=b.device)
        first = float(torch.linalg.vector_norm(r))
        for it in range(1500):
            rho1 = torch.vdot(rh, r)
            p = r + (rho1 / rho) * (alpha / omega) * (p - omega * v)
            v = _apply(E, p)
            alpha = rho1 / torch.vdot(rh, v)
            s = r - alpha * v
            t = _apply(E, s)
            omega = torch.vdot(t, s) / torch.vdot(t, t)
            d = d + alpha * p + omega * s
            r, rho = s - omega * t, rho1
            if it % 8 == 7 and float(torch.linalg.vector_norm(r)) <= max(1e-9 * first, 0.1 * tol * float(nb)):
                break
        x = x + d
    return x


def _sine_solve(m, shift, b):
    """(-Lap_h - shift)^{-1} b by the sine transform of the grid."""
    j = torch.arange(1, m + 1, device=b.device, dtype=torch.float64)
    h = 1.0 / (m + 1)
    V = (math.sqrt(2 * h) * torch.sin(math.pi * h * torch.outer(j, j))).to(C128)
    lam = (4.0 / (h * h)) * torch.sin(j * (math.pi * h / 2.0)) ** 2

    def transform(t):
        t = torch.einsum("ai,ijk->ajk", V, t)
        t = torch.einsum("bj,ajk->abk", V, t)
        return torch.einsum("ck,abk->abc", V, t)

    f = transform(b.reshape(m, m, m))
    f = f / (lam[:, None, None] + lam[None, :, None] + lam[None, None, :] - shift)
    return transform(f).reshape(-1)


def exact(case, seed):
    c, g = case, _gen(seed)
    if c["op"] == "blas1":
        x, y = _cnormal(g, c["n"]), _cnormal(g, c["n"])
        a, b = _cnormal(g, 1), _cnormal(g, 1)
        w = b * (y + a * x)
        return [w, torch.vdot(x, w).reshape(1), torch.linalg.vector_norm(w).reshape(1)]
    if c["op"] in ("spmv", "cspmv", "solve"):
        rowptr, col, val = _operator(c, g)
        n = rowptr.numel() - 1
        if c["op"] == "cspmv":
            val = val.to(torch.complex64).to(C128)
            return _apply(_dense_rows(rowptr, col, val), _cnormal(g, n, torch.complex64).to(C128))
        x = _cnormal(g, n)
        if c["op"] == "solve" and c["grid"] == "fd":
            return _sine_solve(c["nx"], complex(c["k"] ** 2, 0.05 * c["k"] ** 2), x)
        E = _dense_rows(rowptr, col, val)
        return _solve(E, x) if c["op"] == "solve" else _apply(E, x)
    if c["op"] == "sweep":
        return [_sine_solve(m, complex(k * k, 0.05 * k * k), _cnormal(g, m ** 3)) for m, k in _sweep_sizes(c)]
    m = c["nx"]
    k = c.get("k", 0.5 * (m + 1))
    theta = _theta(m, g)
    b, gr = _cnormal(g, m ** 3), _cnormal(g, m ** 3)
    if c["op"] == "adjoint":
        E = _dense_rows(*_fd(m, -k * k * theta))
        x, mu = _solve(E, b), _solve(E, gr.conj().resolve_conj())
        return [x, k * k * (mu * x).conj().resolve_conj(), mu.conj().resolve_conj()]
    theta = theta + 1e-3 * _cnormal(g, m ** 3)
    rowptr, col, val = _fd(m, -k * k * theta)
    y = _apply(_dense_rows(rowptr, col, val), b)
    rows = torch.repeat_interleave(torch.arange(m ** 3, device=b.device), (rowptr[1:] - rowptr[:-1]).to(torch.int64))
    gv = -(gr[rows] * y[col.to(torch.int64)]).conj().resolve_conj()
    return [y, gv, k * k * (gr * y).conj().resolve_conj()]
