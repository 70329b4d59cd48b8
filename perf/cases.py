"""Workloads of the thermoelastic solver, each one call (or one short chain of
calls) through paper_1804_10060_gb300.thermoamg as a user's program makes it.

listed()  the named workloads; draw(rng) one more of the same ranges;
prepare() the meshes, fields, handles and weights a program holds before the
call; run() the call; work() the bytes and operations it cannot do without;
exact() the same results in 64 bits from plain torch (own element integrals,
own assembly, Jacobi-preconditioned Krylov solves), None where there is none.

Meshes come from the package's seeded generators (meshgen); a seed moves the
interior vertices, the fields, the network weights and the rows.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1804_10060_gb300 import meshgen
from paper_1804_10060_gb300 import thermoamg as tam

EDGES = ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))
EXACT_NODES = 100_000  # the largest mesh whose elastic solve exact() repeats


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest whole solve a program asks for (the README's and smoke()'s
        # unit cube, 3,993 DOF) through the one-call host-buffer entry point:
        # copies in, assembly, hierarchy, CG, copy out; bound by latency
        {"name": "host_solve_cube10", "kind": "host_solve", "n": 10, "degree": 1},
        # one application of the preconditioner on a 56k-DOF box: what a program
        # that brings its own Krylov method calls; every level is small
        {"name": "vcycle_box64", "kind": "vcycle", "nx": 64, "ny": 16, "nz": 16, "degree": 1},
        # assembly of the benchmark's 3.26M-DOF two-material box (6.29M linear cells)
        {"name": "assemble_box256", "kind": "assemble", "nx": 256, "ny": 64, "nz": 64, "degree": 1},
        # assembly on quadratic cells (1.39M DOF, the box of the many-load-case study)
        {"name": "assemble_box96_p2", "kind": "assemble", "nx": 96, "ny": 24, "nz": 24, "degree": 2},
        # the multigrid hierarchy of the benchmark's box
        {"name": "setup_box256", "kind": "setup", "nx": 256, "ny": 64, "nz": 64, "degree": 1},
        # the benchmark's solve: FP64 AMG-PCG to 1e-8 from zero
        {"name": "solve_box256", "kind": "solve", "mesh": "box", "nx": 256, "ny": 64, "nz": 64, "degree": 1,
         "precision": 0},
        # a bladed turbine disc of quadratic cells (1.38M DOF) solved with the FP32 hierarchy
        {"name": "solve_disc48_p2_fp32", "kind": "solve", "mesh": "disc", "blades": 48, "theta": 4, "rings": 49,
         "layers": 5, "blade_layers": 8, "degree": 2, "precision": 1},
        # many load cases: eight right-hand sides on each of three meshes of the
        # many-load-case study in one call
        {"name": "batch_3_meshes_8_rhs", "kind": "batch", "meshes": "64x16x16p1,32x8x8p2,128x32x32p1", "n_rhs": 8},
        # the learned guess's network in FP32 on the nodes of a 1.4M-DOF disc
        {"name": "mlp_forward_fp32", "kind": "mlp_forward", "rows": 468864, "width": 128, "depth": 3, "bf16": 0},
        # the same network in BF16 on the 11.6M nodes of the 34.8M-DOF disc
        {"name": "mlp_forward_bf16", "kind": "mlp_forward", "rows": 11606400, "width": 128, "depth": 3, "bf16": 1},
        # one training batch of the network (the training loop's 32,768 rows): loss and gradient
        {"name": "mlp_grad", "kind": "mlp_grad", "rows": 32768, "width": 128, "depth": 3},
        # one implicit heating step of the transient disc (460k unknowns, quadratic
        # cells): Newton with the hierarchy kept between steps
        {"name": "newton_disc48_p2", "kind": "newton", "blades": 48, "theta": 4, "rings": 49, "layers": 5,
         "blade_layers": 8, "degree": 2, "dt": 0.005},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, lo, hi):
    """Hexes of a box about four times as long as wide, odd sizes among them."""
    ny = _log_int(rng, lo, hi)
    nz = max(2, min(hi, ny + rng.randint(-2, 2)))
    nx = max(2, min(4 * hi, int(ny * rng.uniform(2.0, 4.0))))
    return {"nx": nx, "ny": ny, "nz": nz}


def _disc(rng, blades_hi):
    blades = rng.randint(9, blades_hi)
    dth = 2.0 * math.pi / (4 * blades)
    return {"blades": blades, "theta": 4, "rings": max(3, int(round(math.log(5.0) / dth))),
            "layers": max(2, int(round(0.1 / (0.6 * dth)))), "blade_layers": max(1, int(round(math.log(1.3) / dth)))}


def draw(rng):
    kind = rng.choice(["host_solve", "vcycle", "assemble", "setup", "solve", "solve", "batch", "mlp_forward",
                       "mlp_forward", "mlp_grad", "newton"])
    degree = rng.choice([1, 2])
    if kind == "host_solve":
        return {"kind": kind, "n": rng.randint(4, 20 if degree == 1 else 10), "degree": degree}
    if kind == "vcycle":
        return {"kind": kind, **_box(rng, 6, 40 if degree == 1 else 20), "degree": degree}
    if kind in ("assemble", "setup"):
        return {"kind": kind, **_box(rng, 6, 60 if degree == 1 else 24), "degree": degree}
    if kind == "solve":
        precision = rng.choice([0, 1])
        if rng.random() < 0.5:
            return {"kind": kind, "mesh": "box", **_box(rng, 8, 56 if degree == 1 else 22), "degree": degree,
                    "precision": precision}
        return {"kind": kind, "mesh": "disc", **_disc(rng, 40), "degree": degree, "precision": precision}
    if kind == "batch":
        specs = []
        for _ in range(rng.randint(1, 3)):
            p = rng.choice([1, 2])
            b = _box(rng, 6, 28 if p == 1 else 12)
            specs.append("%dx%dx%dp%d" % (b["nx"], b["ny"], b["nz"], p))
        return {"kind": kind, "meshes": ",".join(specs), "n_rhs": rng.randint(1, 16)}
    if kind == "newton":
        return {"kind": kind, **_disc(rng, 40), "degree": degree, "dt": math.exp(rng.uniform(math.log(1e-3), math.log(2e-2)))}
    width, depth = rng.choice([16, 33, 64, 96, 128]), rng.randint(1, 4)
    if kind == "mlp_grad":
        return {"kind": kind, "rows": _log_int(rng, 64, 60000), "width": width, "depth": min(depth, 3)}
    bf16 = rng.choice([0, 1])
    return {"kind": kind, "rows": _log_int(rng, 1, 8000000 if bf16 else 460000), "width": width, "depth": depth,
            "bf16": bf16}


# ---------------------------------------------------------------------------
# meshes and fields
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=6)
def _mesh(kind, *size):
    if kind == "cube":
        return meshgen.unit_cube_problem(size[0], degree=size[1])
    if kind == "box":
        return meshgen.slab_box_problem(*size[:3], degree=size[3])
    blades, theta, rings, layers, blade_layers, degree = size
    return meshgen.bladed_disc_problem(n_r=rings, n_theta_per_blade=theta, n_z=layers, n_blades=blades,
                                       n_r_blade=blade_layers, degree=degree, blade_fraction=0.5)


def _mesh_of(c):
    if c["kind"] == "host_solve":
        return _mesh("cube", c["n"], c["degree"])
    if c["kind"] == "newton" or c.get("mesh") == "disc":
        return _mesh("disc", c["blades"], c["theta"], c["rings"], c["layers"], c["blade_layers"], c["degree"])
    return _mesh("box", c["nx"], c["ny"], c["nz"], c["degree"])


@functools.lru_cache(maxsize=2)
def _thermal_mesh(*size):
    return meshgen.disc_thermal_problem(_mesh("disc", *size), t=0.03)


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _put(a, dt):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=dt)).to(_device())


def _cosines(X, seed, scale):
    """Mean of eight cosines with seeded wave vectors and phases (the generators' smooth field)."""
    rng = np.random.default_rng(seed)
    xt = X / torch.tensor(scale, dtype=torch.float64, device=X.device)
    out = torch.zeros(X.shape[0], dtype=torch.float64, device=X.device)
    n = 0
    while n < 8:
        k = rng.integers(0, 4, size=3)
        if not np.any(k != 0):
            continue
        arg = (xt * torch.tensor(k.astype(np.float64), device=X.device)).sum(1)
        out += torch.cos(np.pi * arg + float(rng.uniform(0.0, 2.0 * np.pi)))
        n += 1
    return out / 8


def _moved(coords, cells, seed):
    """Interior vertices (24 cells) moved by up to 5% of the shortest first edge; mid-edge nodes stay midpoints."""
    v = cells[:, :4].long()
    x = coords.clone()
    interior = torch.bincount(v.reshape(-1), minlength=x.shape[0]) == 24
    h = float((x[v[:, 1]] - x[v[:, 0]]).norm(dim=1).min())
    g = torch.Generator().manual_seed(int(seed))
    d = (torch.rand(x.shape, generator=g, dtype=torch.float64) - 0.5).to(x.device) * (0.1 * h)
    x[interior] += d[interior]
    if cells.shape[1] == 10:
        for k, (a, b) in enumerate(EDGES):
            x[cells[:, 4 + k].long()] = 0.5 * (x[v[:, a]] + x[v[:, b]])
    return x


def _load(pb, x, seed):
    """(T, body force or None) of one load case."""
    if pb.name.startswith("disc"):
        T = 300.0 + 500.0 * (x[:, 0] ** 2 + x[:, 1] ** 2) + 10.0 * _cosines(x, seed, (2.6, 2.6, 0.1))
    else:
        T = _cosines(x, seed, (4.0, 1.0, 1.0))
    omega = float(np.random.default_rng(seed + 77).uniform(0.0, 2.0))
    body = torch.cat([x[:, :2], torch.zeros_like(x[:, :1])], dim=1) * omega ** 2
    return T.contiguous(), body.contiguous()


def _problem(c, seed, pb=None):
    """The device tensors fem_assemble_elasticity takes."""
    pb = _mesh_of(c) if pb is None else pb
    cells = _put(pb.cells, np.int32)
    x = _moved(_put(pb.coords, np.float64), cells, seed)
    T, body = _load(pb, x, seed)
    return dict(coords=x, cells=cells, cell_material=_put(pb.cell_material, np.int32),
                mat_props=_put(pb.mat_props, np.float64), T=T, T_ref=pb.T_ref, body_force=body,
                dirichlet_mask=_put(pb.dirichlet_mask, np.uint8))


def _batch_meshes(c):
    out = []
    for s in c["meshes"].split(","):
        dims, p = s.split("p")
        out.append(_mesh("box", *[int(v) for v in dims.split("x")], int(p)))
    return out


def _batch_loads(c, i, pb, x, seed):
    return [_load(pb, x, seed + 1000 * (i + 1) + k) for k in range(c["n_rhs"])]


def _newton_problem(c, seed):
    tp = _thermal_mesh(c["blades"], c["theta"], c["rings"], c["layers"], c["blade_layers"], c["degree"])
    cells = _put(tp.cells, np.int32)
    x = _moved(_put(tp.coords, np.float64), cells, seed)
    r = torch.hypot(x[:, 0], x[:, 1])
    scale = (2.6, 2.6, 0.1)
    hot = 300.0 + 600.0 * (1.0 - math.exp(-0.06)) + 20.0 * _cosines(x, seed, scale)
    return dict(x=x, cells=cells, mat=_put(tp.cell_material, np.int32), props=tp.thermal_props,
                faces=_put(tp.faces, np.int32), beta=_put(tp.beta, np.float64),
                T_bc=torch.where(r > 0.5, hot, torch.full_like(hot, 300.0)).contiguous(),
                T_old=(310.0 + 10.0 * r + 10.0 * _cosines(x, seed + 1, scale)).contiguous())


def _network(c, seed):
    """(theta, shift, scale, out_scale, X, Y): Glorot weights, small biases, features and targets as the discs give them."""
    rng = np.random.default_rng(seed)
    dims = [8] + [c["width"]] * c["depth"] + [3]
    theta = []
    for a, b in zip(dims, dims[1:]):
        lim = math.sqrt(6.0 / (a + b))
        theta += [rng.uniform(-lim, lim, a * b), rng.uniform(-0.1, 0.1, b)]
    theta = np.concatenate(theta).astype(np.float32)
    g = torch.Generator(device=_device()).manual_seed(int(seed))
    # x, y, z, T, grad T, distance to the bore: their usual centres and spreads
    mean = np.array([0.0, 0.0, 0.0, 580.0, 0.0, 0.0, 0.0, 0.5], np.float32)
    std = np.array([0.55, 0.55, 0.03, 240.0, 550.0, 550.0, 60.0, 0.3], np.float32)
    n = c["rows"]
    X = torch.randn((n, 8), generator=g, device=_device()) * torch.from_numpy(std).to(_device()) + \
        torch.from_numpy(mean).to(_device())
    out_scale = np.array([2e-3, 2e-3, 4e-4], np.float32)
    Y = torch.randn((n, 3), generator=g, device=_device()) * torch.from_numpy(out_scale).to(_device()) \
        if c["kind"] == "mlp_grad" else None
    return dims, theta, mean, (1.0 / std).astype(np.float32), out_scale, X, Y


# ---------------------------------------------------------------------------
def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "host_solve":
        p = _problem(c, seed)
        host = {k: (v.cpu().pin_memory() if isinstance(v, torch.Tensor) else v) for k, v in p.items()}
        return dict(kind=kind, p=host)
    if kind in ("mlp_forward", "mlp_grad"):
        _, theta, shift, scale, out_scale, X, Y = _network(c, seed)
        net = tam.Mlp(8, c["width"], c["depth"], 3, seed=1)
        net.set_normalization(shift, scale, out_scale)
        net.set_params(theta)
        return dict(kind=kind, net=net, X=X, Y=Y, bf16=c.get("bf16", 0))
    if kind == "newton":
        p = _newton_problem(c, seed)
        th = tam.Thermal(p["x"], p["cells"], p["mat"], p["props"], p["faces"])
        return dict(kind=kind, th=th, dt=c["dt"], **{k: p[k] for k in ("beta", "T_bc", "T_old")})
    if kind == "batch":
        prm = tam.amg_params_default(level_precision=1)
        hs, bs = [], []
        for i, pb in enumerate(_batch_meshes(c)):
            p = _problem(c, seed, pb)
            K, _ = tam.fem_assemble_elasticity(**p)
            B = torch.empty((c["n_rhs"], 3 * pb.n_nodes), dtype=torch.float64, device="cuda")
            for k, (T, body) in enumerate(_batch_loads(c, i, pb, p["coords"], seed)):
                tam.fem_assemble_load(K, **dict(p, T=T, body_force=body), out=B[k])
            hs.append(tam.amg_setup(K, p["coords"], prm))
            bs.append(B)
        return dict(kind=kind, H=hs, B=bs)
    p = _problem(c, seed)
    if kind == "assemble":
        return dict(kind=kind, p=p)
    K, rhs = tam.fem_assemble_elasticity(**p)
    if kind == "setup":
        return dict(kind=kind, K=K, coords=p["coords"])
    H = tam.amg_setup(K, p["coords"], tam.amg_params_default(level_precision=c.get("precision", 0)))
    return dict(kind=kind, H=H, rhs=rhs)


def run(state):
    s, kind = state, state["kind"]
    if kind == "host_solve":
        return tam.tam_solve_elasticity_host(**s["p"])[0]
    if kind == "mlp_forward":
        return s["net"].forward(s["X"], bf16=s["bf16"])
    if kind == "mlp_grad":
        loss, grad = s["net"].loss_grad(s["X"], s["Y"])
        return {"loss": np.array(loss), "grad": grad}
    if kind == "newton":
        T = s["T_old"].clone()
        s["th"].newton(T, T_old=s["T_old"], dt=s["dt"], theta=1.0, beta=s["beta"], T_bc=s["T_bc"], rtol=1e-9,
                       lin_rtol=1e-8, reuse=1)
        return T
    if kind == "batch":
        X = [torch.zeros_like(B) for B in s["B"]]
        tam.amg_pcg_solve_batch(s["H"], s["B"], X, rtol=1e-8)
        return X
    if kind == "assemble":
        # the assembled matrix as a program that keeps its own copy reads it
        K, rhs = tam.fem_assemble_elasticity(**s["p"])
        row_ptr, col_idx, vals = tam.tam_matrix_export_bsr(K)
        return {"row_ptr": row_ptr, "col_idx": col_idx, "vals": vals, "rhs": rhs}
    if kind == "setup":
        # the hierarchy and its coarse operators and prolongators
        H = tam.amg_setup(s["K"], s["coords"])
        info = tam.amg_info(H)
        out = {"lambda": np.array(info["lambda"][:-1])}
        for l in range(1, info["n_levels"]):
            for name, level, which in (("A%d" % l, l, 0), ("P%d" % (l - 1), l - 1, 1)):
                e = tam.amg_level_export(H, level, which)
                out[name] = {k: e[k] for k in ("row_ptr", "col_idx", "vals")}
        return out
    if kind == "vcycle":
        return tam.amg_vcycle(s["H"], s["rhs"])
    x = torch.zeros_like(s["rhs"])
    tam.amg_pcg_solve(s["H"], s["rhs"], x, rtol=1e-8, max_iter=1000)
    return x


# ---------------------------------------------------------------------------
# bytes and operations
# ---------------------------------------------------------------------------
def _sizes(c, pb=None):
    """(nodes, cells, nodes per cell, 3x3 blocks of K) of a mesh; blocks per row of a Kuhn mesh's interior, less its surface's."""
    if pb is None and c["kind"] != "host_solve" and not (c["kind"] == "newton" or c.get("mesh") == "disc"):
        nx, ny, nz, p = c["nx"], c["ny"], c["nz"], c["degree"]
        n, m = (p * nx + 1) * (p * ny + 1) * (p * nz + 1), 6 * nx * ny * nz
    else:
        pb = _mesh_of(c) if pb is None else pb
        n, m, p = pb.n_nodes, pb.n_cells, 1 if pb.nodes_per_cell == 4 else 2
    npc = 4 if p == 1 else 10
    return n, m, npc, int(n * (14.0 if p == 1 else 27.0))


def work(case):
    """Inputs once, outputs once, and per operation the products its algorithm needs.

    Solves: K (76 bytes a block) five times an iteration -- the outer product
    and the four of a degree-2 smoothed V-cycle's finest level -- at the
    iteration counts these meshes take (about 25 on linear cells, 60 on
    quadratic ones); FP32 hierarchies read 40 bytes a block in the four."""
    c, kind = case, case["kind"]
    if kind in ("mlp_forward", "mlp_grad"):
        dims = [8] + [c["width"]] * c["depth"] + [3]
        macs = sum(a * b for a, b in zip(dims, dims[1:]))
        par = macs + sum(dims[1:])
        n = c["rows"]
        if kind == "mlp_forward":
            return {"bytes": 44 * n + 4 * par, "flops": 2 * macs * n}
        return {"bytes": 44 * n + 8 * par, "flops": (6 * macs - 2 * 8 * c["width"]) * n}
    if kind == "batch":
        b = f = 0
        for pb in _batch_meshes(c):
            n, m, npc, nnzb = _sizes(c, pb)
            it = 25 if npc == 4 else 45
            b += it * (76 * nnzb + 4 * 40 * nnzb + c["n_rhs"] * n * 24 * 10)
            f += it * 5 * 18 * nnzb * c["n_rhs"]
        return {"bytes": b, "flops": f}
    n, m, npc, nnzb = _sizes(c)
    asm_b = 24 * n + 4 * npc * m + 4 * m + 8 * n + 24 * n + n + 24 * n + 76 * nnzb
    asm_f = m * (16 * 27 if npc == 4 else 4 * 55 * 27)
    if kind == "assemble":
        return {"bytes": asm_b, "flops": asm_f}
    if kind == "setup":
        # K in, the coarse operators and prolongators out (about 0.6 and 0.5 of K's bytes)
        return {"bytes": 76 * nnzb * 2.1, "flops": 2 * nnzb * 300}
    if kind == "newton":
        # three Newton steps: assembly of the scalar Jacobian, about 20 CG iterations each
        return {"bytes": 3 * (44 * m + 12 * nnzb + 20 * 5 * 12 * nnzb), "flops": 3 * (m * 12000 + 20 * 10 * nnzb)}
    it = 25 if npc == 4 else 60
    if kind == "vcycle":
        return {"bytes": 4 * 76 * nnzb + 48 * n, "flops": 4 * 18 * nnzb}
    low = 40 if c.get("precision", 0) else 76
    solve = {"bytes": it * (76 + 4 * low) * nnzb, "flops": it * 5 * 18 * nnzb}
    if kind == "host_solve":
        return {"bytes": asm_b + 76 * nnzb * 2.1 + solve["bytes"], "flops": asm_f + 600 * nnzb + solve["flops"]}
    return solve


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _rule(n):
    """Collapsed Gauss-Legendre rule on the unit tetrahedron: barycentrics [q, 4], weights (sum 1); exact to degree 2 n - 3."""
    t, w = np.polynomial.legendre.leggauss(n)
    t, w = 0.5 * (t + 1.0), 0.5 * w
    a, b, z = (v.ravel() for v in np.meshgrid(t, t, t, indexing="ij"))
    wa, wb, wz = (v.ravel() for v in np.meshgrid(w, w, w, indexing="ij"))
    y = b * (1.0 - z)
    x = a * (1.0 - b) * (1.0 - z)
    W = 6.0 * wa * wb * wz * (1.0 - b) * (1.0 - z) ** 2
    return np.stack([1.0 - x - y - z, x, y, z], axis=1), W


def _basis(npc, L):
    """(phi [q, npc], dphi/dlambda [q, npc, 4]) at barycentric points L."""
    q = L.shape[0]
    if npc == 4:
        return L.copy(), np.broadcast_to(np.eye(4), (q, 4, 4)).copy()
    phi, d = np.zeros((q, 10)), np.zeros((q, 10, 4))
    for a in range(4):
        phi[:, a] = L[:, a] * (2.0 * L[:, a] - 1.0)
        d[:, a, a] = 4.0 * L[:, a] - 1.0
    for k, (a, b) in enumerate(EDGES):
        phi[:, 4 + k] = 4.0 * L[:, a] * L[:, b]
        d[:, 4 + k, a], d[:, 4 + k, b] = 4.0 * L[:, b], 4.0 * L[:, a]
    return phi, d


def _geometry(x, cells):
    v = x[cells[:, :4].long()]
    J = v[:, 1:] - v[:, :1]                                  # rows: edges
    vol = torch.linalg.det(J) / 6.0
    G = torch.linalg.inv(J).transpose(1, 2)                  # rows: gradients of lambda 1..3
    return torch.cat([-G.sum(1, keepdim=True), G], dim=1), vol


def _pattern(n, cells, free):
    """Sorted unique (row, column) keys of the free couplings and every diagonal."""
    c = cells.long()
    npc = c.shape[1]
    diag = torch.arange(n, device=c.device) * (n + 1)
    keys = [diag]
    for a in range(npc):
        for b in range(npc):
            ok = free[c[:, a]] & free[c[:, b]]
            keys.append((c[:, a] * n + c[:, b])[ok])
        keys = [torch.unique(torch.cat(keys))]
    keys = keys[0]
    rows = keys // n
    rp = torch.zeros(n + 1, dtype=torch.int64, device=c.device)
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return keys, rp, keys - rows * n


def _exact_system(p):
    """(row_ptr, col_idx, vals, rhs) of the elastic problem p (no prescribed displacements)."""
    x, cells = p["coords"], p["cells"]
    n, npc, dev = x.shape[0], cells.shape[1], x.device
    free = p["dirichlet_mask"] == 0
    keys, rp, ci = _pattern(n, cells, free)
    vals = torch.zeros((keys.numel(), 9), dtype=torch.float64, device=dev)
    rhs = torch.zeros((n, 3), dtype=torch.float64, device=dev)
    L, W = _rule(4)
    phi, dphi = (torch.from_numpy(v).to(dev) for v in _basis(npc, L))
    w = torch.from_numpy(W).to(dev)
    mass = torch.einsum("q,qa,qb->ab", w, phi, phi)
    stiff = torch.einsum("q,qak,qbl->abkl", w, dphi, dphi)   # on gradients of lambda
    therm = torch.einsum("q,qc,qak->cak", w, phi, dphi)
    E, nu, alpha = (p["mat_props"][:, k][p["cell_material"].long()] for k in range(3))
    mu = E / (2.0 * (1.0 + nu))
    lam = E * nu / ((1.0 + nu) * (1.0 - 2.0 * nu))
    eye = torch.eye(3, dtype=torch.float64, device=dev).reshape(9)
    step = 2_000_000 if npc == 4 else 100_000
    for s in range(0, cells.shape[0], step):
        cc = cells[s:s + step].long()
        g, vol = _geometry(x, cc)
        m_, l_ = mu[s:s + step] * vol, lam[s:s + step] * vol
        for a in range(npc):
            na = cc[:, a]
            for b in range(npc):
                nb = cc[:, b]
                D = torch.einsum("kl,mki,mlj->mij", stiff[a, b], g, g)
                k = l_[:, None] * D.reshape(-1, 9) + m_[:, None] * D.transpose(1, 2).reshape(-1, 9) + \
                    (m_ * torch.diagonal(D, dim1=1, dim2=2).sum(1))[:, None] * eye
                ok = free[na] & free[nb]
                vals.index_add_(0, torch.searchsorted(keys, (na * n + nb)[ok]), k[ok])
        kt = (3.0 * l_ + 2.0 * m_) * alpha[s:s + step]
        f = torch.einsum("mc,cak,mki->mai", p["T"][cc] - p["T_ref"], therm, g) * kt[:, None, None]
        f += torch.einsum("ab,mbi->mai", mass, p["body_force"][cc]) * vol[:, None, None]
        rhs.index_add_(0, cc.reshape(-1), f.reshape(-1, 3))
    fixed = torch.nonzero(~free).reshape(-1)
    vals[torch.searchsorted(keys, fixed * (n + 1))] = eye
    rhs[fixed] = 0.0
    return rp, ci, vals.reshape(-1, 3, 3), rhs


def _csr(rp, ci, vals):
    """Scalar CSR tensor of a block one."""
    n, b = rp.numel() - 1, vals.shape[1]
    cnt = rp[1:] - rp[:-1]
    row = torch.repeat_interleave(torch.arange(n, device=rp.device), cnt)
    k = torch.arange(ci.numel(), device=rp.device) - rp[row]
    i = torch.arange(b, device=rp.device)
    at = (b * b * rp[row] + b * k)[:, None, None] + (b * cnt[row])[:, None, None] * i[None, :, None] + i[None, None, :]
    v = torch.empty(ci.numel() * b * b, dtype=torch.float64, device=rp.device)
    col = torch.empty(v.numel(), dtype=torch.int64, device=rp.device)
    v[at.reshape(-1)] = vals.reshape(-1)
    col[at.reshape(-1)] = (b * ci[:, None, None] + i[None, None, :]).expand(-1, b, b).reshape(-1)
    crow = torch.zeros(n * b + 1, dtype=torch.int64, device=rp.device)
    crow[1:] = torch.cumsum((b * cnt).repeat_interleave(b), 0)
    return torch.sparse_csr_tensor(crow.int(), col.int(), v, size=(n * b, n * b))


def _block_diag_inv(rp, ci, vals):
    n = rp.numel() - 1
    row = torch.repeat_interleave(torch.arange(n, device=rp.device), rp[1:] - rp[:-1])
    return torch.linalg.inv(vals[row == ci])


def _cg(A, dinv, B, tol=1e-11, most=8000):
    """Block-Jacobi-preconditioned CG on A X = B for the columns of B; None when it does not get there."""
    pre = lambda R: torch.einsum("nij,njm->nim", dinv, R.reshape(dinv.shape[0], dinv.shape[1], -1)).reshape(R.shape)
    X, R = torch.zeros_like(B), B.clone()
    Z = pre(R)
    P, rz = Z.clone(), (R * Z).sum(0)
    nb = B.norm(dim=0)
    one = torch.ones_like(rz)
    for k in range(most):
        Q = A @ P
        a = rz / torch.where(rz > 0, (P * Q).sum(0), one)
        X += a * P
        R -= a * Q
        Z = pre(R)
        new = (R * Z).sum(0)
        P = Z + (new / torch.where(rz > 0, rz, one)) * P
        rz = new
        if k % 50 == 49 and bool((R.norm(dim=0) <= tol * nb).all()):
            return X
    return None


def _exact_newton(c, seed):
    """Backward-Euler heating step by Newton, T to the last bits (quadratic or linear cells)."""
    p = _newton_problem(c, seed)
    x, cells = p["x"], p["cells"].long()
    n, npc, dev = x.shape[0], cells.shape[1], x.device
    rho, c0, c1, k0, k1 = (float(v) for v in p["props"][0])
    dt = c["dt"]
    keys, rp, ci = _pattern(n, cells, torch.ones(n, dtype=torch.bool, device=dev))
    L, W = _rule(5)
    phi, dphi = (torch.from_numpy(v).to(dev) for v in _basis(npc, L))
    w = torch.from_numpy(W).to(dev)
    # faces: collapsed rule on the triangle
    t, tw = np.polynomial.legendre.leggauss(4)
    t, tw = 0.5 * (t + 1.0), 0.5 * tw
    fa, fb = (v.ravel() for v in np.meshgrid(t, t, indexing="ij"))
    m = np.stack([1.0 - fa * (1.0 - fb) - fb, fa * (1.0 - fb), fb], axis=1)
    fw = 2.0 * np.outer(tw, tw).ravel() * (1.0 - fb)
    fphi = m if npc == 4 else np.concatenate(
        [m * (2.0 * m - 1.0), np.stack([4.0 * m[:, i] * m[:, j] for i, j in ((0, 1), (1, 2), (2, 0))], axis=1)], axis=1)
    fmass = torch.from_numpy(np.einsum("q,qa,qb->ab", fw, fphi, fphi)).to(dev)
    faces = p["faces"].long()
    e1, e2 = x[faces[:, 1]] - x[faces[:, 0]], x[faces[:, 2]] - x[faces[:, 0]]
    fbw = p["beta"] * 0.5 * torch.linalg.cross(e1, e2).norm(dim=1)
    T, To = p["T_old"].clone(), p["T_old"]
    f0 = None
    for _ in range(12):
        F = torch.zeros(n, dtype=torch.float64, device=dev)
        J = torch.zeros(keys.numel(), dtype=torch.float64, device=dev)
        for s in range(0, cells.shape[0], 40_000):
            cc = cells[s:s + 40_000]
            g, vol = _geometry(x, cc)
            D = torch.einsum("qak,mki->mqai", dphi, g)
            Te, De = T[cc], (T[cc] - To[cc]) / dt
            Tq, Dq = Te @ phi.T, De @ phi.T
            gT = torch.einsum("ma,mqai->mqi", Te, D)
            wv = w[None, :] * vol[:, None]
            kq = (k0 + k1 * Tq) * wv
            mq = rho * wv
            dg = torch.einsum("mqai,mqi->mqa", D, gT)
            f = torch.einsum("mq,mqa->ma", kq, dg) + torch.einsum("mq,qa->ma", mq * (c0 + c1 * Tq) * Dq, phi)
            F.index_add_(0, cc.reshape(-1), f.reshape(-1))
            je = torch.einsum("mqai,mqbi->mab", D * kq[:, :, None, None], D)
            je += k1 * torch.einsum("mqa,qb->mab", dg * wv[:, :, None], phi)
            je += torch.einsum("mq,qa,qb->mab", mq * (c1 * Dq + (c0 + c1 * Tq) / dt), phi, phi)
            pos = torch.searchsorted(keys, (cc[:, :, None] * n + cc[:, None, :]).reshape(-1))
            J.index_add_(0, pos, je.reshape(-1))
        F.index_add_(0, faces.reshape(-1), -(fbw[:, None] * ((T[faces] - p["T_bc"][faces]) @ fmass)).reshape(-1))
        pos = torch.searchsorted(keys, (faces[:, :, None] * n + faces[:, None, :]).reshape(-1))
        J.index_add_(0, pos, -(fbw[:, None, None] * fmass).reshape(-1))
        f0 = F.norm() if f0 is None else f0
        if bool(F.norm() <= 1e-13 * f0):
            break
        # BiCGStab with the diagonal
        A = _csr(rp, ci, J.reshape(-1, 1, 1))
        row = torch.repeat_interleave(torch.arange(n, device=dev), rp[1:] - rp[:-1])
        di = 1.0 / J[row == ci]
        d, r = torch.zeros_like(F), F.clone()
        rs, pv, rho_o = r.clone(), r.clone(), r @ r
        for k in range(3000):
            ph = di * pv
            v = A @ ph
            al = rho_o / (rs @ v)
            sv = r - al * v
            sh = di * sv
            tv = A @ sh
            om = (tv @ sv) / (tv @ tv)
            d += al * ph + om * sh
            r = sv - om * tv
            if k % 10 == 9 and bool(r.norm() <= 1e-10 * F.norm()):
                break
            rn = rs @ r
            pv = r + (rn / rho_o) * (al / om) * (pv - om * v)
            rho_o = rn
        T = T - d
    return T


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("vcycle", "setup"):
        return None  # the hierarchy's own numbers: aggregates and smoothed bases have no outside value
    if kind in ("mlp_forward", "mlp_grad"):
        dims, theta, shift, scale, out_scale, X, Y = _network(c, seed)
        dev = X.device
        th = torch.from_numpy(theta).to(dev).double().requires_grad_(kind == "mlp_grad")
        put = lambda a: torch.from_numpy(a).to(dev).double()

        def net(rows):
            h, off = (rows.double() - put(shift)) * put(scale), 0
            for l, (a, b) in enumerate(zip(dims, dims[1:])):
                h = h @ th[off:off + a * b].reshape(a, b) + th[off + a * b:off + a * b + b]
                off += a * b + b
                h = torch.tanh(h) if l + 2 < len(dims) else h * put(out_scale)
            return h

        if kind == "mlp_forward":
            return torch.cat([net(r) for r in X.split(1_000_000)])
        loss = ((net(X) - Y.double()) ** 2).mean()
        return {"loss": loss.detach(), "grad": torch.autograd.grad(loss, th)[0]}
    if kind == "newton":
        return _exact_newton(c, seed)
    if kind == "batch":
        out = []
        for i, pb in enumerate(_batch_meshes(c)):
            p = _problem(c, seed, pb)
            if pb.n_nodes > EXACT_NODES:
                out.append(None)
                continue
            loads = _batch_loads(c, i, pb, p["coords"], seed)
            rp, ci, vals, _ = _exact_system(p)
            B = torch.stack([_exact_load(dict(p, T=T, body_force=b)).reshape(-1) for T, b in loads], dim=1)
            X = _cg(_csr(rp, ci, vals), _block_diag_inv(rp, ci, vals), B)
            out.append(None if X is None else X.T.contiguous())
        return out
    p = _problem(c, seed)
    if kind == "solve" and p["coords"].shape[0] > EXACT_NODES:
        return None  # thousands of unpreconditioned iterations: over 20 seconds
    rp, ci, vals, rhs = _exact_system(p)
    if kind == "assemble":
        return {"row_ptr": rp.int(), "col_idx": ci.int(), "vals": vals, "rhs": rhs}
    X = _cg(_csr(rp, ci, vals), _block_diag_inv(rp, ci, vals), rhs.reshape(-1, 1))
    return None if X is None else X.reshape(-1, 3)


def _exact_load(p):
    """The load vector alone (another temperature and body force on the same mesh)."""
    x, cells = p["coords"], p["cells"].long()
    npc, dev = cells.shape[1], x.device
    L, W = _rule(4)
    phi, dphi = (torch.from_numpy(v).to(dev) for v in _basis(npc, L))
    w = torch.from_numpy(W).to(dev)
    E, nu, alpha = (p["mat_props"][:, k][p["cell_material"].long()] for k in range(3))
    mu = E / (2.0 * (1.0 + nu))
    lam = E * nu / ((1.0 + nu) * (1.0 - 2.0 * nu))
    g, vol = _geometry(x, cells)
    f = torch.einsum("mc,cak,mki->mai", p["T"][cells] - p["T_ref"],
                     torch.einsum("q,qc,qak->cak", w, phi, dphi), g) * ((3.0 * lam + 2.0 * mu) * alpha * vol)[:, None, None]
    f += torch.einsum("ab,mbi->mai", torch.einsum("q,qa,qb->ab", w, phi, phi), p["body_force"][cells]) * vol[:, None, None]
    rhs = torch.zeros_like(x)
    rhs.index_add_(0, cells.reshape(-1), f.reshape(-1, 3))
    rhs[p["dirichlet_mask"] != 0] = 0.0
    return rhs
