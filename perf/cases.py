"""The calls whose time is watched: what a flow solver, an adjoint or
optimisation loop and a time loop built on this package have it do.

A case is one call through the public Python entry points (`Mesh.assemble`,
`Mesh.assemble_vjp`, `Mesh.assemble_rhs_vjp`, the differentiable `assemble`,
`Mesh.explicit_step`) on a box of hexes cut into 6 tets each: the benchmark's
and the tests' mesh family (8^3, 16^3, 64^3, 128^3, 256^3 hexes), boxes of odd
and unequal sides, boundary-layer boxes whose cells are flat in z, and the
heavily jittered meshes of the precision study. Velocity, pressure, viscosity
and model constants are those of the tests and the benchmark: Taylor-Green
velocity with noise, plus random vectors of up to 10 in the high-Reynolds
case, uniform random pressure, standard normal cotangents.
"""
import math

import torch

import paper_2403_08777_gb300 as ns

# What every case may set, with the package's own defaults.
_DEFAULTS = dict(op="rhs", precision="fp64", nx=8, ny=8, nz=8, jitter=0.1, flat=1.0, order="lex",
                 rho=1.0, mu=1e-2, mag=0.0, c_vreman=0.0, convection="convective", tau="gauss",
                 scatter="auto", geometry="cached")


def _cube(n):
    return dict(nx=n, ny=n, nz=n)


def listed():
    cases = [
        # The smallest call: one right-hand side of the 8^3 parity mesh (3,072
        # tets), as unit tests, examples and coarse levels issue it.
        dict(name="rhs_tiny", **_cube(8)),
        # One SSP-RK3 step of a small mesh (16^3, 24,576 tets): a time loop whose
        # launches count as much as its work. The step starts from a kept state,
        # so that it could be repeated with another dt.
        dict(name="step_small", op="step", **_cube(16)),
        # The same loop in mixed precision with the eddy-viscosity model, on a
        # box of odd, unequal sides (97,092 tets).
        dict(name="step_mixed_odd", op="step", precision="mixed", nx=31, ny=29, nz=18,
             c_vreman=0.07, jitter=0.15),
        # Forward and backward through the differentiable call (an inverse
        # problem's gradient) on the adjoint study's 64^3 mesh (1.57M tets).
        dict(name="grad_64", op="grad", **_cube(64)),
        # A large-eddy simulation's right-hand side: eddy viscosity and the
        # energy-preserving convection, wall-flattened cells, an odd box in
        # random node order (2.56M tets).
        dict(name="rhs_les_odd", nx=97, ny=61, nz=72, jitter=0.15, flat=20.0, order="random",
             mu=1e-4, c_vreman=0.07, convection="skew"),
        # A bitwise reproducible right-hand side (coloured elements), 1.57M tets.
        dict(name="rhs_reproducible", scatter="colour", **_cube(64)),
        # Right-hand side and adjoint at one state in one pass (a steady adjoint
        # solver), random node order, 128^3 (12.6M tets).
        dict(name="rhs_vjp_128", op="rhs_vjp", order="random", **_cube(128)),
        # The same in mixed precision on the precision study's mesh (jitter 0.3).
        dict(name="rhs_vjp_mixed_128", op="rhs_vjp", precision="mixed", jitter=0.3, mu=1e-4,
             mag=10.0, **_cube(128)),
        # The benchmark's workload, 256^3 (100.7M tets, 17.0M nodes), mu = 1e-4,
        # velocities up to 10: the right-hand side ...
        dict(name="rhs_256", mu=1e-4, mag=10.0, **_cube(256)),
        # ... its adjoint ...
        dict(name="vjp_256", op="vjp", mu=1e-4, mag=10.0, **_cube(256)),
        # ... and both in mixed precision.
        dict(name="rhs_mixed_256", precision="mixed", mu=1e-4, mag=10.0, **_cube(256)),
        dict(name="vjp_mixed_256", op="vjp", precision="mixed", mu=1e-4, mag=10.0, **_cube(256)),
    ]
    return [{**_DEFAULTS, **c} for c in cases]


def draw(rng):
    """One more case: any call, precision, formulation, scatter and box of the
    same ranges, its tet count spread evenly over the logarithm."""
    c = dict(_DEFAULTS)
    c["op"] = rng.choice(["rhs", "vjp", "rhs_vjp", "grad", "step"])
    c["precision"] = rng.choice(["fp64", "fp64", "mixed"])
    # hexes: 64 ... 256^3, less where a pass does the work of several calls
    most = 256 ** 3 * {"rhs": 1.0, "vjp": 0.9, "rhs_vjp": 0.7, "grad": 0.5, "step": 0.45}[c["op"]]
    hexes = math.exp(rng.uniform(math.log(64), math.log(0.7 * most)))
    side = hexes ** (1 / 3)
    c["nx"] = max(2, round(side * rng.uniform(0.7, 1.4)))
    c["ny"] = max(2, round(side * rng.uniform(0.7, 1.4)))
    c["nz"] = max(2, round(hexes / (c["nx"] * c["ny"])))
    c["jitter"] = rng.choice([0.05, 0.1, 0.15, 0.3])
    c["flat"] = rng.choice([1.0, 1.0, 5.0, 20.0, 100.0])
    c["order"] = rng.choice(["lex", "lex", "random"])
    c["mu"] = rng.choice([1e-4, 1e-3, 1e-2, 1e-1])
    c["rho"] = rng.choice([1.0, 1.0, 0.8, 1.2])
    c["mag"] = rng.choice([0.0, 10.0])
    c["c_vreman"] = rng.choice([0.0, 0.0, 0.07])
    c["convection"] = rng.choice(["convective", "convective", "skew"])
    c["tau"] = rng.choice(["gauss", "gauss", "element"])
    scatters = ["auto", "auto", "auto", "auto", "block_colour"]
    if c["op"] != "rhs_vjp" and c["precision"] == "fp64":
        scatters.append("colour")
    c["scatter"] = rng.choice(scatters)
    if c["precision"] == "fp64" and c["scatter"] == "auto" and c["op"] != "rhs_vjp":
        c["geometry"] = rng.choice(["cached", "cached", "recompute"])
    return c


# ---- inputs ----

# The 6 tets of a hex share its diagonal: from corner 0 along the axes in every
# order to corner 7; the odd orders swap two nodes for a positive volume.
_PATHS = [((0, 1, 2), 0), ((1, 2, 0), 0), ((2, 0, 1), 0), ((0, 2, 1), 1), ((2, 1, 0), 1),
          ((1, 0, 2), 1)]


def _mesh(case, seed):
    """coords [3, N] float64, conn [4, E] int32 on the GPU."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(1000 * seed + 1)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    sx, sy, sz = 1, nx + 1, (nx + 1) * (ny + 1)
    n_nodes = sz * (nz + 1)
    k, j, i = (torch.arange(n, device=dev, dtype=torch.int32) for n in (nz, ny, nx))
    base = (k[:, None, None] * sz + j[:, None] * sy + i * sx).reshape(-1)
    conn = torch.empty((4, base.numel(), 6), dtype=torch.int32, device=dev)
    step = (sx, sy, sz)
    for t, (axes, odd) in enumerate(_PATHS):
        offs = [0, step[axes[0]], step[axes[0]] + step[axes[1]], sx + sy + sz]
        if odd:
            offs[1], offs[2] = offs[2], offs[1]
        for a in range(4):
            conn[a, :, t] = base + offs[a]
    conn = conn.reshape(4, -1)
    ids = torch.arange(n_nodes, device=dev)
    lat = torch.stack([ids % sy, ids // sy % (ny + 1), ids // sz]).double()
    top = torch.tensor([nx, ny, nz], device=dev, dtype=torch.float64)[:, None]
    inside = ((lat > 0) & (lat < top)).all(0)
    off = (torch.rand((3, n_nodes), generator=gen, device=dev, dtype=torch.float64) * 2 - 1)
    off *= case["jitter"] * inside
    while case["jitter"] > 0.15:  # halve the jitter of nearly flat or inverted tets
        x = lat + off
        bad = torch.zeros(n_nodes, dtype=torch.bool, device=dev)
        for at in range(0, conn.shape[1], 1 << 24):
            cc = conn[:, at:at + (1 << 24)].long()
            e = x[:, cc[1:]] - x[:, cc[:1]]
            det = (e[0, 0] * (e[1, 1] * e[2, 2] - e[2, 1] * e[1, 2])
                   - e[1, 0] * (e[0, 1] * e[2, 2] - e[2, 1] * e[0, 2])
                   + e[2, 0] * (e[0, 1] * e[1, 2] - e[1, 1] * e[0, 2]))
            bad[cc[:, det < 0.05].reshape(-1)] = True
        if not bool(bad.any()):
            break
        off *= torch.where(bad, 0.5, 1.0)
    h = 1.0 / max(nx, ny, nz)
    coords = (lat + off) * torch.tensor([h, h, h / case["flat"]], device=dev)[:, None].double()
    if case["order"] == "random":
        rank = torch.randperm(n_nodes, generator=gen, device=dev)
        moved = torch.empty_like(coords)
        moved[:, rank] = coords
        for a in range(4):
            conn[a] = rank[conn[a].long()].int()
        coords = moved
    return coords.contiguous(), conn.contiguous()


def _fields(case, coords, seed):
    """(u, v, w, p) [4, N] and the cotangent [4, N], float64."""
    dev = coords.device
    gen = torch.Generator(device=dev).manual_seed(1000 * seed + 2)
    n = coords.shape[1]
    x, y, z = coords * (2 * math.pi)
    up = torch.empty((4, n), dtype=torch.float64, device=dev)
    up[0] = x.sin() * y.cos() * z.cos()
    up[1] = -x.cos() * y.sin() * z.cos()
    up[2] = 0.0
    up[:3] += 1e-2 * torch.randn((3, n), generator=gen, device=dev, dtype=torch.float64)
    if case["mag"]:
        d = torch.randn((3, n), generator=gen, device=dev, dtype=torch.float64)
        d /= d.norm(dim=0)
        up[:3] += d * (case["mag"] * torch.rand(n, generator=gen, device=dev, dtype=torch.float64))
    up[3] = torch.rand(n, generator=gen, device=dev, dtype=torch.float64) * 2 - 1
    cot = torch.randn((4, n), generator=gen, device=dev, dtype=torch.float64)
    return up, cot


def _step_size(case):
    """A tenth of the time a particle takes across the smallest cell side."""
    h = 1.0 / max(case["nx"], case["ny"], case["nz"]) / case["flat"]
    return 0.1 * h / (1.0 + case["mag"])


def _params(case):
    return ns.Params(rho=case["rho"], mu=case["mu"], c_vreman=case["c_vreman"],
                     precision=case["precision"], scatter=case["scatter"],
                     convection=case["convection"], tau=case["tau"], geometry=case["geometry"])


def _inputs(case, seed):
    coords, conn = _mesh(case, seed)
    up, cot = _fields(case, coords, seed)
    if case["precision"] == "mixed" and case["op"] != "step":
        up = up.float()
        if case["op"] != "grad":  # the differentiable call takes the float64 RHS's cotangent
            cot = cot.float()
    return coords, conn, up, cot


def prepare(case, seed):
    coords, conn, up, cot = _inputs(case, seed)
    mesh = ns.Mesh(coords, conn, colour=case["scatter"] in ("colour", "block_colour"))
    state = dict(op=case["op"], mesh=mesh, params=_params(case), up=up, cot=cot)
    if case["op"] == "grad":
        state["up"] = up.requires_grad_(True)
    if case["op"] == "step":
        rows = 10 if case["precision"] == "mixed" else 8
        state["now"] = torch.empty_like(up)
        state["work"] = torch.empty((rows, up.shape[1]), dtype=torch.float64, device=up.device)
        state["dt"] = _step_size(case)
    return state


def run(state):
    op, mesh, p = state["op"], state["mesh"], state["params"]
    if op == "rhs":
        return mesh.assemble(state["up"], p)
    if op == "vjp":
        return mesh.assemble_vjp(state["up"], state["cot"], p)
    if op == "rhs_vjp":
        return mesh.assemble_rhs_vjp(state["up"], state["cot"], p)
    if op == "grad":
        rhs = ns.assemble(mesh, state["up"], p)
        (grad,) = torch.autograd.grad(rhs, state["up"], state["cot"])
        return rhs.detach(), grad
    state["now"].copy_(state["up"])
    return mesh.explicit_step(state["now"], state["dt"], "ssprk3", p, work=state["work"])


def work(case):
    """Per pass: connectivity, coordinates and nodal inputs read once, nodal
    outputs written once; the element arithmetic's additions and
    multiplications, and each square root or division, as one each."""
    nodes = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
    tets = 6 * case["nx"] * case["ny"] * case["nz"]
    vreman = case["c_vreman"] > 0
    rhs, vjp, both = (564, 1216, 1507) if vreman else (513, 1095, 1385)
    real = 4 if case["precision"] == "mixed" and case["op"] != "step" else 8
    mesh = 16 * tets + 24 * nodes
    op = case["op"]
    if op == "rhs":
        return {"bytes": mesh + nodes * 4 * (real + 8), "flops": rhs * tets}
    if op == "vjp":
        return {"bytes": mesh + nodes * 4 * (2 * real + 8), "flops": vjp * tets}
    if op == "rhs_vjp":
        return {"bytes": mesh + nodes * 4 * (2 * real + 16), "flops": both * tets}
    if op == "grad":  # the cotangent arrives after the right-hand side is done
        return {"bytes": 2 * mesh + nodes * 4 * (2 * real + 24), "flops": (rhs + vjp) * tets}
    return {"bytes": 3 * mesh + nodes * (3 * 8 + 4 * 6 * 8), "flops": 3 * rhs * tets}


# ---- the same in 64 bits, with torch alone ----

_QA = (5 + 3 * math.sqrt(5)) / 20
_QB = (5 - math.sqrt(5)) / 20


def _element(case, dn, det, U):
    """The element right-hand side F [4, 4, n] of U [4, 4, n] (node, component):
    the weak form at the 4 Gauss points, term by term."""
    rho = case["rho"]
    h = det ** (1 / 3)
    u, p = U[:, :3], U[:, 3]
    G = [[sum(u[a, i] * dn[a][j] for a in range(4)) for j in range(3)] for i in range(3)]
    gp = [sum(p[a] * dn[a][j] for a in range(4)) for j in range(3)]
    div = G[0][0] + G[1][1] + G[2][2]
    mu = torch.full_like(det, case["mu"])
    if case["c_vreman"]:
        b = [[h * h * sum(G[i][m] * G[j][m] for m in range(3)) for j in range(3)] for i in range(3)]
        B = (b[0][0] * b[1][1] - b[0][1] ** 2 + b[0][0] * b[2][2] - b[0][2] ** 2
             + b[1][1] * b[2][2] - b[1][2] ** 2)
        A = sum(G[i][j] ** 2 for i in range(3) for j in range(3))
        on = (A > 0) & (B > 0)
        ratio = torch.where(on, B, torch.ones_like(B)) / torch.where(on, A, torch.ones_like(A))
        mu = mu + torch.where(on, rho * case["c_vreman"] * ratio.sqrt(), torch.zeros_like(mu))
    visc = 4.0 * mu / (h * h)

    def tau_of(v):
        return 1.0 / (visc + 2.0 * rho * (v[0] ** 2 + v[1] ** 2 + v[2] ** 2).sqrt() / h)

    mean = [u[:, i].sum(0) for i in range(3)]
    tau_e = tau_of([0.25 * m for m in mean]) if case["tau"] == "element" else None
    w = det / 24
    F = [[0.0] * 4 for _ in range(4)]
    for g in range(4):
        ug = [_QB * mean[i] + (_QA - _QB) * u[g, i] for i in range(3)]
        pg = _QB * p.sum(0) + (_QA - _QB) * p[g]
        conv = [sum(ug[j] * G[i][j] for j in range(3)) for i in range(3)]
        tau = tau_e if tau_e is not None else tau_of(ug)
        r = [rho * conv[i] + gp[i] for i in range(3)]
        for a in range(4):
            N = _QA if a == g else _QB
            un = sum(ug[j] * dn[a][j] for j in range(3))
            for i in range(3):
                if case["convection"] == "skew":
                    f = -0.5 * rho * (N * conv[i] - un * ug[i])
                else:
                    f = -rho * N * conv[i]
                f = f - mu * sum(dn[a][j] * G[i][j] for j in range(3)) + pg * dn[a][i]
                F[a][i] = F[a][i] + w * (f - tau * rho * un * r[i])
            F[a][3] = F[a][3] + w * (-N * div - tau * sum(dn[a][j] * r[j] for j in range(3)))
    return torch.stack([torch.stack(row) for row in F])


def _whole(case, coords, conn, up, cot, want_rhs, want_vjp):
    """Assembled right-hand side and vector-Jacobian product, chunk by chunk;
    the lumped mass beside them."""
    n = coords.shape[1]
    rhs, grad = (torch.zeros((4, n), dtype=torch.float64, device=up.device) for _ in range(2))
    mass = torch.zeros(n, dtype=torch.float64, device=up.device)
    size = 1 << 20
    for at in range(0, conn.shape[1], size):
        cc = conn[:, at:at + size].long()
        x = coords[:, cc]
        e = x[:, 1:] - x[:, :1]
        cof = []
        for k in range(3):
            a, b = e[:, (k + 1) % 3], e[:, (k + 2) % 3]
            cof.append([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2],
                        a[0] * b[1] - a[1] * b[0]])
        det = sum(e[d, 0] * cof[0][d] for d in range(3))
        dn = [[v / det for v in row] for row in cof]
        dn.insert(0, [-(dn[0][j] + dn[1][j] + dn[2][j]) for j in range(3)])
        flat = cc.reshape(-1)
        mass.index_add_(0, flat, (det / 24).repeat(4))
        U = up[:, cc].transpose(0, 1).contiguous()
        if want_vjp:
            U.requires_grad_(True)
        with torch.set_grad_enabled(want_vjp):
            F = _element(case, dn, det, U)
        if want_rhs:
            rhs.index_add_(1, flat, F.detach().transpose(0, 1).reshape(4, -1))
        if want_vjp:
            W = cot[:, cc].transpose(0, 1)
            (g,) = torch.autograd.grad(F, U, W)
            grad.index_add_(1, flat, g.transpose(0, 1).reshape(4, -1))
    return rhs, grad, mass


def exact(case, seed):
    coords, conn, up, cot = _inputs(case, seed)
    op, up, cot = case["op"], up.double(), cot.double()
    if op == "rhs":
        return _whole(case, coords, conn, up, cot, True, False)[0]
    if op == "vjp":
        return _whole(case, coords, conn, up, cot, False, True)[1]
    if op in ("rhs_vjp", "grad"):
        return _whole(case, coords, conn, up, cot, True, True)[:2]
    # SSP-RK3 of rho m du/dt = F on the velocity rows
    dt = _step_size(case)

    def euler(v):
        F, _, mass = _whole(case, coords, conn, v, cot, True, False)
        out = v.clone()
        out[:3] += dt / case["rho"] * F[:3] / mass
        return out

    s = euler(up)
    s = 0.75 * up + 0.25 * euler(s)
    return up / 3 + 2.0 / 3.0 * euler(s)
