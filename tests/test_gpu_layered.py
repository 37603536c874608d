"""GPU: fields that do not vary across flat cells (a two-dimensional flow on an
extruded boundary-layer mesh, a channel). On a uniform grid of 2^-3 in the plane
the geometry and the double-precision sums over the axes are exact there, at any
aspect ratio, so the fixed-point form has to agree with the double-precision
element routine, which the block scatter runs: 1e-12 norm-wise per component, the
tolerance of every FP64 result. (Not the oracle, which divides the geometry by
detJ first: its rounding puts a variation across the cells.)"""
import numpy as np
import pytest
import torch

import meshgen as mg
import paper_2403_08777_gb300 as ns

pytestmark = pytest.mark.gpu

TOL = 1e-12
N = 8


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ns.load_library()
    return torch.device("cuda:0")


def layered(kind, aspect):
    w = mg.make_workload(N, jitter=0.0, mu=1e-2)
    k, j, i = (a.reshape(-1) for a in np.meshgrid(*[np.arange(N + 1)] * 3, indexing="ij"))
    coords, up = w.coords.copy(), w.up.copy()
    coords[2] /= aspect
    plane = mg.normal((8, (N + 1) ** 2), seed=72)[:, i + (N + 1) * j]
    cot = plane[4:].copy()
    if kind == "plane":
        up[:] = plane[:4]
        up[2] = 0.0
    elif kind == "crossflow":
        up[:] = plane[:4]
        up[2] = 1.0 + 0.1 * plane[2]
    else:  # channel: u(z), p(x)
        z = k / N
        up[:] = 0.0
        up[0] = 4 * z * (1 - z) + 1e-2
        up[3] = 1.0 - i / N
    return coords, w.conn, up, np.ascontiguousarray(cot), w.rho, w.mu


@pytest.mark.parametrize("option", [dict(), dict(scatter="colour"), dict(geometry="recompute")])
@pytest.mark.parametrize("aspect", [20.0, 1e3, 1e4])
@pytest.mark.parametrize("kind", ["plane", "crossflow", "channel"])
def test_layered_fields(dev, kind, aspect, option):
    coords, conn, up, cot, rho, mu = layered(kind, aspect)
    d = [torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in (coords, conn, up, cot)]
    mesh = ns.Mesh(d[0], d[1], colour="scatter" in option)

    def both(**kw):
        p = ns.Params(rho=rho, mu=mu, **kw)
        return mesh.assemble(d[2], p), mesh.assemble_vjp(d[2], d[3], p)

    for x, r in zip(both(**option), both(scatter="block")):
        for k in range(4):
            assert float((x[k] - r[k]).norm()) <= TOL * float(r[k].norm()), k
    mesh.close()
