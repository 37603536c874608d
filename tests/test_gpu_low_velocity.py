"""GPU: FP64 results where the velocity is small and nearly uniform, or differs
from 0 at one node of each element only (beside a no-slip wall), and pressure
differences dominate. The Gauss points' parts of such an element's gradient add
up alike, which takes the last bit that the block fixed-point numbers have.
Tolerance as for every FP64 result: 1e-12 norm-wise against the oracle."""
import numpy as np
import pytest
import torch

import meshgen as mg
import oracle
import paper_2403_08777_gb300 as ns

pytestmark = pytest.mark.gpu

TOL = 1e-12
N = 24


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ns.load_library()
    return torch.device("cuda:0")


@pytest.fixture(scope="module", params=["uniform", "one node"])
def case(request):
    w = mg.make_workload(N, jitter=0.1, mu=1e-4)
    speed = 0.1 * w.mu * N  # cell Reynolds number 0.1
    up = w.up.copy()
    if request.param == "uniform":
        up[:3] = speed * (np.array([[0.3], [-0.7], [1.1]]) + 1e-4 * mg.normal((3, w.n_nodes), seed=61))
    else:  # a tet's nodes have i + j + k = s, s + 1, s + 2, s + 3
        k, j, i = np.meshgrid(*[np.arange(N + 1)] * 3, indexing="ij")
        moving = ((i + j + k) % 4 == 0).reshape(-1)
        up[:3] = speed * mg.normal((3, w.n_nodes), seed=62) * moving
    cot = mg.normal((4, w.n_nodes), seed=mg.SEED_COT)
    ref = oracle.assemble(w.coords, w.conn, up, w.rho, w.mu)
    gref = oracle.vjp(w.coords, w.conn, up, cot, w.rho, w.mu)
    return w, up, cot, ref, gref


@pytest.mark.parametrize("option", [dict(), dict(scatter="colour"), dict(geometry="recompute")])
def test_low_velocity(dev, case, option):
    w, up, cot, ref, gref = case
    d = [torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in (w.coords, w.conn, up, cot)]
    mesh = ns.Mesh(d[0], d[1], colour="scatter" in option)
    p = ns.Params(rho=w.rho, mu=w.mu, **option)
    rhs = mesh.assemble(d[2], p).cpu().numpy()
    grad = mesh.assemble_vjp(d[2], d[3], p).cpu().numpy()
    both = [] if option else [t.cpu().numpy() for t in mesh.assemble_rhs_vjp(d[2], d[3], p)]
    mesh.close()
    for x in [rhs] + both[:1]:
        assert np.linalg.norm(x - ref) <= TOL * np.linalg.norm(ref)
    for x in [grad] + both[1:]:
        for k in range(4):
            assert np.linalg.norm(x[k] - gref[k]) <= TOL * np.linalg.norm(gref[k])
