"""GPU: elements that the FP64 form's block fixed-point arithmetic leaves.

A group of values (an element's velocities of one axis, its pressures, its
cotangents, a column of its cofactors) whose largest is outside 2^-100 ..
2^100 or not finite, or a parameter outside 2^-60 .. 2^60, sends the element,
or the call, to the FP64 pipe. Tolerances as for every FP64 result: 1e-12
norm-wise against the oracle; where values are not finite, the same entries.
"""
import numpy as np
import pytest
import torch

import meshgen as mg
import oracle
import paper_2403_08777_gb300 as ns

pytestmark = pytest.mark.gpu

TOL = 1e-12


def run(coords, conn, up, cot, rho, mu, scatter):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    d = [torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in (coords, conn, up, cot)]
    mesh = ns.Mesh(d[0], d[1], colour=scatter == "colour")
    p = ns.Params(rho=rho, mu=mu, scatter=scatter)
    out = mesh.assemble(d[2], p).cpu().numpy(), mesh.assemble_vjp(d[2], d[3], p).cpu().numpy()
    mesh.close()
    return out


def close(x, ref):
    return np.linalg.norm(x - ref) <= TOL * np.linalg.norm(ref)


@pytest.mark.parametrize("scatter", ["auto", "colour"])
@pytest.mark.parametrize("case", ["huge velocity", "half tiny velocity", "tiny cotangent",
                                  "tiny cells", "tiny density"])
def test_finite_elements_out_of_range(case, scatter):
    w = mg.make_workload(5, jitter=0.1, order="random", mu=1e-2)
    coords, up, rho, mu = w.coords.copy(), w.up.copy(), 1.0, 1e-2
    cot = mg.normal((4, w.n_nodes), seed=mg.SEED_COT)
    if case == "huge velocity":
        up[:3] *= 2.0 ** 110
    elif case == "half tiny velocity":
        up[:3, coords[0] < 0.5] *= 2.0 ** -130
    elif case == "tiny cotangent":
        cot *= 2.0 ** -120
    elif case == "tiny cells":
        coords *= 2.0 ** -52
    else:
        rho = 2.0 ** -70
    rhs, grad = run(coords, w.conn, up, cot, rho, mu, scatter)
    assert close(rhs, oracle.assemble(coords, w.conn, up, rho, mu))
    if case != "half tiny velocity":  # below the oracle's complex step
        assert close(grad, oracle.vjp(coords, w.conn, up, cot, rho, mu))


@pytest.mark.parametrize("row", [0, 3])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_values_that_are_not_finite_stay_at_their_elements(bad, row):
    w = mg.make_workload(5, jitter=0.1, mu=1e-2)
    cot = mg.normal((4, w.n_nodes), seed=mg.SEED_COT)
    node = w.n_nodes // 2
    ref = oracle.assemble(w.coords, w.conn, w.up, w.rho, w.mu)
    gref = oracle.vjp(w.coords, w.conn, w.up, cot, w.rho, w.mu)
    near = np.unique(w.conn[:, (w.conn == node).any(axis=0)])
    far = np.setdiff1d(np.arange(w.n_nodes), near)
    up, bad_cot = w.up.copy(), cot.copy()
    up[row, node] = bad
    bad_cot[row, node] = bad
    rhs, _ = run(w.coords, w.conn, up, cot, w.rho, w.mu, "auto")
    _, grad = run(w.coords, w.conn, w.up, bad_cot, w.rho, w.mu, "auto")
    for x, r in ((rhs, ref), (grad, gref)):
        assert close(x[:, far], r[:, far])
        assert not np.isfinite(x[:, node]).all()
