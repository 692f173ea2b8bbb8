"""The preconditioner in complex double, batches against single right-hand sides: prec_b_kernel sums a
row in four parts for one and two vectors and in one for more, stage K takes 1, 2 or 4 vectors an item
and cuts the batch by its FP64 rule, so a vector is a sum of the same products in another order: sums of
at most 3 q^2 + 24 q^2 products, 1e-12 of the vector (an accumulation in complex float would be 1e-7).
And the complex-float cluster blocks of an order whose systems (2400 rows) take the elimination's widest
shape, at the bar of the smaller ones: 1e-5 of the oracle's inverse."""

import numpy as np
import pytest
import torch

import oracle as O
import paper_2112_02211_gb300 as hps

pytestmark = pytest.mark.gpu


def _medium(xi):
    return 0.4 * np.exp(-9.0 * np.sum((xi - 0.4) ** 2, axis=-1)) + 0.01j * xi[..., 1]


@pytest.mark.parametrize("grid,p", [((3, 2, 3), 6), ((5, 3, 3), 5), ((2, 2, 2), 7), ((4, 4, 2), 8), ((4, 1, 4), 6)])
def test_complex_double(grid, p):
    xi, _ = hps.nodes(*grid, p)
    solver = hps.Solver(*grid, p, kappa=2.5 * max(grid), b=_medium(xi), max_rhs=11, forms=("fp64",), autotune=False)
    g = torch.Generator(device="cuda")
    for nrhs in (2, 3, 4, 7, 8, 11):
        g.manual_seed(nrhs)
        r = torch.randn(nrhs, solver.nf, generator=g, dtype=torch.complex128, device="cuda")
        z = solver.precond(r.reshape(-1)).reshape(nrhs, -1)
        for k in range(nrhs):
            zk = solver.precond(r[k].clone())
            assert float(torch.linalg.vector_norm(z[k] - zk)) <= 1e-12 * float(torch.linalg.vector_norm(zk)), (nrhs, k)
    solver.close()


def test_widest_float_elimination():
    grid, p = (2, 2, 2), 12
    xi, _ = hps.nodes(*grid, p)
    b = _medium(xi)
    solver = hps.Solver(*grid, p, kappa=6.0, b=b, forms=("mixed",), autotune=False)
    g = O.Grid(*grid, p)
    pre = O.Preconditioner(g, O.build_problem(g, 6.0, 6.0, b, homogenized=True).R)
    leaves, J = pre.blocks[0], pre.J[0]
    q2 = solver.q ** 2
    rows = np.concatenate([np.arange(i * solver.nb + f * q2, i * solver.nb + (f + 1) * q2) for i in range(8)
                           for f in range(6) if g.neighbor(leaves[i], f) >= 0])
    ref = np.linalg.inv(J[np.ix_(rows, rows)])
    assert O.relative_error(solver.export("Kc", 0).reshape(ref.shape), ref) <= 1e-5
    solver.close()
