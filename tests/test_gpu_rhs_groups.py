"""Body-load right-hand sides in complex double at the orders where eight interior vectors of a leaf
no longer fit in a CTA's shared memory (p = 14: 12^3 values, 221 KB and more): the same kernel with
fewer of them per launch.

Bar: H^tau s is a sum of n_i <= 2744 products, 86 per lane and 5 exchanges, in complex double: below
1e-13 of sum |H||s|, which for these random vectors is within a factor 100 of the result: 1e-11."""

import numpy as np
import pytest
import torch

import oracle as O
import paper_2112_02211_gb300 as hps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [13, 14, 16])
def test_rhs_of_large_leaves(p):
    solver = hps.Solver(2, 1, 1, p, kappa=5.0, forms=("fp64",), cluster=0, max_rhs=9, autotune=p == 14)
    g = torch.Generator(device="cuda")
    g.manual_seed(p)
    H = [torch.from_numpy(solver.export("H", i).reshape(solver.nb, solver.ni)) for i in range(2)]
    q2 = solver.q ** 2
    for nrhs in (1, 3, 4, 5, 8, 9):
        s = torch.randn(nrhs, 2, solver.ni, generator=g, dtype=torch.complex128, device="cuda")
        b = solver.rhs(s=s.reshape(-1), nrhs=nrhs).reshape(nrhs, 2, 6, q2).cpu()
        sc = s.cpu()
        ref = torch.zeros_like(b)
        ref[:, 1, 0] = -(sc[:, 0] @ H[0].T).reshape(nrhs, 6, q2)[:, 1]
        ref[:, 0, 1] = -(sc[:, 1] @ H[1].T).reshape(nrhs, 6, q2)[:, 0]
        for k in range(nrhs):
            assert O.relative_error(b[k].numpy(), ref[k].numpy()) <= 1e-11, (nrhs, k)
    solver.close()
