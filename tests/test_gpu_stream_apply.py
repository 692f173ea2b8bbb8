"""The complex-float apply with streamed maps against the complex-double one on the same handle, for
grids where its shares of rows, chunks and ring stages end in every possible way: single lines of
leaves, leaves with 1 to 6 neighbours, fewer rows than one chunk, odd q, every group of right-hand
sides, rings of fewer rows per warp (p = 12, 16).

Bar: the maps are rounded to complex float (2^-24 relative per entry) and each row is a sum of n_b
<= 1176 products in at most 10 + 5 rounding steps per lane and exchange, so an entry is within
(1 + 15) 2^-24 sqrt(2) sum |R_ij f_j| / |.|; over random vectors that is below 2e-6 of the norm."""

import pytest
import torch

import paper_2112_02211_gb300 as hps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,p", [((2, 1, 1), 4), ((1, 1, 9), 5), ((3, 2, 2), 6), ((1, 4, 3), 7), ((5, 4, 3), 8),
                                    ((3, 3, 3), 9), ((2, 2, 1), 12), ((2, 1, 1), 16)])
def test_streamed_apply(grid, p):
    solver = hps.Solver(*grid, p, kappa=4.0 * max(grid), cluster=0, max_rhs=40, autotune=False)
    g = torch.Generator(device="cuda")
    g.manual_seed(p)
    for nrhs in (1, 2, 3, 4, 7, 8, 9, 16, 39):
        f = torch.randn(nrhs * solver.nf, generator=g, dtype=torch.complex64, device="cuda")
        y = solver.apply(f).reshape(nrhs, -1)
        ref = solver.apply(f.to(torch.complex128)).reshape(nrhs, -1)
        err = torch.linalg.vector_norm(y - ref, dim=1) / torch.linalg.vector_norm(ref, dim=1)
        assert float(err.max()) <= 2e-6, (nrhs, err)
        one = solver.apply(f.reshape(nrhs, -1)[nrhs - 1].clone())
        assert torch.equal(torch.view_as_real(one), torch.view_as_real(y[nrhs - 1])), nrhs
        if nrhs > 1:  # a vector that starts off a 16-byte boundary
            pad = torch.empty(nrhs * solver.nf + 1, dtype=torch.complex64, device="cuda")
            pad[1:] = f
            assert torch.equal(torch.view_as_real(solver.apply(pad[1:])), torch.view_as_real(y.reshape(-1))), nrhs
    solver.close()
