"""Complex-double applies and body loads where a leaf's rows are cut into the most items (few leaves:
12 and 24 parts at p = 10 and 16), into a face's few rows each, and where three right-hand sides go in
one launch or in two; against the handle's own maps in 64 bits.

Bar: sums of n_b <= 1176 or n_i <= 2744 products in complex double: 1e-11 of the result."""

import numpy as np
import pytest
import torch

import oracle as O
import paper_2112_02211_gb300 as hps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,p", [((2, 2, 1), 10), ((3, 3, 3), 10), ((2, 1, 2), 16), ((3, 2, 2), 4), ((1, 5, 3), 5),
                                    ((4, 4, 4), 7)])
@pytest.mark.parametrize("autotune", [False, True])
def test_items(grid, p, autotune):
    solver = hps.Solver(*grid, p, kappa=3.0 * max(grid), forms=("fp64",), cluster=0, max_rhs=8, autotune=autotune)
    g = O.Grid(*grid, p)
    R = [solver.export("R", i).reshape(solver.nb, solver.nb) for i in range(solver.nl)]
    H = [solver.export("H", i).reshape(solver.nb, solver.ni) for i in range(solver.nl)]
    rng = np.random.default_rng(p)
    for nrhs in (1, 2, 3, 4, 7, 8):
        f = rng.standard_normal((nrhs, solver.nf)) + 1j * rng.standard_normal((nrhs, solver.nf))
        s = rng.standard_normal((nrhs, solver.nl, solver.ni)) + 1j
        y = solver.apply(torch.from_numpy(f).cuda().reshape(-1)).cpu().numpy().reshape(nrhs, -1)
        b = solver.rhs(s=torch.from_numpy(s).cuda().reshape(-1), nrhs=nrhs).cpu().numpy().reshape(nrhs, -1)
        for k in {0, nrhs - 1}:
            assert O.relative_error(y[k], O.apply_face(g, R, f[k])) <= 1e-11, (nrhs, k)
            assert O.relative_error(b[k], O.rhs_face(g, H, s[k], None)) <= 1e-11, (nrhs, k)
    solver.close()
