"""The preconditioner on grids with an axis of one leaf: every cluster is 2x2x1 or 2x1x1, all of one
shape, with 8 q^2 or 2 q^2 internal values.  The FP16 kernels of 2x2x2 clusters do not fit them (8
leaves, 24 slots and three internal faces per leaf), so they take the general ones.

Bars: the FP32 blocks against the oracle's cluster solves at 2e-5 and the FP16 blocks (2^-11 per
entry) at 5e-3, as in the tests of 2x2x2 clusters; blocks shared by 16 and more clusters and 64
right-hand sides run one TF32 product (2^-11 of both operands): 2e-3."""

import numpy as np
import pytest
import torch

import oracle as O
import paper_2112_02211_gb300 as hps

pytestmark = pytest.mark.gpu


# p = 6: 128 and 32 internal values; p = 8: 288 and 72; the last two with 16 and 18 clusters of one
# block (constant medium)
@pytest.mark.parametrize("grid,p,const", [((4, 4, 1), 6, False), ((2, 1, 1), 6, False), ((1, 2, 4), 8, False),
                                          ((2, 1, 6), 8, False), ((8, 1, 8), 6, True), ((1, 36, 1), 6, True)])
def test_flat_grids(grid, p, const):
    xi, _ = hps.nodes(*grid, p)
    b = np.zeros(xi.shape[:-1]) if const else 0.4 * np.exp(-9.0 * np.sum((xi - 0.4) ** 2, axis=-1)) + 0.01j * xi[..., 1]
    kappa = 2.5 * max(grid)
    g = O.Grid(*grid, p)
    pre = O.Preconditioner(g, O.build_problem(g, kappa, kappa, b, homogenized=True).R)
    solver = hps.Solver(*grid, p, kappa=kappa, b=b, max_rhs=64, forms=("mixed",), autotune=False)
    rng = np.random.default_rng(p)
    for nrhs in (1, 2, 5, 64):
        r = (rng.standard_normal((nrhs, solver.nf)) + 1j * rng.standard_normal((nrhs, solver.nf))).astype(np.complex64)
        rd = torch.from_numpy(r.reshape(-1)).cuda()
        for fp16 in (False, True):
            z = solver.precond(rd, fp16_blocks=fp16).cpu().numpy().reshape(nrhs, -1)
            bar = 5e-3 if fp16 else 2e-3 if const or nrhs == 64 else 2e-5
            for k in sorted({0, nrhs // 2, nrhs - 1}):
                assert O.relative_error(z[k], pre(r[k].astype(np.complex128))) <= bar, (nrhs, k, fp16)
    solver.close()
