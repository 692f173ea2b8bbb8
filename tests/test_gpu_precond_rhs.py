"""The preconditioner for every number of right-hand sides: each right-hand side of a batch equals
its own application (alone, or beside one other where blocks of 16 and more clusters are applied
from their complex-FP32 copies for several right-hand sides).  The batch only groups vectors differently (members of a block and
right-hand sides per item of 16 or 64 columns, 1, 2 or 4 vectors per stage-B item, several per pass
of the SIMT kernels); every vector is the same sum in the same order, so the bar is FP32 rounding,
1e-6 of the vector."""

import numpy as np
import pytest
import torch

import paper_2112_02211_gb300 as hps

pytestmark = pytest.mark.gpu


def _solver(grid, p, medium, max_rhs, **kw):
    xi, _ = hps.nodes(*grid, p)
    if medium == "constant":  # one block for all clusters: many vectors per block
        b = np.zeros(xi.shape[:-1])
    else:
        b = 0.4 * np.exp(-9.0 * np.sum((xi - 0.4) ** 2, axis=-1)) + 0.01j * xi[..., 1]
    return hps.Solver(*grid, p, kappa=2.5 * max(grid), b=b, max_rhs=max_rhs, autotune=False, **kw)


def _check(solver, nrhs, dtype, fp16, pair=False):
    g = torch.Generator(device="cuda")
    g.manual_seed(nrhs)
    r = torch.randn(nrhs, solver.nf, generator=g, dtype=dtype, device="cuda")
    z = solver.precond(r.reshape(-1), fp16_blocks=fp16).reshape(nrhs, -1)
    for k in sorted({0, nrhs // 2, nrhs - 1}):
        rk = torch.stack([r[k], r[0]]) if pair else r[k]
        zk = solver.precond(rk.reshape(-1).clone(), fp16_blocks=fp16)[:solver.nf]
        assert float(torch.linalg.vector_norm(z[k] - zk)) <= 1e-6 * float(torch.linalg.vector_norm(zk)), (nrhs, k)


# uniform layout (even grid, even q): the tensor-core path for every count
@pytest.mark.parametrize("grid,p,medium", [((4, 4, 2), 6, "bump"), ((6, 4, 4), 6, "constant"), ((2, 2, 2), 10, "bump"),
                                           ((8, 8, 6), 6, "constant")])
def test_tensor_core_path(grid, p, medium):
    solver = _solver(grid, p, medium, 130, forms=("mixed",))
    for nrhs in (2, 3, 5, 16, 17, 33, 63, 65, 130):
        _check(solver, nrhs, torch.complex64, True, pair=grid == (8, 8, 6))  # 48 clusters, one block
    solver.close()


# odd grids and odd q: SIMT kernels, several right-hand sides per pass, in every precision
@pytest.mark.parametrize("grid,p,medium", [((3, 2, 3), 6, "bump"), ((5, 3, 3), 5, "constant"), ((2, 2, 2), 7, "bump")])
def test_simt_path(grid, p, medium):
    solver = _solver(grid, p, medium, 11, forms=("fp64", "mixed"))
    for nrhs in (2, 3, 7, 8, 11):
        _check(solver, nrhs, torch.complex64, True)
        _check(solver, nrhs, torch.complex64, False)
        _check(solver, nrhs, torch.complex128, False)
    solver.close()
