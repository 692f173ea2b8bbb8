"""Setup's blocked eliminations against the oracle: leaf maps, preconditioner blocks and recovered
leaf solutions at the sizes where the panels, tiles and thread shapes of the elimination change
(rows per thread, a last panel narrower than the others, matrices smaller than one tile), and the
same result from every build of one medium.

Bars: FP64 elimination with partial pivoting of systems with condition number below 1e6 (interior
operators of these leaves) errs by less than 1e6 * 2^-53 ~ 1e-10 relative; complex-float blocks by
less than 1e6 * 2^-24 * (growth) -- the preconditioner's blocks are compared at 1e-3, the precision
their FP16 copies keep."""

import numpy as np
import pytest

import oracle as O
import paper_2112_02211_gb300 as hps

pytestmark = pytest.mark.gpu


def _medium(xi, seed=11):
    rng = np.random.default_rng(seed)
    c, a = rng.uniform(0.2, 0.8, (3, 3)), rng.uniform(-0.4, 0.4, 3)
    return sum(a[i] * np.exp(-20.0 * np.sum((xi - c[i]) ** 2, axis=-1)) for i in range(3)) + 0.02j * xi[..., 0]


# p = 4: a 8 x 8 system; 5: 27 (several partial panels); 7: 125 < 128; 8: 216; 9: 343; 11: 729 (two
# rows per thread); 13: 1331 (six rows per thread, narrow panels)
@pytest.mark.parametrize("grid,p", [((1, 1, 1), 4), ((2, 1, 3), 5), ((2, 2, 1), 7), ((1, 2, 1), 8), ((2, 1, 1), 9),
                                    ((1, 1, 1), 11), ((1, 1, 1), 13)])
def test_leaf_maps_and_recovery(grid, p):
    xi, _ = hps.nodes(*grid, p)
    b = _medium(xi)
    kappa = 3.0 * max(grid)
    solver = hps.Solver(*grid, p, kappa=kappa, b=b, forms=("fp64",), cluster=0, autotune=False)
    g = O.Grid(*grid, p)
    prob = O.build_problem(g, kappa, kappa, b)
    for leaf in range(solver.nl):
        R = solver.export("R", leaf).reshape(solver.nb, solver.nb)
        H = solver.export("H", leaf).reshape(solver.nb, solver.ni)
        assert O.relative_error(R, prob.R[leaf]) <= 1e-10
        assert O.relative_error(H, prob.H[leaf]) <= 1e-10
    import torch
    rng = np.random.default_rng(p)
    for nrhs in (1, 5):
        f = rng.standard_normal((nrhs, solver.nf)) + 1j * rng.standard_normal((nrhs, solver.nf))
        s = rng.standard_normal((nrhs, solver.nl * solver.ni)) + 1j
        u, uf = solver.recover(torch.from_numpy(f).cuda().reshape(-1), s=torch.from_numpy(s).cuda().reshape(-1),
                               nrhs=nrhs, faces=True)
        u, uf = u.cpu().numpy().reshape(nrhs, -1), uf.cpu().numpy().reshape(nrhs, -1)
        for k in range(nrhs):
            ur, ub = O.recover_interior(g, kappa, kappa, b, s[k], f[k], True)
            assert O.relative_error(u[k], ur.reshape(-1)) <= 1e-10
            assert O.relative_error(uf[k], ub.reshape(-1)) <= 1e-10
    solver.close()


# cut-off clusters (1-wide ends, single leaves), odd q, q^2 above 64
@pytest.mark.parametrize("grid,p", [((2, 2, 2), 4), ((3, 2, 3), 6), ((3, 3, 1), 7), ((2, 2, 2), 8), ((2, 1, 2), 11)])
@pytest.mark.parametrize("form", ["fp64", "mixed"])
def test_cluster_inverses(grid, p, form):
    xi, _ = hps.nodes(*grid, p)
    b = _medium(xi, 5)
    kappa = 3.0 * max(grid)
    solver = hps.Solver(*grid, p, kappa=kappa, b=b, forms=(form,), autotune=False)
    g = O.Grid(*grid, p)
    Rt = O.build_problem(g, kappa, kappa, b, homogenized=True).R
    pre = O.Preconditioner(g, Rt)
    q2 = solver.q ** 2
    for c, (leaves, J) in enumerate(zip(pre.blocks, pre.J)):
        slots = [i * solver.nb + f * q2 for i, leaf in enumerate(leaves) for f in range(6)
                 if g.neighbor(leaf, f) in leaves]
        if not slots:
            continue
        rows = np.concatenate([np.arange(s, s + q2) for s in slots])
        ref = np.linalg.inv(J[np.ix_(rows, rows)])
        got = solver.export("Kc", c).reshape(ref.shape)
        assert O.relative_error(got, ref) <= (1e-10 if form == "fp64" else 1e-5)
    solver.close()


def test_builds_of_one_medium_are_the_same():
    """Many matrices in one launch: every build gives the same bits."""
    import torch
    grid, p = (10, 10, 10), 8
    xi, _ = hps.nodes(*grid, p)
    b = _medium(xi)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    first = None
    for _ in range(3):
        solver = hps.Solver(*grid, p, kappa=30.0, b=b, forms=("mixed",), autotune=False)
        r = torch.randn(solver.nf, generator=g.manual_seed(3), dtype=torch.complex64, device="cuda")
        out = (solver.apply(r), solver.precond(r), solver.precond(r, fp16_blocks=True))
        if first is None:
            first = out
        for x, y in zip(first, out):
            assert torch.equal(torch.view_as_real(x), torch.view_as_real(y))
        solver.close()
