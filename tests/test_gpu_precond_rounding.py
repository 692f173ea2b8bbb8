"""The preconditioner with FP16 blocks for 2..63 right-hand sides and ragged multiples of 64: FP32
arithmetic on the FP16 blocks.  The blocks are rebuilt here from the handle's complex-float ones
(each row divided by its largest component in FP32 and rounded to FP16, as setup does) and applied
in 64 bits, so the FP16 rounding of the blocks, a hundred times larger, is on both sides.

Bar: one component of t is a chain of 6 q^2 fused multiply-adds (3 q^2 complex columns of B) and one
of z_int a chain of 48 q^2 / 32 of them per lane, 5 exchanges and a scale.  Rounding errors of u =
2^-24 / sqrt(3) (rms) relative to partial sums whose squares grow linearly add up to u sqrt(N / 2) of
the result, so z is within u sqrt(3 q^2 + 0.75 q^2 + 8) of the exact product; 1.5 times that is
allowed.  The tensor cores' truncating sums (one right-hand side and multiples of 64) would not pass."""

import numpy as np
import pytest
import torch

import oracle as O
import paper_2112_02211_gb300 as hps

pytestmark = pytest.mark.gpu


def _fp16_rows(M):
    M = M.astype(np.complex64)
    s = np.maximum(np.abs(M.real), np.abs(M.imag)).max(axis=1)
    s = np.where(s > 0, s, np.float32(1)).astype(np.float32)
    inv = (np.float32(1) / s).astype(np.float32)[:, None]
    h = (M.real * inv).astype(np.float16).astype(np.float64) + 1j * (M.imag * inv).astype(np.float16).astype(np.float64)
    return h * s.astype(np.float64)[:, None]


class _Exact:
    """z = J^{-1} r in 64 bits with the handle's FP16 blocks."""

    def __init__(self, solver, grid, p):
        g = O.Grid(*grid, p)
        q2 = solver.q ** 2
        self.nf, self.parts = solver.nf, []
        B = [_fp16_rows(solver.export("B", i).reshape(3 * q2, 3 * q2)) for i in range(solver.nl)]
        for c, leaves in enumerate(O.clusters(g)):
            members = set(leaves)
            slots = [(i, f) for i in leaves for f in range(6) if g.neighbor(i, f) in members]
            where = {s: k for k, s in enumerate(slots)}
            K = _fp16_rows(solver.export("Kc", c).reshape(24 * q2, 24 * q2))
            rows = [np.arange(i * solver.nb + f * q2, i * solver.nb + (f + 1) * q2) for i, f in slots]
            bs = []
            for i in leaves:
                inner = [f for f in range(6) if g.neighbor(i, f) in members]
                out = [where[(g.neighbor(i, f), f ^ 1)] for f in inner]  # where leaf i's rows arrive
                ext = np.concatenate([np.arange(i * solver.nb + f * q2, i * solver.nb + (f + 1) * q2)
                                      for f in range(6) if f not in inner])
                bs.append((B[i], out, ext))
            self.parts.append((K, np.concatenate(rows), bs, q2))

    def __call__(self, r):
        z = r.copy()
        for K, rows, bs, q2 in self.parts:
            t = r[rows].copy()
            for B, out, ext in bs:
                y = B @ r[ext]
                for k, o in enumerate(out):
                    t[o * q2:(o + 1) * q2] -= y[k * q2:(k + 1) * q2]
            z[rows] = K @ t
        return z


# 384, 864 and 1536 internal values; leaves of different media, so blocks of one member
@pytest.mark.parametrize("grid,p", [((4, 2, 2), 6), ((2, 4, 2), 8), ((2, 2, 2), 10)])
def test_fp32_arithmetic(grid, p):
    xi, _ = hps.nodes(*grid, p)
    b = 0.4 * np.exp(-9.0 * np.sum((xi - 0.4) ** 2, axis=-1)) + 0.01j * xi[..., 1]
    solver = hps.Solver(*grid, p, kappa=2.5 * max(grid), b=b, max_rhs=70, forms=("mixed",), autotune=False)
    exact = _Exact(solver, grid, p)
    bar = 1.5 * 2.0 ** -24 / np.sqrt(3.0) * np.sqrt(3.75 * solver.q ** 2 + 8)
    g = torch.Generator(device="cuda")
    for nrhs in (2, 3, 7, 16, 63, 65):
        g.manual_seed(nrhs)
        r = torch.randn(nrhs * solver.nf, generator=g, dtype=torch.complex64, device="cuda")
        z = solver.precond(r, fp16_blocks=True).cpu().numpy().reshape(nrhs, -1)
        rn = r.cpu().numpy().reshape(nrhs, -1).astype(np.complex128)
        for k in sorted({0, nrhs // 2, nrhs - 1}):
            assert O.relative_error(z[k], exact(rn[k])) <= bar, (nrhs, k)
    solver.close()


# blocks of 16 and more clusters: one TF32 product of their complex-float copies in a launch of their
# own (both operands rounded to 2^-11: 2e-3), against the oracle
@pytest.mark.parametrize("grid,p", [((8, 4, 4), 6), ((4, 8, 6), 4)])
def test_widely_shared_blocks(grid, p):
    kappa = 2.5 * max(grid)
    solver = hps.Solver(*grid, p, kappa=kappa, max_rhs=65, forms=("mixed",), autotune=False)
    assert solver.precond_info()[:2] == (grid[0] * grid[1] * grid[2] // 8, 1)
    g = O.Grid(*grid, p)
    hom = O.build_problem(g, kappa, kappa, np.zeros((solver.nl, solver.ni), complex), homogenized=True)
    pre = O.Preconditioner(g, hom.R)
    rng = np.random.default_rng(p)
    for nrhs in (2, 17, 63, 65):
        r = (rng.standard_normal((nrhs, solver.nf)) + 1j * rng.standard_normal((nrhs, solver.nf))).astype(np.complex64)
        z = solver.precond(torch.from_numpy(r.reshape(-1)).cuda(), fp16_blocks=True).cpu().numpy().reshape(nrhs, -1)
        for k in sorted({0, nrhs // 2, nrhs - 1}):
            assert O.relative_error(z[k], pre(r[k].astype(np.complex128))) <= 2e-3, (nrhs, k)
    solver.close()
