"""Stage B of the general preconditioner kernels at the largest order with as many leaves as leave two
CTAs for each: 588 rows of a leaf in two parts, more than a CTA has threads.

Bar: z_int = K_c (r_int - B r_ext) with the handle's own blocks in complex double: sums of 588 and
4704 products, 1e-11 of the result."""

import numpy as np
import pytest
import torch

import oracle as O
import paper_2112_02211_gb300 as hps

pytestmark = pytest.mark.gpu


def test_stage_b_in_two_parts():
    grid, p = (2, 2, 26), 16  # 104 leaves
    solver = hps.Solver(*grid, p, kappa=10.0, forms=("fp64",), max_rhs=3, autotune=False)
    g = O.Grid(*grid, p)
    q2, nb = solver.q ** 2, solver.nb
    leaves = O.clusters(g)[5]
    members = set(leaves)
    slots = [(i, f) for i in leaves for f in range(6) if g.neighbor(i, f) in members]
    where = {s: k for k, s in enumerate(slots)}
    K = solver.export("Kc", 5).reshape(24 * q2, 24 * q2)
    gen = torch.Generator(device="cuda")
    for nrhs in (1, 3):
        gen.manual_seed(nrhs)
        r = torch.randn(nrhs, solver.nf, generator=gen, dtype=torch.complex128, device="cuda")
        z = solver.precond(r.reshape(-1)).reshape(nrhs, -1).cpu().numpy()
        face = lambda v, i, f: v[i * nb + f * q2:i * nb + (f + 1) * q2]
        for k in range(nrhs):
            rk = r[k].cpu().numpy()
            t = np.concatenate([face(rk, i, f) for i, f in slots])
            for i in leaves:
                inner = [f for f in range(6) if g.neighbor(i, f) in members]
                ext = np.concatenate([face(rk, i, f) for f in range(6) if f not in inner])
                y = solver.export("B", i).reshape(3 * q2, 3 * q2) @ ext
                for n, f in enumerate(inner):
                    o = where[(g.neighbor(i, f), f ^ 1)]
                    t[o * q2:(o + 1) * q2] -= y[n * q2:(n + 1) * q2]
            got = np.concatenate([face(z[k], i, f) for i, f in slots])
            assert O.relative_error(got, K @ t) <= 1e-11, (nrhs, k)
    solver.close()
