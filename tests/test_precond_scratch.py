"""Device memory of the preconditioner's scratch: one array of 16 bytes per cluster-internal value and
right-hand side (complex double, or the four FP16 operand rows of the tensor-core stage K in its
place) and 4 per cluster, whatever the options; and hps_precond_noalloc, which brings its own array,
does not depend on the handle's."""

import ctypes

import numpy as np
import pytest

import paper_2112_02211_gb300 as hps
from paper_2112_02211_gb300 import _native as N


def _estimate(L, p, max_rhs, **opts):
    lib = N.load()
    o = N.Options()
    lib.hps_default_options(ctypes.byref(o))
    o.max_rhs = max_rhs
    for k, v in opts.items():
        setattr(o, k, v)
    return lib.hps_setup_bytes(ctypes.byref(N.Grid(L, L, L, p, p - 2)), ctypes.byref(o), 1)


# the estimate grows by the scratch and the staged host inputs of 63 right-hand sides, no more
@pytest.mark.parametrize("opts", [dict(), dict(forms=N.HPS_FORM_FP64), dict(tc_apply=0), dict(precond_fp16=0)])
@pytest.mark.parametrize("L,p", [(4, 8), (16, 12)])
def test_estimate_per_right_hand_side(L, p, opts):
    q = p - 2
    internal, clusters = (L // 2) ** 3 * 24 * q * q, (L // 2) ** 3
    per = 16 * internal + 4 * clusters + 16 * L ** 3 * (q ** 3 + 6 * q * q)
    got = _estimate(L, p, 64, **opts) - _estimate(L, p, 1, **opts)
    assert 0 <= got <= 63 * per + 16 * 16 * 64


@pytest.mark.gpu
@pytest.mark.parametrize("grid,p", [((4, 4, 2), 6), ((2, 2, 2), 8)])
def test_handle_memory_per_right_hand_side(grid, p):
    nbytes = []
    for max_rhs in (1, 64):
        s = hps.Solver(*grid, p, kappa=10.0, max_rhs=max_rhs, autotune=False, forms=("mixed",))
        nbytes.append(s.memory_bytes)
        s.close()
    clusters = grid[0] * grid[1] * grid[2] // 8
    per = clusters * (16 * 24 * (p - 2) ** 2 + 4)
    assert nbytes[1] - nbytes[0] <= 63 * per + 16 * 16 * 64


@pytest.mark.gpu
@pytest.mark.parametrize("nrhs", [1, 5, 64])
def test_noalloc_on_its_own_array(nrhs):
    import torch
    grid, p = (4, 4, 2), 6
    xi, _ = hps.nodes(*grid, p)
    b = 0.4 * np.exp(-9.0 * np.sum((xi - 0.4) ** 2, axis=-1)) + 0.01j * xi[..., 1]
    out = []
    for max_rhs in (1, 64):
        s = hps.Solver(*grid, p, kappa=10.0, b=b, max_rhs=max_rhs, autotune=False, forms=("mixed",))
        g = torch.Generator(device="cuda")
        g.manual_seed(nrhs)
        r = torch.randn(nrhs * s.nf, generator=g, dtype=torch.complex64, device="cuda")
        z = torch.full_like(r, float("nan"))
        N.check(N.load().hps_precond_noalloc(s.handle, N.HPS_C64_H16, ctypes.c_void_p(r.data_ptr()),
                                             ctypes.c_void_p(z.data_ptr()), nrhs,
                                             ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
        if max_rhs == 64:
            assert torch.equal(torch.view_as_real(z), torch.view_as_real(s.precond(r, fp16_blocks=True)))
        out.append(z.cpu())
        s.close()
    assert torch.equal(torch.view_as_real(out[0]), torch.view_as_real(out[1]))
