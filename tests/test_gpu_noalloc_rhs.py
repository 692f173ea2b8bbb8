"""hps_precond_noalloc with 2..63 right-hand sides leaves the handle's own scratch alone, so it runs
the same kernels whatever options.max_rhs is: the same bits from a handle that holds fewer
right-hand sides (no operand rows for them) and one that holds enough."""

import ctypes

import numpy as np
import pytest
import torch

import paper_2112_02211_gb300 as hps
from paper_2112_02211_gb300 import _native as N

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [2, 3, 7])
def test_independent_of_max_rhs(nrhs):
    grid, p = (4, 4, 2), 6
    xi, _ = hps.nodes(*grid, p)
    b = 0.4 * np.exp(-9.0 * np.sum((xi - 0.4) ** 2, axis=-1)) + 0.01j * xi[..., 1]
    out = []
    for max_rhs in (1, 8):
        s = hps.Solver(*grid, p, kappa=10.0, b=b, max_rhs=max_rhs, autotune=False, forms=("mixed",))
        g = torch.Generator(device="cuda")
        g.manual_seed(nrhs)
        r = torch.randn(nrhs * s.nf, generator=g, dtype=torch.complex64, device="cuda")
        z = torch.full_like(r, float("nan"))
        rc = N.load().hps_precond_noalloc(s.handle, N.HPS_C64_H16, ctypes.c_void_p(r.data_ptr()),
                                          ctypes.c_void_p(z.data_ptr()), nrhs,
                                          ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == N.HPS_OK, N.load().hps_last_error()
        torch.cuda.synchronize()
        out.append(z.cpu())
        s.close()
    assert torch.isfinite(torch.view_as_real(out[0])).all()
    assert torch.equal(out[0], out[1])
