"""Time-outs of the streamed applies (complex float, other than 64, 128, ... right-hand sides), which
wait on mbarriers: an asynchronous call reports them through hps_status, a solve itself, and a solve
keeps an earlier call's time-out for hps_status.  The test hook leaves out one arrival of CTA 0's
first chunk (a grid with many more chunks per CTA than ring stages), with a short wait limit; nothing
hangs or faults, and with the hook cleared the same handle gives the same bits as before."""

import numpy as np
import pytest
import torch

import paper_2112_02211_gb300 as hps
from paper_2112_02211_gb300 import _native as N

pytestmark = pytest.mark.gpu


def _inject(solver, on):
    N.check(N.load().hps_test_inject(solver.handle, N.HPS_INJECT_SKIP_ARRIVAL if on else N.HPS_INJECT_NONE,
                                     4096 if on else 0))


def _timed_out(solver):
    with pytest.raises(hps.HPSError) as err:
        solver.check()
    assert err.value.code == N.HPS_ETIMEOUT
    solver.check()  # reported once


@pytest.mark.parametrize("nrhs", [1, 5])
def test_apply_reports_through_the_status(nrhs):
    solver = hps.Solver(8, 8, 8, 8, kappa=20.0, forms=("mixed",), cluster=0, max_rhs=nrhs, autotune=False)
    f = torch.randn(nrhs * solver.nf, dtype=torch.complex64, device="cuda")
    ref = solver.apply(f)
    solver.check()
    _inject(solver, True)
    y = torch.zeros_like(f)
    solver.apply(f, out=y)
    _timed_out(solver)
    assert not torch.equal(y, ref)
    _inject(solver, False)
    assert torch.equal(torch.view_as_real(solver.apply(f)), torch.view_as_real(ref))
    solver.check()
    solver.close()


def test_solves_report_their_own_and_keep_an_earlier_one():
    xi, _ = hps.nodes(8, 8, 8, 8)
    solver = hps.Solver(8, 8, 8, 8, kappa=20.0, forms=("mixed",), autotune=False)
    s = torch.from_numpy(np.exp(-400.0 * np.sum((xi - 0.37) ** 2, axis=-1)).astype(complex).reshape(-1)).cuda()
    ref, info = solver.solve(s=s, tol=1e-6, form="mixed")
    _inject(solver, True)
    with pytest.raises(hps.HPSError) as err:
        solver.solve(s=s, tol=1e-6, form="mixed")
    assert err.value.code == N.HPS_ETIMEOUT
    solver.check()  # the solve's own report
    solver.apply(torch.randn(solver.nf, dtype=torch.complex64, device="cuda"))
    torch.cuda.synchronize()
    _inject(solver, False)
    f, info2 = solver.solve(s=s, tol=1e-6, form="mixed")
    assert info2["iterations"] == info["iterations"] and torch.equal(f, ref)
    _timed_out(solver)  # the apply's
    solver.close()


def test_status_rejects_a_null_handle():
    assert N.load().hps_status(None, None) == N.HPS_EINVAL
