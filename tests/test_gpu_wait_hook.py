"""The failure-test hook stmg_test_wait_timeout, smoother by smoother, without a GPU fault.  Surrogate patches
(0): a block in place of the sweep waits for bytes that are never sent.  Exact patches (2): the staging
barrier of every patch expects 16 bytes more than are copied.  Both waits are bounded: the sweep returns
STMG_ERR_TIMEOUT with the correction as it was (zero when it starts from zero), and the handle then gives
the sweep of a fresh one.  The diagonal sweep (1) has no wait and is not affected."""
import ctypes

import pytest

from tests.helpers import build_and_load, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a CUDA GPU")]


def _handle(d, smoother, prec):
    import torch
    from paper_2602_13841_gb300 import inputs, stmg
    build_and_load()
    n = 4
    p = stmg.default_params(dim=d, n_cells_1d=n, r=1, k=1, nu=1e-2, tau=0.05, problem="TG2D" if d == 2 else "TG3D",
                            precond_precision=prec, smoother=smoother)
    S = stmg.Solver(p, inputs.vertices(d, n, 0.1, 3))
    S.smoother_build(torch.tensor(inputs.uniform(S.levels[0]["Nst"], 5), dtype=torch.float64, device="cuda"))
    return S


# (3D: one call of the exact sweep would wait 2 s in each of eight colours)
@pytest.mark.parametrize("d,smoother,prec", [(2, 0, 1), (2, 0, 0), (3, 0, 1), (2, 1, 1), (2, 2, 1)])
@pytest.mark.parametrize("zero_start", [0, 1])
def test_timed_out_sweep_leaves_the_correction(d, smoother, prec, zero_start):
    import torch
    from paper_2602_13841_gb300 import inputs
    S, ref = _handle(d, smoother, prec), _handle(d, smoother, prec)
    n, lib = S.levels[0]["Nst"], S.lib
    rhs = torch.tensor(inputs.uniform(n, 11), dtype=S.pdtype, device="cuda")
    d0 = torch.tensor(inputs.uniform(n, 12), dtype=S.pdtype, device="cuda")
    want = d0.clone()
    ref.smoother_sweep(0, rhs, want, 1, zero_start=bool(zero_start))

    def sweep():
        z = d0.clone()
        st = lib.stmg_smoother_sweep(S.h, 0, ctypes.c_void_p(rhs.data_ptr()), ctypes.c_void_p(z.data_ptr()), 1, zero_start)
        torch.cuda.synchronize()
        return st, z
    assert lib.stmg_test_wait_timeout(S.h, 1) == 0
    st, z = sweep()
    if smoother == 1:
        assert st == 0 and torch.equal(z, want)
    else:
        assert st == 6, st                              # STMG_ERR_TIMEOUT
        assert torch.equal(z, torch.zeros_like(d0) if zero_start else d0)
    assert lib.stmg_test_wait_timeout(S.h, 0) == 0
    st, z = sweep()
    assert st == 0 and torch.equal(z, want) and float((z - d0).abs().max()) > 0.0
