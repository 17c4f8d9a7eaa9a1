"""Rounding error of the FP32 patch inverses of large (blocked) patches: one sweep of a hierarchy rebuilt in
FP32 against the same in FP64, below eight units in the last place of FP32 (8 * 2^-24 relative, in norm).
Column by column the elimination stays at about that; panel products rounded at the size of the entries
they are added to do not."""
import pytest

from paper_2602_13841_gb300 import inputs
from tests.helpers import build_and_load, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("n,r,k", [(4, 2, 1), (4, 2, 2), (6, 1, 1)])
def test_fp32_patch_inverses_round_like_columnwise_elimination(n, r, k):
    import torch
    from paper_2602_13841_gb300 import stmg
    build_and_load()
    out = []
    for prec in (stmg.STMG_FP64, stmg.STMG_FP32):
        S = stmg.Solver(stmg.default_params(dim=3, n_cells_1d=n, r=r, k=k, nu=1.0 / 400, tau=0.01, problem="TG3D",
                                            precond_precision=prec), inputs.vertices(3, n, 0.1, 3))
        L = S.levels[0]
        V0 = torch.empty(L["Nv"], dtype=torch.float64, device="cuda")
        U = torch.empty(L["Nst"], dtype=torch.float64, device="cuda")
        S.initial_condition(V0)
        S.initial_guess(V0 + 0.01 * torch.tensor(inputs.uniform(L["Nv"], 8), device="cuda"), U)
        S.smoother_build(U)
        rhs = torch.tensor(inputs.uniform(L["Nst"], 9), device="cuda").float()
        z = torch.empty(L["Nst"], dtype=S.pdtype, device="cuda")
        S.smoother_sweep(0, rhs.to(S.pdtype), z, 1, zero_start=True)
        torch.cuda.synchronize()
        out.append(z.double())
    err = float((out[1] - out[0]).norm() / out[0].norm())
    assert err < 8 * 2.0 ** -24, err
