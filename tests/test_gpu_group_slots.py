"""A slot of a group computes what a lone handle computes, whichever slots are ready and with whatever
viscosity the group was created: one attached handle, its viscosity not the group's, gives the bits of the same
solve without a group (in slot 0 and in a later one, in groups of one and of several slots)."""
import numpy as np
import pytest

from tests.helpers import build_and_load, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("slots,slot,prec", [(3, 0, 1), (3, 2, 1), (1, 0, 1), (2, 0, 0)])
def test_lone_slot_uses_its_own_viscosity(slots, slot, prec):
    import torch
    from paper_2602_13841_gb300 import inputs, stmg
    build_and_load()
    verts = inputs.vertices(2, 8, 0.1, 3)

    def params(nu):
        return stmg.default_params(dim=2, n_cells_1d=8, r=2, k=1, nu=nu, tau=0.05, problem="TG2D", precond_precision=prec,
                                   newton_rtol=1e-10, newton_atol=1e-14, nu1=2, nu2=2)

    def solver(nu):
        return stmg.Solver(params(nu), verts, stream=torch.cuda.Stream().cuda_stream)

    def solve(S):
        with torch.cuda.stream(torch.cuda.ExternalStream(S.stream)):
            V0 = torch.empty(S.levels[0]["Nv"], dtype=torch.float64, device="cuda")
            U = torch.empty(S.levels[0]["Nst"], dtype=torch.float64, device="cuda")
            S.initial_condition(V0)
            S.initial_guess(V0, U)
            rc, st = S.slab_solve(0.1, V0, U, check=False)
            torch.cuda.current_stream().synchronize()
        return rc, st["gmres_its_total"], U.cpu().numpy()
    alone = solver(1.0 / 900)
    want = solve(alone)
    alone.close()
    G = stmg.Group(params(1.0 / 20), verts, slots=slots)
    others = [solver(1.0 / 20) for _ in range(slot)]        # hold the lower slots, solve nothing
    S = solver(1.0 / 900)
    for o in others + [S]:
        G.attach(o)
    got = solve(S)
    for o in others + [S]:
        G.detach(o)
        o.close()
    G.close()
    assert want[0] == 0 and got[0] == 0
    assert got[1] == want[1]
    assert np.array_equal(got[2], want[2])
