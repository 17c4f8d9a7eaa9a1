"""A batched V-cycle of a group launches every kernel once, however many slots it carries: as many launches
for a handle in the last of eight slots (all eight are carried) as for one in a group of one, at a size whose
cell-wise results for eight slots exceed the least work space of a handle; with the same bits."""
import numpy as np
import pytest

from tests.helpers import build_and_load, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("d,n,r,k", [(2, 128, 1, 2), (3, 16, 1, 2)])
def test_launches_do_not_depend_on_the_slots(d, n, r, k):
    import torch
    from paper_2602_13841_gb300 import inputs, stmg
    build_and_load()
    verts = inputs.vertices(d, n, 0.1, 3)
    p = stmg.default_params(dim=d, n_cells_1d=n, r=r, k=k, nu=0.01, tau=0.05, problem="TG2D" if d == 2 else "TG3D",
                            precond_precision=stmg.STMG_FP32, newton_rtol=1e-4, newton_atol=0.0)
    per_round, result = [], []
    for slots in (1, 8):
        G = stmg.Group(p, verts, slots=slots)
        handles = [stmg.Solver(p, verts, stream=torch.cuda.Stream().cuda_stream) for _ in range(slots)]
        for S in handles:
            G.attach(S)
        S = handles[-1]
        with torch.cuda.stream(torch.cuda.ExternalStream(S.stream)):
            V0 = torch.empty(S.levels[0]["Nv"], dtype=torch.float64, device="cuda")
            U = torch.empty(S.levels[0]["Nst"], dtype=torch.float64, device="cuda")
            S.initial_condition(V0)
            S.initial_guess(V0, U)
            S.slab_solve(0.0, V0, U)
            torch.cuda.current_stream().synchronize()
        result.append(U.cpu().numpy())
        st = G.stats()
        assert st["launches"] % st["rounds"] == 0
        per_round.append(st["launches"] // st["rounds"])
        for S in handles:
            G.detach(S)
            S.close()
        G.close()
    assert per_round[0] == per_round[1], per_round
    assert np.array_equal(result[0], result[1])
