"""Calls whose cell-wise results exceed the cell buffer run in chunks of cell planes (a ring of P planes, the
last one of a chunk kept for the next), batched calls in several passes over the columns.  With the buffer
limited (stmg_test_cell_buffer) to rings of two and three planes, and to one and two columns, every call gives
the bits that it gives with room for everything."""
import numpy as np
import pytest

from paper_2602_13841_gb300 import inputs
from tests.helpers import build_and_load, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a CUDA GPU")]


def _column(d, n, r, k, es):
    """(bytes of one plane of cell-wise results, of one column) of a level."""
    plane = es * (k + 1) * d * n ** (d - 1) * (r + 2) ** d
    return plane, plane * n


def _params(d, n, r, k, prec, **kw):
    from paper_2602_13841_gb300 import stmg
    return stmg.default_params(dim=d, n_cells_1d=n, r=r, k=k, nu=0.01, tau=0.05, problem="MMS2D" if d == 2 else "MMS3D",
                               precond_precision=prec, **kw)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("planes", [2, 3])
@pytest.mark.parametrize("d,n,r,k", [(2, 9, 2, 2), (2, 8, 1, 0), (2, 6, 3, 1), (3, 6, 1, 1), (3, 4, 2, 2)])
def test_chunks_of_planes_give_the_same_bits(d, n, r, k, planes, prec):
    import torch
    from paper_2602_13841_gb300 import stmg
    build_and_load()
    S = stmg.Solver(_params(d, n, r, k, prec), inputs.vertices(d, n, 0.1, 3))
    L = S.levels[0]
    f64 = lambda m, seed: torch.tensor(inputs.uniform(m, seed), dtype=torch.float64, device="cuda")  # noqa: E731
    U, x, vp, d0 = f64(L["Nst"], 1), f64(L["Nst"], 2), f64(L["Nv"], 3), f64(L["Nst"], 4)
    S.smoother_build(U)

    def limit(es):
        b = planes * _column(d, n, r, k, es)[0] if es else 0
        assert S.lib.stmg_test_cell_buffer(S.h, b) == 0

    def calls(on):
        out = []
        for p, dt in ((stmg.STMG_FP64, torch.float64), (stmg.STMG_FP32, torch.float32)):
            limit(on and (8 if p == stmg.STMG_FP64 else 4))
            y = torch.full((L["Nst"],), float("nan"), dtype=dt, device="cuda")
            S.apply(U.to(dt), x.to(dt), y, 0, p)
            out.append(y)
        limit(on and 8)
        R, M = torch.full_like(U, float("nan")), torch.full_like(U, float("nan"))
        S.residual(0.3, U, vp, R)
        S.mass(x, M)
        out += [R, M]
        limit(on and (8 if prec == 0 else 4))
        for zero in (True, False):                      # two sweeps: the second forms rhs - J d through the ring
            z = d0.to(S.pdtype)
            S.smoother_sweep(0, x.to(S.pdtype), z, 2, zero_start=zero)
            out.append(z)
        limit(0)
        torch.cuda.synchronize()
        return out
    for i, (a, b) in enumerate(zip(calls(0), calls(1))):
        assert torch.isfinite(a).all() and torch.equal(a, b), i


@pytest.mark.parametrize("d,n,r,k", [(2, 8, 1, 1), (3, 4, 1, 1)])
def test_batched_columns_in_several_passes_give_the_same_bits(d, n, r, k):
    """The coarse matrix is assembled by one batched apply to the identity (FP64 columns of the coarsest level)."""
    import torch
    from paper_2602_13841_gb300 import stmg
    build_and_load()
    out = []
    for limited in (False, True):
        S = stmg.Solver(_params(d, n, r, k, stmg.STMG_FP64), inputs.vertices(d, n, 0.1, 3))
        m, c = S.levels[0]["Nst"], S.levels[-1]
        if limited:                                     # seven coarse columns a pass; the levels above in rings or whole
            need = max(2 * _column(d, L["n"], L["r"], L["k"], 8)[0] for L in S.levels)
            assert S.lib.stmg_test_cell_buffer(S.h, max(need, 7 * _column(d, c["n"], c["r"], c["k"], 8)[1])) == 0
        S.smoother_build(torch.tensor(inputs.uniform(m, 1), device="cuda"))
        z = torch.empty(m, dtype=torch.float64, device="cuda")
        S.vcycle(torch.tensor(inputs.uniform(m, 2), device="cuda"), z)
        torch.cuda.synchronize()
        out.append(z)
    assert torch.isfinite(out[0]).all() and torch.equal(out[0], out[1])


@pytest.mark.parametrize("columns", [0.5, 1, 2])        # half a column: rings of planes, slot by slot
@pytest.mark.parametrize("d,n,r,k", [(2, 8, 2, 1), (3, 8, 1, 1)])
def test_group_slots_in_several_passes_give_the_same_bits(d, n, r, k, columns):
    import torch
    from paper_2602_13841_gb300 import stmg
    build_and_load()
    verts = inputs.vertices(d, n, 0.1, 3)
    p = _params(d, n, r, k, stmg.STMG_FP32, newton_rtol=1e-8, newton_atol=0.0, nu1=2, nu2=2)

    def solver():
        return stmg.Solver(p, verts, stream=torch.cuda.Stream().cuda_stream)

    def solve(S):
        with torch.cuda.stream(torch.cuda.ExternalStream(S.stream)):
            V0 = torch.tensor(inputs.uniform(S.levels[0]["Nv"], 6), dtype=torch.float64, device="cuda") * 0.1
            U = torch.empty(S.levels[0]["Nst"], dtype=torch.float64, device="cuda")
            S.initial_guess(V0, U)
            rc, st = S.slab_solve(0.1, V0, U, check=False)
            torch.cuda.current_stream().synchronize()
        return rc, st["gmres_its_total"], U.cpu().numpy()
    S = solver()
    want = solve(S)
    S.close()
    G = stmg.Group(p, verts, slots=3)
    handles = [solver() for _ in range(3)]
    for h in handles:
        G.attach(h)
    S = handles[2]                                      # the last slot: all three are carried
    assert S.lib.stmg_test_cell_buffer(S.h, int(columns * _column(d, n, r, k, 4)[1])) == 0
    # (the limit holds for the handle's own FP64 calls too, in rings)
    got = solve(S)
    for h in handles:
        G.detach(h)
        h.close()
    G.close()
    assert want[0] == got[0] == 0 and want[1] == got[1]
    assert np.array_equal(want[2], got[2])
