"""GPU parity of the cell kernels at the sizes where their blocks are cut: meshes of one to three cells
(every cell on the boundary, one on two opposite sides), blocks whose last cells are missing, each time
degree; and the order of chained launches.

Tolerances as for the other operator comparisons with the FP64 oracle: FP64 1e-12, FP32 2e-5.
"""
import numpy as np
import pytest

from oracle import forms, problems
from oracle.mesh import Mesh, Space
from oracle.reference import TimeData
from paper_2602_13841_gb300 import inputs
from tests.helpers import build_and_load, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a CUDA GPU")]


def _solver(d, n, r, k, pname):
    from paper_2602_13841_gb300 import stmg
    build_and_load()
    verts = inputs.vertices(d, n, 0.1, 11)
    return stmg.Solver(stmg.default_params(dim=d, n_cells_1d=n, r=r, k=k, nu=0.01, tau=0.05, problem=pname), verts), verts


def _rel(a, b):
    return np.abs(a.double().cpu().numpy() - b).max() / np.abs(b).max()


@pytest.mark.parametrize("d,n,r,k", [(2, 1, 1, 0), (2, 1, 3, 2), (2, 2, 2, 1), (2, 3, 1, 2), (2, 13, 2, 2), (2, 17, 1, 1),
                                     (3, 1, 1, 1), (3, 1, 3, 0), (3, 2, 1, 0), (3, 5, 1, 1), (3, 2, 3, 2)])
def test_apply_and_residual_at_block_edges(d, n, r, k):
    import torch
    from paper_2602_13841_gb300 import stmg
    pname = "MMS2D" if d == 2 else "MMS3D"
    S, verts = _solver(d, n, r, k, pname)
    sp, td = Space(Mesh(d, n, verts), r), TimeData(k, S.params.tau)
    lay = forms.SlabLayout(sp, k)
    U, x, vp = inputs.uniform(lay.Nst, 1), inputs.uniform(lay.Nst, 2), inputs.uniform(lay.Nv, 3)
    want = forms.jacobian(sp, td, U, S.params.nu) @ x
    for prec, dt, tol in ((stmg.STMG_FP64, torch.float64, 1e-12), (stmg.STMG_FP32, torch.float32, 2e-5)):
        y = torch.full((lay.Nst,), float("nan"), dtype=dt, device="cuda")
        S.apply(torch.tensor(U, dtype=dt, device="cuda"), torch.tensor(x, dtype=dt, device="cuda"), y, 0, prec)
        assert _rel(y, want) < tol, dt
    R = torch.full((lay.Nst,), float("nan"), dtype=torch.float64, device="cuda")
    S.residual(0.3, torch.tensor(U, device="cuda"), torch.tensor(vp, device="cuda"), R)
    assert _rel(R, forms.residual(sp, td, U, vp, problems.make(pname, S.params.nu), 0.3)) < 1e-12


@pytest.mark.parametrize("d,n,r", [(2, 8, 1), (2, 48, 2), (3, 4, 1)])
def test_chained_launches_keep_their_order(d, n, r):
    """Applies that feed one another give the same bits whether or not the host waits between them."""
    import torch
    from paper_2602_13841_gb300 import stmg
    S, _ = _solver(d, n, r, 1, "TG2D" if d == 2 else "TG3D")
    m = S.levels[0]["Nst"]
    for prec, dt in ((stmg.STMG_FP64, torch.float64), (stmg.STMG_FP32, torch.float32)):
        U = torch.tensor(inputs.uniform(m, 4), dtype=dt, device="cuda")
        x0 = torch.tensor(inputs.uniform(m, 5), dtype=dt, device="cuda")
        out = []
        for wait in (True, False):
            a, b = x0.clone(), torch.empty_like(x0)
            torch.cuda.synchronize()
            for _ in range(8):
                S.apply(U, a, b, 0, prec)
                if wait:
                    torch.cuda.synchronize()
                a, b = b, a
            torch.cuda.synchronize()
            out.append(a.clone())
        assert torch.isfinite(out[0]).all()
        assert torch.equal(out[0], out[1])
