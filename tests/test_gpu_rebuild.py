"""GPU parity of the smoother rebuild at the sizes where its kernels change form: patches that stay in
registers (2D, up to 60 rows) and patches eliminated in panels (more than 64 rows, or FP64 with 60),
in shared memory and in the global workspace; coarse systems of more than 1024 and 2048 unknowns.

Tolerances as for the other sweeps and V-cycles against the FP64 oracle: FP64 1e-9 (sweeps) and
1e-11 (V-cycle), FP32 2e-3.
"""
import numpy as np
import pytest

from oracle import multigrid
from paper_2602_13841_gb300 import inputs
from tests.helpers import build_and_load, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a CUDA GPU")]


def _rel(a, b):
    return np.abs(a - b).max() / np.abs(b).max()


@pytest.mark.parametrize("d,n,r,k,prec", [
    (2, 5, 3, 2, "fp32"), (2, 4, 3, 2, "fp64"),     # m = 60: registers in FP32, panels of 16 in FP64
    (2, 3, 2, 0, "fp32"), (2, 7, 2, 1, "fp64"),     # m = 38, the last block of cells not full
    (3, 3, 1, 2, "fp64"),                           # m = 85: real and complex, matrix on chip
    (2, 9, 2, 2, "fp64"), (2, 11, 2, 1, "fp32"),    # coarse systems of 1932 and 2844 unknowns
])
def test_rebuild_sweep_and_vcycle_match_oracle(d, n, r, k, prec):
    import torch
    from paper_2602_13841_gb300 import stmg
    build_and_load()
    verts = inputs.vertices(d, n, 0.1, 21)
    p = stmg.default_params(dim=d, n_cells_1d=n, r=r, k=k, nu=0.01, tau=0.05, problem="TG2D" if d == 2 else "MMS3D",
                            precond_precision=stmg.STMG_FP64 if prec == "fp64" else stmg.STMG_FP32)
    S = stmg.Solver(p, verts)
    mg = multigrid.Multigrid(d, n, r, k, verts, 0.05, 0.01)
    tol_s, tol_v = (1e-9, 1e-11) if prec == "fp64" else (2e-3, 2e-3)
    n0 = mg.levels[0].Nst
    U = inputs.uniform(n0, 3)
    mg.setup(U)
    S.smoother_build(torch.tensor(U, device="cuda"))
    for l in range(len(mg.levels) - 1):
        m = mg.levels[l].Nst
        rhs, d0 = inputs.uniform(m, 5 + l), inputs.uniform(m, 15 + l)
        got = torch.tensor(d0, dtype=S.pdtype, device="cuda")
        S.smoother_sweep(l, torch.tensor(rhs, dtype=S.pdtype, device="cuda"), got, 1)
        assert _rel(got.double().cpu().numpy(), mg.smoothers[l].sweep(mg.J[l], rhs, d0)) < tol_s, l
    r0 = inputs.uniform(n0, 77)
    z = torch.empty(n0, dtype=torch.float64, device="cuda")
    S.vcycle(torch.tensor(r0, device="cuda"), z)
    assert _rel(z.cpu().numpy(), mg.vcycle(r0)) < tol_v


def test_singular_patch_is_reported():
    """A state of NaN makes every patch matrix NaN: no pivot qualifies, on every path."""
    import torch
    from paper_2602_13841_gb300 import stmg
    build_and_load()
    for d, n, r, prec in ((2, 4, 2, stmg.STMG_FP32), (3, 4, 1, stmg.STMG_FP32), (3, 2, 2, stmg.STMG_FP64)):
        p = stmg.default_params(dim=d, n_cells_1d=n, r=r, k=1, nu=0.01, tau=0.05,
                                problem="TG2D" if d == 2 else "MMS3D", precond_precision=prec)
        S = stmg.Solver(p)
        U = torch.full((S.levels[0]["Nst"],), float("nan"), dtype=torch.float64, device="cuda")
        with pytest.raises(stmg.StmgError) as e:
            S.smoother_build(U)
        assert e.value.status == 5
        S.smoother_build(torch.zeros_like(U))
