"""GPU parity of the grid transfers at the sizes where their tiles are cut: levels smaller than a tile, last
tiles of one and of all but one node, windows that reach past a tile on both sides, each pair of orders and
time degrees.  Tolerances as in the other comparison of transfers with the FP64 oracle: FP64 1e-13, FP32 2e-6."""
import numpy as np
import pytest

from oracle import multigrid
from paper_2602_13841_gb300 import inputs
from tests.helpers import build_and_load, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-13), ("fp32", 2e-6)])
@pytest.mark.parametrize("d,n,r,k,keep", [(2, 32, 1, 1, 0), (2, 30, 2, 2, 0), (2, 15, 3, 0, 0), (2, 8, 3, 2, 1), (3, 4, 1, 0, 0),
                                          (3, 8, 1, 2, 0), (3, 7, 2, 1, 0), (3, 6, 2, 2, 1), (3, 4, 3, 1, 0)])
def test_transfers_at_tile_edges(d, n, r, k, keep, prec, tol):
    import torch
    from paper_2602_13841_gb300 import stmg
    build_and_load()
    verts = inputs.vertices(d, n, 0.1, 3)
    S = stmg.Solver(stmg.default_params(dim=d, n_cells_1d=n, r=r, k=k, nu=0.01, tau=0.05, problem="TG2D" if d == 2 else "TG3D",
                                        precond_precision=stmg.STMG_FP64 if prec == "fp64" else stmg.STMG_FP32,
                                        keep_time_degree=keep), verts)
    mg = multigrid.Multigrid(d, n, r, k, verts, 0.05, 0.01, keep_k=bool(keep))
    for l, (P, I) in enumerate(zip(mg.P, mg.I)):
        nf, nc = S.levels[l]["Nst"], S.levels[l + 1]["Nst"]
        nvf, nvc = (S.levels[i]["Nv"] * (S.levels[i]["k"] + 1) for i in (l, l + 1))
        xf, xc = inputs.uniform(nf, 200 + l), inputs.uniform(nc, 100 + l)
        for op, x, want in ((0, xc, P @ xc), (1, xf, P.T @ xf), (2, xf, I @ xf[:nvf])):
            out = torch.full((nf if op == 0 else nc,), float("nan"), dtype=S.pdtype, device="cuda")
            S.transfer(l, op, torch.tensor(x, dtype=S.pdtype, device="cuda"), out)
            got = out.double().cpu().numpy()[:nvc if op == 2 else None]
            assert np.abs(got - want).max() < tol * np.abs(want).max(), (l, op)
