"""Grid transfers keep a non-finite velocity entry to the output entries that depend on it: an infinity in one
input entry makes exactly those outputs non-finite that the same unit entry changes, although a row of the
1D operators is stored as a window of columns that may hold zeros (a node at which the basis function of a
coarse vertex vanishes lies between nodes at which it does not)."""
import pytest

from tests.helpers import build_and_load, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a CUDA GPU")]


# (n, r): h-transfers of Q2/P1, p-transfers Q3/P2 -> Q2/P1 and Q4/P3 -> Q2/P1
@pytest.mark.parametrize("d,n,r", [(2, 4, 1), (2, 2, 2), (2, 2, 3), (3, 4, 1), (3, 2, 2), (3, 2, 3)])
@pytest.mark.parametrize("prec", [0, 1])
def test_infinity_reaches_only_dependent_entries(d, n, r, prec):
    import torch
    from paper_2602_13841_gb300 import inputs, stmg
    build_and_load()
    p = stmg.default_params(dim=d, n_cells_1d=n, r=r, k=0, nu=0.01, tau=0.05, problem="TG2D" if d == 2 else "TG3D",
                            precond_precision=prec)
    S = stmg.Solver(p, inputs.vertices(d, n, 0.1, 3))
    for op in (0, 1, 2):
        src, dst = (S.levels[1], S.levels[0]) if op == 0 else (S.levels[0], S.levels[1])
        n1 = (src["r"] + 1) * src["n"] + 1
        # entries around the middle of the mesh along every axis, and the last one
        mid = [sum((n1 // 2 + s) * n1 ** l for l in range(d)) for s in (-2, -1, 0, 1, 2)]
        for e in sorted({i for i in mid if 0 <= i < src["Nv"]} | {src["Nv"] - 1}):
            out = []
            for val in (1.0, float("inf")):
                x = torch.zeros(src["Nst"], dtype=S.pdtype, device="cuda")
                x[e] = val
                y = torch.zeros(dst["Nst"], dtype=S.pdtype, device="cuda")
                S.transfer(0, op, x, y)
                torch.cuda.synchronize()
                out.append(y)
            assert torch.equal(torch.isfinite(out[1]), out[0] == 0), (op, e)
