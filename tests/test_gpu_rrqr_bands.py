"""The streaming RRQR at the sizes where its branches change: columns of up to
512, 1024 and 2048 FP32 rows (half of that in FP64) held in registers by a pivot
step and taller ones, heights that are no multiple of a vector, more reflectors
than one block, and columns too tall for the band pass's shared memory.

One elimination level (depth 1) over a grid of n_r rings makes the two radial
separators the only interfaces, of n = 4 (p+1)^2 n_r unknowns each.
FP64 ranks are the oracle's and one apply equals the oracle's to 1e-9: the
factors differ from it by rounding (1e-16) times the cut's amplification
(1 / eps = 1e3) times the growth of the triangular inverses (below 1e3 on these
matrices).  In mixed precision ranks may move at the cut by FP32 rounding: 2 %;
the solve is refined to the FP64 residual whatever the ranks.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import dg, spand  # noqa: E402
from synth import modal_state, naca_ogrid  # noqa: E402


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__ as g
    g.build()
    import paper_2101_01763_gb300 as m
    return m


def _system(nt, nr, p):
    X = naca_ogrid(nt, nr, 100 + nr)
    u = modal_state(X, p, 0.6, 2.0, 0.1, 100 + nr)
    rhs, bsr, _ = dg.assemble(X, p, u, 0.6, 2.0, 10.0)
    return rhs, bsr


# n = 16 n_r (p=1), 36 n_r (p=2), 64 n_r (p=3)
@pytest.mark.parametrize("nt,nr,p,eps", [(6, 1, 1, 1e-3), (8, 5, 1, 1e-2), (6, 7, 2, 1e-3), (6, 8, 3, 1e-3),
                                         (5, 9, 3, 1e-3), (6, 29, 2, 1e-3), (4, 17, 3, 1e-2)])
def test_one_level_matches_oracle(sg, nt, nr, p, eps):
    rhs, bsr = _system(nt, nr, p)
    B = 4 * (p + 1) ** 2
    A = sg.BSR.from_host(*bsr)
    Fo = spand.factor(bsr, nt, nr, 1, eps)
    F = sg.Factor(sg.Plan(nt, nr, B, 1), A, eps, "fp64")
    want = [sum(r for _, r in lv) for lv in Fo.ranks]
    assert F.stats()["sum_r"][:len(want)] == want
    zo = spand.apply(Fo, rhs)
    z = F.apply(torch.as_tensor(rhs, device="cuda")).cpu().numpy()
    assert np.linalg.norm(z - zo) <= 1e-9 * np.linalg.norm(zo)
    Fm = sg.Factor(sg.Plan(nt, nr, B, 1), A, eps, "mixed")
    got = Fm.stats()["sum_r"][:len(want)]
    assert all(abs(a - b) <= 0.02 * max(b, 50) for a, b in zip(got, want))
    x, st = sg.sstep_gmres(A, Fm, torch.as_tensor(rhs, device="cuda"), s=4, restart=40, tol=1e-10)
    S = dg.bsr_to_scipy(*bsr).tocsr()
    assert st["converged"] and np.linalg.norm(S @ x.cpu().numpy() - rhs) <= 2e-10 * np.linalg.norm(rhs)


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("mixed", 1e-5)])
@pytest.mark.parametrize("nr", [33, 64])
def test_tall_columns_direct_solve(sg, nr, prec, tol):
    """n = 2,112 and 4,096 rows, every one a pivot (eps = 0): the factorization is
    a direct solve whatever the pivots, as long as every reflector reached every
    column once (the bounds of the small direct-solve test)."""
    rhs, bsr = _system(4, nr, 3)
    A = sg.BSR.from_host(*bsr)
    F = sg.Factor(sg.Plan(4, nr, 64, 1), A, 0.0, prec)
    st = F.stats()
    assert st["sum_r"] == st["sum_n"]
    z = F.apply(torch.as_tensor(rhs, device="cuda")).cpu().numpy()
    S = dg.bsr_to_scipy(*bsr).tocsr()
    scale = np.sqrt(abs(S).sum(0).max() * abs(S).sum(1).max())     # >= the 2-norm
    assert np.linalg.norm(S @ z - rhs) <= tol * (scale * np.linalg.norm(z) + np.linalg.norm(rhs))
