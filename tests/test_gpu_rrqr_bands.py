"""The streaming RRQR at the sizes where its branches change: columns of up to
512, 1024 and 2048 FP32 rows (half of that in FP64) held in registers by a pivot
step and taller ones, heights that are no multiple of a vector, more reflectors
than one block, and columns too tall for the band pass's shared memory.

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
from synth.lowrank import lowrank_coupled  # noqa: E402


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


# tallest interface: 48, 64, 128, 576, 1024 and 1008 rows; depth 3 adds an inner level
@pytest.mark.parametrize("nt,nr,p,depth,eps", [(8, 3, 1, 2, 1e-3), (8, 5, 1, 2, 1e-2), (9, 17, 2, 2, 1e-3),
                                               (8, 17, 3, 2, 1e-3), (8, 29, 2, 2, 1e-3), (12, 9, 2, 3, 1e-3)])
def test_levels_match_oracle(sg, nt, nr, p, depth, eps):
    rhs, bsr = _system(nt, nr, p)
    B = 4 * (p + 1) ** 2
    A = sg.BSR.from_host(*bsr)
    Fo = spand.factor(bsr, nt, nr, depth, eps)
    F = sg.Factor(sg.Plan(nt, nr, B, depth), A, eps, "fp64")
    want = [sum(r for _, r in lv) for lv in Fo.ranks]
    assert want[0] > 0
    assert F.stats()["sum_r"][:len(want)] == want
    zo = spand.apply(Fo, rhs)
    z = F.apply(torch.as_tensor(rhs, device="cuda")).cpu().numpy()
    assert np.linalg.norm(z - zo) <= 1e-9 * np.linalg.norm(zo)
    Fm = sg.Factor(sg.Plan(nt, nr, B, depth), A, eps, "mixed")
    got = Fm.stats()["sum_r"][:len(want)]
    assert all(abs(a - b) <= 0.02 * max(b, 50) for a, b in zip(got, want))
    x, st = sg.sstep_gmres(A, Fm, torch.as_tensor(rhs, device="cuda"), s=4, restart=40, tol=1e-10)
    S = dg.bsr_to_scipy(*bsr).tocsr()
    assert st["converged"] and np.linalg.norm(S @ x.cpu().numpy() - rhs) <= 2e-10 * np.linalg.norm(rhs)


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("mixed", 1e-5)])
@pytest.mark.parametrize("nr,p,depth", [(33, 3, 2), (64, 3, 2), (67, 2, 1)])
def test_tall_columns_direct_solve(sg, nr, p, depth, prec, tol):
    """Interfaces of 2,048 and 4,032 rows and nothing cut (eps = 0: as many pivots
    as rows or columns), and an undivided box of 2,412: the factorization is a
    direct solve whatever the pivots, as long as every reflector reached every
    column once (the bounds of the small direct-solve test)."""
    nt = 8 if depth == 2 else 4
    rhs, bsr = _system(nt, nr, p)
    A = sg.BSR.from_host(*bsr)
    F = sg.Factor(sg.Plan(nt, nr, 4 * (p + 1) ** 2, depth), A, 0.0, prec)
    st = F.stats()
    assert depth == 1 or 0 < st["sum_r"][0] <= st["sum_n"][0]
    z = F.apply(torch.as_tensor(rhs, device="cuda")).cpu().numpy()
    S = dg.bsr_to_scipy(*bsr).tocsr()
    scale = np.sqrt(abs(S).sum(0).max() * abs(S).sum(1).max())     # >= the 2-norm
    assert np.linalg.norm(S @ z - rhs) <= tol * (scale * np.linalg.norm(z) + np.linalg.norm(rhs))


# ranks 2k per element of an interface: 96; 320 and 384; 672 (of 768 rows)
@pytest.mark.parametrize("k,nr", [(4, 13), (16, 12), (28, 13)])
def test_reflector_products_of_many_columns(sg, k, nr):
    """An exact rank: what FP64 drops at eps = 1e-12 is rounding, so the solve is
    direct up to eps times the number of interfaces (5).  The mixed solve is
    refined to the FP64 residual."""
    nt, B = 16, 64
    bsr = lowrank_coupled(nt, nr, B, k, 7, coupling=3.0)
    A = sg.BSR.from_host(*bsr)
    F = sg.Factor(sg.Plan(nt, nr, B, 2), A, 1e-12, "fp64")
    assert F.stats()["sum_r"][0] == sum(r for _, r in spand.factor(bsr, nt, nr, 2, 1e-12).ranks[0])
    S = dg.bsr_to_scipy(*bsr).tocsr()
    scale = np.sqrt(abs(S).sum(0).max() * abs(S).sum(1).max())
    b = np.random.default_rng(k).standard_normal(nt * nr * B)
    bt = torch.as_tensor(b, device="cuda")
    for tr, M in ((False, S), (True, S.T)):
        z = F.apply(bt, transpose=tr).cpu().numpy()
        assert np.linalg.norm(M @ z - b) <= 1e-11 * (scale * np.linalg.norm(z) + np.linalg.norm(b))
    x, st = sg.sstep_gmres(A, sg.Factor(sg.Plan(nt, nr, B, 2), A, 1e-4, "mixed"), bt, s=4, restart=40, tol=1e-10)
    assert st["converged"] and np.linalg.norm(S @ x.cpu().numpy() - b) <= 2e-10 * np.linalg.norm(b)
