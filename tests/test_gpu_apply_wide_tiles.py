"""Apply sweeps in phases of 2,432 and more 32-row tiles, where a CTA takes 64
rows: whole tiles (96 x 48 p=2 at its own depth) and tiles cut into pieces (72 x 36
p=2 at depth 4, boxes of 4,000 and more unknowns), row counts that are no multiple
of 64, both precisions and directions.  The tile counts are checked first.

Bounds on |r - A z| / (|A| |z| + |r|) of an eps = 0 factor, a direct solve: 1e-12
as in the other direct-solve tests; 1e-5 for factors in FP32, whose rounding unit
is 5.4e8 times that of FP64 (1e-5 is 170 of them).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import dg, nd  # noqa: E402
from synth import modal_state, naca_ogrid  # noqa: E402

MANY, PIECE = 2432, 64


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__ as g
    g.build()
    import paper_2101_01763_gb300 as m
    return m


def _leaf_rows(nt, nr, B, depth):
    return [len(c["elems"]) * B for c in nd.build_hierarchy(nt, nr, depth)[1][0] if c["interior"]]


@pytest.mark.parametrize("precision,bound", [("fp64", 1e-12), ("mixed", 1e-5)])
@pytest.mark.parametrize("nt,nr,p,depth,pieces", [(96, 48, 2, 0, False), (72, 36, 2, 4, True)])
def test_apply_64_row_tiles(sg, nt, nr, p, depth, pieces, precision, bound):
    B = 4 * (p + 1) ** 2
    plan = sg.Plan(nt, nr, B, depth)
    rows = _leaf_rows(nt, nr, B, plan.export()["D"])
    assert sum(-(-n // 32) for n in rows) >= MANY            # 64-row tiles at the leaf
    assert any(n % 64 for n in rows)
    # L^-1: a tile at row r0 has min(n, r0 + 64) columns, in chunks of 32
    tiles = [-(-min(n, r0 + 64) // 32) for n in rows for r0 in range(0, n, 64)]
    assert (max(tiles) > max(PIECE, sum(tiles) // MANY)) == pieces
    X = naca_ogrid(nt, nr, 21)
    u = modal_state(X, p, 0.5, 2.0, 0.05, 21)
    _, bsr, _ = dg.assemble(X, p, u, 0.5, 2.0, 10.0)
    F = sg.Factor(plan, sg.BSR.from_host(*bsr), 0.0, precision)
    S = dg.bsr_to_scipy(*bsr).tocsr()
    r = np.random.default_rng(3).standard_normal(S.shape[0])
    for tr, M in ((False, S), (True, S.T)):
        z = F.apply(torch.as_tensor(r, device="cuda"), transpose=tr).cpu().numpy()
        assert np.linalg.norm(M @ z - r) <= bound * np.linalg.norm(abs(M) @ abs(z) + abs(r))
