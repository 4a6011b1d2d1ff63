"""FP64 products of operands whose entries differ in scale: an eps = 0 FP64 factor
of a matrix with scaled columns, or with a diagonal of very different entries,
solves as exactly as one of unscaled unknowns does.

Bound: block elimination in FP64 multiply-adds with explicit inverses (what the
factor computes) leaves |r - A z| / (|A| |z| + |r|) of 1.5e-16 to 3.1e-16 in norm
on every one of these systems, at depth 1 where no interface is rotated; 1e-14 is
30 times that.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import dg  # noqa: E402
from synth import modal_state, naca_ogrid  # noqa: E402

NT, NR, P = 16, 4, 2
B = 4 * (P + 1) ** 2


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__ as g
    g.build()
    import paper_2101_01763_gb300 as m
    return m


@pytest.fixture(scope="module")
def system():
    X = naca_ogrid(NT, NR, 7)
    u = modal_state(X, P, 0.5, 2.0, 0.05, 7)
    return dg.assemble(X, P, u, 0.5, 2.0, 10.0)[1]


def _backward_error(sg, bsr, C):
    """Of the factor's solve with the matrix times diag(C), in unscaled unknowns."""
    rp, col, val = bsr
    A = sg.BSR.from_host(rp, col, val * C[col[:, None] * B + np.arange(B)][:, None, :])
    F = sg.Factor(sg.Plan(NT, NR, B, 1), A, 0.0, "fp64")
    S = dg.bsr_to_scipy(rp, col, val).tocsr()
    for tr, M in ((False, S), (True, S.T)):
        r = np.random.default_rng(3).standard_normal(len(C))
        # A C z = r, or C A^T z = C r
        z = F.apply(torch.as_tensor(r * C if tr else r, device="cuda"), transpose=tr).cpu().numpy()
        if not tr:
            z = z * C
        yield np.linalg.norm(M @ z - r) / np.linalg.norm(abs(M) @ abs(z) + abs(r))


@pytest.mark.parametrize("scales", ["none", "si", 10, 20, 30, 450])
def test_scaled_columns(sg, system, scales):
    n = NT * NR * B
    C = np.ones(n)
    if scales == "si":                        # density, momentum and energy in SI units
        C = np.tile([1.2, 400.0, 400.0, 1.7e5], n // 4)
    elif scales != "none":
        C = 2.0 ** np.random.default_rng(1).integers(-scales, scales + 1, n)
    for e in _backward_error(sg, system, C):
        assert e <= 1e-14


@pytest.mark.parametrize("lo,hi", [(0, 10), (0, 20)])
def test_diagonal_of_different_scales(sg, system, lo, hi):
    rp, col, val = system
    val, rng = val.copy(), np.random.default_rng(1)
    for e in range(len(rp) - 1):
        for k in range(rp[e], rp[e + 1]):
            if col[k] == e:
                val[k] += np.diag(10.0 ** rng.uniform(lo, hi, B))
    for e in _backward_error(sg, (rp, col, val), np.ones(NT * NR * B)):
        assert e <= 1e-14
