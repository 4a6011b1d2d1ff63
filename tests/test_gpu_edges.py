"""Sizes and alignments at which a kernel changes branch: the transposed block
SpMV (its block sizes, others, values off a 16-byte boundary), the assembly (one
and two rings, values off a 16-byte boundary) and the apply sweeps (phases of
enough tiles for 64-row tiles; odd sizes), against the oracle or the matrix.

Bounds: sums of FP64 products in another order, 1e-12 relative (as the existing
assembly and SpMV tests); an eps = 0 FP64 factor is a direct solve, 1e-12
backward.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import dg  # noqa: E402
from synth import modal_state, naca_ogrid  # noqa: E402
from synth.lowrank import grid_pattern  # noqa: E402


@pytest.fixture(scope="module")
def sg():
    import __graft_entry__ as g
    g.build()
    import paper_2101_01763_gb300 as m
    return m


def _shifted(t, by):
    """The same values `by` elements into a larger buffer (8-byte aligned only, for odd `by`)."""
    buf = torch.empty(t.numel() + by, dtype=t.dtype, device=t.device)
    buf[by:] = t
    return buf[by:]


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("B", [4, 16, 20, 36, 64])
def test_spmv_transposed(sg, B, shift):
    rp, col = grid_pattern(7, 5)
    rng = np.random.default_rng(B)
    val = rng.standard_normal((len(col), B, B))
    S = dg.bsr_to_scipy(rp, col, val).tocsr()
    A = sg.BSR.from_host(rp, col, val)
    A.val = _shifted(A.val, shift)
    x = rng.standard_normal(35 * B)
    xt = torch.as_tensor(x, device="cuda")
    for tr, M in ((False, S), (True, S.T)):
        y = sg.spmv(A, xt, transpose=tr).cpu().numpy()
        ref = M @ x
        assert np.abs(y - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("bc", ["wall", "farfield"])
@pytest.mark.parametrize("nt,nr,p", [(4, 1, 3), (5, 1, 1), (6, 2, 2), (7, 3, 3), (9, 2, 1)])
def test_assembly_few_rings(sg, nt, nr, p, bc):
    X = naca_ogrid(nt, nr, 7)
    u = modal_state(X, p, 0.6, 2.0, 0.05, 7)
    rhs_o, bsr, dtau_o = dg.assemble(X, p, u, 0.6, 2.0, 10.0, bc_mode=bc)
    rhs, A, dtau = sg.assemble(torch.as_tensor(X, device="cuda"), p, torch.as_tensor(u, device="cuda"), 0.6, 2.0, 10.0,
                               bc=bc)
    assert np.array_equal(A.row_ptr.cpu().numpy(), bsr[0]) and np.array_equal(A.col.cpu().numpy(), bsr[1])
    assert abs(dtau - dtau_o) <= 1e-13 * dtau_o
    assert np.abs(rhs.cpu().numpy() - rhs_o).max() <= 1e-12 * np.abs(rhs_o).max()
    assert np.abs(A.blocks_rowmajor() - bsr[2]).max() <= 1e-12 * np.abs(bsr[2]).max()


def test_assembly_values_off_a_16_byte_boundary(sg):
    import ctypes as C
    from paper_2101_01763_gb300 import _lib as L
    X = naca_ogrid(6, 3, 9)
    u = modal_state(X, 2, 0.6, 2.0, 0.05, 9)
    Xt, ut = torch.as_tensor(X, device="cuda"), torch.as_tensor(u, device="cuda")
    rhs, A, _ = sg.assemble(Xt, 2, ut, 0.6, 2.0, 10.0)
    A2 = sg.BSR.empty(A.K, A.B, A.nnzb)
    A2.val = torch.empty(A2.val.numel() + 1, dtype=torch.float64, device="cuda")[1:]
    r2, dt = torch.empty_like(rhs), C.c_double(0.0)
    mesh, flow, st = L.DgMesh(6, 3, Xt.data_ptr()), L.DgFlow(1.4, 0.6, 2.0, 10.0, L.BC_WALL), A2.struct()
    L.check(L.lib().dg_assemble_jacobian(C.byref(mesh), 2, C.c_void_p(ut.data_ptr()), C.byref(flow),
                                         C.c_void_p(r2.data_ptr()), C.byref(st), C.byref(dt),
                                         C.c_void_p(torch.cuda.current_stream().cuda_stream)), "assemble")
    assert torch.equal(A2.val, A.val) and torch.equal(r2, rhs)


def _direct(sg, A, S, nt, nr, B, depth, r):
    F = sg.Factor(sg.Plan(nt, nr, B, depth), A, 0.0, "fp64")
    scale = np.sqrt(abs(S).sum(0).max() * abs(S).sum(1).max())
    for tr, M in ((False, S), (True, S.T)):
        z = F.apply(torch.as_tensor(r, device="cuda"), transpose=tr).cpu().numpy()
        assert np.linalg.norm(M @ z - r) <= 1e-12 * (scale * np.linalg.norm(z) + np.linalg.norm(r))


# 72 x 36 p=2: more than 2,432 32-row tiles in the leaf phases; the others have odd sizes in every phase
@pytest.mark.parametrize("nt,nr,p,depth", [(72, 36, 2, 0), (7, 5, 1, 2), (11, 9, 2, 3), (13, 6, 3, 2)])
def test_apply_both_directions_direct_solve(sg, nt, nr, p, depth):
    X = naca_ogrid(nt, nr, 21)
    u = modal_state(X, p, 0.5, 2.0, 0.05, 21)
    rhs, bsr, _ = dg.assemble(X, p, u, 0.5, 2.0, 10.0)
    A = sg.BSR.from_host(*bsr)
    _direct(sg, A, dg.bsr_to_scipy(*bsr).tocsr(), nt, nr, 4 * (p + 1) ** 2, depth,
            np.random.default_rng(3).standard_normal(len(rhs)))

