"""The barycentric far quadrature against the general form: with identity CBF
blocks the reduced matrix is the RWG matrix itself, which the conventional MoM
assembly forms with the general quadrature.

Tolerances, relative to the largest entry.  FP64: both sides sum the same 49
point pairs; rounding of k R (a few units of 1e-16 at k R < 20) and of sums that
cancel to a tenth of their terms stay below 1e-13.  FP32: 6e-8 per operation on
the same sums, k R rounded once (1e-6 rad at k R = 16), TF32 pairs of 2^-21 in
the projection: 5e-6.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()
    from paper_2111_11058_gb300 import build as B
    B.build()
    import paper_2111_11058_gb300 as pkg
    return pkg


# triangle counts around the tiles of 32 trial triangles: 12, 20, 80, 108, 192
@pytest.mark.parametrize("shape", ["cube1", "ico0", "ico1", "cube3", "cube4"])
@pytest.mark.parametrize("eps", [2.5, 4.0 - 0.7j])
def test_identity_blocks_are_the_rwg_matrix(P, shape, eps):
    n = int(shape[-1])
    g = W.cube(n, 0.4 + 0.2 * n) if shape.startswith("cube") else W.icosphere(n, 0.5)
    nc = 1 if n <= 1 else 3
    gm = P.mesh(g.verts, g.tris, nc, eps, partition="rcb")
    cell = gm.cells()
    blocks = [np.eye(k, dtype=complex) for k in np.bincount(cell, minlength=nc)]
    order = np.argsort(cell, kind="stable")   # CBFs follow the cells, RWG functions the mesh
    order = np.concatenate([order, len(cell) + order])
    Z = P.assemble_mom(gm).export()[np.ix_(order, order)]
    cb = P.cbf_import(gm, blocks, blocks)
    for prec, tol in ((P.FP64, 1e-13), (P.MIXED_UNFUSED, 5e-6)):
        A = P.assemble_reduced(gm, cb, prec).export()
        assert A.shape == Z.shape
        assert np.abs(A - Z).max() < tol * np.abs(Z).max(), prec


# fused form: many cells with fewer triangles than a warp has lanes, single CBFs, cell pairs with the
# conjugate lanes (L <= 16) up to their limit and beyond it, one cell, tiles close to N = 256
@pytest.mark.parametrize("shape,nc,L", [("cube4", 60, 1), ("cube4", 24, 3), ("ico2", 9, 16), ("ico2", 4, 17),
                                        ("ico2", 2, 8), ("cube3", 1, 16), ("ico2", 6, 32)])
def test_fused_cell_pairs(P, shape, nc, L):
    """Fused against unfused, both FP32 quadrature and split TF32: 5e-6 of the largest entry (above)."""
    n = int(shape[-1])
    g = W.cube(n, 0.8) if shape.startswith("cube") else W.icosphere(n, 0.5)
    gm = P.mesh(g.verts, g.tris, nc, 3.0 - 0.1j, partition="rcb")
    Ns = np.bincount(gm.cells(), minlength=nc)
    CM, CJ = W.random_cbfs(Ns, [min(L, k) for k in Ns], seed=3)
    cb = P.cbf_import(gm, CM, CJ)
    Af = P.assemble_reduced(gm, cb, P.MIXED_FUSED).export()
    Au = P.assemble_reduced(gm, cb, P.MIXED_UNFUSED).export()
    assert np.isfinite(Af).all()
    assert np.abs(Af - Au).max() < 5e-6 * np.abs(Au).max()
