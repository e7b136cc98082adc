"""Which products of a solve may be cut into digits of row-scaled fixed point (the tensor-core FP64 form), and what
depends on it.

A digit product is off by about 2^-56 of the largest entries of a row and a column, an FP64 sum by 2^-53 of the
products it adds: rows whose entries differ by orders of magnitude lose digits in the first form that
the second keeps.
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


def _launches(P, call):
    """Kernels launched by a call, name -> launches."""
    P.profile(True)
    P.profile_read()
    try:
        call()
        return {k: v["launches"] for k, v in P.profile_read().items()}
    finally:
        P.profile(False)


def test_mom_block_solve_converges(P):
    """Restarted block GMRES on the conventional MoM system (924 unknowns, 16 right-hand sides): about 1000 block
    iterations with FP64 sums, more than 3000 where the operator's and the Hessenberg matrix's products lose digits."""
    g = W.cylinder(0.2, 0.5, 14, 8, 2)
    mom = P.assemble_mom(P.mesh(g.verts, g.tris, 2, 3.0), P.FP64)
    P.tdiag_setup(mom, jacobi=True)
    exc = W.plane_wave_set(W.fibonacci_dirs(8))
    s = P.solve(mom, exc, tol=1e-6, maxit=2000, restart=200, precond=P.PC_TDIAG, solver=P.BLOCK, monostatic=True,
                allow_noconv=True)
    assert s.resid.max() <= 1e-6 and (s.iters > 0).all()


@pytest.mark.parametrize("pc", ["none", "inexact", "tdiag"])
def test_fp64_sums_without_the_cmp(P, pc):
    g = W.cube(5, 0.6)
    m = P.mesh(g.verts, g.tris, 3, 2.5)
    exc = W.plane_wave_set(W.fibonacci_dirs(20))
    kw = dict(tol=1e-6, maxit=20, restart=300, solver=P.BLOCK, monostatic=True, allow_noconv=True)
    if pc == "tdiag":
        r = P.assemble_mom(m, P.FP64)
        P.tdiag_setup(r, jacobi=True)
        kw["precond"] = P.PC_TDIAG
    else:
        r = P.assemble_reduced(m, P.build_cbfs(m, W.plane_wave_set(W.fibonacci_dirs(24))), P.FP64)
        P.cmp_setup(r, inexact=pc == "inexact", inner_tol=1e-5)
        kw["precond"] = P.PC_NONE if pc == "none" else P.PC_CMP_INEXACT
    n = _launches(P, lambda: P.solve(r, exc, **kw))
    assert n.get("k_oz_gemm", 0) == 0 and n.get("k_gemm_dir", 0) == 0


def test_one_cell_products_keep_fp64_sums(P):
    """FP64 products with identity CBF blocks are exact (one term of every sum is not zero), so A is Z entry by entry
    whatever the number of cells, also where the entries of a row differ by 1e5."""
    g = W.cube(4, 0.8)
    A = []
    for nc in (1, 3):
        m = P.mesh(g.verts, g.tris, nc, 2.5 - 0.1j)
        cell = m.cells()
        blocks = [np.eye(k, dtype=complex) for k in np.bincount(cell, minlength=nc)]
        r = P.assemble_reduced(m, P.cbf_import(m, blocks, blocks), P.FP64)
        order = np.argsort(np.argsort(cell, kind="stable"))   # CBFs follow the cells, RWG functions the mesh
        order = np.concatenate([order, len(cell) + order])
        A.append(r.export()[np.ix_(order, order)])
        if nc == 1:   # right-hand sides and currents of the one cell
            exc = W.plane_wave_set(W.fibonacci_dirs(20))
            n = _launches(P, lambda: P.solve(r, exc, maxit=2, precond=P.PC_NONE, monostatic=True, allow_noconv=True))
    assert np.array_equal(A[0], A[1])
    assert n.get("k_oz_gemm", 0) == 0


def test_fp64_operator_keeps_fp64_sums(P):
    """B = A (G^CBF)^{-1} of an FP64 system, its product with the basis vectors and the recovery: the sizes are such that
    the operator's products (5 n^2 > 2e6) are the only ones of the solve large enough for the tensor cores."""
    g = W.cube(8, 1.0)
    m = P.mesh(g.verts, g.tris, 16, 2.5)
    r = P.assemble_reduced(m, P.build_cbfs(m, W.plane_wave_set(W.fibonacci_dirs(64))), P.FP64)
    assert 5 * r.n ** 2 > 2e6 and 5 * (r.n // 2) ** 2 < 2e6
    assert _launches(P, lambda: P.cmp_setup(r)).get("k_oz_gemm", 0) == 0
    exc = W.plane_wave_set(W.fibonacci_dirs(3))[:5]
    n = _launches(P, lambda: P.solve(r, exc, tol=1e-8, maxit=20, restart=r.n + 256, solver=P.BLOCK, monostatic=True,
                                     allow_noconv=True))
    assert n.get("k_oz_gemm", 0) == 0
