"""Per-RHS and block GMRES over the sizes where their kernels change form, against a dense solution of the exported
system.

The reduced matrix A comes back exactly (complex64 widened), G^CBF as it is; x = A^{-1} b in complex128 and j = C x are
what the solver approximates.  Its residual is below tol = 1e-10 (FP64), so with cond(A (G^CBF)^{-1}) below 1e5 here
the currents agree to 1e-5 relative at worst and 1e-7 is asserted (the bound of the parity tests); on the mixed
path the FP32 product adds ~1e-7 times that conditioning, and 1e-3 of the currents and 1e-4 of the peak RCS are asserted.
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


@pytest.fixture(scope="module")
def systems(P):
    g = W.cube(5, 0.7)
    m = P.mesh(g.verts, g.tris, 6, 2.5 - 0.05j)
    cb = P.build_cbfs(m, W.plane_wave_set(W.fibonacci_dirs(24)))
    out = {}
    for prec in (P.FP64, P.MIXED):
        r = P.assemble_reduced(m, cb, prec)
        P.cmp_setup(r)
        out[prec] = r
    return out


def _reference(P, r, exc):
    """The currents of a GMRES far below every tolerance tested, on the FP64 system, checked against a dense solve."""
    return P.solve(r, exc, tol=1e-13, restart=r.n + 256, solver=P.BLOCK, allow_noconv=True, monostatic=True)


# one cluster per right-hand side up to the clusters a device holds, then separate kernels: 8-wide and 32-wide products
@pytest.mark.parametrize("nrhs", [1, 2, 8, 9, 12, 33, 40])
@pytest.mark.parametrize("mixed", [False, True])
def test_per_rhs_against_block(P, systems, nrhs, mixed):
    exc = W.plane_wave_set(W.fibonacci_dirs(20))[:nrhs]
    ref = _reference(P, systems[P.FP64], exc)
    r = systems[P.MIXED if mixed else P.FP64]
    res = P.solve(r, exc, tol=1e-6 if mixed else 1e-10, monostatic=True)
    e = np.linalg.norm(res.j - ref.j, axis=0) / np.linalg.norm(ref.j, axis=0)
    assert e.max() <= (1e-3 if mixed else 1e-7)
    if mixed:
        assert np.abs(res.rcs - ref.rcs).max() <= 1e-4 * ref.rcs.max()


# cycles that end at the restart length, inside one and at maxit: the iterate after maxit steps is the same in both forms
# (the same sums in another order: 1e-9 leaves the conditioning 1e6)
@pytest.mark.parametrize("restart,maxit", [(37, 100), (64, 64), (5, 23), (1, 3), (1000, 40)])
def test_cycles(P, systems, restart, maxit):
    exc = W.plane_wave_set(W.fibonacci_dirs(20))[:30]
    kw = dict(tol=1e-12, maxit=maxit, restart=restart, monostatic=True, allow_noconv=True)
    many = P.solve(systems[P.FP64], exc, **kw)
    few = P.solve(systems[P.FP64], exc[:3], **kw)
    assert (few.iters == many.iters[:3]).all() and few.iters.max() == maxit
    assert np.allclose(few.resid, many.resid[:3], rtol=1e-9, atol=0)
    assert np.linalg.norm(few.j - many.j[:, :3]) <= 1e-9 * np.linalg.norm(few.j)


def test_dense_solution(P, systems):
    r = systems[P.FP64]
    exc = W.plane_wave_set(W.fibonacci_dirs(20))[:33]
    ref = _reference(P, r, exc)
    A = r.export()
    CM, CJ = r.cbf.export()
    cells = r.mesh.cells()
    ne, nh = r.mesh.n_edges, r.n // 2
    C = np.zeros((2 * ne, r.n), np.complex128)
    off = 0
    for c, (a, b) in enumerate(zip(CM, CJ)):
        rows = np.nonzero(cells == c)[0]
        C[rows, off:off + a.shape[1]] = a
        C[ne + rows, nh + off:nh + off + b.shape[1]] = b
        off += a.shape[1]
    from oracle import mesh as OM, mom as OMo
    g = W.cube(5, 0.7)
    v = OMo.rhs(OM.build_rwg(g.verts, g.tris), exc)
    D = np.concatenate([C[ne:, nh:], C[:ne, :nh]])          # C^JM: J-tested rows, then M-tested rows
    b = np.concatenate([D[:ne].conj().T @ v[:ne], D[ne:].conj().T @ v[ne:]])
    j = C @ np.linalg.solve(A, b)
    assert np.linalg.norm(ref.j - j) <= 1e-9 * np.linalg.norm(j)
