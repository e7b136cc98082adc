"""CBF generation near the largest cell it takes (2048 RWG functions: the LU kernel's column and pivots fill 128 KB of
shared memory), beyond it, and with many small cells (four, two and one CTA per system).  Reference: the dense FP64
solution with the conventional MoM matrix, which is Z_mm of a single cell, on the host; for many cells the
oracle's.  Tolerances of test_build_cbfs_gpu.py (both sides solve Z_mm J = V in FP64).
"""
import numpy as np
import pytest

import workloads as W
from oracle import cbfm as OC, mesh as OM, mom as OMo

pytestmark = pytest.mark.gpu
GEN = W.plane_wave_set(W.fibonacci_dirs(3))


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


def test_large_cell(P):
    g = W.cube(10, 1.0)
    m = OM.build_rwg(g.verts, g.tris)
    assert m.ne == 1800
    gm = P.mesh(g.verts, g.tris, 1, 2.5 - 0.1j)
    J = np.linalg.solve(P.assemble_mom(gm, P.FP64).export(), OMo.rhs(m, GEN))
    Gf = OC.rwg_gram(m)
    sig = np.linalg.svd(J[:m.ne].conj().T @ (Gf @ J[m.ne:]), compute_uv=False)
    cb = P.build_cbfs(gm, GEN, 1e-6)
    L = int(cb.L[0])
    assert L == int((sig / sig[0] >= 1e-6).sum())
    assert np.abs(cb.sigma[0, :L] - sig[:L] / sig[0]).max() < 1e-9
    CM, CJ = cb.export()
    D = CM[0].conj().T @ (Gf @ CJ[0])
    assert np.abs(D - np.diag(sig[:L])).max() < 1e-9 * sig[0]


def test_larger_cell_is_refused(P):
    g = W.cube(12, 1.0)   # 2592 RWG functions
    with pytest.raises(P.CbfmError) as e:
        P.build_cbfs(P.mesh(g.verts, g.tris, 1, 2.5), GEN)
    assert e.value.status == 1


@pytest.mark.parametrize("shape,nc,s", [("cube7", 100, 5), ("cube7", 100, 40), ("cube9", 200, 8), ("ico4", 640, 8)])
def test_many_cells(P, shape, nc, s):
    n = int(shape[-1])
    g = W.cube(n, 0.8) if shape.startswith("cube") else W.icosphere(n, 0.5)
    m = OM.build_rwg(g.verts, g.tris)
    cell = OM.cells_rcb(m, nc)
    gen = W.plane_wave_set(W.fibonacci_dirs((s + 1) // 2))[:s]
    v = OMo.rhs(m, gen)
    cb = P.build_cbfs(P.mesh(g.verts, g.tris, nc, 3.0 - 0.1j, partition="rcb"), gen, 1e-2)
    for c in range(0, nc, nc // 14):
        lam = np.nonzero(cell == c)[0]
        Ks, Ta, Tb = OMo.pmchwt_blocks(m, 3.0 - 0.1j, rows=lam, cols=lam)
        J = np.linalg.solve(np.block([[Ks, Ta], [Tb, Ks]]), np.vstack([v[lam], v[m.ne + lam]]))
        ref = OC.cell_dual_cbfs(m, lam, J[:len(lam)], J[len(lam):], 1e-2)
        assert cb.L[c] == ref.L
        assert np.abs(cb.sigma[c, :ref.L] - ref.sigma[:ref.L] / ref.sigma[0]).max() < 1e-9
