"""CBF generation (batched LU solve over a cluster, Jacobi SVD with the columns in
registers or read again) against the oracle at the edges of its tiles: one
excitation, odd counts, more columns than the registers hold (128), cells of one
block of eight columns and of sizes that are not multiples of eight.

Tolerances as in the full parity test: singular values 1e-9 of the largest (both
sides solve Z_mm J = V in FP64, condition 1e4, and form the Gram of 1e-13
relative accuracy), the diagonal of C^M^H G C^J 1e-9 of its largest entry.
"""
import numpy as np
import pytest

import workloads as W
from oracle import cbfm as OC, mesh as OM

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


@pytest.mark.parametrize("shape,nc,s", [("cube1", 1, 1), ("cube1", 1, 9), ("ico1", 3, 33), ("ico1", 1, 128),
                                        ("ico1", 2, 141)])
def test_build_cbfs_tiles(P, shape, nc, s):
    n = int(shape[-1])
    g = W.cube(n, 0.6) if shape.startswith("cube") else W.icosphere(n, 0.4)
    m = OM.build_rwg(g.verts, g.tris)
    cell = OM.cells_rcb(m, nc)
    gen = W.plane_wave_set(W.fibonacci_dirs((s + 1) // 2))[:s]
    ref = OC.primary_cbfs(m, cell, nc, 3.0 - 0.1j, gen, 1e-3)
    gm = P.mesh(g.verts, g.tris, nc, 3.0 - 0.1j, partition="rcb")
    cb = P.build_cbfs(gm, gen, 1e-3)
    assert cb.L.tolist() == [c.L for c in ref]
    CM, CJ = cb.export()
    for c in range(nc):
        L = ref[c].L
        assert np.abs(cb.sigma[c, :L] - ref[c].sigma[:L] / ref[c].sigma[0]).max() < 1e-9
        lam = ref[c].edges
        D = CM[c].conj().T @ OC.rwg_gram(m, lam, lam) @ CJ[c]
        sig = ref[c].sigma[:L]
        assert np.abs(D - np.diag(sig)).max() < 1e-9 * sig[0]
