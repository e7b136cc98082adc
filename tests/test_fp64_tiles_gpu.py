"""The FP64 product of the per-RHS solver without the CMP in its two forms: rows for few right-hand sides, tiles of 32
for many.  Both add ascending k in one chain of FMAs per component, so a right-hand side gets the same bits alone and
among others, whichever form its call takes.
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


# n = 60, 324 and 900, not multiples of 16 or 32 but the last takes the tiles: full ones, ragged ones and two waves
@pytest.mark.parametrize("shape,nrhs", [("ico0", 100), ("cube3", 33), ("cube3", 100), ("cube5", 64), ("cube5", 100)])
def test_same_bits_alone_and_among_many(P, shape, nrhs):
    n = int(shape[-1])
    g = W.cube(n, 0.5) if shape.startswith("cube") else W.icosphere(n, 0.2)
    mom = P.assemble_mom(P.mesh(g.verts, g.tris, 1, 2.5), P.FP64)
    P.tdiag_setup(mom, jacobi=True)
    exc = W.plane_wave_set(W.fibonacci_dirs(50))[:nrhs]
    kw = dict(tol=1e-8, maxit=12, restart=6, precond=P.PC_TDIAG, monostatic=True, allow_noconv=True)
    many = P.solve(mom, exc, **kw)
    for k in (0, nrhs // 2, nrhs - 1):
        alone = P.solve(mom, exc[k:k + 1], **kw)
        assert np.array_equal(many.j[:, k], alone.j[:, 0]) and many.iters[k] == alone.iters[0]
    assert np.isfinite(many.j).all() and (many.resid < 1.0).all()
