"""The FP32 barycentric far quadrature and the shorter near forms against the general FP64 forms, entry by entry, and
which of the two forms a system takes.

CBF blocks.  C^M is the identity and column l of C^J adds RWG l and a neighbour pi(l) of it (pi a permutation of
the cell with a large Gram entry <f_pi(l), n x f_l>), so that the diagonal of G^CBF is even (spread far below 300:
the shorter forms) and the reduced matrix holds Tb as it is, Ks with rows added in pairs and Ta with rows and
columns added in pairs.  The expected matrix is formed from the conventional MoM matrix (general FP64 forms).

Tolerances, relative to the largest entry compared in a block.  Far entries: k R rounded once in FP32 (6e-8 k R,
below 1e-6 at these sizes), 49 terms of one sign per moment, and differences of four local entries that cancel to a
tenth: 1e-5, doubled: 2e-5.  All entries: 2e-5, as in the parity test of the FP32 MoM matrix.
"""
import numpy as np
import pytest
from scipy.optimize import linear_sum_assignment

import workloads as W
from oracle import cbfm as OC, mesh as OM

pytestmark = pytest.mark.gpu
TOL = 2e-5


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()
    from paper_2111_11058_gb300 import build as B
    B.build()
    import paper_2111_11058_gb300 as pkg
    g = W.icosphere(1, 0.3)   # the far tasks' width is timed on the first FP32 call of a process
    pkg.assemble_mom(pkg.mesh(g.verts, g.tris, 1, 2.0), pkg.MIXED)
    return pkg


def _kernels(P, call):
    P.profile(True)
    P.profile_read()
    try:
        r = call()
        return r, {k: v["launches"] for k, v in P.profile_read().items() if v["launches"]}
    finally:
        P.profile(False)


def _far_rwg(m, alpha):
    """RWG pairs none of whose triangle pairs is near."""
    p = m.verts[m.tris]
    cen, h = p.mean(1), np.linalg.norm(p - np.roll(p, 1, 1), axis=2).max(1)
    near = np.linalg.norm(cen[:, None] - cen[None], axis=2) < 1.001 * alpha * np.maximum(h[:, None], h[None])
    near |= (m.tris[:, None, :, None] == m.tris[None, :, None, :]).any(3).any(2)
    t = m.edge_tri
    return ~np.any([near[t[:, a]][:, t[:, b]] for a in range(2) for b in range(2)], axis=0)


# triangle counts around the tiles of 32 trial triangles: 12, 20, 80, 108, 192, 320; near factor 2 (the default) and
# 0.5, where nearly all pairs without a common vertex are far
@pytest.mark.parametrize("shape", ["cube1", "ico0", "ico1", "cube3", "cube4", "ico2"])
@pytest.mark.parametrize("eps,alpha", [(2.5, 0.5), (4.0 - 0.7j, 0.5), (2.5, 2.0)])
def test_entries(P, shape, eps, alpha):
    n = int(shape[-1])
    g = W.cube(n, 0.2 + 0.15 * n) if shape.startswith("cube") else W.icosphere(n, 0.3)
    m = OM.build_rwg(g.verts, g.tris)
    gm = P.mesh(g.verts, g.tris, 1 if n <= 1 else 2, eps, alpha=alpha)
    cell, nc = gm.cells(), gm.n_cells
    G = OC.rwg_gram(m)
    CM, CJ = [], []
    for c in range(nc):
        lam = np.nonzero(cell == c)[0]
        Gc = np.abs(G[np.ix_(lam, lam)])
        l, pi = linear_sum_assignment(-Gc.T)   # pi[l]: the row of column l
        CM.append(np.eye(len(lam), dtype=complex))
        CJ.append(np.eye(len(lam), dtype=complex))
        CJ[c][pi, l] += 1.0
        d = np.abs(np.einsum("il,il->l", CJ[c], G[np.ix_(lam, lam)].astype(complex)))
        assert d.max() < 100 * d.min()
    cb = P.cbf_import(gm, CM, CJ)
    r, ran = _kernels(P, lambda: P.assemble_reduced(gm, cb, P.MIXED_UNFUSED))
    assert ran["k_far"] == 1 and "k_near_blocks" not in ran   # both kinds of pairs in one launch: the shorter forms
    A = r.export()
    ne = m.ne
    Z = P.assemble_mom(gm).export()
    order = np.argsort(cell, kind="stable")   # CBFs follow the cells, RWG functions the mesh
    cj = np.zeros((ne, ne))
    o = 0
    for c in range(nc):
        k = len(CM[c])
        cj[np.ix_(order[o:o + k], np.arange(o, o + k))] = CJ[c].real
        o += k
    cm = np.eye(ne)[:, order]
    far = _far_rwg(m, alpha)
    rows = lambda C, X: (np.abs(C).T @ (~X).astype(float)) == 0   # noqa: E731  no near RWG pair among the rows added
    for name, (R, C), X in (("Ks", (cj, cm), Z[:ne, :ne]), ("Ta", (cj, cj), Z[:ne, ne:]), ("Tb", (cm, cm), Z[ne:, :ne]),
                            ("Ks2", (cm, cj), Z[:ne, :ne])):
        r0, c0 = {"Ks": (0, 0), "Ta": (0, ne), "Tb": (ne, 0), "Ks2": (ne, ne)}[name]
        ref = R.T @ X @ C
        err = np.abs(A[r0:r0 + ne, c0:c0 + ne] - ref)
        assert err.max() <= TOL * np.abs(ref).max(), name
        f = rows(C, rows(R, far).T).T
        if f.any():
            assert err[f].max() <= TOL * np.abs(ref[f]).max(), name + " far"
        else:
            assert n <= 1 or alpha == 2.0


def test_general_forms_above_the_limit(P):
    """Generated CBFs (singular values kept to 1e-3 of the largest) spread over the limit: near pairs in their own
    launch on the unfused path.  The fused form takes the shorter forms for them too; its matrix is as close to
    the FP64 one (1e-5 of its norm: FP32 entries 5e-6 as above, TF32 pairs 2^-21, doubled)."""
    g = W.cube(8, 0.6)
    gm = P.mesh(g.verts, g.tris, 10, 2.5)
    cb = P.build_cbfs(gm, W.plane_wave_set(W.fibonacci_dirs(64)), 1e-3)
    ref = P.assemble_reduced(gm, cb, P.FP64)
    P.cmp_setup(ref)
    d = np.abs(np.diag(ref.gram()))
    assert d.max() > 300 * d.min()
    A = ref.export()
    r, ran = _kernels(P, lambda: P.assemble_reduced(gm, cb, P.MIXED_UNFUSED))
    assert ran["k_far"] == 1 and ran["k_near_blocks"] == 1
    assert np.linalg.norm(r.export() - A) <= 1e-5 * np.linalg.norm(A)
    f, ran = _kernels(P, lambda: P.assemble_reduced(gm, cb, P.MIXED_FUSED))
    assert ran["k_fused"] == 1
    assert np.linalg.norm(f.export() - A) <= 1e-5 * np.linalg.norm(A)
