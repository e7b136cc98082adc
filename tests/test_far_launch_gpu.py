"""Near and far pairs in one launch of the FP32 assembly (shorter entry forms): the first call of a process, which times
the far tasks' widths, and later ones run the same code, and the profile credits work to launches that were made."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = r"""
import numpy as np
import paper_2111_11058_gb300 as P
import workloads as W

g = W.%s
m = P.mesh(g.verts, g.tris, 4, %s)
# Gaussian blocks of few CBFs: their spread lies below the limit of the shorter forms
CM, CJ = W.random_cbfs(np.bincount(m.cells(), minlength=4), [3] * 4, seed=2)
cb = P.cbf_import(m, CM, CJ)
A = []
for call in range(3):
    P.profile(True)
    P.profile_read()
    r = P.assemble_reduced(m, cb, P.MIXED_UNFUSED)
    prof = P.profile_read()
    P.profile(False)
    A.append(r.export())
    for name in ("k_far", "k_near_blocks"):
        rec = prof.get(name)
        assert rec is None or rec["flop"] == 0 or rec["launches"] > 0, (call, name, rec)
P.cmp_setup(r)
d = np.abs(np.diag(r.gram()))
assert d.max() / d.min() < 300, d.max() / d.min()
# tuned calls of the shorter forms make one launch for both kinds of pairs
assert prof["k_far"]["launches"] == 1 and "k_near_blocks" not in prof, prof
assert np.array_equal(A[0], A[1]) and np.array_equal(A[1], A[2])
"""


@pytest.mark.parametrize("shape,eps", [("cube(5, 0.6)", "2.5"), ("icosphere(2, 0.4)", "3.0 - 0.2j")])
def test_first_and_later_calls(shape, eps):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2111_11058_gb300 import build as B
    B.build()
    code = "import torch; torch.cuda.init()\n" + CODE % (shape, eps)
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, PYTHONPATH=ROOT),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
