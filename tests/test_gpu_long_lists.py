"""Head entries of block-arrow SDPs at the number of cliques from which they take
a warp of their own (16, 17 and more), with cliques small and large enough for
both splits of Algorithm 2's clique updates: the first 20 FP64 iterates of every
form against the oracle's (rtol 1e-7: the two differ by rounding order, about
1e-12 an iterate, and the iteration is nonexpansive)."""
import dataclasses

import numpy as np
import pytest

from oracle import admm
from paper_1707_05058_gb300 import workloads as W

pytestmark = pytest.mark.gpu


SMALL = [(16, 4, 2), (17, 4, 2), (40, 3, 3)]
LARGE = (18, 20, 6)  # Algorithms 1 and 2: its tau in Algorithm 3 passes near zero, where the residuals lose digits


@pytest.mark.parametrize("form,l,d,h", [(f, *s) for s in SMALL for f in ("primal", "dual", "hsde")]
                         + [("primal", *LARGE), ("dual", *LARGE)])
def test_head_entries(form, l, d, h):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_05058_gb300 import cdsdp
    p = W.block_arrow(l, d, h, 12, seed=l + d)
    w = np.where(p.C_row == p.C_col, 1.0, 2.0)
    p = dataclasses.replace(p, C_val=p.C_val / np.sqrt(np.sum(w * p.C_val ** 2)), b=p.b / np.linalg.norm(p.b))
    run = {"primal": admm.primal_admm, "dual": admm.dual_admm, "hsde": admm.hsde_admm}[form]
    ref = run(admm.decompose(p), eps=0.0, max_iter=20)
    out = cdsdp.Problem(p).bind(max_iter=20).solve(form, eps=0.0, max_iter=20, precision="fp64")
    np.testing.assert_allclose(out["hist"][:, :6], ref.hist[:, :6], rtol=1e-7, atol=1e-10)
