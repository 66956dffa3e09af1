"""Constraint matrices with few nonzeros a row and a pattern entry, on both
sides of the averages where the kernels that walk them change (32 a row, 2 an
entry): the first 20 FP64 iterates of every form
against the oracle's (rtol 1e-7: the two differ by rounding order, about 1e-12
an iterate, and the iteration is nonexpansive)."""
import numpy as np
import pytest

from oracle import admm
from paper_1707_05058_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = [(60, 3, 12, 2), (60, 3, 14, 32), (60, 3, 14, 33), (60, 3, 13, 36), (60, 3, 15, 36)]


def _problem(n, w, m, k):
    """A band whose m constraints hold k pattern entries each, unit norms of b and C."""
    rng = np.random.default_rng(n + 7 * k + m)
    base = W.banded(n, w, 1, seed=n, density=1.0)
    r = np.concatenate([np.arange(j, min(n, j + w + 1)) for j in range(n)])
    c = np.concatenate([np.full(min(n, j + w + 1) - j, j) for j in range(n)])
    e = np.concatenate([rng.choice(len(r), k, replace=False) for _ in range(m)])
    con, row, col, val = np.repeat(np.arange(m), k), r[e], c[e], rng.standard_normal(m * k)
    b = rng.random(m) + 0.5
    wgt = np.where(base.C_row == base.C_col, 1.0, 2.0)
    i32 = lambda a: np.asarray(a, np.int32)
    return W.SDPProblem(n, m, i32(con), i32(row), i32(col), val, b / np.linalg.norm(b), base.C_row, base.C_col,
                        base.C_val / np.sqrt(np.sum(wgt * base.C_val ** 2)), i32(r[r != c]), i32(c[r != c]))


@pytest.mark.parametrize("form", ["primal", "dual", "hsde"])
@pytest.mark.parametrize("case", CASES, ids=str)
def test_iterates(case, form):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_05058_gb300 import cdsdp
    p = _problem(*case)
    run = {"primal": admm.primal_admm, "dual": admm.dual_admm, "hsde": admm.hsde_admm}[form]
    ref = run(admm.decompose(p), eps=0.0, max_iter=20)
    P = cdsdp.Problem(p).bind(max_iter=20)
    out = P.solve(form, eps=0.0, max_iter=20, precision="fp64")
    np.testing.assert_allclose(out["hist"][:, :6], ref.hist[:, :6], rtol=1e-7, atol=1e-10)
    np.testing.assert_allclose(out["y"], ref.y, rtol=1e-7, atol=1e-9)
