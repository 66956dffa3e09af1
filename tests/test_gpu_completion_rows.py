"""The one-launch form of the maximum-determinant completion (patterns whose
rows are independent chains) at the sizes where its row blocks, its ring of
recent entries and its stages end, against the oracle; and patterns that keep
the step-by-step form."""
import numpy as np
import pytest

from oracle import completion
from paper_1707_05058_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [  # orders around 16 rows a block, 64 ring entries, 32 steps a stage; lists of 1 .. 44 neighbours
    [W.banded(n, w, 1, seed=n + w, density=1.0) for n, w in ((2, 1), (15, 3), (16, 15), (17, 2), (33, 32))],
    [W.banded(n, w, 1, seed=n + w, density=1.0) for n, w in ((63, 5), (64, 33), (65, 1), (66, 40), (81, 8), (130, 44))],
    [W.block_arrow(l, d, h, 1, seed=l + d) for l, d, h in ((1, 1, 1), (30, 3, 2), (6, 20, 20), (5, 36, 8))],
    [W.maxcut(60, 3, 3), W.banded(40, 4, 1, seed=1, density=1.0)],  # fill in a random order: rows depend on each other
]


@pytest.mark.parametrize("parts", SIZES, ids=["short", "ring", "arrow", "general"])
def test_rows_match_oracle(parts):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_05058_gb300 import cdsdp
    prob = W.direct_sum(parts)
    P = cdsdp.Problem(prob, cache_factor=False)
    r, c = P.pattern()
    X = W.pd_on_pattern(prob.n, r, c, 3)
    _, welems, offs = P.completion_sizes()
    out = torch.full((welems,), float("nan"), dtype=torch.float64, device="cuda")  # nothing may be read before it is written
    Wg, ld = P.complete(X, out=out)
    Wo, schur, ok = completion.maxdet_completion(prob.n, list(zip(r.tolist(), c.tolist())), X)
    assert ok
    vc, _ = P.components()
    Wh = Wg.cpu().numpy()
    for k in range(int(P.info["ncomp"])):
        v = np.flatnonzero(vc == k)
        B = Wh[offs[k]:offs[k + 1]].reshape(len(v), len(v))
        assert np.abs(B - Wo[np.ix_(v, v)]).max() <= 1e-10 * np.abs(Wo).max(), k
        np.testing.assert_allclose(ld[k], np.sum(np.log(schur[v])), rtol=1e-11, atol=1e-11)
