"""What a completion call writes into its scratch: the tables of the one-launch
form only for a dense result on a pattern whose rows are independent, and a
scratch that ends before them still serves the same call.  The tables hold, per
off-diagonal pattern entry, two integers (8 bytes)."""
import numpy as np
import pytest

from paper_1707_05058_gb300 import workloads as W

pytestmark = pytest.mark.gpu

BAND, GENERAL = [W.banded(300, 9, 1, seed=2, density=1.0), W.banded(77, 5, 1, seed=3, density=1.0)], [W.maxcut(80, 3, 3)]


def _case(parts):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_05058_gb300 import cdsdp
    prob = W.direct_sum(parts)
    P = cdsdp.Problem(prob, cache_factor=False)
    r, c = P.pattern()
    return torch, P, W.pd_on_pattern(prob.n, r, c, 3), 8 * (len(r) - prob.n)


@pytest.mark.parametrize("parts,dense,tables", [(BAND, False, False), (GENERAL, False, False), (GENERAL, True, False),
                                                (BAND, True, True)], ids=["logdet", "general-logdet", "general", "rows"])
def test_tables_only_where_they_are_read(parts, dense, tables):
    torch, P, X, table_bytes = _case(parts)
    need, _, _ = P.completion_sizes()
    scratch = torch.full((need,), 0xA5, dtype=torch.uint8, device="cuda")
    P.complete(X, dense=dense, scratch=scratch)
    kept = int((scratch == 0xA5).sum())  # bytes nothing was written to (padding, a few values by chance)
    assert (kept < table_bytes) if tables else (kept >= table_bytes), (kept, table_bytes)


@pytest.mark.parametrize("dense", [False, True])
def test_scratch_without_the_tables(dense):
    torch, P, X, table_bytes = _case(BAND)
    need, welems, offs = P.completion_sizes()
    Wf, ld = P.complete(X, dense=dense)
    Wg, lg = P.complete(X, dense=dense, scratch=torch.empty(need - table_bytes, dtype=torch.uint8, device="cuda"))
    np.testing.assert_array_equal(ld, lg)
    if dense:  # the same recurrence, its sums in another order (bound of the oracle comparison, 1e-10)
        a, b = Wf.cpu().numpy(), Wg.cpu().numpy()
        assert np.abs(a - b).max() <= 1e-10 * np.abs(a).max()
