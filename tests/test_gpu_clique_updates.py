"""Algorithm 2's clique update at the clique orders where the entries a lane
keeps in flight change (fewer than 32, 64 and 128 entries a warp, then more; a
block a clique above order 22, with fewer than 512 entries and more): the first
20 FP64 iterates against the oracle's (rtol 1e-7: the two differ by rounding
order, about 1e-12 an iterate, and the iteration is nonexpansive)."""
import numpy as np
import pytest

from oracle import admm
from paper_1707_05058_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [2, 7, 8, 11, 12, 15, 16, 22, 23, 31, 32])
def test_orders(order):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_05058_gb300 import cdsdp
    p = W.banded(order + 25, order - 1, 4, seed=order, density=0.5)
    ref = admm.dual_admm(admm.decompose(p), eps=0.0, max_iter=20)
    out = cdsdp.Problem(p).bind(max_iter=20).solve("dual", eps=0.0, max_iter=20, precision="fp64")
    np.testing.assert_allclose(out["hist"][:, :6], ref.hist[:, :6], rtol=1e-7, atol=1e-10)
