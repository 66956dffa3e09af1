"""More independent components than a grid's y and z axes take (65,535) in one
solve: every component of 70,000 SDPs of order 2 against the same SDP among a
few.  A component's sums run over its own entries in an order of their own, so
only the order of a few atomics differs, on integers: the FP64 iterates agree to
rounding (1e-12)."""
import numpy as np
import pytest

from paper_1707_05058_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KINDS, COUNT = 7, 70000


def _order2(count):
    """min <C, X> s.t. X_11 = 1: SDP j has the C of kind j mod KINDS."""
    v = np.arange(count)
    c = 0.2 + 0.1 * (v % KINDS)
    i32 = lambda a: np.asarray(a, np.int32)
    return W.SDPProblem(2 * count, count, i32(v), i32(2 * v), i32(2 * v), np.ones(count), np.ones(count),
                        i32(np.concatenate([2 * v, 2 * v + 1, 2 * v + 1])), i32(np.concatenate([2 * v, 2 * v, 2 * v + 1])),
                        np.concatenate([c, 0.5 - c, 0.4 + 0 * c]), i32([]), i32([]))


@pytest.mark.parametrize("form", ["primal", "dual", "hsde"])
def test_many_components(form):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_05058_gb300 import cdsdp
    outs = []
    for count in (KINDS, COUNT):
        P = cdsdp.Problem(_order2(count))
        assert P.info["ncomp"] == count
        o = P.solve(form, eps=0.0, max_iter=12, precision="fp64")
        assert o["iters"] == 12
        r, c = P.pattern()
        outs.append((o["X"].reshape(count, -1), o["Z"].reshape(count, -1), o["y"].reshape(count, -1),
                     P.component_results()[2].reshape(count, -1)))
    for few, many in zip(*outs):
        np.testing.assert_allclose(many, few[np.arange(COUNT) % KINDS], rtol=1e-12, atol=1e-13)
