"""The tensor-core projection of blocks above order 1000 against float64: random
blocks, blocks of a graded scale, block-diagonal ones whose halves differ by 1e4, and
their eigenvalues' signs through the invariants of a projection.

Bound: an accumulation in float32 that cuts each of its order / 16 partial sums at
2^-23 is off by order * 2^-27 = 7.5e-9 order, relative to the product's norm; the last
three products of the iteration pass such an error on, so 2.5e-8 order ||W||_F
(Frobenius)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _block(kind, s):
    rng = np.random.default_rng(s)
    A = rng.standard_normal((s, s))
    if kind == "graded":
        g = 10.0 ** -np.linspace(0, 4, s)
        A = g[:, None] * A * g[None, :]
    if kind == "halves":
        h = s // 2
        A[h:, :h] = 0
        A[h:, h:] *= 1e-4
    A = np.tril(A).astype(np.float32).astype(np.float64)
    return A + np.tril(A, -1).T


@pytest.mark.parametrize("kind", ["normal", "graded", "halves"])
@pytest.mark.parametrize("order", [1100, 1500])
def test_error(kind, order):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_05058_gb300 import cdsdp
    W = _block(kind, order)
    iu = np.triu_indices(order)
    x = cdsdp.psd_project_large(torch.tensor(W[iu].astype(np.float32), device="cuda"), [order]).cpu().numpy()
    X = np.zeros_like(W)
    X[iu] = x
    X = X + np.triu(X, 1).T
    lam, V = np.linalg.eigh(W)
    nrm, bound = np.linalg.norm(W), 2.5e-8 * order
    assert np.linalg.norm(X - (V * np.maximum(lam, 0)) @ V.T) <= bound * nrm
    assert abs(np.sum((X - W) * X)) <= bound * nrm ** 2  # orthogonality of the two parts
