"""The projection of blocks of order 1 to 4 in both precisions, in a batch of their
own and among larger ones: the mean error over many random blocks, in units of
u ||W||_F.  Bounds: the means of a float32 replay of the sweeps with exactly
rounded square roots and quotients (0.69, 1.31, 1.68 at orders 2, 3, 4) and four
standard errors of the mean (0.01 for 4,096 blocks of order 2, 0.025 and 0.03 for
1,024 of orders 3 and 4), rounded up."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BOUND = {1: 0.0, 2: 0.74, 3: 1.41, 4: 1.80}


@pytest.mark.parametrize("with_larger", [False, True])
@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_mean_error(dtype, with_larger):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_05058_gb300 import cdsdp
    rng = np.random.default_rng(31)
    sizes = np.concatenate([np.repeat([1, 2, 3, 4], [64, 4096, 1024, 1024]), [7, 16, 29, 32] if with_larger else []]).astype(np.int32)
    rng.shuffle(sizes)
    off = np.concatenate([[0], np.cumsum(sizes * (sizes + 1) // 2)]).astype(np.int32)
    W = rng.standard_normal(off[-1]).astype(np.float32)
    X = cdsdp.psd_project(torch.tensor(W, dtype=getattr(torch, dtype), device="cuda"), torch.tensor(off, device="cuda"),
                          torch.tensor(sizes, device="cuda")).cpu().numpy()
    u = 2.0 ** (-24 if dtype == "float32" else -53)
    ld = np.longdouble if np.finfo(np.longdouble).eps < 2e-17 else np.float64  # 64 bits or more where there is a wider type
    for s in BOUND:
        if dtype == "float64" and (s > 2 or ld is np.float64):
            continue  # the reference has to be wider than the result: order 2 in closed form only
        err = []
        iu = np.tril_indices(s)
        for k in np.flatnonzero(sizes == s):
            A = np.zeros((s, s), ld)
            A.T[np.triu_indices(s)] = W[off[k]:off[k + 1]]
            A = A + np.tril(A, -1).T
            P = _psd2(A) if s <= 2 else _psd(A)
            B = np.zeros((s, s), ld)
            B.T[np.triu_indices(s)] = X[off[k]:off[k + 1]]
            d = (B - P)[iu]
            w = np.where(iu[0] == iu[1], 1, 2)
            err.append(float(np.sqrt((w * d * d).sum()) / np.sqrt((A * A).sum()) / u))
        assert np.mean(err) <= BOUND[s], (s, np.mean(err))


def _psd(A):
    lam, V = np.linalg.eigh(A.astype(np.float64))
    return (V * np.maximum(lam, 0)) @ V.T


def _psd2(A):
    """max(A, 0) of order 1 or 2: with m the mean and r the half difference of the eigenvalues, by cases."""
    if A.shape[0] == 1:
        return np.maximum(A, 0)
    m, h, q = (A[0, 0] + A[1, 1]) / 2, (A[0, 0] - A[1, 1]) / 2, A[1, 0]
    r = np.sqrt(h * h + q * q)
    if m >= r:
        return A
    if m <= -r:
        return np.zeros_like(A)
    J = np.array([[h, q], [q, -h]], dtype=A.dtype) / r
    return (m + r) / 2 * (np.eye(2, dtype=A.dtype) + J)
