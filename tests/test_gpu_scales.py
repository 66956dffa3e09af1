"""Blocks whose entries' squares leave the range of their type, beside ordinary and
zero ones in the same batch: the projection and the eigenvalues scale with the
block.  Both sides are within a few times the order's root in u ||W||_F of the
exact result (order 32: 7 u in float, 9 u in double), so 64 u bounds their
difference."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = np.array([1, 2, 3, 4, 7, 8, 12, 16, 20, 27, 32, 5], np.int32)


@pytest.mark.parametrize("eig", [False, True])
@pytest.mark.parametrize("dtype,power", [("float32", k) for k in (-110, -90, -75, 0, 62, 100)]
                         + [("float64", k) for k in (-900, -520, 505, 900)])
def test_scales(dtype, power, eig):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_05058_gb300 import cdsdp
    rng = np.random.default_rng(5)
    dt = getattr(torch, dtype)
    u = 2.0 ** (-24 if dtype == "float32" else -53)
    off = np.concatenate([[0], np.cumsum(SIZES * (SIZES + 1) // 2)]).astype(np.int32)
    eo = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int32)
    vo = np.concatenate([[0], np.cumsum(SIZES * SIZES)]).astype(np.int32)
    W = rng.standard_normal(off[-1]).astype(np.float32).astype(np.float64)
    W[off[-2]:] = 0.0  # a zero block
    scaled = np.where(np.arange(len(W)) < off[-3], W * 2.0 ** power, W)  # the last but one as it is
    t = lambda a: torch.tensor(a, device="cuda")

    def run(w):
        a = (torch.tensor(w, dtype=dt, device="cuda"), t(off), t(SIZES))
        if not eig:
            return cdsdp.psd_project(*a).cpu().numpy().astype(np.float64), None
        X, lam, _ = cdsdp.psd_project(*a, t(eo), t(vo), want_eig=True)
        return X.cpu().numpy().astype(np.float64), lam.cpu().numpy().astype(np.float64)

    ref, lref = run(W)
    got, lgot = run(scaled)
    for k, s in enumerate(SIZES):
        f = 2.0 ** power if k < len(SIZES) - 2 else 1.0
        i, j = slice(off[k], off[k + 1]), slice(eo[k], eo[k + 1])
        bound = 64 * u * max(np.sqrt(2) * np.linalg.norm(W[i]), 1e-300)
        assert np.isfinite(got[i]).all() and np.abs(got[i] / f - ref[i]).max() <= bound, (k, s)
        if eig:
            assert np.abs(np.sort(lgot[j]) / f - np.sort(lref[j])).max() <= bound, (k, s)
