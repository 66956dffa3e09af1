"""cdsdp_psd_project on batches whose orders differ, at the edges of its kernel
families (orders 4, 8, 16 and 32 for lanes per block, 33, 64, 65, 96, 97 and
128 for thread blocks) and of its runs of entries, against numpy's float64
eigendecomposition.  Bound: 40 u sqrt(s) ||W||_F (u the unit roundoff): a few
tens of roundings of size u per eigenvector row."""
import numpy as np
import pytest

from paper_1707_05058_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = [([1], 32), ([2, 1, 3, 4, 5], 32), ([8, 9, 16, 17, 1, 32, 31, 20, 21, 24, 25, 28, 29], 32),
         (list(range(1, 33)) * 11, 32), ([7] * 700, 32), ([11] * 305, 32), ([33, 32, 64, 1, 36, 37, 60, 61, 40, 41, 52], 32),
         ([65, 64, 33, 96, 97, 128, 12, 100], 32), ([1, 2, 3], 64), (list(range(1, 33)), 64),
         ([33, 2, 64, 40, 17], 64), ([12, 16, 13, 5], 64)]


@pytest.mark.parametrize("sizes,bits", CASES, ids=lambda v: f"{len(v)}x{max(v)}" if isinstance(v, list) else f"f{v}")
def test_ragged_orders(sizes, bits):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_05058_gb300 import cdsdp
    sizes = np.asarray(sizes)
    off = np.concatenate([[0], np.cumsum(sizes * (sizes + 1) // 2)])
    rng = np.random.default_rng(int(sizes.sum()))
    w = W._f32(rng.standard_normal(int(off[-1])))
    if len(sizes) > 2:
        w[off[1]:off[2]] = 0.0  # a zero block
    dt = torch.float64 if bits == 64 else torch.float32
    dev = lambda a, t: torch.tensor(a, dtype=t, device="cuda")  # noqa: E731
    got = cdsdp.psd_project(dev(w, dt), dev(off, torch.int32), dev(sizes, torch.int32)).cpu().numpy().astype(float)
    u = 2.0 ** (-53 if bits == 64 else -24)
    for k, s in enumerate(sizes):
        i, j = np.tril_indices(s)
        o = np.lexsort((i, j))
        i, j = i[o], j[o]
        B = np.zeros((s, s))
        B[i, j] = B[j, i] = w[off[k]:off[k + 1]]
        lam, V = np.linalg.eigh(B)
        P = (V * np.maximum(lam, 0.0)) @ V.T
        G = np.zeros((s, s))
        G[i, j] = G[j, i] = got[off[k]:off[k + 1]]
        assert np.linalg.norm(G - P) <= 40 * u * np.sqrt(s) * np.linalg.norm(B) + 1e-300, (k, s)
