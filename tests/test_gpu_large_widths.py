"""cdsdp_psd_project_large over its choices of tile width (32, 64 or 128 columns,
or two of them in a batch) and at the edges of a 128-row tile: a block's result
alone and in a batch, where its tiles have another width, bit for bit (an entry
is the same sum at each width), and the same block at other scales."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BATCHES = [[127, 128, 129], [1, 256, 257], [385, 640, 385], [900, 500], [1300, 1052, 943, 245, 129, 1], [700] * 9,
           [512] * 70]


def _blocks(sizes):
    rng = np.random.default_rng(sum(sizes))
    return [rng.standard_normal(s * (s + 1) // 2).astype(np.float32) for s in sizes]


def _project(torch, cdsdp, blocks, sizes):
    got = cdsdp.psd_project_large(torch.tensor(np.concatenate(blocks), device="cuda"), sizes).cpu().numpy()
    return np.split(got, np.cumsum([b.size for b in blocks])[:-1])


@pytest.mark.parametrize("sizes", BATCHES, ids=lambda s: f"{len(s)}x{max(s)}")
def test_widths(sizes):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_05058_gb300 import cdsdp
    blocks = _blocks(sizes)
    out = _project(torch, cdsdp, blocks, sizes)
    for k in range(min(len(sizes), 6)):
        alone = _project(torch, cdsdp, [blocks[k]], [sizes[k]])[0]
        assert np.isfinite(alone).all() and np.array_equal(out[k], alone), (k, sizes[k])


def test_scales_of_the_input():
    """Blocks of very small and very large entries: P(a W) = a P(W) for a power of two, exactly."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_05058_gb300 import cdsdp
    (w,), s = _blocks([200]), [200]
    ref = _project(torch, cdsdp, [w], s)[0]
    for e in (-80, -30, 30, 100):
        a = np.float32(2.0) ** e
        np.testing.assert_array_equal(_project(torch, cdsdp, [w * a], s)[0], ref * a)
