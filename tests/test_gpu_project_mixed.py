"""The standalone projection of batches that several kernels share (orders up to
32, 33..64, 65..96 and 97..128): the kernels run beside each other, so a batch of
few blocks takes less than its parts one after the other; the blocks of a kernel
equal those of a batch that it has to itself, bit for bit, also in place, in a
captured graph, and read by the next operation on the stream."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _batch(torch, sizes, dtype, seed):
    sizes = np.asarray(sizes, np.int32)
    off = np.concatenate([[0], np.cumsum(sizes.astype(np.int64) * (sizes + 1) // 2)]).astype(np.int32)
    W = np.random.default_rng(seed).standard_normal(off[-1])
    return (torch.tensor(W, dtype=getattr(torch, dtype), device="cuda"), torch.tensor(off, device="cuda"),
            torch.tensor(sizes, device="cuda"))


def _torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _time(torch, f):
    for _ in range(3):
        f()
    ts = []
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(5):
            f()
        b.record()
        b.synchronize()
        ts.append(a.elapsed_time(b))
    return min(ts)


@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_parts_run_beside_each_other(dtype):
    torch = _torch()
    from paper_1707_05058_gb300 import cdsdp
    small, large = [32, 31, 20, 25] * 3, [40, 38, 33, 36] * 2
    t = {k: _time(torch, lambda b=_batch(torch, s, dtype, 3): cdsdp.psd_project(*b))
         for k, s in (("small", small), ("large", large), ("both", small + large))}
    assert t["both"] <= 0.85 * (t["small"] + t["large"]), t


@pytest.mark.parametrize("dtype,sizes", [("float32", [128, 97, 96, 65, 64, 33, 32, 9, 2, 1] * 3), ("float32", [70, 5] * 200),
                                         ("float64", [64, 49, 33, 32, 17, 8, 2, 1] * 4), ("float64", [34, 3] * 300)])
def test_parts_equal_their_own_batch(dtype, sizes):
    torch = _torch()
    from paper_1707_05058_gb300 import cdsdp
    W, off, sz = _batch(torch, sizes, dtype, 4)
    X = cdsdp.psd_project(W, off, sz)
    twice = X * 2  # the next operation on the stream
    o, n = off.cpu().numpy(), np.asarray(sizes)
    for lo, hi in ((1, 32), (33, 64), (65, 96), (97, 128)):
        ks = np.flatnonzero((n >= lo) & (n <= hi))
        if not len(ks):
            continue
        ent = torch.tensor(np.concatenate([np.arange(o[k], o[k + 1]) for k in ks]), device="cuda")
        po = np.concatenate([[0], np.cumsum([o[k + 1] - o[k] for k in ks])]).astype(np.int32)
        part = cdsdp.psd_project(W[ent], torch.tensor(po, device="cuda"), torch.tensor(n[ks].astype(np.int32), device="cuda"))
        assert torch.equal(X[ent], part) and torch.equal(twice[ent], part * 2), (lo, hi)


def test_in_a_captured_graph():
    torch = _torch()
    from paper_1707_05058_gb300 import cdsdp
    import ctypes
    W, off, sz = _batch(torch, [128, 96, 64, 40, 32, 7] * 4, "float32", 5)
    ref = cdsdp.psd_project(W, off, sz)
    Y, Z = W.clone(), torch.empty_like(W)
    p = lambda t: ctypes.c_void_p(t.data_ptr())

    def body():  # in place, then read
        st = cdsdp._lib.cdsdp_psd_project(sz.numel(), p(off), p(sz), 128, p(Y), p(Y), None, None, None, None, cdsdp.FP32,
                                          30, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert st == 0
        Z.copy_(Y)

    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        body()
    for _ in range(3):
        Y.copy_(W)
        g.replay()
        assert torch.equal(Z, ref)
