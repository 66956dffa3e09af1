"""Where the sweeps of a projection end: nearly diagonal blocks W = diag(l) + F on
both sides of the line sum over i < j of F_ij^2 / (|l_i| + |l_j|) = u ||W||_F / 2,
with eigenvalues that straddle zero in pairs, cluster at zero or are spread out.

Below the line no sweep runs and the result is P(W) to first order in F, from V =
I, so its rounding is that of one entry.  The second-order term is sum over k of
F_ik F_kj f[l_i, l_k, l_j] with f = max(., 0), and its divided difference is at
most 1 / sqrt((|l_i| + |l_k|) (|l_k| + |l_j|)), so the term's Frobenius norm is at
most twice that sum, u ||W||_F; with one u for the rounding and the terms after it
the bound is 2 u ||W||_F.  Above the line sweeps run: (4 + order / 4) u ||W||_F (a
random block of order 32 is 7 u off, of order 128 18 u).

The reference has more digits than the type: float64 for float, 40 decimal digits
for double."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _blocks(dtype, sizes, times, rng):
    """Blocks whose sum is `times` u ||W||_F / 2."""
    u = 2.0 ** (-24 if dtype == "float32" else -53)
    out = []
    for s in sizes:
        for kind in ("straddle", "cluster", "spread"):
            if kind == "straddle":
                a = 10.0 ** rng.uniform(np.log10(u) - 1, 0, (s + 1) // 2)
                lam = np.concatenate([a, -a])[:s] * 10.0 ** rng.uniform(-0.3, 0.3, s)
                lam[0] = 1.0
            elif kind == "cluster":
                lam = 3 * u * rng.standard_normal(s)
                lam[:max(1, s // 2)] = rng.uniform(0.1, 1.0, max(1, s // 2))
            else:
                lam = rng.standard_normal(s)
            lam /= np.linalg.norm(lam)
            w = np.abs(lam)[:, None] + np.abs(lam)[None, :]
            F = np.tril(rng.standard_normal((s, s)) * np.sqrt(w), -1)
            F *= np.sqrt(times * u / 2 / np.sum(F * F / w))
            M = (np.diag(lam) + F).astype(dtype).astype(np.float64)
            out.append(M + np.tril(M, -1).T)
    return out


def _exact(M, dtype):
    """P(M) as an array of objects or float64, wide enough to measure a result of `dtype`."""
    if dtype == "float32":
        lam, V = np.linalg.eigh(M)
        return (V * np.maximum(lam, 0)) @ V.T
    mp = pytest.importorskip("mpmath")
    with mp.workdps(40):
        E, Q = mp.eigsy(mp.matrix(M.tolist()))
        Q = np.array(Q.tolist(), dtype=object).reshape(len(M), -1)
        return (Q * np.array([e if e > 0 else mp.mpf(0) for e in E], dtype=object)) @ Q.T


@pytest.mark.parametrize("times", [0.9, 4.0])
@pytest.mark.parametrize("dtype,sizes", [("float32", (3, 4, 5, 8, 12, 17, 24, 32)), ("float32", (33, 48, 64, 90, 128)),
                                         ("float64", (3, 4, 5, 8, 12))])
def test_nearly_diagonal(dtype, sizes, times):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1707_05058_gb300 import cdsdp
    blocks = _blocks(dtype, sizes, times, np.random.default_rng(len(sizes)))
    n = np.array([len(B) for B in blocks], np.int32)
    off = np.concatenate([[0], np.cumsum(n * (n + 1) // 2)]).astype(np.int32)
    W = np.concatenate([B[np.triu_indices(len(B))] for B in blocks])  # symmetric: upper rows are lower columns
    X = cdsdp.psd_project(torch.tensor(W, dtype=getattr(torch, dtype), device="cuda"), torch.tensor(off, device="cuda"),
                          torch.tensor(n, device="cuda")).cpu().numpy().astype(np.float64)
    u = 2.0 ** (-24 if dtype == "float32" else -53)
    for k, B in enumerate(blocks):
        s = len(B)
        iu = np.triu_indices(s)
        d = X[off[k]:off[k + 1]] - _exact(B, dtype)[iu]
        err = float(sum(np.where(iu[0] == iu[1], 1, 2) * d * d)) ** 0.5 / np.linalg.norm(B) / u
        assert err <= (2.0 if times < 1 else 4.0 + s / 4), (s, k % 3, err)
