"""Algorithm 3 on a direct sum whose larger summands have several blocks each in
the per-component reductions (from 1,024 pattern entries on), one of them with a
last part that is no multiple of the others, next to summands with one block;
against the oracle's Algorithm 3 on each summand alone (FP64; data normalised).
Residual rows, tau and kappa after 20 iterations: rtol 1e-7 (the two differ by
rounding order, about 1e-12 an iterate, and the iteration is nonexpansive); runs
to 1e-3, where a component that has stopped stays as it is while others go on."""
import dataclasses

import numpy as np
import pytest

from oracle import admm
from paper_1707_05058_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _normalised(q):
    w = np.where(q.C_row == q.C_col, 1.0, 2.0)
    return dataclasses.replace(q, C_val=q.C_val / np.sqrt(np.sum(w * q.C_val ** 2)), b=q.b / np.linalg.norm(q.b))


def _parts():
    return [_normalised(q) for q in (W.banded(400, 5, 8, seed=1), W.banded(12, 3, 2, seed=2, density=0.5),
                                     W.block_arrow(40, 5, 6, 10, seed=3), W.banded(171, 6, 5, seed=4))]


def _torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_twenty_iterations():
    _torch()
    from paper_1707_05058_gb300 import cdsdp
    parts = _parts()
    P = cdsdp.Problem(W.direct_sum(parts)).bind(max_iter=20)
    out = P.solve("hsde", eps=0.0, max_iter=20, precision="fp64")
    it, st, res = P.component_results()
    r, c = P.pattern()
    vo = mo = 0
    for j, q in enumerate(parts):
        dp = admm.decompose(q)
        ref = admm.hsde_admm(dp, eps=0.0, max_iter=20)
        assert it[j] == 20
        np.testing.assert_allclose(res[j, :6], ref.hist[-1, :6], rtol=1e-7, atol=1e-10)
        np.testing.assert_allclose(out["y"][mo:mo + q.m], ref.y, rtol=1e-7, atol=1e-9)
        mask = (c >= vo) & (c < vo + q.n)
        np.testing.assert_allclose(out["X"][mask], dp.lower_values(ref.X), rtol=1e-7, atol=1e-9)
        vo += q.n
        mo += q.m


def test_components_that_stop():
    _torch()
    from paper_1707_05058_gb300 import cdsdp
    parts = _parts()
    P = cdsdp.Problem(W.direct_sum(parts)).bind(max_iter=3000)
    out = P.solve("hsde", eps=1e-3, max_iter=3000, precision="fp64")
    it, st, res = P.component_results()
    mo = 0
    for j, q in enumerate(parts):
        _, ref = admm.solve(q, "hsde", eps=1e-3, max_iter=3000)
        assert st[j] == ref.status and abs(int(it[j]) - ref.iters) <= 1, (j, it[j], ref.iters)
        if int(it[j]) == ref.iters:
            np.testing.assert_allclose(out["y"][mo:mo + q.m], ref.y, rtol=1e-6, atol=1e-8)
        mo += q.m
    assert len(set(it.tolist())) > 1  # some stopped while others went on
