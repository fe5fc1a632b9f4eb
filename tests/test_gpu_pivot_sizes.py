"""Pivot clusters whose CTAs hold the most quads that shared memory takes (2b =
184 and 186 on 2 CTAs, 224 on 3: more than 2048 quads each): a forced size that
fits is used, to the oracle's step (FP64), and to the bits of a larger cluster
(low precision: every entry is computed by the same operations whatever the
cluster).  The block sizes beside them take the next smaller instance."""
from __future__ import annotations

import numpy as np
import pytest

import jacobi_inputs as gen
import oracle

pytestmark = pytest.mark.gpu

SIZES = [(91, 2), (92, 2), (93, 2), (92, 3), (111, 3), (112, 3), (113, 3)]


@pytest.fixture(scope="module")
def jg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_28952_gb300 as m
    m.lib()
    return m


@pytest.mark.parametrize("b,cl", SIZES)
def test_largest_shares(jg, monkeypatch, b, cl):
    import torch
    monkeypatch.setenv("JACOBI_PIVOT_CLUSTER", str(cl))
    np_, s = 4 * b, 1
    A0 = np.asfortranarray(np.diag(np.linspace(1.0, 2.0 * np_, np_)) + 0.05 * gen.sym_gaussian(np_, 3300 + b))
    A_or, Q_or, _ = oracle.syev_step(A0, np.eye(np_), b, oracle.ordering(0, np_ // b)[s])
    A, Q = (jg.colmajor(x, device="cuda", dtype=torch.float64) for x in (A0, np.eye(np_)))
    assert jg.jacobi_syev_step(A, Q, s, jg.params(b=b)) == 0
    # the bounds of the step parity tests: rounding, on pivots whose eigenvalues are a unit apart
    assert np.abs(A.cpu().numpy() - A_or).max() <= 1e-13 * np.abs(A0).max()
    assert np.abs(Q.cpu().numpy() - Q_or).max() <= 1e-13


@pytest.mark.parametrize("b,cl", SIZES)
def test_largest_shares_lowp(jg, monkeypatch, b, cl):
    import torch
    A0 = gen.sym_gaussian(4 * b, 3400 + b).astype(np.float32)
    out = []
    for c in (cl, 4):
        monkeypatch.setenv("JACOBI_PIVOT_CLUSTER", str(c))
        A, Q = (jg.colmajor(x, device="cuda", dtype=torch.float32) for x in (A0, np.eye(4 * b, dtype=np.float32)))
        for s in (0, 1):
            assert jg.jacobi_syev_step_lowp(A, Q, s, jg.params(b=b, precision=jg.PREC_MIXED_BF16X3)) == 0
        out.append((A, Q))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
