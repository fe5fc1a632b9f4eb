"""The pivot solves over the cluster sizes, powers of two or not, with several inner
sweeps and with V in FP32: one result, bit for bit, and (FP64) the oracle's
step."""
from __future__ import annotations

import numpy as np
import pytest

import jacobi_inputs as gen
import oracle

pytestmark = pytest.mark.gpu

SIZES = {32: (1, 2, 3, 4, 5, 7, 8), 64: (1, 2, 3, 5, 6, 7, 8, 11, 13, 16)}


@pytest.fixture(scope="module")
def jg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_28952_gb300 as m
    m.lib()
    return m


@pytest.mark.parametrize("b", [32, 64])
def test_fp64_steps_with_several_inner_sweeps(jg, monkeypatch, b):
    import torch
    np_, s = 4 * b, 1
    A0 = np.asfortranarray(np.diag(np.linspace(1.0, 2.0 * np_, np_)) + 0.05 * gen.sym_gaussian(np_, 3500 + b))
    A_or, Q_or, _ = oracle.syev_step(A0, np.eye(np_), b, oracle.ordering(0, np_ // b)[s], inner_max=3)
    first = None
    for C in SIZES[b]:
        monkeypatch.setenv("JACOBI_PIVOT_CLUSTER", str(C))
        A, Q = (jg.colmajor(x, device="cuda", dtype=torch.float64) for x in (A0, np.eye(np_)))
        assert jg.jacobi_syev_step(A, Q, s, jg.params(b=b, inner_max_sweeps=3)) == 0
        # the bounds of the step parity tests: rounding, on pivots whose eigenvalues are a unit apart
        assert np.abs(A.cpu().numpy() - A_or).max() <= 1e-13 * np.abs(A0).max(), C
        assert np.abs(Q.cpu().numpy() - Q_or).max() <= 1e-13, C
        first = first or (A, Q)
        assert torch.equal(A, first[0]) and torch.equal(Q, first[1]), C


@pytest.mark.parametrize("b", [32, 64])
def test_lowp_steps(jg, monkeypatch, b):
    import torch
    A0 = gen.sym_gaussian(4 * b, 3600 + b).astype(np.float32)
    first = None
    for C in SIZES[b]:
        monkeypatch.setenv("JACOBI_PIVOT_CLUSTER", str(C))
        A, Q = (jg.colmajor(x, device="cuda", dtype=torch.float32) for x in (A0, np.eye(4 * b, dtype=np.float32)))
        for s in (0, 1):
            assert jg.jacobi_syev_step_lowp(A, Q, s, jg.params(b=b, precision=jg.PREC_MIXED_BF16X3)) == 0
        first = first or (A, Q)
        assert torch.equal(A, first[0]) and torch.equal(Q, first[1]), C
