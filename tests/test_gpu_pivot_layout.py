"""The pivot solves' position layout (k_pivot_pos.cu): quads that move from
round to round, over the edges of the layout: the smallest pivots (one and two
pairs), odd block sizes, quad counts just below and above a thread's share
(128, 256, 512, 1024 quads per CTA), one and two buffers of the quads, and
every cluster size, against the oracle's step on well separated pivots; and, on
the CPU, the moves themselves against the round-robin order's definition."""
from __future__ import annotations

import numpy as np
import pytest

import jacobi_inputs as gen
import oracle


@pytest.fixture(scope="module")
def jg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_28952_gb300 as m
    m.lib()
    return m


@pytest.mark.gpu
@pytest.mark.parametrize("cl", [None, 1, 2, 4, 8, 16])
@pytest.mark.parametrize("b", [1, 2, 3, 8, 16, 17, 24, 32, 33, 45, 46, 64, 72, 128])
def test_step_at_the_layouts_edges(jg, monkeypatch, b, cl):
    import torch
    if cl is not None:
        monkeypatch.setenv("JACOBI_PIVOT_CLUSTER", str(cl))   # (an unusable size falls back to the automatic one)
    np_, s = 4 * b, 1
    A0 = np.asfortranarray(np.diag(np.linspace(1.0, 2.0 * np_, np_)) + 0.05 * gen.sym_gaussian(np_, 3100 + b))
    pairs = oracle.ordering(0, np_ // b)[s]
    A_or, Q_or, _ = oracle.syev_step(A0, np.eye(np_), b, pairs)
    A, Q = (jg.colmajor(x, device="cuda", dtype=torch.float64) for x in (A0, np.eye(np_)))
    assert jg.jacobi_syev_step(A, Q, s, jg.params(b=b)) == 0
    # the bounds of the step parity tests: rounding, on pivots whose eigenvalues are a unit apart
    assert np.abs(A.cpu().numpy() - A_or).max() <= 1e-13 * np.abs(A0).max()
    assert np.abs(Q.cpu().numpy() - Q_or).max() <= 1e-13


def _quad_number(i, j, h):
    m, K = i + j, 2 * (h - 1)
    off = m * m // 4 if m <= h - 1 else h * (h - 1) // 2 - (K - m + 1) ** 2 // 4
    return off + ((j - i - 1) >> 1)


def _next(t, e, h):
    """Side and pair of the position that the index at (t, e) moves to."""
    if h == 1:
        return t, e
    p = e if t == 0 else 2 * h - 1 - e
    if p > 0:
        p = 2 * h - 1 if p == 1 else p - 1
    return (1, 2 * h - 1 - p) if p >= h else (0, p)


@pytest.mark.parametrize("h", [1, 2, 3, 4, 5, 16, 33, 64, 128])
def test_moves_follow_the_round_robin_order(h):
    k = 2 * h
    index = lambda pos, r: 0 if pos == 0 else 1 + (pos - 1 + r) % (k - 1)  # noqa: E731
    quads = sorted(_quad_number(i, j, h) for j in range(h) for i in range(j))
    assert quads == list(range(h * (h - 1) // 2))
    sides = [(t, e) for t in (0, 1) for e in range(h)]
    to = {s: _next(*s, h) for s in sides}
    assert sorted(to.values()) == sorted(sides)
    pos = lambda t, e: e if t == 0 else k - 1 - e  # noqa: E731
    for s, d in to.items():
        for r in range(0, k - 1, max(1, k // 5)):
            assert index(pos(*s), r) == index(pos(*d), r + 1)
    source = {d: s for s, d in to.items()}
    for e in range(h if h > 1 else 0):     # the entry of the next round's pair e: one entry of one quad
        (ta, a), (tb, c) = source[(0, e)], source[(1, e)]
        want = ((0, 0), (0, 1)) if e == 0 else ((1, h - 1), (1, h - 2)) if e == h - 1 else ((0, e + 1), (1, e - 1))
        assert ((ta, a), (tb, c)) == want
