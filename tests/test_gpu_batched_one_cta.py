"""The blocked batched EVD in FP64 with one CTA per matrix against several: a batch
of equal orders, a multiple of what the GPU holds at once, for which the rule
(played through here) takes one CTA each whatever the occupancy, holds the
matrices of a small batch, which takes several; and the small batch against
LAPACK."""
from __future__ import annotations

import heapq

import numpy as np
import pytest

import jacobi_inputs as gen

SMS, N = 152, 353      # order above the other routes' (320), no multiple of the block


def _ctas(orders, grid):
    """blk_cluster's rule for FP64: the fewest CTAs per matrix whose queue, longest
    first, ends within 0.9 of the best so far."""
    best = pick = None
    for C, gain in ((1, 1.0), (2, 1.96), (4, 3.25), (8, 4.85)):
        ends = []
        for n in sorted(orders, reverse=True):
            t = n ** 2.93 / gain
            heapq.heappush(ends, t + (heapq.heappop(ends) if len(ends) == max(1, grid // C) else 0.0))
        if best is None or max(ends) < 0.9 * best:
            best, pick = max(ends), C
    return pick


def _few():
    few = [gen.sym_gaussian(N + 32 * i, 43, i) for i in range(3)]
    few[1][5, 3] = np.nan
    return few


def _many(sms):
    return _few() + [gen.sym_gaussian(N, 44)] * (12 * sms - 3)      # 12: a multiple of 1, 2, 3 and 4 CTAs per SM


@pytest.mark.parametrize("sms", [148, SMS, 160])
@pytest.mark.parametrize("per_sm", [1, 2, 3, 4])
def test_the_batches_take_one_and_several(sms, per_sm):
    assert _ctas([a.shape[0] for a in _many(sms)], sms * per_sm) == 1
    assert _ctas([a.shape[0] for a in _few()], sms * per_sm) == 8


@pytest.mark.gpu
@pytest.mark.parametrize("vec", [True, False])
def test_one_cta_each_gives_the_same_bits(vec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_28952_gb300 as jg
    dt = torch.float64

    def solve(mats, max_sweeps):
        dev = {id(a): jg.colmajor(a, device="cuda", dtype=dt) for a in mats}      # (A is read only)
        As = [dev[id(a)] for a in mats]
        ws = [torch.empty(a.shape[0], dtype=dt, device="cuda") for a in mats]
        Qs = [jg.colmajor_empty(a.shape[0], a.shape[0], dt, "cuda") for a in mats] if vec else None
        info = torch.full((len(mats),), -7, dtype=torch.int32, device="cuda")
        rc, _ = jg.jacobi_syev_batched(As, ws, Qs, info, jg.params(want_vectors=int(vec), max_sweeps=max_sweeps))
        assert rc == 0
        return ws, Qs, info.cpu().tolist()

    few, many = _few(), _many(torch.cuda.get_device_properties(0).multi_processor_count)
    ws1, Qs1, i1 = solve(few, 2)
    ws2, Qs2, i2 = solve(many, 2)
    assert i1 == [2, -100, 2] and i2[:3] == i1 and all(v == 2 for v in i2[3:])
    for i in (0, 2):
        assert torch.equal(ws1[i], ws2[i])
        assert not vec or torch.equal(Qs1[i], Qs2[i])
    del ws2, Qs2
    ws, Qs, info = solve(few, 60)
    assert info == [0, -100, 0]
    for i in (0, 2):      # a few hundred roundings of the norm, as the batched tests take it
        A = torch.from_numpy(np.tril(few[i]) + np.tril(few[i], -1).T).cuda()
        norm = float(torch.linalg.matrix_norm(A))
        assert float((ws[i] - torch.linalg.eigvalsh(A)).abs().max()) <= 1e-13 * norm
        if vec:
            assert float(torch.linalg.matrix_norm(A @ Qs[i] - Qs[i] * ws[i])) <= 1e-12 * norm
            eye = torch.eye(A.shape[0], dtype=dt, device="cuda")
            assert float(torch.linalg.matrix_norm(Qs[i].T @ Qs[i] - eye)) <= 1e-13 * A.shape[0]
