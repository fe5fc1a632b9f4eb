"""The statistics of a solve whose Q (V) updates run beside the pivot solves: their
time and launches count with the other updates', so flops_update / ms_update stays
a rate that the FP64 unit can reach."""
from __future__ import annotations

import pytest

import bench

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def jg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_28952_gb300 as m
    m.lib()
    return m


@pytest.mark.parametrize("n,b,emu", [(1536, 64, False), (1000, 32, False), (1024, 64, True)])
def test_evd(jg, n, b, emu):
    import torch
    M = torch.randn((n, n), generator=torch.Generator().manual_seed(n), dtype=torch.float64)
    A = (0.5 * (M + M.t())).cuda()
    kw = dict(b=b, **(dict(precision=jg.PREC_FP64_EMU) if emu else {}))
    jg.syev(A.clone(), **kw)
    st = jg.syev(A.clone(), **kw)[-1]
    S = bench.padded_np(n, b) // b - 1
    assert st.update_launches == 2 * S * st.sweeps and st.pivot_launches == S * st.sweeps
    # a step: pivots, A, Q and (but for the last) the pause; a sweep: the stop sums; a call: four more
    assert st.launches == (4 * S - 1 + 1) * st.sweeps + 4
    if not emu:
        assert st.flops_update / st.ms_update / 1e9 <= bench.FP64_PEAK_TFLOPS, st
    # Q's share of the updates' flops is a third or more: without it the time is less
    A_only = jg.syev(A.clone(), want_vectors=False, **kw)[-1]
    assert st.ms_update / st.sweeps >= 1.3 * A_only.ms_update / A_only.sweeps


def test_svd(jg):
    import torch
    m, n, b = 2000, 512, 32
    G = torch.randn((m, n), generator=torch.Generator().manual_seed(n), dtype=torch.float64).cuda()
    jg.gesvd(G.clone(), b=b, svd_qr=0)
    st = jg.gesvd(G.clone(), b=b, svd_qr=0)[-1]
    S = n // b - 1
    assert st.update_launches == 3 * S * st.sweeps and st.pivot_launches == S * st.sweeps
    assert st.launches == (6 * S - 1) * st.sweeps + 4
    assert st.flops_update / st.ms_update / 1e9 <= bench.FP64_PEAK_TFLOPS, st


@pytest.mark.parametrize("n,b,emu", [(1536, 64, False), (2048, 64, True)])
def test_update_time_within_the_call(jg, n, b, emu):
    """Q's and A's updates that run at the same time count it once: the updates' time
    is no more than the call's."""
    import torch
    M = torch.randn((n, n), generator=torch.Generator().manual_seed(n), dtype=torch.float64)
    A = (0.5 * (M + M.t())).cuda()
    kw = dict(b=b, **(dict(precision=jg.PREC_FP64_EMU) if emu else {}))
    jg.syev(A.clone(), **kw)
    st = jg.syev(A.clone(), **kw)[-1]
    assert 0 < st.ms_update <= st.ms_total and 0 < st.ms_pivot <= st.ms_total
