"""The FP64 Gram blocks' sums are fixed by the shape: a call whose workspace has
room only for one partial per 512 rows gives the bits of one that has room for
every panel's (64 to 256 rows each)."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,b", [(1000, 200, 16), (700, 48, 8), (513, 160, 40), (3000, 72, 12)])
def test_same_bits_at_any_room(monkeypatch, m, n, b):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_28952_gb300 as jg
    G = torch.randn((m, n), generator=torch.Generator().manual_seed(m), dtype=torch.float64).cuda()

    def call():
        U = jg.colmajor(G.clone())
        s = torch.empty(n, dtype=torch.float64, device="cuda")
        V = jg.colmajor_empty(n, n, torch.float64, "cuda")
        rc, st = jg.jacobi_gesvd(U, s, V, jg.params(b=b, svd_qr=0))
        return rc, (U, s, V), st

    rc, want, st = call()
    assert rc == 0
    lo, hi = 0, 1 << 28
    while hi - lo > 4096:      # the least workspace that the call runs in
        mid = (lo + hi) // 2
        monkeypatch.setenv("JACOBI_WORKSPACE_LIMIT", str(mid))
        lo, hi = (lo, mid) if call()[0] == 0 else (mid, hi)
    monkeypatch.setenv("JACOBI_WORKSPACE_LIMIT", str(hi))
    rc, got, st1 = call()
    assert rc == 0 and st1.sweeps == st.sweeps
    for x, y in zip(want, got):
        assert torch.equal(x, y)
