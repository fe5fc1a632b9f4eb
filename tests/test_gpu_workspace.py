"""The workspace pool: calls from several host threads on streams of their own
share it and give the results of calls made one after the other."""
from __future__ import annotations

import threading

import numpy as np
import pytest

import jacobi_inputs as gen

pytestmark = pytest.mark.gpu


def test_threads_and_streams_share_the_pool():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_28952_gb300 as jg
    mats = [gen.sym_gaussian(n, 51, n) for n in (96, 130, 200, 257)]
    want = [jg.syev(a, b=16) for a in mats]
    got, errors = [None] * len(mats), []

    def work(i):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for _ in range(3):
                    got[i] = jg.syev(mats[i], b=16, stream=s)
            s.synchronize()
        except Exception as e:   # noqa: BLE001 (reported below)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(mats))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for a, b in zip(want, got):
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
        assert np.isfinite(b[0].cpu().numpy()).all()


def _least_limit(monkeypatch, call, alloc_err):
    """The smallest workspace cap under which `call` still runs, to 4 KB."""
    lo, hi = 0, 1 << 30
    while hi - lo > 4096:
        mid = (lo + hi) // 2
        monkeypatch.setenv("JACOBI_WORKSPACE_LIMIT", str(mid))
        rc = call()
        assert rc in (0, alloc_err)
        lo, hi = (lo, mid) if rc == 0 else (mid, hi)
    monkeypatch.setenv("JACOBI_WORKSPACE_LIMIT", str(hi))
    assert call() == 0
    return hi


def test_evd_runs_without_room_for_the_overlap_buffers(monkeypatch):
    """n = 512, b = 32 overlaps Q's update with the next pivots through a second
    set of transforms (8 pairs x 2 x 64 x 64 doubles).  A call that has room for
    one set only runs one after the other, to the same bits: beyond the four
    matrices and one set it asks for less than a quarter of a set."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_28952_gb300 as jg
    n, b = 512, 32
    A = torch.from_numpy(gen.sym_gaussian(n, 61, n)).cuda()
    want = jg.syev(A.clone(), b=b)   # (a column-major argument is solved in place)
    out = {}

    def call():
        w = torch.empty(n, dtype=torch.float64, device="cuda")
        Q = jg.colmajor_empty(n, n, torch.float64, "cuda")
        rc, _ = jg.jacobi_syev(jg.colmajor(A.clone()), w, Q, jg.params(b=b))
        out.update(w=w, Q=Q)
        return rc

    one = 8 * (n // (2 * b)) * 2 * (2 * b) ** 2
    assert _least_limit(monkeypatch, call, jg.ERR_ALLOC) < 4 * 8 * n * n + one + one // 4
    assert torch.equal(out["w"], want[0]) and torch.equal(out["Q"], want[1])


def test_svd_runs_without_room_for_small_gram_panels(monkeypatch):
    """1000 x 200, b = 16 takes 64-row Gram panels; with room for 512-row ones
    only (two per pair), it takes those."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_28952_gb300 as jg
    m, n, b = 1000, 200, 16
    G = torch.randn((m, n), generator=torch.Generator().manual_seed(5), dtype=torch.float64).cuda()
    out = {}

    def call():
        U = jg.colmajor(G.clone())
        s = torch.empty(n, dtype=torch.float64, device="cuda")
        V = jg.colmajor_empty(n, n, torch.float64, "cuda")
        rc, _ = jg.jacobi_gesvd(U, s, V, jg.params(b=b, svd_qr=0))
        out.update(U=U, s=s, V=V)
        return rc

    npad, k = 224, 2 * b
    pairs = npad // k
    need = 8 * (2 * m * npad + 2 * npad * npad + pairs * 2 * k * k + pairs * 2 * k * k)
    assert _least_limit(monkeypatch, call, jg.ERR_ALLOC) < need + 16384
    # one-sided Jacobi in FP64: a few hundred roundings of each column's norm
    ref = torch.linalg.svdvals(G)
    assert float((out["s"] - ref).abs().max()) <= 1e3 * 2.0 ** -53 * float(ref[0])
    back = (out["U"] * out["s"]) @ out["V"].t()
    assert float((back - G).norm()) <= 1e3 * 2.0 ** -53 * n ** 0.5 * float(ref[0])
