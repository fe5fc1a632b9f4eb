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
