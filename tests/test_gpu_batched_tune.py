"""The autotuner's choice for an FP64 batch larger than its sample repeats: the
sample is timed so that the candidates differ (group after group), not by the
longest matrix alone, where the choice was noise."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu


def test_the_choice_repeats(monkeypatch, tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import numpy as np

    import jacobi_inputs as gen
    import paper_2608_28952_gb300 as jg
    monkeypatch.setenv("JACOBI_TUNE_CACHE", str(tmp_path / "cache"))
    ns = np.random.default_rng(5).integers(8, 513, 400).tolist()     # the sample is two matrices per SM
    dev = torch.device("cuda", 0)
    flat, X, _ = gen.batch_flat_torch([(n, n) for n in ns], 3, dev, torch.float64, symmetric=True)
    Y = [torch.empty(n, dtype=torch.float64, device=dev) for n in ns]
    Z = [jg.colmajor_empty(n, n, torch.float64, dev) for n in ns]
    info = torch.zeros(len(ns), dtype=torch.int32, device=dev)
    chosen = []
    for _ in range(3):
        plan = jg.Plan(0, jg.PREC_FP64, ns, p=jg.params(max_sweeps=1))
        plan.autotune(X, Y, Z, info)
        chosen.append(plan.blocking())
        plan.close()
    assert chosen[0] == chosen[1] == chosen[2], chosen
