"""The blocked batched EVD with several CTAs per matrix (small batches of large
orders): every item is computed by the same operations whichever CTA takes it,
so eigenvalues and vectors are those of one CTA per matrix, bit for bit.  A
batch large enough to be played through with one CTA each holds the same
matrices as small ones; ragged orders, a non-finite matrix, both types, with
and without vectors."""
from __future__ import annotations

import numpy as np
import pytest

import jacobi_inputs as gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def jg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2608_28952_gb300 as m
    m.lib()
    return m


def _solve(jg, mats, dt, vec):
    import torch
    As = [jg.colmajor(a, device="cuda", dtype=dt) for a in mats]
    ws = [torch.empty(a.shape[0], dtype=dt, device="cuda") for a in mats]
    Qs = [jg.colmajor_empty(a.shape[0], a.shape[0], dt, "cuda") for a in mats] if vec else None
    info = torch.full((len(mats),), -7, dtype=torch.int32, device="cuda")
    rc, _ = jg.jacobi_syev_batched(As, ws, Qs, info, jg.params(want_vectors=int(vec), max_sweeps=4),
                                   f32=dt == torch.float32)
    assert rc == 0
    return ws, Qs, info.cpu().tolist()


@pytest.mark.parametrize("f32", [True, False])
@pytest.mark.parametrize("vec", [True, False])
def test_split_matrices_match_one_cta_each(jg, f32, vec):
    import torch
    dt = torch.float32 if f32 else torch.float64
    n = 353 if not f32 else 321      # above the other routes' orders; no multiple of the block
    few = [gen.sym_gaussian(n + 32 * i, 41, i) for i in range(3)]
    few[1][5, 3] = np.nan
    many = few + [few[0]] * 330       # more than two per CTA of the GPU: one CTA each
    ws1, Qs1, i1 = _solve(jg, few, dt, vec)
    ws2, Qs2, i2 = _solve(jg, many, dt, vec)
    assert i1 == [4, -100, 4] and i2[:3] == i1 and all(v == 4 for v in i2[3:])
    for i in (0, 2):
        assert torch.equal(ws1[i], ws2[i])
        if vec:
            assert torch.equal(Qs1[i], Qs2[i])
    assert torch.equal(ws1[0], ws2[-1])
