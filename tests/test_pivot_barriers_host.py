"""k_pivot_pos.cu's roles (bulk, chain, auxiliary warps) each run the rounds in a
branch of their own: what they meet at inside them has a thread count, and is no
__syncthreads(), which the whole block has to reach in one place."""
from __future__ import annotations

import os
import re

SRC = os.path.join(os.path.dirname(__file__), "..", "paper_2608_28952_gb300", "csrc", "k_pivot_pos.cu")


def test_no_syncthreads_inside_the_roles():
    src = open(SRC).read()
    lambdas = dict(re.findall(r"auto (\w+) = \[&\][^{]*\{(.*?)\n    \};", src, re.S))
    assert {"sync_all", "loaded", "may_store", "rounds", "rotate_v"} <= set(lambdas)
    with_bar = {k for k, v in lambdas.items() if "__syncthreads" in v}
    roles = src[src.index("if (role == 0) {"):src.index("// ---- the final diagonal, hi + lo rounded once")]
    assert "__syncthreads" not in roles
    for name in re.findall(r"\b(\w+)\(", roles + lambdas["rounds"]):
        assert name not in with_bar, name
