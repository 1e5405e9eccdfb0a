"""Output entries of the longest allowed length on one CTA each.  A plan of
few entries shares them out over units of a few products, so that the folds
of the lazily reduced sums (every 255 or 256 products of a unit) are reached
only by plans of many long entries; a workspace without room for the units'
partial sums makes the plan keep whole entries, which runs them at 1024
products here.  An unfolded sum of d0 and d1 would pass 2^64."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_common import coeff_of, gpu_ctx, gpu_modules
import workloads as W

pytestmark = pytest.mark.gpu


def _whole_plan(api, S, ctx, A, B, C):
    """a plan whose workspace is one step short of what sharing-out needs"""
    import torch
    args = [A.desc()], [B.desc()]
    n = S.sfhe_matmul_workspace_size(ctx.h, *args, S.SFHE_EXEC_PERSISTENT)
    work = torch.empty(n - 256, dtype=torch.uint8, device="cuda")
    return S.sfhe_plan_create(ctx.h, *args, [C.desc()], S.SFHE_EXEC_PERSISTENT, work), work


@pytest.mark.parametrize("N,L,n,cols", [(4096, 2, 1024, 2), (4096, 8, 1024, 1), (8192, 4, 1024, 2),
                                        (8192, 8, 512, 1), (16384, 8, 1024, 1)])
def test_whole_long_entries_equal_the_plain_path(N, L, n, cols):
    api, S = gpu_modules()
    ctx = gpu_ctx(N, L, 4)
    A = W.sparse_int_matrix(1, n, 0.0, -7, 7, 81)
    B = W.dense_int_matrix(n, cols, -7, 7, 82)
    Ae, Be = api.encrypt_matrix(ctx, A, "csr", 1), api.encrypt_matrix(ctx, B, "dense", 2)
    C = api.result_matrix(ctx, 1, cols)
    plan, work = _whole_plan(api, S, ctx, Ae, Be, C)
    try:
        st = S.sfhe_plan_stats(plan)
        assert st["products"] == n * cols and st["entries"] == st["ctas"] == cols  # one CTA per whole entry
        S.sfhe_plan_execute(plan)
        S.sfhe_matmul_check(work)
        got = coeff_of(api, ctx, C)
    finally:
        S.sfhe_plan_destroy(plan)
    assert (got == coeff_of(api, ctx, api.matmul(ctx, Ae, Be, mode="plain"))).all()
    want = ((A @ B + W.T_PLAIN // 2) % W.T_PLAIN) - W.T_PLAIN // 2
    assert (api.decrypt(ctx, C) == want).all()
