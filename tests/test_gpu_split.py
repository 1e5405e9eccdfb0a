"""Output entries whose products are shared out over several units (few
entries): bit-identical to the plain per-product path, to the oracle's grouped
mode when grouped, over several executions, with empty entries, and stopped
and resumed."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W
from gpu_common import coeff_of, gpu_ctx, gpu_modules, oracle_ctx
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,L,shape,s", [(4096, 2, (1, 301, 1), 0.0), (4096, 3, (3, 17, 2), 0.4),
                                         (8192, 4, (2, 9, 3), 0.3), (8192, 4, (1, 2, 1), 0.0), (16384, 8, (1, 5, 2), 0.0)])
def test_shared_out_entries_equal_the_plain_path(N, L, shape, s):
    api, S = gpu_modules()
    ctx = gpu_ctx(N, L, 6)
    M, K, Nc = shape
    A = W.sparse_int_matrix(M, K, s, -16, 16, 71)
    if M > 2:
        A[1] = 0  # an empty entry among shared-out ones
    B = W.dense_int_matrix(K, Nc, -16, 16, 72)
    Ae, Be = api.encrypt_matrix(ctx, A, "csr", 1), api.encrypt_matrix(ctx, B, "dense", 2)
    ref = coeff_of(api, ctx, api.matmul(ctx, Ae, Be, mode="plain"))
    for graph in (False, True):
        plan = api.Plan(ctx, [Ae], [Be], graph=graph)
        assert plan.stats["entries"] == M * Nc and plan.stats["products"] == int((A != 0).sum()) * Nc
        assert plan.stats["ctas"] > M * Nc  # more units than entries
        for _ in range(3):
            plan.Cs[0].ct.fill_(3)
            plan.execute()
            assert (coeff_of(api, ctx, plan.Cs[0]) == ref).all()
        plan.close()


def test_grouped_mode_keeps_its_groups():
    """N = 8192, L = 4: groups of 15; 40 products in groups of 15, 15, 10"""
    api, S = gpu_modules()
    ctx = gpu_ctx(8192, 4, 6)
    assert ctx.lazy_group == 15
    A = W.sparse_int_matrix(1, 40, 0.0, -16, 16, 73)
    B = W.dense_int_matrix(40, 1, -16, 16, 74)
    Ae, Be = api.encrypt_matrix(ctx, A, "csr", 1), api.encrypt_matrix(ctx, B, "dense", 2)
    plan = api.Plan(ctx, [Ae], [Be], mode="lazy")
    assert plan.stats["ctas"] == 3
    plan.execute()
    parts = [api.matmul(ctx, api.EncMatrix(1, k1 - k0, S.SFHE_ENC_DENSE, k1 - k0, ct=Ae.ct[k0:k1], ext=Ae.ext[k0:k1]),
                        api.EncMatrix(k1 - k0, 1, S.SFHE_ENC_DENSE, k1 - k0, ct=Be.ct[k0:k1], ext=Be.ext[k0:k1]),
                        mode="lazy") for k0, k1 in ((0, 15), (15, 30), (30, 40))]
    q = np.array(ctx.q, dtype=np.uint64)[None, None, :, None]
    want = sum(coeff_of(api, ctx, p) for p in parts) % q  # one group each; the groups are added
    assert (coeff_of(api, ctx, plan.Cs[0]) == want).all()
    plan.close()


def test_stopped_and_resumed():
    api, S = gpu_modules()
    import torch
    ctx = gpu_ctx(4096, 2, 6)
    A = W.sparse_int_matrix(3, 60, 0.2, -16, 16, 75)
    B = W.dense_int_matrix(60, 4, -16, 16, 76)
    Ae, Be = api.encrypt_matrix(ctx, A, "csr", 1), api.encrypt_matrix(ctx, B, "dense", 2)
    ref = coeff_of(api, ctx, api.matmul(ctx, Ae, Be, mode="plain"))
    plan = api.Plan(ctx, [Ae], [Be])
    stop = torch.ones(1, dtype=torch.int32, device="cuda")
    S.sfhe_plan_set_stop(plan.h, stop)
    plan.execute()
    assert S.sfhe_plan_progress(plan.h) == 0
    stop.zero_()
    S.sfhe_plan_resume(plan.h)
    assert S.sfhe_plan_progress(plan.h) == 12
    assert (coeff_of(api, ctx, plan.Cs[0]) == ref).all()
    plan.close()
