"""A launch that stops with output entries half done: some of an entry's units
have left their sums in its slots, the others have not run.  The stop word
here is the launch's own unit counter (the first word of the workspace): it
is zero until the first unit is taken, so every CTA takes about one unit and
stops, whatever the timing, and a plan of more units than CTAs is always cut
short.  How many units it took by then, from one to the number of CTAs, is left
to timing.  At 24 products an entry's units are alike and follow one another,
so that entries are complete when the launch stops; at 23 the last one is
shorter and units go longest first, so that any number of units taken leaves
entries half done."""
from __future__ import annotations

import pytest

import workloads as W
from gpu_common import coeff_of, gpu_ctx, gpu_modules

pytestmark = pytest.mark.gpu
MARK = 3


@pytest.mark.parametrize("K", [24, 23])
@pytest.mark.parametrize("N,L,M,Nc", [(4096, 2, 20, 10), (8192, 4, 10, 10), (16384, 8, 10, 10)])
def test_half_done_entries_survive_a_stop(N, L, M, Nc, K):
    import torch
    api, S = gpu_modules()
    ctx = gpu_ctx(N, L, 6)
    A = W.sparse_int_matrix(M, K, 0.0, -16, 16, 77)
    B = W.dense_int_matrix(K, Nc, -16, 16, 78)
    Ae, Be = api.encrypt_matrix(ctx, A, "csr", 1), api.encrypt_matrix(ctx, B, "dense", 2)
    ref = coeff_of(api, ctx, api.matmul(ctx, Ae, Be, mode="plain"))
    plan = api.Plan(ctx, [Ae], [Be])
    C, n, grid = plan.Cs[0].ct, plan.stats["entries"], plan.stats["ctas"]
    counter = plan.work[:4].view(torch.int32)
    plan.execute()
    torch.cuda.synchronize()
    # every CTA's last fetch goes past the end: units = counter - CTAs, p an entry
    units = int(counter) - grid
    p = units // n
    assert units == n * p and p > 1 and units > grid
    assert K == 23 or K % p == 0
    for _ in range(3):
        C.fill_(MARK)
        S.sfhe_plan_set_stop(plan.h, counter)
        plan.execute()
        done, taken = S.sfhe_plan_progress(plan.h), int(counter)
        assert 0 < taken <= grid
        if K == 24:
            assert done == taken // p
        else:  # the n (p - 1) longer units come first, p - 1 an entry
            assert done == max(0, taken - n * (p - 1)) < min(n, -(-taken // (p - 1)))  # entries begun
        written = [not bool((C[e] == MARK).all()) for e in range(n)]
        assert sum(written) == done  # the others' C is untouched
        S.sfhe_plan_set_stop(plan.h, None)
        S.sfhe_plan_resume(plan.h)
        assert S.sfhe_plan_progress(plan.h) == n
        assert (coeff_of(api, ctx, plan.Cs[0]) == ref).all()
    plan.close()
