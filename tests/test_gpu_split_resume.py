"""A launch that stops with output entries half done: some of an entry's units
have left their sums in its slots, the others have not run.  The stop word
here is the launch's own unit counter (the first word of the workspace): it
is zero until the first unit is taken, so every CTA takes about one unit and
stops, whatever the timing, and a plan of more units than CTAs is always cut
short."""
from __future__ import annotations

import pytest

import workloads as W
from gpu_common import coeff_of, gpu_ctx, gpu_modules

pytestmark = pytest.mark.gpu
MARK = 3


@pytest.mark.parametrize("N,L,M,Nc", [(4096, 2, 20, 10), (8192, 4, 10, 10), (16384, 8, 10, 10)])
def test_half_done_entries_survive_a_stop(N, L, M, Nc):
    import torch
    api, S = gpu_modules()
    ctx = gpu_ctx(N, L, 6)
    A = W.sparse_int_matrix(M, 24, 0.0, -16, 16, 77)
    B = W.dense_int_matrix(24, Nc, -16, 16, 78)
    Ae, Be = api.encrypt_matrix(ctx, A, "csr", 1), api.encrypt_matrix(ctx, B, "dense", 2)
    ref = coeff_of(api, ctx, api.matmul(ctx, Ae, Be, mode="plain"))
    plan = api.Plan(ctx, [Ae], [Be])
    C, n, grid = plan.Cs[0].ct, plan.stats["entries"], plan.stats["ctas"]
    counter = plan.work[:4].view(torch.int32)
    plan.execute()
    torch.cuda.synchronize()
    # every CTA's last fetch goes past the end: units = counter - CTAs.  The
    # entries are alike, so their units come one after another, p each
    units = int(counter) - grid
    p = units // n
    assert units == n * p and p > 1 and units > grid
    half = 0
    for _ in range(20):
        C.fill_(MARK)
        S.sfhe_plan_set_stop(plan.h, counter)
        plan.execute()
        done, taken = S.sfhe_plan_progress(plan.h), int(counter)
        assert 0 < taken <= grid and done == taken // p
        written = [not bool((C[e] == MARK).all()) for e in range(n)]
        assert sum(written) == done  # the others' C is untouched
        S.sfhe_plan_set_stop(plan.h, None)
        S.sfhe_plan_resume(plan.h)
        assert S.sfhe_plan_progress(plan.h) == n
        assert (coeff_of(api, ctx, plan.Cs[0]) == ref).all()
        if 0 < done and taken % p:
            half += 1
            break
    assert half
    plan.close()
