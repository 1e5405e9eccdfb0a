"""Which plans share the products of their entries out: not those that it
makes slower, because the entries are short (the units then end with more
relinearisations than fit beside one another) or because the units of a small
ring come to lie two on an SM.  Measured, shared out against whole, on the
GB300: 0.84 (8192, 4), 0.74 (4096, 2), 0.75 (4096, 8) and 0.88 (16384, 8) for
100 entries of 2 products; 0.90 for 128 entries of 16 products in groups of
15; 1.3 for 64 entries of 4 products."""
from __future__ import annotations

import pytest

import workloads as W
from gpu_common import coeff_of, gpu_ctx, gpu_modules

pytestmark = pytest.mark.gpu


def _plan(N, L, M, K, Nc, mode):
    api, S = gpu_modules()
    ctx = gpu_ctx(N, L, 6)
    A, B = W.sparse_int_matrix(M, K, 0.0, -16, 16, 91), W.dense_int_matrix(K, Nc, -16, 16, 92)
    Ae, Be = api.encrypt_matrix(ctx, A, "csr", 1), api.encrypt_matrix(ctx, B, "dense", 2)
    return api, ctx, Ae, Be, api.Plan(ctx, [Ae], [Be], mode=mode)


@pytest.mark.parametrize("N,L,M,K,Nc,mode", [(8192, 4, 10, 2, 10, "persistent"), (8192, 4, 10, 6, 10, "persistent"),
                                             (4096, 2, 10, 2, 10, "persistent"), (4096, 8, 10, 2, 10, "persistent"),
                                             (16384, 8, 10, 2, 10, "persistent"), (8192, 4, 8, 16, 16, "lazy")])
def test_entries_stay_whole_where_sharing_out_is_slower(N, L, M, K, Nc, mode):
    plan = _plan(N, L, M, K, Nc, mode)[-1]
    assert plan.stats["ctas"] == plan.stats["entries"] == M * Nc  # as many units as entries
    plan.close()


@pytest.mark.parametrize("N,L", [(4096, 2), (8192, 4), (16384, 8)])
def test_entries_are_shared_out_where_sms_would_idle(N, L):
    api, ctx, Ae, Be, plan = _plan(N, L, 8, 4, 8, "persistent")
    assert plan.stats["ctas"] > plan.stats["entries"] == 64
    plan.execute()
    assert (coeff_of(api, ctx, plan.Cs[0]) == coeff_of(api, ctx, api.matmul(ctx, Ae, Be, mode="plain"))).all()
    plan.close()


@pytest.mark.parametrize("L", [3, 4])
def test_a_grouped_launch_has_as_many_ctas_as_are_resident(L):
    """N = 4096, L = 3 and 4: two CTAs of the per-product kernel fit on an SM,
    one of the grouped kernel (its registers); a launch of more would run the
    rest after the others, and the schedule would count on them"""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for mode, per_sm in (("persistent", 2), ("lazy", 1)):
        api, ctx, Ae, Be, plan = _plan(4096, L, 20, 3, 20, mode)
        assert plan.stats["entries"] == 400 and plan.stats["ctas"] == per_sm * sms, mode
        plan.execute()
        if mode == "lazy":  # one group per entry
            want = ((W.sparse_int_matrix(20, 3, 0.0, -16, 16, 91) @ W.dense_int_matrix(3, 20, -16, 16, 92) + 32768)
                    % W.T_PLAIN) - 32768
            assert (api.decrypt(ctx, plan.Cs[0]) == want).all()
        plan.close()
