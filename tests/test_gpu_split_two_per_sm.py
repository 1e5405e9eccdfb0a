"""Which units the entries are cut into where two CTAs fit on an SM: a grid
beyond the SMs puts long units beside long ones.  56 entries of 5 products on
the GB300 at (4096, 2): 303 us in 280 units of one product, 413 in 168 of two;
72 entries: 348 in 144 units of three, 428 in 216 of two."""
from __future__ import annotations

import pytest

import workloads as W
from gpu_common import gpu_ctx, gpu_modules

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [2, 3])
@pytest.mark.parametrize("M,Nc,units", [(7, 8, 280), (8, 9, 144)])
def test_units_of_entries_of_five_products(L, M, Nc, units):
    api, S = gpu_modules()
    ctx = gpu_ctx(4096, L, 6)
    A, B = W.sparse_int_matrix(M, 5, 0.0, -16, 16, 91), W.dense_int_matrix(5, Nc, -16, 16, 92)
    plan = api.Plan(ctx, [api.encrypt_matrix(ctx, A, "csr", 1)], [api.encrypt_matrix(ctx, B, "dense", 2)])
    assert plan.stats["ctas"] == units
