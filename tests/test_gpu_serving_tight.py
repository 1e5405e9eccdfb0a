"""A budget that holds a request only beside workspaces without the slots of
shared-out entries: the request still runs, with the same ciphertexts."""
from __future__ import annotations

import pytest

import workloads as W
from gpu_common import gpu_ctx, gpu_modules

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lazy", [False, True])
def test_request_beside_whole_entry_workspaces(lazy):
    api, S = gpu_modules()
    from paper_2503_09184_gb300 import serving as SV
    ctx = gpu_ctx(4096, 2, 0)
    A, B = W.operands(W.MatmulShape(6, 16, 4, 0.4, -16, 16, 301))
    req = SV.Request(3, A, B, arrival=0.0)
    ct_b, ext_b = 2 * ctx.L * ctx.N * 8, 2 * ctx.K * ctx.N * 4
    flags = S.SFHE_EXEC_PERSISTENT | (S.SFHE_EXEC_LAZY if lazy else 0)
    whole = S.sfhe_matmul_workspace_bound_whole(ctx.h, 1024, 256, 256, flags)
    ex = SV.GpuExecutor(ctx, lazy=lazy, wave_products=256)
    assert ex.reserved_bytes > whole
    # one column of B and of C beside A
    budget = int((A != 0).sum()) * (ct_b + ext_b) + 16 * (ct_b + ext_b) + 6 * ct_b + whole
    out = SV.serve([req], ex, budget, wave_products=256, ct_bytes=ct_b, ext_bytes=ext_b, keep_results=True)
    assert out["done"] == 1 and req.state == "done"
    assert out["reserved_bytes"] == ex.reserved_bytes == whole
    alone = api.matmul(ctx, api.encrypt_matrix(ctx, A, "csr", 2 * req.rid + 1),
                       api.encrypt_matrix(ctx, B, "dense", 2 * req.rid + 2), mode="lazy" if lazy else "persistent")
    want = api.to_coeff(ctx, alone.ct, 24).reshape(6, 4, 2, ctx.L, ctx.N)
    for c in range(4):
        tile = api.to_coeff(ctx, ex.result(req, c).ct, 6).reshape(6, 2, ctx.L, ctx.N)
        assert (tile == want[:, c]).all(), c
