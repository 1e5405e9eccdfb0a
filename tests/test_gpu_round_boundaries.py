"""The exact scale-and-round inside plans at L = 8, where the plans round on
the tensor cores and the plain path on the CUDA cores: tensor coefficients on
and beside the half-integers, where the tensor-core form leaves the decision
to the exact one (within 2^-27 of a half-integer, about one coefficient in
2^26 otherwise).

With constant a0 = m0, a1 = m1 the tensor is x0 = m0 b0, x1 = m0 b1 + m1 b0,
x2 = m1 b1, so that any fraction of t x / Q can be chosen coefficient by
coefficient: t m b = r (mod Q) for b = r (t m)^-1.  The neighbours in a warp
are far from a half-integer, or all of them close."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_common import coeff_of, gpu_ctx, gpu_modules
import textbook as tb

pytestmark = pytest.mark.gpu
T = 65537
RINGS = [(4096, 8), (8192, 8), (16384, 8)]


def _fractions(Q):
    """distances from a half-integer: 1 / (2 Q), inside, on both sides of and
    just outside the band, in units of 1 / (2 Q)"""
    band = (2 * Q) >> 27
    out = [1, -1]
    for d in (band - (band >> 10), band + (band >> 10), band - (band >> 11), band + (band >> 11), band >> 1, 2 * band,
              band >> 13, (2 * Q) >> 54, (2 * Q) >> 39):
        out += [d, -d]
    return out


def _operands(q, N, large, dense, seed):
    """(a, b, expected d) in coefficient form; large: m0, m1 of Q's size"""
    rng = np.random.default_rng(seed)
    Q = tb.prod(q)

    def big():
        return int.from_bytes(rng.bytes((Q.bit_length() + 7) // 8 + 8), "little") % Q

    m = [tb.centred(big(), Q) if large else 1 for _ in range(2)]
    inv = [pow(T * m[p], -1, Q) for p in range(2)]
    fr = _fractions(Q)
    b0, b1, d = [], [], [[], [], []]
    for k in range(N):
        def near():
            return ((Q + fr[int(rng.integers(0, len(fr)))]) // 2) % Q
        hit = dense or rng.integers(0, 4) == 0
        kind = int(rng.integers(0, 3))
        x0 = near() * inv[0] % Q if hit else big()
        if hit and kind == 0:      # x2 on the boundary
            x1 = near() * inv[1] % Q
        elif hit and kind == 1:    # x1 on the boundary
            x1 = (near() - T * m[1] * tb.centred(x0, Q)) * inv[0] % Q
        else:
            x1 = big()
        b0.append(x0)
        b1.append(x1)
        c0, c1 = tb.centred(x0, Q), tb.centred(x1, Q)
        for p, x in enumerate((m[0] * c0, m[0] * c1 + m[1] * c0, m[1] * c1)):
            d[p].append((2 * T * x + Q) // (2 * Q) % Q)
    const = [tb.from_int_poly([m[p]] + [0] * (N - 1), q) for p in range(2)]
    return (np.stack(const), np.stack([tb.from_int_poly(b0, q), tb.from_int_poly(b1, q)]),
            np.stack([tb.from_int_poly(x, q) for x in d]))


@pytest.mark.parametrize("N,L", RINGS)
@pytest.mark.parametrize("large,dense", [(False, False), (True, False), (True, True)])
def test_plans_round_boundary_coefficients_exactly(N, L, large, dense):
    import torch
    api, S = gpu_modules()
    ctx = gpu_ctx(N, L, 1)
    a, b, d = _operands(ctx.q, N, large, dense, 17 * N + L)
    M = api.import_coeff(ctx, np.stack([a, b]))
    # the plain path's rounding against big integers
    got = torch.empty((3, L, N), dtype=torch.int64, device="cuda")
    work = torch.empty(3 * ctx.K * N * 4, dtype=torch.uint8, device="cuda")
    S.sfhe_ct_tensor_scale(ctx.h, M.ext[0], M.ext[1], got, work)
    assert (api.to_numpy_u64(got) == d).all()
    # plans of one product against the plain path's relinearised product
    Am = api.EncMatrix(1, 1, S.SFHE_ENC_DENSE, 1, ct=M.ct[0:1], ext=M.ext[0:1])
    Bm = api.EncMatrix(1, 1, S.SFHE_ENC_DENSE, 1, ct=M.ct[1:2], ext=M.ext[1:2])
    ref = coeff_of(api, ctx, api.matmul(ctx, Am, Bm, mode="plain"))
    for mode in ("persistent", "lazy"):
        assert (coeff_of(api, ctx, api.matmul(ctx, Am, Bm, mode=mode)) == ref).all(), mode


@pytest.mark.parametrize("N,L", [(4096, 8), (16384, 8)])
def test_sums_over_boundary_products(N, L):
    """three products of one entry, whole and shared out"""
    import torch
    api, S = gpu_modules()
    ctx = gpu_ctx(N, L, 1)
    ops = [_operands(ctx.q, N, True, False, 40 + i) for i in range(3)]
    MA = api.import_coeff(ctx, np.stack([o[0] for o in ops]))
    MB = api.import_coeff(ctx, np.stack([o[1] for o in ops]))
    MB.rows, MB.cols = 3, 1
    ref = coeff_of(api, ctx, api.matmul(ctx, MA, MB, mode="plain"))
    assert (coeff_of(api, ctx, api.matmul(ctx, MA, MB)) == ref).all()
    n = S.sfhe_matmul_workspace_size(ctx.h, [MA.desc()], [MB.desc()], S.SFHE_EXEC_PERSISTENT)
    C = api.result_matrix(ctx, 1, 1)
    work = torch.empty(n - 256, dtype=torch.uint8, device="cuda")
    plan = S.sfhe_plan_create(ctx.h, [MA.desc()], [MB.desc()], [C.desc()], S.SFHE_EXEC_PERSISTENT, work)
    try:
        S.sfhe_plan_execute(plan)
        assert (coeff_of(api, ctx, C) == ref).all()
    finally:
        S.sfhe_plan_destroy(plan)
