"""The ciphertext-prime transforms at the extremes of their lazy ranges: every
coefficient q - 1, alternating 0 and q - 1, and the monomial X, in every ring,
against closed forms (all slots of X are the evaluation points z, z^N = -1;
a constant coefficient vector v gives v (z^N - 1) / (z - 1)), and back."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_common import gpu_ctx, gpu_modules

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,L", [(4096, 2), (4096, 8), (8192, 4), (8192, 8), (16384, 2), (16384, 8)])
def test_transforms_at_the_ends_of_the_range(N, L):
    api, S = gpu_modules()
    import torch
    ctx = gpu_ctx(N, L, 5)
    q = np.array(ctx.q, dtype=np.uint64)
    x = np.zeros((3, L, N), dtype=np.uint64)
    x[0, :, 1] = 1
    x[1] = (q - np.uint64(1))[:, None]
    x[2, :, 1::2] = (q - np.uint64(1))[:, None]
    src = torch.from_numpy(x.view(np.int64)).cuda()
    f, back = torch.empty_like(src), torch.empty_like(src)
    S.sfhe_from_coeff(ctx.h, src, 3, f)
    S.sfhe_to_coeff(ctx.h, f, 3, back)
    assert bool((back == src).all())
    got = api.to_numpy_u64(f)
    slots = np.unique(np.r_[0, 1, 31, 32, N // 2 - 1, N // 2, N - 2, N - 1, np.random.default_rng(N + L).integers(0, N, 40)])
    for i in range(L):
        p = ctx.q[i]
        assert len(np.unique(got[0, i])) == N
        for s in slots:
            z = int(got[0, i, s])
            assert pow(z, N, p) == p - 1
            assert int(got[1, i, s]) == (p - 1) * -2 * pow(z - 1, -1, p) % p
            assert int(got[2, i, s]) == (p - 1) * z * -2 * pow(z * z - 1, -1, p) % p
