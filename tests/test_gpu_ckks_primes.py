"""CKKS contexts over other prime sizes than the paper's: the pseudo-Mersenne
transforms at the ends of their range (33 and 54 bits) and the Shoup ones
outside it (a 30-bit and a 58-bit prime): encryption, product and rescale limb
for limb against the oracle."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_common import gpu_modules
from oracle import ckks as CK

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,special", [((54, 33, 50, 54), 54), ((33, 33, 34, 33), 33), ((54, 54, 53, 54), 33),
                                          ((50, 30, 40, 40), 40), ((58, 40, 40, 40), 40)])
def test_other_prime_sizes(bits, special):
    api, S = gpu_modules()
    import torch
    N = 64
    h = S.sfhe_ckks_ctx_create(N=N, bits=bits, special_bits=special, log_scale=20, seed=9)
    ck = CK.OracleCkks(N=N, bits=bits, special_bits=special, log_scale=20, seed=9)
    q, P, _ = S.sfhe_ckks_ctx_primes(h, 4)
    assert q == ck.q and P == ck.P
    work = torch.empty(S.sfhe_ckks_workspace_size(h) + 4 * 4 * N * 8 + 10 * N * 8 * 4, dtype=torch.uint8, device="cuda")

    def ct():
        return torch.zeros((1, 2, 4, N), dtype=torch.int64, device="cuda")

    def coeff(x, level):
        out = ct()
        S.sfhe_ckks_to_coeff(h, x, level, 1, out)
        return out.cpu().numpy().view(np.uint64)[0]

    rng = np.random.default_rng(3)
    m = [rng.integers(-(1 << 20), 1 << 20, N) for _ in range(2)]
    a, b, x = ct(), ct(), ct()
    for t, p, mid in ((a, m[0], 1), (b, m[1], 2)):
        S.sfhe_ckks_encrypt(h, p[None], np.array([[2, 3]], dtype=np.int32), mid, t)
    oa, ob = ck.encrypt(m[0], 1, 2, 3), ck.encrypt(m[1], 2, 2, 3)
    assert (coeff(a, 3) == oa).all()
    S.sfhe_ckks_mul_relin(h, a, b, 3, x, work)
    prod = ck.mul_relin(oa, ob, 3)
    assert (coeff(x, 3) == prod).all()
    S.sfhe_ckks_rescale(h, x, 3, 1, x, work)
    assert (coeff(x, 2)[:, :3] == ck.rescale(prod, 3)[:, :3]).all()
    S.sfhe_ckks_ctx_destroy(h)
