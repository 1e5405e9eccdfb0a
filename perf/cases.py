"""Performance cases of the encrypted sparse matmul: what a user's program has
the library do, over the rings, shapes, sparsities, encodings and execution
modes of the workloads and tests.

A case's "kind" is the entry point a program calls:
  product  one ciphertext product with relinearisation (sfhe_ct_mul_relin)
  plan     a kept matmul plan, executed (Plan.execute)
  call     a one-shot matmul and the decryption of its result
  client   encryption of a matrix, its lift and a decryption
  host     a matmul over ciphertexts in host memory (sfhe_matmul_host)
  chunked  the chunked product of Alg. 1 (c values per ciphertext) in BFV
  ckks     the chunked product under the paper's CKKS parameter set
"""
from __future__ import annotations

import numpy as np
import torch

from paper_2503_09184_gb300 import api
from paper_2503_09184_gb300 import sfhe as S
import workloads as W

T = W.T_PLAIN
# CKKS: four data primes of 50, 40, 40 and 40 bits at N = 8192, one digit per prime
CKKS_N, CKKS_L = 8192, 4


def _mm(name, M, K, Nc, s, N, L, enc, mode="persistent", kind="plan", sb=0.0, count=1, graph=False):
    return {"name": name, "kind": kind, "N": N, "L": L, "M": M, "K": K, "Nc": Nc, "sparsity": s, "b_sparsity": sb,
            "encoding": enc, "mode": mode, "count": count, "graph": graph}


def listed():
    return [
        # the smallest call: one product, as a program that drives Alg. 1's inner loop itself makes it; launches count
        {"name": "product_one", "kind": "product", "N": 8192, "L": 4},
        # the tiny workload, a replayed graph plan: far fewer output entries than SMs
        _mm("tiny_graph", 8, 8, 8, 0.5, 4096, 2, "csr", graph=True),
        # a ragged one-shot call (work list built and uploaded in the call) and the decryption of its result
        _mm("call_ragged", 13, 29, 7, 0.7, 8192, 4, "ell", kind="call"),
        # the sparsity sweep's headline point: A at 50% zeros
        _mm("sweep_50", 64, 64, 64, 0.5, 8192, 4, "csr"),
        # zero masks on both operands: few products per output entry
        _mm("sweep_masks_70", 64, 64, 64, 0.7, 8192, 4, "mask", sb=0.7),
        # a pruned network layer: encrypted weights times a batch of activations
        _mm("layer_90", 128, 256, 16, 0.9, 8192, 4, "csr"),
        # two matmuls of the mixed workload in one plan, the largest ring
        _mm("mixed_batch", 32, 64, 16, 0.6, 16384, 8, "csr", count=2),
        # the opt-in grouped accumulate-then-round mode on the sweep's shape
        _mm("sweep_50_grouped", 64, 64, 64, 0.5, 8192, 4, "csr", mode="lazy"),
        # the data owner's side: encrypt and lift a matrix, decrypt one
        {"name": "client_24x40", "kind": "client", "N": 8192, "L": 4, "rows": 24, "cols": 40},
        # end to end from host memory: upload, lift, matmul, download
        _mm("host_32", 32, 32, 32, 0.5, 8192, 4, "csr", kind="host"),
        # eight values per ciphertext: rotations and masks around the product
        {"name": "chunked_16", "kind": "chunked", "N": 8192, "L": 4, "M": 16, "K": 16, "Nc": 16, "sparsity": 0.5,
         "c": 8, "fused": True},
        # the paper's CKKS set, term by term in batches
        {"name": "ckks_8", "kind": "ckks", "M": 8, "K": 8, "Nc": 8, "sparsity": 0.5, "c": 8},
    ]


# relative cost of one product in a ring (N = 8192, L = 4: 1), for draw()
def _ring_cost(N, L):
    return (N / 8192) * (L / 4) ** 1.3


def _between(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["plan"] * 9 + ["call"] * 3 + ["host"] * 2 + ["client"] * 2 + ["product", "chunked", "ckks"])
    if kind == "product":
        N, L = rng.choice([(4096, 2), (4096, 3), (4096, 4), (8192, 2), (8192, 3), (16384, 4), (16384, 8)])
        return {"kind": kind, "N": N, "L": L}
    if kind == "client":
        N, L = rng.choice([(4096, 2), (8192, 3), (8192, 4), (16384, 8)])
        most = 2048 if N < 16384 else 512
        rows = _between(rng, 1, 64)
        return {"kind": kind, "N": N, "L": L, "rows": rows, "cols": _between(rng, 1, max(1, min(64, most // rows)))}
    if kind == "chunked":
        return {"kind": kind, "N": 8192, "L": 4, "M": _between(rng, 4, 24), "K": _between(rng, 4, 24),
                "Nc": _between(rng, 4, 24), "sparsity": round(rng.uniform(0.3, 0.8), 2), "c": rng.choice([4, 8]),
                "fused": rng.random() < 0.7}
    if kind == "ckks":
        return {"kind": kind, "M": _between(rng, 3, 12), "K": _between(rng, 3, 12), "Nc": _between(rng, 3, 12),
                "sparsity": round(rng.uniform(0.3, 0.8), 2), "c": rng.choice([4, 8])}
    while True:
        N, L = rng.choice([(4096, 2), (4096, 2), (8192, 3), (8192, 4), (8192, 4), (8192, 4), (16384, 8), (16384, 8)])
        M, K, Nc = _between(rng, 3, 128), _between(rng, 3, 256), _between(rng, 3, 64)
        s = round(rng.uniform(0.0, 0.95), 2)
        sb = round(rng.uniform(0.3, 0.9), 2) if rng.random() < 0.25 else 0.0
        products = M * K * Nc * (1 - s) * (1 - sb)
        stored = (M * K + K * Nc + M * Nc) * (N / 8192) * (L / 4)
        most = 60000 if kind == "plan" else 12000
        if 4 <= products * _ring_cost(N, L) <= most and stored <= (12000 if kind == "plan" else 4000):
            break
    mode = "persistent" if kind != "plan" else rng.choice(["persistent"] * 4 + ["lazy"])
    encoding = rng.choice(["csr", "ell", "mask"] + (["dense"] if s == 0.0 else []))
    c = _mm("", M, K, Nc, s, N, L, encoding, mode=mode, kind=kind, sb=sb, graph=kind == "plan" and rng.random() < 0.3)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs ---
def _values(case, seed, m=0):
    """the m-th pair of plaintext operands"""
    rng = np.random.default_rng([seed, m])
    s1, s2 = (int(x) for x in rng.integers(0, 1 << 31, size=2))
    A = W.sparse_int_matrix(case["M"], case["K"], case["sparsity"], -16, 16, s1)
    B = W.dense_int_matrix(case["K"], case["Nc"], -16, 16, s2)
    if case.get("b_sparsity", 0.0) > 0.0:
        B = W.sparsify(B, case["b_sparsity"], s2 + 1)
    return A, B


def _b_encoding(case):
    return "mask" if case.get("b_sparsity", 0.0) > 0.0 else "dense"


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.kind = case["kind"]
    if s.kind == "ckks":
        return _prepare_ckks(s, case, seed)
    s.ctx = api.Context(case["N"], case["L"], seed=seed)
    if s.kind == "product":
        rng = np.random.default_rng(seed)
        s.ops = api.encrypt_matrix(s.ctx, rng.integers(-16, 17, size=(1, 2)), "dense", 1)
        N, L, K = s.ctx.N, s.ctx.L, s.ctx.K
        s.work = torch.empty(3 * K * N * 4 + 256 + (3 * L + (L + 2) * L) * N * 8, dtype=torch.uint8, device="cuda")
        s.out = torch.empty((2, L, N), dtype=torch.int64, device="cuda")
    elif s.kind == "client":
        rng = np.random.default_rng(seed)
        s.values = rng.integers(-16, 17, size=(case["rows"], case["cols"]))
        s.seed = seed
    elif s.kind == "chunked":
        A, B = _values(case, seed)
        s.A = api.encrypt_chunked(s.ctx, A, case["c"], 1)
        s.B = api.encrypt_chunked(s.ctx, B, case["c"], 2)
        s.rk = api.RotationKeys(s.ctx, case["c"])
        s.fused = case["fused"]
        if s.fused:
            az, bz = s.A.zero.reshape(-1), s.B.zero.reshape(-1)
            n = S.sfhe_matmul_chunked_fused_workspace_size(s.ctx.h, case["c"], case["M"], case["K"], case["Nc"], az, bz)
        else:
            n = S.sfhe_matmul_chunked_workspace_size(s.ctx.h)
        s.work = torch.empty(n, dtype=torch.uint8, device="cuda")
    else:
        lift = s.kind != "host"
        s.As, s.Bs = [], []
        for m in range(case["count"]):
            A, B = _values(case, seed, m)
            s.As.append(api.encrypt_matrix(s.ctx, A, case["encoding"], 2 * m + 1, lift=lift))
            s.Bs.append(api.encrypt_matrix(s.ctx, B, _b_encoding(case), 2 * m + 2, lift=lift))
        s.mode = case["mode"]
        if s.kind == "plan":
            s.plan = api.Plan(s.ctx, s.As, s.Bs, mode=s.mode, graph=case["graph"])
        elif s.kind == "host":
            s.h_a = [M.ct.cpu().pin_memory() for M in s.As]
            s.h_b = [M.ct.cpu().pin_memory() for M in s.Bs]
            s.h_c = [torch.empty((M.rows * B.cols, 2, case["L"], case["N"]), dtype=torch.int64, pin_memory=True)
                     for M, B in zip(s.As, s.Bs)]
            s.hp = _HostPlan(s.ctx, s.As, s.Bs)
    return s


class _HostPlan:
    def __init__(self, ctx, As, Bs):
        self.ctx = ctx
        self.h = S.sfhe_host_plan_create(ctx.h, [a.desc() for a in As], [b.desc() for b in Bs], api.PERSISTENT, 2)

    def __del__(self):
        torch.cuda.synchronize()
        S.sfhe_host_plan_destroy(self.h)


class _Ckks:
    def __init__(self, seed):
        self.h = S.sfhe_ckks_ctx_create(N=CKKS_N, seed=seed)
        self.scale = S.sfhe_ckks_ctx_primes(self.h, CKKS_L)[2]

    def __del__(self):
        torch.cuda.synchronize()
        S.sfhe_ckks_ctx_destroy(self.h)


class _CkksKeys:
    def __init__(self, ctx, c):
        self.ctx = ctx
        self.h = S.sfhe_ckks_rotkeys_create(ctx.h, c)

    def __del__(self):
        torch.cuda.synchronize()
        S.sfhe_ckks_rotkeys_destroy(self.h)


def _prepare_ckks(s, case, seed):
    s.ctx = _Ckks(seed)
    A, B = _values(case, seed)
    c = case["c"]
    ops = []
    for mid, V in ((1, A), (2, B)):
        flat = V.reshape(-1).astype(np.float64)
        n = -(-flat.size // c)
        polys = np.stack([S.sfhe_ckks_encode(s.ctx.h, CKKS_N, flat[q * c:(q + 1) * c], s.ctx.scale) for q in range(n)])
        ct = torch.empty((n, 2, CKKS_L, CKKS_N), dtype=torch.int64, device="cuda")
        S.sfhe_ckks_encrypt(s.ctx.h, polys, np.stack([np.arange(n), np.zeros(n)], axis=1).astype(np.int32), mid, ct)
        ops.append(ct)
    s.A, s.B = ops
    s.shape = (case["M"], case["K"], case["Nc"])
    s.az, s.bz = ((V == 0).astype(np.uint8).reshape(-1) for V in (A, B))
    s.rk = _CkksKeys(s.ctx, c)
    nC = -(-(case["M"] * case["Nc"]) // c)
    s.C = torch.zeros((nC, 2, CKKS_L, CKKS_N), dtype=torch.int64, device="cuda")
    s.work = torch.empty(S.sfhe_ckks_matmul_chunked_workspace_size(s.ctx.h), dtype=torch.uint8, device="cuda")
    return s


# -------------------------------------------------------------------- pass ---
def run(s):
    if s.kind == "product":
        S.sfhe_ct_mul_relin(s.ctx.h, s.ops.ext[0], s.ops.ext[1], s.out, s.work)
        return s.out
    if s.kind == "plan":
        s.plan.execute()
        return [C.ct for C in s.plan.Cs]
    if s.kind == "call":
        C = api.matmul(s.ctx, s.As[0], s.Bs[0], mode=s.mode)
        return [C.ct, api.decrypt(s.ctx, C)]
    if s.kind == "client":
        M = api.encrypt_matrix(s.ctx, s.values, "dense", 1 + s.seed % 1000)
        return [M.ct, M.ext, api.decrypt(s.ctx, M)]
    if s.kind == "host":
        S.sfhe_matmul_host(s.hp.h, s.h_a, s.h_b, s.h_c)
        return s.h_c
    if s.kind == "chunked":
        return api.matmul_chunked(s.ctx, s.A, s.B, s.rk, skip_zeros=True, fused=s.fused, work=s.work)[0].ct
    S.sfhe_ckks_matmul_chunked(s.ctx.h, s.rk.h, *s.shape, s.A, s.B, s.C, s.az, s.bz, s.work)
    return s.C[:, :, :2]  # the result's level: two of the four limbs remain after the two rescales


# -------------------------------------------------------------------- work ---
def _log2(n):
    return n.bit_length() - 1


def work(case):
    """Bytes: each stored operand (for a host matmul its upload) read once, the
    result written once.  "flops": modular multiplications of a ciphertext
    word, each counted as two operations: the pointwise products of the tensor
    for every product, the transforms and key products of one relinearisation
    for every output."""
    kind = case["kind"]
    if kind == "ckks":
        N, L = CKKS_N, CKKS_L
    else:
        N, L = case["N"], case["L"]
    ct = 2 * L * N * 8
    ext = 2 * ((10 * (_log2(N) + 108 * L + 1) + 298) // 299) * N * 4
    tensor = 4 * L * N
    relin = L * (L + 2) * (N // 2) * _log2(N) + 2 * L * L * N
    if kind == "product":
        return {"bytes": 2 * ext + ct, "flops": 2 * (tensor + relin)}
    if kind == "client":
        n = case["rows"] * case["cols"]
        return {"bytes": n * (2 * ct + ext + 16), "flops": 2 * n * (4 * L) * (N // 2) * _log2(N)}
    M, K, Nc = case["M"], case["K"], case["Nc"]
    keep = 1 - case["sparsity"]
    if kind in ("chunked", "ckks"):
        products, c = M * K * Nc * keep, case["c"]
        n = (M * K + K * Nc + M * Nc) / c
        return {"bytes": int(n * ct), "flops": int(2 * (products * tensor + M * Nc * relin))}
    products = case["count"] * M * K * Nc * keep * (1 - case["b_sparsity"])
    stored = M * K * (keep if case["encoding"] in ("csr", "ell") else 1) + K * Nc
    return {"bytes": int(case["count"] * (stored * (ct if kind == "host" else ext) + M * Nc * ct)),
            "flops": int(2 * (products * tensor + case["count"] * M * Nc * relin))}


def _centred(x):
    return ((x + T // 2) % T) - T // 2


def exact(case, seed):
    """The decrypted values; ciphertext words are whole numbers without a 64-bit counterpart."""
    if case["kind"] == "call":
        A, B = _values(case, seed)
        return [None, _centred(A @ B)]
    if case["kind"] == "client":
        rng = np.random.default_rng(seed)
        return [None, None, rng.integers(-16, 17, size=(case["rows"], case["cols"]))]
    return None
