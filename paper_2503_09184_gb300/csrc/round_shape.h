// round_shape.h -- columns and sizes of the rounding's matrix product
// (round_mma.cuh), shared with the host code that builds its right operand.
#pragma once

// the rings that take it: more than 16 tensor-base primes (round_mma.cuh has
// both sides' figures)
constexpr bool round_on_tensor_cores(int K) { return K > 16; }

// columns of the right operand: 0 v, 1..6 F, then 6 per prime: primes 0..3 at
// 7, primes 4..7 at 32 (so that a 32-column load covers whole primes)
constexpr int round_mma_col(int i) { return i < 4 ? 7 + 6 * i : 32 + 6 * (i - 4); }

// contraction length (4 K bytes and a constant, padded to 16) and columns (padded to 16)
struct RoundShape {
    int kc, nc;
};
constexpr RoundShape round_shape(int L, int K)
{
    return RoundShape{(4 * K + 1 + 15) / 16 * 16, (round_mma_col(L - 1) + 6 + 15) / 16 * 16};
}

// The accumulators hold integers D, |D| < 2^22, in a float whose last place
// is 1: the constant row adds 1.5 2^23 = 2048 x 6144, so that the float's bits
// are ROUND_MAGIC + D.
constexpr unsigned ROUND_MAGIC = 0x4B400000u;
