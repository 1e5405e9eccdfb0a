// round_mma.cuh -- the exact scale-and-round as a matrix product on the
// tensor cores.
//
// For a tensor coefficient x with residues x~_k (see scale_round_m), every
// quantity of the rounding is linear in the bytes of the x~_k: with byte a of
// x~_k and 2^(8a) t (B/b_k) = A_ka Q + R_ka, |R_ka| <= Q/2,
//   t x / Q = sum byte_ka A_ka - v alpha_B + F,
//   F = (sum byte_ka R_ka - v r_B) / Q.
// One row of the left operand holds a coefficient's 4 K bytes less 128 (fp16
// integers), the columns of the right one hold signed 9-bit digits (fp16
// integers in [-256, 256]) of [A_ka]_{q_i} (centred, six digits per prime), of
// R_ka 2^54 / Q (six digits) and 2^40 / b_k, 2^32 / b_k at the top two bytes
// (v).  Every sum is an integer below 31 4 128 256 < 2^22, exact in the fp32
// accumulator; one more row of the right operand adds the constant that makes
// the float's bits an integer (round_shape.h).  CUDA cores only spread the
// bytes (two byte permutes and two subtractions per residue) and recombine
// the digits' sums.
//
// Why and where: the CUDA-core form spends 2 K (L + 1) wide multiplies (4.25
// issue cycles each) per coefficient, 540 at L = 8 (K = 30), where this one
// spends about 10 (L + 1): as a contraction of length 4 K with 6 L + 7 columns
// its products cost the tensor pipe a few per cent of the stage, a third of
// the kernel at L = 8.  Plans of 50% zeros before the 64-bit folds and this
// rounding against now (GB300): N = 16384, 32 x 64 x 16, 199.4 -> 168.9 ms;
// N = 8192, 32 x 32 x 16, 51.0 -> 40.1 ms; N = 4096, 32 x 32 x 32, 45.8 ->
// 39.9 ms, there with one CTA on an SM in place of two (the runtime reports
// one for any kernel that allocates tensor memory).  Two 32 x 64 x 16 matmuls
// at 60% zeros: 294 -> 246 ms, of which this rounding 267 -> 241 when it came.
// At L <= 4 (K <= 16) the two forms issue about as many instructions, 450 per
// coefficient and warp, and the stage waits for its residues and sums instead
// (2.3 MB of scratch per CTA, more than the CTAs' share of L2): measured with
// byte subnormals, bulk-copied residues and double-buffered tiles 64^3 gained
// 2.5% and the small ring (N = 4096) lost 20%, so those rings keep the
// CUDA-core form.
//
// The left operand is written to tensor memory by the thread that owns the
// row (no shared-memory layout), the right one sits in shared memory
// (K-major, no swizzle: core matrices of 8 columns x 16 bytes, 128 bytes
// apart along K), the accumulators come back by tcgen05.ld to the same thread.
#pragma once
#include "device_math.cuh"
#include "round_shape.h"

// ------------------------------------------------------ tensor memory -----
// The tcgen05 instructions with .sync.aligned are the warp's: PTX leaves them
// undefined unless all 32 lanes execute them together, which independent
// thread scheduling does not give after a branch or a spin that lanes leave
// at different times.  So every sequence of them starts with a __syncwarp()
// (tmem_alloc, tmem_dealloc, RoundMma::store_row, RoundMma::load_row).
// one warp; COLS a power of two, at least 32 (an immediate: with a register
// the occupancy calculation assumes all 512 columns)
template <int COLS>
SFHE_DEV void tmem_alloc(u32* slot)
{
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(slot)), "n"(COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
template <int COLS>
SFHE_DEV void tmem_dealloc(u32 base)  // the same warp
{
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "n"(COLS) : "memory");
}
SFHE_DEV void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
SFHE_DEV void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
SFHE_DEV void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// Waits for the warp's loads into w.  The registers hold the columns only
// behind the wait, which has no operands of its own: the empty statements make
// every use of w depend on it.
template <int NR>
SFHE_DEV void tmem_wait_ld(u32 (&w)[NR])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < NR; i++) asm volatile("" : "+r"(w[i]));
}
// eight columns of the calling warp's lanes
SFHE_DEV void tmem_st8(u32 addr, const u32* w)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(addr), "r"(w[0]),
                 "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                 : "memory");
}
SFHE_DEV void tmem_ld8(u32 (&w)[8], u32 addr)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                 : "r"(addr));
}
// D[128][NC] (+)= A[128][16] (tensor memory) B[NC][16]^T (shared memory), fp16 in, fp32 out
SFHE_DEV void mma_f16_ts(u32 d, u32 a, u64 bdesc, u32 idesc, u32 accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
        "r"(a), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// one arrival on bar when the issuing thread's earlier MMAs are complete
SFHE_DEV void mma_commit(u64* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
                 : "memory");
}

// ------------------------------------------------------------ rounding ----
template <int L, int K>
struct RoundMma {
    static constexpr int KC = round_shape(L, K).kc, NC = round_shape(L, K).nc;
    static constexpr int ACOLS = KC / 2;       // tensor-memory columns of a tile's left operand
    static constexpr int BYTES = NC * KC * 2;  // right operand
    static constexpr u32 IDESC = (1u << 4) | ((u32)(NC >> 3) << 17) | ((128u >> 4) << 24);
    static_assert(KC <= 128 && NC <= 64, "exactness: sums below 2^22");

    // two words (fp16 pairs) of x~: its bytes less 128 (0x64bb is the fp16
    // integer 1024 + bb, 0x6480 is 1152)
    SFHE_DEV static void pack(u32 x, u32& w0, u32& w1)
    {
        w0 = __byte_perm(x, 0x64646464u, 0x5140), w1 = __byte_perm(x, 0x64646464u, 0x5342);
        asm("sub.f16x2 %0, %0, %1;" : "+r"(w0) : "r"(0x64806480u));
        asm("sub.f16x2 %0, %0, %1;" : "+r"(w1) : "r"(0x64806480u));
    }
    // the coefficient's row: residues at src[k * stride] into the columns at
    // `a`; by whole warps
    SFHE_DEV static void store_row(const u32* __restrict__ src, size_t stride, u32 a)
    {
        u32 x[K];
#pragma unroll
        for (int k = 0; k < K; k++) x[k] = src[(size_t)k * stride];
        __syncwarp();
#pragma unroll
        for (int k0 = 0; k0 < KC / 4; k0 += 4) {
            u32 w[8];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                if (k0 + k < K) pack(x[k0 + k], w[2 * k], w[2 * k + 1]);
                else w[2 * k] = k0 + k == K ? 0x6800u : 0, w[2 * k + 1] = 0;  // the constant's 2048
            }
            tmem_st8(a + 2 * k0, w);
        }
        tmem_wait_st();
    }
    // one thread: the tile's product
    SFHE_DEV static void issue(u32 d, u32 a, u32 smem_b)
    {
        u64 desc = (u64)((smem_b >> 4) & 0x3FFF) | ((u64)(128 >> 4) << 16) | ((u64)((KC / 8 * 128) >> 4) << 32) | (1ull << 46);
#pragma unroll
        for (int ks = 0; ks < KC / 16; ks++, desc += 256 >> 4) mma_f16_ts(d, a + 8 * ks, desc, IDESC, ks);
    }
    // one wide multiply-add; the powers of two come from the kernel's
    // parameters, since a known one would be taken apart into shifts and adds
    SFHE_DEV static u64 madu(u32 a, u32 b, u64 c)
    {
        u64 d;
        asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
        return d;
    }
    // three digits' sums: c0 + u0 + 2^9 u1 + 2^18 u2
    SFHE_DEV static u64 join(u64 c0, u32 u0, u32 u1, u32 u2, const RnsConsts& c)
    {
        return madu(u2, c.mm_p18, madu(u1, c.mm_p9, c0 + u0));
    }
    // The accumulators of a row at d: r[i] = round(t x / Q) mod q_i for every
    // prime i, congruent and below 2^55.3; returns false when F is too close
    // to a half-integer to round (bits 27..53 of its fraction all equal after
    // adding a half; its error is below 2^15 units of 2^-54), and r is then
    // not valid.  By whole warps.
    template <int NP>  // NP = L
    SFHE_DEV static bool load_row(u32 d, const RnsConsts& c, u64 (&out)[NP])
    {
        u32 r[32];
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 4; q++) tmem_ld8(reinterpret_cast<u32(&)[8]>(r[8 * q]), d + 8 * q);
        tmem_wait_ld(r);
        const u32 v = (r[0] + c.mm_vc) >> 16;
        // F + 2^20 (the offset keeps it positive), in units of 2^-54: g0 + 2^27 g1
        const i64 g0 = mad_wide((int)v, c.mm_rb0n, (i64)join(c.mm_g0, r[1], r[2], r[3], c));
        const i64 g1 = mad_wide((int)v, c.mm_rb1n, (i64)join(c.mm_g1, r[4], r[5], r[6], c));
        const i64 s = g1 + (g0 >> 27) + (1 << 26);
        const u32 m = (u32)(s >> 27);  // round(F) + 2^20
        const bool ok = (((u32)s + 1) & ((1u << 27) - 1)) > 1;
#pragma unroll
        for (int i = 0; i < NP; i++) {
            if (i == 4) {
#pragma unroll
                for (int q = 0; q < (NC > 32 ? 3 : 0); q++) tmem_ld8(reinterpret_cast<u32(&)[8]>(r[8 * q]), d + 32 + 8 * q);
                tmem_wait_ld(r);
            }
            constexpr int COL[8] = {7, 13, 19, 25, 0, 6, 12, 18};  // round_mma_col(i) mod 32
            const int o = COL[i];
            const u64 p1 = madu(v, c.mm_nab_hi[i], join(0, r[o + 3], r[o + 4], r[o + 5], c));
            u64 p0 = madu(v, c.mm_nab_lo[i], join(c.mm_cq[i] + m, r[o], r[o + 1], r[o + 2], c));
            // p0 + 2^27 p1, 2^54 = c: p1 below 2^51
            p0 = madu((u32)(p1 >> 27), (u32)pm_c(c.m[i].q), p0);
            out[i] = madu((u32)p1 & ((1u << 27) - 1), c.mm_p27, p0);
        }
        return ok;
    }
};
