// The fp32-grade chunk engine: 16-token chunks whose products run on the tensor cores with every fp32 operand split
// into an fp16 head and an fp16 tail (22 significant bits; the three significant of the four partial products are
// added in fp32).  Used by the fp32 forward (sfda_forward_f32.cu) and the backward pass (sfda_backward.cu).
//
// Why split fp16: measured per SM and clock, mma.sync does 970 multiply-adds in fp16 and 484 in TF32, so three fp16
// products (323 effective) are twice as fast as 3 x TF32 (161) and 2.5 times the fp32 pipe (128), at the same 22 bits.
// fp16's exponent range is covered by powers of two: a chunk's tile of keys or queries is scaled so that its largest
// magnitude comes to lie at 2^14, a state, R, U and what else has value channels for rows channel by channel (RowScale).
// Entries down to 2^-16 of that largest one keep all 22 bits, smaller ones an absolute error of 2^-39 of it.
//
// Why chunks of 16: the state-sized products cost the same per token at any chunk size, the products inside a chunk
// grow with it, and inside 16 tokens the decays divide safely unless a coordinate loses more than 2^-16, which is
// checked per chunk (a slow exact path takes over then).
//
// Roles in a CTA: PREP warps make the operand tiles of a chunk into a ring of shared-memory slots, SOLVE warps the two
// Gram matrices and the inverse of the triangular system, and each CHAIN warp owns 16 value columns of the state in the
// accumulator layout of m16n8 with the value channel as the row.  That layout is also the A-operand layout of the next product,
// so a chain warp that has all keys goes R = V - W^* S -> U = M R -> S = gamma_C S + Y U with no exchange with other warps at
// all.  In blocks of 32 columns two warps have half of the keys each and exchange their parts of W^* S (and Q^* S) through
// shared memory once per chunk.  Blocks of columns of one pair are clusters, whose CTAs make the tiles in turn for all (Chain).
//
// Code counts: mma.sync holds its scheduler (sfda_forward_f32.cu), so every other instruction adds to the time, and
// unrolled code streams from the instruction caches (the first version was 93 KB for the forward).  So the operands of
// the Gram products come from the planes by ldmatrix instead of being split again, and every loop over key tiles is
// rolled.  Registers cannot be indexed at run time, hence the state lives in tensor memory -- a thread's accumulator
// fragment in consecutive columns of its lane -- and passes through registers 16 columns at a time, requested one step
// ahead; that also frees the 64 registers per thread it took.
#pragma once
#include <cstdlib>
#include "sfda_common.cuh"

namespace sfda {
namespace c16 {

constexpr int kC = 16;                       // tokens per chunk
constexpr int kSlots = 4;                    // operand tiles in flight
constexpr int kBarAux = 1, kBarFull = 2, kBarDone = 6, kBarFree = 10;   // hardware barriers; the last three: + slot

__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
#ifdef SFDA_WS_CHAOS
__device__ __forceinline__ void pause(uint32_t salt)              // of a warp (see chaos)
{
    chaos(salt);
    __syncwarp();
}
#else
__device__ __forceinline__ void pause(uint32_t) {}
#endif
__device__ __forceinline__ void bar_arrive(int id, int n)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
    pause(id);
}

// ---- tensor-core primitives ---------------------------------------------------------------------
__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// d = a b
__device__ __forceinline__ void mma_f16_z(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ void ldsm(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm_t(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ uint32_t transpose8x8(uint32_t a)
{
    uint32_t d;
    asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}
__device__ __forceinline__ uint32_t pack_f16(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ float2 unpack_f16(uint32_t x)
{
    float2 r;
    asm("{\n.reg .b16 a, b;\nmov.b32 {a, b}, %2;\ncvt.f32.f16 %0, a;\ncvt.f32.f16 %1, b;\n}" : "=f"(r.x), "=f"(r.y) : "r"(x));
    return r;
}
// re += Re(conj(b) a), im += Im(conj(b) a) for split complex operands (h: head, l: tail) and NT column tiles of b, tile n in
// registers 2 n and 2 n + 1.  An accumulator's next product is at least four instructions away, b's tails come first (their
// registers are free after a third of the products).  Two accumulators less by negating b's imaginary part: 543 us
// instead of 422 for the fp32 forward at B = 2, T = 2001, H = 16.
//
// The tensor core truncates its sums: with all 24 products of a 64-key sum in one accumulator the outputs were 1.7 times as
// far from 64-bit arithmetic as with sums rounded to nearest (5.3e-7, the CUDA-core kernel 3.1e-7).  So 16 keys at a time
// start from zero, small terms first, and are added with fp32 additions: 2.1e-7.  (415 -> 422 us at those sizes.)
template <int NT>
__device__ __forceinline__ void add_products(float (&re)[NT][4], float (&im)[NT][4], const uint32_t (&arh)[4], const uint32_t (&arl)[4],
                                             const uint32_t (&aih)[4], const uint32_t (&ail)[4], const uint32_t (&brh)[2 * NT],
                                             const uint32_t (&brl)[2 * NT], const uint32_t (&bih)[2 * NT], const uint32_t (&bil)[2 * NT])
{
    float x[NT][4], y[NT][4], z[NT][4], x2[NT][4];                 // Ar Br (+ Ai Bi), Ai Br, Ar Bi; one tile: Ai Bi by itself
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const uint32_t(&ar)[4] = k == 1 ? arl : arh;
        const uint32_t(&ai)[4] = k == 1 ? ail : aih;
        const uint32_t(&br)[2 * NT] = k == 0 ? brl : brh;
        const uint32_t(&bi)[2 * NT] = k == 0 ? bil : bih;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            if (k == 0) mma_f16_z(x[n], ar, br[2 * n], br[2 * n + 1]);
            else mma_f16(x[n], ar, br[2 * n], br[2 * n + 1]);
        }
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            if (k == 0) mma_f16_z(y[n], ai, br[2 * n], br[2 * n + 1]);
            else mma_f16(y[n], ai, br[2 * n], br[2 * n + 1]);
        }
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            if (NT > 1) mma_f16(x[n], ai, bi[2 * n], bi[2 * n + 1]);
            else if (k == 0) mma_f16_z(x2[n], ai, bi[2 * n], bi[2 * n + 1]);
            else mma_f16(x2[n], ai, bi[2 * n], bi[2 * n + 1]);
        }
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            if (k == 0) mma_f16_z(z[n], ar, bi[2 * n], bi[2 * n + 1]);
            else mma_f16(z[n], ar, bi[2 * n], bi[2 * n + 1]);
        }
    }
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            re[n][i] += NT > 1 ? x[n][i] : x[n][i] + x2[n][i];
            im[n][i] += y[n][i] - z[n][i];
        }
}
// head and tail of two values (already scaled)
__device__ __forceinline__ void split_f16(float x, float y, uint32_t &h, uint32_t &l)
{
    h = pack_f16(x, y);
    const float2 f = unpack_f16(h);
    l = pack_f16(x - f.x, y - f.y);
}
// Power of two that brings this magnitude into [2^14, 2^15), and its inverse.
__device__ __forceinline__ float scale_for(float largest, float &inv)
{
    const int e = max((int)(__float_as_uint(largest) >> 23) - 127, -100);
    inv = __uint_as_float((uint32_t)(113 + e) << 23);
    return __uint_as_float((uint32_t)(141 - e) << 23);
}
__device__ __forceinline__ float warp_max(float x) { return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(x))); }   // x >= 0
__device__ __forceinline__ float max_nan(float x, float y)     // NaN where either is
{
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(x), "f"(y));
    return r;
}
// Largest magnitudes of a fragment's two rows (value channels: lane >> 2, + 8) in this thread.
template <int N>
__device__ __forceinline__ float2 max_abs(const float (&x)[N][4], float2 m = make_float2(0.f, 0.f))
{
#pragma unroll
    for (int n = 0; n < N; ++n) {
        m.x = max_nan(m.x, max_nan(fabsf(x[n][0]), fabsf(x[n][1])));
        m.y = max_nan(m.y, max_nan(fabsf(x[n][2]), fabsf(x[n][3])));
    }
    return m;
}
// Scales of a fragment's rows, given the largest magnitudes in this thread.  Value channels do not interact, so every row has
// a scale of its own: an entry's precision does not depend on other channels, and one that is not finite spoils none.
// kStep: exponents go in steps of 1 or 4 (the largest entry of a row comes to lie in [2^14, 2^15) or [2^11, 2^15)); with
// steps neighbouring channels mostly share a scale all the same, which the gradients' sums over the channels are for.
struct RowScale {
    float inv[2];
};
template <int kStep>
__device__ __forceinline__ RowScale row_scale(float2 m)
{
    // both rows' leading 16 bits (all the exponent) at once through the row's four lanes
    uint32_t x = __byte_perm(__float_as_uint(m.x), __float_as_uint(m.y), 0x7632);
    x = __vmaxu2(x, __shfl_xor_sync(0xffffffffu, x, 1));
    x = __vmaxu2(x, __shfl_xor_sync(0xffffffffu, x, 2));
    RowScale r;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        // exponent + 1; that of an infinity or NaN counts as the smallest, so that it does not decide a shared scale
        const uint32_t e = max((i ? x >> 23 : (x << 16) >> 23) + 1u & 255u, 28u);
        r.inv[i] = __uint_as_float(kStep == 1 ? (e - 15u) << 23 : ((e + (kStep - 1) & ~(uint32_t)(kStep - 1)) - 15u) << 23);
    }
    return r;
}
__device__ __forceinline__ float scale_of(float inv) { return __uint_as_float(0x7f000000u - __float_as_uint(inv)); }   // 1 / a power of two
// A-operand registers (16 x 16) of two neighbouring accumulator tiles, scaled and split
__device__ __forceinline__ void split_tiles(const float *x, const float *y, const RowScale &r, uint32_t (&h)[4], uint32_t (&l)[4])
{
    const float s0 = scale_of(r.inv[0]), s1 = scale_of(r.inv[1]);
    split_f16(x[0] * s0, x[1] * s0, h[0], l[0]);
    split_f16(x[2] * s1, x[3] * s1, h[1], l[1]);
    split_f16(y[0] * s0, y[1] * s0, h[2], l[2]);
    split_f16(y[2] * s1, y[3] * s1, h[3], l[3]);
}
// cos / sin of a phase in 2^-32 turns: the quadrant is the two leading bits, the rest lies in [-pi/4, pi/4], where the
// Taylor polynomials to x^9 and x^10 are off by 2e-9 (half the code of sincospif, and code is what costs here)
__device__ __forceinline__ void cos_sin(uint32_t turns, float &c, float &s)
{
    const uint32_t q = (turns + 0x20000000u) >> 30;
    const float x = (float)(int32_t)(turns - (q << 30)) * 1.4629180792671596e-9f, y = x * x;
    float p = fmaf(y, 2.7557319e-6f, -1.9841270e-4f), r = fmaf(y, -2.7557319e-7f, 2.4801587e-5f);
    p = fmaf(y, p, 8.3333333e-3f);
    r = fmaf(y, r, -1.3888889e-3f);
    p = fmaf(y, p, -0.16666667f);
    r = fmaf(y, r, 4.1666667e-2f);
    p = fmaf(x * y, p, x);
    r = fmaf(y, fmaf(y, r, -0.5f), 1.f);
    const float cc = q & 1 ? p : r, ss = q & 1 ? r : p;
    c = (q + 1) & 2 ? -cc : cc;
    s = q & 2 ? -ss : ss;
}

// ---- inputs that are not finite -------------------------------------------------------------------
// The products over a chunk's tokens multiply by the zeros of triangular matrices, and zero times NaN is NaN: a token that
// is not finite would reach the outputs of the tokens before it, and the gradients of those behind it.  So it goes in as
// zeros (PREP: the keys' side for all channels, CHAIN: v and the cotangents channel by channel), and what it does reach in
// the recurrence becomes NaN explicitly: a channel's outputs from the token on and its state behind it, or, on the way
// back, its cotangents up to the token.  PREP sees it in the maxima that the scales need anyway and then does the chunk
// over; CHAIN takes its few values out as they come and asks only after the products whether there was one.  (PREP
// looking at its inputs first: 528 us instead of 444 for the fp32 forward at B = 2, T = 2001, H = 16; CHAIN branching in
// front of its products: 472 us, doing a step over: 567 us.)
// Tokens that are not finite in this thread's share of the two rows become zero; their bits, for every_lanes
__device__ __forceinline__ uint32_t take_out(float (&x)[2][4])
{
    uint32_t m = 0;
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const bool on = fabsf(x[n][i]) <= 3.402823466e38f;
            m |= on ? 0u : 1u << (8 * n + (i & 1) + 16 * (i >> 1));
            x[n][i] = on ? x[n][i] : 0.f;
        }
    return m;
}
// bit t: the row lane >> 2, bit 16 + t: the row + 8
__device__ __forceinline__ uint32_t every_lanes(uint32_t m, int lane)
{
    m <<= 2 * (lane & 3);
    m |= __shfl_xor_sync(0xffffffffu, m, 1);
    return m | __shfl_xor_sync(0xffffffffu, m, 2);
}
__device__ __forceinline__ uint32_t from_first(uint32_t m) { return m ? 0xffffu & ~((m & (0u - m)) - 1u) : 0u; }    // 16 tokens
__device__ __forceinline__ uint32_t to_last(uint32_t m) { return m ? 0xffffffffu >> __clz(m) : 0u; }
__device__ __forceinline__ uint32_t both(uint32_t m) { return m | m << 16; }
// (t0: the first tile's first token, 0 or 8)
template <int NT>
__device__ __forceinline__ void put_nan(float (&x)[NT][4], uint32_t m, int lane, int t0 = 0)
{
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (m >> (t0 + 8 * n + 2 * (lane & 3) + (i & 1) + 16 * (i >> 1)) & 1) x[n][i] = __int_as_float(0x7fc00000);
}
__device__ __forceinline__ void put_nan(float (&inv)[2], uint32_t m)      // the rows' scales: a state update with them is NaN
{
    if (m & 0xffffu) inv[0] = __int_as_float(0x7fc00000);
    if (m >> 16) inv[1] = __int_as_float(0x7fc00000);
}

// ---- the state in tensor memory: 16 columns of the thread's lane = two key tiles, [re 4, im 4] each ------------------
__device__ __forceinline__ void tm_load(float (&x)[16], uint32_t addr)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]), "=f"(x[4]), "=f"(x[5]), "=f"(x[6]), "=f"(x[7]), "=f"(x[8]),
                   "=f"(x[9]), "=f"(x[10]), "=f"(x[11]), "=f"(x[12]), "=f"(x[13]), "=f"(x[14]), "=f"(x[15])
                 : "r"(addr));
}
// the loaded registers pass through the wait, so that no use of them can be moved in front of it
__device__ __forceinline__ void tm_wait_load(float (&x)[16])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(x[0]), "+f"(x[1]), "+f"(x[2]), "+f"(x[3]), "+f"(x[4]), "+f"(x[5]), "+f"(x[6]), "+f"(x[7]), "+f"(x[8]),
                   "+f"(x[9]), "+f"(x[10]), "+f"(x[11]), "+f"(x[12]), "+f"(x[13]), "+f"(x[14]), "+f"(x[15])
                 :
                 : "memory");
}
__device__ __forceinline__ void tm_store(uint32_t addr, const float (&x)[16])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
                 ::"r"(addr), "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]), "f"(x[4]), "f"(x[5]), "f"(x[6]), "f"(x[7]), "f"(x[8]),
                 "f"(x[9]), "f"(x[10]), "f"(x[11]), "f"(x[12]), "f"(x[13]), "f"(x[14]), "f"(x[15])
                 : "memory");
}
__device__ __forceinline__ void tm_wait_store() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tm_alloc(uint32_t *where, int columns)     // one warp; columns: a power of two >= 32
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(where)), "r"(columns) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tm_free(uint32_t base, int columns)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(columns));
}

// ---- operand tiles of a chunk in shared memory --------------------------------------------------
// Complex matrices as four planes (Re head, Re tail, Im head, Im tail) of fp16 [16 tokens][keys] (or [16][16]), rows
// padded to an odd number of 16-byte units so that ldmatrix is free of bank conflicts:
//   W[t][j] = conj(gamma_t) k_t     Y[t][j] = (gamma_C/gamma_t) beta_t k_t     Q[t][j] = conj(gamma_t) q_t
//   Mt[t][i] = (I + K D_beta)^{-1}  Ab[t][i] = beta_i A^{qk}[t][i]             (unit lower / lower triangular)
template <int DK>
struct Tile {
    static constexpr int M = DK / 2, KT = M / 8, KS = M / 16;
    static constexpr int LDB = (M + 8) * 2;                       // bytes per row
    static constexpr int PL = 16 * LDB, BIG = 4 * PL;
    static constexpr int LDS = 48, PS = 16 * LDS, SMALL = 4 * PS;
    static constexpr int oW = 0, oY = BIG, oQ = 2 * BIG, oM = 3 * BIG, oA = oM + SMALL, oG = oA + SMALL, oS = oG + 8 * M;
    // oG: gamma_C float2 [M]; oS: inverse scales of W, Y, Q, M, A, Kb, then whether the chunk is fast, then its tokens that
    // are not finite (bit t: k, alpha, theta or beta, bit 16 + t: q); oB: beta [16]
    static constexpr int oB = oS + 32, bytes = (oB + 64 + 127) / 128 * 128;
};

// ---- CHAIN --------------------------------------------------------------------------------------
// acc[x] = products conj(X_x)^T S of NX tiles with the state at `st`, value channels in rows, tokens in columns, for
// each of two token tiles: [0] = Re = Xr Sr + Xi Si, [1] = Im = Xr Si - Xi Sr; scaled by s and the tiles' scales.
// KN: steps of 16 keys (all of them, or a warp's share).  pub(kk, rh, rl, ih, il) sees the split state of every step.
template <int DK, int NX, int KN, typename Pub>
__device__ __forceinline__ void keys_product(float (&acc)[NX][2][2][4], uint32_t st, const RowScale &s, const uint32_t (&tile)[NX],
                                             int lane, Pub pub)
{
    using TL = Tile<DK>;
#pragma unroll
    for (int x = 0; x < NX; ++x)
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[x][c][n][i] = 0.f;
    uint32_t at = (uint32_t)(((lane & 7) + ((lane >> 4) << 3)) * TL::LDB + ((lane >> 3) & 1) * 16);
    float x[16];
    tm_load(x, st);
    tm_wait_load(x);
#pragma unroll 1
    for (int kk = 0; kk < KN; ++kk, at += 32) {
        uint32_t rh[4], rl[4], ih[4], il[4];
        split_tiles(x, x + 8, s, rh, rl);
        split_tiles(x + 4, x + 12, s, ih, il);
        const bool more = kk + 1 < KN;
        if (more) tm_load(x, st + 16 * (kk + 1));
        pub(kk, rh, rl, ih, il);
#pragma unroll
        for (int t = 0; t < NX; ++t) {
            uint32_t brh[4], brl[4], bih[4], bil[4];
            const uint32_t p = tile[t] + at;
            ldsm(brl, p + TL::PL);
            ldsm(bil, p + 3 * TL::PL);
            ldsm(brh, p);
            ldsm(bih, p + 2 * TL::PL);
            if constexpr (NX == 1) {                              // (a column tile at a time: eight registers fewer)
#pragma unroll
                for (int n = 0; n < 2; ++n) {
                    const uint32_t h0[2] = {brh[2 * n], brh[2 * n + 1]}, l0[2] = {brl[2 * n], brl[2 * n + 1]};
                    const uint32_t h1[2] = {bih[2 * n], bih[2 * n + 1]}, l1[2] = {bil[2 * n], bil[2 * n + 1]};
                    add_products<1>(reinterpret_cast<float(&)[1][4]>(acc[t][0][n]), reinterpret_cast<float(&)[1][4]>(acc[t][1][n]), rh, rl,
                                    ih, il, h0, l0, h1, l1);
                }
            } else {
                add_products<2>(acc[t][0], acc[t][1], rh, rl, ih, il, brh, brl, bih, bil);
            }
        }
        if (more) tm_wait_load(x);
    }
}

// A-operand registers of a complex [value x 16 tokens] matrix
struct TokFrag {
    uint32_t rh[4], rl[4], ih[4], il[4];
};

// B-operand registers (all four planes) of a [16][16] tile; kT: k runs over the tile's rows instead of its columns
template <bool kT>
__device__ __forceinline__ void load_small(TokFrag &b, uint32_t tile, int lane)
{
    constexpr int LD = 48, PS = 16 * LD;
    if constexpr (kT) {
        const uint32_t p = tile + (uint32_t)(((lane & 7) + (((lane >> 3) & 1) << 3)) * LD + (lane >> 4) * 16);
        ldsm_t(b.rh, p);
        ldsm_t(b.rl, p + PS);
        ldsm_t(b.ih, p + 2 * PS);
        ldsm_t(b.il, p + 3 * PS);
    } else {
        const uint32_t p = tile + (uint32_t)(((lane & 7) + ((lane >> 4) << 3)) * LD + ((lane >> 3) & 1) * 16);
        ldsm(b.rh, p);
        ldsm(b.rl, p + PS);
        ldsm(b.ih, p + 2 * PS);
        ldsm(b.il, p + 3 * PS);
    }
}

// out = a b (kConj: a conj(b)) over 16 tokens, both complex, unscaled by f and the rows' inv; NT column tiles of b
template <bool kConj, int NT>
__device__ __forceinline__ void product_small(float (&re)[NT][4], float (&im)[NT][4], const TokFrag &a, const TokFrag &b, const float (&inv)[2], float f)
{
    float rr[NT][4], ii[NT][4], ir[NT][4], ri[NT][4];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const uint32_t(&ar)[4] = k == 0 ? a.rl : a.rh;
        const uint32_t(&ai)[4] = k == 0 ? a.il : a.ih;
        const uint32_t(&br)[4] = k == 1 ? b.rl : b.rh;
        const uint32_t(&bi)[4] = k == 1 ? b.il : b.ih;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            if (k == 0) {
                mma_f16_z(rr[n], ar, br[2 * n], br[2 * n + 1]);
                mma_f16_z(ii[n], ai, bi[2 * n], bi[2 * n + 1]);
                mma_f16_z(ir[n], ai, br[2 * n], br[2 * n + 1]);
                mma_f16_z(ri[n], ar, bi[2 * n], bi[2 * n + 1]);
            } else {
                mma_f16(rr[n], ar, br[2 * n], br[2 * n + 1]);
                mma_f16(ii[n], ai, bi[2 * n], bi[2 * n + 1]);
                mma_f16(ir[n], ai, br[2 * n], br[2 * n + 1]);
                mma_f16(ri[n], ar, bi[2 * n], bi[2 * n + 1]);
            }
        }
    }
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            re[n][i] = (inv[i >> 1] * f) * (kConj ? rr[n][i] + ii[n][i] : rr[n][i] - ii[n][i]);
            im[n][i] = (inv[i >> 1] * f) * (kConj ? ir[n][i] - ri[n][i] : ir[n][i] + ri[n][i]);
        }
}

// scale and split a [value x 16 tokens] matrix
__device__ __forceinline__ RowScale make_frag(TokFrag &f, const float (&re)[2][4], const float (&im)[2][4])
{
    const RowScale r = row_scale<1>(max_abs(im, max_abs(re)));
    split_tiles(re[0], re[1], r, f.rh, f.rl);
    split_tiles(im[0], im[1], r, f.ih, f.il);
    return r;
}
// The inverse of the scale for sums over a warp's channels: that of its largest row; own: some row has another.
__device__ __forceinline__ float shared_scale(const RowScale &r, bool &own)
{
    const float all = warp_max(fmaxf(r.inv[0], r.inv[1]));
    own = __any_sync(0xffffffffu, r.inv[0] != all || r.inv[1] != all);
    return all;
}
// Split operands from the rows' scales to the shared one (a power of two: exact unless bits fall off the end)
__device__ __forceinline__ void to_shared_scale(uint32_t (&x)[4], const RowScale &r, float all)
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float f = r.inv[i & 1] * scale_of(all);
        const uint32_t f2 = pack_f16(f, f);
        asm("mul.rn.f16x2 %0, %0, %1;" : "+r"(x[i]) : "r"(f2));
    }
}

// re, im (two key tiles of eight) = a X with tokens as k: X the tile at `at` (B operand by transposed loads);
// nih, nil = the imaginary registers of `a` negated
template <int DK>
__device__ __forceinline__ void tokens_product(float (&re)[2][4], float (&im)[2][4], const TokFrag &a, const uint32_t (&nih)[4],
                                               const uint32_t (&nil)[4], uint32_t at)
{
    using TL = Tile<DK>;
    uint32_t brh[4], brl[4], bih[4], bil[4];
    ldsm_t(brh, at);
    ldsm_t(bih, at + 2 * TL::PL);
    ldsm_t(brl, at + TL::PL);
    ldsm_t(bil, at + 3 * TL::PL);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const uint32_t(&ar)[4] = k == 0 ? a.rl : a.rh;
        const uint32_t(&ai)[4] = k == 0 ? a.il : a.ih;
        const uint32_t(&an)[4] = k == 0 ? nil : nih;
        const uint32_t(&br)[4] = k == 1 ? brl : brh;
        const uint32_t(&bi)[4] = k == 1 ? bil : bih;
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            if (k == 0) mma_f16_z(re[n], ar, br[2 * n], br[2 * n + 1]);
            else mma_f16(re[n], ar, br[2 * n], br[2 * n + 1]);
        }
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            if (k == 0) mma_f16_z(im[n], ai, br[2 * n], br[2 * n + 1]);
            else mma_f16(im[n], ai, br[2 * n], br[2 * n + 1]);
        }
#pragma unroll
        for (int n = 0; n < 2; ++n) mma_f16(re[n], an, bi[2 * n], bi[2 * n + 1]);
#pragma unroll
        for (int n = 0; n < 2; ++n) mma_f16(im[n], ar, bi[2 * n], bi[2 * n + 1]);
    }
}

// The thread's 16 elements (token 8 n + (i & 1), column + 8 (i >> 1)) of a [token][column] array: `p` points at the
// first, `step` is a token's distance, `left` the number of tokens from p's on.
template <typename T>
__device__ __forceinline__ void load_rows(float (&x)[2][4], const T *p, size_t step, int left)
{
#pragma unroll
    for (int n = 0; n < 2; ++n, p += 8 * step)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const T *r = p + (e ? step : 0);
            const bool on = 8 * n + e < left;
            x[n][e] = on ? ld_val(r, 0) : 0.f;
            x[n][e + 2] = on ? ld_val(r, 8) : 0.f;
        }
}
template <typename T, int NT>
__device__ __forceinline__ void store_rows(T *p, const float (&x)[NT][4], size_t step, int left)
{
#pragma unroll
    for (int n = 0; n < NT; ++n, p += 8 * step)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            T *r = p + (e ? step : 0);
            if (8 * n + e < left) {
                st_val(r, 0, x[n][e]);
                st_val(r, 8, x[n][e + 2]);
            }
        }
}

// The thread's fragment of a state [d_k][dv] (paired rows) at `p` (its key pair 2 (lane & 3), its column); returns the
// largest magnitudes of its two rows.  p = NULL: zeros.
template <int KN>
__device__ __forceinline__ float2 state_from_memory(uint32_t st, const float *p, int dv)
{
    float2 largest = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int n = 0; n < KN; ++n) {
        float x[16];
#pragma unroll
        for (int i = 0; i < 16; ++i)                              // [key tile][Re / Im][column half][key]
            x[i] = p ? p[(size_t)(32 * n + 16 * (i >> 3) + 2 * (i & 1) + ((i >> 2) & 1)) * dv + 8 * ((i >> 1) & 1)] : 0.f;
        largest = max_abs(reinterpret_cast<const float(&)[4][4]>(x), largest);
        tm_store(st + 16 * n, x);
    }
    tm_wait_store();
    return largest;
}
template <int KN>
__device__ __forceinline__ void state_to_memory(uint32_t st, float *p, int dv)
{
#pragma unroll 1
    for (int n = 0; n < KN; ++n) {
        float x[16];
        tm_load(x, st + 16 * n);
        tm_wait_load(x);
#pragma unroll
        for (int i = 0; i < 16; ++i) p[(size_t)(32 * n + 16 * (i >> 3) + 2 * (i & 1) + ((i >> 2) & 1)) * dv + 8 * ((i >> 1) & 1)] = x[i];
    }
}

// S <- gamma_C S + f inv a Y, the state at `st`, inv per row; returns the largest magnitudes of the new state's rows
template <int DK, int KN>
__device__ __forceinline__ float2 state_update(uint32_t st, const TokFrag &a, const float (&inv)[2], float f, uint32_t tile, const float4 *gamma, int lane)
{
    using TL = Tile<DK>;
    uint32_t nih[4], nil[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        nih[i] = a.ih[i] ^ 0x80008000u;
        nil[i] = a.il[i] ^ 0x80008000u;
    }
    uint32_t at = tile + (uint32_t)(((lane & 7) + (((lane >> 3) & 1) << 3)) * TL::LDB + (lane >> 4) * 16);
    gamma += lane & 3;
    const float fr[2] = {inv[0] * f, inv[1] * f};
    float2 largest = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int np = 0; np < KN; ++np, at += 32, gamma += 8, st += 16) {
        float x[16], re[2][4], im[2][4];
        tm_load(x, st);
        tokens_product<DK>(re, im, a, nih, nil, at);
        tm_wait_load(x);
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            const float4 g = gamma[4 * n];                       // gamma_C of keys 8 n + 2 (lane & 3), + 1
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float gr = (i & 1) ? g.z : g.x, gi = (i & 1) ? g.w : g.y, u = x[8 * n + i], v = x[8 * n + 4 + i];
                x[8 * n + i] = fmaf(fr[i >> 1], re[n][i], gr * u - gi * v);
                x[8 * n + 4 + i] = fmaf(fr[i >> 1], im[n][i], gr * v + gi * u);
            }
        }
        largest = max_abs(reinterpret_cast<const float(&)[4][4]>(x), largest);
        tm_store(st, x);
    }
    tm_wait_store();
    return largest;
}

// ---- PREP and SOLVE ------------------------------------------------------------------------------
// PREP (PW warps): a thread owns two neighbouring keys and kC / NG consecutive tokens, so that global rows are read and
// operand rows written in whole words.  The decays' products and the phases' sums cross the token groups through
// shared memory.  SOLVE: one warp per Gram matrix, straight from the operand planes.
template <int DK, int PW>
struct PrepMap {
    static constexpr int M = DK / 2, PAIRS = M / 2, NG = 32 * PW / PAIRS, TPT = kC / NG;
    static_assert(NG * PAIRS == 32 * PW && TPT * NG == kC && TPT >= 1, "token groups must tile the chunk");
    static constexpr int scan_bytes = NG * PAIRS * 16 + 5 * PW * 4;          // products, phase sums, the warps' maxima and tokens taken out
    static constexpr int slow_bytes = kC * (M + 4) * 8 * 3;                 // k', q', alpha of a chunk that is not fast
};

template <typename T> struct KeyPair;
template <> struct KeyPair<float> {
    float4 v;
    __device__ __forceinline__ void zero() { v = make_float4(0.f, 0.f, 0.f, 0.f); }
    __device__ __forceinline__ void load(const float *p) { v = *reinterpret_cast<const float4 *>(p); }
    __device__ __forceinline__ float4 get() const { return v; }
};
template <> struct KeyPair<__nv_bfloat16> {
    uint2 v;
    __device__ __forceinline__ void zero() { v = make_uint2(0u, 0u); }
    __device__ __forceinline__ void load(const __nv_bfloat16 *p) { v = *reinterpret_cast<const uint2 *>(p); }
    __device__ __forceinline__ float4 get() const
    {
        return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                           __uint_as_float(v.y & 0xffff0000u));
    }
};

template <int TPT, typename T>
struct PrepRaw {
    KeyPair<T> k[TPT], q[TPT];
    float2 al[TPT], th[TPT];
    float be[TPT];
};

template <int DK, int PW, typename T>
__device__ __forceinline__ void prep_fetch(PrepRaw<PrepMap<DK, PW>::TPT, T> &in, const T *__restrict__ q, const T *__restrict__ k,
                                           const float *__restrict__ alpha, const float *__restrict__ theta,
                                           const float *__restrict__ beta, size_t row0, int H, int t0, int T_, bool needq, int tid)
{
    using PM = PrepMap<DK, PW>;
    const int pair = tid % PM::PAIRS, t1 = t0 + tid / PM::PAIRS * PM::TPT;
#pragma unroll
    for (int x = 0; x < PM::TPT; ++x) {
        in.k[x].zero();
        in.q[x].zero();
        in.al[x] = make_float2(1.f, 1.f);
        in.th[x] = make_float2(0.f, 0.f);
        in.be[x] = 0.f;
        if (t1 + x < T_) {
            const size_t row = row0 + (size_t)(t1 + x) * H;
            in.k[x].load(k + row * DK + 4 * pair);
            if (needq) in.q[x].load(q + row * DK + 4 * pair);
            in.al[x] = *reinterpret_cast<const float2 *>(alpha + row * PM::M + 2 * pair);
            in.th[x] = *reinterpret_cast<const float2 *>(theta + row * PM::M + 2 * pair);
            in.be[x] = beta[row];
        }
    }
}

// The rare path: a thread's tokens that are not finite in any of the warp's keys become zeros (alpha 1); the bits of the
// warp's tokens are returned
template <int TPT, typename T>
__device__ __forceinline__ uint32_t take_out(PrepRaw<TPT, T> &in, int t)
{
    uint32_t m = 0;
#pragma unroll
    for (int x = 0; x < TPT; ++x) {
        const float4 k = in.k[x].get(), q = in.q[x].get();
        const float zk = fmaf(k.x, 0.f, fmaf(k.y, 0.f, fmaf(k.z, 0.f, k.w * 0.f))), zq = fmaf(q.x, 0.f, fmaf(q.y, 0.f, fmaf(q.z, 0.f, q.w * 0.f)));
        const float za = fmaf(in.al[x].x, 0.f, fmaf(in.al[x].y, 0.f, fmaf(in.th[x].x, 0.f, fmaf(in.th[x].y, 0.f, fmaf(in.be[x], 0.f, zk)))));
        if (za != 0.f) m |= 1u << (t + x);
        if (zq != 0.f) m |= 0x10000u << (t + x);
    }
    m = __reduce_or_sync(0xffffffffu, m);
    if (m) {
#pragma unroll
        for (int x = 0; x < TPT; ++x) {
            if (m >> (t + x) & 1) {
                in.k[x].zero();
                in.al[x] = make_float2(1.f, 1.f);
                in.th[x] = make_float2(0.f, 0.f);
                in.be[x] = 0.f;
            }
            if (m >> (16 + t + x) & 1) in.q[x].zero();
        }
    }
    return m;
}

// two keys of one token into the four planes
__device__ __forceinline__ void put_planes(unsigned char *p, int pl, float r0, float i0, float r1, float i1)
{
    uint32_t h, l;
    split_f16(r0, r1, h, l);
    *reinterpret_cast<uint32_t *>(p) = h;
    *reinterpret_cast<uint32_t *>(p + pl) = l;
    split_f16(i0, i1, h, l);
    *reinterpret_cast<uint32_t *>(p + 2 * pl) = h;
    *reinterpret_cast<uint32_t *>(p + 3 * pl) = l;
}

// Operand planes of one chunk: W, Y (and Q, with needq) into the slot, Kb_i = beta_i k_i / gamma_i into `kb` for the Gram products.
// `vals` (or NULL) receives what the gradients need again, a float4 per (token, key): prod alpha up to the token and after
// it, e^{i phi}.  Called by all 32 PW threads (BAR: their barrier); the planes are
// complete for other threads only after a barrier of the caller's.
//
// The division by gamma_i is bounded by 2^16 inside a fast chunk (every coordinate keeps at least 2^-16 over the 16
// tokens): Kb's entries then reach 2^16, the smaller ones keep an absolute error of 2^-39 of that, 2^-23 beside the
// unit-sized entries of W they meet.  Stronger decays take slow_gram.  Returns whether the chunk is fast, or -1 where it
// is not finite -- unless kAgain: this has been seen to, by leaving out the tokens `out` (the same value in every thread).
template <int DK, int PW, int BAR, bool kAgain, typename T>
__device__ __forceinline__ int prep_planes(const PrepRaw<PrepMap<DK, PW>::TPT, T> &in, float4 *vals, unsigned char *slot,
                                           unsigned char *kb, unsigned char *scan, bool needq, int tid, uint32_t out)
{
    using PM = PrepMap<DK, PW>;
    using TL = Tile<DK>;
    constexpr int M = PM::M, PAIRS = PM::PAIRS, NG = PM::NG, TPT = PM::TPT;
    const int pair = tid % PAIRS, grp = tid / PAIRS, lane = tid & 31, warp = tid >> 5;
    float2 *sp = reinterpret_cast<float2 *>(scan);
    uint2 *su = reinterpret_cast<uint2 *>(scan + NG * PAIRS * 8);
    uint32_t *red = reinterpret_cast<uint32_t *>(scan + NG * PAIRS * 16);

    float2 p[TPT], sf[TPT];
    uint2 u[TPT];
#pragma unroll
    for (int x = 0; x < TPT; ++x) {
        p[x] = make_float2(fmaf(in.th[x].x, 0.f, in.al[x].x), fmaf(in.th[x].y, 0.f, in.al[x].y));   // (NaN where theta is not finite)
        u[x] = make_uint2(phase_to_turns(in.th[x].x), phase_to_turns(in.th[x].y));
        if (x) {
            p[x] = make_float2(p[x - 1].x * p[x].x, p[x - 1].y * p[x].y);
            u[x] = make_uint2(u[x - 1].x + u[x].x, u[x - 1].y + u[x].y);
        }
    }
    sf[TPT - 1] = make_float2(1.f, 1.f);
#pragma unroll
    for (int x = TPT - 2; x >= 0; --x) sf[x] = make_float2(sf[x + 1].x * in.al[x + 1].x, sf[x + 1].y * in.al[x + 1].y);
    sp[grp * PAIRS + pair] = p[TPT - 1];
    su[grp * PAIRS + pair] = u[TPT - 1];
    bar_sync(BAR, 32 * PW);
    float2 pre = make_float2(1.f, 1.f), suf = pre, aC = pre;
    uint2 ub = make_uint2(0u, 0u), uc = ub;
#pragma unroll 2
    for (int gg = 0; gg < NG; ++gg) {                              // the same order in every thread: aC decides `fast`
        const float2 f = sp[gg * PAIRS + pair];
        const uint2 v = su[gg * PAIRS + pair];
        aC = make_float2(aC.x * f.x, aC.y * f.y);
        uc = make_uint2(uc.x + v.x, uc.y + v.y);
        if (gg < grp) {
            pre = make_float2(pre.x * f.x, pre.y * f.y);
            ub = make_uint2(ub.x + v.x, ub.y + v.y);
        }
        if (gg > grp) suf = make_float2(suf.x * f.x, suf.y * f.y);
    }
    const bool fast = __reduce_min_sync(0xffffffffu, __float_as_uint(fminf(aC.x, aC.y))) >= 0x37800000u;   // 2^-16
    float2 gc0, gc1;                                              // e^{i phi_C}
    cos_sin(uc.x, gc0.x, gc0.y);
    cos_sin(uc.y, gc1.x, gc1.y);
    if (grp == 0)
        reinterpret_cast<float4 *>(slot + TL::oG)[pair] = make_float4(aC.x * gc0.x, aC.x * gc0.y, aC.y * gc1.x, aC.y * gc1.y);

    float4 kk[TPT], qq[TPT];
    float2 av[TPT], yf[TPT], bi[TPT];
    float mw = 0.f, my = 0.f, mq = 0.f, mb = 0.f;
    if (pair == 0) {
#pragma unroll
        for (int x = 0; x < TPT; ++x) reinterpret_cast<float *>(slot + TL::oB)[grp * TPT + x] = in.be[x];
    }
#pragma unroll
    for (int x = 0; x < TPT; ++x) {
        const int t = grp * TPT + x;
        av[x] = make_float2(pre.x * p[x].x, pre.y * p[x].y);
        sf[x] = make_float2(sf[x].x * suf.x, sf[x].y * suf.y);
        yf[x] = make_float2(sf[x].x * in.be[x], sf[x].y * in.be[x]);
        float c0, s0, c1, s1;
        cos_sin(ub.x + u[x].x, c0, s0);
        cos_sin(ub.y + u[x].y, c1, s1);
        float4 r = in.k[x].get();
        kk[x] = make_float4(r.x * c0 + r.y * s0, r.y * c0 - r.x * s0, r.z * c1 + r.w * s1, r.w * c1 - r.z * s1);
        qq[x] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (needq) {
            r = in.q[x].get();
            qq[x] = make_float4(r.x * c0 + r.y * s0, r.y * c0 - r.x * s0, r.z * c1 + r.w * s1, r.w * c1 - r.z * s1);
            if (vals) {
                float4 *o = vals + t * M + 2 * pair;
                o[0] = make_float4(av[x].x, sf[x].x, c0, s0);
                o[1] = make_float4(av[x].y, sf[x].y, c1, s1);
            }
            qq[x] = make_float4(av[x].x * qq[x].x, av[x].x * qq[x].y, av[x].y * qq[x].z, av[x].y * qq[x].w);
            mq = max_nan(max_nan(mq, max_nan(fabsf(qq[x].x), fabsf(qq[x].y))), max_nan(fabsf(qq[x].z), fabsf(qq[x].w)));
        }
        bi[x] = fast ? make_float2(__fdividef(in.be[x], av[x].x), __fdividef(in.be[x], av[x].y)) : make_float2(0.f, 0.f);
        const float n0 = fabsf(kk[x].x) + fabsf(kk[x].y), n1 = fabsf(kk[x].z) + fabsf(kk[x].w);   // bounds both parts
        mw = max_nan(mw, max_nan(av[x].x * n0, av[x].y * n1));
        my = max_nan(my, max_nan(fabsf(yf[x].x) * n0, fabsf(yf[x].y) * n1));
        mb = max_nan(mb, max_nan(fabsf(bi[x].x) * n0, fabsf(bi[x].y) * n1));
    }
    uint32_t m[4] = {__float_as_uint(mw), __float_as_uint(my), __float_as_uint(mq), __float_as_uint(mb)};   // all >= 0
#pragma unroll
    for (int i = 0; i < 4; ++i)
        m[i] = __reduce_max_sync(0xffffffffu, m[i]);
    if (lane == 0) {
        *reinterpret_cast<uint4 *>(red + 4 * warp) = make_uint4(m[0], m[1], m[2], m[3]);
        if (kAgain) red[4 * PW + warp] = out;
    }
    bar_sync(BAR, 32 * PW);
#pragma unroll 2
    for (int w = 0; w < PW; ++w) {
        const uint4 r = *reinterpret_cast<const uint4 *>(red + 4 * w);
        m[0] = max(m[0], r.x);
        m[1] = max(m[1], r.y);
        m[2] = max(m[2], r.z);
        m[3] = max(m[3], r.w);
    }
    if (!kAgain && max(max(m[0], m[1]), max(m[2], m[3])) >= 0x7f800000u) return -1;
    float iw, iy, iq, ib;
    const float sw = scale_for(__uint_as_float(m[0]), iw), sy = scale_for(__uint_as_float(m[1]), iy);
    const float sq = scale_for(__uint_as_float(m[2]), iq), sb = scale_for(__uint_as_float(m[3]), ib);
    if (tid == 0) {
        float *inv = reinterpret_cast<float *>(slot + TL::oS);
        inv[0] = iw;
        inv[1] = iy;
        inv[2] = iq;
        inv[5] = ib;
        reinterpret_cast<int *>(inv)[6] = fast;
        uint32_t all = 0;
        if (kAgain)
            for (int w = 0; w < PW; ++w) all |= red[4 * PW + w];
        reinterpret_cast<uint32_t *>(inv)[7] = all;
    }
#pragma unroll
    for (int x = 0; x < TPT; ++x) {
        const int at = (grp * TPT + x) * TL::LDB + 4 * pair;
        const float w0 = av[x].x * sw, w1 = av[x].y * sw, y0 = yf[x].x * sy, y1 = yf[x].y * sy;
        put_planes(slot + TL::oW + at, TL::PL, w0 * kk[x].x, w0 * kk[x].y, w1 * kk[x].z, w1 * kk[x].w);
        put_planes(slot + TL::oY + at, TL::PL, y0 * (gc0.x * kk[x].x - gc0.y * kk[x].y), y0 * (gc0.x * kk[x].y + gc0.y * kk[x].x),
                   y1 * (gc1.x * kk[x].z - gc1.y * kk[x].w), y1 * (gc1.x * kk[x].w + gc1.y * kk[x].z));
        if (needq) put_planes(slot + TL::oQ + at, TL::PL, sq * qq[x].x, sq * qq[x].y, sq * qq[x].z, sq * qq[x].w);
        if (fast) {
            const float b0 = bi[x].x * sb, b1 = bi[x].y * sb;
            put_planes(kb + at, TL::PL, b0 * kk[x].x, b0 * kk[x].y, b1 * kk[x].z, b1 * kk[x].w);
        }
    }
    return fast;
}

// prep_planes for a chunk that is not finite: once more, without the tokens that are not
template <int DK, int PW, int BAR, typename T>
__device__ __noinline__ bool prep_again(const T *q, const T *k, const float *alpha, const float *theta, const float *beta, size_t row0, int H, int t0,
                                        int T_, float4 *vals, unsigned char *slot, unsigned char *kb, unsigned char *scan, bool needq, int tid)
{
    using PM = PrepMap<DK, PW>;
    PrepRaw<PM::TPT, T> in;
    prep_fetch<DK, PW, T>(in, q, k, alpha, theta, beta, row0, H, t0, T_, needq, tid);
    const uint32_t out = take_out<PM::TPT, T>(in, tid / PM::PAIRS * PM::TPT);
    return prep_planes<DK, PW, BAR, true, T>(in, vals, slot, kb, scan, needq, tid, out) != 0;
}
// the chunk at t0, whose inputs are in `in`
template <int DK, int PW, int BAR, typename T>
__device__ __forceinline__ bool prep_chunk(const PrepRaw<PrepMap<DK, PW>::TPT, T> &in, const T *q, const T *k, const float *alpha, const float *theta,
                                           const float *beta, size_t row0, int H, int t0, int T_, float4 *vals, unsigned char *slot,
                                           unsigned char *kb, unsigned char *scan, bool needq, int tid)
{
    const int fast = prep_planes<DK, PW, BAR, false, T>(in, vals, slot, kb, scan, needq, tid, 0);
    return fast < 0 ? prep_again<DK, PW, BAR, T>(q, k, alpha, theta, beta, row0, H, t0, T_, vals, slot, kb, scan, needq, tid) : fast != 0;
}

// The Gram matrices of a chunk whose decays are too strong to divide by: every pair's decay as a running product.  Called
// by all 32 PW threads after prep_planes returned false; `slow` is a scratch of PrepMap::slow_bytes nobody else uses.
// Reads its inputs again: passed on, they would not stay in registers on the common path.
template <int DK, int PW, int BAR, typename T>
__device__ __noinline__ void slow_gram(const T *q, const T *k, const float *alpha, const float *theta, const float *beta,
                                       size_t row0, int H, int t0, int T_, unsigned char *slow, const unsigned char *scan,
                                       float2 *gk, float2 *gq, bool needq, int tid)
{
    using PM = PrepMap<DK, PW>;
    PrepRaw<PM::TPT, T> in;
    prep_fetch<DK, PW, T>(in, q, k, alpha, theta, beta, row0, H, t0, T_, needq, tid);
    constexpr int M = PM::M, PAIRS = PM::PAIRS, TPT = PM::TPT, LD = M + 4;
    const int pair = tid % PAIRS, grp = tid / PAIRS, lane = tid & 31, warp = tid >> 5;
    take_out<PM::TPT, T>(in, grp * TPT);
    const uint2 *su = reinterpret_cast<const uint2 *>(scan + PM::NG * PAIRS * 8);
    float2 *sk = reinterpret_cast<float2 *>(slow), *sq = sk + kC * LD, *sa = sq + kC * LD;   // sa: (alpha, beta)
    uint2 ub = make_uint2(0u, 0u);
    for (int gg = 0; gg < grp; ++gg) ub = make_uint2(ub.x + su[gg * PAIRS + pair].x, ub.y + su[gg * PAIRS + pair].y);
#pragma unroll
    for (int x = 0; x < TPT; ++x) {
        const int at = (grp * TPT + x) * LD + 2 * pair;
        ub = make_uint2(ub.x + phase_to_turns(in.th[x].x), ub.y + phase_to_turns(in.th[x].y));
        float c0, s0, c1, s1;
        cos_sin(ub.x, c0, s0);
        cos_sin(ub.y, c1, s1);
        float4 r = in.k[x].get();
        sk[at] = make_float2(r.x * c0 + r.y * s0, r.y * c0 - r.x * s0);
        sk[at + 1] = make_float2(r.z * c1 + r.w * s1, r.w * c1 - r.z * s1);
        if (needq) {
            r = in.q[x].get();
            sq[at] = make_float2(r.x * c0 + r.y * s0, r.y * c0 - r.x * s0);
            sq[at + 1] = make_float2(r.z * c1 + r.w * s1, r.w * c1 - r.z * s1);
        }
        sa[at] = make_float2(in.al[x].x, in.be[x]);
        sa[at + 1] = make_float2(in.al[x].y, in.be[x]);
    }
    bar_sync(BAR, 32 * PW);
    for (int t = warp; t < kC; t += PW) {
        float w[M / 32];
#pragma unroll
        for (int e = 0; e < M / 32; ++e) w[e] = 1.f;
        for (int i = t; i >= 0; --i) {
            float s[4] = {0.f, 0.f, 0.f, 0.f};
            float be = 0.f;
#pragma unroll
            for (int e = 0; e < M / 32; ++e) {
                const int j = lane + 32 * e;
                const float2 b = sk[i * LD + j], x = sk[t * LD + j], ab = sa[i * LD + j];
                const float br = w[e] * b.x, bim = w[e] * b.y;
                s[0] += x.x * br + x.y * bim;
                s[1] += x.x * bim - x.y * br;
                if (needq) {
                    const float2 y = sq[t * LD + j];
                    s[2] += y.x * br + y.y * bim;
                    s[3] += y.x * bim - y.y * br;
                }
                w[e] *= ab.x;
                be = ab.y;
            }
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1)
#pragma unroll
                for (int e = 0; e < 4; ++e) s[e] += __shfl_xor_sync(0xffffffffu, s[e], d);
            if (lane == 0) {
                gk[t * 17 + i] = make_float2(be * s[0], be * s[1]);
                if (needq) gq[t * 17 + i] = make_float2(be * s[2], be * s[3]);
            }
        }
    }
}

// X^* Kb (X = W or Q) for the columns 8 nt0 .. of NT tiles of eight, by one warp, into [17] float2 rows
template <int DK, int NT>
__device__ __forceinline__ void gram_tiles(uint32_t x, uint32_t kb, float f, float2 *out, int nt0, int lane)
{
    using TL = Tile<DK>;
    const int g = lane >> 2, t4 = lane & 3;
    uint32_t pa = x + (uint32_t)(((lane & 7) + (((lane >> 3) & 1) << 3)) * TL::LDB + (lane >> 4) * 16);
    // B registers of both halves of a k-step for the heads (lanes 0-15) and the tails (lanes 16-31)
    uint32_t pb = kb + (uint32_t)((8 * nt0 + (lane & 7)) * TL::LDB + ((lane >> 3) & 1) * 16 + (lane >> 4) * TL::PL);
    float re[NT][4], im[NT][4];                     // im: of a conj(b), negated at the end
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) re[n][i] = im[n][i] = 0.f;
#pragma unroll 1
    for (int kk = 0; kk < TL::KS; ++kk, pa += 32, pb += 32) {
        uint32_t rh[4], rl[4], ih[4], il[4], br[NT][4], bi[NT][4];
        ldsm(rh, pa);
        ldsm(ih, pa + 2 * TL::PL);
        ldsm(rl, pa + TL::PL);
        ldsm(il, pa + 3 * TL::PL);
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            ldsm(br[n], pb + n * 8 * TL::LDB);
            ldsm(bi[n], pb + n * 8 * TL::LDB + 2 * TL::PL);
        }
        uint32_t brh[2 * NT], brl[2 * NT], bih[2 * NT], bil[2 * NT];
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                brh[2 * n + i] = br[n][i];
                brl[2 * n + i] = br[n][2 + i];
                bih[2 * n + i] = bi[n][i];
                bil[2 * n + i] = bi[n][2 + i];
            }
        add_products<NT>(re, im, rh, rl, ih, il, brh, brl, bih, bil);
    }
    out += g * 17 + 8 * nt0 + 2 * t4;
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) out[8 * 17 * (i >> 1) + 8 * n + (i & 1)] = make_float2(f * re[n][i], -f * im[n][i]);
}

// Inverse of I + N (16 x 16 complex, [17] float2 rows, only the strictly lower part of N is read) by one warp, in place:
// the 4 x 4 diagonal blocks by substitution, then X21 = -X22 N21 X11 twice (4 -> 8 -> 16).  A rolled loop over block
// sizes 1 to 8 is a quarter of the code and took 3.5 k cycles instead of 1.7 k.
__device__ __forceinline__ void invert_unit_lower16(float2 *N, int lane)
{
    {
        const int blk = lane >> 3, c = (lane >> 1) & 3, part = lane & 1;      // a lane: half (Re / Im) of one column
        float2 *B = N + blk * 4 * 18;
        const float2 n10 = B[17], n20 = B[34], n21 = B[35], n30 = B[51], n31 = B[52], n32 = B[53];
        float x[4][2];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            float s = (t == c && part == 0) ? 1.f : 0.f;
#pragma unroll
            for (int i = 0; i < t; ++i) {
                const float2 n = t == 1 ? n10 : t == 2 ? (i ? n21 : n20) : (i == 0 ? n30 : i == 1 ? n31 : n32);
                s -= part ? n.x * x[i][1] + n.y * x[i][0] : n.x * x[i][0] - n.y * x[i][1];
            }
            const float o = __shfl_xor_sync(0xffffffffu, s, 1);
            x[t][0] = part ? o : s;
            x[t][1] = part ? s : o;
        }
        __syncwarp();
        if (part == 0) {
#pragma unroll
            for (int t = 0; t < 4; ++t) B[t * 17 + c] = make_float2(x[t][0], x[t][1]);
        } else if ((blk & 1) == 0) {                                          // the block right of it is zero
#pragma unroll
            for (int t = 0; t < 4; ++t) B[t * 17 + 4 + c] = make_float2(0.f, 0.f);
        }
        __syncwarp();
    }
    {
        const int r = (lane >> 2) & 3, c = lane & 3;
        float2 *B = N + (lane >> 4) * 8 * 18;
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            float2 acc = make_float2(0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 l = B[(4 + r) * 17 + 4 * pass + i], x = B[(4 * pass + i) * 17 + c];
                acc.x += l.x * x.x - l.y * x.y;
                acc.y += l.x * x.y + l.y * x.x;
            }
            __syncwarp();
            B[(4 + r) * 17 + c] = pass ? make_float2(-acc.x, -acc.y) : acc;
            __syncwarp();
        }
    }
    const int r = lane >> 2, c0 = 2 * (lane & 3);
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        float2 acc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        const float2 *L = N + (8 + r) * 17 + 8 * pass, *R = N + 8 * 17 * pass;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float2 l = L[i];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float2 x = R[i * 17 + c0 + e];
                acc[e].x += l.x * x.x - l.y * x.y;
                acc[e].y += l.x * x.y + l.y * x.x;
            }
        }
        __syncwarp();
#pragma unroll
        for (int e = 0; e < 2; ++e) N[(8 + r) * 17 + c0 + e] = pass ? make_float2(-acc[e].x, -acc[e].y) : acc[e];
        __syncwarp();
    }
}

// The lower triangle (diagonal included) of a [17] float2 matrix into the four planes of a small tile, by one warp
__device__ __forceinline__ void store_lower(unsigned char *tile, const float2 *A, float *inv_out, int lane)
{
    const int i0 = 2 * (lane & 7), r0 = lane >> 3;                            // a lane: two columns, every fourth row
    const float2 *p = A + r0 * 17 + i0;
    float m = 0.f;
#pragma unroll
    for (int r = 0; r < 16; r += 4) {
        const float2 x = p[r * 17], y = p[r * 17 + 1];
        if (i0 <= r0 + r) m = fmaxf(m, fmaxf(fabsf(x.x), fabsf(x.y)));
        if (i0 + 1 <= r0 + r) m = fmaxf(m, fmaxf(fabsf(y.x), fabsf(y.y)));
    }
    float inv;
    const float s = scale_for(warp_max(m), inv);
    tile += r0 * 48 + i0 * 2;
#pragma unroll 1
    for (int r = 0; r < 16; r += 4, tile += 4 * 48) {
        const float2 zero = make_float2(0.f, 0.f);
        const float2 x = i0 <= r0 + r ? p[r * 17] : zero, y = i0 + 1 <= r0 + r ? p[r * 17 + 1] : zero;
        put_planes(tile, 768, x.x * s, x.y * s, y.x * s, y.y * s);
    }
    if (lane == 0) *inv_out = inv;
}

// ---- a cluster's shared memory ---------------------------------------------------------------------
// Barriers in shared memory: FULL (a slot's tile is complete) in every CTA, EMPTY (all CTAs are through with it) in the CTA
// that makes the slot's tiles.  Every wait has a limit (never reached, unless a CTA is stuck).  The warp that gives up raises
// a flag in all CTAs of the cluster and nobody waits any more: tiles may be overwritten while they are read.  So all
// results of the pair are replaced by NaN at the end, what was computed before the wait included.
constexpr uint32_t kWaitTicks = 1u << 31;                        // of the SM's clock, about a second
#ifdef SFDA_WS_CHAOS
// Development builds only: with SFDA_WITHHOLD in the environment some arrivals at these barriers are withheld and the limit is
// short, so that waits run out.
constexpr bool kWithhold = true;
inline uint32_t wait_limit() { return getenv("SFDA_WITHHOLD") ? 1u << 18 : kWaitTicks; }
#else
constexpr bool kWithhold = false;
inline uint32_t wait_limit() { return kWaitTicks; }
#endif
struct Wait {
    uint32_t flag, limit;                                        // the CTA's flag (shared memory); SM-clock ticks
    __device__ __forceinline__ bool raised() const
    {
        uint32_t x;
        asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(x) : "r"(flag) : "memory");
        return x != 0;
    }
    __device__ __forceinline__ bool withheld() const { return kWithhold && limit != kWaitTicks; }
};
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count)); }
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// By whole warps, which leave together (what follows is for whole warps); false: given up, by this warp or another.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, const Wait &w)
{
    const uint32_t start = (uint32_t)clock(), limit = kWithhold ? w.limit : kWaitTicks;
    do {
        if (__all_sync(0xffffffffu, mbar_try(bar, parity))) return true;
    } while (!__any_sync(0xffffffffu, (uint32_t)clock() - start >= limit || w.raised()));
    return false;
}
__device__ __forceinline__ uint32_t in_cta(uint32_t addr, uint32_t rank)       // the same place in another CTA of the cluster
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// A warp of a cluster of CL waits; where the wait runs out every CTA learns of it.
template <int CL>
__device__ __forceinline__ bool cluster_wait(uint32_t bar, uint32_t parity, const Wait &w, int lane)
{
    if (mbar_wait(bar, parity, w)) {
        pause(bar);
        return true;
    }
    if (lane < CL) asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], 1;" ::"r"(in_cta(w.flag, lane)) : "memory");
    __syncwarp();
    return false;
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) { asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory"); }
__device__ __forceinline__ void warp_arrive(uint32_t bar, uint32_t rank, int lane)   // once for the warp, when all of it is here
{
    __syncwarp();
    if (lane == 0) asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(in_cta(bar, rank)) : "memory");
    __syncwarp();
    pause(bar + rank);
}
// `bytes` from this CTA's shared memory to the same place in another's, counted by the barrier there
__device__ __forceinline__ void copy_to_cta(uint32_t from, uint32_t bytes, uint32_t bar, uint32_t rank)
{
    const uint32_t to = in_cta(from, rank), there = in_cta(bar, rank);
    asm volatile("mbarrier.arrive.expect_tx.release.cluster.shared::cluster.b64 _, [%0], %1;" ::"r"(there), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(to), "r"(from), "r"(bytes), "r"(there) : "memory");
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() { asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// ---- kernels that run a chain and nothing else: PREP, SOLVE, CHAIN -----------------------------------
// A pair's CTAs (blocks of NB value columns) are clusters of CL (mostly one cluster): the tile of chunk c is made by CTA c % CL alone and copied
// to the others' shared memory, so that the preparation, which does not depend on the columns, is done once per pair.  It
// had been half of what a CTA of 32 columns issued (13.4 k of 27.6 k issue cycles per chunk; mma.sync holds its scheduler
// for 8.2 cycles, and 0.7 more for every other instruction issued meanwhile).  With 32 columns two warps share a block of
// 16, half of the keys each (KSP), and add up their parts of the products over the keys: every scheduler has one chain
// warp, with less work.  fp32 forward, B = 2, T = 2001, H = 16, d = 128: 457 -> 334 us, 326 now (at 334: one warp per block of 16 columns 431,
// eight PREP warps instead of four 371, the planes handed out with the rest of a tile 387).
template <int DK, int NB, int CL>
struct Chain {
    static constexpr int KSP = NB == 32 ? 2 : 1, KN = Tile<DK>::KS / KSP;
    static constexpr int prep_warps = NB == 32 ? 4 : 8, kPrep = 32 * prep_warps, kSolve = 128, warps = NB / 16 * KSP, kChain = 32 * warps;
    static constexpr int threads = kPrep + kSolve + kChain;
    static_assert(kSlots % CL == 0, "a slot's tiles are made by one CTA");
    using PM = PrepMap<DK, prep_warps>;
    static constexpr int own = kSlots / CL;                      // slots whose tiles this CTA makes
    static constexpr int kb = kSlots * Tile<DK>::bytes;          // Kb planes, one for each of them,
    static constexpr int gram = kb + own * Tile<DK>::BIG;        // the two Gram matrices likewise
    static constexpr int gram_bytes = 2 * 16 * 17 * 8;
    static constexpr int scan = gram + own * gram_bytes;
    static constexpr int slow = scan + (PM::scan_bytes + 127) / 128 * 128;   // its first word also passes the tensor-memory address on
    static constexpr int part = slow + (PM::slow_bytes + 127) / 128 * 128;   // KSP: [chunk parity][warp][6][lane] float4
    static constexpr int bars = part + (KSP - 1) * 2 * warps * 3072;
    static constexpr int sent = bars + 2 * kSlots * 8;           // per slot: tiles handed out; then the flag of a wait that ran out
    static constexpr int flag = sent + kSlots * 4, bytes = flag + 16;
    static_assert(bytes <= 232448, "shared memory");
    // 8 KT / KSP columns for every four warps
    static constexpr int need = (warps + 3) / 4 * Tile<DK>::KT * 8 / KSP, columns = need < 32 ? 32 : need;
};
constexpr int kBarPlanes = kBarFree, kBarPair = 2, kBarHalf = 4;  // planes ready: + slot; SOLVE: + parity; chain halves: + block

template <int DK, int NB, int CL>
__device__ __forceinline__ void chain_begin(unsigned char *smem, int tid)
{
    using L = Chain<DK, NB, CL>;
    if (tid < 32) tm_alloc(reinterpret_cast<uint32_t *>(smem + L::slow), L::columns);
    if (CL > 1 && tid == 32) {                                   // (without a cluster nothing uses them)
        const uint32_t bars = (uint32_t)__cvta_generic_to_shared(smem + L::bars);
        uint32_t *sent = reinterpret_cast<uint32_t *>(smem + L::sent);
        for (int i = 0; i < kSlots; ++i) {
            mbar_init(bars + 8 * i, 2);
            mbar_init(bars + 8 * (kSlots + i), CL * L::warps);
            sent[i] = 0;
        }
        sent[kSlots] = 0;                                        // the flag
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if constexpr (CL > 1) cluster_sync();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
template <int DK, int NB, int CL>
__device__ __forceinline__ Wait chain_limit(const unsigned char *smem, uint32_t limit)
{
    return {(uint32_t)__cvta_generic_to_shared(smem + Chain<DK, NB, CL>::flag), limit};
}
// Nobody leaves before the others are through.  Every CTA's copies have arrived when its chain is; where a wait has run out
// (the answer, the same in all CTAs) that is waited for here: the last tile sent into a slot is the last phase of its FULL.
template <int DK, int NB, int CL>
__device__ __forceinline__ bool chain_end(unsigned char *smem, uint32_t tmem, const Wait &wait, int tid)
{
    using L = Chain<DK, NB, CL>;
    bool gave_up = false;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if constexpr (CL > 1) {
        cluster_sync();
        gave_up = wait.raised();
        if (gave_up) {
            const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem);
            if (tid < kSlots) {
                uint32_t sent;
                asm volatile("ld.relaxed.cluster.shared::cluster.u32 %0, [%1];" : "=r"(sent) : "r"(in_cta(base + L::sent + 4 * tid, tid % CL)) : "memory");
#pragma unroll 1
                for (uint32_t i = 0; sent && i < 1u << 20 && !mbar_try(base + L::bars + 8 * tid, (sent - 1) & 1);) ++i;
            }
            __syncwarp();
            cluster_sync();
        }
    }
    if (tid < 32) tm_free(tmem, L::columns);
    return gave_up;
}

// PREP of the chunks of rank `rank`, in the order of the chain (back: last to first)
template <int DK, int NB, int CL, typename T>
__device__ __forceinline__ void chain_prep(unsigned char *smem, const T *q, const T *k, const float *alpha, const float *theta, const float *beta,
                                           size_t row0, int H, int T_, int nch, bool back, bool needq, int rank, const Wait &wait, int tid)
{
    using L = Chain<DK, NB, CL>;
    constexpr int PW = L::prep_warps;
    const uint32_t empty = (uint32_t)__cvta_generic_to_shared(smem + L::bars) + 8 * kSlots;
    PrepRaw<L::PM::TPT, T> in;
    prep_fetch<DK, PW, T>(in, q, k, alpha, theta, beta, row0, H, max(back ? nch - 1 - rank : rank, 0) * kC, T_, needq, tid);
    bool ok = true;
#pragma unroll 1
    for (int c = rank; c < nch; c += CL) {
        const int slot = c % kSlots, at = back ? nch - 1 - c : c, nx = back ? max(at - CL, 0) : at + CL;
        if (CL == 1 && c >= kSlots) bar_sync(kBarDone + slot, L::kPrep + L::kChain);
        if (CL > 1 && c >= kSlots) ok = ok && cluster_wait<CL>(empty + 8 * slot, (c / kSlots - 1) & 1, wait, tid & 31) && !wait.raised();
        PrepRaw<L::PM::TPT, T> next;
        prep_fetch<DK, PW, T>(next, q, k, alpha, theta, beta, row0, H, nx * kC, T_, needq, tid);
        unsigned char *tile = smem + slot * Tile<DK>::bytes, *kb = smem + L::kb + slot / CL * Tile<DK>::BIG;
        float2 *gk = reinterpret_cast<float2 *>(smem + L::gram + slot / CL * L::gram_bytes);
        if (!prep_chunk<DK, PW, kBarAux, T>(in, q, k, alpha, theta, beta, row0, H, at * kC, T_, nullptr, tile, kb, smem + L::scan, needq, tid))
            slow_gram<DK, PW, kBarAux, T>(q, k, alpha, theta, beta, row0, H, at * kC, T_, smem + L::slow, smem + L::scan, gk, gk + 16 * 17, needq, tid);
        if (CL > 1 && ok && tid == 0) reinterpret_cast<uint32_t *>(smem + L::sent)[slot] = c / kSlots + 1;   // only into a slot that all are through with
        if constexpr (CL > 1) fence_async_smem();
        bar_arrive(kBarPlanes + slot, L::kPrep + 64);
        in = next;
    }
}

// SOLVE: warps 0, 1 the system's inverse of this CTA's even / odd chunks, warps 2, 3 the outputs' Gram matrix of them
// (needq); they also hand the tile out, its large planes first.  (With a single slot to make tiles in, warps 0 and 2 do it
// alone: two chunks would meet at the slot's barrier.)
template <int DK, int NB, int CL>
__device__ __forceinline__ void chain_solve(unsigned char *smem, int nch, bool needq, int rank, int tid)
{
    using L = Chain<DK, NB, CL>;
    using TL = Tile<DK>;
    constexpr int pairs = L::own > 1 ? 2 : 1;
    const int lane = tid & 31, w = tid >> 5, out = w >> 1;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem), full = base + L::bars;
    if ((w & 1) >= pairs) return;
#pragma unroll 1
    for (int c = rank + CL * (w & 1); c < nch; c += pairs * CL) {
        const int slot = c % kSlots;
        unsigned char *tile = smem + slot * TL::bytes;
        float *inv = reinterpret_cast<float *>(tile + TL::oS);
        float2 *gm = reinterpret_cast<float2 *>(smem + L::gram + slot / CL * L::gram_bytes) + out * 16 * 17;
        const uint32_t bar = full + 8 * slot, from = base + slot * TL::bytes;
        bar_sync(kBarPlanes + slot, L::kPrep + 64);
        const bool send = CL > 1 && reinterpret_cast<const uint32_t *>(smem + L::sent)[slot] == c / kSlots + 1;
        const bool other = send && lane < CL && lane != rank;    // a lane per CTA to hand out to
        if (out && other) copy_to_cta(from, TL::oM, bar, lane);
        __syncwarp();
        if (needq || !out) {
            if (reinterpret_cast<const int *>(inv)[6])
                gram_tiles<DK, 2>(base + slot * TL::bytes + (out ? TL::oQ : TL::oW), base + L::kb + slot / CL * TL::BIG, inv[out ? 2 : 0] * inv[5], gm, 0, lane);
            __syncwarp();
            if (!out) invert_unit_lower16(gm, lane);
            store_lower(tile + (out ? TL::oA : TL::oM), gm, inv + 3 + out, lane);
        }
        if constexpr (CL == 1) {
            bar_arrive(kBarFull + slot, 64 + L::kChain);
            continue;
        }
        fence_async_smem();
        if (out) {
            bar_arrive(kBarPair + (w & 1), 64);
        } else {
            bar_sync(kBarPair + (w & 1), 64);
            if (other) copy_to_cta(from + TL::oM, TL::bytes - TL::oM, bar, lane);
        }
        if (send) warp_arrive(bar, rank, lane);
    }
}

// CHAIN: until chunk c's tile is there; and when the warp is through with it.  (A CTA by itself has hardware barriers for FULL and
// EMPTY: a warp that waits at one in shared memory resumes a few hundred cycles late, 36.3 us instead of 34.8 for the forward of
// B = 20, T = 104, H = 7, d_k = 64, d_v = 128.)
template <int DK, int NB, int CL>
__device__ __forceinline__ void chain_wait(uint32_t full, int c, const Wait &wait, int lane)
{
    const int slot = c % kSlots;
    if constexpr (CL > 1) cluster_wait<CL>(full + 8 * slot, (c / kSlots) & 1, wait, lane);
    else bar_sync(kBarFull + slot, 64 + Chain<DK, NB, CL>::kChain);
}
template <int DK, int NB, int CL>
__device__ __forceinline__ void chain_release(uint32_t full, int c, int nch, const Wait &wait, int lane)
{
    const int slot = c % kSlots;
    if (c + kSlots >= nch) return;
    if (CL > 1 && wait.withheld() && c % CL == 0) return;        // (the others learn of it by the flag)
    if constexpr (CL > 1) warp_arrive(full + 8 * (kSlots + slot), c % CL, lane);
    else bar_arrive(kBarDone + slot, Chain<DK, NB, CL>::kPrep + Chain<DK, NB, CL>::kChain);
}

// A chain warp's place: its half of the keys (KSP = 2), and where the halves exchange their parts
struct Half {
    int half, bar;
    float4 *mine;             // this chunk's (offset by the lane); the other half's lies `other` float4 further
    int other;
};
// x += the other half's x; N a multiple of 4.  `out` goes to the other half, which sends its own in return.
template <int N>
__device__ __forceinline__ void add_other(float (&x)[N], const float (&out)[N], const Half &h)
{
#pragma unroll
    for (int i = 0; i < N / 4; ++i) h.mine[32 * i] = make_float4(out[4 * i], out[4 * i + 1], out[4 * i + 2], out[4 * i + 3]);
    bar_sync(h.bar, 64);
#pragma unroll
    for (int i = 0; i < N / 4; ++i) {
        const float4 v = h.mine[h.other + 32 * i];
        x[4 * i] += v.x;
        x[4 * i + 1] += v.y;
        x[4 * i + 2] += v.z;
        x[4 * i + 3] += v.w;
    }
}
template <int DK, int NB, int CL>
__device__ __forceinline__ Half chain_half(unsigned char *smem, int w, int c, int lane)
{
    using L = Chain<DK, NB, CL>;
    const int half = w & 1, block = w >> 1;
    float4 *p = reinterpret_cast<float4 *>(smem + L::part) + ((c & 1) * L::warps + w) * 192 + lane;
    return {half, kBarHalf + block, p, half ? -192 : 192};
}

// Value columns per CTA for `walks` sequences that a chain kernel takes at once, and CTAs per cluster: all columns, halved (down
// to 32) while the CTAs fit the SMs.  Clusters of two fit all SMs (74), of clusters of four 33 at a time (asked of the driver; 32
// here, as other parts may have lost other SMs).  So 33 to 37 sequences of 128 columns have two clusters of two each, and every
// chunk is prepared twice: 37 sequences of 520 tokens 126 us at d_k = 128, 74 us at 64, with blocks of 64 columns 138 and 95,
// with CTAs that prepare everything for themselves 125 and 76.  (Only where every decay is too strong to divide by are 64 columns
// better, 166 us instead of 207; without clusters 303.)  On a device with other SMs the blocks are merely not the best ones.
struct Blocks {
    int columns, cluster;
};
inline Blocks chain_blocks(long long walks, int d_v)
{
    Blocks b = {d_v, 1};
    while (b.columns > 32 && walks * (2 * d_v / b.columns) <= 148) b.columns /= 2;
    b.cluster = d_v / b.columns;
    if (b.cluster == 4 && walks > 32) b.cluster = 2;
    return b;
}
template <typename Args>
cudaError_t launch_clusters(void (*kern)(Args), const Args &a, dim3 grid, int cluster, int threads, int bytes, cudaStream_t stream)
{
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = cluster;                          // neighbouring blocks of columns of a pair
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 1 : 0;
    const cudaError_t launched = cudaLaunchKernelEx(&cfg, kern, a);
    const cudaError_t last = cudaGetLastError();                 // (a refused launch is this call's error, not a later one's)
    return launched != cudaSuccess ? launched : last;
}

}  // namespace c16
}  // namespace sfda
