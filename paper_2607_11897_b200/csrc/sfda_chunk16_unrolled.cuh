// The backward pass's chunk engine: 16-token chunks at fp32 precision on the tensor cores (see sfda_chunk16.cuh for the
// arithmetic; this one keeps the state in registers and everything unrolled): every fp32 operand split
// into an fp16 head and an fp16 tail (22 significant bits; the three significant of the four partial products are
// added in fp32).  Used by the fp32 forward (sfda_forward_f32.cu) and the backward pass (sfda_backward.cu).
//
// Why split fp16: measured per SM and clock, mma.sync does 970 multiply-adds in fp16 and 484 in TF32, so three fp16
// products (323 effective) are twice as fast as 3 x TF32 (161) and 2.5 times the fp32 pipe (128), at the same 22 bits.
// fp16's exponent range is covered by scaling every operand tile by a power of two that puts its largest magnitude
// at 2^14: entries down to 2^-16 of the largest keep all 22 bits, smaller ones an absolute error of 2^-39 of it.
// Where an operand's range is not bounded (keys divided by the cumulative decay) 3 x TF32 is used instead.
//
// Why chunks of 16: the state-sized products cost the same per token at any chunk size, the products inside a chunk
// grow with it, and inside 16 tokens the decays divide safely unless a coordinate loses more than 2^-80, which is
// checked per chunk (a slow exact path takes over then).
//
// Roles in a CTA: eight AUX warps prepare the operand tiles of a chunk (PREP) into a ring of shared-memory slots;
// CHAIN warps own 16 value columns of the state each, for all keys, in the accumulator layout of m16n8 with the value
// channel as the row.  That layout is also the A-operand layout of the next product, so a chain warp goes
// R = V - W^* S -> U = M R -> S = gamma_C S + Y U with no exchange with other warps at all.
#pragma once
#include "sfda_common.cuh"

namespace sfda {
namespace c16 {

constexpr int kC = 16;                       // tokens per chunk
constexpr int kAuxWarps = 8, kAux = 32 * kAuxWarps;
constexpr int kSlots = 4;                    // operand tiles in flight
constexpr int kBarAux = 1, kBarFull = 2, kBarDone = 6, kBarFree = 10;   // hardware barriers; the last three: + slot

__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// ---- tensor-core primitives ---------------------------------------------------------------------
__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_tf32(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// d += (ah + al)(bh + bl) without the product of the tails, smallest terms first
__device__ __forceinline__ void mma3(float (&d)[4], const uint32_t (&ah)[4], const uint32_t (&al)[4], uint32_t bh0,
                                     uint32_t bh1, uint32_t bl0, uint32_t bl1)
{
    mma_f16(d, al, bh0, bh1);
    mma_f16(d, ah, bl0, bl1);
    mma_f16(d, ah, bh0, bh1);
}
__device__ __forceinline__ void mma3_tf32(float (&d)[4], const uint32_t (&ah)[4], const uint32_t (&al)[4],
                                          const uint32_t (&bh)[2], const uint32_t (&bl)[2])
{
    mma_tf32(d, al, bh[0], bh[1]);
    mma_tf32(d, ah, bl[0], bl[1]);
    mma_tf32(d, ah, bh[0], bh[1]);
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
// head and tail of two values (already scaled)
__device__ __forceinline__ void split_f16(float x, float y, uint32_t &h, uint32_t &l)
{
    h = pack_f16(x, y);
    const float2 f = unpack_f16(h);
    l = pack_f16(x - f.x, y - f.y);
}
// TF32 head = the value cut to ten mantissa bits; the tail is passed as it is (the tensor core reads its leading bits)
__device__ __forceinline__ void split_tf32(float x, uint32_t &h, uint32_t &l)
{
    h = __float_as_uint(x) & 0xffffe000u;
    l = __float_as_uint(x - __uint_as_float(h));
}
// Power of two that brings a magnitude with these bits into [2^14, 2^15), and its inverse.
__device__ __forceinline__ float scale_for(uint32_t max_bits, float &inv)
{
    const int e = max((int)(max_bits >> 23) - 127, -100);
    inv = __uint_as_float((uint32_t)(113 + e) << 23);
    return __uint_as_float((uint32_t)(141 - e) << 23);
}
__device__ __forceinline__ uint32_t abs_bits(float x) { return __float_as_uint(x) & 0x7fffffffu; }
template <int N>
__device__ __forceinline__ uint32_t max_bits4(const float (&x)[N][4])
{
    uint32_t m = 0;
#pragma unroll
    for (int n = 0; n < N; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) m = max(m, abs_bits(x[n][i]));
    return m;
}
// A-operand registers (16 x 16) of two neighbouring accumulator tiles, scaled and split
__device__ __forceinline__ void split_tiles(const float (&x)[4], const float (&y)[4], float s, uint32_t (&h)[4], uint32_t (&l)[4])
{
    split_f16(x[0] * s, x[1] * s, h[0], l[0]);
    split_f16(x[2] * s, x[3] * s, h[1], l[1]);
    split_f16(y[0] * s, y[1] * s, h[2], l[2]);
    split_f16(y[2] * s, y[3] * s, h[3], l[3]);
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
    static constexpr int bytes = (oS + 32 + 127) / 128 * 128;     // oG: gamma_C float2 [M]; oS: inverse scales W Y Q M A
};

// ---- CHAIN --------------------------------------------------------------------------------------
// acc[x] = products conj(X_x)^T S of NX tiles with the state, value channels in rows, tokens in columns, for each of
// two token tiles: [0] = Xr Sr + Xi Si, [1] = Xr Si, [2] = Xi Sr (Im = [1] - [2]); scaled by s and the tiles' scales.
// With kPub the split state is also left in `pub` as the B operand (value channel, key) of products over the columns.
template <int DK, int NX, bool kPub>
__device__ __forceinline__ void product_over_keys(float (&acc)[NX][3][2][4], const float (&sr)[DK / 16][4],
                                                  const float (&si)[DK / 16][4], float s, const uint32_t (&tile)[NX],
                                                  int lane, uint4 *pub)
{
    using TL = Tile<DK>;
#pragma unroll
    for (int x = 0; x < NX; ++x)
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[x][c][n][i] = 0.f;
    const uint32_t at = (uint32_t)(((lane & 7) + ((lane >> 4) << 3)) * TL::LDB + ((lane >> 3) & 1) * 16);
#pragma unroll
    for (int kk = 0; kk < TL::KS; ++kk) {
        uint32_t rh[4], rl[4], ih[4], il[4];
        split_tiles(sr[2 * kk], sr[2 * kk + 1], s, rh, rl);
        split_tiles(si[2 * kk], si[2 * kk + 1], s, ih, il);
        if constexpr (kPub) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                pub[((2 * kk + e) * 2 + 0) * 32 + lane] = make_uint4(transpose8x8(rh[2 * e]), transpose8x8(rh[2 * e + 1]),
                                                                   transpose8x8(rl[2 * e]), transpose8x8(rl[2 * e + 1]));
                pub[((2 * kk + e) * 2 + 1) * 32 + lane] = make_uint4(transpose8x8(ih[2 * e]), transpose8x8(ih[2 * e + 1]),
                                                                   transpose8x8(il[2 * e]), transpose8x8(il[2 * e + 1]));
            }
        }
#pragma unroll
        for (int x = 0; x < NX; ++x) {
            uint32_t brh[4], brl[4], bih[4], bil[4];
            const uint32_t p = tile[x] + at + kk * 32;
            ldsm(brh, p);
            ldsm(brl, p + TL::PL);
            ldsm(bih, p + 2 * TL::PL);
            ldsm(bil, p + 3 * TL::PL);
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                mma3(acc[x][0][n], rh, rl, brh[2 * n], brh[2 * n + 1], brl[2 * n], brl[2 * n + 1]);
                mma3(acc[x][1][n], ih, il, brh[2 * n], brh[2 * n + 1], brl[2 * n], brl[2 * n + 1]);
                mma3(acc[x][2][n], rh, rl, bih[2 * n], bih[2 * n + 1], bil[2 * n], bil[2 * n + 1]);
                mma3(acc[x][0][n], ih, il, bih[2 * n], bih[2 * n + 1], bil[2 * n], bil[2 * n + 1]);
            }
        }
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

// out = a b (kConj: a conj(b)) over 16 tokens, both complex, unscaled by f
template <bool kConj>
__device__ __forceinline__ void product_small(float (&re)[2][4], float (&im)[2][4], const TokFrag &a, const TokFrag &b, float f)
{
#pragma unroll
    for (int n = 0; n < 2; ++n) {
        float rr[4] = {0.f, 0.f, 0.f, 0.f}, ii[4] = {0.f, 0.f, 0.f, 0.f}, ir[4] = {0.f, 0.f, 0.f, 0.f}, ri[4] = {0.f, 0.f, 0.f, 0.f};
        mma3(rr, a.rh, a.rl, b.rh[2 * n], b.rh[2 * n + 1], b.rl[2 * n], b.rl[2 * n + 1]);
        mma3(ii, a.ih, a.il, b.ih[2 * n], b.ih[2 * n + 1], b.il[2 * n], b.il[2 * n + 1]);
        mma3(ir, a.ih, a.il, b.rh[2 * n], b.rh[2 * n + 1], b.rl[2 * n], b.rl[2 * n + 1]);
        mma3(ri, a.rh, a.rl, b.ih[2 * n], b.ih[2 * n + 1], b.il[2 * n], b.il[2 * n + 1]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            re[n][i] = f * (kConj ? rr[i] + ii[i] : rr[i] - ii[i]);
            im[n][i] = f * (kConj ? ir[i] - ri[i] : ir[i] + ri[i]);
        }
    }
}

// scale and split a [value x 16 tokens] matrix; returns the inverse scale
__device__ __forceinline__ float make_frag(TokFrag &f, const float (&re)[2][4], const float (&im)[2][4])
{
    float inv;
    const float s = scale_for(__reduce_max_sync(0xffffffffu, max(max_bits4(re), max_bits4(im))), inv);
    split_tiles(re[0], re[1], s, f.rh, f.rl);
    split_tiles(im[0], im[1], s, f.ih, f.il);
    return inv;
}

// S <- gamma_C S + sum_t a[., t] X[t][.]   (X: W-like tile read with tokens as k), unscaled by f
template <int DK>
__device__ __forceinline__ void state_update(float (&sr)[DK / 16][4], float (&si)[DK / 16][4], const TokFrag &a, float f,
                                             uint32_t tile, const float4 *__restrict__ gamma, int lane)
{
    using TL = Tile<DK>;
    const uint32_t at = tile + (uint32_t)(((lane & 7) + (((lane >> 3) & 1) << 3)) * TL::LDB + (lane >> 4) * 16);
#pragma unroll
    for (int np = 0; np < TL::KT; np += 2) {
        uint32_t brh[4], brl[4], bih[4], bil[4];
        ldsm_t(brh, at + np * 16);
        ldsm_t(brl, at + np * 16 + TL::PL);
        ldsm_t(bih, at + np * 16 + 2 * TL::PL);
        ldsm_t(bil, at + np * 16 + 3 * TL::PL);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            float rr[4] = {0.f, 0.f, 0.f, 0.f}, ii[4] = {0.f, 0.f, 0.f, 0.f}, im[4] = {0.f, 0.f, 0.f, 0.f};
            mma3(rr, a.rh, a.rl, brh[2 * e], brh[2 * e + 1], brl[2 * e], brl[2 * e + 1]);
            mma3(im, a.ih, a.il, brh[2 * e], brh[2 * e + 1], brl[2 * e], brl[2 * e + 1]);
            mma3(ii, a.ih, a.il, bih[2 * e], bih[2 * e + 1], bil[2 * e], bil[2 * e + 1]);
            mma3(im, a.rh, a.rl, bih[2 * e], bih[2 * e + 1], bil[2 * e], bil[2 * e + 1]);
            const int n = np + e;
            const float4 g = gamma[4 * n + (lane & 3)];           // gamma_C of keys 8 n + 2 (lane & 3), + 1
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float gr = (i & 1) ? g.z : g.x, gi = (i & 1) ? g.w : g.y;
                const float x = sr[n][i], y = si[n][i];
                sr[n][i] = fmaf(f, rr[i] - ii[i], gr * x - gi * y);
                si[n][i] = fmaf(f, im[i], gr * y + gi * x);
            }
        }
    }
}

// ---- PREP ---------------------------------------------------------------------------------------
// Thread of AUX warp w: key 8 w + (lane >> 2), tokens 4 (lane & 3) .. + 3 of a chunk.
struct PrepIn {
    float kr[4], ki[4], qr[4], qi[4], al[4], th[4], be[4];
};
struct PrepVals {                             // what the gradients of a chunk need again
    float kr[4], ki[4], qr[4], qi[4];         // rotated key and query (phases inside the chunk)
    float a[4], sfx[4], cs[4], sn[4];         // prod alpha up to the token / after it; e^{i phi}
};

__device__ __forceinline__ float2 ld_pair(const float *p, size_t i) { return *reinterpret_cast<const float2 *>(p + i); }
__device__ __forceinline__ float2 ld_pair(const __nv_bfloat16 *p, size_t i)
{
    const uint32_t u = *reinterpret_cast<const uint32_t *>(p + i);
    return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
}

// q may be NULL (keys only)
template <int DK, typename T>
__device__ __forceinline__ void prep_load(PrepIn &in, const T *__restrict__ q, const T *__restrict__ k,
                                          const float *__restrict__ alpha, const float *__restrict__ theta,
                                          const float *__restrict__ beta, size_t row0, int H, int t0, int T_, int key, int t4)
{
    constexpr int M = DK / 2;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const int t = t0 + 4 * t4 + x;
        in.kr[x] = in.ki[x] = in.qr[x] = in.qi[x] = in.th[x] = in.be[x] = 0.f;
        in.al[x] = 1.f;
        if (t < T_ && key < M) {
            const size_t row = row0 + (size_t)t * H;
            const float2 kk = ld_pair(k, row * DK + 2 * key);
            in.kr[x] = kk.x;
            in.ki[x] = kk.y;
            if (q) {
                const float2 qq = ld_pair(q, row * DK + 2 * key);
                in.qr[x] = qq.x;
                in.qi[x] = qq.y;
            }
            in.al[x] = alpha[row * M + key];
            in.th[x] = theta[row * M + key];
            in.be[x] = beta[row];
        }
    }
}

// Scratch of PREP: fp32 copies of W, K = k' / a, Q for the Gram products, the two Gram matrices, the warps' maxima.
template <int DK>
struct PrepSmem {
    static constexpr int M = DK / 2, LDF = M + 4;                 // float2 per token row
    static constexpr int gram = 16 * 17;                          // float2
    static constexpr int stage_bytes = 3 * 16 * LDF * 8;
    static constexpr int small_bytes = 2 * (2 * gram * 8 + 4 * kAuxWarps * 4 + 16 * 4);   // two chunks deep
};

// Inverse of I + N (16 x 16 complex, N strictly lower, [17] float2 rows) by one warp: the two 8 x 8 diagonal blocks by
// substitution (a lane owns half -- Re or Im -- of one column), then X21 = -X22 N21 X11.  The result replaces N.
__device__ __forceinline__ void invert_unit_lower16(float2 *N, int lane)
{
    const int blk = (lane >> 3) & 1, c = lane & 7, part = lane >> 4;
    float2 *B = N + blk * 8 * 17 + blk * 8;
    float xr[8], xi[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        float s0 = 0.f, s1 = 0.f;
#pragma unroll
        for (int i = 0; i < t; ++i) {
            const float2 n = B[t * 17 + i];
            // Re: nr xr - ni xi; Im: nr xi + ni xr
            s0 = fmaf(n.x, part ? xi[i] : xr[i], s0);
            s1 = fmaf(part ? n.y : -n.y, part ? xr[i] : xi[i], s1);
        }
        const float own = ((t == c && part == 0) ? 1.f : 0.f) - (s0 + s1);
        const float other = __shfl_xor_sync(0xffffffffu, own, 16);
        xr[t] = part ? other : own;
        xi[t] = part ? own : other;
    }
    __syncwarp();
    if (part == 0) {
#pragma unroll
        for (int t = 0; t < 8; ++t) B[t * 17 + c] = make_float2(xr[t], xi[t]);
    }
    __syncwarp();
    // T = N21 X11, then X21 = -X22 T: a lane owns row lane >> 2, columns 2 (lane & 3), + 1
    const int r = lane >> 2, c0 = 2 * (lane & 3);
    float2 acc[2];
#pragma unroll
    for (int pass = 0; pass < 2; ++pass) {
        acc[0] = acc[1] = make_float2(0.f, 0.f);
        const float2 *L = pass == 0 ? N + (8 + r) * 17 : N + (8 + r) * 17 + 8;
        const float2 *R = pass == 0 ? N : N + 8 * 17;
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
        for (int e = 0; e < 2; ++e)
            N[(8 + r) * 17 + c0 + e] = pass == 0 ? acc[e] : make_float2(-acc[e].x, -acc[e].y);
        __syncwarp();
    }
}

// Splits a [16][16] matrix held by one warp ([17] float2 rows) into the four planes of a small tile.  Element (t, i)
// is kept for i < t (strict == true) or i <= t, multiplied by w[i] when w is given.
__device__ __forceinline__ void store_small(unsigned char *tile, const float2 *A, const float *w, bool mask, float *inv_out, int lane)
{
    // lane: column pair 2 (lane & 7), rows 4 (lane >> 3) .. + 3
    const int i0 = 2 * (lane & 7), r0 = 4 * (lane >> 3);
    float2 v[4][2];
    uint32_t m = 0;
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            float2 a = A[(r0 + x) * 17 + i0 + e];
            if (mask) {
                const float f = w[i0 + e];
                const bool keep = i0 + e <= r0 + x;
                a = keep ? make_float2(a.x * f, a.y * f) : make_float2(0.f, 0.f);
            }
            v[x][e] = a;
            m = max(m, max(abs_bits(a.x), abs_bits(a.y)));
        }
    float inv;
    const float s = scale_for(__reduce_max_sync(0xffffffffu, m), inv);
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        uint32_t h, l;
        unsigned char *p = tile + (r0 + x) * 48 + i0 * 2;
        split_f16(v[x][0].x * s, v[x][1].x * s, h, l);
        *reinterpret_cast<uint32_t *>(p) = h;
        *reinterpret_cast<uint32_t *>(p + 768) = l;
        split_f16(v[x][0].y * s, v[x][1].y * s, h, l);
        *reinterpret_cast<uint32_t *>(p + 2 * 768) = h;
        *reinterpret_cast<uint32_t *>(p + 3 * 768) = l;
    }
    if (lane == 0) *inv_out = inv;
}

// One value pair (keys 2 p, 2 p + 1 of a token) would need an exchange between lanes; single 16-bit stores instead.
__device__ __forceinline__ void store_planes(unsigned char *p, int pl, float re, float im)
{
    uint32_t h, l;
    split_f16(re, im, h, l);
    *reinterpret_cast<uint16_t *>(p) = (uint16_t)h;
    *reinterpret_cast<uint16_t *>(p + pl) = (uint16_t)l;
    *reinterpret_cast<uint16_t *>(p + 2 * pl) = (uint16_t)(h >> 16);
    *reinterpret_cast<uint16_t *>(p + 3 * pl) = (uint16_t)(l >> 16);
}

// Builds the operand tile of one chunk.  All AUX threads call it; the caller announces the slot afterwards.  `stage`
// and `small` are PrepSmem; par alternates from chunk to chunk.  kNeedQ == false: W, Y, M only.
// Returns whether the chunk took the fast path (no coordinate decays below 2^-80 inside it).
template <int DK, bool kNeedQ>
__device__ __forceinline__ bool prep_chunk(const PrepIn &in, PrepVals &pv, unsigned char *slot, float2 *stage,
                                           unsigned char *small, int par, int tid)
{
    using TL = Tile<DK>;
    using PS = PrepSmem<DK>;
    constexpr int M = TL::M;
    const int lane = tid & 31, warp = tid >> 5, g = lane >> 2, t4 = lane & 3, key = 8 * warp + g;
    const bool own = key < M;
    unsigned char *sm = small + par * (PS::small_bytes / 2);
    float2 *gk = reinterpret_cast<float2 *>(sm), *gq = gk + PS::gram;
    float *red = reinterpret_cast<float *>(gq + PS::gram), *bsm = red + 4 * kAuxWarps;
    float2 *sW = stage, *sK = stage + 16 * PS::LDF, *sQ = stage + 32 * PS::LDF;

    // products of alpha and sums of the phase: inside the thread's four tokens, then over the key's four lanes
    float p[4], sf[4];
    uint32_t u[4];
    p[0] = in.al[0];
    u[0] = phase_to_turns(in.th[0]);
#pragma unroll
    for (int x = 1; x < 4; ++x) {
        p[x] = p[x - 1] * in.al[x];
        u[x] = u[x - 1] + phase_to_turns(in.th[x]);
    }
    sf[3] = 1.f;
#pragma unroll
    for (int x = 2; x >= 0; --x) sf[x] = sf[x + 1] * in.al[x + 1];
    float inc = p[3], dec = p[3];
    uint32_t ut = u[3];
#pragma unroll
    for (int d = 1; d < 4; d <<= 1) {
        const float up = __shfl_up_sync(0xffffffffu, inc, d, 4), dn = __shfl_down_sync(0xffffffffu, dec, d, 4);
        const uint32_t uu = __shfl_up_sync(0xffffffffu, ut, d, 4);
        if (t4 >= d) {
            inc *= up;
            ut += uu;
        }
        if (t4 + d < 4) dec *= dn;
    }
    float pre = __shfl_up_sync(0xffffffffu, inc, 1, 4), suf = __shfl_down_sync(0xffffffffu, dec, 1, 4);
    uint32_t ub = __shfl_up_sync(0xffffffffu, ut, 1, 4);
    if (t4 == 0) {
        pre = 1.f;
        ub = 0u;
    }
    if (t4 == 3) suf = 1.f;
    const float aC = __shfl_sync(0xffffffffu, inc, 3, 4);

    float Wr[4], Wi[4], Qr[4], Qi[4];
    uint32_t mk = 0, my = 0, mq = 0;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        pv.a[x] = pre * p[x];
        pv.sfx[x] = sf[x] * suf;
        turns_to_cos_sin(ub + u[x], &pv.cs[x], &pv.sn[x]);
        pv.kr[x] = in.kr[x] * pv.cs[x] + in.ki[x] * pv.sn[x];
        pv.ki[x] = in.ki[x] * pv.cs[x] - in.kr[x] * pv.sn[x];
        Wr[x] = pv.a[x] * pv.kr[x];
        Wi[x] = pv.a[x] * pv.ki[x];
        mk = max(mk, max(abs_bits(Wr[x]), abs_bits(Wi[x])));
        if constexpr (kNeedQ) {
            pv.qr[x] = in.qr[x] * pv.cs[x] + in.qi[x] * pv.sn[x];
            pv.qi[x] = in.qi[x] * pv.cs[x] - in.qr[x] * pv.sn[x];
            Qr[x] = pv.a[x] * pv.qr[x];
            Qi[x] = pv.a[x] * pv.qi[x];
            mq = max(mq, max(abs_bits(Qr[x]), abs_bits(Qi[x])));
        }
    }
    const float gcs = __shfl_sync(0xffffffffu, pv.cs[3], 3, 4), gsn = __shfl_sync(0xffffffffu, pv.sn[3], 3, 4);
    float Yr[4], Yi[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const float f = pv.sfx[x] * in.be[x];
        Yr[x] = f * (gcs * pv.kr[x] - gsn * pv.ki[x]);
        Yi[x] = f * (gcs * pv.ki[x] + gsn * pv.kr[x]);
        my = max(my, max(abs_bits(Yr[x]), abs_bits(Yi[x])));
    }
    if (own) {
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int t = 4 * t4 + x;
            const float ia = __frcp_rn(pv.a[x]);
            sW[t * PS::LDF + key] = make_float2(Wr[x], Wi[x]);
            sK[t * PS::LDF + key] = make_float2(pv.kr[x] * ia, pv.ki[x] * ia);
            if constexpr (kNeedQ) sQ[t * PS::LDF + key] = make_float2(Qr[x], Qi[x]);
        }
        if (t4 == 3) reinterpret_cast<float2 *>(slot + TL::oG)[key] = make_float2(aC * gcs, aC * gsn);
    }
    if (warp == 0 && g == 0) {
#pragma unroll
        for (int x = 0; x < 4; ++x) bsm[4 * t4 + x] = in.be[x];
    }
    mk = __reduce_max_sync(0xffffffffu, mk);
    my = __reduce_max_sync(0xffffffffu, my);
    mq = __reduce_max_sync(0xffffffffu, mq);
    const uint32_t lo = __reduce_min_sync(0xffffffffu, own ? __float_as_uint(aC) : 0x3f800000u);
    if (lane == 0) {
        red[warp] = __uint_as_float(mk);
        red[8 + warp] = __uint_as_float(my);
        red[16 + warp] = __uint_as_float(mq);
        red[24 + warp] = __uint_as_float(lo);
    }
    bar_sync(kBarAux, kAux);
    mk = my = mq = 0;
    float amin = 1.f;
#pragma unroll
    for (int w = 0; w < kAuxWarps; ++w) {
        mk = max(mk, __float_as_uint(red[w]));
        my = max(my, __float_as_uint(red[8 + w]));
        mq = max(mq, __float_as_uint(red[16 + w]));
        amin = fminf(amin, red[24 + w]);
    }
    const bool fast = amin >= 0x1p-80f;
    float *inv = reinterpret_cast<float *>(slot + TL::oS);
    float ik, iy, iq;
    const float sk = scale_for(mk, ik), sy = scale_for(my, iy), sq = scale_for(mq, iq);
    if (tid == 0) {
        inv[0] = ik;
        inv[1] = iy;
        inv[2] = iq;
    }
    if (own) {
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            unsigned char *row = slot + (4 * t4 + x) * TL::LDB + 2 * key;
            store_planes(row + TL::oW, TL::PL, Wr[x] * sk, Wi[x] * sk);
            store_planes(row + TL::oY, TL::PL, Yr[x] * sy, Yi[x] * sy);
            if constexpr (kNeedQ) store_planes(row + TL::oQ, TL::PL, Qr[x] * sq, Qi[x] * sq);
        }
    }
    if (fast) {
        // K[t][i] = W_t^* K_i and A[t][i] = Q_t^* K_i, 3 x TF32: warp = (matrix, half of the columns, Re / Im)
        const int which = warp & 1, nt = (warp >> 1) & 1, part = warp >> 2;
        if (kNeedQ || which == 0) {
            const float2 *A = which ? sQ : sW;
            float acc0[4] = {0.f, 0.f, 0.f, 0.f}, acc1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int kk = 0; kk < TL::KT; ++kk) {
                const float2 a0 = A[g * PS::LDF + 8 * kk + t4], a1 = A[(g + 8) * PS::LDF + 8 * kk + t4];
                const float2 a2 = A[g * PS::LDF + 8 * kk + t4 + 4], a3 = A[(g + 8) * PS::LDF + 8 * kk + t4 + 4];
                const float2 b0 = sK[(8 * nt + g) * PS::LDF + 8 * kk + t4], b1 = sK[(8 * nt + g) * PS::LDF + 8 * kk + t4 + 4];
                uint32_t rh[4], rl[4], ih[4], il[4], ch[2], cl[2], dh[2], dl[2];
                split_tf32(a0.x, rh[0], rl[0]);
                split_tf32(a1.x, rh[1], rl[1]);
                split_tf32(a2.x, rh[2], rl[2]);
                split_tf32(a3.x, rh[3], rl[3]);
                split_tf32(a0.y, ih[0], il[0]);
                split_tf32(a1.y, ih[1], il[1]);
                split_tf32(a2.y, ih[2], il[2]);
                split_tf32(a3.y, ih[3], il[3]);
                // Re: Ar Kr + Ai Ki;  Im: Ar Ki - Ai Kr
                split_tf32(part ? b0.y : b0.x, ch[0], cl[0]);
                split_tf32(part ? b1.y : b1.x, ch[1], cl[1]);
                split_tf32(part ? -b0.x : b0.y, dh[0], dl[0]);
                split_tf32(part ? -b1.x : b1.y, dh[1], dl[1]);
                mma3_tf32(acc0, rh, rl, ch, cl);
                mma3_tf32(acc1, ih, il, dh, dl);
            }
            float *dst = reinterpret_cast<float *>(which ? gq : gk) + part;
            const int i = 8 * nt + 2 * t4;
            dst[2 * (g * 17 + i)] = acc0[0] + acc1[0];
            dst[2 * (g * 17 + i + 1)] = acc0[1] + acc1[1];
            dst[2 * ((g + 8) * 17 + i)] = acc0[2] + acc1[2];
            dst[2 * ((g + 8) * 17 + i + 1)] = acc0[3] + acc1[3];
        }
    } else {
        // A coordinate decays too far to divide: every pair's decay as a running product.  The staging now takes k',
        // q' and alpha; a warp does rows warp and warp + 8, a lane keys lane, lane + 32.
        bar_sync(kBarAux, kAux);
        if (own) {
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const int t = 4 * t4 + x;
                sW[t * PS::LDF + key] = make_float2(pv.kr[x], pv.ki[x]);
                sK[t * PS::LDF + key] = make_float2(in.al[x], 0.f);
                if constexpr (kNeedQ) sQ[t * PS::LDF + key] = make_float2(pv.qr[x], pv.qi[x]);
            }
        }
        bar_sync(kBarAux, kAux);
        for (int t = warp; t < 16; t += 8) {
            float w[2] = {1.f, 1.f};
            for (int i = t; i >= 0; --i) {
                float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int e = 0; e < M / 32; ++e) {
                    const int j = lane + 32 * e;
                    const float2 b = sW[i * PS::LDF + j], x = sW[t * PS::LDF + j];
                    const float br = w[e] * b.x, bi = w[e] * b.y;
                    s[0] += x.x * br + x.y * bi;
                    s[1] += x.x * bi - x.y * br;
                    if constexpr (kNeedQ) {
                        const float2 y = sQ[t * PS::LDF + j];
                        s[2] += y.x * br + y.y * bi;
                        s[3] += y.x * bi - y.y * br;
                    }
                    w[e] *= sK[i * PS::LDF + j].x;
                }
#pragma unroll
                for (int d = 16; d >= 1; d >>= 1)
#pragma unroll
                    for (int e = 0; e < 4; ++e) s[e] += __shfl_xor_sync(0xffffffffu, s[e], d);
                if (lane == 0) {
                    gk[t * 17 + i] = make_float2(s[0], s[1]);
                    if constexpr (kNeedQ) gq[t * 17 + i] = make_float2(s[2], s[3]);
                }
            }
        }
    }
    bar_sync(kBarAux, kAux);
    if (warp == 0) {
        // N = K D_beta, strictly lower; only its lower part is read
        for (int e = lane; e < 256; e += 32) {
            const int t = e >> 4, i = e & 15;
            const float2 x = gk[t * 17 + i];
            const float f = i < t ? bsm[i] : 0.f;
            gk[t * 17 + i] = i < t ? make_float2(x.x * f, x.y * f) : make_float2(0.f, 0.f);
        }
        __syncwarp();
        invert_unit_lower16(gk, lane);
        store_small(slot + TL::oM, gk, nullptr, false, inv + 3, lane);
    } else if (kNeedQ && warp == 1) {
        store_small(slot + TL::oA, gq, bsm, true, inv + 4, lane);
    }
    return fast;
}

}  // namespace c16
}  // namespace sfda
