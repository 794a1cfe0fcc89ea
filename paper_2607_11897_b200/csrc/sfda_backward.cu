// sfda_backward: reverse-mode derivative of the recurrence of Section 3 (Eq. "sfda") with o_t = S_t^* q_t, chunk by
// chunk (16 tokens) at fp32 precision on the tensor cores.  (The paper asks for the backward pass only as something to
// be timed, App. E; what it computes is the adjoint of Eq. "sfda".)  Complex cotangents Xb mean dL = Re sum conj(Xb) dX,
// i.e. the ordinary gradient with respect to the (Re, Im) pair; yb_t = do_re + i do_im.
//
// Per chunk, with W, Y, Q, M, A^{qk} of sfda_chunk16_unrolled.cuh, S_0 the state before the chunk and G_C the cotangent of the
// state after it:
//
//   forward    U = M (V - W^* S_0)  (rows u_t^T = v_t^T - k_t^* Lambda_t S_{t-1}),   S_C = gamma_C S_0 + Y U
//   backward   Bc = M^H (Y^* G_C + (A^{qk} D_beta)^H Yb^*)   (rows beta_t p_t^*, p_t = G_t^* k_t),   dv_t = Re Bc_t
//              G_0 = conj(gamma_C) G_C + Q^T Yb^* - W^T Bc
//   gradients  dq_t = S_t yb_t,   f_t = G_t conj(u_t),   z_t = Lambda_t S_{t-1} (beta_t p_t),
//              dk_t = beta_t f_t - z_t,   dbeta_t = Re(f_t^* k_t),
//              D_t = D_{t+1} + q_t conj(dq_t) - beta_t conj(k_t) f_t - k_t conj(z_t)    (D_{T+1} = rowdot(S_T, G_T)),
//              dalpha_t = Re D_t / alpha_t,   dtheta_t = Im D_t
//
// where S_t, G_t inside a chunk are S_0, G_C plus rank-16 corrections, so dq, f, z come from three products with the
// boundary matrices (S_0 Yb^T, S_0 B^T, G_C U^H), two 16 x 16 matrices U Yb^T, U B^T and triangular products with the
// decayed keys and queries.  Where alpha_t < 1/16 the division would lose digits: dalpha comes from its definition,
// sum_c conj(S_{t-1,jc}) Zb_jc, rebuilt for that (token, coordinate) alone.
//
// One CTA per (batch, head) pair and block of value columns (all of them, or with few sequences 64 or 32: the columns
// never interact, and a second kernel adds the blocks' shares of the sums over the columns in a fixed order).  The
// CHAIN warps walk the sequence forward once, keeping the state every 64 tokens, then per segment of 64 tokens, last to
// first: forward again from the checkpoint, backward through it.  They leave S_0, U, G_C, Bc of a chunk in a scratch
// ring as the operand registers of the gradients' products.  The AUX warps prepare the chunks' operand tiles and turn
// what the chain leaves into gradients one chunk behind it.  The two meet at hardware barriers, one per slot:
//   FULL  operand tile ready       DONE  the chain is through with a chunk       FREE  its gradients are written
#include <type_traits>

#include "sfda_chunk16_unrolled.cuh"
#include "sfda_internal.h"

namespace sfda {
namespace {

using namespace c16;

constexpr int kSeg = 64;                    // tokens between checkpoints
constexpr int kSegChunks = kSeg / kC;
static_assert(kSegChunks == kSlots, "a segment's operand tiles fill the ring");

struct BwdArgsDev {
    const void *q, *k, *v, *d_o, *d_o_im;
    const float *alpha, *theta, *beta, *S0, *dS_T;
    void *dq, *dk, *dv;
    float *dalpha, *dtheta, *dbeta, *dS0;
    float *dq_p, *dk_p, *dalpha_p, *dtheta_p, *dbeta_p;   // shares of the column blocks: [blocks][rows][...] fp32
    float *check, *scratch;
    size_t rows;
    int T, H, NS;
};

// One slot of the scratch ring (global memory, one ring per CTA), all of it in the order of the consumer's registers:
// S_0, G_C as B operands [chain warp][key tile][Re / Im][lane] uint4 (two heads, two tails); U, Bc as A operands
// [chain warp][plane][lane] uint4; then the chunk's rotated keys and queries, decays and phases, 8 floats per
// (token, key).
template <int DK, int NB>
struct BwdScratch {
    static constexpr int NCW = NB / 16, KT = DK / 16, M = DK / 2;
    static constexpr int oS = 0, oU = oS + NCW * KT * 1024, oG = oU + NCW * 2048, oB = oG + NCW * KT * 1024;
    static constexpr int oV = oB + NCW * 2048, slot = oV + 16 * M * 32;
    static_assert((size_t)slot * kSlots <= (size_t)kSeg * DK * NB * 4, "the scratch ring must fit the workspace");
};

template <int DK, int NB>
struct BwdSmem {
    static constexpr int NCW = NB / 16, M = DK / 2;
    static constexpr int frag_bytes = 3 * NCW * 2048;             // Yb, Bc, U of the chunk as A operands
    static constexpr int stage = kSlots * Tile<DK>::bytes;        // PREP's staging and the gradients' operands share a place
    static constexpr int stage_bytes = frag_bytes > PrepSmem<DK>::stage_bytes ? frag_bytes : PrepSmem<DK>::stage_bytes;
    static constexpr int small = stage + stage_bytes;
    static constexpr int tri = small + PrepSmem<DK>::small_bytes; // the triangular factors of the corrections, 8 x 4 uint4 [32]
    static constexpr int uy = tri + 8 * 4 * 512;                  // U Yb^T, U B^T: float2 [2][16][17]
    static constexpr int scal = uy + 2 * 16 * 17 * 8;             // inverse scales [slot][NCW] (S, U, G, B), [NCW] Yb
    static constexpr int rg = scal + kSlots * NCW * 16 + NCW * 4 + (16 - NCW * 4 % 16) % 16;   // rowdot(S, G): float2 [2][NCW][M]
    static constexpr int db = rg + 2 * NCW * M * 8;               // dbeta: [8][16] floats
    static constexpr int flag = db + 8 * 16 * 4;                  // fast flag per slot
    static constexpr int bytes = flag + 16;
};

__device__ __forceinline__ int ring_slot(int r, int c) { return (r & 1) ? kSlots - 1 - c : c; }

// d += a (bh + bl); the head of `a` alone where its values are exact in fp16 (kExact)
template <bool kExact>
__device__ __forceinline__ void mma3x(float (&d)[4], const uint32_t (&ah)[4], const uint32_t (&al)[4], uint32_t bh0,
                                      uint32_t bh1, uint32_t bl0, uint32_t bl1)
{
    if constexpr (!kExact) mma_f16(d, al, bh0, bh1);
    mma_f16(d, ah, bl0, bl1);
    mma_f16(d, ah, bh0, bh1);
}
template <bool kExact>
__device__ __forceinline__ void product_small_conj(float (&re)[2][4], float (&im)[2][4], const TokFrag &a, const TokFrag &b,
                                                   float f, bool has_im)
{
#pragma unroll
    for (int n = 0; n < 2; ++n) {
        float rr[4] = {0.f, 0.f, 0.f, 0.f}, ir[4] = {0.f, 0.f, 0.f, 0.f}, ri[4] = {0.f, 0.f, 0.f, 0.f};
        mma3x<kExact>(rr, a.rh, a.rl, b.rh[2 * n], b.rh[2 * n + 1], b.rl[2 * n], b.rl[2 * n + 1]);
        mma3x<kExact>(ri, a.rh, a.rl, b.ih[2 * n], b.ih[2 * n + 1], b.il[2 * n], b.il[2 * n + 1]);
        if (has_im) {
            mma3x<kExact>(rr, a.ih, a.il, b.ih[2 * n], b.ih[2 * n + 1], b.il[2 * n], b.il[2 * n + 1]);
            mma3x<kExact>(ir, a.ih, a.il, b.rh[2 * n], b.rh[2 * n + 1], b.rl[2 * n], b.rl[2 * n + 1]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            re[n][i] = fmaf(f, rr[i], re[n][i]);
            im[n][i] = fmaf(f, ir[i] - ri[i], im[n][i]);
        }
    }
}

// the [value x token] operand as the A operand (token, value) of products over the value columns
__device__ __forceinline__ void publish_frag(uint4 *p, const TokFrag &f, int lane)
{
    p[0 * 32 + lane] = make_uint4(transpose8x8(f.rh[0]), transpose8x8(f.rh[2]), transpose8x8(f.rh[1]), transpose8x8(f.rh[3]));
    p[1 * 32 + lane] = make_uint4(transpose8x8(f.rl[0]), transpose8x8(f.rl[2]), transpose8x8(f.rl[1]), transpose8x8(f.rl[3]));
    p[2 * 32 + lane] = make_uint4(transpose8x8(f.ih[0]), transpose8x8(f.ih[2]), transpose8x8(f.ih[1]), transpose8x8(f.ih[3]));
    p[3 * 32 + lane] = make_uint4(transpose8x8(f.il[0]), transpose8x8(f.il[2]), transpose8x8(f.il[1]), transpose8x8(f.il[3]));
}

template <int KT>
__device__ __forceinline__ void store_state(float4 *p, const float (&sr)[KT][4], const float (&si)[KT][4], int lane)
{
#pragma unroll
    for (int n = 0; n < KT; ++n) {
        p[(2 * n) * 32 + lane] = make_float4(sr[n][0], sr[n][1], sr[n][2], sr[n][3]);
        p[(2 * n + 1) * 32 + lane] = make_float4(si[n][0], si[n][1], si[n][2], si[n][3]);
    }
}
template <int KT>
__device__ __forceinline__ void load_state(const float4 *p, float (&sr)[KT][4], float (&si)[KT][4], int lane)
{
#pragma unroll
    for (int n = 0; n < KT; ++n) {
        const float4 x = p[(2 * n) * 32 + lane], y = p[(2 * n + 1) * 32 + lane];
        sr[n][0] = x.x; sr[n][1] = x.y; sr[n][2] = x.z; sr[n][3] = x.w;
        si[n][0] = y.x; si[n][1] = y.y; si[n][2] = y.z; si[n][3] = y.w;
    }
}

__device__ __forceinline__ void st_val4(float *p, float4 x) { *reinterpret_cast<float4 *>(p) = x; }
__device__ __forceinline__ void st_val4(__nv_bfloat16 *p, float4 x)
{
    const __nv_bfloat162 lo = __floats2bfloat162_rn(x.x, x.y), hi = __floats2bfloat162_rn(x.z, x.w);
    *reinterpret_cast<uint2 *>(p) = make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
}

__device__ __forceinline__ float2 cmul(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) { return make_float2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x); }   // conj(a) b

// one 16-bit half of the head and of the tail, added
__device__ __forceinline__ float join_half(uint32_t h, uint32_t l, int half)
{
    const float2 x = unpack_f16(h), y = unpack_f16(l);
    return half ? x.y + y.y : x.x + y.x;
}

// ---- AUX: the gradients of one chunk --------------------------------------------------------------
template <int DK, int DVT, int NB, typename T>
__device__ __forceinline__ void chunk_gradients(const BwdArgsDev &a, unsigned char *smem, unsigned char *scr, int slot, int rpar,
                                             bool first, int t0, size_t row0, float2 (&carry)[2], int tid)
{
    using L = BwdSmem<DK, NB>;
    using SC = BwdScratch<DK, NB>;
    constexpr int NCW = L::NCW, M = L::M, KT = M / 8, NSL = DVT / NB;
    constexpr bool kExact = sizeof(T) == 2;
    const int lane = tid & 31, warp = tid >> 5, g = lane >> 2, t4 = lane & 3, c0 = blockIdx.y * NB;
    const bool has_im = a.d_o_im != nullptr;
    uint4 *frag = reinterpret_cast<uint4 *>(smem + L::stage);                     // [Yb, Bc, U][NCW][4][32]
    uint4 *tri = reinterpret_cast<uint4 *>(smem + L::tri);
    float2 *uy = reinterpret_cast<float2 *>(smem + L::uy);
    float *scal = reinterpret_cast<float *>(smem + L::scal), *yscal = scal + kSlots * NCW * 4;
    const float *sc = scal + slot * NCW * 4;
    float *db = reinterpret_cast<float *>(smem + L::db);
    const uint4 *pS = reinterpret_cast<const uint4 *>(scr + SC::oS), *pG = reinterpret_cast<const uint4 *>(scr + SC::oG);
    const float4 *vals = reinterpret_cast<const float4 *>(scr + SC::oV);

    // operands over the value columns: Yb from the caller's arrays, Bc and U from the ring
    for (int w = warp; w < NCW; w += kAuxWarps) {
        float2 y[2][4];
        uint32_t m = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int t = t0 + g + 8 * (i & 1);
            y[0][i] = y[1][i] = make_float2(0.f, 0.f);
            if (t < a.T) {
                const size_t at = (row0 + (size_t)t * a.H) * DVT + c0 + 16 * w + 2 * t4 + 8 * (i >> 1);
                y[0][i] = ld_pair(static_cast<const T *>(a.d_o), at);
                if (has_im) y[1][i] = ld_pair(static_cast<const T *>(a.d_o_im), at);
            }
            m = max(m, max(max(abs_bits(y[0][i].x), abs_bits(y[0][i].y)), max(abs_bits(y[1][i].x), abs_bits(y[1][i].y))));
        }
        const uint4 *pB = reinterpret_cast<const uint4 *>(scr + SC::oB) + w * 128, *pU = reinterpret_cast<const uint4 *>(scr + SC::oU) + w * 128;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            frag[((NCW + w) * 4 + p) * 32 + lane] = pB[p * 32 + lane];
            frag[((2 * NCW + w) * 4 + p) * 32 + lane] = pU[p * 32 + lane];
        }
        float inv;
        const float s = scale_for(__reduce_max_sync(0xffffffffu, m), inv);
        if (lane == 0) yscal[w] = inv;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            uint32_t h[4], l[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) split_f16(y[c][i].x * s, y[c][i].y * s, h[i], l[i]);
            frag[(w * 4 + 2 * c) * 32 + lane] = make_uint4(h[0], h[1], h[2], h[3]);
            frag[(w * 4 + 2 * c + 1) * 32 + lane] = make_uint4(l[0], l[1], l[2], l[3]);
        }
    }
    bar_sync(kBarAux, kAux);

    // U Yb^T (index [i][t]: u_i . yb_t) and U B^T (b_t = beta_t p_t = conj of the rows of Bc): warp = (matrix, half of
    // the columns, Re / Im); the A-operand registers of tokens 0-7 / 8-15 are the B operand of that half
    {
        const int mat = warp & 1, nt = (warp >> 1) & 1, part = warp >> 2;
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        const float sx = (mat && part) ? -1.f : 1.f, sz = (!mat && !part) ? -1.f : 1.f;
#pragma unroll 2
        for (int w = 0; w < NCW; ++w) {
            const uint4 *fu = frag + (2 * NCW + w) * 128 + lane, *fx = frag + (mat * NCW + w) * 128 + lane;
            const uint4 urh = fu[0], url = fu[32], uih = fu[64], uil = fu[96];
            const uint4 xh = fx[part * 64], xl = fx[part * 64 + 32], zh = fx[64 - part * 64], zl = fx[96 - part * 64];
            const uint32_t ar[4] = {urh.x, urh.y, urh.z, urh.w}, arl[4] = {url.x, url.y, url.z, url.w};
            const uint32_t ai[4] = {uih.x, uih.y, uih.z, uih.w}, ail[4] = {uil.x, uil.y, uil.z, uil.w};
            float p[4] = {0.f, 0.f, 0.f, 0.f}, z[4] = {0.f, 0.f, 0.f, 0.f};
            mma3(p, ar, arl, nt ? xh.y : xh.x, nt ? xh.w : xh.z, nt ? xl.y : xl.x, nt ? xl.w : xl.z);
            mma3(z, ai, ail, nt ? zh.y : zh.x, nt ? zh.w : zh.z, nt ? zl.y : zl.x, nt ? zl.w : zl.z);
            const float f = sc[4 * w + 1] * (mat ? sc[4 * w + 3] : yscal[w]);
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i] = fmaf(f, fmaf(sx, p[i], sz * z[i]), acc[i]);
        }
        float *dst = reinterpret_cast<float *>(uy + mat * 16 * 17) + part;
        const int t = 8 * nt + 2 * t4;
        dst[2 * (g * 17 + t)] = acc[0];
        dst[2 * (g * 17 + t + 1)] = acc[1];
        dst[2 * ((g + 8) * 17 + t)] = acc[2];
        dst[2 * ((g + 8) * 17 + t + 1)] = acc[3];
    }

    // X1 = S_0 yb_t, X2 = S_0 b_t, X3 = G_C conj(u_t) for the keys of tile `warp` (accumulator layout: token g (+ 8),
    // keys 2 t4, + 1); every chain warp's 16 columns come with scales of their own
    float x1r[4] = {0.f, 0.f, 0.f, 0.f}, x1i[4] = {0.f, 0.f, 0.f, 0.f}, x2r[4] = {0.f, 0.f, 0.f, 0.f};
    float x2i[4] = {0.f, 0.f, 0.f, 0.f}, x3r[4] = {0.f, 0.f, 0.f, 0.f}, x3i[4] = {0.f, 0.f, 0.f, 0.f};
    if (warp < KT) {
#pragma unroll 1
        for (int w = 0; w < NCW; ++w) {
            const uint4 s0 = pS[((w * KT + warp) * 2) * 32 + lane], s1 = pS[((w * KT + warp) * 2 + 1) * 32 + lane];
            const uint4 g0 = pG[((w * KT + warp) * 2) * 32 + lane], g1 = pG[((w * KT + warp) * 2 + 1) * 32 + lane];
            {
                const uint4 *fy = frag + w * 128 + lane;
                const uint4 h = fy[0], l = fy[32];
                const uint32_t ah[4] = {h.x, h.y, h.z, h.w}, al[4] = {l.x, l.y, l.z, l.w};
                float pr[4] = {0.f, 0.f, 0.f, 0.f}, pi[4] = {0.f, 0.f, 0.f, 0.f}, mr[4] = {0.f, 0.f, 0.f, 0.f};
                mma3x<kExact>(pr, ah, al, s0.x, s0.y, s0.z, s0.w);
                mma3x<kExact>(pi, ah, al, s1.x, s1.y, s1.z, s1.w);
                if (has_im) {
                    const uint4 h2 = fy[64], l2 = fy[96];
                    const uint32_t bh[4] = {h2.x, h2.y, h2.z, h2.w}, bl[4] = {l2.x, l2.y, l2.z, l2.w};
                    mma3x<kExact>(mr, bh, bl, s1.x, s1.y, s1.z, s1.w);
                    mma3x<kExact>(pi, bh, bl, s0.x, s0.y, s0.z, s0.w);
                }
                const float f = sc[4 * w] * yscal[w];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    x1r[i] = fmaf(f, pr[i] - mr[i], x1r[i]);
                    x1i[i] = fmaf(f, pi[i], x1i[i]);
                }
            }
            auto conj_product = [&](const uint4 *fx, const uint4 &b0, const uint4 &b1, float f, float (&xr)[4], float (&xi)[4]) {
                const uint4 h = fx[0], l = fx[32], h2 = fx[64], l2 = fx[96];
                const uint32_t rh[4] = {h.x, h.y, h.z, h.w}, rl[4] = {l.x, l.y, l.z, l.w};
                const uint32_t ih[4] = {h2.x, h2.y, h2.z, h2.w}, il[4] = {l2.x, l2.y, l2.z, l2.w};
                float pr[4] = {0.f, 0.f, 0.f, 0.f}, pi[4] = {0.f, 0.f, 0.f, 0.f}, mi[4] = {0.f, 0.f, 0.f, 0.f};
                mma3(pr, rh, rl, b0.x, b0.y, b0.z, b0.w);
                mma3(pi, rh, rl, b1.x, b1.y, b1.z, b1.w);
                mma3(mi, ih, il, b0.x, b0.y, b0.z, b0.w);
                mma3(pr, ih, il, b1.x, b1.y, b1.z, b1.w);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    xr[i] = fmaf(f, pr[i], xr[i]);
                    xi[i] = fmaf(f, pi[i] - mi[i], xi[i]);
                }
            };
            conj_product(frag + (NCW + w) * 128 + lane, s0, s1, sc[4 * w] * sc[4 * w + 3], x2r, x2i);
            conj_product(frag + (2 * NCW + w) * 128 + lane, g0, g1, sc[4 * w + 2] * sc[4 * w + 1], x3r, x3i);
        }
    }
    bar_sync(kBarAux, kAux);

    // the triangular factors of the corrections as TF32 A operands: warp = (sum, step of eight tokens); the k index of
    // a step runs over tokens 4 t4 + 2 step (slot t4) and + 1 (slot t4 + 4), PREP's order of tokens
    const float *beta_row = a.beta + row0;
    {
        const int sum = warp >> 1, i0 = 4 * t4 + 2 * (warp & 1);
        uint32_t rh[4], rl[4], ih[4], il[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int t = g + 8 * (e & 1), i = i0 + (e >> 1);
            float2 x = make_float2(0.f, 0.f);
            if (sum < 2) {
                if (sum == 0 ? i <= t : i < t) {
                    const float be = t0 + i < a.T ? beta_row[(size_t)(t0 + i) * a.H] : 0.f;
                    x = uy[sum * 272 + i * 17 + t];
                    x = make_float2(be * x.x, be * x.y);
                }
            } else if (sum == 2 ? i >= t : i > t) {
                x = uy[(sum - 2) * 272 + t * 17 + i];
                x = sum == 2 ? make_float2(x.x, -x.y) : make_float2(-x.x, x.y);
            }
            split_tf32(x.x, rh[e], rl[e]);
            split_tf32(x.y, ih[e], il[e]);
        }
        uint4 *p = tri + warp * 128 + lane;
        p[0] = make_uint4(rh[0], rh[1], rh[2], rh[3]);
        p[32] = make_uint4(rl[0], rl[1], rl[2], rl[3]);
        p[64] = make_uint4(ih[0], ih[1], ih[2], ih[3]);
        p[96] = make_uint4(il[0], il[1], il[2], il[3]);
    }
    bar_sync(kBarAux, kAux);

    if (warp < KT) {
        const bool fast = reinterpret_cast<const int *>(smem + L::flag)[slot] != 0;
        float z1r[4] = {0.f, 0.f, 0.f, 0.f}, z1i[4] = {0.f, 0.f, 0.f, 0.f}, z2r[4] = {0.f, 0.f, 0.f, 0.f};
        float z2i[4] = {0.f, 0.f, 0.f, 0.f}, z3r[4] = {0.f, 0.f, 0.f, 0.f}, z3i[4] = {0.f, 0.f, 0.f, 0.f};
        if (fast) {
            auto tri_product = [&](int sum, int step, const float2 &b0, const float2 &b1, float (&zr)[4], float (&zi)[4]) {
                const uint4 *p = tri + (2 * sum + step) * 128 + lane;
                const uint4 h = p[0], l = p[32], h2 = p[64], l2 = p[96];
                const uint32_t rh[4] = {h.x, h.y, h.z, h.w}, rl[4] = {l.x, l.y, l.z, l.w};
                const uint32_t ih[4] = {h2.x, h2.y, h2.z, h2.w}, il[4] = {l2.x, l2.y, l2.z, l2.w};
                uint32_t brh[2], brl[2], bih[2], bil[2], nih[2], nil[2];
                split_tf32(b0.x, brh[0], brl[0]);
                split_tf32(b1.x, brh[1], brl[1]);
                split_tf32(b0.y, bih[0], bil[0]);
                split_tf32(b1.y, bih[1], bil[1]);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    nih[i] = bih[i] ^ 0x80000000u;
                    nil[i] = bil[i] ^ 0x80000000u;
                }
                mma3_tf32(zr, rh, rl, brh, brl);
                mma3_tf32(zi, rh, rl, bih, bil);
                mma3_tf32(zr, ih, il, nih, nil);
                mma3_tf32(zi, ih, il, brh, brl);
            };
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                float2 kh[2], qw[2], wv[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float4 *p = vals + ((4 * t4 + 2 * s + e) * M + 8 * warp + g) * 2;
                    const float4 x = p[0], y = p[1];
                    const float ia = __frcp_rn(y.x);
                    kh[e] = make_float2(x.x * ia, x.y * ia);
                    wv[e] = make_float2(x.x * y.x, x.y * y.x);
                    qw[e] = make_float2(x.z * y.x, x.w * y.x);
                }
                tri_product(0, s, kh[0], kh[1], z1r, z1i);
                tri_product(1, s, kh[0], kh[1], z2r, z2i);
                tri_product(2, s, qw[0], qw[1], z3r, z3i);
                tri_product(3, s, wv[0], wv[1], z3r, z3i);
            }
        }
        float2 dqv[4], dkv[4], dd[4];
        float al[4], dbp[2] = {0.f, 0.f};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = i >> 1, e = i & 1, tl = g + 8 * r, t = t0 + tl, key = 8 * warp + 2 * t4 + e;
            const size_t row = row0 + (size_t)t * a.H;
            const float4 x = vals[(tl * M + key) * 2], y = vals[(tl * M + key) * 2 + 1];
            const float4 last = vals[(15 * M + key) * 2 + 1];                     // e^{i phi_C}
            const float2 kp = make_float2(x.x, x.y), qp = make_float2(x.z, x.w), ph = make_float2(y.z, y.w);
            const float be = t < a.T ? a.beta[row] : 0.f;
            al[i] = t < a.T ? a.alpha[row * M + key] : 1.f;
            const float2 x3 = cmulc(make_float2(last.z, last.w), make_float2(x3r[i], x3i[i]));
            float2 qb, zb, fb;
            if (fast) {
                const float ia = __frcp_rn(y.x);
                qb = make_float2(y.x * (x1r[i] + z1r[i]), y.x * (x1i[i] + z1i[i]));
                zb = make_float2(y.x * (x2r[i] + z2r[i]), y.x * (x2i[i] + z2i[i]));
                fb = make_float2(fmaf(y.y, x3.x, ia * z3r[i]), fmaf(y.y, x3.y, ia * z3i[i]));
            } else {
                // decays too strong to divide by: running products, token by token
                float w = 1.f;
                qb = zb = fb = make_float2(0.f, 0.f);
                for (int j = tl; j >= 0; --j) {
                    const size_t rj = row0 + (size_t)(t0 + j) * a.H;
                    const float4 kj = vals[(j * M + key) * 2];
                    const float bj = t0 + j < a.T ? w * a.beta[rj] : 0.f;
                    const float2 kk = make_float2(bj * kj.x, bj * kj.y);
                    const float2 p = cmul(kk, uy[j * 17 + tl]), s = cmul(kk, uy[272 + j * 17 + tl]);
                    qb = make_float2(qb.x + p.x, qb.y + p.y);
                    if (j < tl) zb = make_float2(zb.x + s.x, zb.y + s.y);
                    w *= t0 + j < a.T ? a.alpha[rj * M + key] : 1.f;
                }
                qb = make_float2(fmaf(w, x1r[i], qb.x), fmaf(w, x1i[i], qb.y));
                zb = make_float2(fmaf(w, x2r[i], zb.x), fmaf(w, x2i[i], zb.y));
                w = 1.f;
                for (int l = tl; l < 16; ++l) {
                    const float4 kl = vals[(l * M + key) * 2];
                    const float2 p = cmulc(uy[tl * 17 + l], make_float2(w * kl.z, w * kl.w));
                    fb = make_float2(fb.x + p.x, fb.y + p.y);
                    if (l > tl) {
                        const float2 s = cmulc(uy[272 + tl * 17 + l], make_float2(w * kl.x, w * kl.y));
                        fb = make_float2(fb.x - s.x, fb.y - s.y);
                    }
                    if (l < 15 && t0 + l + 1 < a.T) w *= a.alpha[(row0 + (size_t)(t0 + l + 1) * a.H) * M + key];
                }
                fb = make_float2(fmaf(w, x3.x, fb.x), fmaf(w, x3.y, fb.y));
            }
            const float2 dkp = make_float2(be * fb.x - zb.x, be * fb.y - zb.y);
            dqv[i] = cmul(ph, qb);
            dkv[i] = cmul(ph, dkp);
            dbp[r] += fb.x * kp.x + fb.y * kp.y;
            const float2 p = cmulc(qb, qp), s = cmulc(kp, make_float2(be * fb.x, be * fb.y)), z = cmulc(zb, kp);
            dd[i] = make_float2(p.x - s.x - z.x, p.y - s.y - z.y);
        }
        // D: sums over the tokens behind, down to each token (tokens 8-15 in i = 2, 3, tokens 0-7 in i = 0, 1)
        if (first) {
            const float2 *rg = reinterpret_cast<const float2 *>(smem + L::rg) + rpar * NCW * M;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                carry[e] = make_float2(0.f, 0.f);
                for (int w = 0; w < NCW; ++w) {
                    const float2 x = rg[w * M + 8 * warp + 2 * t4 + e];
                    carry[e] = make_float2(carry[e].x + x.x, carry[e].y + x.y);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int d = 4; d < 32; d <<= 1) {
                const float ox = __shfl_down_sync(0xffffffffu, dd[i].x, d), oy = __shfl_down_sync(0xffffffffu, dd[i].y, d);
                if (lane + d < 32) dd[i] = make_float2(dd[i].x + ox, dd[i].y + oy);
            }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            dd[2 + e] = make_float2(dd[2 + e].x + carry[e].x, dd[2 + e].y + carry[e].y);
            dd[e] = make_float2(dd[e].x + __shfl_sync(0xffffffffu, dd[2 + e].x, t4), dd[e].y + __shfl_sync(0xffffffffu, dd[2 + e].y, t4));
            carry[e] = make_float2(__shfl_sync(0xffffffffu, dd[e].x, t4), __shfl_sync(0xffffffffu, dd[e].y, t4));
        }
        float dal[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) dal[i] = __fdiv_rn(dd[i].x, al[i]);
        // small alpha: from the definition, one (token, key) at a time
#pragma unroll 1
        for (int i = 0; i < 4; ++i) {
            unsigned todo = __ballot_sync(0xffffffffu, (i == 0 ? al[0] : i == 1 ? al[1] : i == 2 ? al[2] : al[3]) < 0.0625f);
            while (todo) {
                const int src = __ffs(todo) - 1;
                todo &= todo - 1;
                const int tl = (src >> 2) + 8 * (i >> 1), kl = 2 * (src & 3) + (i & 1), key = 8 * warp + kl;
                float sum = 0.f;
                float cst = 1.f, snt = 0.f;
                for (int val = lane; val < NB; val += 32) {
                    const int w = val >> 4, vl = val & 15, hf = vl & 1;
                    auto state = [&](const uint4 *base, float inv) {
                        const uint32_t *p = reinterpret_cast<const uint32_t *>(base + ((w * KT + warp) * 2) * 32 + 4 * kl + ((vl & 7) >> 1)) + (vl >> 3);
                        return make_float2(inv * join_half(p[0], p[2], hf), inv * join_half(p[128], p[130], hf));
                    };
                    auto token = [&](int mat, int tok, float inv) {
                        const uint32_t *p = reinterpret_cast<const uint32_t *>(frag + (mat * NCW + w) * 128 + 4 * (tok & 7) + ((vl & 7) >> 1)) + (tok >> 3) + 2 * (vl >> 3);
                        return make_float2(inv * join_half(p[0], p[128], hf), inv * join_half(p[256], p[384], hf));
                    };
                    float2 s = state(pS, sc[4 * w]), z = state(pG, sc[4 * w + 2]);
                    for (int j = 0; j < 16; ++j) {           // S_{t-1}
                        if (j >= tl) break;
                        const size_t rj = row0 + (size_t)(t0 + j) * a.H;
                        const float4 x = vals[(j * M + key) * 2], y = vals[(j * M + key) * 2 + 1];
                        float sn, cs;
                        sincosf(a.theta[rj * M + key], &sn, &cs);
                        const float aj = a.alpha[rj * M + key], bj = a.beta[rj];
                        const float2 kj = cmul(make_float2(y.z, y.w), make_float2(bj * x.x, bj * x.y)), u = token(2, j, sc[4 * w + 1]);
                        s = cmul(make_float2(aj * cs, aj * sn), s);
                        const float2 p = cmul(kj, u);
                        s = make_float2(s.x + p.x, s.y + p.y);
                    }
                    for (int l = 15; l >= tl; --l) {         // the cotangent of Lambda_t S_{t-1}
                        if (t0 + l >= a.T) continue;
                        const size_t rl = row0 + (size_t)(t0 + l) * a.H;
                        const float4 x = vals[(l * M + key) * 2], y = vals[(l * M + key) * 2 + 1];
                        const float2 ph = make_float2(y.z, y.w), ql = cmul(ph, make_float2(x.z, x.w)), kj = cmul(ph, make_float2(x.x, x.y));
                        const float2 yb = token(0, l, yscal[w]), bc = token(1, l, sc[4 * w + 3]);
                        const float2 p = cmulc(yb, ql), m = cmul(kj, bc);
                        z = make_float2(z.x + p.x - m.x, z.y + p.y - m.y);
                        float sn, cs;
                        sincosf(a.theta[rl * M + key], &sn, &cs);
                        if (l > tl) {
                            const float aj = a.alpha[rl * M + key];
                            z = cmulc(make_float2(aj * cs, aj * sn), z);
                        } else {
                            cst = cs;
                            snt = sn;
                        }
                    }
                    const float2 lb = cmulc(s, z);
                    sum += lb.x * cst + lb.y * snt;          // Re(conj(lambda bar) e^{i theta})
                }
#pragma unroll
                for (int d = 16; d >= 1; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
                if (lane == src) {
                    if (i == 0) dal[0] = sum;
                    else if (i == 1) dal[1] = sum;
                    else if (i == 2) dal[2] = sum;
                    else dal[3] = sum;
                }
            }
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int t = t0 + g + 8 * r;
            if (t < a.T) {
                const size_t row = row0 + (size_t)t * a.H;
                const size_t ak = row * DK + 2 * (8 * warp + 2 * t4), am = row * M + 8 * warp + 2 * t4;
                const float4 q4 = make_float4(dqv[2 * r].x, dqv[2 * r].y, dqv[2 * r + 1].x, dqv[2 * r + 1].y);
                const float4 k4 = make_float4(dkv[2 * r].x, dkv[2 * r].y, dkv[2 * r + 1].x, dkv[2 * r + 1].y);
                const float2 a2 = make_float2(dal[2 * r], dal[2 * r + 1]), th2 = make_float2(dd[2 * r].y, dd[2 * r + 1].y);
                if constexpr (NSL == 1) {
                    st_val4(static_cast<T *>(a.dq) + ak, q4);
                    st_val4(static_cast<T *>(a.dk) + ak, k4);
                    *reinterpret_cast<float2 *>(a.dalpha + am) = a2;
                    *reinterpret_cast<float2 *>(a.dtheta + am) = th2;
                } else {
                    const size_t off = (size_t)blockIdx.y * a.rows;
                    st_val4(a.dq_p + off * DK + ak, q4);
                    st_val4(a.dk_p + off * DK + ak, k4);
                    *reinterpret_cast<float2 *>(a.dalpha_p + off * M + am) = a2;
                    *reinterpret_cast<float2 *>(a.dtheta_p + off * M + am) = th2;
                }
            }
            float x = dbp[r];
            x += __shfl_xor_sync(0xffffffffu, x, 1);
            x += __shfl_xor_sync(0xffffffffu, x, 2);
            if (t4 == 0) db[warp * 16 + g + 8 * r] = x;
        }
    }
    bar_sync(kBarAux, kAux);
    if (tid < 16 && t0 + tid < a.T) {
        float x = 0.f;
#pragma unroll
        for (int w = 0; w < KT; ++w) x += db[w * 16 + tid];
        const size_t row = row0 + (size_t)(t0 + tid) * a.H;
        if constexpr (NSL == 1) a.dbeta[row] = x;
        else a.dbeta_p[(size_t)blockIdx.y * a.rows + row] = x;
    }
}

template <int DK, int DVT, int NB, typename T>
__global__ void __launch_bounds__(kAux + 2 * NB, 1) sfda_backward_kernel(const BwdArgsDev a)
{
    using TL = Tile<DK>;
    using L = BwdSmem<DK, NB>;
    using SC = BwdScratch<DK, NB>;
    constexpr int kAll = kAux + 2 * NB, NCW = NB / 16, M = DK / 2, KT = TL::KT;
    constexpr bool kExact = sizeof(T) == 2;
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, bh = blockIdx.x, h = bh % a.H, b = bh / a.H, c0 = blockIdx.y * NB;
    const size_t row0 = (size_t)b * a.T * a.H + h;                       // row of token t: row0 + t H
    const int nch = (a.T + kC - 1) / kC, NS = a.NS;
    unsigned char *ring = reinterpret_cast<unsigned char *>(a.scratch + ((size_t)bh * DVT + c0) * kSeg * DK);
    const int last_nch = nch - (NS - 1) * kSegChunks;                    // chunks of the last segment

    if (tid < kAux) {
        if constexpr (NB == 128) asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
        const int lane = tid & 31, warp = tid >> 5, g = lane >> 2, t4 = lane & 3, key = 8 * warp + g;
        const T *q = static_cast<const T *>(a.q), *k = static_cast<const T *>(a.k);
        float2 *stage = reinterpret_cast<float2 *>(smem + L::stage);
        int par = 0;
        for (int c = 0; c < nch; ++c) {                                  // first sweep: keys only
            const int slot = c % kSlots;
            if (c >= kSlots) bar_sync(kBarDone + slot, kAll);
            PrepIn in;
            PrepVals pv;
            prep_load<DK, T>(in, nullptr, k, a.alpha, a.theta, a.beta, row0, a.H, c * kC, a.T, key, t4);
            prep_chunk<DK, false>(in, pv, smem + slot * TL::bytes, stage, smem + L::small, par, tid);
            bar_arrive(kBarFull + slot, kAll);
            par ^= 1;
        }
        for (int c = max(nch - kSlots, 0); c < nch; ++c) bar_sync(kBarDone + c % kSlots, kAll);
        // Second sweep.  Chunks are prepared in the order the chain goes forward through the segments (last segment
        // first) and their gradients follow in the order it comes back; the ring's slots are assigned so that the
        // p-th chunk prepared takes the slot of gradient p - 4.
        float2 carry[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        for (int p = 0; p < nch + kSlots; ++p) {
            if (p >= kSlots) {
                const int n = p - kSlots, r = n < last_nch ? 0 : 1 + (n - last_nch) / kSegChunks;
                const int nc = r == 0 ? last_nch : kSegChunks, at = r == 0 ? n : (n - last_nch) % kSegChunks, c = nc - 1 - at;
                const int slot = ring_slot(r, c);
                bar_sync(kBarDone + slot, kAll);
                chunk_gradients<DK, DVT, NB, T>(a, smem, ring + (size_t)slot * SC::slot, slot, r & 1, at == 0,
                                                (NS - 1 - r) * kSeg + c * kC, row0, carry, tid);
                if (p < nch) bar_arrive(kBarFree + slot, kAll);
            }
            if (p < nch) {
                const int r = p < last_nch ? 0 : 1 + (p - last_nch) / kSegChunks, c = r == 0 ? p : (p - last_nch) % kSegChunks;
                const int slot = ring_slot(r, c);
                PrepIn in;
                PrepVals pv;
                prep_load<DK, T>(in, q, k, a.alpha, a.theta, a.beta, row0, a.H, (NS - 1 - r) * kSeg + c * kC, a.T, key, t4);
                const bool fast = prep_chunk<DK, true>(in, pv, smem + slot * TL::bytes, stage, smem + L::small, par, tid);
                bar_arrive(kBarFull + slot, kAll);
                par ^= 1;
                if (tid == 0) reinterpret_cast<int *>(smem + L::flag)[slot] = fast;
                if (key < M) {
                    float4 *vals = reinterpret_cast<float4 *>(ring + (size_t)slot * SC::slot + SC::oV) + (4 * t4 * M + key) * 2;
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        vals[x * M * 2] = make_float4(pv.kr[x], pv.ki[x], pv.qr[x], pv.qi[x]);
                        vals[x * M * 2 + 1] = make_float4(pv.a[x], pv.sfx[x], pv.cs[x], pv.sn[x]);
                    }
                }
            }
        }
        return;
    }

    if constexpr (NB == 128) asm volatile("setmaxnreg.inc.sync.aligned.u32 168;");
    const int lane = tid & 31, w = (tid - kAux) >> 5, g = lane >> 2, t4 = lane & 3;
    const int col = c0 + 16 * w + g;                                     // and col + 8
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem);
    float *scal = reinterpret_cast<float *>(smem + L::scal);
    auto checkpoint = [&](int s) {
        return reinterpret_cast<float4 *>(a.check + (((size_t)bh * NS + s) * DVT + c0 + 16 * w) * DK);
    };
    auto state_at = [&](int n, int i) {                                  // Re of (key, column) of accumulator element (n, i)
        return ((size_t)bh * DK + 2 * (8 * n + 2 * t4 + (i & 1))) * DVT + col + 8 * (i >> 1);
    };
    auto load_tokens = [&](const void *p, int t0, float sign, float (&x)[2][4]) {
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int t = t0 + 8 * n + 2 * t4 + (i & 1);
                x[n][i] = p && t < a.T ? sign * ld_val(static_cast<const T *>(p), (row0 + (size_t)t * a.H) * DVT + col + 8 * (i >> 1)) : 0.f;
            }
    };
    float sr[KT][4], si[KT][4];
#pragma unroll
    for (int n = 0; n < KT; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            sr[n][i] = a.S0 ? a.S0[state_at(n, i)] : 0.f;
            si[n][i] = a.S0 ? a.S0[state_at(n, i) + DVT] : 0.f;
        }

    // forward through one chunk: U = M (V - W^* S), S <- gamma_C S + Y U
    auto forward_chunk = [&](int slot, int t0, auto pub, bool update) {
        constexpr bool kPub = decltype(pub)::value;
        unsigned char *scr = ring + (size_t)slot * SC::slot;
        float rr[2][4], ri[2][4];
        load_tokens(a.v, t0, 1.f, rr);
        bar_sync(kBarFull + slot, kAll);
        const uint32_t tile = base + slot * TL::bytes;
        const float *inv = reinterpret_cast<const float *>(smem + slot * TL::bytes + TL::oS);
        float isv;
        const float ss = scale_for(__reduce_max_sync(0xffffffffu, max(max_bits4(sr), max_bits4(si))), isv);
        float acc[1][3][2][4];
        const uint32_t tiles[1] = {tile + TL::oW};
        product_over_keys<DK, 1, kPub>(acc, sr, si, ss, tiles, lane, reinterpret_cast<uint4 *>(scr + SC::oS) + w * KT * 64);
        const float fw = isv * inv[0];
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                rr[n][i] = fmaf(-fw, acc[0][0][n][i], rr[n][i]);
                ri[n][i] = -fw * (acc[0][1][n][i] - acc[0][2][n][i]);
            }
        TokFrag fr, fb;
        const float ir = make_frag(fr, rr, ri);
        load_small<false>(fb, tile + TL::oM, lane);
        product_small<false>(rr, ri, fr, fb, ir * inv[3]);
        const float iu = make_frag(fr, rr, ri);
        if constexpr (kPub) {
            publish_frag(reinterpret_cast<uint4 *>(scr + SC::oU) + w * 128, fr, lane);
            if (lane == 0) {
                scal[(slot * NCW + w) * 4] = isv;
                scal[(slot * NCW + w) * 4 + 1] = iu;
            }
        }
        if (update)
            state_update<DK>(sr, si, fr, iu * inv[1], tile + TL::oY, reinterpret_cast<const float4 *>(smem + slot * TL::bytes + TL::oG), lane);
    };

    for (int c = 0; c < nch; ++c) {
        if (c % kSegChunks == 0) store_state<KT>(checkpoint(c / kSegChunks), sr, si, lane);
        forward_chunk(c % kSlots, c * kC, std::false_type{}, true);
        bar_arrive(kBarDone + c % kSlots, kAll);
    }

    float gr[KT][4], gi[KT][4];
    for (int r = 0; r < NS; ++r) {
        const int s = NS - 1 - r, nc = r == 0 ? last_nch : kSegChunks, p0 = r == 0 ? 0 : last_nch + kSegChunks * (r - 1);
        // rowdot(conj S, G) at the segment's end, this warp's columns; G then waits where that state was kept
        {
            float2 *rg = reinterpret_cast<float2 *>(smem + L::rg) + ((r & 1) * NCW + w) * M;
            if (r == 0) {
#pragma unroll
                for (int n = 0; n < KT; ++n)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        gr[n][i] = a.dS_T ? a.dS_T[state_at(n, i)] : 0.f;
                        gi[n][i] = a.dS_T ? a.dS_T[state_at(n, i) + DVT] : 0.f;
                    }
            } else {
                load_state<KT>(checkpoint(s + 1), sr, si, lane);
            }
#pragma unroll
            for (int n = 0; n < KT; ++n)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    float x = sr[n][e] * gr[n][e] + si[n][e] * gi[n][e] + sr[n][e + 2] * gr[n][e + 2] + si[n][e + 2] * gi[n][e + 2];
                    float y = sr[n][e] * gi[n][e] - si[n][e] * gr[n][e] + sr[n][e + 2] * gi[n][e + 2] - si[n][e + 2] * gr[n][e + 2];
#pragma unroll
                    for (int d = 4; d < 32; d <<= 1) {
                        x += __shfl_xor_sync(0xffffffffu, x, d);
                        y += __shfl_xor_sync(0xffffffffu, y, d);
                    }
                    if (g == 0) rg[8 * n + 2 * t4 + e] = make_float2(x, y);
                }
            if (r > 0) store_state<KT>(checkpoint(s + 1), gr, gi, lane);
        }
        load_state<KT>(checkpoint(s), sr, si, lane);
        for (int c = 0; c < nc; ++c) {
            const int slot = ring_slot(r, c);
            if (p0 + c >= kSlots) bar_sync(kBarFree + slot, kAll);
            forward_chunk(slot, s * kSeg + c * kC, std::true_type{}, c + 1 < nc);
        }
        if (r == 0) {
#pragma unroll
            for (int n = 0; n < KT; ++n)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    gr[n][i] = a.dS_T ? a.dS_T[state_at(n, i)] : 0.f;
                    gi[n][i] = a.dS_T ? a.dS_T[state_at(n, i) + DVT] : 0.f;
                }
        } else {
            load_state<KT>(checkpoint(s + 1), gr, gi, lane);
        }
        for (int c = nc - 1; c >= 0; --c) {
            const int slot = ring_slot(r, c), t0 = s * kSeg + c * kC;
            unsigned char *scr = ring + (size_t)slot * SC::slot;
            const bool has_im = a.d_o_im != nullptr;
            float yr[2][4], yi[2][4];
            load_tokens(a.d_o, t0, 1.f, yr);
            load_tokens(a.d_o_im, t0, -1.f, yi);
            const uint32_t tile = base + slot * TL::bytes;
            const float *inv = reinterpret_cast<const float *>(smem + slot * TL::bytes + TL::oS);
            float ig;
            const float sg = scale_for(__reduce_max_sync(0xffffffffu, max(max_bits4(gr), max_bits4(gi))), ig);
            float acc[1][3][2][4];
            const uint32_t tiles[1] = {tile + TL::oY};
            product_over_keys<DK, 1, true>(acc, gr, gi, sg, tiles, lane, reinterpret_cast<uint4 *>(scr + SC::oG) + w * KT * 64);
            TokFrag fy, fp, fb;
            const float iy = make_frag(fy, yr, yi);
            float pr[2][4], pi[2][4];
            const float fg = ig * inv[1];
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    pr[n][i] = fg * acc[0][0][n][i];
                    pi[n][i] = fg * (acc[0][1][n][i] - acc[0][2][n][i]);
                }
            load_small<true>(fb, tile + TL::oA, lane);
            product_small_conj<kExact>(pr, pi, fy, fb, iy * inv[4], has_im);
            const float ip = make_frag(fp, pr, pi);
            load_small<true>(fb, tile + TL::oM, lane);
            product_small<true>(pr, pi, fp, fb, ip * inv[3]);
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int t = t0 + 8 * n + 2 * t4 + (i & 1);
                    if (t < a.T) st_val(static_cast<T *>(a.dv), (row0 + (size_t)t * a.H) * DVT + col + 8 * (i >> 1), pr[n][i]);
                }
            const float ib = make_frag(fp, pr, pi);
            publish_frag(reinterpret_cast<uint4 *>(scr + SC::oB) + w * 128, fp, lane);
            if (lane == 0) {
                scal[(slot * NCW + w) * 4 + 2] = ig;
                scal[(slot * NCW + w) * 4 + 3] = ib;
            }
            // G <- conj(gamma_C) G + Q^T Yb^* - W^T Bc
            const float fq = iy * inv[2], fw = ib * inv[0];
            const float4 *gamma = reinterpret_cast<const float4 *>(smem + slot * TL::bytes + TL::oG);
            const uint32_t at = tile + (uint32_t)(((lane & 7) + (((lane >> 3) & 1) << 3)) * TL::LDB + (lane >> 4) * 16);
#pragma unroll
            for (int np = 0; np < KT; np += 2) {
                uint32_t qrh[4], qrl[4], qih[4], qil[4], wrh[4], wrl[4], wih[4], wil[4];
                ldsm_t(qrh, at + TL::oQ + np * 16);
                ldsm_t(qrl, at + TL::oQ + np * 16 + TL::PL);
                ldsm_t(qih, at + TL::oQ + np * 16 + 2 * TL::PL);
                ldsm_t(qil, at + TL::oQ + np * 16 + 3 * TL::PL);
                ldsm_t(wrh, at + TL::oW + np * 16);
                ldsm_t(wrl, at + TL::oW + np * 16 + TL::PL);
                ldsm_t(wih, at + TL::oW + np * 16 + 2 * TL::PL);
                ldsm_t(wil, at + TL::oW + np * 16 + 3 * TL::PL);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int n = np + e;
                    float qr_[4] = {0.f, 0.f, 0.f, 0.f}, qn[4] = {0.f, 0.f, 0.f, 0.f}, qm[4] = {0.f, 0.f, 0.f, 0.f};
                    float wr_[4] = {0.f, 0.f, 0.f, 0.f}, wn[4] = {0.f, 0.f, 0.f, 0.f}, wm[4] = {0.f, 0.f, 0.f, 0.f};
                    mma3(wr_, fp.rh, fp.rl, wrh[2 * e], wrh[2 * e + 1], wrl[2 * e], wrl[2 * e + 1]);
                    mma3(wm, fp.ih, fp.il, wrh[2 * e], wrh[2 * e + 1], wrl[2 * e], wrl[2 * e + 1]);
                    mma3(wn, fp.ih, fp.il, wih[2 * e], wih[2 * e + 1], wil[2 * e], wil[2 * e + 1]);
                    mma3x<kExact>(qr_, fy.rh, fy.rl, qrh[2 * e], qrh[2 * e + 1], qrl[2 * e], qrl[2 * e + 1]);
                    mma3x<kExact>(qm, fy.rh, fy.rl, qih[2 * e], qih[2 * e + 1], qil[2 * e], qil[2 * e + 1]);
                    mma3(wm, fp.rh, fp.rl, wih[2 * e], wih[2 * e + 1], wil[2 * e], wil[2 * e + 1]);
                    if (has_im) {
                        mma3x<kExact>(qn, fy.ih, fy.il, qih[2 * e], qih[2 * e + 1], qil[2 * e], qil[2 * e + 1]);
                        mma3x<kExact>(qm, fy.ih, fy.il, qrh[2 * e], qrh[2 * e + 1], qrl[2 * e], qrl[2 * e + 1]);
                    }
                    const float4 gm = gamma[4 * n + t4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float cr = (i & 1) ? gm.z : gm.x, ci = (i & 1) ? gm.w : gm.y, x = gr[n][i], y = gi[n][i];
                        gr[n][i] = fmaf(fq, qr_[i] - qn[i], fmaf(-fw, wr_[i] - wn[i], cr * x + ci * y));
                        gi[n][i] = fmaf(fq, qm[i], fmaf(-fw, wm[i], cr * y - ci * x));
                    }
                }
            }
            bar_arrive(kBarDone + slot, kAll);
        }
    }
#pragma unroll
    for (int n = 0; n < KT; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            a.dS0[state_at(n, i)] = gr[n][i];
            a.dS0[state_at(n, i) + DVT] = gi[n][i];
        }
}

// ---- the sums over the column blocks: out[i] = share_0[i] + share_1[i] + ... in that order, one thread per four
// consecutive elements.  HBM-bound and small beside the sweeps.
constexpr int kSumThreads = 256;

template <int NSL, typename T>
__global__ void __launch_bounds__(kSumThreads)
sfda_backward_sum_kernel(const float *__restrict__ dq_p, const float *__restrict__ dk_p, const float *__restrict__ dal_p,
                         const float *__restrict__ dth_p, const float *__restrict__ dbe_p, T *__restrict__ dq,
                         T *__restrict__ dk, float *__restrict__ dalpha, float *__restrict__ dtheta,
                         float *__restrict__ dbeta, size_t n_key, size_t n_coord, size_t rows)
{
    // work items in float4 units: [dq | dk | dalpha | dtheta] then dbeta one by one
    const size_t q4 = n_key / 4, c4 = n_coord / 4, total = 2 * q4 + 2 * c4 + rows;
    for (size_t i = (size_t)blockIdx.x * kSumThreads + threadIdx.x; i < total; i += (size_t)gridDim.x * kSumThreads) {
        if (i < 2 * q4 + 2 * c4) {
            const float *src;
            size_t n, at;
            int which;
            if (i < q4) { src = dq_p; n = n_key; at = i; which = 0; }
            else if (i < 2 * q4) { src = dk_p; n = n_key; at = i - q4; which = 1; }
            else if (i < 2 * q4 + c4) { src = dal_p; n = n_coord; at = i - 2 * q4; which = 2; }
            else { src = dth_p; n = n_coord; at = i - 2 * q4 - c4; which = 3; }
            float4 acc = *reinterpret_cast<const float4 *>(src + 4 * at);
#pragma unroll
            for (int sl = 1; sl < NSL; ++sl) {
                const float4 x = *reinterpret_cast<const float4 *>(src + (size_t)sl * n + 4 * at);
                acc.x += x.x; acc.y += x.y; acc.z += x.z; acc.w += x.w;
            }
            if (which >= 2) {
                *reinterpret_cast<float4 *>((which == 2 ? dalpha : dtheta) + 4 * at) = acc;
            } else {
                st_val4((which == 0 ? dq : dk) + 4 * at, acc);
            }
        } else {
            const size_t at = i - 2 * q4 - 2 * c4;
            float acc = dbe_p[at];
#pragma unroll
            for (int sl = 1; sl < NSL; ++sl) acc += dbe_p[(size_t)sl * rows + at];
            dbeta[at] = acc;
        }
    }
}

// Value columns per CTA: all of them while the (batch, head) pairs alone fill the SMs; halved (down to 32) while the
// grid still fits the SMs of a B200, so that few sequences use the whole device.  (A fixed count rather than the
// device's: the workspace size must not depend on where it is asked for.)
constexpr int kBwdTargetCtas = 148;

int bwd_cols(int B, int H, int d_v)
{
    int cols = d_v;
    while (cols > 32 && (long long)B * H * (d_v / (cols / 2)) <= kBwdTargetCtas) cols /= 2;
    return cols;
}

// workspace: checkpoints, the S_{t-1} of one segment, then (more than one column block only) the blocks' shares of
// dq, dk, dalpha, dtheta, dbeta
struct BwdWorkspace {
    size_t check, scratch, dq, dk, dalpha, dtheta, dbeta, total;   // offsets and size in floats
};

BwdWorkspace bwd_workspace(int B, int T, int H, int d_k, int d_v)
{
    const size_t bhn = (size_t)B * H, ns = (size_t)(T + kSeg - 1) / kSeg, state = (size_t)d_k * d_v;
    const size_t rows = bhn * T, nsl = (size_t)(d_v / bwd_cols(B, H, d_v)), shares = nsl > 1 ? nsl * rows : 0;
    BwdWorkspace w;
    w.check = 0;
    w.scratch = w.check + bhn * ns * state;
    w.dq = w.scratch + bhn * kSeg * state;
    w.dk = w.dq + shares * d_k;
    w.dalpha = w.dk + shares * d_k;
    w.dtheta = w.dalpha + shares * (d_k / 2);
    w.dbeta = w.dtheta + shares * (d_k / 2);
    w.total = w.dbeta + ((shares + 3) & ~(size_t)3);
    return w;
}

template <int DK, int DVT, int DV, typename T>
cudaError_t launch_cols(const BackwardArgs &x, void *workspace, cudaStream_t stream, int *launches)
{
    using L = BwdSmem<DK, DV>;
    constexpr int NSL = DVT / DV;
    auto kern = sfda_backward_kernel<DK, DVT, DV, T>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::bytes);
    if (e != cudaSuccess) return e;
    const BwdWorkspace w = bwd_workspace(x.B, x.T, x.H, DK, DVT);
    float *ws = static_cast<float *>(workspace);
    BwdArgsDev a;
    a.q = x.q; a.k = x.k; a.v = x.v; a.d_o = x.d_o; a.d_o_im = x.d_o_im;
    a.alpha = x.alpha; a.theta = x.theta; a.beta = x.beta; a.S0 = x.S0; a.dS_T = x.dS_T;
    a.dq = x.dq; a.dk = x.dk; a.dv = x.dv; a.dalpha = x.dalpha; a.dtheta = x.dtheta; a.dbeta = x.dbeta; a.dS0 = x.dS0;
    a.T = x.T; a.H = x.H; a.NS = (x.T + kSeg - 1) / kSeg;
    const size_t bhn = (size_t)x.B * x.H;
    a.rows = bhn * x.T;
    a.check = ws + w.check; a.scratch = ws + w.scratch;
    a.dq_p = ws + w.dq; a.dk_p = ws + w.dk; a.dalpha_p = ws + w.dalpha; a.dtheta_p = ws + w.dtheta; a.dbeta_p = ws + w.dbeta;
    kern<<<dim3((unsigned)bhn, NSL), kAux + 2 * DV, L::bytes, stream>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (launches) ++*launches;
    if constexpr (NSL > 1) {
        const size_t n_key = a.rows * DK, n_coord = a.rows * (DK / 2);
        const size_t items = n_key / 2 + n_coord / 2 + a.rows;
        size_t blocks = (items + kSumThreads - 1) / kSumThreads;
        if (blocks > 148 * 8 * 8) blocks = 148 * 8 * 8;
        sfda_backward_sum_kernel<NSL, T><<<(unsigned)blocks, kSumThreads, 0, stream>>>(
            a.dq_p, a.dk_p, a.dalpha_p, a.dtheta_p, a.dbeta_p, static_cast<T *>(x.dq), static_cast<T *>(x.dk), x.dalpha,
            x.dtheta, x.dbeta, n_key, n_coord, a.rows);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (launches) ++*launches;
    }
    return cudaSuccess;
}

template <int DK, int DV, typename T>
cudaError_t launch_typed(const BackwardArgs &x, void *workspace, cudaStream_t stream, int *launches)
{
    const int cols = bwd_cols(x.B, x.H, DV);
    if (cols == DV) return launch_cols<DK, DV, DV, T>(x, workspace, stream, launches);
    if constexpr (DV > 64) {
        if (cols == 64) return launch_cols<DK, DV, 64, T>(x, workspace, stream, launches);
    }
    return launch_cols<DK, DV, 32, T>(x, workspace, stream, launches);
}

}  // namespace

size_t backward_workspace_bytes(int B, int T, int H, int d_k, int d_v)
{
    return bwd_workspace(B, T, H, d_k, d_v).total * sizeof(float);
}

cudaError_t launch_backward(const BackwardArgs &a, void *workspace, cudaStream_t stream, int *launches)
{
    cudaError_t e = cudaErrorInvalidValue;
    if (a.dtype == 1) {
        if (a.d_k == 128 && a.d_v == 128) e = launch_typed<128, 128, __nv_bfloat16>(a, workspace, stream, launches);
        else if (a.d_k == 128 && a.d_v == 64) e = launch_typed<128, 64, __nv_bfloat16>(a, workspace, stream, launches);
        else if (a.d_k == 64 && a.d_v == 128) e = launch_typed<64, 128, __nv_bfloat16>(a, workspace, stream, launches);
        else if (a.d_k == 64 && a.d_v == 64) e = launch_typed<64, 64, __nv_bfloat16>(a, workspace, stream, launches);
    } else {
        if (a.d_k == 128 && a.d_v == 128) e = launch_typed<128, 128, float>(a, workspace, stream, launches);
        else if (a.d_k == 128 && a.d_v == 64) e = launch_typed<128, 64, float>(a, workspace, stream, launches);
        else if (a.d_k == 64 && a.d_v == 128) e = launch_typed<64, 128, float>(a, workspace, stream, launches);
        else if (a.d_k == 64 && a.d_v == 64) e = launch_typed<64, 64, float>(a, workspace, stream, launches);
    }
    return e;
}

}  // namespace sfda
