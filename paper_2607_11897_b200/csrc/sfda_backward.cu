// sfda_backward: reverse-mode derivative of the recurrence of Section 3 (Eq. "sfda") with o_t = S_t^* q_t, chunk by
// chunk (16 tokens) at fp32 precision on the tensor cores.  (The paper asks for the backward pass only as something to
// be timed, App. E; what it computes is the adjoint of Eq. "sfda".)  Complex cotangents Xb mean dL = Re sum conj(Xb) dX,
// i.e. the ordinary gradient with respect to the (Re, Im) pair; yb_t = do_re + i do_im.
//
// Per chunk, with W, Y, Q, M, A^{qk} of sfda_chunk16.cuh, S_0 the state before the chunk and G_C the cotangent of the
// state after it:
//
//   forward    U = M (V - W^* S_0)  (rows u_t^T = v_t^T - k_t^* Lambda_t S_{t-1}),   S_C = gamma_C S_0 + Y U
//   backward   Bc = M^H (Y^* G_C + (A^{qk} D_beta)^H Yb^*)   (rows beta_t p_t^*, p_t = G_t^* k_t),   dv_t = Re Bc_t
//              G_0 = conj(gamma_C) G_C + Q^T Yb^* - W^T Bc
//   gradients  dq_t = S_t yb_t,   f_t = G_t conj(u_t),   z_t = Lambda_t S_{t-1} (beta_t p_t),
//              dk_t = beta_t f_t - z_t,   dbeta_t = Re(f_t^* k_t),
//              D_t = D_{t+1} + q_t conj(dq_t) - beta_t conj(k_t) f_t - k_t conj(z_t)    (behind a chunk: rowdot(S_C, G_C)),
//              dalpha_t = Re D_t / alpha_t,   dtheta_t = Im D_t
//
// where S_t, G_t inside a chunk are S_0, G_C plus rank-16 corrections, so dq, f, z come from three products with the
// boundary matrices (S_0 Yb^T, S_0 B^T, G_C U^H), two 16 x 16 matrices U Yb^T, U B^T and triangular products with the
// decayed keys and queries.  Where alpha_t < 1/16 the division would lose digits: dalpha comes from its definition,
// sum_c conj(S_{t-1,jc}) Zb_jc, written out over the chunk's own products (from_definition).  D is made anew behind every
// chunk from sum_c conj(S_0) G_C: it runs over at most 16 tokens (over 64: dalpha 5.4e-7 from 64 bits instead of 3.3e-7).
//
// A (batch, head) pair is walked forward once, keeping the state every 64 tokens, then per segment of 64 tokens, last to
// first: forward again from the kept state, backward through it; the walks of all pairs are cut into one equal piece per
// SM.  With few sequences the two chains run by themselves first, in blocks of value columns, and every segment is then a
// unit of its own.  The CHAIN warps leave S_0, U, G_C, Bc of a chunk in a scratch ring as the operand registers of the
// gradients' products.  PREP warps prepare the chunks' operand tiles and stage what the gradients need of the tokens;
// GRAD warps turn all that into gradients one chunk behind the chain.  They meet at hardware barriers, one per slot: FULL
// (a tile is complete), DONE (the chain came back through the chunk); READY (the gradients are through with the slot),
// STAGED and TAKEN (the tokens are there, and free again).  In the units also at two barriers in shared memory, one per place
// of G_C: GFREE (the place is free again).
//
// What bounds it: about 60 k cycles per 16 tokens of a pair at d_k = d_v = 128 (57 k, 12.6 k of them in the first sweep, with
// mma.sync holding 29 % of the tensor pipe's time and issue slots 33 % used, before sums over the keys were rounded to
// nearest and channels had scales of their own): the latency of the two chains under roles that share the schedulers.
// Training step on raw inputs, B = 8, T = 8192, H = 32, bf16: 28.3 ms (the token-level adjoint on the CUDA cores: 148 ms);
// B = 4, T = 4096, H = 16: 4.2 ms (21.8).
#include "sfda_chunk16.cuh"
#include "sfda_internal.h"

namespace sfda {
namespace {

using namespace c16;

constexpr int kSeg = 64;                    // tokens between checkpoints
constexpr int kSegChunks = kSeg / kC;
static_assert(kSegChunks == kSlots, "a segment's operand tiles fill the ring");
constexpr int kGradWarps = 8, kGrad = 32 * kGradWarps, kPrepWarps = 8, kPrep = 32 * kPrepWarps;   // of the walk with gradients
constexpr int kBarGrad = kBarAux, kBarPrep = 14, kBarReady = 10, kBarTaken = 12, kBarStaged = 13, kBarTri = 15;   // READY: + parity

struct BwdArgsDev {
    const void *q, *k, *v, *d_o, *d_o_im;
    const float *alpha, *theta, *beta, *S0, *dS_T;
    void *dq, *dk, *dv;
    float *dalpha, *dtheta, *dbeta, *dS0;
    // kept states: S at the start of segment s of pair bh at keep_s + (bh * pitch + s) * d_k * d_v, the final state in the
    // place after the last; G at the end of segment s likewise at keep_g (few sequences only)
    float *keep_s, *keep_g;
    unsigned char *ring;      // the CTAs' scratch rings, ring_bytes apart
    size_t ring_bytes;
    int T, H, NS, pitch, units;
    long long work;           // of all pairs' walks, in the units of walk_cut
    unsigned *status;         // first word of the workspace: 1 where a wait ran out
    unsigned *flags;          // per CTA of the walk: the piece it hands on is written (null where none is); of the chains: a wait ran out
    int chain_ctas;           // CTAs of the chains that write such a flag
    unsigned long long wait_ticks;   // SM-clock ticks after which a wait gives up
    int withhold;             // diagnostic: pieces are never announced
};

// The head of the workspace: the status word and, 256 bytes behind it, the flags of at most kBwdTargetCtas CTAs.
constexpr int kBwdTargetCtas = 148;
constexpr size_t kHeadBytes = 1024;
constexpr unsigned long long kChunkTicks = 1ull << 22;           // more than any chunk takes
static_assert(256 + kBwdTargetCtas * sizeof(unsigned) <= kHeadBytes, "the flags follow the status block");   // (the chains: at most 2 x 74)

// The scratch ring (global memory, one per CTA), all of it in the order of the consumer's registers.  A slot for every chunk
// of a segment: S_0 as B operand [chain warp][key tile][Re / Im][lane] uint4 (two heads, two tails); U as A operand [chain warp]
// [plane][lane] uint4; the chunk's decays and phases, 4 floats per (token, key).  Behind the slots slow_gram's scratch and four
// or two places in turn for G_C and Bc likewise.  With two the chain that comes back waits until the gradients have used up
// what lies there (GFREE); see ring_places.  The rotated keys and queries, which only the rare paths want, are made again there (Rotated):
// 704 KB (and 25 of slow_gram's scratch) with four places for d_k = d_v = 128 instead of 768, of which every chunk writes and reads 176 instead of 192.
// Training step at the headline sizes 29.5 -> 28.2 ms, B = 4, T = 4096, H = 16: 4.43 -> 4.29 ms.
template <int DK, int NB>
struct BwdScratch {
    static constexpr int NCW = NB / 16, KT = DK / 16, M = DK / 2;
    static constexpr int oS = 0, oU = oS + NCW * KT * 1024, oV = oU + NCW * 2048, slot = oV + 16 * M * 16;
    static constexpr int oSlow = slot * kSlots, oG = (oSlow + PrepMap<DK, kPrepWarps>::slow_bytes + 255) / 256 * 256;
    static constexpr int oB = oG + NCW * KT * 1024, place = NCW * KT * 1024 + NCW * 2048;
    static constexpr size_t bytes(int places) { return (size_t)oG + (size_t)places * place; }
    static_assert(place % 256 == 0 && kHeadBytes + bytes(4) + DK * NB * 4 <= (size_t)kSeg * DK * NB * 4, "head, ring and final state must fit a pair's scratch");
};
// Two for the units: B = 2, T = 333, H = 4, d = 64 has 48 segments, for which the workspace has room for 59 rings (47 with four places, 41 before; one
// round instead of two, 187 -> 158 us), and B = 4, T = 4096, H = 16 has its rings in 80 MB of L2 instead of 104 (4.29 -> 4.22 ms).
// Four for the walk, whose gradients have all of the way forward to catch up in: 28.2 ms at the headline sizes, 28.8 with two.
constexpr int ring_places(bool units) { return units ? 2 : 4; }
// Which of the places chunk c of a segment has: they take turns in the order in which the chain comes back
__device__ __forceinline__ int back_place(int c, int places) { return (kSegChunks - 1 - c) & (places - 1); }

template <int DK, int NB>
struct BwdSmem {
    using PM = PrepMap<DK, kPrepWarps>;
    static constexpr int NCW = NB / 16, M = DK / 2;
    static constexpr int up(int x) { return (x + 127) / 128 * 128; }
    static constexpr int kb = kSlots * Tile<DK>::bytes;           // PREP: Kb planes,
    static constexpr int gram = kb + Tile<DK>::BIG;               // the two Gram matrices,
    static constexpr int scan = gram + 2 * 16 * 17 * 8;           // the scan's scratch
    static constexpr int frag = up(scan + PM::scan_bytes);        // GRAD: Yb, Bc, U of the chunk as A operands,
    static constexpr int uy = up(frag + 3 * NCW * 2048);          // U Yb^T, U B^T in two halves over the columns: float2 [2][2][16][17]
    static constexpr int uy_bytes = 4 * 16 * 17 * 8;
    static constexpr int tri = uy + uy_bytes;                     // the corrections' triangular factors: 4 x 4 uint4 [32]
    static constexpr int scal = tri + 4 * 4 * 512;                // inverse scales [slot][NCW] (S, U, G, B), [NCW] Yb, [4] tri
    static constexpr int db = scal + kSlots * NCW * 16 + 48;      // dbeta: [8][16] floats
    static constexpr int word = db + 8 * 16 * 4;                  // tensor-memory address
    static constexpr int job = word + 16;                         // the walk's current piece: pair, first and last position, gave up
    static constexpr int gfree = job + 16;                        // GFREE: two barriers in shared memory, and the flag of a wait that ran out
    static constexpr int bytes = gfree + 32;
    static_assert(bytes <= 232448, "shared memory");
    static constexpr int columns = (NB + 63) / 64 * DK < 32 ? 32 : (NB + 63) / 64 * DK;   // S and G
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

// the [value x token] operand as the A operand (token, value) of products over the value columns, at their
// shared scale, whose inverse is returned; NaN at the tokens `off`
__device__ __forceinline__ float publish_frag(uint4 *p, const TokFrag &f, const RowScale &r, bool odd, uint32_t off, int lane)
{
    bool own;
    const float all = shared_scale(r, own);                      // (nearly always some row has another)
    auto put = [&](int plane, const uint32_t(&v)[4]) {
        uint32_t x[4] = {v[0], v[1], v[2], v[3]};
        to_shared_scale(x, r, all);
        if (plane == 0 && odd) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t m = off >> (8 * (i >> 1) + 2 * (lane & 3) + 16 * (i & 1));
                x[i] |= (m & 1 ? 0x7e00u : 0u) | (m & 2 ? 0x7e000000u : 0u);
            }
        }
        p[plane * 32 + lane] = make_uint4(transpose8x8(x[0]), transpose8x8(x[2]), transpose8x8(x[1]), transpose8x8(x[3]));
    };
    put(0, f.rh);
    put(1, f.rl);
    put(2, f.ih);
    put(3, f.il);
    return all;
}

// Gradients and kept states pass through L2 first to go (4.30 -> 4.25 ms for the training step at B = 4, T = 4096, H = 16): the rings
// want to stay in it.
__device__ __forceinline__ void st_val4(float *p, float4 x) { __stcs(reinterpret_cast<float4 *>(p), x); }
__device__ __forceinline__ void st_val4(__nv_bfloat16 *p, float4 x)
{
    const __nv_bfloat162 lo = __floats2bfloat162_rn(x.x, x.y), hi = __floats2bfloat162_rn(x.z, x.w);
    __stcs(reinterpret_cast<uint2 *>(p), make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi)));
}

__device__ __forceinline__ float2 cmul(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) { return make_float2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x); }   // conj(a) b

// ---- the gradients where decays are too strong to divide by, or alpha too small -----------------------------
// The rotated keys and queries (k'_t, q'_t) of a warp's eight keys, as PREP made them: from the caller's arrays and the phases in
// `vals`; zero behind the sequence and where PREP took a token out (`out`, see Tile).  They lie where the warp has read its key
// tile of S_0: tokens 0-7 in the first chain warp's kilobyte, 8-15 in the second's.  Made again at each use, element
// by element in the loops below, they cost a quarter: 200 sequences of 1000 tokens with alpha ~ U(0, 1) 14.2 ms, 10.9 ms so (11.3
// when PREP wrote them for every chunk), a not finite token in each 9.8 and 8.4 (8.3); 148 of 333 with alpha = 0.01 3.31 and 2.60 (2.65).
template <int DK>
struct Rotated {
    float4 *at;
    __device__ __forceinline__ float4 &operator()(int t, int key) const { return at[(t >> 3) * Tile<DK>::KT * 64 + (t & 7) * 8 + (key & 7)]; }
    template <typename T>
    __device__ __forceinline__ void make(const BwdArgsDev &a, const float4 *vals, size_t row0, int t0, uint32_t out, int warp, int lane) const
    {
#pragma unroll 1
        for (int i = lane; i < 128; i += 32) {
            const int t = i >> 3, key = 8 * warp + (i & 7);
            const size_t x = (row0 + (size_t)(t0 + t) * a.H) * DK + 2 * key;
            const bool on = t0 + t < a.T;
            const float4 v = vals[t * (DK / 2) + key];           // -, -, cos, sin
            float2 k = make_float2(0.f, 0.f), q = k;
            if (on && !(out >> t & 1)) k = make_float2(ld_val(static_cast<const T *>(a.k), x), ld_val(static_cast<const T *>(a.k), x + 1));
            if (on && !(out >> (16 + t) & 1)) q = make_float2(ld_val(static_cast<const T *>(a.q), x), ld_val(static_cast<const T *>(a.q), x + 1));
            (*this)(t, key) = make_float4(k.x * v.z + k.y * v.w, k.y * v.z - k.x * v.w, q.x * v.z + q.y * v.w, q.y * v.z - q.x * v.w);
        }
        __syncwarp();
    }
};

// The corrections of one (token, key) where the decays are too strong to divide by: running products, token by token.
// uy: U Yb^T and U B^T (two halves each); x1, x2, x3: the products with the boundary matrices.
struct SlowOut {
    float2 qb, zb, fb;
};
template <int DK>
__device__ __forceinline__ SlowOut slow_corrections(const Rotated<DK> &rotated, const float2 *uy, const float *alpha, const float *beta,
                                                 size_t row0, int H, int t0, int T_, int tl, int key, float2 x1, float2 x2, float2 x3)
{
    auto at = [&](int mat, int i, int t) {
        const float2 x = uy[mat * 272 + i * 17 + t], y = uy[544 + mat * 272 + i * 17 + t];
        return make_float2(x.x + y.x, x.y + y.y);
    };
    constexpr int M = DK / 2;
    SlowOut o;
    float w = 1.f;
    o.qb = o.zb = o.fb = make_float2(0.f, 0.f);
    for (int j = tl; j >= 0; --j) {
        const size_t rj = row0 + (size_t)(t0 + j) * H;
        const float4 kj = rotated(j, key);
        const float bj = t0 + j < T_ ? w * beta[rj] : 0.f;
        const float2 kk = make_float2(bj * kj.x, bj * kj.y);
        const float2 p = cmul(kk, at(0, j, tl)), s = cmul(kk, at(1, j, tl));
        o.qb = make_float2(o.qb.x + p.x, o.qb.y + p.y);
        if (j < tl) o.zb = make_float2(o.zb.x + s.x, o.zb.y + s.y);
        w *= t0 + j < T_ ? alpha[rj * M + key] : 1.f;
    }
    o.qb = make_float2(fmaf(w, x1.x, o.qb.x), fmaf(w, x1.y, o.qb.y));
    o.zb = make_float2(fmaf(w, x2.x, o.zb.x), fmaf(w, x2.y, o.zb.y));
    w = 1.f;
    for (int l = tl; l < 16; ++l) {
        const float4 kl = rotated(l, key);
        const float2 p = cmulc(at(0, tl, l), make_float2(w * kl.z, w * kl.w));
        o.fb = make_float2(o.fb.x + p.x, o.fb.y + p.y);
        if (l > tl) {
            const float2 s = cmulc(at(1, tl, l), make_float2(w * kl.x, w * kl.y));
            o.fb = make_float2(o.fb.x - s.x, o.fb.y - s.y);
        }
        if (l < 15 && t0 + l + 1 < T_) w *= alpha[(row0 + (size_t)(t0 + l + 1) * H) * M + key];
    }
    o.fb = make_float2(fmaf(w, x3.x, o.fb.x), fmaf(w, x3.y, o.fb.y));
    return o;
}

// dalpha and dtheta from their definition instead of from D, by a warp for the keys of its tile:  Re H and alpha Im H with
// H = sum_c conj(S'_c) Z'_c over the value columns, where e^{i phi_{t-1}} S' is the state before token t and e^{i phi_t} Z'
// the cotangent of Lambda_t S_{t-1}.  Written out over S_0, the tokens before t, G_C and the tokens from t on, every sum
// over the columns is one that the chunk's products have already made (X1, X2, X3 before they are corrected, U Yb^T, U B^T)
// or r0 = sum_c conj(S_0) G_C; decays come as running products.  x: the thread's tokens g, g + 8 and keys 2 t4, + 1.
// redo: bit 2 r + e says that this element is wanted; it goes to the caller's arrays.
// (Rebuilding both matrices per element, column by column, took 6.4 M cycles a chunk where every alpha is small.)
template <int DK>
__device__ __forceinline__ void from_definition(const BwdArgsDev &a, const Rotated<DK> &rotated, const float4 *vals, const float2 *uy, const float2 (&r0)[2],
                                                const float (&x1r)[4], const float (&x1i)[4], const float (&x2r)[4], const float (&x2i)[4],
                                                const float (&x3r)[4], const float (&x3i)[4], unsigned redo, size_t row0, int t0, int kt, int lane)
{
    constexpr int M = DK / 2;
    const int g = lane >> 2, t4 = lane & 3, key = 8 * kt + 2 * t4, left = a.T - t0;
    // an element (token, key 2 t4 + e) of another thread's tile
    auto other = [&](const float(&re)[4], const float(&im)[4], int t, int e) {
        const int src = 4 * (t & 7) + t4;
        const float u = t < 8 ? re[e] : re[2 + e], v = t < 8 ? im[e] : im[2 + e];
        return make_float2(__shfl_sync(0xffffffffu, u, src), __shfl_sync(0xffffffffu, v, src));
    };
    float2 wt[16][2];
#pragma unroll 1
    for (int r = 0; r < 2; ++r) {
        const int t = g + 8 * r;
        float pw[2] = {1.f, 1.f}, pz[2] = {1.f, 1.f};
        float2 h[2], sx[2], su[2];                                // with S_0, with G_C and u_i, with u_i and the tokens from t on
#pragma unroll
        for (int e = 0; e < 2; ++e) h[e] = sx[e] = su[e] = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int i = 14; i >= 0; --i) {                           // prod alpha behind i up to t - 1, beta_i conj(k'_i)
            const float2 x3[2] = {other(x3r, x3i, i, 0), other(x3r, x3i, i, 1)};
            if (i >= t || i >= left) continue;
            const size_t row = row0 + (size_t)(t0 + i) * a.H;
            const float be = a.beta[row];
            const float2 al = *reinterpret_cast<const float2 *>(a.alpha + row * M + key);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float4 v = rotated(i, key + e);
                const float2 w = make_float2(pw[e] * be * v.x, -pw[e] * be * v.y), p = cmul(w, x3[e]);
                wt[i][e] = w;
                sx[e] = make_float2(sx[e].x + p.x, sx[e].y + p.y);
                pw[e] *= e ? al.y : al.x;
            }
        }
#pragma unroll 1
        for (int l = 0; l < 16; ++l) {                            // prod alpha behind t up to l
            const float2 x1[2] = {other(x1r, x1i, l, 0), other(x1r, x1i, l, 1)}, x2[2] = {other(x2r, x2i, l, 0), other(x2r, x2i, l, 1)};
            if (l < t || l >= left) continue;
            if (l > t) {
                const float2 al = *reinterpret_cast<const float2 *>(a.alpha + (row0 + (size_t)(t0 + l) * a.H) * M + key);
                pz[0] *= al.x;
                pz[1] *= al.y;
            }
            float2 q[2], k[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float4 v = rotated(l, key + e);
                k[e] = make_float2(pz[e] * v.x, pz[e] * v.y);
                q[e] = make_float2(pz[e] * v.z, pz[e] * v.w);
                const float2 p = cmulc(x1[e], q[e]), m = cmulc(x2[e], k[e]);
                h[e] = make_float2(h[e].x + p.x - m.x, h[e].y + p.y - m.y);
            }
#pragma unroll 1
            for (int i = 0; i < t; ++i) {
                const float2 *u = uy + i * 17 + l;
                const float2 y = make_float2(u[0].x + u[544].x, u[0].y + u[544].y), b = make_float2(u[272].x + u[816].x, u[272].y + u[816].y);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float2 p = cmulc(y, q[e]), m = cmulc(b, k[e]), x = cmul(wt[i][e], make_float2(p.x - m.x, p.y - m.y));
                    su[e] = make_float2(su[e].x + x.x, su[e].y + x.y);
                }
            }
        }
        if (t >= left) continue;
        const size_t row = row0 + (size_t)(t0 + t) * a.H;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float4 v = vals[15 * M + key + e];               // -, -, e^{i phi_C}
            const float2 end = make_float2(pz[e] * v.z, -pz[e] * v.w), z0 = cmul(end, r0[e]), zx = cmul(end, sx[e]);
            const float hr = fmaf(pw[e], h[e].x + z0.x, su[e].x + zx.x), hi = fmaf(pw[e], h[e].y + z0.y, su[e].y + zx.y);
            if (redo >> (2 * r + e) & 1) {
                a.dalpha[row * M + key + e] = hr;
                a.dtheta[row * M + key + e] = a.alpha[row * M + key + e] * hi;
            }
        }
    }
}

// ---- PREP, second task: what the gradients of a chunk need of its tokens -----------------------------------
// Yb, Bc, U into shared memory (STAGED), U Yb^T and U B^T, and the triangular factors of the corrections (TRI).
template <int DK, int NB, typename T>
__device__ __forceinline__ void stage_tokens(const BwdArgsDev &a, unsigned char *smem, const unsigned char *ring, int slot, int place, int t0, size_t row0, int tid)
{
    using L = BwdSmem<DK, NB>;
    using SC = BwdScratch<DK, NB>;
    constexpr int NCW = L::NCW;
    const int lane = tid & 31, warp = tid >> 5, g = lane >> 2, t4 = lane & 3;
    const bool has_im = a.d_o_im != nullptr;
    uint4 *frag = reinterpret_cast<uint4 *>(smem + L::frag);                      // [Yb, Bc, U][NCW][4][32]
    uint4 *tri = reinterpret_cast<uint4 *>(smem + L::tri);
    float2 *uy = reinterpret_cast<float2 *>(smem + L::uy);
    float *scal = reinterpret_cast<float *>(smem + L::scal), *yscal = scal + kSlots * NCW * 4, *tscal = yscal + 8;
    const float *sc = scal + slot * NCW * 4;

    // operands over the value columns: Yb from the caller's arrays, Bc and U from the ring
    if (warp < NCW) {
        const int w = warp;
        const uint4 *pB = reinterpret_cast<const uint4 *>(ring + SC::oB + place * SC::place) + w * 128 + lane;
        const uint4 *pU = reinterpret_cast<const uint4 *>(ring + slot * SC::slot + SC::oU) + w * 128 + lane;
        uint4 x[8];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            x[p] = pB[p * 32];
            x[4 + p] = pU[p * 32];
        }
        float2 y[2][4];
        float m = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int t = t0 + g + 8 * (i & 1);
            y[0][i] = y[1][i] = make_float2(0.f, 0.f);
            if (t < a.T) {
                const size_t at = (row0 + (size_t)t * a.H) * NB + 16 * w + 2 * t4 + 8 * (i >> 1);
                y[0][i] = make_float2(ld_val(static_cast<const T *>(a.d_o), at), ld_val(static_cast<const T *>(a.d_o), at + 1));
                if (has_im) y[1][i] = make_float2(ld_val(static_cast<const T *>(a.d_o_im), at), ld_val(static_cast<const T *>(a.d_o_im), at + 1));
            }
            m = fmaxf(fmaxf(m, fmaxf(fabsf(y[0][i].x), fabsf(y[0][i].y))), fmaxf(fabsf(y[1][i].x), fabsf(y[1][i].y)));
        }
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            frag[((NCW + w) * 4 + p) * 32 + lane] = x[p];
            frag[((2 * NCW + w) * 4 + p) * 32 + lane] = x[4 + p];
        }
        if (__any_sync(0xffffffffu, m > 3.402823466e38f)) {              // an infinity does not decide the others' scale
            m = 0.f;
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float ax = fabsf(y[c][i].x), ay = fabsf(y[c][i].y);
                    m = fmaxf(m, fmaxf(ax <= 3.402823466e38f ? ax : 0.f, ay <= 3.402823466e38f ? ay : 0.f));
                }
        }
        float inv;
        const float s = scale_for(warp_max(m), inv);
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
    bar_sync(kBarPrep, kPrep);
    bar_arrive(kBarStaged, kPrep + kGrad);

    // U Yb^T (index [i][t]: u_i . yb_t) and U B^T (b_t = beta_t p_t = conj of the rows of Bc): warp = (matrix, half of
    // the tokens t, half of the value columns); the A-operand registers of tokens 0-7 / 8-15 are that half's B operand
    {
        const int mat = warp & 1, nt = (warp >> 1) & 1, wh = warp >> 2;
        float re[4] = {0.f, 0.f, 0.f, 0.f}, im[4] = {0.f, 0.f, 0.f, 0.f};
        const float sg = mat ? 1.f : -1.f;
#pragma unroll 1
        for (int w = wh; w < NCW; w += 2) {
            const uint4 *fu = frag + (2 * NCW + w) * 128 + lane, *fx = frag + (mat * NCW + w) * 128 + lane;
            const uint4 u0 = fu[0], u1 = fu[32], u2 = fu[64], u3 = fu[96], x0 = fx[0], x1 = fx[32], x2 = fx[64], x3 = fx[96];
            const uint32_t rh[4] = {u0.x, u0.y, u0.z, u0.w}, rl[4] = {u1.x, u1.y, u1.z, u1.w};
            const uint32_t ih[4] = {u2.x, u2.y, u2.z, u2.w}, il[4] = {u3.x, u3.y, u3.z, u3.w};
            const uint32_t xr[2] = {nt ? x0.y : x0.x, nt ? x0.w : x0.z}, xrl[2] = {nt ? x1.y : x1.x, nt ? x1.w : x1.z};
            const uint32_t xi[2] = {nt ? x2.y : x2.x, nt ? x2.w : x2.z}, xil[2] = {nt ? x3.y : x3.x, nt ? x3.w : x3.z};
            float rr[4], ii[4], ri[4], ir[4];
            mma_f16_z(rr, rl, xr[0], xr[1]);
            mma_f16_z(ii, il, xi[0], xi[1]);
            mma_f16_z(ri, rl, xi[0], xi[1]);
            mma_f16_z(ir, il, xr[0], xr[1]);
            mma_f16(rr, rh, xrl[0], xrl[1]);
            mma_f16(ii, ih, xil[0], xil[1]);
            mma_f16(ri, rh, xil[0], xil[1]);
            mma_f16(ir, ih, xrl[0], xrl[1]);
            mma_f16(rr, rh, xr[0], xr[1]);
            mma_f16(ii, ih, xi[0], xi[1]);
            mma_f16(ri, rh, xi[0], xi[1]);
            mma_f16(ir, ih, xr[0], xr[1]);
            const float f = sc[4 * w + 1] * (mat ? sc[4 * w + 3] : yscal[w]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                re[i] = fmaf(f, fmaf(sg, ii[i], rr[i]), re[i]);
                im[i] = fmaf(f, fmaf(-sg, ri[i], ir[i]), im[i]);
            }
        }
        float2 *dst = uy + (wh * 2 + mat) * 272 + g * 17 + 8 * nt + 2 * t4;
        dst[0] = make_float2(re[0], im[0]);
        dst[1] = make_float2(re[1], im[1]);
        dst[8 * 17] = make_float2(re[2], im[2]);
        dst[8 * 17 + 1] = make_float2(re[3], im[3]);
    }

    bar_sync(kBarPrep, kPrep);

    // the triangular factors of the corrections as A operands (t, i), a warp each:
    //   0: u_i . yb_t (i <= t)   1: u_i . b_t (i < t)   2: conj(u_t . yb_i) (i >= t)   3: -conj(u_t . b_i) (i > t)
    if (warp < 4) {
        float2 x[4][2];
        float m = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int t = g + 8 * (e & 1), i = 2 * t4 + 8 * (e >> 1) + j;
                const float2 *p = uy + (warp & 1) * 272 + (warp < 2 ? i * 17 + t : t * 17 + i);
                const bool on = (warp & 1) ? (warp < 2 ? i < t : i > t) : (warp < 2 ? i <= t : i >= t);
                const float2 u = p[0], v = p[544];
                const float sr = warp == 3 ? -1.f : 1.f, si = warp == 2 ? -1.f : 1.f;
                x[e][j] = on ? make_float2(sr * (u.x + v.x), si * (u.y + v.y)) : make_float2(0.f, 0.f);
                m = fmaxf(m, fmaxf(fabsf(x[e][j].x), fabsf(x[e][j].y)));
            }
        float inv;
        const float s = scale_for(warp_max(m), inv);
        if (lane == 0) tscal[warp] = inv;
        uint32_t h[4], l[4];
        uint4 *p = tri + warp * 128 + lane;
#pragma unroll
        for (int e = 0; e < 4; ++e) split_f16(x[e][0].x * s, x[e][1].x * s, h[e], l[e]);
        p[0] = make_uint4(h[0], h[1], h[2], h[3]);
        p[32] = make_uint4(l[0], l[1], l[2], l[3]);
#pragma unroll
        for (int e = 0; e < 4; ++e) split_f16(x[e][0].y * s, x[e][1].y * s, h[e], l[e]);
        p[64] = make_uint4(h[0], h[1], h[2], h[3]);
        p[96] = make_uint4(l[0], l[1], l[2], l[3]);
    }
    bar_arrive(kBarTri, kPrep + kGrad);
}

// ---- GRAD: the gradients of one chunk -----------------------------------------------------------------
template <int DK, int NB, typename T>
__device__ __forceinline__ void chunk_gradients(const BwdArgsDev &a, unsigned char *smem, unsigned char *ring, int slot, int place, bool gfree, bool last_one, int t0,
                                                size_t row0, int tid)
{
    using L = BwdSmem<DK, NB>;
    using SC = BwdScratch<DK, NB>;
    using TL = Tile<DK>;
    constexpr int NCW = L::NCW, M = L::M, KT = M / 8;
    constexpr bool kExact = sizeof(T) == 2;
    const int lane = tid & 31, warp = tid >> 5, g = lane >> 2, t4 = lane & 3;
    const bool has_im = a.d_o_im != nullptr;
    uint4 *frag = reinterpret_cast<uint4 *>(smem + L::frag);                      // [Yb, Bc, U][NCW][4][32]
    uint4 *tri = reinterpret_cast<uint4 *>(smem + L::tri);
    float2 *uy = reinterpret_cast<float2 *>(smem + L::uy);
    float *scal = reinterpret_cast<float *>(smem + L::scal), *yscal = scal + kSlots * NCW * 4, *tscal = yscal + 8;
    const float *sc = scal + slot * NCW * 4;
    float *db = reinterpret_cast<float *>(smem + L::db);
    unsigned char *scr = ring + slot * SC::slot;
    const uint4 *pS = reinterpret_cast<const uint4 *>(scr + SC::oS), *pG = reinterpret_cast<const uint4 *>(ring + SC::oG + place * SC::place);
    const float4 *vals = reinterpret_cast<const float4 *>(scr + SC::oV);

    bar_sync(kBarStaged, kPrep + kGrad);

    // X1 = S_0 yb_t, X2 = S_0 b_t, X3 = G_C conj(u_t) for the keys of tile `warp` (accumulator layout: token g (+ 8),
    // keys 2 t4, + 1); every chain warp's 16 columns come with scales of their own
    float x1r[4] = {0.f, 0.f, 0.f, 0.f}, x1i[4] = {0.f, 0.f, 0.f, 0.f}, x2r[4] = {0.f, 0.f, 0.f, 0.f};
    float x2i[4] = {0.f, 0.f, 0.f, 0.f}, x3r[4] = {0.f, 0.f, 0.f, 0.f}, x3i[4] = {0.f, 0.f, 0.f, 0.f};
    float2 r0[2];
    if (warp < KT) {
        auto conj_product = [&](const uint4 *fx, const uint4 &b0, const uint4 &b1, float f, float (&xr)[4], float (&xi)[4]) {
            const uint4 h = fx[0], l = fx[32], h2 = fx[64], l2 = fx[96];
            const uint32_t rh[4] = {h.x, h.y, h.z, h.w}, rl[4] = {l.x, l.y, l.z, l.w};
            const uint32_t ih[4] = {h2.x, h2.y, h2.z, h2.w}, il[4] = {l2.x, l2.y, l2.z, l2.w};
            float pr[4], pi[4], qr[4], mi[4];
            mma_f16_z(pr, rl, b0.x, b0.y);
            mma_f16_z(pi, rl, b1.x, b1.y);
            mma_f16_z(mi, il, b0.x, b0.y);
            mma_f16_z(qr, il, b1.x, b1.y);
            mma_f16(pr, rh, b0.z, b0.w);
            mma_f16(pi, rh, b1.z, b1.w);
            mma_f16(mi, ih, b0.z, b0.w);
            mma_f16(qr, ih, b1.z, b1.w);
            mma_f16(pr, rh, b0.x, b0.y);
            mma_f16(pi, rh, b1.x, b1.y);
            mma_f16(mi, ih, b0.x, b0.y);
            mma_f16(qr, ih, b1.x, b1.y);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                xr[i] = fmaf(f, pr[i] + qr[i], xr[i]);
                xi[i] = fmaf(f, pi[i] - mi[i], xi[i]);
            }
        };
        // the ring's operands are requested a step ahead (more of them in registers cost more in spills than they hid)
        const uint4 *p = pS + warp * 64 + lane;
        uint4 n0 = p[0], n1 = p[32];
#pragma unroll 1
        for (int w = 0; w < NCW; ++w) {
            const uint4 s0 = n0, s1 = n1;
            p = w + 1 < NCW ? p + KT * 64 : pG + warp * 64 + lane;
            n0 = p[0];
            n1 = p[32];
            {
                const uint4 *fy = frag + w * 128 + lane;
                const uint4 h = fy[0], l = fy[32];
                const uint32_t ah[4] = {h.x, h.y, h.z, h.w}, al[4] = {l.x, l.y, l.z, l.w};
                float pr[4] = {0.f, 0.f, 0.f, 0.f}, pi[4] = {0.f, 0.f, 0.f, 0.f}, mr[4] = {0.f, 0.f, 0.f, 0.f}, mi[4] = {0.f, 0.f, 0.f, 0.f};
                mma3x<kExact>(pr, ah, al, s0.x, s0.y, s0.z, s0.w);
                mma3x<kExact>(pi, ah, al, s1.x, s1.y, s1.z, s1.w);
                if (has_im) {
                    const uint4 h2 = fy[64], l2 = fy[96];
                    const uint32_t bh[4] = {h2.x, h2.y, h2.z, h2.w}, bl[4] = {l2.x, l2.y, l2.z, l2.w};
                    mma3x<kExact>(mr, bh, bl, s1.x, s1.y, s1.z, s1.w);
                    mma3x<kExact>(mi, bh, bl, s0.x, s0.y, s0.z, s0.w);
                }
                const float f = sc[4 * w] * yscal[w];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    x1r[i] = fmaf(f, pr[i] - mr[i], x1r[i]);
                    x1i[i] = fmaf(f, pi[i] + mi[i], x1i[i]);
                }
            }
            conj_product(frag + (NCW + w) * 128 + lane, s0, s1, sc[4 * w] * sc[4 * w + 3], x2r, x2i);
        }
        // ... and sum_c conj(S_0) G_C: S with Re and Im in the rows, the diagonal of what that gives with Re G and Im G
        const uint4 *ps = pS + warp * 64 + lane;
        float sre[2] = {0.f, 0.f}, sim[2] = {0.f, 0.f};
#pragma unroll 1
        for (int w = 0; w < NCW; ++w, ps += KT * 64) {
            const uint4 g0 = n0, g1 = n1, s0 = ps[0], s1 = ps[32];
            if (w + 1 < NCW) {
                p += KT * 64;
                n0 = p[0];
                n1 = p[32];
            }
            conj_product(frag + (2 * NCW + w) * 128 + lane, g0, g1, sc[4 * w + 2] * sc[4 * w + 1], x3r, x3i);
            const uint32_t ah[4] = {s0.x, s1.x, s0.y, s1.y}, al[4] = {s0.z, s1.z, s0.w, s1.w};
            float d1[4] = {0.f, 0.f, 0.f, 0.f}, d2[4] = {0.f, 0.f, 0.f, 0.f};
            mma3x<false>(d1, ah, al, g0.x, g0.y, g0.z, g0.w);
            mma3x<false>(d2, ah, al, g1.x, g1.y, g1.z, g1.w);
            const float f = sc[4 * w] * sc[4 * w + 2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                sre[e] = fmaf(f, d1[e] + d2[2 + e], sre[e]);
                sim[e] = fmaf(f, d2[e] - d1[2 + e], sim[e]);
            }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int src = 4 * (2 * t4 + e) + t4;                 // row = column = 2 t4 + e
            r0[e] = make_float2(__shfl_sync(0xffffffffu, sre[e], src), __shfl_sync(0xffffffffu, sim[e], src));
        }
    }
    __syncwarp();
    if (gfree && lane == 0) mbar_arrive((uint32_t)__cvta_generic_to_shared(smem + L::gfree) + 8 * place);   // (Bc has been staged, G_C is in X3 and r0)
    // what the elements need besides, requested here: it comes from L2 and memory (prod alpha up to the token and after it)
    float2 va[4], al2[2];
    if (warp < KT) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int t = t0 + g + 8 * r;
            const float4 *p = vals + (g + 8 * r) * M + 8 * warp + 2 * t4;
            va[2 * r] = *reinterpret_cast<const float2 *>(p);
            va[2 * r + 1] = *reinterpret_cast<const float2 *>(p + 1);
            al2[r] = t < a.T ? *reinterpret_cast<const float2 *>(a.alpha + (row0 + (size_t)t * a.H) * M + 8 * warp + 2 * t4) : make_float2(1.f, 1.f);
        }
    }
    bar_sync(kBarTri, kPrep + kGrad);

    if (warp < KT) {
        // D behind the chunk, sum_c conj(S_C) G_C = conj(gamma_C) (sum_c conj(S_0) G_C) + sum_t conj(Y_t) X3_t
        float2 carry[2];
        {
            const unsigned char *py = smem + slot * TL::bytes + TL::oY + g * TL::LDB + 2 * (8 * warp + 2 * t4);
            float2 yr[2], yi[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                auto both = [&](int off) {
                    const uint32_t *h = reinterpret_cast<const uint32_t *>(py + 8 * r * TL::LDB + off);
                    const float2 x = unpack_f16(h[0]), y = unpack_f16(h[TL::PL / 4]);
                    return make_float2(x.x + y.x, x.y + y.y);
                };
                yr[r] = both(0);
                yi[r] = both(2 * TL::PL);
            }
            const float f = reinterpret_cast<const float *>(smem + slot * TL::bytes + TL::oS)[1];
            const float4 gm = reinterpret_cast<const float4 *>(smem + slot * TL::bytes + TL::oG)[4 * warp + t4];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float2 d = make_float2(0.f, 0.f);
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const float2 x = cmulc(e ? make_float2(yr[r].y, yi[r].y) : make_float2(yr[r].x, yi[r].x), make_float2(x3r[2 * r + e], x3i[2 * r + e]));
                    d = make_float2(d.x + x.x, d.y + x.y);
                }
#pragma unroll
                for (int i = 4; i < 32; i <<= 1) {
                    d.x += __shfl_xor_sync(0xffffffffu, d.x, i);
                    d.y += __shfl_xor_sync(0xffffffffu, d.y, i);
                }
                const float2 z = cmulc(e ? make_float2(gm.z, gm.w) : make_float2(gm.x, gm.y), r0[e]);
                carry[e] = make_float2(fmaf(f, d.x, z.x), fmaf(f, d.y, z.y));
            }
        }
        // D / alpha loses digits where alpha is small, and D takes up all that is not finite up to the chunk's end: those
        // elements come from the definition
        constexpr float kSmall = 0.0625f;
        unsigned redo = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float x = i & 1 ? al2[i >> 1].y : al2[i >> 1].x, d = (carry[i & 1].x + carry[i & 1].y) * 0.f;
            if (x < kSmall || d != 0.f) redo |= 1u << i;
        }
        const bool some = __any_sync(0xffffffffu, redo != 0);
        const float *inv = reinterpret_cast<const float *>(smem + slot * TL::bytes + TL::oS);
        const uint32_t out = reinterpret_cast<const uint32_t *>(inv)[7];
        const bool fast = reinterpret_cast<const int *>(inv)[6] != 0;
        const Rotated<DK> rotated = {reinterpret_cast<float4 *>(scr + SC::oS) + warp * 64};
        if (some || !fast) rotated.template make<T>(a, vals, row0, t0, out, warp, lane);
        if (some)
            from_definition<DK>(a, rotated, vals, uy, r0, x1r, x1i, x2r, x2i, x3r, x3i, redo, row0, t0, warp, lane);
        const unsigned char *slot_at = smem + slot * TL::bytes;
        // from here on x1, x2, x3 become S_t yb_t, Lambda_t S_{t-1} b_t, G_t conj(u_t) in the rotated frame
        if (fast) {
            // B operand: tokens as k, the warp's eight keys; heads in registers 0, 1 and tails in 2, 3
            const uint32_t tile = (uint32_t)__cvta_generic_to_shared(slot_at) + (uint32_t)((lane & 15) * TL::LDB + warp * 16 + (lane >> 4) * TL::PL);
            auto tri_product = [&](int sum, uint32_t at, float (&zr)[4], float (&zi)[4]) {
                const uint4 *p = tri + sum * 128 + lane;
                const uint4 h = p[0], l = p[32], h2 = p[64], l2 = p[96];
                const uint32_t rh[4] = {h.x, h.y, h.z, h.w}, rl[4] = {l.x, l.y, l.z, l.w};
                const uint32_t ih[4] = {h2.x, h2.y, h2.z, h2.w}, il[4] = {l2.x, l2.y, l2.z, l2.w};
                uint32_t br[4], bi[4];
                ldsm_t(br, tile + at);
                ldsm_t(bi, tile + at + 2 * TL::PL);
                float nr[4], ni[4];
                mma_f16_z(zr, rl, br[0], br[1]);
                mma_f16_z(zi, rl, bi[0], bi[1]);
                mma_f16_z(nr, il, bi[0], bi[1]);
                mma_f16_z(ni, il, br[0], br[1]);
                mma_f16(zr, rh, br[2], br[3]);
                mma_f16(zi, rh, bi[2], bi[3]);
                mma_f16(nr, ih, bi[2], bi[3]);
                mma_f16(ni, ih, br[2], br[3]);
                mma_f16(zr, rh, br[0], br[1]);
                mma_f16(zi, rh, bi[0], bi[1]);
                mma_f16(nr, ih, bi[0], bi[1]);
                mma_f16(ni, ih, br[0], br[1]);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    zr[i] -= nr[i];
                    zi[i] += ni[i];
                }
            };
            const float4 gm = reinterpret_cast<const float4 *>(slot_at + TL::oG)[4 * warp + t4];   // gamma_C of the two keys
            // 1 / |gamma_C|^2 and 1 / |gamma_C|, the latter with a Newton step (the instruction is good to 23 bits)
            const float n2[2] = {gm.x * gm.x + gm.y * gm.y, gm.z * gm.z + gm.w * gm.w};
            const float i2[2] = {__frcp_rn(n2[0]), __frcp_rn(n2[1])};
            float i1[2] = {rsqrtf(n2[0]), rsqrtf(n2[1])};
#pragma unroll
            for (int e = 0; e < 2; ++e) i1[e] = fmaf(0.5f * i1[e], fmaf(-n2[e] * i1[e], i1[e], 1.f), i1[e]);
            float zr[4], zi[4];
            // a_t (X + conj(gamma_C) Z / |gamma_C|^2), the scale f of Z included
            auto fold = [&](float f, float (&xr)[4], float (&xi)[4]) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int e = i & 1;
                    const float w = f * i2[e];
                    const float2 z = cmulc(e ? make_float2(gm.z, gm.w) : make_float2(gm.x, gm.y), make_float2(w * zr[i], w * zi[i]));
                    xr[i] = va[i].x * (xr[i] + z.x);
                    xi[i] = va[i].x * (xi[i] + z.y);
                }
            };
            tri_product(0, TL::oY, zr, zi);
            fold(tscal[0] * inv[1], x1r, x1i);
            tri_product(1, TL::oY, zr, zi);
            fold(tscal[1] * inv[1], x2r, x2i);
            float wr[4], wi[4];
            tri_product(2, TL::oQ, zr, zi);
            tri_product(3, TL::oW, wr, wi);
            const float f2 = tscal[2] * inv[2], f3 = tscal[3] * inv[0];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int e = i & 1;
                const float s = va[i].y * i1[e], down = __frcp_rn(va[i].x);      // 1 / a_t: at most 2^16
                const float2 z = cmulc(e ? make_float2(gm.z, gm.w) : make_float2(gm.x, gm.y), make_float2(x3r[i], x3i[i]));
                x3r[i] = fmaf(s, z.x, down * fmaf(f2, zr[i], f3 * wr[i]));
                x3i[i] = fmaf(s, z.y, down * fmaf(f2, zi[i], f3 * wi[i]));
            }
        } else {
#pragma unroll 1
            for (int i = 0; i < 4; ++i) {                          // (no function and no indexed registers: both cost the common path)
                auto pick = [&](const float(&v)[4]) { return i == 0 ? v[0] : i == 1 ? v[1] : i == 2 ? v[2] : v[3]; };
                auto put = [&](float(&v)[4], float x) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) v[j] = i == j ? x : v[j];
                };
                const int tl = g + 8 * (i >> 1), key = 8 * warp + 2 * t4 + (i & 1);
                const float4 lv = vals[15 * M + key];              // -, -, e^{i phi_C}
                const SlowOut o = slow_corrections<DK>(rotated, uy, a.alpha, a.beta, row0, a.H, t0, a.T, tl, key, make_float2(pick(x1r), pick(x1i)),
                                                   make_float2(pick(x2r), pick(x2i)), cmulc(make_float2(lv.z, lv.w), make_float2(pick(x3r), pick(x3i))));
                put(x1r, o.qb.x);
                put(x1i, o.qb.y);
                put(x2r, o.zb.x);
                put(x2i, o.zb.y);
                put(x3r, o.fb.x);
                put(x3i, o.fb.y);
            }
        }
        if (!last_one) bar_arrive(kBarTaken, kGrad + kPrep);
        float2 dqv[4], dkv[4], dd[4];
        float al[4], dbp[2] = {0.f, 0.f};
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            // rotated key and query of the two keys: from the planes (W = a k', Q = a q'), or as above
            const int tl = g + 8 * r;
            const float4 *p = vals + tl * M + 8 * warp + 2 * t4;
            float2 kr, ki, qr, qi;
            if (fast) {
                const unsigned char *pw = slot_at + tl * TL::LDB + 2 * (8 * warp + 2 * t4);
                auto both = [&](int off, float2 f) {
                    const float2 h = unpack_f16(*reinterpret_cast<const uint32_t *>(pw + off)), l = unpack_f16(*reinterpret_cast<const uint32_t *>(pw + off + TL::PL));
                    return make_float2(f.x * (h.x + l.x), f.y * (h.y + l.y));
                };
                const float2 fw = make_float2(__fdividef(inv[0], va[2 * r].x), __fdividef(inv[0], va[2 * r + 1].x));
                const float2 fq = make_float2(__fdividef(inv[2], va[2 * r].x), __fdividef(inv[2], va[2 * r + 1].x));
                kr = both(TL::oW, fw);
                ki = both(TL::oW + 2 * TL::PL, fw);
                qr = both(TL::oQ, fq);
                qi = both(TL::oQ + 2 * TL::PL, fq);
            } else {
                const float4 u = rotated(tl, 8 * warp + 2 * t4), v = rotated(tl, 8 * warp + 2 * t4 + 1);
                kr = make_float2(u.x, v.x);
                ki = make_float2(u.y, v.y);
                qr = make_float2(u.z, v.z);
                qi = make_float2(u.w, v.w);
            }
            const float be = reinterpret_cast<const float *>(slot_at + TL::oB)[tl];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int i = 2 * r + e;
                const float2 ph = *(reinterpret_cast<const float2 *>(p + e) + 1);          // e^{i phi}
                const float2 kp = e ? make_float2(kr.y, ki.y) : make_float2(kr.x, ki.x), qp = e ? make_float2(qr.y, qi.y) : make_float2(qr.x, qi.x);
                const float2 qb = make_float2(x1r[i], x1i[i]), zb = make_float2(x2r[i], x2i[i]), fb = make_float2(x3r[i], x3i[i]);
                al[i] = e ? al2[r].y : al2[r].x;
                const float2 dkp = make_float2(be * fb.x - zb.x, be * fb.y - zb.y);
                dqv[i] = cmul(ph, qb);
                dkv[i] = cmul(ph, dkp);
                dbp[r] += fb.x * kp.x + fb.y * kp.y;
                const float2 y = cmulc(qb, qp), s = cmulc(kp, make_float2(be * fb.x, be * fb.y)), z = cmulc(zb, kp);
                dd[i] = make_float2(y.x - s.x - z.x, y.y - s.y - z.y);
            }
        }
        // D: sums over the tokens behind, down to each token (tokens 8-15 in i = 2, 3, tokens 0-7 in i = 0, 1)
#pragma unroll
        for (int d = 4; d < 32; d <<= 1)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float ox = __shfl_down_sync(0xffffffffu, dd[i].x, d), oy = __shfl_down_sync(0xffffffffu, dd[i].y, d);
                if (lane + d < 32) dd[i] = make_float2(dd[i].x + ox, dd[i].y + oy);
            }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            dd[2 + e] = make_float2(dd[2 + e].x + carry[e].x, dd[2 + e].y + carry[e].y);
            dd[e] = make_float2(dd[e].x + __shfl_sync(0xffffffffu, dd[2 + e].x, t4), dd[e].y + __shfl_sync(0xffffffffu, dd[2 + e].y, t4));
        }
        float dal[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) dal[i] = __fdividef(dd[i].x, al[i]);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int t = t0 + g + 8 * r;
            if (t < a.T) {
                const size_t row = row0 + (size_t)t * a.H;
                const size_t ak = row * DK + 2 * (8 * warp + 2 * t4), am = row * M + 8 * warp + 2 * t4;
                const float4 q4 = make_float4(dqv[2 * r].x, dqv[2 * r].y, dqv[2 * r + 1].x, dqv[2 * r + 1].y);
                const float4 k4 = make_float4(dkv[2 * r].x, dkv[2 * r].y, dkv[2 * r + 1].x, dkv[2 * r + 1].y);
                float2 a2 = make_float2(dal[2 * r], dal[2 * r + 1]), th2 = make_float2(dd[2 * r].y, dd[2 * r + 1].y);
                if (some) {                                        // (written by this thread, above)
                    if (redo >> 2 * r & 1) a2.x = a.dalpha[am], th2.x = a.dtheta[am];
                    if (redo >> 2 * r & 2) a2.y = a.dalpha[am + 1], th2.y = a.dtheta[am + 1];
                }
                st_val4(static_cast<T *>(a.dq) + ak, q4);
                st_val4(static_cast<T *>(a.dk) + ak, k4);
                __stcs(reinterpret_cast<float2 *>(a.dalpha + am), a2);
                __stcs(reinterpret_cast<float2 *>(a.dtheta + am), th2);
            }
            float x = dbp[r];
            x += __shfl_xor_sync(0xffffffffu, x, 1);
            x += __shfl_xor_sync(0xffffffffu, x, 2);
            // (a query that was taken out is missing from its own token's sum)
            if (t4 == 0) db[warp * 16 + g + 8 * r] = out >> (16 + g + 8 * r) & 1 ? __int_as_float(0x7fc00000) : x;
        }
    } else if (!last_one) {
        bar_arrive(kBarTaken, kGrad + kPrep);
    }
    bar_sync(kBarGrad, kGrad);
    if (tid < 16 && t0 + tid < a.T) {
        float x = 0.f;
#pragma unroll
        for (int w = 0; w < KT; ++w) x += db[w * 16 + tid];
        const size_t row = row0 + (size_t)(t0 + tid) * a.H;
        a.dbeta[row] = x;
    }
}

// ---- CHAIN helpers -----------------------------------------------------------------------------------
// the state's 16-column pieces to and from the checkpoint [piece][4][lane] float4
template <int KN>
__device__ __forceinline__ void keep_state(float4 *p, uint32_t st)
{
#pragma unroll 1
    for (int n = 0; n < KN; ++n, p += 128) {
        float x[16];
        tm_load(x, st + 16 * n);
        tm_wait_load(x);
#pragma unroll
        for (int j = 0; j < 4; ++j) __stcs(p + 32 * j, make_float4(x[4 * j], x[4 * j + 1], x[4 * j + 2], x[4 * j + 3]));
    }
}
__device__ __forceinline__ void read_piece(const float4 *p, float (&x)[16])
{
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float4 v = __ldcs(p + 32 * j);
        x[4 * j] = v.x;
        x[4 * j + 1] = v.y;
        x[4 * j + 2] = v.z;
        x[4 * j + 3] = v.w;
    }
}

// A kept state back into tensor memory; the largest entries of this thread's rows
template <int DK>
__device__ __forceinline__ float2 state_from_kept(uint32_t st, const float4 *p)
{
    float2 largest = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int n = 0; n < Tile<DK>::KS; ++n, p += 128) {
        float x[16];
        read_piece(p, x);
        largest = max_abs(reinterpret_cast<const float(&)[4][4]>(x), largest);
        tm_store(st + 16 * n, x);
    }
    tm_wait_store();
    return largest;
}

// The split state of a step of keys_product as the B operand (value channel, key) of the gradients' products
__device__ __forceinline__ void publish_split(uint4 *p, int kk, const uint32_t (&rh)[4], const uint32_t (&rl)[4], const uint32_t (&ih)[4], const uint32_t (&il)[4])
{
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        p[(4 * kk + 2 * e) * 32] = make_uint4(transpose8x8(rh[2 * e]), transpose8x8(rh[2 * e + 1]), transpose8x8(rl[2 * e]), transpose8x8(rl[2 * e + 1]));
        p[(4 * kk + 2 * e + 1) * 32] = make_uint4(transpose8x8(ih[2 * e]), transpose8x8(ih[2 * e + 1]), transpose8x8(il[2 * e]), transpose8x8(il[2 * e + 1]));
    }
}

// The same at the shared scale of all channels
__device__ __forceinline__ void publish_state(uint4 *p, int kk, const uint32_t (&rh)[4], const uint32_t (&rl)[4], const uint32_t (&ih)[4], const uint32_t (&il)[4],
                                              const RowScale &r, float all, bool own)
{
    if (!own) {
        publish_split(p, kk, rh, rl, ih, il);
        return;
    }
    uint32_t x[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        x[0][i] = rh[i];
        x[1][i] = rl[i];
        x[2][i] = ih[i];
        x[3][i] = il[i];
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) to_shared_scale(x[c], r, all);
    publish_split(p, kk, x[0], x[1], x[2], x[3]);
}

// Where a chain warp leaves a chunk's operands for the gradients; ps = NULL: nowhere
struct Publish {
    uint4 *ps, *pt;           // the state's (offset by the lane), the [value x token] operand's
    float *scale;             // two inverse scales
};

// The products over the keys of both halves, scaled by f and added
__device__ __forceinline__ void whole_sum(float (&acc)[2][2][4], const float (&f)[2], const Half &hf)
{
    float x[16], y[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = y[i] = f[(i & 3) >> 1] * acc[i >> 3][(i >> 2) & 1][i & 3];
    add_other(x, y, hf);
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i >> 3][(i >> 2) & 1][i & 3] = x[i];
}

// forward through one chunk whose tile is at `slot` (shared memory): U = M (V - W^* S), S <- gamma_C S + Y U unless
// `update` is false.  wait(): until the tile is there; load(rr): the chunk's rows of v.  KSP = 2: by one of two warps, for half
// of the keys.  Returns the largest magnitudes of S.
template <int DK, int KSP, typename Load, typename Wait>
__device__ __forceinline__ float2 forward_step(uint32_t st, float2 big, unsigned char *slot, Wait wait, Load load, const Publish &pub, bool update, int lane,
                                               const Half &hf = Half())
{
    using TL = Tile<DK>;
    constexpr int KN = TL::KS / KSP;
    float rr[2][4], ri[2][4];
    load(rr);
    uint32_t off;                                                // tokens whose v is not finite; below, all behind them too
    const RowScale sr = row_scale<4>(big);
    bool own = false;
    const float all = pub.ps ? shared_scale(sr, own) : 0.f;
    wait();
    const uint32_t tile = (uint32_t)__cvta_generic_to_shared(slot), keys = KSP > 1 ? 32 * KN * hf.half : 0;
    const float *inv = reinterpret_cast<const float *>(slot + TL::oS);
    const uint32_t tiles[1] = {tile + TL::oW + keys};
    TokFrag fr;
    {
        float acc[1][2][2][4];
        keys_product<DK, 1, KN>(acc, st, sr, tiles, lane, [&](int kk, const uint32_t(&rh)[4], const uint32_t(&rl)[4], const uint32_t(&ih)[4], const uint32_t(&il)[4]) {
            if (pub.ps) publish_state(pub.ps, kk, rh, rl, ih, il, sr, all, own);
        });
        const float fw[2] = {sr.inv[0] * inv[0], sr.inv[1] * inv[0]};
        off = take_out(rr);
        if constexpr (KSP > 1) whole_sum(acc[0], fw, hf);
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                rr[n][i] = KSP > 1 ? rr[n][i] - acc[0][0][n][i] : fmaf(-fw[i >> 1], acc[0][0][n][i], rr[n][i]);
                ri[n][i] = KSP > 1 ? -acc[0][1][n][i] : -fw[i >> 1] * acc[0][1][n][i];
            }
    }
    {
        TokFrag fb;
        const RowScale r = make_frag(fr, rr, ri);
        load_small<false>(fb, tile + TL::oM, lane);
        product_small<false, 2>(rr, ri, fr, fb, r.inv, inv[3]);
    }
    RowScale ru = make_frag(fr, rr, ri);
    const uint32_t out = reinterpret_cast<const uint32_t *>(inv)[7];
    const bool odd = __any_sync(0xffffffffu, (off | out) != 0);
    if (odd) {
        off = every_lanes(off, lane);
        off = from_first(off & 0xffffu) | from_first(off >> 16) << 16 | both(from_first(out & 0xffffu));
    }
    if (pub.ps) {
        const float all_u = publish_frag(pub.pt, fr, ru, odd, off, lane);
        if (lane == 0) {
            pub.scale[0] = all;
            pub.scale[1] = all_u;
        }
    }
    if (odd) put_nan(ru.inv, off);
    return update ? state_update<DK, KN>(st, fr, ru.inv, inv[1], tile + TL::oY + keys, reinterpret_cast<const float4 *>(slot + TL::oG) + keys / 4, lane) : big;
}

// backward through one chunk: Bc = M^H (Y^* G + (A D_beta)^H Yb^*), G <- conj(gamma_C) G + Q^T Yb^* - W^T Bc.  load(yr, yi):
// the chunk's rows of Yb^* (yi zero without has_im).  Leaves Re Bc (the rows of dv) in pr; returns the largest magnitudes of G.
template <int DK, int KSP, bool kExact, typename Load>
__device__ __forceinline__ float2 backward_step(uint32_t sg, float2 big, unsigned char *slot, Load load, bool has_im, float (&pr)[2][4],
                                                const Publish &pub, int lane, const Half &hf = Half())
{
    using TL = Tile<DK>;
    constexpr int KN = TL::KS / KSP;
    const int t4 = lane & 3;
    uint32_t off;                                                // tokens whose cotangents are not finite; below, all before them too
    TokFrag fy;
    RowScale ry;
    {
        float yr[2][4], yi[2][4];
        load(yr, yi);
        off = take_out(yr);
        if (has_im) off |= take_out(yi);
        ry = make_frag(fy, yr, yi);
    }
    const uint32_t tile = (uint32_t)__cvta_generic_to_shared(slot), keys = KSP > 1 ? 32 * KN * hf.half : 0;
    const float *inv = reinterpret_cast<const float *>(slot + TL::oS);
    const RowScale sr = row_scale<4>(big);
    bool own = false;
    const float all = pub.ps ? shared_scale(sr, own) : 0.f;
    float acc[1][2][2][4];
    const uint32_t tiles[1] = {tile + TL::oY + keys};
    keys_product<DK, 1, KN>(acc, sg, sr, tiles, lane, [&](int kk, const uint32_t(&rh)[4], const uint32_t(&rl)[4], const uint32_t(&ih)[4], const uint32_t(&il)[4]) {
        if (pub.ps) publish_state(pub.ps, kk, rh, rl, ih, il, sr, all, own);
    });
    float pi[2][4];
    {
        TokFrag fb;
        load_small<true>(fb, tile + TL::oA, lane);
        float fg[2] = {sr.inv[0] * inv[1], sr.inv[1] * inv[1]};
        if constexpr (KSP > 1) {
            whole_sum(acc[0], fg, hf);
            fg[0] = fg[1] = 1.f;
        }
        const float fa[2] = {ry.inv[0] * inv[4], ry.inv[1] * inv[4]};
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            float re[4] = {0.f, 0.f, 0.f, 0.f}, im[4] = {0.f, 0.f, 0.f, 0.f}, ni[4] = {0.f, 0.f, 0.f, 0.f};
            mma3x<kExact>(re, fy.rh, fy.rl, fb.rh[2 * n], fb.rh[2 * n + 1], fb.rl[2 * n], fb.rl[2 * n + 1]);
            mma3x<kExact>(ni, fy.rh, fy.rl, fb.ih[2 * n], fb.ih[2 * n + 1], fb.il[2 * n], fb.il[2 * n + 1]);
            if (has_im) {
                mma3x<kExact>(re, fy.ih, fy.il, fb.ih[2 * n], fb.ih[2 * n + 1], fb.il[2 * n], fb.il[2 * n + 1]);
                mma3x<kExact>(im, fy.ih, fy.il, fb.rh[2 * n], fb.rh[2 * n + 1], fb.rl[2 * n], fb.rl[2 * n + 1]);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                pr[n][i] = fmaf(fa[i >> 1], re[i], fg[i >> 1] * acc[0][0][n][i]);
                pi[n][i] = fmaf(fa[i >> 1], im[i] - ni[i], fg[i >> 1] * acc[0][1][n][i]);
            }
        }
    }
    TokFrag fp;
    {
        TokFrag fb;
        const RowScale r = make_frag(fp, pr, pi);
        load_small<true>(fb, tile + TL::oM, lane);
        product_small<true, 2>(pr, pi, fp, fb, r.inv, inv[3]);
    }
    const RowScale rb = make_frag(fp, pr, pi);
    const uint32_t out = reinterpret_cast<const uint32_t *>(inv)[7];
    const bool odd = __any_sync(0xffffffffu, (off | out) != 0);
    if (odd) {
        off = every_lanes(off, lane);
        off = to_last(off & 0xffffu) | to_last(off >> 16) << 16 | both(to_last((out | out >> 16) & 0xffffu));
        put_nan(pr, off, lane);
        put_nan(ry.inv, off);
    }
    if (pub.ps) {
        const float all_b = publish_frag(pub.pt, fp, rb, odd, off, lane);
        if (lane == 0) {
            pub.scale[0] = all;
            pub.scale[1] = all_b;
        }
    }
    const float fq[2] = {ry.inv[0] * inv[2], ry.inv[1] * inv[2]}, fw[2] = {-rb.inv[0] * inv[0], -rb.inv[1] * inv[0]};
    const float4 *gamma = reinterpret_cast<const float4 *>(slot + TL::oG) + t4 + keys / 4;
    uint32_t at = tile + keys + (uint32_t)(((lane & 7) + (((lane >> 3) & 1) << 3)) * TL::LDB + (lane >> 4) * 16);
    uint32_t nih[4], nil[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        nih[i] = fp.ih[i] ^ 0x80008000u;
        nil[i] = fp.il[i] ^ 0x80008000u;
    }
    big = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int np = 0; np < KN; ++np, at += 32, gamma += 8) {
        float x[16];
        tm_load(x, sg + 16 * np);
        uint32_t qh[4], ql[4], jh[4], jl[4];
        ldsm_t(qh, at + TL::oQ);
        ldsm_t(jh, at + TL::oQ + 2 * TL::PL);
        ldsm_t(ql, at + TL::oQ + TL::PL);
        ldsm_t(jl, at + TL::oQ + 3 * TL::PL);
        float qr[2][4], qi[2][4];
#pragma unroll
        for (int n = 0; n < 2; ++n) {
#pragma unroll
            for (int i = 0; i < 4; ++i) qr[n][i] = qi[n][i] = 0.f;
            mma3x<kExact>(qr[n], fy.rh, fy.rl, qh[2 * n], qh[2 * n + 1], ql[2 * n], ql[2 * n + 1]);
            mma3x<kExact>(qi[n], fy.rh, fy.rl, jh[2 * n], jh[2 * n + 1], jl[2 * n], jl[2 * n + 1]);
        }
        if (has_im) {
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                float ni[4] = {0.f, 0.f, 0.f, 0.f};
                mma3x<kExact>(ni, fy.ih, fy.il, jh[2 * n], jh[2 * n + 1], jl[2 * n], jl[2 * n + 1]);
                mma3x<kExact>(qi[n], fy.ih, fy.il, qh[2 * n], qh[2 * n + 1], ql[2 * n], ql[2 * n + 1]);
#pragma unroll
                for (int i = 0; i < 4; ++i) qr[n][i] -= ni[i];
            }
        }
        tm_wait_load(x);
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            const float4 gm = gamma[4 * n];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float cr = (i & 1) ? gm.z : gm.x, ci = (i & 1) ? gm.w : gm.y, u = x[8 * n + i], v = x[8 * n + 4 + i];
                x[8 * n + i] = fmaf(fq[i >> 1], qr[n][i], cr * u + ci * v);
                x[8 * n + 4 + i] = fmaf(fq[i >> 1], qi[n][i], cr * v - ci * u);
            }
        }
        tokens_product<DK>(qr, qi, fp, nih, nil, at + TL::oW);
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                x[8 * n + i] = fmaf(fw[i >> 1], qr[n][i], x[8 * n + i]);
                x[8 * n + 4 + i] = fmaf(fw[i >> 1], qi[n][i], x[8 * n + 4 + i]);
            }
        big = max_abs(reinterpret_cast<const float(&)[4][4]>(x), big);
        tm_store(sg + 16 * np, x);
    }
    tm_wait_store();
    return big;
}

// the rows of Yb^* of a chunk
template <typename T>
__device__ __forceinline__ void load_cotangents(float (&yr)[2][4], float (&yi)[2][4], const void *re, const void *im, size_t at, size_t step, int left)
{
    load_rows(yr, static_cast<const T *>(re) + at, step, left);
    load_rows(yi, static_cast<const T *>(im) + at, step, im ? left : 0);
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) yi[n][i] = -yi[n][i];
}

// a chain warp's part of a kept state: [piece][4][lane] float4
template <int DK>
__device__ __forceinline__ float4 *kept(float *keep, int bh, int pitch, int s, int dv, int col0, int lane)
{
    return reinterpret_cast<float4 *>(keep + (((size_t)bh * pitch + s) * dv + col0) * DK) + lane;
}

// ---- few sequences: the two chains alone, side by side (blockIdx.z) -------------------------------------
// With less than half as many sequences as SMs the walk of one CTA per sequence leaves the device idle.  But the
// cotangent's chain needs neither S nor U: so S walks forward and G backward at the same time, each in blocks of value
// columns (NB), both kept every 64 tokens; then every segment's gradients are a unit of their own (kUnits below).
template <int DK, int NB, int CL, int DVT, typename T>
__global__ void __launch_bounds__(Chain<DK, NB, CL>::threads, 1) sfda_backward_chain_kernel(const BwdArgsDev a)
{
    using TL = Tile<DK>;
    using L = Chain<DK, NB, CL>;
    constexpr int KN = L::KN;
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, bh = blockIdx.x, h = bh % a.H, b = bh / a.H, rank = blockIdx.y % CL, c0 = blockIdx.y * NB;
    const bool back = blockIdx.z != 0;
    const size_t row0 = (size_t)b * a.T * a.H + h;
    const int nch = (a.T + kC - 1) / kC;
    chain_begin<DK, NB, CL>(smem, tid);
    const uint32_t tmem = *reinterpret_cast<const uint32_t *>(smem + L::slow);
    const Wait limit = chain_limit<DK, NB, CL>(smem, (uint32_t)a.wait_ticks);
    if (tid == 0 && blockIdx.x + blockIdx.y + blockIdx.z == 0) *a.status = 0;     // (set, if at all, by the launch behind this one)
    __syncthreads();

    if (tid < L::kPrep) {
        if constexpr (NB == 128) asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
        chain_prep<DK, NB, CL, T>(smem, static_cast<const T *>(a.q), static_cast<const T *>(a.k), a.alpha, a.theta, a.beta, row0, a.H, a.T, nch, back, back,
                                  rank, limit, tid);
    } else if (tid < L::kPrep + L::kSolve) {
        if constexpr (NB == 128) asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
        chain_solve<DK, NB, CL>(smem, nch, back, rank, tid - L::kPrep);
    } else {
        if constexpr (NB == 128) asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
        const int lane = tid & 31, w = (tid - L::kPrep - L::kSolve) >> 5, half = L::KSP > 1 ? w & 1 : 0, g = lane >> 2, t4 = lane & 3;
        const int col0 = c0 + 16 * (w / L::KSP), col = col0 + g;
        const uint32_t st = tmem + ((uint32_t)(w & 3) << 21) + (w >> 2) * 16 * KN, full = (uint32_t)__cvta_generic_to_shared(smem + L::bars);
        const size_t state_at = ((size_t)bh * DK + 32 * KN * half + 4 * t4) * DVT + col, step = (size_t)a.H * DVT;
        const Publish none = {nullptr, nullptr, nullptr};
        const float *from = back ? a.dS_T : a.S0;
        float2 big = state_from_memory<KN>(st, from ? from + state_at : nullptr, DVT);
#pragma unroll 1
        for (int c = 0; c < nch; ++c) {
            const int slot = c % kSlots, cc = back ? nch - 1 - c : c, left = a.T - cc * kC - 2 * t4;
            unsigned char *tile = smem + slot * TL::bytes;
            const size_t at = (row0 + (size_t)(cc * kC + 2 * t4) * a.H) * DVT + col;
            const Half hf = L::KSP > 1 ? chain_half<DK, NB, CL>(smem, w, c, lane) : Half();
            auto wait = [&] { chain_wait<DK, NB, CL>(full, c, limit, lane); };
            auto kept_at = [&](float *keep) { return kept<DK>(keep, bh, a.pitch, cc / kSegChunks, DVT, col0, lane) + 128 * KN * half; };
            if (!back) {
                if (cc % kSegChunks == 0) keep_state<KN>(kept_at(a.keep_s), st);
                auto rows = [&](float(&x)[2][4]) { load_rows(x, static_cast<const T *>(a.v) + at, step, left); };
                big = forward_step<DK, L::KSP>(st, big, tile, wait, rows, none, true, lane, hf);
            } else {
                if (c == 0 || cc % kSegChunks == kSegChunks - 1) keep_state<KN>(kept_at(a.keep_g), st);
                float pr[2][4];
                auto rows = [&](float(&x)[2][4], float(&y)[2][4]) { load_cotangents<T>(x, y, a.d_o, a.d_o_im, at, step, left); };
                wait();
                big = backward_step<DK, L::KSP, sizeof(T) == 2>(st, big, tile, rows, a.d_o_im != nullptr, pr, none, lane, hf);
            }
            chain_release<DK, NB, CL>(full, c, nch, limit, lane);
        }
        if (back) state_to_memory<KN>(st, a.dS0 + state_at, DVT);
    }
    // where a wait ran out the kept states become NaN, so that all gradients that depend on them do (dv not on S), and dS0
    const bool gave_up = chain_end<DK, NB, CL>(smem, tmem, limit, tid);
    if (CL > 1 && tid == 0) a.flags[blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)] = gave_up;
    if (gave_up) {
        const float nan = __int_as_float(0x7fc00000);
        float *keep = (back ? a.keep_g : a.keep_s) + ((size_t)bh * a.pitch * DVT + c0) * DK;
#pragma unroll 1
        for (size_t i = tid; i < (size_t)a.NS * NB * DK; i += L::threads) keep[i / (NB * DK) * DVT * DK + i % (NB * DK)] = nan;
#pragma unroll 1
        for (int i = tid; back && i < DK * NB; i += L::threads) a.dS0[((size_t)bh * DK + i / NB) * DVT + c0 + i % NB] = nan;
    }
}

// ---- the walk with gradients ------------------------------------------------------------------------------
// kUnits == false: a pair is walked forward (keeping S), then its segments last to first: 2 NS positions.  The pairs'
// positions, one pair after the other, are cut into as many equal pieces as there are CTAs, so that no SM is idle while
// others work through a last round of whole pairs.  A pair that a cut falls into is begun by the CTA before the cut, as the
// first thing it does, and finished by the next one, as its last: S or G goes from one to the other through the place of
// the kept final state, and a CTA only waits for what the CTA before it in the grid does first.  256 pairs of 8192 tokens
// on 148 SMs, with the forward and the passes around it: 30.5 ms as two rounds of whole pairs, 27.5 ms cut.
// The launch is cooperative, so that both CTAs run, and the wait is bounded by what the other's part can take at most: a
// chunk takes 60 k cycles, and 250 k where every alpha is below 1/16.  Where it runs out all the same, the status
// word is set and the part is not walked: its gradients become NaN.  (Signs of life instead of a bound, one store per
// segment, cost 1.3 % of the walk, in the chain's warps as in the gradients'.)
// kUnits == true: S and G are kept already; a CTA takes units (pair, segment) blockIdx.x, + gridDim.x, ...
// Either way the second sweep is a list of segments, each of kSegChunks chunks (a ragged last one is completed with
// neutral tokens), pipelined over its borders.

// a position's share of the work: 12.6k cycles per chunk in the first sweep, 44.6k on the way back (d_k = d_v = 128)
constexpr int kSweepCost = 2, kBackCost = 7;

// Where CTA c's piece begins: pair * 2 NS + position
__device__ __forceinline__ long long walk_cut(long long work, int c, int ctas, int NS)
{
    const long long x = work * c / ctas;
    const int whole = (kSweepCost + kBackCost) * NS, pair = (int)(x / whole), rest = (int)(x - (long long)pair * whole);
    return (long long)pair * 2 * NS + (rest < kSweepCost * NS ? rest / kSweepCost : NS + (rest - kSweepCost * NS) / kBackCost);
}

// The j-th part of CTA c's piece: the pair that the next CTA finishes, whole pairs, the pair that the CTA before has begun.
// (pair, first position, position behind the last), or pair -1 behind the last part.
__device__ __forceinline__ int3 walk_part(long long work, int c, int ctas, int NS, int j)
{
    const int len = 2 * NS;
    const long long from = walk_cut(work, c, ctas, NS), to = walk_cut(work, c + 1, ctas, NS);
    const int head = (int)(to % len), tail = (int)(from % len);
    const int first = (int)((from + len - 1) / len), last = (int)(to / len);
    if (head && j-- == 0) return make_int3(last, 0, head);
    if (j < last - first) return make_int3(first + j, 0, len);
    if (tail && j == last - first) return make_int3(first - 1, tail, len);
    return make_int3(-1, 0, 0);
}

// NaN for every gradient of `tokens` tokens from t0 on of pair bh and, with `state`, for dS0, by all threads of the CTA
template <int DK, int NB, typename T>
__device__ __forceinline__ void give_up(const BwdArgsDev &a, int bh, int t0, int tokens, bool state, int tid, int threads)
{
    const float nan = __int_as_float(0x7fc00000);
    const size_t row0 = (size_t)(bh / a.H) * a.T * a.H + bh % a.H + (size_t)t0 * a.H;
#pragma unroll 1
    for (int i = tid; i < tokens * DK; i += threads) {
        const size_t row = row0 + (size_t)(i / DK) * a.H;
        const int x = i % DK;
        st_val(static_cast<T *>(a.dq), row * DK + x, nan);
        st_val(static_cast<T *>(a.dk), row * DK + x, nan);
        if (x < DK / 2) a.dalpha[row * (DK / 2) + x] = a.dtheta[row * (DK / 2) + x] = nan;
        if (x == 0) a.dbeta[row] = nan;
    }
#pragma unroll 1
    for (int i = tid; i < tokens * NB; i += threads) st_val(static_cast<T *>(a.dv), (row0 + (size_t)(i / NB) * a.H) * NB + i % NB, nan);
#pragma unroll 1
    for (int i = tid; state && i < DK * NB; i += threads) a.dS0[(size_t)bh * DK * NB + i] = nan;
}

template <int DK, int NB, typename T, bool kUnits>
__global__ void __launch_bounds__(kGrad + kPrep + 2 * NB, 1) sfda_backward_kernel(const BwdArgsDev a)
{
    using TL = Tile<DK>;
    using L = BwdSmem<DK, NB>;
    using SC = BwdScratch<DK, NB>;
    constexpr int kChain = 2 * NB, NCW = NB / 16, KT = TL::KT;
    constexpr bool kExact = sizeof(T) == 2;
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, NS = a.NS, nch = (a.T + kC - 1) / kC;
    unsigned char *ring = a.ring + blockIdx.x * a.ring_bytes;
    constexpr int places = ring_places(kUnits);
    volatile int *job = reinterpret_cast<volatile int *>(smem + L::job);
    // The next part of the walk, for all threads at once (a part leaves none of its barriers pending).
    auto next_part = [&](int j) {
        if constexpr (kUnits) return j == 0;
        bar_sync(0, kGrad + kPrep + kChain);
        if (tid == 0) {
            // the first part is what the next CTA waits for
            if (j == 1 && a.flags && !a.withhold) asm volatile("fence.acq_rel.gpu;\n\tst.relaxed.gpu.global.u32 [%0], 1;" ::"l"(a.flags + blockIdx.x) : "memory");
            const int3 p = walk_part(a.work, blockIdx.x, gridDim.x, NS, j);
            int gave_up = 0;
            if (p.x >= 0 && p.y) {
                uint32_t seen, before = (uint32_t)clock();
                unsigned long long spent = 0;
                while (true) {
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(a.flags + blockIdx.x - 1) : "memory");
                    if (seen) break;
                    const uint32_t now = (uint32_t)clock();
                    spent += min(now - before, 1u << 16);                // (a pause of the whole SM counts as one look)
                    before = now;
                    if (spent >= a.wait_ticks) {
                        gave_up = 1;
                        atomicOr(a.status, 1u);
                        break;
                    }
                    __nanosleep(200);
                }
                __threadfence();
            }
            job[0] = p.x;
            job[1] = p.y;
            job[2] = p.z;
            job[3] = gave_up;
        }
        bar_sync(0, kGrad + kPrep + kChain);
        return job[0] >= 0 && !job[3];                                   // (only the last part can be given up)
    };
    auto segments_of = [&] { return kUnits ? (a.units - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : max(0, job[2] - max(job[1], NS)); };
    // the r-th segment of this CTA's list: pair and segment; row of token t of a pair: row0 + t H
    auto segment = [&](int r, int &bh, int &s) {
        if constexpr (kUnits) {
            const int u = blockIdx.x + r * gridDim.x;
            bh = u / NS;
            s = u - bh * NS;
        } else {
            bh = job[0];
            s = 2 * NS - 1 - max(job[1], NS) - r;
        }
    };
    auto row_of = [&](int bh) { return (size_t)(bh / a.H) * a.T * a.H + bh % a.H; };
    // the status word: cleared by the launcher where pieces are handed over, by the chains before units
    if (!kUnits && !a.flags && blockIdx.x == 0 && tid == 0) *a.status = 0;
    const Wait limit = {(uint32_t)__cvta_generic_to_shared(smem + L::gfree + 16), (uint32_t)a.wait_ticks};   // (of GFREE)
    if (tid < 32) tm_alloc(reinterpret_cast<uint32_t *>(smem + L::word), L::columns);
    if (places == 2 && tid == 32) {
        const uint32_t bar = (uint32_t)__cvta_generic_to_shared(smem + L::gfree);
        mbar_init(bar, kGradWarps);
        mbar_init(bar + 8, kGradWarps);
        *reinterpret_cast<uint32_t *>(smem + L::gfree + 16) = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *reinterpret_cast<const uint32_t *>(smem + L::word);

    // Where a wait for GFREE ran out: NaN for all gradients of this CTA's segments.  By the gradients' warps with 128 value columns, by
    // all threads with 64: at the end of the kernel it costs the former's code 1 % (training step at B = 4, T = 4096, H = 16 4.22 -> 4.17
    // ms), among the gradients it costs the latter's 2 % (fp32 segments of 64 / 64 at B H = 8, T = 333 101 us instead of 99).
    auto give_up_units = [&](int threads) {
        if (places != 2 || !limit.raised()) return;
        if (tid == 0) atomicOr(a.status, 1u);
#pragma unroll 1
        for (int r = 0; r < segments_of(); ++r) {
            int bh, s;
            segment(r, bh, s);
            give_up<DK, NB, T>(a, bh, s * kSeg, min(kSeg, a.T - s * kSeg), false, tid, threads);
        }
    };

    // register shares: 256 x (88 + 64 + 88) of 768 x 80 with 128 value columns; 256 x (104 + 80) + 128 x 112 of 640 x 96
    // with 64
    if (tid < kGrad) {
        if constexpr (NB == 128) asm volatile("setmaxnreg.inc.sync.aligned.u32 88;");
        if constexpr (NB == 64) asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
        if (kUnits && blockIdx.x == 0 && tid < a.chain_ctas && a.flags[tid]) atomicOr(a.status, 1u);
        __syncwarp();
#pragma unroll 1
        for (int j = 0; next_part(j); ++j) {
            const int total = segments_of() * kSegChunks;
#pragma unroll 1
            for (int n = 0; n < total; ++n) {
                const int r = n / kSegChunks, at = n % kSegChunks, c = kSegChunks - 1 - at, slot = ring_slot(r, c);
                int bh, s;
                segment(r, bh, s);
                chunk_gradients<DK, NB, T>(a, smem, ring, slot, back_place(c, places), places == 2 && !limit.withheld(), n + 1 == total, s * kSeg + c * kC, row_of(bh), tid);
                if (n + kSlots < total) bar_arrive(kBarReady + (n & 1), kGrad + kPrep);
            }
        }
        if constexpr (NB == 128) {                               // (the chain is through with what these warps have used)
            bar_sync(kBarGrad, kGrad);
            give_up_units(kGrad);
        }
    } else if (tid < kGrad + kPrep) {
        if constexpr (NB == 128) asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
        if constexpr (NB == 64) asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        const T *q = static_cast<const T *>(a.q), *k = static_cast<const T *>(a.k);
        const int ptid = tid - kGrad, lane = tid & 31, w = ptid >> 5;
        const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem);
        float2 *gram = reinterpret_cast<float2 *>(smem + L::gram);
        // One list of steps, two tasks each.  First sweep: chunk p is prepared once the chain is through with chunk p - 4.
        // Second sweep: the tokens of chunk m = p - 3 (in the order the chain comes back) are staged for the gradients
        // and chunk p (in the order it goes forward) is prepared once those of chunk p - 4 are written.  The chain needs
        // a whole segment prepared before it can come back, so that a segment's first chunk is staged second.
#pragma unroll 1
        for (int j = 0; next_part(j);)
#pragma unroll 1
        for (int sweep = kUnits ? 1 : 0; sweep < 2; j += sweep++) {
            const int c0 = sweep ? 0 : min(job[1], NS) * kSegChunks;
            const int np = sweep ? segments_of() * kSegChunks : min(nch, job[2] * kSegChunks) - c0;
#pragma unroll 1
            for (int u = 0; u < 2 * (np + (sweep ? 3 : kSlots)); ++u) {
                const int p = u >> 1, m = sweep ? p - 3 : -1;
                int bh, s;
                if (m < 0 ? (u & 1) != 0 : ((u & 1) == 0) != (m % kSegChunks == 0)) {
                    if (m < 0) continue;
                    const int r = m / kSegChunks, c = kSegChunks - 1 - m % kSegChunks, slot = ring_slot(r, c);
                    segment(r, bh, s);
                    bar_sync(kBarDone + slot, kPrep + kChain);
                    if (m) bar_sync(kBarTaken, kGrad + kPrep);
                    stage_tokens<DK, NB, T>(a, smem, ring, slot, back_place(c, places), s * kSeg + c * kC, row_of(bh), ptid);
                    continue;
                }
                if (!sweep && p >= kSlots) bar_sync(kBarDone + p % kSlots, kPrep + kChain);
                if (p >= np) continue;
                const int r = p / kSegChunks, at = p % kSegChunks, slot = sweep ? ring_slot(r, at) : at;
                if (sweep && p >= kSlots) bar_sync(kBarReady + (p & 1), kGrad + kPrep);
                segment(sweep ? r : 0, bh, s);
                const size_t row0 = row_of(bh);
                const int t0 = sweep ? s * kSeg + at * kC : (c0 + p) * kC;
                const bool needq = sweep;
                unsigned char *tile = smem + slot * TL::bytes;
                float *inv = reinterpret_cast<float *>(tile + TL::oS);
                PrepRaw<L::PM::TPT, T> in;
                prep_fetch<DK, kPrepWarps, T>(in, q, k, a.alpha, a.theta, a.beta, row0, a.H, t0, a.T, needq, ptid);
                float4 *vals = sweep ? reinterpret_cast<float4 *>(ring + (size_t)slot * SC::slot + SC::oV) : nullptr;
                const bool fast = prep_chunk<DK, kPrepWarps, kBarPrep, T>(in, q, k, a.alpha, a.theta, a.beta, row0, a.H, t0, a.T, vals, tile, smem + L::kb,
                                                                          smem + L::scan, needq, ptid);
                if (!fast)
                    slow_gram<DK, kPrepWarps, kBarPrep, T>(q, k, a.alpha, a.theta, a.beta, row0, a.H, t0, a.T, ring + SC::oSlow,
                                                           smem + L::scan, gram, gram + 16 * 17, needq, ptid);
                bar_sync(kBarPrep, kPrep);
                if (fast && w < (needq ? 4 : 2))                 // the two Gram matrices, a column tile per warp (a matrix
                                                                 // per warp: 27.5 ms instead of 27.35 for the training step)
                    gram_tiles<DK, 1>(base + slot * TL::bytes + (w >> 1 ? TL::oQ : TL::oW), base + L::kb, inv[w >> 1 ? 2 : 0] * inv[5],
                                      gram + (w >> 1) * 16 * 17, w & 1, lane);
                bar_sync(kBarPrep, kPrep);
                if (w == 0 || (needq && w == 1)) {               // the system's inverse; the outputs' Gram matrix
                    float2 *gm = gram + w * 16 * 17;
                    if (!w) invert_unit_lower16(gm, lane);
                    store_lower(tile + (w ? TL::oA : TL::oM), gm, inv + 3 + w, lane);
                }
                bar_arrive(kBarFull + slot, kPrep + kChain);
            }
        }
    } else {
        if constexpr (NB == 128) asm volatile("setmaxnreg.inc.sync.aligned.u32 88;");
        if constexpr (NB == 64) asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
        const int lane = tid & 31, w = (tid - kGrad - kPrep) >> 5, g = lane >> 2, t4 = lane & 3;
        const int col = 16 * w + g;                                      // and col + 8
        const uint32_t ss = tmem + ((uint32_t)(w & 3) << 21) + (w >> 2) * 16 * KT, sg = ss + 8 * KT;   // S and G
        float *scal = reinterpret_cast<float *>(smem + L::scal);
        const size_t step = (size_t)a.H * NB;
        float2 big_s = make_float2(0.f, 0.f), big_g = big_s;
#pragma unroll 1
        for (int j = 0; next_part(j); ++j)
#pragma unroll 1
        for (int r = kUnits ? 0 : -1, segments = segments_of(); r < segments; ++r) {   // -1: the first sweep
            int bh, s;
            segment(max(r, 0), bh, s);
            const size_t state_at = ((size_t)bh * DK + 4 * t4) * NB + col, row0 = row_of(bh);
            const int from = kUnits ? 0 : job[1], to = kUnits ? 0 : job[2], c0 = r < 0 ? from * kSegChunks : 0;
            if (r < 0) {
                if (from >= NS) continue;
                big_s = from ? state_from_kept<DK>(ss, kept<DK>(a.keep_s, bh, a.pitch, NS, NB, 16 * w, lane))
                             : state_from_memory<TL::KS>(ss, a.S0 ? a.S0 + state_at : nullptr, NB);
            } else {
                if (!kUnits && r == 0)
                    big_g = from > NS ? state_from_kept<DK>(sg, kept<DK>(a.keep_s, bh, a.pitch, NS, NB, 16 * w, lane))
                                      : state_from_memory<TL::KS>(sg, a.dS_T ? a.dS_T + state_at : nullptr, NB);
                const float4 *start = kept<DK>(a.keep_s, bh, a.pitch, s, NB, 16 * w, lane), *kg = kept<DK>(a.keep_g, bh, a.pitch, s, NB, 16 * w, lane);
                big_s = make_float2(0.f, 0.f);
                if (kUnits) big_g = make_float2(0.f, 0.f);
#pragma unroll 1
                for (int n = 0; n < TL::KS; ++n, start += 128, kg += 128) {
                    float x[16];
                    if constexpr (kUnits) {
                        read_piece(kg, x);
                        tm_store(sg + 16 * n, x);
                        big_g = max_abs(reinterpret_cast<const float(&)[4][4]>(x), big_g);
                    }
                    read_piece(start, x);
                    tm_store(ss + 16 * n, x);
                    big_s = max_abs(reinterpret_cast<const float(&)[4][4]>(x), big_s);
                }
                tm_wait_store();
            }
#pragma unroll 1
            for (int c = c0, n = r < 0 ? min(nch, to * kSegChunks) : kSegChunks; c < n; ++c) {
                const int slot = r < 0 ? c % kSlots : ring_slot(r, c), t0 = (r < 0 ? 0 : s * kSeg) + c * kC;
                if (r < 0 && c % kSegChunks == 0) keep_state<TL::KS>(kept<DK>(a.keep_s, bh, a.pitch, c / kSegChunks, NB, 16 * w, lane), ss);
                unsigned char *scr = ring + (size_t)slot * SC::slot;
                Publish pub = {nullptr, nullptr, nullptr};
                if (r >= 0) pub = {reinterpret_cast<uint4 *>(scr + SC::oS) + w * KT * 64 + lane, reinterpret_cast<uint4 *>(scr + SC::oU) + w * 128, scal + (slot * NCW + w) * 4};
                auto rows = [&](float(&x)[2][4]) {
                    load_rows(x, static_cast<const T *>(a.v) + (row0 + (size_t)(t0 + 2 * t4) * a.H) * NB + col, step, a.T - t0 - 2 * t4);
                };
                auto full = [&] { bar_sync(kBarFull + slot, kPrep + kChain); };
                big_s = forward_step<DK, 1>(ss, big_s, smem + slot * TL::bytes, full, rows, pub, r < 0 || c + 1 < kSegChunks, lane);
                if (r < 0) bar_arrive(kBarDone + slot, kPrep + kChain);
            }
            if (r < 0) {                                                 // the final state, or where the next CTA begins
                keep_state<TL::KS>(kept<DK>(a.keep_s, bh, a.pitch, NS, NB, 16 * w, lane), ss);
                continue;
            }
#pragma unroll 1
            for (int c = kSegChunks - 1; c >= 0; --c) {
                const int slot = ring_slot(r, c), t0 = s * kSeg + c * kC, left = a.T - t0 - 2 * t4;
                const size_t at = (row0 + (size_t)(t0 + 2 * t4) * a.H) * NB + col;
                const int n = r * kSegChunks + kSegChunks - 1 - c;
                unsigned char *scr = ring + (n & (places - 1)) * SC::place;
                const Publish pub = {reinterpret_cast<uint4 *>(scr + SC::oG) + w * KT * 64 + lane, reinterpret_cast<uint4 *>(scr + SC::oB) + w * 128, scal + (slot * NCW + w) * 4 + 2};
                // (where this wait runs out the place is overwritten while it is read, and all of the CTA's gradients become NaN)
                if constexpr (places == 2) cluster_wait<1>(limit.flag - 16 + 8 * (n & 1), ((n >> 1) + 1) & 1, limit, lane);
                float pr[2][4];
                auto rows = [&](float(&x)[2][4], float(&y)[2][4]) { load_cotangents<T>(x, y, a.d_o, a.d_o_im, at, step, left); };
                big_g = backward_step<DK, 1, kExact>(sg, big_g, smem + slot * TL::bytes, rows, a.d_o_im != nullptr, pr, pub, lane);
                store_rows(static_cast<T *>(a.dv) + at, pr, step, left);
                bar_arrive(kBarDone + slot, kPrep + kChain);
            }
            if (!kUnits && r + 1 == segments) {
                if (to == 2 * NS) state_to_memory<TL::KS>(sg, a.dS0 + state_at, NB);
                else keep_state<TL::KS>(kept<DK>(a.keep_s, bh, a.pitch, NS, NB, 16 * w, lane), sg);
            }
        }
    }
    if constexpr (!kUnits) {
        if (job[3]) give_up<DK, NB, T>(a, job[0], 0, min(a.T, (2 * NS - max(job[1], NS)) * kSeg), true, tid, kGrad + kPrep + kChain);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if constexpr (NB == 64) give_up_units(kGrad + kPrep + kChain);
    if (tid < 32) tm_free(tmem, L::columns);
}

// All value columns while the (batch, head) pairs alone fill the SMs: then there is only the walk with gradients.  Fewer with few
// sequences: the chains by themselves, then units; how many fewer only says how large the workspace is (the chains' blocks are
// those of chain_blocks).  (A fixed count rather than the
// device's: the workspace size must not depend on where it is asked for.)
int bwd_cols(int B, int H, int d_v)
{
    int cols = d_v;
    while (cols > 32 && (long long)B * H * (d_v / (cols / 2)) <= kBwdTargetCtas) cols /= 2;
    return cols;
}

// Workspace in floats: with many sequences the kept states (one per segment of 64 tokens and pair) and 64 states per
// pair, which hold a CTA's ring and the final state.  With few sequences as much again and 3 d_k + 1 floats per row and
// block of columns: room for both chains' kept states and one ring for as many CTAs as fit (never less than one).
size_t bwd_workspace(int B, int T, int H, int d_k, int d_v)
{
    const size_t bhn = (size_t)B * H, ns = (size_t)(T + kSeg - 1) / kSeg, state = (size_t)d_k * d_v;
    const size_t rows = bhn * T, nsl = (size_t)(d_v / bwd_cols(B, H, d_v)), shares = nsl > 1 ? nsl * rows : 0;
    return bhn * (ns + kSeg) * state + shares * 3 * d_k + ((shares + 3) & ~(size_t)3);
}

template <int DK, int DV, typename T, bool kUnits>
cudaError_t launch_walk(const BwdArgsDev &a, int grid, cudaStream_t stream, int *launches)
{
    auto kern = sfda_backward_kernel<DK, DV, T, kUnits>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BwdSmem<DK, DV>::bytes);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kGrad + kPrep + 2 * DV);
    cfg.dynamicSmemBytes = BwdSmem<DK, DV>::bytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = !kUnits && a.flags ? 1 : 0;                 // CTAs that wait for one another run together (one per SM)
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kern, a);
    const cudaError_t last = cudaGetLastError();                 // (cleared also where the launch was refused)
    if (e != cudaSuccess) return e;
    if (launches) ++*launches;
    return last;
}

template <int DK, int NB, int CL, int DV, typename T>
cudaError_t launch_chains(const BwdArgsDev &a, int pairs, cudaStream_t stream, int *launches)
{
    using L = Chain<DK, NB, CL>;
    if (launches) ++*launches;
    return launch_clusters(sfda_backward_chain_kernel<DK, NB, CL, DV, T>, a, dim3((unsigned)pairs, DV / NB, 2), CL, L::threads, L::bytes, stream);
}

template <int DK, int DV, typename T>
cudaError_t launch_typed(const BackwardArgs &x, void *workspace, cudaStream_t stream, int *launches)
{
    using SC = BwdScratch<DK, DV>;
    const size_t state = (size_t)DK * DV;
    const int pairs = x.B * x.H, cols = bwd_cols(x.B, x.H, DV);
    float *ws = reinterpret_cast<float *>(static_cast<char *>(workspace) + kHeadBytes);
    BwdArgsDev a;
    a.q = x.q; a.k = x.k; a.v = x.v; a.d_o = x.d_o; a.d_o_im = x.d_o_im;
    a.alpha = x.alpha; a.theta = x.theta; a.beta = x.beta; a.S0 = x.S0; a.dS_T = x.dS_T;
    a.dq = x.dq; a.dk = x.dk; a.dv = x.dv; a.dalpha = x.dalpha; a.dtheta = x.dtheta; a.dbeta = x.dbeta; a.dS0 = x.dS0;
    a.T = x.T; a.H = x.H; a.NS = (x.T + kSeg - 1) / kSeg;
    a.units = pairs * a.NS;
    a.keep_s = ws;
    a.pitch = a.NS + 1;
    a.keep_g = ws + (size_t)pairs * a.pitch * state;
    a.ring_bytes = SC::bytes(ring_places(cols != DV));
    a.status = static_cast<unsigned *>(workspace);
    a.flags = nullptr;
    a.chain_ctas = 0;
    a.wait_ticks = x.wait_ticks ? x.wait_ticks : 1ull << 31;     // about a second, more for long sequences
    if (!x.wait_ticks && (unsigned long long)a.NS * kSegChunks * kChunkTicks > a.wait_ticks) a.wait_ticks = (unsigned long long)a.NS * kSegChunks * kChunkTicks;
    a.withhold = x.withhold;
    if (cols == DV) {
        int dev = 0, sms = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        const int most = sms < kBwdTargetCtas ? sms : kBwdTargetCtas, grid = pairs < most ? pairs : most;
        a.ring = reinterpret_cast<unsigned char *>(a.keep_g);
        a.work = (long long)pairs * a.NS * (kSweepCost + kBackCost);
        if (pairs % grid) {
            a.flags = a.status + 64;
            if ((e = cudaMemsetAsync(a.status, 0, kHeadBytes, stream)) != cudaSuccess) return e;
        } else if (a.withhold) {
            return cudaErrorInvalidValue;                        // no pair is cut
        }
        return launch_walk<DK, DV, T, false>(a, grid, stream, launches);
    }
    if (a.withhold) return cudaErrorInvalidValue;
    float *rings = a.keep_g + (size_t)pairs * a.pitch * state;
    a.ring = reinterpret_cast<unsigned char *>(rings);
    const size_t room = bwd_workspace(x.B, x.T, x.H, DK, DV) * sizeof(float) - kHeadBytes - (size_t)(rings - ws) * sizeof(float);
    int grid = a.units < kBwdTargetCtas ? a.units : kBwdTargetCtas;
    if ((size_t)grid * a.ring_bytes > room) grid = (int)(room / a.ring_bytes);
    const Blocks b = chain_blocks(2LL * pairs, DV);              // both chains of all pairs at once
    a.flags = a.status + 64;
    a.chain_ctas = b.cluster > 1 ? 2 * pairs * (DV / b.columns) : 0;
    a.wait_ticks = wait_limit();
    cudaError_t e;
    if (b.columns == DV) e = launch_chains<DK, DV, 1, DV, T>(a, pairs, stream, launches);
    else if (b.columns == 64) e = launch_chains<DK, 64, DV / 64, DV, T>(a, pairs, stream, launches);
    else if (b.cluster == 2) e = launch_chains<DK, 32, 2, DV, T>(a, pairs, stream, launches);
    else e = launch_chains<DK, 32, DV / 32, DV, T>(a, pairs, stream, launches);
    return e == cudaSuccess ? launch_walk<DK, DV, T, true>(a, grid, stream, launches) : e;
}

}  // namespace

bool backward_hands_over(int B, int H, int d_v)
{
    const long long pairs = (long long)B * H;
    return bwd_cols(B, H, d_v) == d_v && pairs > kBwdTargetCtas && pairs % kBwdTargetCtas != 0;
}

size_t backward_workspace_bytes(int B, int T, int H, int d_k, int d_v)
{
    return bwd_workspace(B, T, H, d_k, d_v) * sizeof(float);
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
