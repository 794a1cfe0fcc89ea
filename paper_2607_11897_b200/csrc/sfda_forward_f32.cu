// fp32 chunk-WY forward for every supported d_k, d_v and dtype: the path of fp32 inputs and of the shapes the bf16
// tensor-core kernel does not take.  Same algebra as the other forwards (Theorem "Constructive left-to-right chunk-WY
// recursion", Eq. "apply-transfer", Theorem "Prefix outputs inside a chunk") in chunks of 16 tokens:
//
//   R = V - W^* S_0,  U = M R,  rho = Q^* S_0 + (A^{qk} D_beta) U,  o = conj(rho),  S_C = gamma_C S_0 + Y U
//
// One CTA per (batch, head) pair and block of value columns, the blocks of a pair a cluster that shares the preparation of
// the chunks; sfda_chunk16.cuh describes the arithmetic (split fp16 on the tensor cores) and the roles, which are pipelined
// over a ring of operand tiles.
//
// What bounds it: with few pairs the latency of the chain (B = 2, T = 2001, H = 16, d = 128, fp32: 5.0 k cycles of a chunk's 5.1 k are
// left without any preparation), with many the schedulers' issue slots, which mma.sync holds.  326 us at those sizes (457
// while each of a pair's four CTAs prepared every chunk for itself and a warp had all keys of its 16 columns; the unrolled
// first version 665, the CUDA-core kernel 3154); B = 1, T = 256, H = 2, d = 64: 37 us (39, 61, 201).
#include "sfda_chunk16.cuh"
#include "sfda_internal.h"

namespace sfda {
namespace {

using namespace c16;

struct FwdArgsDev {
    const void *q, *k, *v;
    const float *alpha, *theta, *beta, *S0;
    void *o, *o_im;
    float *S_T;
    int T, H, dv;
    uint32_t wait_ticks;                                         // limit of the waits on another CTA
};

template <int DK, int NB, int CL, typename T>
__global__ void __launch_bounds__(Chain<DK, NB, CL>::threads, 1) sfda_forward_f32_kernel(const FwdArgsDev a)
{
    using TL = Tile<DK>;
    using L = Chain<DK, NB, CL>;
    constexpr int KN = L::KN;
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, bh = blockIdx.x, h = bh % a.H, b = bh / a.H, c0 = blockIdx.y * NB, rank = blockIdx.y % CL;
    const size_t row0 = (size_t)b * a.T * a.H + h;               // row of token t: row0 + t H
    const int nch = (a.T + kC - 1) / kC;
    chain_begin<DK, NB, CL>(smem, tid);
    const uint32_t tmem = *reinterpret_cast<const uint32_t *>(smem + L::slow);
    const Wait wait = chain_limit<DK, NB, CL>(smem, a.wait_ticks);
    __syncthreads();

    // register shares with all 128 value columns: 256 x 88 + 128 x 72 + 256 x 112 of the launch's 640 x 96
    if (tid < L::kPrep) {
        if constexpr (NB == 128) asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
        chain_prep<DK, NB, CL, T>(smem, static_cast<const T *>(a.q), static_cast<const T *>(a.k), a.alpha, a.theta, a.beta, row0, a.H, a.T, nch, false, true,
                                  rank, wait, tid);
    } else if (tid < L::kPrep + L::kSolve) {
        if constexpr (NB == 128) asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
        chain_solve<DK, NB, CL>(smem, nch, true, rank, tid - L::kPrep);
    } else {
        if constexpr (NB == 128) asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
        const int lane = tid & 31, w = (tid - L::kPrep - L::kSolve) >> 5, half = L::KSP > 1 ? w & 1 : 0, g = lane >> 2, t4 = lane & 3;
        const int col = c0 + 16 * (w / L::KSP) + g;              // and col + 8
        const uint32_t st = tmem + ((uint32_t)(w & 3) << 21) + (w >> 2) * 16 * KN;       // this warp's lanes and columns
        const size_t state_at = ((size_t)bh * DK + 32 * KN * half + 4 * t4) * a.dv + col;
        float2 largest = state_from_memory<KN>(st, a.S0 ? a.S0 + state_at : nullptr, a.dv);
        const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem), keys = 32 * KN * half;   // (bytes of a row in front of this half)
        const size_t step = (size_t)a.H * a.dv;
        size_t at = (row0 + (size_t)(2 * t4) * a.H) * a.dv + col;
#pragma unroll 1
        for (int c = 0; c < nch; ++c, at += 16 * step) {
            const int slot = c % kSlots, left = a.T - c * kC - 2 * t4;
            float rr[2][4], ri[2][4];
            load_rows(rr, static_cast<const T *>(a.v) + at, step, left);
            const RowScale sr = row_scale<4>(largest);
            chain_wait<DK, NB, CL>(base + L::bars, c, wait, lane);
            const uint32_t tile = base + slot * TL::bytes;
            const float *inv = reinterpret_cast<const float *>(smem + slot * TL::bytes + TL::oS);
            float acc[2][2][2][4];
            const uint32_t tiles[2] = {tile + TL::oW + keys, tile + TL::oQ + keys};
            keys_product<DK, 2, KN>(acc, st, sr, tiles, lane, [](int, const uint32_t(&)[4], const uint32_t(&)[4], const uint32_t(&)[4], const uint32_t(&)[4]) {});
            const float fw[2] = {sr.inv[0] * inv[0], sr.inv[1] * inv[0]}, fq[2] = {sr.inv[0] * inv[2], sr.inv[1] * inv[2]};
            uint32_t off = take_out(rr);                         // tokens whose v is not finite; below, all behind them too
            // R in rr, ri; the outputs' part from S in pr, pi: all tokens, or the eight of this half
            constexpr int NT = 2 / L::KSP;
            float pr[NT][4], pi[NT][4];
            if constexpr (L::KSP == 1) {
#pragma unroll
                for (int n = 0; n < 2; ++n)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        rr[n][i] = fmaf(-fw[i >> 1], acc[0][0][n][i], rr[n][i]);
                        ri[n][i] = -fw[i >> 1] * acc[0][1][n][i];
                        pr[n][i] = fq[i >> 1] * acc[1][0][n][i];
                        pi[n][i] = fq[i >> 1] * acc[1][1][n][i];
                    }
            } else {
                float x[24], y[24];                              // W^* S of all tokens, Q^* S of this half's (y: the other's)
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    x[i] = y[i] = fw[(i & 3) >> 1] * acc[0][0][i >> 2][i & 3];
                    x[8 + i] = y[8 + i] = fw[(i & 3) >> 1] * acc[0][1][i >> 2][i & 3];
                    const float u = acc[1][i >> 2][0][i & 3], v = acc[1][i >> 2][1][i & 3], f = fq[(i & 3) >> 1];
                    x[16 + i] = f * (half ? v : u);
                    y[16 + i] = f * (half ? u : v);
                }
                add_other(x, y, chain_half<DK, NB, CL>(smem, w, c, lane));
#pragma unroll
                for (int i = 0; i < 4; ++i) {
#pragma unroll
                    for (int n = 0; n < 2; ++n) {
                        rr[n][i] -= x[4 * n + i];
                        ri[n][i] = -x[8 + 4 * n + i];
                    }
                    pr[0][i] = x[16 + i];
                    pi[0][i] = x[20 + i];
                }
            }
            TokFrag fr, fb;
            const RowScale r = make_frag(fr, rr, ri);            // U = M R
            load_small<false>(fb, tile + TL::oM, lane);
            product_small<false, 2>(rr, ri, fr, fb, r.inv, inv[3]);
            RowScale ru = make_frag(fr, rr, ri);                 // (A^{qk} D_beta) U
            load_small<false>(fb, tile + TL::oA, lane);
            float ur[NT][4], ui[NT][4];
            if (L::KSP > 1 && half) {                            // the second token tile's registers
#pragma unroll
                for (int i = 0; i < 2; ++i) fb.rh[i] = fb.rh[2 + i], fb.rl[i] = fb.rl[2 + i], fb.ih[i] = fb.ih[2 + i], fb.il[i] = fb.il[2 + i];
            }
            product_small<false, NT>(ur, ui, fr, fb, ru.inv, inv[4]);
            const uint32_t out = reinterpret_cast<const uint32_t *>(inv)[7];
            const bool odd = __any_sync(0xffffffffu, (off | out) != 0);
            if (odd) {
                off = every_lanes(off, lane);
                off = from_first(off & 0xffffu) | from_first(off >> 16) << 16 | both(from_first(out & 0xffffu));
                put_nan(ru.inv, off);
            }
            largest = state_update<DK, KN>(st, fr, ru.inv, inv[1], tile + TL::oY + keys, reinterpret_cast<const float4 *>(smem + slot * TL::bytes + TL::oG) + 8 * KN * half, lane);
            chain_release<DK, NB, CL>(base + L::bars, c, nch, wait, lane);
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    pr[n][i] += ur[n][i];
                    pi[n][i] = -(pi[n][i] + ui[n][i]);
                }
            if (odd) {
                put_nan(pr, off | both(out >> 16), lane, 8 * half);
                put_nan(pi, off | both(out >> 16), lane, 8 * half);
            }
            const size_t to = at + (L::KSP > 1 ? 8 * half * step : 0);
            store_rows(static_cast<T *>(a.o) + to, pr, step, left - 8 * half);
            if (a.o_im) store_rows(static_cast<T *>(a.o_im) + to, pi, step, left - 8 * half);
        }
        if (a.S_T) state_to_memory<KN>(st, a.S_T + state_at, a.dv);
    }
    if (chain_end<DK, NB, CL>(smem, tmem, wait, tid)) {          // NaN for all of this CTA's results
        const float nan = __int_as_float(0x7fc00000);
#pragma unroll 1
        for (size_t i = tid; i < (size_t)a.T * NB; i += L::threads) {
            const size_t at = (row0 + i / NB * a.H) * a.dv + c0 + i % NB;
            st_val(static_cast<T *>(a.o), at, nan);
            if (a.o_im) st_val(static_cast<T *>(a.o_im), at, nan);
        }
#pragma unroll 1
        for (int i = tid; a.S_T && i < DK * NB; i += L::threads) a.S_T[((size_t)bh * DK + i / NB) * a.dv + c0 + i % NB] = nan;
    }
}

template <int DK, int NB, int CL, typename T>
cudaError_t launch_nb(const ForwardArgs &x, cudaStream_t stream)
{
    using L = Chain<DK, NB, CL>;
    FwdArgsDev a;
    a.q = x.q; a.k = x.k; a.v = x.v; a.alpha = x.alpha; a.theta = x.theta; a.beta = x.beta; a.S0 = x.S0;
    a.o = x.o; a.o_im = x.o_im; a.S_T = x.S_T;
    a.T = x.T; a.H = x.H; a.dv = x.d_v;
    a.wait_ticks = wait_limit();
    return launch_clusters(sfda_forward_f32_kernel<DK, NB, CL, T>, a, dim3((unsigned)(x.B * x.H), x.d_v / NB), CL, L::threads, L::bytes, stream);
}

// A sequence of one chunk, or of up to four where the blocks have 64 columns anyway, takes blocks of 64 without a cluster: there is
// little or nothing to share, and a cluster's start, its two meetings and the copies cost 1 to 2 us.  74 sequences, d_v = 128:
// 14.2 -> 12.5 us at T = 16, 20.6 -> 18.9 at 48, 24.1 -> 23.0 at 64; one sequence of 16 tokens 11.8 -> 11.6; with blocks of 32 columns
// clusters are better from two chunks on (T = 48: 16.5 us, 18.6 without).
template <int DK, typename T>
cudaError_t launch_typed(const ForwardArgs &x, cudaStream_t stream)
{
    Blocks b = chain_blocks((long long)x.B * x.H, x.d_v);
    if (b.cluster > 1 && x.T <= (b.columns == 64 ? 4 * kC : kC)) b = {64, 1};
    if (b.columns == 128) return launch_nb<DK, 128, 1, T>(x, stream);
    if (b.columns == 64) return b.cluster == 2 ? launch_nb<DK, 64, 2, T>(x, stream) : launch_nb<DK, 64, 1, T>(x, stream);
    return b.cluster == 4 ? launch_nb<DK, 32, 4, T>(x, stream) : launch_nb<DK, 32, 2, T>(x, stream);
}

}  // namespace

cudaError_t launch_forward_f32(const ForwardArgs &a, cudaStream_t stream, int *launches)
{
    cudaError_t e;
    if (a.dtype == 1) e = a.d_k == 128 ? launch_typed<128, __nv_bfloat16>(a, stream) : launch_typed<64, __nv_bfloat16>(a, stream);
    else e = a.d_k == 128 ? launch_typed<128, float>(a, stream) : launch_typed<64, float>(a, stream);
    if (e == cudaSuccess && launches) ++*launches;
    return e;
}

}  // namespace sfda
