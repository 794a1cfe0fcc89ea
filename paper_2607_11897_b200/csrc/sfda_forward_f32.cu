// fp32 chunk-WY forward for every supported d_k, d_v and dtype: the path of fp32 inputs and of the shapes the bf16
// tensor-core kernel does not take.  Same algebra as the other forwards (Theorem "Constructive left-to-right chunk-WY
// recursion", Eq. "apply-transfer", Theorem "Prefix outputs inside a chunk") in chunks of 16 tokens:
//
//   R = V - W^* S_0,  U = M R,  rho = Q^* S_0 + (A^{qk} D_beta) U,  o = conj(rho),  S_C = gamma_C S_0 + Y U
//
// One CTA per (batch, head) pair and block of value columns; sfda_chunk16.cuh describes the arithmetic (split fp16 on
// the tensor cores) and the two roles, which are pipelined over a ring of operand tiles.
//
// What bounds it: the schedulers' issue slots, which mma.sync holds (see ChainRoles), and the latency of the chain.
// B = 2, T = 2001, H = 16, d = 128, fp32: 457 us, 6.9 k cycles per 16 tokens with 32 value columns per CTA (the unrolled first
// version 665 us, the CUDA-core kernel 3154 us); B = 1, T = 256, H = 2, d = 64: 39 us (61, 201).
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
};

template <int DK, int NB, typename T>
__global__ void __launch_bounds__(ChainRoles<DK, NB>::threads, 1) sfda_forward_f32_kernel(const FwdArgsDev a)
{
    using TL = Tile<DK>;
    using L = ChainSmem<DK, NB>;
    constexpr int kChain = 2 * NB, kPrepWarps = ChainRoles<DK, NB>::prep_warps, kPrep = ChainRoles<DK, NB>::kPrep;
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, bh = blockIdx.x, h = bh % a.H, b = bh / a.H, c0 = blockIdx.y * NB;
    const size_t row0 = (size_t)b * a.T * a.H + h;               // row of token t: row0 + t H
    const int nch = (a.T + kC - 1) / kC;
    if (tid < 32) tm_alloc(reinterpret_cast<uint32_t *>(smem + L::slow), L::columns);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *reinterpret_cast<const uint32_t *>(smem + L::slow);
    __syncthreads();

    const ChainRoles<DK, NB> role(tid);
    if (role.prep >= 0) {
        // register shares with all 128 value columns: 256 x 88 + 128 x 72 + 256 x 112 of the launch's 640 x 96
        if constexpr (NB == 128) asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
        const T *q = static_cast<const T *>(a.q), *k = static_cast<const T *>(a.k);
        PrepRaw<L::PM::TPT, T> in;
        prep_fetch<DK, kPrepWarps, T>(in, q, k, a.alpha, a.theta, a.beta, row0, a.H, 0, a.T, true, role.prep);
        for (int c = 0; c < nch; ++c) {
            const int slot = c % kSlots;
            if (c >= kSlots) bar_sync(kBarDone + slot, kPrep + kChain);
            PrepRaw<L::PM::TPT, T> next;
            prep_fetch<DK, kPrepWarps, T>(next, q, k, a.alpha, a.theta, a.beta, row0, a.H, (c + 1) * kC, a.T, true, role.prep);
            float2 *gk = reinterpret_cast<float2 *>(smem + L::gram + slot * L::gram_bytes);
            if (!prep_chunk<DK, kPrepWarps, kBarAux, T>(in, q, k, a.alpha, a.theta, a.beta, row0, a.H, c * kC, a.T, nullptr, smem + slot * TL::bytes,
                                                        smem + L::kb + slot * TL::BIG, smem + L::scan, true, role.prep))
                slow_gram<DK, kPrepWarps, kBarAux, T>(q, k, a.alpha, a.theta, a.beta, row0, a.H, c * kC, a.T, smem + L::slow, smem + L::scan,
                                                   gk, gk + 16 * 17, true, role.prep);
            bar_arrive(kBarPlanes + slot, kPrep + 64);
            in = next;
        }
    } else if (role.solve >= 0) {
        // warps 0, 1: the system's inverse of even / odd chunks; warps 2, 3: the outputs' Gram matrix of them
        if constexpr (NB == 128) asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
        const int lane = tid & 31, w = role.solve >> 5, out = w >> 1;
        const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem);
        for (int c = w & 1; c < nch; c += 2) {
            const int slot = c % kSlots;
            unsigned char *tile = smem + slot * TL::bytes;
            float *inv = reinterpret_cast<float *>(tile + TL::oS);
            float2 *gm = reinterpret_cast<float2 *>(smem + L::gram + slot * L::gram_bytes) + out * 16 * 17;
            bar_sync(kBarPlanes + slot, kPrep + 64);
            if (reinterpret_cast<const int *>(inv)[6])
                gram_tiles<DK, 2>(base + slot * TL::bytes + (out ? TL::oQ : TL::oW), base + L::kb + slot * TL::BIG, inv[out ? 2 : 0] * inv[5], gm, 0, lane);
            __syncwarp();
            if (!out) invert_unit_lower16(gm, lane);
            store_lower(tile + (out ? TL::oA : TL::oM), gm, inv + 3 + out, lane);
            bar_arrive(kBarFull + slot, 64 + kChain);
        }
    } else if (role.chain >= 0) {
        if constexpr (NB == 128) asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
        const int lane = tid & 31, w = role.chain >> 5, g = lane >> 2, t4 = lane & 3;
        const int col = c0 + 16 * w + g;                         // and col + 8
        const uint32_t st = tmem + ((uint32_t)(w & 3) << 21) + (w >> 2) * 8 * TL::KT;    // this warp's lanes and columns
        const size_t state_at = ((size_t)bh * DK + 4 * t4) * a.dv + col;
        float2 largest = state_from_memory<DK>(st, a.S0 ? a.S0 + state_at : nullptr, a.dv);
        const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem);
        const size_t step = (size_t)a.H * a.dv;
        size_t at = (row0 + (size_t)(2 * t4) * a.H) * a.dv + col;
        for (int c = 0; c < nch; ++c, at += 16 * step) {
            const int slot = c % kSlots, left = a.T - c * kC - 2 * t4;
            float rr[2][4], ri[2][4];
            load_rows(rr, static_cast<const T *>(a.v) + at, step, left);
            const RowScale sr = row_scale<4>(largest);
            bar_sync(kBarFull + slot, 64 + kChain);
            const uint32_t tile = base + slot * TL::bytes;
            const float *inv = reinterpret_cast<const float *>(smem + slot * TL::bytes + TL::oS);
            float acc[2][2][2][4];
            const uint32_t tiles[2] = {tile + TL::oW, tile + TL::oQ};
            keys_product<DK, 2>(acc, st, sr, tiles, lane, [](int, const uint32_t(&)[4], const uint32_t(&)[4], const uint32_t(&)[4], const uint32_t(&)[4]) {});
            const float fw[2] = {sr.inv[0] * inv[0], sr.inv[1] * inv[0]}, fq[2] = {sr.inv[0] * inv[2], sr.inv[1] * inv[2]};
            uint32_t off = take_out(rr);                         // tokens whose v is not finite; below, all behind them too
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    rr[n][i] = fmaf(-fw[i >> 1], acc[0][0][n][i], rr[n][i]);
                    ri[n][i] = -fw[i >> 1] * acc[0][1][n][i];
                }
            TokFrag fr;
            RowScale ru;
#pragma unroll 1
            for (int pass = 0; pass < 2; ++pass) {               // U = M R, then (A^{qk} D_beta) U
                TokFrag fb;
                ru = make_frag(fr, rr, ri);
                load_small<false>(fb, tile + (pass ? TL::oA : TL::oM), lane);
                product_small<false>(rr, ri, fr, fb, ru.inv, inv[3 + pass]);
            }
            const uint32_t out = reinterpret_cast<const uint32_t *>(inv)[7];
            const bool odd = __any_sync(0xffffffffu, (off | out) != 0);
            if (odd) {
                off = every_lanes(off, lane);
                off = from_first(off & 0xffffu) | from_first(off >> 16) << 16 | both(from_first(out & 0xffffu));
                put_nan(ru.inv, off);
            }
            largest = state_update<DK>(st, fr, ru.inv, inv[1], tile + TL::oY, reinterpret_cast<const float4 *>(smem + slot * TL::bytes + TL::oG), lane);
            if (c + kSlots < nch) bar_arrive(kBarDone + slot, kPrep + kChain);
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    rr[n][i] = fmaf(fq[i >> 1], acc[1][0][n][i], rr[n][i]);
                    ri[n][i] = -fmaf(fq[i >> 1], acc[1][1][n][i], ri[n][i]);
                }
            if (odd) {
                put_nan(rr, off | both(out >> 16), lane);
                put_nan(ri, off | both(out >> 16), lane);
            }
            store_rows(static_cast<T *>(a.o) + at, rr, step, left);
            if (a.o_im) store_rows(static_cast<T *>(a.o_im) + at, ri, step, left);
        }
        if (a.S_T) state_to_memory<DK>(st, a.S_T + state_at, a.dv);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid < 32) tm_free(tmem, L::columns);
}

template <int DK, int NB, typename T>
cudaError_t launch_nb(const ForwardArgs &x, cudaStream_t stream)
{
    auto kern = sfda_forward_f32_kernel<DK, NB, T>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, ChainSmem<DK, NB>::bytes);
    if (e != cudaSuccess) return e;
    FwdArgsDev a;
    a.q = x.q; a.k = x.k; a.v = x.v; a.alpha = x.alpha; a.theta = x.theta; a.beta = x.beta; a.S0 = x.S0;
    a.o = x.o; a.o_im = x.o_im; a.S_T = x.S_T;
    a.T = x.T; a.H = x.H; a.dv = x.d_v;
    kern<<<dim3((unsigned)(x.B * x.H), (unsigned)(x.d_v / NB)), ChainRoles<DK, NB>::threads, ChainSmem<DK, NB>::bytes, stream>>>(a);
    return cudaGetLastError();
}

// Value columns per CTA: all of them when the (batch, head) pairs fill the SMs, halved (down to 32) while the grid
// still fits: every block of columns repeats the chunk preparation, which runs beside the chain.  (148: the SMs of a B200.
// On another device the blocks are merely not the best ones.)
template <int DK, typename T>
cudaError_t launch_typed(const ForwardArgs &x, cudaStream_t stream)
{
    int nb = x.d_v;
    while (nb > 32 && (long long)x.B * x.H * (x.d_v / (nb / 2)) <= 148) nb /= 2;
    if (nb == 128) return launch_nb<DK, 128, T>(x, stream);
    if (nb == 64) return launch_nb<DK, 64, T>(x, stream);
    return launch_nb<DK, 32, T>(x, stream);
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
