// fp32 chunk-WY forward for every supported d_k, d_v and dtype: the path of fp32 inputs and of the shapes the bf16
// tensor-core kernel does not take.  Same algebra as the other forwards (Theorem "Constructive left-to-right chunk-WY
// recursion", Eq. "apply-transfer", Theorem "Prefix outputs inside a chunk") in chunks of 16 tokens:
//
//   R = V - W^* S_0,  U = M R,  rho = Q^* S_0 + (A^{qk} D_beta) U,  o = conj(rho),  S_C = gamma_C S_0 + Y U
//
// One CTA per (batch, head) pair and block of value columns; sfda_chunk16.cuh describes the arithmetic (split fp16 on
// the tensor cores) and the two roles, which are pipelined over a ring of operand tiles.
//
// What bounds it: the latency of a chunk's dependent steps (scan, Gram products, inverse in the AUX warps; the three
// products in the chain warps), not memory.  B = 2, T = 2001, H = 16, d = 128, fp32: 3154 us with the CUDA-core
// kernel (an exponential per pair and coordinate, loops over shared memory), 665 us with this one; B = 1, T = 256,
// H = 2, d = 64: 201 -> 61 us.
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

template <int DK>
struct FwdSmem {
    static constexpr int stage = kSlots * Tile<DK>::bytes;
    static constexpr int small = stage + PrepSmem<DK>::stage_bytes;
    static constexpr int bytes = small + PrepSmem<DK>::small_bytes;
};

template <int DK, int NB, typename T>
__global__ void __launch_bounds__(kAux + 2 * NB, 1) sfda_forward_f32_kernel(const FwdArgsDev a)
{
    using TL = Tile<DK>;
    constexpr int kAll = kAux + 2 * NB;
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, bh = blockIdx.x, h = bh % a.H, b = bh / a.H, c0 = blockIdx.y * NB;
    const size_t row0 = (size_t)b * a.T * a.H + h;               // row of token t: row0 + t H
    const int nch = (a.T + kC - 1) / kC;

    if (tid < kAux) {
        if constexpr (NB == 128) asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        const int key = 8 * (tid >> 5) + ((tid & 31) >> 2), t4 = tid & 3;
        const T *q = static_cast<const T *>(a.q), *k = static_cast<const T *>(a.k);
        PrepIn in;
        prep_load<DK, T>(in, q, k, a.alpha, a.theta, a.beta, row0, a.H, 0, a.T, key, t4);
        for (int c = 0; c < nch; ++c) {
            const int slot = c % kSlots;
            if (c >= kSlots) bar_sync(kBarDone + slot, kAll);
            PrepIn next = in;
            if (c + 1 < nch) prep_load<DK, T>(next, q, k, a.alpha, a.theta, a.beta, row0, a.H, (c + 1) * kC, a.T, key, t4);
            PrepVals pv;
            prep_chunk<DK, true>(in, pv, smem + slot * TL::bytes, reinterpret_cast<float2 *>(smem + FwdSmem<DK>::stage),
                                 smem + FwdSmem<DK>::small, c & 1, tid);
            bar_arrive(kBarFull + slot, kAll);
            in = next;
        }
        return;
    }

    if constexpr (NB == 128) asm volatile("setmaxnreg.inc.sync.aligned.u32 176;");
    const int lane = tid & 31, w = (tid - kAux) >> 5, g = lane >> 2, t4 = lane & 3;
    const int col = c0 + 16 * w + g;                             // and col + 8
    const T *v = static_cast<const T *>(a.v);
    float sr[TL::KT][4], si[TL::KT][4];
#pragma unroll
    for (int n = 0; n < TL::KT; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const size_t at = ((size_t)bh * DK + 2 * (8 * n + 2 * t4 + (i & 1))) * a.dv + col + 8 * (i >> 1);
            sr[n][i] = a.S0 ? a.S0[at] : 0.f;
            si[n][i] = a.S0 ? a.S0[at + a.dv] : 0.f;
        }
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem);
    for (int c = 0; c < nch; ++c) {
        const int slot = c % kSlots;
        float rr[2][4], ri[2][4];
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int t = c * kC + 8 * n + 2 * t4 + (i & 1);
                rr[n][i] = t < a.T ? ld_val(v, (row0 + (size_t)t * a.H) * a.dv + col + 8 * (i >> 1)) : 0.f;
            }
        bar_sync(kBarFull + slot, kAll);
        const uint32_t tile = base + slot * TL::bytes;
        const float *inv = reinterpret_cast<const float *>(smem + slot * TL::bytes + TL::oS);
        float isv;
        const float ss = scale_for(__reduce_max_sync(0xffffffffu, max(max_bits4(sr), max_bits4(si))), isv);
        float acc[2][3][2][4];
        const uint32_t tiles[2] = {tile + TL::oW, tile + TL::oQ};
        product_over_keys<DK, 2, false>(acc, sr, si, ss, tiles, lane, nullptr);
        const float fw = isv * inv[0], fq = isv * inv[2];
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
        float ur[2][4], ui[2][4];
        product_small<false>(ur, ui, fr, fb, ir * inv[3]);
        const float iu = make_frag(fr, ur, ui);
        load_small<false>(fb, tile + TL::oA, lane);
        product_small<false>(rr, ri, fr, fb, iu * inv[4]);
        state_update<DK>(sr, si, fr, iu * inv[1], tile + TL::oY, reinterpret_cast<const float4 *>(smem + slot * TL::bytes + TL::oG), lane);
        if (c + kSlots < nch) bar_arrive(kBarDone + slot, kAll);
        T *o = static_cast<T *>(a.o), *oi = static_cast<T *>(a.o_im);
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int t = c * kC + 8 * n + 2 * t4 + (i & 1);
                if (t < a.T) {
                    const size_t at = (row0 + (size_t)t * a.H) * a.dv + col + 8 * (i >> 1);
                    st_val(o, at, fmaf(fq, acc[1][0][n][i], rr[n][i]));
                    if (oi) st_val(oi, at, -fmaf(fq, acc[1][1][n][i] - acc[1][2][n][i], ri[n][i]));
                }
            }
    }
    if (a.S_T) {
#pragma unroll
        for (int n = 0; n < TL::KT; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const size_t at = ((size_t)bh * DK + 2 * (8 * n + 2 * t4 + (i & 1))) * a.dv + col + 8 * (i >> 1);
                a.S_T[at] = sr[n][i];
                a.S_T[at + a.dv] = si[n][i];
            }
    }
}

template <int DK, int NB, typename T>
cudaError_t launch_nb(const ForwardArgs &x, cudaStream_t stream)
{
    auto kern = sfda_forward_f32_kernel<DK, NB, T>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, FwdSmem<DK>::bytes);
    if (e != cudaSuccess) return e;
    FwdArgsDev a;
    a.q = x.q; a.k = x.k; a.v = x.v; a.alpha = x.alpha; a.theta = x.theta; a.beta = x.beta; a.S0 = x.S0;
    a.o = x.o; a.o_im = x.o_im; a.S_T = x.S_T;
    a.T = x.T; a.H = x.H; a.dv = x.d_v;
    kern<<<dim3((unsigned)(x.B * x.H), (unsigned)(x.d_v / NB)), kAux + 2 * NB, FwdSmem<DK>::bytes, stream>>>(a);
    return cudaGetLastError();
}

// Value columns per CTA: all of them when the (batch, head) pairs fill the SMs, halved (down to 32) while the grid
// still fits: every block of columns repeats the chunk preparation, which runs beside the chain.
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
