// sw_ramp.cu -- ramp filter and positive/negative split of the projections
// for the ramp-filtered sliced W2 (Sec. 2.1 "High-pass filter (optional)",
// Eq. 1d_ift_ramp and Eq. line_decomp; the negative part is taken as the
// absolute value max(-mu~, 0), as in the appendix on ramp-filtered
// distances, and each part is normalised later by its own mass).
//
// Each projection row U[0..B) is filtered circularly on its bin grid:
//   Ut = IDFT_B( |xi_j| DFT_B(U) ),  |xi_j| = min(j, B - j),
// then split into Ut+ = max(Ut, 0) and Ut- = max(-Ut, 0).
//
// Design (GB300): one CTA per image; rows are taken 2*nsig at a time, two
// real rows packed into one complex signal.  The filter is real and even, so
// filtering the packed signal filters both rows at once (the real part holds
// one filtered row, the imaginary part the other): forward FFT, scale by
// |xi_j| / B, inverse FFT, all in shared memory with the Stockham FFT.
#include "sw_forms.h"
#include "sw_internal.cuh"

namespace swk {
namespace {

constexpr int kRampThreads = 256;
#ifndef RAMP_NSIG_MAX
#define RAMP_NSIG_MAX 8
#endif

// PAIRS: FFT stages in pairs (ramp_pairs: rows of 128 bins and more).  LANES:
// threads that copy a row, 16 for rows of at most 16 bins (1500 images at n =
// 360, B = 10: 165 us by warps, 128 us so; the index arithmetic of a run-time choice
// cost 13% at B = 120).
template <int nsig, bool PAIRS, int LANES = 32>
__global__ void __launch_bounds__(kRampThreads, PAIRS ? 4 : 8)
k_ramp(const float *__restrict__ proj, int nh, int B, FftPlan plan,
       const float2 *__restrict__ tw, float *__restrict__ parts)
{
    extern __shared__ float2 smr[];
    float2 *b0 = smr;
    float2 *b1 = b0 + B * nsig;
    float2 *tws = b1 + B * nsig;                            // [B]
    float *tile = reinterpret_cast<float *>(tws + B);       // [2 nsig][B + 1] rows of the chunk
    chain_wait();
    const int TS = B + 1;  // odd row stride (B is even): column reads hit distinct banks
    for (int i = threadIdx.x; i < B; i += blockDim.x) tws[i] = tw[i];
    const int grp = threadIdx.x / LANES, lane = threadIdx.x % LANES;
    constexpr int ngrp = kRampThreads / LANES;
    const int img = blockIdx.x;
    const float *U = proj + (size_t)img * nh * B;
    float *Pp = parts + (size_t)img * 2 * nh * B;  // part 0 (positive)
    float *Pm = Pp + (size_t)nh * B;                // part 1 (negative)
    const float invB = 1.f / (float)B;
    for (int r0 = 0; r0 < nh; r0 += 2 * nsig) {
        const int rows = min(2 * nsig, nh - r0);
        // ---- load the chunk's rows (coalesced), then pack: signal s =
        // rows (2s, 2s + 1) as (re, im), element-major for the FFT
        // (no division by B per element)
        for (int r = grp; r < 2 * nsig; r += ngrp) {
            const float *row = U + (size_t)(r0 + r) * B;
#pragma unroll 4
            for (int b = lane; b < B; b += LANES) tile[r * TS + b] = r < rows ? __ldg(row + b) : 0.f;
        }
        __syncthreads();
        for (int t = threadIdx.x; t < B * nsig; t += blockDim.x) {
            const int b = t / nsig, sg = t % nsig;
            b0[t] = make_float2(tile[(2 * sg) * TS + b], tile[(2 * sg + 1) * TS + b]);
        }
        __syncthreads();
        float2 *X = fft_smem<nsig, -1, PAIRS>(b0, b1, plan, tws);
        float2 *Y = X == b0 ? b1 : b0;
        for (int t = threadIdx.x; t < B * nsig; t += blockDim.x) {
            const int j = t / nsig;
            const float w = (float)min(j, B - j) * invB;
            X[t] = make_float2(w * X[t].x, w * X[t].y);
        }
        __syncthreads();
        const float2 *R = fft_smem<nsig, +1, PAIRS>(X, Y, plan, tws);
        // ---- unpack to rows, then split and write (coalesced)
        for (int t = threadIdx.x; t < B * nsig; t += blockDim.x) {
            const int b = t / nsig, sg = t % nsig;
            const float2 v = R[t];
            tile[(2 * sg) * TS + b] = v.x;
            tile[(2 * sg + 1) * TS + b] = v.y;
        }
        __syncthreads();
        for (int r = grp; r < rows; r += ngrp) {
            float *pp = Pp + (size_t)(r0 + r) * B, *pm = Pm + (size_t)(r0 + r) * B;
#pragma unroll 4
            for (int b = lane; b < B; b += LANES) {
                const float v = tile[r * TS + b];
                pp[b] = fmaxf(v, 0.f);
                pm[b] = fmaxf(-v, 0.f);
            }
        }
        __syncthreads();
    }
}

}  // namespace

cudaError_t launch_ramp(const float *proj, int nb, int nh, int B, const FftPlan &plan,
                        const float2 *tw, float *parts, cudaStream_t st)
{
    if (nb <= 0) return cudaSuccess;
    if (plan.n != B) return cudaErrorInvalidValue;
    // the widest signal batch (up to RAMP_NSIG_MAX) whose buffers fit 200 KB
    auto smem_of = [&](int ns) {
        return sizeof(float2) * ((size_t)2 * B * ns + B) + sizeof(float) * (size_t)2 * ns * (B + 1);
    };
    int nsig = RAMP_NSIG_MAX;
    while (nsig > 2 && smem_of(nsig) > 200 * 1024) nsig /= 2;
    if (smem_of(nsig) > 200 * 1024) return cudaErrorInvalidValue;
    const size_t smem = smem_of(nsig);
#define SW_RAMP_LAUNCH(...)                                                                    \
    do {                                                                                      \
        cudaFuncSetAttribute(k_ramp<__VA_ARGS__>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                             200 * 1024);                                                     \
        return launch_chained(k_ramp<__VA_ARGS__>, dim3(nb), dim3(kRampThreads), smem, st, 1, \
                              proj, nh, B, plan, tw, parts);                                  \
    } while (0)
    if (nsig == 16) SW_RAMP_LAUNCH(16, true);
    else if (nsig == 8 && B <= 16) SW_RAMP_LAUNCH(8, false, 16);
    else if (nsig == 8 && !ramp_pairs(B)) SW_RAMP_LAUNCH(8, false);
    else if (nsig == 8) SW_RAMP_LAUNCH(8, true);
    else if (nsig == 4) SW_RAMP_LAUNCH(4, true);
    else SW_RAMP_LAUNCH(2, true);
#undef SW_RAMP_LAUNCH
}

}  // namespace swk
