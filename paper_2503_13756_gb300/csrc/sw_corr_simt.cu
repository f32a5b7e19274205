// sw_corr_simt.cu -- FP32 correlation of angle spectra on the CUDA cores:
// the "products summed over rows" step of the FFT cross-correlation of
// Sec. 2.3 ("Fast computation over rotations"), written as one complex
// product-sum per frequency and pair:
//   C_ij(k') = sum_p Qhat_i(k', p) conj(Qhat_j(k', p))
//            = sum_p (a_i a_j + b_i b_j) + i (b_i a_j - a_i b_j),  Qhat = a + i b.
// This is a batched GEMM over frequencies; the FP32 path keeps it on FFMA
// so that the accumulation is full single precision.
//
// Design: 64 x 64 pair tile per CTA, 4 x 4 pairs per thread, levels staged
// 16 at a time in shared memory (transposed so that each thread reads four
// consecutive queries or templates as one float4), register double-buffer
// of the next stage.
#include <algorithm>

#include "sw_forms.h"
#include "sw_internal.cuh"

namespace swk {
namespace {

constexpr int TM = 64, TN = 64, KP = 16;

__global__ void __launch_bounds__(256)
k_corr_simt(const float *__restrict__ X, size_t xf, const float *__restrict__ Y, size_t yf,
            int Nq, int Nt, int M, float2 *__restrict__ C)
{
    __shared__ __align__(16) float qa[KP][TM], qb[KP][TM], ta[KP][TN], tb[KP][TN];
    chain_wait();
    const int f = blockIdx.z;
    const int i0 = blockIdx.y * TM, j0 = blockIdx.x * TN;
    const float *Xf = X + (size_t)f * xf;
    const float *Yf = Y + (size_t)f * yf;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    // loader mapping: row r = t / 4 (0..63), levels (t % 4) * 4 .. +3
    const int lr = threadIdx.x >> 2, lp = (threadIdx.x & 3) * 4;
    const int gi = i0 + lr, gj = j0 + lr;
    const float *xrow = gi < Nq ? Xf + (size_t)gi * 2 * M : nullptr;
    const float *yrow = gj < Nt ? Yf + (size_t)gj * 2 * M : nullptr;

    float vqa[4], vqb[4], vta[4], vtb[4];
    auto fetch = [&](int p0) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int p = p0 + lp + u;
            const bool okp = p < M;
            vqa[u] = (xrow && okp) ? __ldg(xrow + p) : 0.f;
            vqb[u] = (xrow && okp) ? __ldg(xrow + M + p) : 0.f;
            vta[u] = (yrow && okp) ? __ldg(yrow + p) : 0.f;
            vtb[u] = (yrow && okp) ? __ldg(yrow + M + p) : 0.f;
        }
    };

    float re[4][4], im[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) re[a][b] = im[a][b] = 0.f;

    fetch(0);
    for (int p0 = 0; p0 < M; p0 += KP) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            qa[lp + u][lr] = vqa[u];
            qb[lp + u][lr] = vqb[u];
            ta[lp + u][lr] = vta[u];
            tb[lp + u][lr] = vtb[u];
        }
        __syncthreads();
        if (p0 + KP < M) fetch(p0 + KP);
#pragma unroll
        for (int p = 0; p < KP; ++p) {
            const float4 xa = *reinterpret_cast<const float4 *>(&qa[p][ty * 4]);
            const float4 xb = *reinterpret_cast<const float4 *>(&qb[p][ty * 4]);
            const float4 ya = *reinterpret_cast<const float4 *>(&ta[p][tx * 4]);
            const float4 yb = *reinterpret_cast<const float4 *>(&tb[p][tx * 4]);
            const float A[4] = {xa.x, xa.y, xa.z, xa.w}, Bq[4] = {xb.x, xb.y, xb.z, xb.w};
            const float Ca[4] = {ya.x, ya.y, ya.z, ya.w}, Cb[4] = {yb.x, yb.y, yb.z, yb.w};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    re[a][b] = fmaf(A[a], Ca[b], fmaf(Bq[a], Cb[b], re[a][b]));
                    im[a][b] = fmaf(Bq[a], Ca[b], fmaf(-A[a], Cb[b], im[a][b]));
                }
        }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int i = i0 + ty * 4 + a;
        if (i >= Nq) continue;
        float2 *crow = C + ((size_t)f * Nq + i) * Nt;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int j = j0 + tx * 4 + b;
            if (j < Nt) crow[j] = make_float2(re[a][b], im[a][b]);
        }
    }
}

// A few pairs (a single pair above all): one thread per frequency and pair, in
// the tile kernel's order of operations.  Where the 64 x 64 tile is nearly
// all padding its time is the latency of its stages (a pair at n = 360, M =
// 128: 31 us); here a CTA copies the rows of `fb` frequencies to shared memory
// at once and each thread runs one chain of 2 M dependent FMAs per component
// (8 us).  Rows are 2 M floats; a frequency's rows take an odd number of
// floats, so that the threads of adjacent frequencies read distinct banks.
__global__ void __launch_bounds__(256)
k_corr_few(const float *__restrict__ X, size_t xf, const float *__restrict__ Y, size_t yf, int Nq,
           int Nt, int M, int nf, int fb, float2 *__restrict__ C)
{
    extern __shared__ float sm[];
    chain_wait();
    const int M2 = 2 * M, rows = Nq + Nt, FS = rows * M2 + 1;
    const int f0 = blockIdx.x * fb, nb = min(fb, nf - f0);
    for (int fl = 0; fl < nb; ++fl) {
        const float *Xf = X + (size_t)(f0 + fl) * xf, *Yf = Y + (size_t)(f0 + fl) * yf;
#pragma unroll 4
        for (int e = threadIdx.x; e < rows * M2; e += blockDim.x)
            sm[fl * FS + e] = e < Nq * M2 ? __ldg(Xf + e) : __ldg(Yf + e - Nq * M2);
    }
    __syncthreads();
    const int pairs = Nq * Nt;
    for (int t = threadIdx.x; t < nb * pairs; t += blockDim.x) {
        const int fl = t / pairs, pr = t % pairs, i = pr / Nt, j = pr % Nt;
        const float *x = sm + fl * FS + i * M2, *y = sm + fl * FS + (Nq + j) * M2;
        float re = 0.f, im = 0.f;
#pragma unroll 8
        for (int p = 0; p < M; ++p) {
            const float a = x[p], b = x[M + p], c = y[p], d = y[M + p];
            re = fmaf(a, c, fmaf(b, d, re));
            im = fmaf(b, c, fmaf(-a, d, im));
        }
        C[((size_t)(f0 + fl) * Nq + i) * Nt + j] = make_float2(re, im);
    }
}

}  // namespace

cudaError_t launch_corr_simt(const float *X, size_t xf, const float *Y, size_t yf, int Nq,
                             int Nt, int M, int nf, float2 *C, cudaStream_t st)
{
    if (Nq <= 0 || Nt <= 0 || nf <= 0) return cudaSuccess;
    // few pairs: frequencies per CTA so that its rows fit 48 KB and the chip
    // has a CTA or two per SM (see k_corr_few).  Few and tile form in us, at n =
    // 360, M = 256: 1 x 1 9 and 57, 4 x 4 17 and 57, 8 x 8 26 and 57, 16 x 4 28 and 57, 4
    // x 16 34 and 57; at n = 256, M = 32 5 to 8 and 8; at n = 60, M = 16 5 to 6 and 6.
    const DeviceForm *dev;
    const cudaError_t e = device_form(&dev);
    if (e != cudaSuccess) return e;
    const size_t per_f = sizeof(float) * ((size_t)(Nq + Nt) * 2 * M + 1);
    if (Nq <= 16 && Nt <= 16 && Nq * Nt <= 64 && per_f <= 48 * 1024) {
        const int fb = (int)std::max<size_t>(
            1, std::min<size_t>({48 * 1024 / per_f, (size_t)((nf + dev->sms - 1) / dev->sms), (size_t)8}));
        return launch_chained(k_corr_few, dim3((nf + fb - 1) / fb), dim3(256), per_f * fb, st, 1, X,
                              xf, Y, yf, Nq, Nt, M, nf, fb, C);
    }
    dim3 grid((Nt + TN - 1) / TN, (Nq + TM - 1) / TM, nf);
    return launch_chained(k_corr_simt, grid, dim3(256), 0, st, 1, X, xf, Y, yf, Nq, Nt, M, C);
}

}  // namespace swk
