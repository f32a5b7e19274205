// sw_spectrum.cu -- angle spectra of the quantile functions: the first half
// of the FFT cross-correlation of Sec. 2.3 ("Fast computation over
// rotations": the correlation along angle of every row of U_I and V_I is
// computed with the FFT), plus the translation centring.
//
// For level p, the quantiles u_pk (k = 0..n-1) are transformed over k:
//   Qhat(k', p) = sum_k u~_pk e^{-2 pi i k k'/n},  u~_pk = u_pk - <a, theta_k>,
// with a = (2/n) sum_k ubar_k theta_k.  Centring only changes k' = 1 (and
// n-1): Qhat(1, p) -= c1 with c1 = mean_p Qhat_u(1, p) = (n/2)(a_x - i a_y),
// so it is applied after the transform with no second pass over the data.
// The k' = 0 term (n times the mean over angle of each level, the "profile")
// is kept apart, so that the rotation-invariant part of the distance is
// computed later as a direct difference instead of a cancelling sum.
//
// Design (GB300): one CTA per image, or a cluster of them when there are few;
// levels are taken 2*nsig at a time, two
// real levels packed into one complex signal, FFT'd by the shared-memory
// Stockham FFT and unpacked by Hermitian symmetry.  The batches are staged
// by cp.async into two buffers, so that batch b + 1 is in flight while batch
// b is transformed and written.  Norms are compensated FP32 sums.
// Optional BF16/FP16 copies feed the tensor-core GEMM, with their norms taken
// from the rounded values so that self-distances cancel.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "sw_forms.h"
#include "sw_internal.cuh"

namespace swk {
namespace {

namespace cg = cooperative_groups;

template <typename T>
__device__ __forceinline__ T to_lp(float x);
template <>
__device__ __forceinline__ __nv_bfloat16 to_lp<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }
template <>
__device__ __forceinline__ __half to_lp<__half>(float x) { return __float2half_rn(x); }
template <typename T>
__device__ __forceinline__ float from_lp(T x);
template <>
__device__ __forceinline__ float from_lp<__nv_bfloat16>(__nv_bfloat16 x) { return __bfloat162float(x); }
template <>
__device__ __forceinline__ float from_lp<__half>(__half x) { return __half2float(x); }

struct SpecOut {
    float *spec32;
    size_t fstride;
    void *lp_q;
    size_t lpq_fstride;
    void *lp_t;
    size_t lpt_fstride;
    int Nq;
    int ldk;    // low-precision segment length (>= 2M, zero padded)
    int lp;     // write low-precision copies (queries to lp_q, templates to lp_t)
    int split;  // FP16 hi/lo split: rows of 2 segments [hi | lo]
};

// Compensated (Kahan) sum of nonnegative terms, kept as (sum, -compensation):
// the value is a.hi + a.lo, within about 2 ulp of the exact sum.
__device__ __forceinline__ void kahan_add(DF &a, float x)
{
    const float y = x + a.lo;
    const float t = a.hi + y;
    a.lo = y - (t - a.hi);
    a.hi = t;
}

// Writes Qhat(kf, p) (kf >= 1) for image img and returns its |.|^2 (weight w)
// for the norm: of the low-precision values where the GEMM sees only those
// (BF16, FP16), of the FP32 values otherwise.
template <typename T>
__device__ __forceinline__ float emit(const SpecOut &o, int img, int M, int kf, int p, float2 X,
                                      float w)
{
    const float term = w * fmaf(X.x, X.x, X.y * X.y);
    if (!o.lp) {
        float *row = o.spec32 + (size_t)(kf - 1) * o.fstride + (size_t)img * 2 * M;
        row[p] = X.x;
        row[M + p] = X.y;
        return term;
    }
    const T re = to_lp<T>(X.x), im = to_lp<T>(X.y);
    const float rf = from_lp<T>(re), imf = from_lp<T>(im);
    const T nim = to_lp<T>(-imf);
    const bool tmpl = img >= o.Nq;
    const int seg = o.ldk;                     // one [re|im|0] segment
    const int row_len = o.split ? 2 * seg : seg;
    T *r = tmpl ? reinterpret_cast<T *>(o.lp_t) + (size_t)(kf - 1) * o.lpt_fstride +
                      (size_t)(2 * (img - o.Nq)) * row_len
                : reinterpret_cast<T *>(o.lp_q) + (size_t)(kf - 1) * o.lpq_fstride +
                      (size_t)img * row_len;
    if (!o.split) {
        r[p] = re;
        r[M + p] = im;
        if (tmpl) {
            r[row_len + p] = nim;  // row 2j+1: [ -im | re | 0 ]
            r[row_len + M + p] = re;
        }
        return w * fmaf(rf, rf, imf * imf);
    }
    // FP16 split: lo = x - hi, exact in FP32, rounded to FP16; rows [hi | lo]
    // (the correlation reads segments hi hi, hi lo, lo hi of its operands)
    const T rel = to_lp<T>(X.x - rf), iml = to_lp<T>(X.y - imf);
    r[p] = re;
    r[M + p] = im;
    r[seg + p] = rel;
    r[seg + M + p] = iml;
    if (tmpl) {  // row 2j+1: [-im | re]
        const T nrel = to_lp<T>(-(X.y - imf));
        T *r2 = r + row_len;
        r2[p] = nim;
        r2[M + p] = re;
        r2[seg + p] = nrel;
        r2[seg + M + p] = rel;
    }
    return term;
}

// Two values as one packed pair of the type, and back.
template <typename T>
struct Pair2;
template <>
struct Pair2<__half> {
    using V = __half2;
    static __device__ __forceinline__ V pack(float a, float b) { return __floats2half2_rn(a, b); }
    static __device__ __forceinline__ float2 unpack(V v) { return __half22float2(v); }
};
template <>
struct Pair2<__nv_bfloat16> {
    using V = __nv_bfloat162;
    static __device__ __forceinline__ V pack(float a, float b) { return __floats2bfloat162_rn(a, b); }
    static __device__ __forceinline__ float2 unpack(V v) { return __bfloat1622float2(v); }
};

// emit for the two levels pa (even) and pa + 1 of one frequency at once, M
// even: every row segment then takes the pair as one 4-byte store (FP32
// rows: one 8-byte store), the same values as two emit calls.
template <typename T>
__device__ __forceinline__ float2 emit2(const SpecOut &o, int img, int M, int kf, int pa,
                                        float2 Xa, float2 Xb, float w)
{
    const float2 term = make_float2(w * fmaf(Xa.x, Xa.x, Xa.y * Xa.y),
                                    w * fmaf(Xb.x, Xb.x, Xb.y * Xb.y));
    if (!o.lp) {
        float *row = o.spec32 + (size_t)(kf - 1) * o.fstride + (size_t)img * 2 * M;
        *reinterpret_cast<float2 *>(row + pa) = make_float2(Xa.x, Xb.x);
        *reinterpret_cast<float2 *>(row + M + pa) = make_float2(Xa.y, Xb.y);
        return term;
    }
    using P = Pair2<T>;
    using V = typename P::V;
    const V re2 = P::pack(Xa.x, Xb.x), im2 = P::pack(Xa.y, Xb.y);  // (pa, pa + 1)
    const float2 rf = P::unpack(re2), imf = P::unpack(im2);
    const bool tmpl = img >= o.Nq;
    const int seg = o.ldk;
    const int row_len = o.split ? 2 * seg : seg;
    T *r = tmpl ? reinterpret_cast<T *>(o.lp_t) + (size_t)(kf - 1) * o.lpt_fstride +
                      (size_t)(2 * (img - o.Nq)) * row_len
                : reinterpret_cast<T *>(o.lp_q) + (size_t)(kf - 1) * o.lpq_fstride +
                      (size_t)img * row_len;
    auto put = [](T *dst, V v) { *reinterpret_cast<V *>(dst) = v; };
    if (!o.split) {
        put(r + pa, re2);
        put(r + M + pa, im2);
        if (tmpl) {
            put(r + row_len + pa, __hneg2(im2));  // row 2j+1: [ -im | re | 0 ]
            put(r + row_len + M + pa, re2);
        }
        return make_float2(w * fmaf(rf.x, rf.x, imf.x * imf.x),
                           w * fmaf(rf.y, rf.y, imf.y * imf.y));
    }
    // FP16 split: lo = x - hi, exact in FP32, rounded to FP16
    const V rel2 = P::pack(Xa.x - rf.x, Xb.x - rf.y);
    const V iml2 = P::pack(Xa.y - imf.x, Xb.y - imf.y);
    put(r + pa, re2);  // [hi | lo]
    put(r + M + pa, im2);
    put(r + seg + pa, rel2);
    put(r + seg + M + pa, iml2);
    if (tmpl) {  // row 2j+1: [-im | re] (rounding is symmetric)
        T *r2 = r + row_len;
        put(r2 + pa, __hneg2(im2));
        put(r2 + M + pa, re2);
        put(r2 + seg + pa, __hneg2(iml2));
        put(r2 + seg + M + pa, rel2);
    }
    return term;
}

__device__ __forceinline__ void cpa16(void *dst, const void *src, int src_bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(__cvta_generic_to_global(src)), "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cpa4(void *dst, const void *src, int src_bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(__cvta_generic_to_global(src)), "r"(src_bytes)
                 : "memory");
}

// Issue the copies of the level batch [p0, p0 + 2 nsig) of image qi into
// buf: signal s of angle k is buf[k nsig + s] = (level p0 + 2s, p0 + 2s + 1);
// levels past M are zero-filled.  With whole groups of four levels per part
// every angle's slice is 16-byte chunks, each within one part; otherwise one
// 4-byte copy per level.
template <int nsig>
__device__ __forceinline__ void stage_levels(const float *__restrict__ qi, int n, int M, int Mp,
                                             int parts, int p0, float2 *buf)
{
    if ((Mp & 3) == 0) {
        constexpr int CH = nsig / 2;  // 16-byte chunks (4 levels) per angle
        for (int c = threadIdx.x; c < n * CH; c += blockDim.x) {
            const int k = c / CH, h = c % CH;
            const int p = p0 + 4 * h;
            const int valid = min(max(M - p, 0), 4);
            // level p of part p / Mp (the parts' arrays lie one after the other)
            const bool second = parts == 2 && p >= Mp;
            const float *src = valid ? qi + (size_t)(second ? n + k : k) * Mp + (second ? p - Mp : p)
                                     : qi;
            cpa16(buf + k * nsig + 2 * h, src, 4 * valid);
        }
    } else {
        for (int c = threadIdx.x; c < n * 2 * nsig; c += blockDim.x) {
            const int k = c / (2 * nsig), e = c % (2 * nsig);
            const int p = p0 + e;
            const float *src = qi;
            if (p < M)
                src = parts == 1 ? qi + (size_t)k * M + p
                                 : qi + (size_t)(p / Mp) * n * Mp + (size_t)k * Mp + p % Mp;
            cpa4(reinterpret_cast<float *>(buf + k * nsig) + e, src, p < M ? 4 : 0);
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// Forms.  The norm of an image is a sum of 256 Kahan sums, one per class c of
// terms: with NSC signals to a batch, signal c mod NSC of each batch at the
// frequencies k' = c / NSC + (256 / NSC) i in increasing order, batch after
// batch; every form keeps that order.
//  - plain: batches of NSC signals, one thread per class, three or four CTAs
//    per SM.
//  - HB: half batches of NSC / 2 signals, so half of the buffers and more CTAs on
//    an SM, for many images whose plain buffers leave room for fewer than three.
//    Lanes l and l + 16 of a warp take alternate frequencies of a class and
//    exchange their terms, so both hold its sum, and a thread keeps two classes,
//    one per half of the batch.  10,001 images at n = 512, M = 256: 5.2 ms plain
//    (one CTA of 8 warps per SM), 4.9 ms with 512 threads on full batches, 3.9 ms
//    in this form.
//  - CL: few images; the CTAs of a cluster share an image, CTA r taking the
//    level batches r, r + S, ...; the terms wait in shared memory, and after
//    the cluster's barrier CTA 0 adds them in order and finishes the image.
// Which one a launch takes is spectrum_form's choice (sw_forms.h).
template <typename T, int NSC, bool HB, bool CL, int CTAS = CL ? 2 : 3>
__global__ void __launch_bounds__(kSpecThreads, CTAS)
k_spectrum(const float *__restrict__ q, int n, int M, FftPlan plan, const float2 *__restrict__ tw,
           SpecOut o, float *__restrict__ prof, double *__restrict__ center,
           double *__restrict__ norm32, double *__restrict__ norm16, int parts,
           int *__restrict__ clear)
{
    constexpr int nsig = HB ? NSC / 2 : NSC;  // signals transformed at a time
    // M levels in all; with parts = 2 (ramp-filtered distance) the levels
    // [0, M/2) and [M/2, M) are the quantiles of the positive and negative
    // parts, stored as [parts][n][M/2], and each part is centred by its own
    // vector.
    extern __shared__ __align__(16) float2 smc[];
    // two batch buffers: the staged input of the FFT and its other buffer;
    // once a batch's transform is done, the buffer it did not end in takes
    // the next batch's copies while the unpack reads the result
    float2 *bufA = smc;                  // [n nsig]
    float2 *bufB = bufA + n * nsig;      // [n nsig]
    float2 *x1 = bufB + n * nsig;        // [M] Qhat(1, p) before centring (CTA 0's)
    float2 *tws = x1 + M;                // [n] twiddles
    float2 *terms = tws + n;             // CL: [batches here][NI][256] of levels (pa, pa + 1)
    constexpr int NW = kSpecThreads / 32;
    __shared__ double red[2][NW];
    __shared__ double s_c1[2][2];
    const int Mp = M / parts;  // levels per part
    int S = 1, rank = 0;
    if constexpr (CL) {
        S = (int)cg::this_cluster().num_blocks();
        rank = (int)cg::this_cluster().block_rank();
    }
    const int img = blockIdx.x / S;
    const float *qi = q + (size_t)img * n * M;
    const int nbatch = (M + 2 * nsig - 1) / (2 * nsig);
    chain_wait();
    stage_levels<nsig>(qi, n, M, Mp, parts, rank * 2 * nsig, bufA);
    for (int i = threadIdx.x; i < n; i += blockDim.x) tws[i] = tw[i];
    if (clear && blockIdx.x == 0 && threadIdx.x == 0) *clear = 0;
    if constexpr (CL) cg::this_cluster().sync();  // CTA 0 has started: its x1 can be written
    float2 *x1o = x1;
    if constexpr (CL) x1o = cg::this_cluster().map_shared_rank(x1, 0);
    const int nh = n / 2;
    // this thread's class (HB: the first of two) and share of it
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cls = HB ? warp * 16 + (lane & 15) : (int)threadIdx.x;
    const int sub = HB ? lane >> 4 : 0;
    const int s = cls % nsig, a = cls / nsig;
    constexpr int NA = kSpecThreads / NSC;
    const int NI = nh / NA + 1;  // frequencies of a class at most
    // norms as compensated (Kahan) FP32 sums: FP64 arithmetic is scarce on
    // this part
    DF acc = {0.f, 0.f}, acc_other = {0.f, 0.f};  // HB: this half's and the other half's class
    const float invn = 1.f / (float)n;

    float2 *cur = bufA, *oth = bufB;
    for (int bt = rank; bt < nbatch; bt += S) {
        const int p0 = bt * 2 * nsig;
        // ---- batch: levels (p0 + 2s, p0 + 2s + 1) as signal s (re, im)
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        float2 *R = fft_smem<nsig, -1, true>(cur, oth, plan, tws);
        // the next batch goes to the buffer the transform did not end in
        // (fft_smem ends with a block barrier: both buffers' readers are done)
        float2 *nxt = R == cur ? oth : cur;
        if (bt + S < nbatch)
            stage_levels<nsig>(qi, n, M, Mp, parts, (bt + S) * 2 * nsig, nxt);
        cur = nxt;
        oth = R;
        // ---- unpack two real spectra per signal, k' = 0..n/2
        const int pa = p0 + 2 * s, pb = pa + 1;
        for (int i0 = 0; i0 < NI; i0 += HB ? 2 : 1) {
            const int i = i0 + sub, kf = a + NA * i;
            float2 term = make_float2(0.f, 0.f);
            if (kf <= nh) {
                const float2 Z = R[kf * nsig + s];
                const float2 Zc = cconj(R[(kf ? n - kf : 0) * nsig + s]);
                // Xa = (Z + conj Z(n-k))/2, Xb = (Z - conj Z(n-k)) / (2i)
                float2 Xa = make_float2(0.5f * (Z.x + Zc.x), 0.5f * (Z.y + Zc.y));
                const float2 dz = make_float2(0.5f * (Z.x - Zc.x), 0.5f * (Z.y - Zc.y));
                float2 Xb = make_float2(dz.y, -dz.x);
                if (kf >= 2) {
                    if (kf == nh) Xa.y = Xb.y = 0.f;  // Nyquist term of a real signal
                    const float w = kf == nh ? 1.f : 2.f;
                    if ((M & 1) == 0) {
                        // both levels at once (pa even, M even: 4-byte aligned pairs)
                        if (pb < M) {
                            term = emit2<T>(o, img, M, kf, pa, Xa, Xb, w);
                            if constexpr (!CL && !HB) {
                                kahan_add(acc, term.x);
                                kahan_add(acc, term.y);
                            }
                        }
                    } else {
                        if (pa < M) {
                            term.x = emit<T>(o, img, M, kf, pa, Xa, w);
                            if constexpr (!CL && !HB) kahan_add(acc, term.x);
                        }
                        if (pb < M) {
                            term.y = emit<T>(o, img, M, kf, pb, Xb, w);
                            if constexpr (!CL && !HB) kahan_add(acc, term.y);
                        }
                    }
                } else if (kf == 1) {
                    if (pa < M) x1o[pa] = Xa;
                    if (pb < M) x1o[pb] = Xb;
                } else {
                    if (pa < M) prof[(size_t)img * M + pa] = Xa.x * invn;
                    if (pb < M) prof[(size_t)img * M + pb] = Xb.x * invn;
                }
            }
            if constexpr (CL) {
                terms[((bt / S) * NI + i) * kSpecThreads + cls] = term;
            } else if constexpr (HB) {
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const float2 tu =
                        make_float2(__shfl_sync(0xffffffffu, term.x, (lane & 15) + 16 * u),
                                    __shfl_sync(0xffffffffu, term.y, (lane & 15) + 16 * u));
                    const int ku = a + NA * (i0 + u);
                    if (ku >= 2 && ku <= nh) {
                        if (pa < M) kahan_add(acc, tu.x);
                        if (pb < M) kahan_add(acc, tu.y);
                    }
                }
            }
        }
        if constexpr (HB) {  // the next half batch adds to the other class
            const DF t = acc;
            acc = acc_other;
            acc_other = t;
        }
        __syncthreads();
    }
    if constexpr (HB) {
        if (nbatch & 1) {  // acc: the first half's class again
            const DF t = acc;
            acc = acc_other;
            acc_other = t;
        }
    }
    const bool tmpl = img >= o.Nq;
    // ---- zero padding of the low-precision rows: [2M, ldk) of every segment
    if (o.lp && o.ldk > 2 * M) {
        const int pad = o.ldk - 2 * M;
        const int nseg = o.split ? 2 : 1;
        const int row_len = nseg * o.ldk;
        const int rows = tmpl ? 2 : 1;
        const int per_f = rows * nseg * pad;
        for (int t = rank * blockDim.x + threadIdx.x; t < nh * per_f; t += S * blockDim.x) {
            const int kf = 1 + t / per_f, rem = t % per_f;
            const int rr = rem / (nseg * pad), sg = (rem / pad) % nseg, e = 2 * M + rem % pad;
            T *r = tmpl ? reinterpret_cast<T *>(o.lp_t) + (size_t)(kf - 1) * o.lpt_fstride +
                              (size_t)(2 * (img - o.Nq) + rr) * row_len
                        : reinterpret_cast<T *>(o.lp_q) + (size_t)(kf - 1) * o.lpq_fstride +
                              (size_t)img * row_len;
            r[sg * o.ldk + e] = to_lp<T>(0.f);
        }
    }
    if constexpr (CL) {
        cg::this_cluster().sync();  // every batch's terms and x1 are in place
        if (rank == 0) {
            for (int bt = 0; bt < nbatch; ++bt) {
                const int pa = bt * 2 * nsig + 2 * s, pb = pa + 1;
                const float2 *tr = cg::this_cluster().map_shared_rank(terms, bt % S) +
                                   (size_t)(bt / S) * NI * kSpecThreads + cls;
#pragma unroll 8
                for (int i = 0; i < NI; ++i) {
                    const int ku = a + NA * i;
                    const float2 tu = tr[i * kSpecThreads];
                    if (ku >= 2 && ku <= nh) {
                        if (pa < M) kahan_add(acc, tu.x);
                        if (pb < M) kahan_add(acc, tu.y);
                    }
                }
            }
        }
        cg::this_cluster().sync();  // CTA 0 has read the other CTAs' terms
        if (rank != 0) return;
    }
    // ---- centring, per part: c1 = mean_p Qhat_u(1, p);  a = (2/n)(Re c1, -Im c1)
    for (int part = 0; part < parts; ++part) {
        double cr = 0.0, ci = 0.0;
        for (int p = part * Mp + threadIdx.x; p < (part + 1) * Mp; p += blockDim.x) {
            cr += x1[p].x;
            ci += x1[p].y;
        }
#pragma unroll
        for (int off = 16; off; off >>= 1) {
            cr += __shfl_xor_sync(0xffffffffu, cr, off);
            ci += __shfl_xor_sync(0xffffffffu, ci, off);
        }
        if (lane == 0) {
            red[0][warp] = cr;
            red[1][warp] = ci;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double sr = 0.0, si = 0.0;
            for (int w = 0; w < NW; ++w) {
                sr += red[0][w];
                si += red[1][w];
            }
            s_c1[part][0] = sr / Mp;
            s_c1[part][1] = si / Mp;
            double *cimg = center + 2 * ((size_t)img * parts + part);
            cimg[0] = 2.0 * s_c1[part][0] / n;
            cimg[1] = -2.0 * s_c1[part][1] / n;
        }
        __syncthreads();
    }
    // k' = 1 (n >= 4: 1 < n/2), last in each class: level p is class p mod 256's
    auto first_frequency = [&](int c, DF &sum) {
        for (int p = c; p < M; p += kSpecThreads) {
            const int part = p / Mp;
            const float c1r = (float)s_c1[part][0], c1i = (float)s_c1[part][1];
            const float2 X = make_float2(x1[p].x - c1r, x1[p].y - c1i);
            kahan_add(sum, emit<T>(o, img, M, 1, p, X, 2.f));
        }
    };
    if (sub == 0) {
        first_frequency(a * NSC + s, acc);
        if constexpr (HB) first_frequency(a * NSC + s + nsig, acc_other);
    }
    // ---- norms: Parseval over k' != 0 of the centred spectra, / n
    double an = (double)acc.hi + (double)acc.lo;
    if constexpr (HB)
        an = sub == 0 ? an + ((double)acc_other.hi + (double)acc_other.lo) : 0.0;
#pragma unroll
    for (int off = 16; off; off >>= 1) an += __shfl_xor_sync(0xffffffffu, an, off);
    __syncthreads();
    if (lane == 0) red[0][warp] = an;
    __syncthreads();
    if (threadIdx.x == 0) {
        double sn = 0.0;
        for (int w = 0; w < NW; ++w) sn += red[0][w];
        (o.lp && !o.split ? norm16 : norm32)[img] = sn / n;
    }
}

}  // namespace

cudaError_t launch_spectrum(const float *q, int nb, int n, int M, const FftPlan &plan,
                            const float2 *tw, float *spec32, size_t fstride, int lp_kind,
                            void *lp_q, size_t lpq_fstride, void *lp_t, size_t lpt_fstride,
                            int Nq, float *prof, double *center, double *norm32,
                            double *norm16, cudaStream_t st, int nsig_req, int parts,
                            int *clear)
{
    if (parts != 1 && (parts != 2 || M % 2)) return cudaErrorInvalidValue;
    if (nb <= 0) return cudaSuccess;
    const DeviceForm *dev;
    cudaError_t e = device_form(&dev);
    if (e != cudaSuccess) return e;
    SpecOut o{spec32, fstride, lp_q, lpq_fstride, lp_t, lpt_fstride, Nq, tc_ldk(M),
              lp_kind != 0, lp_kind == 3};
    // zeros of a template's two rows where there are templates, of a query's one elsewhere
    const long long zeros = o.lp ? (long long)(n / 2) * (o.ldk - 2 * M) * (o.split ? 2 : 1) *
                                       (Nq < nb ? 2 : 1)
                                 : 0;
    SpectrumForm f;
    if (!spectrum_form(nb, n, M, nsig_req, zeros, *dev, &f)) return cudaErrorInvalidValue;
    auto run = [&](auto kern) {
        cudaError_t er = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)f.smem);
        if (er != cudaSuccess) return er;
        return launch_chained(kern, dim3((unsigned)(nb * f.cluster)), dim3(kSpecThreads), f.smem,
                              st, f.cluster, q, n, M, plan, tw, o, prof, center, norm32, norm16,
                              parts, clear);
    };
#define SW_SPEC_FORMS(T, NS)                                                  \
    return f.cluster > 1 ? run(k_spectrum<T, NS, false, true>)                \
           : f.half      ? run(k_spectrum<T, NS, (NS > 4), false>)            \
           : f.dense     ? run(k_spectrum<T, NS, false, false, 4>)            \
                         : run(k_spectrum<T, NS, false, false>)
    if (lp_kind == 2 || lp_kind == 3) {
        if (f.nsig == 16) SW_SPEC_FORMS(__half, 16);
        if (f.nsig == 8) SW_SPEC_FORMS(__half, 8);
        SW_SPEC_FORMS(__half, 4);
    }
    if (f.nsig == 16) SW_SPEC_FORMS(__nv_bfloat16, 16);
    if (f.nsig == 8) SW_SPEC_FORMS(__nv_bfloat16, 8);
    SW_SPEC_FORMS(__nv_bfloat16, 4);
#undef SW_SPEC_FORMS
}

}  // namespace swk
