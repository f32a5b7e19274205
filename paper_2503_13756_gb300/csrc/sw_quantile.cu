// sw_quantile.cu -- quantile functions of the projections (Sec. 2.3
// "Computation": CDF by cumulative sum, ICDF by linear interpolation;
// Eq. inv_cdf read with the ">=" of App. A.1.1).
//
// For one projection U[0..B) with nodes e_j = (j - B/2) h:
//   F_0 = 0, F_j = sum_{b<j} U_b,  tau_p = z_p F_B,
//   j* = min{ j >= 1 : F_j >= tau_p },
//   Q(z_p) = e_{j*-1} + h (tau_p - F_{j*-1}) / U_{j*-1};
// at tau = 0 (level p = 0 under the p/M rule) every t qualifies and Q is the
// left end of the domain, e_0.
//
// Design (GB300): one warp per projection; one resident set of warps shares
// the batch's projections evenly, each warp taking its share one after the
// other (the next one's bins are loaded into registers while the current one
// is computed).  The CDF is a warp scan of double-float
// partial sums (TwoSum-compensated FP32), so that tau - F_{j-1} keeps ~48
// bits even where it cancels.  The levels are not searched for: every bin
// counts the levels below its right node and the bins whose count grows put
// their index at their first level; a warp maximum scan over the levels then
// gives every level its bin, without divergence.  No FP64 on this path.
#include <cooperative_groups.h>

#include <algorithm>

#include "sw_forms.h"
#include "sw_internal.cuh"

namespace swk {
namespace {

namespace cg = cooperative_groups;

constexpr int kQThreads = 256;  // 8 warps

// a + b for double-floats of non-negative value (every partial sum of a
// projection row): TwoSum of the leading parts, then the tails, then a
// Fast2Sum renormalisation -- exact, since without cancellation the tail
// sum is below an ulp and a half of the leading sum, which Fast2Sum needs.
// The same (hi, lo) as df_add with its second TwoSum, in three fewer flops.
__device__ __forceinline__ DF df_add_nonneg(DF a, DF b)
{
    const DF s = df_two_sum(a.hi, b.hi);
    const float e = s.lo + (a.lo + b.lo);
    const float hi = s.hi + e;
    return {hi, e - (hi - s.hi)};
}

// a + x for one value of a row (a double-float with no tail).
__device__ __forceinline__ DF df_add_value(DF a, float x)
{
    const DF s = df_two_sum(a.hi, x);
    const float e = s.lo + a.lo;
    const float hi = s.hi + e;
    return {hi, e - (hi - s.hi)};
}

// The levels tau_q = z_q F_B of one row, numbered from 1.
struct Levels {
    DF total;        // F_B
    float dz, inv_dz;
    int rule;        // 0: z = (2 q - 1) / (2 M); 1: z = q / M
    // kz = z_q dz: 2 q - 1 (midpoints) or q
    __device__ __forceinline__ DF at(float kz) const
    {
        return df_scale_ratio(total, kz, dz, inv_dz);
    }
    __device__ __forceinline__ DF tau(int q) const
    {
        return at(rule == 0 ? 2.f * (float)q - 1.f : (float)q);
    }
};

// df_scale_ratio for two values of k at once, in two-wide FP32 operations (one
// instruction for both; the same roundings).
__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    return __fadd2_rn(a, make_float2(-b.x, -b.y));
}
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2 &s, float2 &e)
{
    s = __fadd2_rn(a, b);
    const float2 v = sub2(s, a);
    e = __fadd2_rn(sub2(a, sub2(s, v)), sub2(b, v));
}
__device__ __forceinline__ void scale_ratio2(DF t, float2 k, float d, float inv_d, float2 &hi,
                                             float2 &lo)
{
    const float2 th = make_float2(t.hi, t.hi), tl = make_float2(t.lo, t.lo);
    const float2 iv = make_float2(inv_d, inv_d), nd = make_float2(-d, -d);
    const float2 p = __fmul2_rn(th, k);
    const float2 e = __ffma2_rn(th, k, make_float2(-p.x, -p.y));
    float2 nh, nl;
    two_sum2(p, __ffma2_rn(tl, k, e), nh, nl);
    const float2 qq = __fmul2_rn(nh, iv);
    const float2 r = __ffma2_rn(nd, qq, nh);
    two_sum2(qq, __fmul2_rn(__fadd2_rn(r, nl), iv), hi, lo);
}

// Number of levels q in 1..qmax with tau_q <= F, by bisection (exact).  Out
// of line (rarely needed) and by value, so that the levels stay in registers.
__device__ __noinline__ int count_levels(Levels lv, int qmax, DF F)
{
    int lo = 0, hi = qmax;  // tau_q <= F for q <= lo; not for q > hi
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (df_ge(F, lv.tau(mid))) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// *dst = v in shared memory where ok, as one predicated store (a branch per
// store costs more than the store).
__device__ __forceinline__ void store_if(bool ok, int *dst, int v)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.s32 p, %0, 0;\n @p st.shared.s32 [%1], %2;\n}" ::"r"((int)ok),
        "r"((uint32_t)__cvta_generic_to_shared(dst)), "r"(v)
        : "memory");
}

// Bins [c0, c0 + C) of a row (u[i] = row bin c0 + i, read backwards in a
// mirrored row), zero past B.  C even: 8-byte loads (B is even and the rows
// are 16-byte aligned, so every even element is 8-byte aligned).
template <int C>
__device__ __forceinline__ void load_bins(float (&u)[C], const float *__restrict__ row, int B,
                                          int c0, bool mirror)
{
    if (C % 2 == 0 && c0 + C <= B) {
        const float2 *src = reinterpret_cast<const float2 *>(row + (mirror ? B - c0 - C : c0));
#pragma unroll
        for (int i = 0; i < C / 2; ++i) {
            const float2 v = __ldg(src + i);
            u[mirror ? C - 1 - 2 * i : 2 * i] = v.x;
            u[mirror ? C - 2 - 2 * i : 2 * i + 1] = v.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < C; ++i) {
            const int b = c0 + i;
            u[i] = b < B ? __ldg(row + (mirror ? B - 1 - b : b)) : 0.f;
        }
    }
}

// C: bins per lane (ceil(B / 32)) in registers, or 0 for the run-time form
// that reads its bins twice (B > 384).  LV: adjacent levels per lane of each
// group of 32 LV levels.
//
// Bound by instruction issue (614 warp instructions per row at B = 192, M =
// 128; 1,174 with a binary search per lane and forward walks).  4352 images
// at n = 256, B = 192, M = 128: 353 us, 584 us before; 10,001 at n = 512, M =
// 256: 2.01 ms, 4.32 ms before; 3 at n = 360, B = 384, M = 256: 16 us, 55 us
// before.  What each choice is for:
//  - bins in registers, C a template parameter: no loop control, and one
//    read per bin instead of three;
//  - one 16-byte record per bin, (F_{j-1} hi, lo, U_{j-1}, e_{j-1}), so that a
//    level reads all it needs in one load; lanes' record groups are an odd
//    number of records apart (no bank conflicts);
//  - the level counts: M F_j / F_B in FP32 rounded to the nearest count, exact
//    unless it lands within its rounding error of a boundary between two
//    counts (count_edge); a warp in which one does (about one row in a hundred) recounts
//    its row, that node by a double-float comparison with the one level
//    (by bisection over the levels it took a quarter of the kernel's time);
//  - two levels at a time in two-wide FP32 operations, and predicated slot
//    stores (a branch each took 7% more instructions).
// CTAs per SM: four (64 registers) to C = 8, three (80) above.  Three and four in us
// of 1000 images, n = 360, M = 256: C = 6 165 and 159, 7 170 and 180, 8 182 and 180, 9
// 209 and 208, 10 198 and 200, 11 240 and 262; of 300 images C = 8 59 and 61, 9 68
// and 69, 10 65 and 69, 11 77 and 86.
constexpr int quantile_ctas(int C) { return C >= 9 ? 3 : 4; }
template <int C, int LV>
__global__ void __launch_bounds__(kQThreads, quantile_ctas(C))
k_quantiles(const float *__restrict__ proj, int n, int B, int M, float h, int level_rule,
            int half, int mirror_out, long long nrow, float *__restrict__ q,
            int32_t *__restrict__ status, int status_shift)
{
    extern __shared__ float4 smq[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nw = blockDim.x >> 5;
    chain_wait();
    const int nh = n / 2;
    const int nrows = mirror_out ? nh : n;  // rows computed per image
    // this warp's rows (images' rows in a row), as even a share as possible
    const long long gw = (long long)blockIdx.x * nw + warp, W = (long long)gridDim.x * nw;
    const long long r0 = nrow * gw / W;
    int left = (int)(nrow * (gw + 1) / W - r0);
    if (left == 0) return;  // whole warp leaves; no block barrier below
    int imgi = (int)(r0 / nrows), k = (int)(r0 % nrows);
    const int Cr = C > 0 ? C : (B + 31) / 32;
    const int RS = Cr | 1;                       // records per lane, odd
    constexpr int GL = 32 * LV;                  // levels per group
    const int ngrp = (M + GL - 1) / GL;
    // per warp: records [32 RS], then the level slots [ngrp GL]
    float4 *rec = smq + (size_t)warp * (32 * RS + ngrp * GL / 4);
    int *slot = reinterpret_cast<int *>(rec + 32 * RS);
    const int c0 = min(B, lane * Cr);
    const int c1 = min(B, c0 + Cr);
    const int last_lane = (B - 1) / Cr;          // owner of the last bin
    const int qmax = level_rule == 0 ? M : M - 1;
    const int qoff = level_rule == 0 ? 1 : 0;    // level of number q is p = q - qoff
    Levels lv;
    lv.dz = level_rule == 0 ? 2.f * M : (float)M;
    lv.inv_dz = 1.f / lv.dz;
    lv.rule = level_rule;
    const float coff = level_rule == 0 ? 0.f : -0.5f;
    const float kstep = level_rule == 0 ? 2.f : 1.f, kofs = level_rule == 0 ? -1.f : 0.f;
    const float edge = count_edge(M);
    const float e0 = ((float)c0 - 0.5f * (float)B);

    for (int g = 0; g < ngrp; ++g)
#pragma unroll
        for (int v = 0; v < LV; ++v) slot[g * GL + lane * LV + v] = 0;
    __syncwarp();

    auto row_of = [&](int img, int kk, bool &mirror) {
        mirror = half && kk >= nh;
        return half ? proj + ((size_t)img * nh + (mirror ? kk - nh : kk)) * B
                    : proj + ((size_t)img * n + kk) * B;
    };
    constexpr int CA = C > 0 ? C : 1;
    float u[CA], un[CA];
    bool mir;
    const float *row = row_of(imgi, k, mir);
    if (C > 0) load_bins<CA>(u, row, B, c0, mir);

    for (; left > 0; --left) {
        bool mir_next = false;
        const float *row_next = row;
        const bool wrap = k + 1 == nrows;
        const int img_next = wrap ? imgi + 1 : imgi, k_next = wrap ? 0 : k + 1;
        if (left > 1) {
            row_next = row_of(img_next, k_next, mir_next);
            if (C > 0) load_bins<CA>(un, row_next, B, c0, mir_next);
        }
        auto bin = [&](int i) {  // run-time form
            return __ldg(row + (mir ? B - 1 - c0 - i : c0 + i));
        };

        // ---- compensated prefix sums: lane owns bins [c0, c1)
        DF s = {0.f, 0.f};
        if (C > 0) {
            s.hi = u[0];
#pragma unroll
            for (int i = 1; i < CA; ++i) s = df_add_value(s, u[i]);
        } else {
            for (int i = 0; i < c1 - c0; ++i) s = df_add_value(s, bin(i));
        }
        // inclusive warp scan of the lane sums
        DF inc = s;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            DF o;
            o.hi = __shfl_up_sync(0xffffffffu, inc.hi, off);
            o.lo = __shfl_up_sync(0xffffffffu, inc.lo, off);
            const DF t = df_add_nonneg(o, inc);
            inc.hi = lane >= off ? t.hi : inc.hi;
            inc.lo = lane >= off ? t.lo : inc.lo;
        }
        DF run;
        run.hi = __shfl_up_sync(0xffffffffu, inc.hi, 1);
        run.lo = __shfl_up_sync(0xffffffffu, inc.lo, 1);
        if (lane == 0) run = {0.f, 0.f};
        // running sums; record i holds F before bin i (record 0: below)
        float4 *myrec = rec + lane * RS;
        float fh[CA];
        float u0 = 0.f;
        if (C > 0) {
            u0 = u[0];
#pragma unroll
            for (int i = 0; i < CA; ++i) {
                if (i > 0)
                    myrec[i] = make_float4(run.hi, run.lo, u[i], (e0 + (float)i) * h);
                run = df_add_value(run, u[i]);
                fh[i] = run.hi;
            }
        } else {
            for (int i = 0; i < c1 - c0; ++i) {
                const float x = bin(i);
                if (i == 0) u0 = x;
                else myrec[i] = make_float4(run.hi, run.lo, x, (e0 + (float)i) * h);
                run = df_add_value(run, x);
            }
        }
        const float phi = __shfl_up_sync(0xffffffffu, run.hi, 1);
        const float plo = __shfl_up_sync(0xffffffffu, run.lo, 1);
        myrec[0] = make_float4(lane ? phi : 0.f, lane ? plo : 0.f, u0, e0 * h);
        lv.total.hi = __shfl_sync(0xffffffffu, run.hi, last_lane);
        lv.total.lo = __shfl_sync(0xffffffffu, run.lo, last_lane);
        const float total = lv.total.hi;
        float *qo = q + ((size_t)imgi * n + k) * M;
        float *qm = qo + (size_t)nh * M;
        if (!(total > 0.f) || !isfinite(total)) {
            for (int p = lane; p < M; p += 32) qo[p] = __int_as_float(0x7fc00000);
            if (mirror_out)
                for (int p = lane; p < M; p += 32) qm[p] = __int_as_float(0x7fc00000);
            if (lane == 0) atomicOr(status + (imgi >> status_shift), 1);
        } else {
            // ---- counts at the bins' right nodes; a bin whose count grows
            // takes the levels from its left count on
            bool near = total < 1e-30f || total > 1e30f || C == 0;
            if (!near) {
                const float sc = __fdividef((float)M, total);
                int c[CA];
                // (the unsigned minimum also bounds what a row that is no
                // projection, with negative sums, could give)
                auto count = [&](int i) {
                    const float x = fmaf(fh[i], sc, coff);
                    const float y = x + 12582912.f;  // 1.5 2^23: rounds to an integer
                    c[i] = (int)min((unsigned)(__float_as_int(y) - 0x4b400000), (unsigned)qmax);
                    return fabsf(x - (y - 12582912.f)) > edge;
                };
                if (level_rule == 0) {
#pragma unroll
                    for (int i = 0; i < CA; ++i) near |= count(i);
                } else {  // z = q / M: F = 0 and F = F_B lie on boundaries without a level
#pragma unroll
                    for (int i = 0; i < CA; ++i)
                        near |= count(i) & (fh[i] > 0.f) & (fh[i] < total);
                }
                near = __any_sync(0xffffffffu, near);
                if (!near) {
                    int cp = __shfl_up_sync(0xffffffffu, c[CA - 1], 1);
                    if (lane == 0) cp = 0;
#pragma unroll
                    for (int i = 0; i < CA; ++i) {
                        store_if(c[i] > cp, slot + (cp + 1 - qoff), lane * RS + i + 1);
                        cp = c[i];
                    }
                }
            }
            if (near) {
                // the same, with the count of a node on the edge taken from
                // the comparison of the node with the one level it may hold
                const bool odd_scale = total < 1e-30f || total > 1e30f;
                const float sc = odd_scale ? 0.f : __fdividef((float)M, total);
                auto count = [&](DF F) {
                    if (odd_scale) return count_levels(lv, qmax, F);
                    const float x = fmaf(F.hi, sc, coff);
                    const float y = x + 12582912.f;
                    const float d = x - (y - 12582912.f);
                    int c = (int)min((unsigned)(__float_as_int(y) - 0x4b400000), (unsigned)qmax);
                    if (fabsf(d) > edge) {
                        const int qc = __float_as_int(y) - 0x4b400000 + (d > 0.f);
                        if (qc >= 1 && qc <= qmax) c = df_ge(F, lv.tau(qc)) ? qc : qc - 1;
                    }
                    return c;
                };
                __syncwarp();
                const int cl = c1 > c0 ? count(run) : 0;  // the next lane's left count
                int cp = __shfl_up_sync(0xffffffffu, cl, 1);
                if (lane == 0) cp = 0;
                for (int i = 0; i < c1 - c0; ++i) {
                    DF F = run;
                    if (i + 1 < c1 - c0) {
                        const float4 r = myrec[i + 1];
                        F = {r.x, r.y};
                    }
                    const int ci = count(F);
                    if (ci > cp) slot[cp + 1 - qoff] = lane * RS + i + 1;
                    cp = ci;
                }
            }
            __syncwarp();
            // ---- levels: the running maximum of the slots is the record
            int carry = 1;
            for (int g = 0; g < ngrp; ++g) {
                int *sl = slot + g * GL + lane * LV;
                int j[LV];
                if (LV == 4) {
                    const int4 t = *reinterpret_cast<const int4 *>(sl);
                    *reinterpret_cast<int4 *>(sl) = make_int4(0, 0, 0, 0);
                    j[0] = t.x;
                    j[1 % LV] = t.y;
                    j[2 % LV] = t.z;
                    j[3 % LV] = t.w;
                } else {
                    const int2 t = *reinterpret_cast<const int2 *>(sl);
                    *reinterpret_cast<int2 *>(sl) = make_int2(0, 0);
                    j[0] = t.x;
                    j[1 % LV] = t.y;
                }
#pragma unroll
                for (int v = 1; v < LV; ++v) j[v] = max(j[v], j[v - 1]);
                int m = max(j[LV - 1], carry);
#pragma unroll
                for (int off = 1; off < 32; off <<= 1)
                    m = max(m, __shfl_up_sync(0xffffffffu, m, off));
                int ex = __shfl_up_sync(0xffffffffu, m, 1);
                if (lane == 0) ex = carry;
                carry = __shfl_sync(0xffffffffu, m, 31);
                const int p0 = g * GL + lane * LV;
                const float kz0 = fmaf((float)(p0 + qoff), kstep, kofs);
                float Q[LV];
#pragma unroll
                for (int v = 0; v < LV; v += 2) {
                    float2 th, tl;
                    scale_ratio2(lv.total,
                                 make_float2(kz0 + (float)v * kstep, kz0 + (float)(v + 1) * kstep),
                                 lv.dz, lv.inv_dz, th, tl);
                    const float4 ra = rec[max(j[v], ex) - 1], rb = rec[max(j[v + 1], ex) - 1];
                    const float2 num = __fadd2_rn(sub2(th, make_float2(ra.x, rb.x)),
                                                  sub2(tl, make_float2(ra.y, rb.y)));
                    // the fraction only scales h: a fast divide (error ~2 ulp) is ample
                    float fa = __fdividef(num.x, ra.z), fb = __fdividef(num.y, rb.z);
                    fa = __saturatef(ra.z > 0.f ? fa : 0.f);
                    fb = __saturatef(rb.z > 0.f ? fb : 0.f);
                    Q[v] = fmaf(h, fa, ra.w);
                    Q[v + 1] = fmaf(h, fb, rb.w);
                }
                // tau = 0: inf{t : F(t) >= 0} is the domain's left end e_0
                if (level_rule == 1 && p0 == 0) Q[0] = -0.5f * (float)B * h;
                // theta + pi: the mirrored histogram has Q'(z) = -Q(1 - z), and
                // with midpoint levels 1 - z_p = z_{M-1-p}
                if ((M % LV) == 0) {
                    if (p0 < M) {
                        if (LV == 4) {
                            *reinterpret_cast<float4 *>(qo + p0) =
                                make_float4(Q[0], Q[1 % LV], Q[2 % LV], Q[3 % LV]);
                            if (mirror_out)
                                *reinterpret_cast<float4 *>(qm + M - 4 - p0) =
                                    make_float4(-Q[3 % LV], -Q[2 % LV], -Q[1 % LV], -Q[0]);
                        } else {
                            *reinterpret_cast<float2 *>(qo + p0) = make_float2(Q[0], Q[1 % LV]);
                            if (mirror_out)
                                *reinterpret_cast<float2 *>(qm + M - 2 - p0) =
                                    make_float2(-Q[1 % LV], -Q[0]);
                        }
                    }
                } else {
                    // rows of any alignment: through the group's slots, which
                    // only this group's lanes use, so that the stores coalesce
                    float *st = reinterpret_cast<float *>(slot + g * GL);
                    __syncwarp();
#pragma unroll
                    for (int v = 0; v < LV; ++v) st[lane * LV + v] = Q[v];
                    __syncwarp();
#pragma unroll
                    for (int v = 0; v < LV; ++v) {
                        const int p = g * GL + 32 * v + lane;
                        const float x = st[32 * v + lane];
                        if (p < M) {
                            qo[p] = x;
                            if (mirror_out) qm[M - 1 - p] = -x;
                        }
                    }
                    __syncwarp();
#pragma unroll
                    for (int v = 0; v < LV; ++v) st[lane * LV + v] = 0.f;
                }
            }
        }
        __syncwarp();  // the records and slots are free for the next projection
        if (C > 0) {
#pragma unroll
            for (int i = 0; i < CA; ++i) u[i] = un[i];
        }
        row = row_next;
        mir = mir_next;
        imgi = img_next;
        k = k_next;
    }
}

// Centring vector and centred norm (public sw_quantiles outputs), FP64
// accumulation.  A cluster of CTAs per image shares its rows; the partial
// sums meet in the shared memory of the cluster's CTAs, added in rank order
// by every CTA.  Bound by FP64 issue, so a row costs only the additions of
// its quantiles and two fused multiply-adds (no division or warp reduction
// per row: those were four fifths of the instructions), the norm is skipped
// when it is not wanted, and every SM has rows (64 images on one CTA each
// left 88 of 152 SMs idle).
__global__ void __launch_bounds__(256)
k_center_norm(const float *__restrict__ q, int n, int M, const double2 *__restrict__ cs64,
              double *__restrict__ center, double *__restrict__ norm)
{
    __shared__ double red[3][32];
    __shared__ double part[3];  // this CTA's sums: a (x, y), norm
    chain_wait();
    cg::cluster_group cl = cg::this_cluster();
    const int S = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int imgi = blockIdx.x / S;
    const float *qi = q + (size_t)imgi * n * M;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    // a = (2/n) sum_k ubar_k (cos, sin),  ubar_k = mean_p q[k][p]: every lane
    // weights its own share of each row's sum
    double ax = 0.0, ay = 0.0;
    for (int k = rank * nw + warp; k < n; k += S * nw) {
        double s = 0.0;
        for (int p = lane; p < M; p += 32) s += (double)qi[(size_t)k * M + p];
        ax += s * cs64[k].x;
        ay += s * cs64[k].y;
    }
#pragma unroll
    for (int off = 16; off; off >>= 1) {
        ax += __shfl_xor_sync(0xffffffffu, ax, off);
        ay += __shfl_xor_sync(0xffffffffu, ay, off);
    }
    if (lane == 0) {
        red[0][warp] = ax;
        red[1][warp] = ay;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double sx = 0.0, sy = 0.0;
        for (int w = 0; w < nw; ++w) {
            sx += red[0][w];
            sy += red[1][w];
        }
        part[0] = sx;
        part[1] = sy;
    }
    cl.sync();
    double a0 = 0.0, a1 = 0.0;
    for (int r = 0; r < S; ++r) {
        const double *o = cl.map_shared_rank(part, r);
        a0 += o[0];
        a1 += o[1];
    }
    a0 = a0 * 2.0 / ((double)n * M);
    a1 = a1 * 2.0 / ((double)n * M);
    if (norm) {
        double acc = 0.0;
        for (int k = rank * nw + warp; k < n; k += S * nw) {
            const double off = a0 * cs64[k].x + a1 * cs64[k].y;
            for (int p = lane; p < M; p += 32) {
                const double d = (double)qi[(size_t)k * M + p] - off;
                acc += d * d;
            }
        }
#pragma unroll
        for (int off = 16; off; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (lane == 0) red[2][warp] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int w = 0; w < nw; ++w) s += red[2][w];
            part[2] = s;
        }
        cl.sync();
    }
    if (rank == 0 && threadIdx.x == 0) {
        if (center) {
            center[2 * imgi] = a0;
            center[2 * imgi + 1] = a1;
        }
        if (norm) {
            double s = 0.0;
            for (int r = 0; r < S; ++r) s += cl.map_shared_rank(part, r)[2];
            norm[imgi] = s;
        }
    }
    cl.sync();  // no CTA leaves while its sums may still be read
}

}  // namespace

cudaError_t launch_quantiles(const float *proj, int nb, int n, int B, int M, float h,
                             int level_rule, int half, float *q, int32_t *status,
                             cudaStream_t st, int status_shift)
{
    if (nb <= 0) return cudaSuccess;
    // with half projections and midpoint levels, angles k and k + n/2 come
    // from one quantile computation
    const int mirror = half && level_rule == 0;
    const int nang = mirror ? n / 2 : n;
    int C = (B + 31) / 32;
    const int LV = M <= 64 ? 2 : 4;
    const int GL = 32 * LV;
    const size_t per_warp = 16 * (size_t)(32 * (C | 1)) + 4 * (size_t)((M + GL - 1) / GL * GL);
    int nw = kQThreads / 32;
    while (nw > 1 && nw * per_warp > 200 * 1024) nw /= 2;
    const size_t smem = nw * per_warp;
    // Every warp takes an even share of the rows, so that all but its first
    // are in flight before they are needed: one resident set of warps, or
    // several short ones where that leaves each warp some 16 rows (a row's
    // time varies a little, and short shares even that out: 4352 images at
    // n = 256, M = 128 take 374 us in one set, 353 us in 4 to 7 and 374 us in
    // 16; 128 images at n = 360, M = 256, six rows a warp, 34.7 us in one set
    // and 36.8 us in two).
    const DeviceForm *dev;
    cudaError_t e = device_form(&dev);
    if (e != cudaSuccess) return e;
    const long long nrow = (long long)nb * nang;
    const int per_sm = std::max(1, std::min(quantile_ctas(C), (int)(220 * 1024 / smem)));
    const long long set = (long long)dev->sms * per_sm;
    const long long share = nrow / (set * nw);
    const long long sets = std::min<long long>(12, std::max<long long>(1, (share + 8) / 16));
    const int grid = (int)std::min<long long>((nrow + nw - 1) / nw, set * sets);
    auto run = [&](auto kern) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             200 * 1024);
        if (e != cudaSuccess) return e;
        return launch_chained(kern, dim3(grid), dim3(32 * nw), smem, st, 1, proj, n, B, M, h,
                              level_rule, half, mirror, nrow, q, status, status_shift);
    };
    if (C > 12) C = 0;
    switch (C) {
#define SW_Q(c) case c: return LV == 2 ? run(k_quantiles<c, 2>) : run(k_quantiles<c, 4>)
        SW_Q(1);
        SW_Q(2);
        SW_Q(3);
        SW_Q(4);
        SW_Q(5);
        SW_Q(6);
        SW_Q(7);
        SW_Q(8);
        SW_Q(9);
        SW_Q(10);
        SW_Q(11);
        SW_Q(12);
#undef SW_Q
    default: return LV == 2 ? run(k_quantiles<0, 2>) : run(k_quantiles<0, 4>);
    }
}

cudaError_t launch_center_norm(const float *q, int nb, int n, int M, const double2 *cs64,
                               double *center, double *norm, cudaStream_t st)
{
    if (nb <= 0) return cudaSuccess;
    // CTAs per image: enough for four on each SM, eight (the portable
    // cluster size) at most, and at least four rows to a warp (below that the
    // reductions cost more than the rows: 151 images at n = 96)
    const DeviceForm *dev;
    const cudaError_t e = device_form(&dev);
    if (e != cudaSuccess) return e;
    int S = 1;
    while (S < 8 && (long long)nb * S < 4 * dev->sms && 64 * S <= n) S *= 2;
    return launch_chained(k_center_norm, dim3((unsigned)(nb * S)), dim3(256), 0, st, S, q, n, M, cs64,
                          center, norm);
}

}  // namespace swk
