// sw_msw.cu -- max-sliced W2 over rotations (Eq. max_sliced_wasserstein):
//   D(l) = max_k (1/M) sum_p (u_pk - v_{p,(k-l) mod n})^2
// over the (optionally centred) quantiles of two images.  The cyclic
// cross-correlation does not apply to a maximum, so every (k, k') column
// pair is formed: O(n^2 M) per pair.
//
// Design (GB300): the per-angle terms are squared differences summed
// directly in FP32 (no Gram-matrix cancellation), level by level.  One CTA
// takes one pair and a tile of 64 rows k of the query against 64 CC <= 256
// columns k' of the template (all of them up to n = 256), staged 32 levels at
// a time; a warp owns eight of the rows and each lane 2 CC columns, as CC
// adjacent pairs, so that the difference and the square of two columns are
// one two-wide FP32 operation each.  The query values are staged twice side
// by side (the two-wide operand without a move) and the template's negated,
// columns transposed.  The tile's terms then go to shared memory, each thread
// takes rotations l = t, t + 256, ... and the maximum over the tile's rows of
// E[k][(k - l) mod n], and the tiles of a pair meet in an atomic max on the
// pair's curve (the terms are >= 0, so their float bits order as integers;
// the maximum does not depend on the order).  A second kernel takes the
// argmin per pair.
//
// Bound: two FP32 operations per level and column pair (k, k').
#include "sw_internal.cuh"
#include "swalign.h"

namespace swk {
namespace {

constexpr int kMswThreads = 256;
constexpr int kMswPC = 32;     // levels per stage (even)
constexpr int kMswWR = 8;      // rows per warp
constexpr int kMswR = kMswWR * kMswThreads / 32;  // rows per CTA

constexpr int kMswUS = kMswR + 2;  // staged row stride (16-byte rows, few bank conflicts)

// Shared memory: the staged tiles Us [PC][R + 2] of (u, u) and Vt [PC][64 CC + 2]
// of -v, then, in the same place, the terms Eb [R][64 CC]; and the template
// columns' offsets [64 CC].
size_t msw_smem(int CC)
{
    const size_t stage = 8 * (size_t)kMswPC * kMswUS + 4 * (size_t)kMswPC * (64 * CC + 2);
    const size_t terms = 4 * (size_t)kMswR * 64 * CC;
    return (stage > terms ? stage : terms) + 4 * (size_t)64 * CC;
}

template <int CC>
__global__ void __launch_bounds__(kMswThreads, 2)
k_msw(MswArgs A)
{
    constexpr int W = 64 * CC, R = kMswR, VS = W + 2;
    extern __shared__ __align__(16) float sms[];
    const int n = A.n, M = A.M;
    float2 *Us = reinterpret_cast<float2 *>(sms);  // [kMswPC][kMswUS]
    float *Vt = sms + 2 * kMswPC * kMswUS;              // [kMswPC][VS]
    float *Eb = sms;                               // [R][W]
    constexpr int kStage = 2 * kMswPC * kMswUS + kMswPC * VS, kTerms = R * W;
    float *offt = sms + (kStage > kTerms ? kStage : kTerms);  // [W]
    __shared__ float offq[R];
    const int pair = blockIdx.x;
    const int i = pair / A.Nt, j = pair % A.Nt;
    const int k0 = blockIdx.y * R, c0 = blockIdx.z * W;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const float *Qi = A.q + (size_t)i * n * M;
    const float *Qj = A.t + (size_t)j * n * M;
    // centring offsets <a, e_k> (translation): subtracted in the staging
    // below (FP64 is scarce: once per column, not once per staged level)
    const double2 *cs = A.cs64;
    const double aix = A.translation ? A.ctr_q[2 * i] : 0.0;
    const double aiy = A.translation ? A.ctr_q[2 * i + 1] : 0.0;
    const double ajx = A.translation ? A.ctr_t[2 * j] : 0.0;
    const double ajy = A.translation ? A.ctr_t[2 * j + 1] : 0.0;
    if (t < R) {
        const int k = k0 + t;
        offq[t] = k < n ? (float)(aix * cs[k].x + aiy * cs[k].y) : 0.f;
    }
    for (int c = t; c < W; c += kMswThreads) {
        const int kk = c0 + c;
        offt[c] = A.translation && kk < n ? (float)(ajx * cs[kk].x + ajy * cs[kk].y) : 0.f;
    }
    float2 acc[kMswWR][CC];
#pragma unroll
    for (int r = 0; r < kMswWR; ++r)
#pragma unroll
        for (int c = 0; c < CC; ++c) acc[r][c] = make_float2(0.f, 0.f);
    __syncthreads();
    const bool vec = (M & 3) == 0;  // every row starts on 16 bytes
    for (int p0 = 0; p0 < M; p0 += kMswPC) {
        const int pc = min(kMswPC, M - p0);
        // (u, u) and -v, centred, zero outside (zeros add nothing); four
        // levels per load where the rows keep 16-byte alignment
        constexpr int P4 = kMswPC / 4;
        for (int e = t; e < (R + W) * P4; e += kMswThreads) {
            const int row = e / P4, p = 4 * (e % P4);
            const bool is_q = row < R;
            const int c = is_q ? row : row - R;
            const int kk = (is_q ? k0 : c0) + c;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            if (kk < n && p < pc) {
                const float *src = (is_q ? Qi : Qj) + (size_t)kk * M + p0 + p;
                const float o = is_q ? offq[c] : offt[c];
                if (vec) {
                    x = __ldg(reinterpret_cast<const float4 *>(src));
                    x = make_float4(x.x - o, x.y - o, x.z - o, x.w - o);
                } else {
                    x.x = src[0] - o;
                    if (p + 1 < pc) x.y = src[1] - o;
                    if (p + 2 < pc) x.z = src[2] - o;
                    if (p + 3 < pc) x.w = src[3] - o;
                }
            }
            if (is_q) {
                Us[p * kMswUS + c] = make_float2(x.x, x.x);
                Us[(p + 1) * kMswUS + c] = make_float2(x.y, x.y);
                Us[(p + 2) * kMswUS + c] = make_float2(x.z, x.z);
                Us[(p + 3) * kMswUS + c] = make_float2(x.w, x.w);
            } else {
                Vt[p * VS + c] = -x.x;
                Vt[(p + 1) * VS + c] = -x.y;
                Vt[(p + 2) * VS + c] = -x.z;
                Vt[(p + 3) * VS + c] = -x.w;
            }
        }
        __syncthreads();
#pragma unroll 2
        for (int p = 0; p < pc; ++p) {
            float2 v[CC];
#pragma unroll
            for (int c = 0; c < CC; ++c)
                v[c] = *reinterpret_cast<const float2 *>(Vt + p * VS + 64 * c + 2 * lane);
            const float4 *up = reinterpret_cast<const float4 *>(Us + p * kMswUS + kMswWR * warp);
#pragma unroll
            for (int r2 = 0; r2 < kMswWR / 2; ++r2) {
                const float4 uu = up[r2];  // two rows
#pragma unroll
                for (int c = 0; c < CC; ++c) {
                    const float2 d0 = __fadd2_rn(make_float2(uu.x, uu.y), v[c]);
                    acc[2 * r2][c] = __ffma2_rn(d0, d0, acc[2 * r2][c]);
                    const float2 d1 = __fadd2_rn(make_float2(uu.z, uu.w), v[c]);
                    acc[2 * r2 + 1][c] = __ffma2_rn(d1, d1, acc[2 * r2 + 1][c]);
                }
            }
        }
        __syncthreads();
    }
    // ---- tile terms to shared memory, then diagonal maxima per rotation
#pragma unroll
    for (int r = 0; r < kMswWR; ++r)
#pragma unroll
        for (int c = 0; c < CC; ++c)
            *reinterpret_cast<float2 *>(Eb + (kMswWR * warp + r) * W + 64 * c + 2 * lane) =
                acc[r][c];
    __syncthreads();
    const int rows = min(R, n - k0), cols = min(W, n - c0);
    unsigned *curve = reinterpret_cast<unsigned *>(A.curve) + (size_t)pair * n;
    for (int l = t; l < n; l += kMswThreads) {
        float mx = 0.f;
        // row r takes the template column (k0 + r - l) mod n: the tile's
        // rows where it lies in the tile form at most two runs
        int cb = k0 - l - c0;
        cb += k0 < l ? n : 0;
#pragma unroll
        for (int h = 0; h < 2; ++h, cb -= n) {
            const int r0 = max(0, -cb), r1 = min(rows, cols - cb);
            const float *Er = Eb + cb;
#pragma unroll 4
            for (int r = r0; r < r1; ++r) mx = fmaxf(mx, Er[r * (W + 1)]);
        }
        atomicMax(curve + l, __float_as_uint(mx));
    }
}

// argmin over l (lowest l on ties), one warp per pair
__global__ void k_msw_decide(MswArgs A)
{
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    const int pairs = A.Nq * A.Nt;
    if (warp >= pairs) return;
    const int i = warp / A.Nt, j = warp % A.Nt, n = A.n;
    const float *cv = A.curve + (size_t)warp * n;
    float best = __int_as_float(0x7f800000);
    int bl = 0x7fffffff;
    for (int l = lane; l < n; l += 32) {
        const float v = cv[l];
        if (v < best) {  // l increases: ties keep the lowest
            best = v;
            bl = l;
        }
    }
#pragma unroll
    for (int off = 16; off; off >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, off);
        const int ol = __shfl_xor_sync(0xffffffffu, bl, off);
        if (ob < best || (ob == best && ol < bl)) {
            best = ob;
            bl = ol;
        }
    }
    const double invM = 1.0 / A.M;
    const int st = A.st_q[i] ? 1 : (A.st_t[j] ? 2 : 0);
    auto shift_at = [&](int l, double &sx, double &sy) {
        sx = sy = 0.0;
        if (A.translation) {
            const double2 c = A.cs64[l];
            const double ajx = A.ctr_t[2 * j], ajy = A.ctr_t[2 * j + 1];
            sx = A.ctr_q[2 * i] - (c.x * ajx - c.y * ajy);
            sy = A.ctr_q[2 * i + 1] - (c.y * ajx + c.x * ajy);
        }
    };
    if (lane == 0) {
        sw_result r;
        if (st || bl >= n) {
            const double nan = __longlong_as_double(0x7ff8000000000000ULL);
            r.best_l = -1;
            r.status = st ? st : 1;
            r.angle_rad = __int_as_float(0x7fc00000);
            r.shift[0] = r.shift[1] = nan;
            r.d2 = nan;
        } else {
            r.best_l = bl;
            r.status = 0;
            r.angle_rad = (float)(A.dalpha * bl);
            shift_at(bl, r.shift[0], r.shift[1]);
            r.d2 = (double)best * invM;
        }
        r.template_index = j;
        reinterpret_cast<sw_result *>(A.out)[warp] = r;
    }
    if (A.full && warp == 0) {
        const int bad = st != 0;
        for (int l = lane; l < n; l += 32) {
            A.full[l] = bad ? __longlong_as_double(0x7ff8000000000000ULL) : (double)cv[l] * invM;
            if (A.shifts) shift_at(l, A.shifts[2 * l], A.shifts[2 * l + 1]);
        }
    }
}

template <int CC>
cudaError_t launch_tiles(const MswArgs &a, int nblk, cudaStream_t st)
{
    const size_t smem = msw_smem(CC);
    cudaError_t e = cudaFuncSetAttribute(k_msw<CC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    const dim3 grid(a.Nq * a.Nt, (a.n + kMswR - 1) / kMswR, nblk);
    k_msw<CC><<<grid, kMswThreads, smem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_msw(const MswArgs &args, cudaStream_t st)
{
    if (args.Nq <= 0 || args.Nt <= 0) return cudaSuccess;
    if (args.n > 1024 || (size_t)args.Nq * args.Nt > 0x7fffffffu) return cudaErrorInvalidValue;
    MswArgs a = args;
    a.dalpha = 6.283185307179586 / a.n;
    cudaError_t e = cudaMemsetAsync(a.curve, 0, sizeof(float) * (size_t)a.Nq * a.Nt * a.n, st);
    if (e != cudaSuccess) return e;
    // the columns in equal blocks of at most 256
    const int nblk = (a.n + 255) / 256;
    switch ((a.n + 64 * nblk - 1) / (64 * nblk)) {
    case 1: e = launch_tiles<1>(a, nblk, st); break;
    case 2: e = launch_tiles<2>(a, nblk, st); break;
    case 3: e = launch_tiles<3>(a, nblk, st); break;
    default: e = launch_tiles<4>(a, nblk, st); break;
    }
    if (e != cudaSuccess) return e;
    const int threads = 256;
    const long long warps = (long long)a.Nq * a.Nt;
    k_msw_decide<<<(unsigned)((warps * 32 + threads - 1) / threads), threads, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace swk
