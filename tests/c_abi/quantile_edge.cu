// The quantile kernel counts the levels below a node of the CDF in FP32 and
// trusts a count that is not within count_edge of a boundary between two.  Here
// every rounding of that count takes its worst allowed value: tails of half an
// ulp in F and F_B, a quotient off by two ulps (the bound of the fast division),
// on mantissas where an ulp is largest; a trusted count has to be the exact one.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>

#include "sw_internal.cuh"

static uint64_t state = 0x9e3779b97f4a7c15ull;
static double uniform()
{
    state ^= state << 13;
    state ^= state >> 7;
    state ^= state << 17;
    return (double)(state >> 11) * 0x1p-53;
}

static long long trusted = 0, wrong = 0;

// Counts at boundaries of M levels, `its` draws per level rule: F_B = th + tl with
// th in [1, th_max), the boundary c - 1/2 with c in (c_min M, M].
static void check(int M, int its, double th_max, double c_min)
{
    const float edge = swk::count_edge(M);
    for (int rule = 0; rule < 2; ++rule) {
        const float coff = rule == 0 ? 0.f : -0.5f;
        for (int it = 0; it < its; ++it) {
            const float th = (float)(1.0 + (th_max - 1.0) * uniform());
            const double tl = (it & 1 ? 1 : -1) * 0.5 * ((double)nextafterf(th, 4.f) - th);
            const double total = (double)th + tl;
            const int c = M - (int)((1.0 - c_min) * uniform() * M);
            // a node F with M F / F_B + coff = c - 1/2, and the floats around it,
            // with a tail to either side
            const double at = ((double)c - 0.5 - (double)coff) * total / M;
            if (!(at > 0.0) || at > total) continue;
            float fh = (float)at;
            const int away = (int)(uniform() * 11.0) - 5;
            for (int s = 0; s < abs(away); ++s) fh = nextafterf(fh, away < 0 ? 0.f : 4.f);
            const double half = 0.5 * ((double)nextafterf(fh, 4.f) - fh);
            const double quot = (double)M / (double)th;
            const float q0 = (float)quot;
            const double ulp = (double)nextafterf(q0, 1e30f) - q0;
            for (int side = -1; side <= 1; side += 2) {
                const double x64 = (double)M * ((double)fh + side * half) / total + (double)coff;
                const int exact = (int)std::floor(x64 + 0.5);
                for (int e = -2; e <= 2; ++e) {
                    float q = q0;
                    for (int s = 0; s < abs(e); ++s) q = nextafterf(q, e < 0 ? 0.f : 1e30f);
                    if (std::fabs((double)q - quot) > 2.0 * ulp) continue;
                    const float x = fmaf(fh, q, coff);
                    const float y = x + 12582912.f;  // rounds to an integer, as the kernel does
                    const float d = x - (y - 12582912.f);
                    if (fabsf(d) > edge) continue;
                    ++trusted;
                    wrong += (int)(y - 12582912.f) != exact;
                }
            }
        }
    }
}

int main()
{
    for (int M = 1; M <= 1024; M = M < 40 ? M + 1 : M + 1 + M / 16) check(M, 30000, 2.0, 0.0);
    // just above a power of two the mantissas of F_B, F, M / F_B and the count are
    // near 1 at once, where every half ulp is a whole unit of the bound
    for (int k = 5; k <= 9; ++k)
        for (int M = (1 << k) + (1 << k) / 128 + 1; M <= (1 << k) * 33 / 32; M += 1 + (1 << k) / 256)
            check(M, 200000, (double)M / (1 << k), (double)(1 << k) / M);
    printf("%lld trusted counts, %lld wrong\n", trusted, wrong);
    if (wrong || trusted < 1000) return 1;
    printf("ok\n");
    return 0;
}
