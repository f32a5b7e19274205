// sw_forms.h -- which form of a kernel a launch takes, from the call's sizes
// and the device alone.  Host code without CUDA, so that the rules can be
// checked without a device.
#pragma once

#include <algorithm>
#include <cstddef>

namespace swk {

// What the rules ask of the device: its multiprocessors, and how many clusters
// of w CTAs it holds at once where p CTAs fit an SM (clusters[p - 1][w], p = 1,
// 2, w = 1..8; 0: none).  The runtime knows the latter: a cluster stays within
// a GPC, and the GPCs of a part differ (a GB300 of 152 SMs holds 76, 46, 36,
// 28, 23, 15 and 15 clusters of 2..8 CTAs of one per SM, not 8 floor(19 / w)).
struct DeviceForm {
    int sms;
    int clusters[2][9];
};

// CTAs per image (a power of two, at most the portable cluster size 8) of the
// slice projector with a grid of N x N points in shared memory, one CTA per SM,
// and nh angles of nj samples: the widest cluster with room for all nb images at
// once.  A cluster too many runs after the others: 16 images in clusters of 8, of
// which 15 are resident, took 25 us at L = 64, n = 8, and 15 us in clusters of 4.
// The barriers and the copies of rows take some us, so an image of little work
// (the grid's FFTs and the samples, about us of one CTA) stays on its CTA.  Us
// alone and in clusters of 4 for 20 images, and of 2 for 46: L = 32, n = 8 10 and
// 12, 10 and 13; L = 16, n = 360 19 and 12, 20 and 22; L = 64, n = 60 15 and 14, 16
// and 17; L = 64, n = 180 27 and 16, 27 and 22.
inline int slice_cluster(int nb, int N, int nh, int nj, const DeviceForm &d)
{
    const double work = 0.00035 * N * N + 0.0032 * nj * nh;
    for (int P = 8; P > 1; P /= 2)
        if (nb <= d.clusters[0][P]) return work >= (P == 2 ? 10.5 : 5.0) ? P : 1;
    return 1;
}

// The same for its global grid build, two CTAs per SM.  Two CTAs of an SM
// share its pipes, so clusters of 8 and 4 gain until they fill two thirds of
// their places (of the time on one CTA per image, L = 160..256: 20 images 0.49
// in clusters of 8 and 0.51 in clusters of 4, 36 images 0.57 and 0.55; 37
// images 0.70 in clusters of 4 and 2, 72 images 0.78 and 0.75; 152 images 0.99
// in clusters of 2).
inline int slice_grid_cluster(int nb, const DeviceForm &d)
{
    for (int P = 8; P > 2; P /= 2)
        if (3 * nb <= 2 * d.clusters[1][P]) return P;
    return nb <= d.clusters[1][2] ? 2 : 1;
}

// The angle spectra (k_spectrum).
constexpr int kSpecThreads = 256;
constexpr size_t kSmemOptIn = 227 * 1024 - 512;  // dynamic shared memory of a CTA, beside the static
// An SM's 228 KB hold k CTAs of smem bytes (beside each the system's 1 KB and the static).
inline bool spectrum_fits(int k, size_t smem) { return k * (smem + 1536) <= 228 * 1024; }

struct SpectrumForm {
    int nsig;      // signals per FFT batch
    int cluster;   // CTAs per image
    bool half;     // half batches
    bool dense;    // four CTAs per SM (plain form)
    size_t smem;   // dynamic shared memory of a CTA
};

// Form for nb images of n angles and M levels; false if an image does not fit
// a CTA.  nsig_req: a requested batch width (0: none).  zeros: elements of zero
// padding written per image (the low-precision rows').
inline bool spectrum_form(int nb, int n, int M, int nsig_req, long long zeros, const DeviceForm &d,
                          SpectrumForm *f)
{
    // signals per FFT batch: 16 by default, 8 at n = 1024; a requested
    // width is taken when its buffers fit (2 n nsig complex values)
    int nsig = n <= 512 ? 16 : 8;
    if ((nsig_req == 4 || nsig_req == 8 || nsig_req == 16) && (size_t)n * nsig_req <= 8192)
        nsig = nsig_req;
    // two batch buffers (the staged input and the FFT's other buffer),
    // within the 227 KB a CTA can hold
    auto smem_of = [&](int ns) { return 8 * ((size_t)2 * n * ns + M + n); };
    while (nsig > 4 && smem_of(nsig) > kSmemOptIn) nsig /= 2;
    const size_t smem = smem_of(nsig);
    if (smem > kSmemOptIn) return false;
    *f = SpectrumForm{nsig, 1, false, false, smem};
    const int nbatch = (M + 2 * nsig - 1) / (2 * nsig);

    // A cluster per image where it is expected to save a tenth of the time, by
    // the times of a launch in us on a GB300 (fitted at n = 8..1024, M = 64..1024;
    // nine in ten of 11,658 measured launches from 10% below to 7% above): 7.5 + b
    // nbatch + z with a CTA per image, b the time of a batch and z that of the
    // padding; 5 + 5 + 0.86 b ceil(nbatch / w) + 0.29 b nbatch + z / w in
    // clusters of w CTAs (two barriers, the longest CTA's batches, the ordered
    // sum of the terms), the batches 1.16 times longer where CTAs share an SM,
    // and all but the launch again for every further set of resident clusters:
    // 48 images at n = 360, M = 256 take 65 us alone, 51 us in clusters of 2, and
    // 79 us in clusters of 3, of which 46 are resident.
    const double b = nsig / 16.0 * (nsig == 16 ? 1.0 + 0.0168 * n : 3.5 + 0.0156 * n) *
                     (M & 1 ? 1.5 : 1.0);  // odd M: copies and stores level by level
    const double z = 0.0012 * (double)zeros;
    const size_t per_batch = 8 * (size_t)((n / 2) / (kSpecThreads / nsig) + 1) * kSpecThreads;
    double best = 0.9 * (7.5 + b * nbatch + z);
    for (int w = 2; w <= std::min(8, nbatch) && nb <= d.sms; ++w) {
        const int per = (nbatch + w - 1) / w;
        const size_t need = smem + per_batch * per;
        const int fit = need > kSmemOptIn ? 0 : d.clusters[spectrum_fits(2, need) ? 1 : 0][w];
        if (fit == 0) continue;
        const int sets = (nb + fit - 1) / fit;
        const double shared = std::min(nb, fit) * w > d.sms ? 1.16 : 1.0;
        const double t = 5 + sets * (5 + shared * b * (0.86 * per + 0.29 * nbatch) + z / w);
        if (t < best) {
            best = t;
            f->cluster = w;
            f->smem = need;
        }
    }
    if (f->cluster > 1) return true;

    // Half batches, where the plain form's buffers leave room for fewer than
    // three CTAs per SM and the images take more than one wave.  Of the plain
    // form's time: batches of 16 with one plain CTA per SM (n > 440) 0.55..0.92;
    // with two, only where the half form takes a wave fewer and wastes none of a
    // batch or the batches are few (M = 64 0.98 and 0.94, M = 100 0.91, but M =
    // 128..256 1.02..1.08 at 310 and 420 images, and 1.05..1.21 at 600, which fill
    // two plain waves).  Batches of 8 (n > 512) halve to rows of 16 bytes per store,
    // and many images then write parts of sectors (1.24 at 420 images and M = 100,
    // 1.43..1.84 at 420 to 600 and M = 64): only with one plain CTA per SM and at
    // most two waves, or few levels.  Levels of one half batch always gain.
    const int ctas = smem > kSmemOptIn / 2 ? 1 : 2, slots = d.sms * ctas;
    const int halves = (M + nsig - 1) / nsig;  // half batches
    if (nsig >= 8 && smem > kSmemOptIn / 3 && nb > slots) {
        const int waves = (nb + slots - 1) / slots, waves_half = (nb + 3 * d.sms - 1) / (3 * d.sms);
        const bool odd = halves & 1;
        f->half = halves == 1 ||
                  (nsig == 16 ? ctas == 1 || (waves_half < waves && (M <= 64 || odd))
                              : ctas == 1 && (M <= 40 || (odd && waves <= 2)));
        if (f->half) f->smem = smem_of(nsig / 2);
    }

    // Four CTAs per SM, by 64 registers a thread instead of 80, where shared
    // memory holds them (n <= 200) and three do not hold all images.  Of the time
    // at three: n = 8..32 0.69..0.76 at 520 and 600 images, 0.80..0.84 at 1000, n =
    // 128 0.91 and 0.93, n = 200 0.94 and 0.96; up to 456 images 0.99..1.04.
    f->dense = !f->half && spectrum_fits(4, smem) && nb > 3 * d.sms;
    return true;
}

// The ramp filter (k_ramp) of rows of B bins: FFT stages in pairs?  Pairs save
// passes and barriers but hold twice the registers (64 against 32, four CTAs per
// SM against eight) and leave most threads of a short row's pass idle.  Time in
// pairs over single stages, 24 and 1500 images at n = 360: B = 32 1.39 and 1.60, B
// = 64 1.34 and 1.50, B = 120 1.15 and 1.26; B = 128 1.19 and 1.08, B = 192 1.10
// and 1.07, B = 256 1.01 and 0.92, B = 384 0.94 and 0.94.  At 600 images, one wave
// in pairs, 0.95..1.00 at B = 108..192 and 0.89..0.94 above.
inline bool ramp_pairs(int B) { return B >= 128; }

// The best template of Nq queries among Nt (k_best_template): a block per query
// instead of a warp?  A warp reads its results in chains of Nt / 32, a block in
// chains of Nt / 256 but with eight warps and a barrier per query, so the block
// gains while the chip is not filled with blocks.  Block and warp in us: 150 queries
// of 129 and 1000 templates 4 and 4, 8 and 10; 600 of 129 and 1000 8 and 4, 10
// and 10; 4000 of 129 and 1000 31 and 10, 51 and 39; 1000 of 2000 21 and 22; 4000
// of 4000 113 and 131.
inline bool best_by_block(int Nq, int Nt, const DeviceForm &d)
{
    return Nt > 128 && (Nq <= d.sms + Nt / 2 || Nt >= 4000);
}

}  // namespace swk
