// Prints the launch rules' choices (sw_forms.h) for sizes read from standard
// input, one query a line, on the device given by the arguments: the SMs, then
// the resident clusters of 1..8 CTAs at one and at two CTAs per SM.
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "sw_forms.h"

int main(int argc, char **argv)
{
    if (argc != 18) return 2;
    swk::DeviceForm d{};
    d.sms = atoi(argv[1]);
    for (int p = 0; p < 2; ++p)
        for (int w = 1; w <= 8; ++w) d.clusters[p][w] = atoi(argv[1 + 8 * p + w]);
    char kind[32];
    int a, b, c, e;
    while (scanf("%31s %d %d %d %d", kind, &a, &b, &c, &e) == 5) {
        if (!strcmp(kind, "slice")) {
            printf("%d\n", swk::slice_cluster(a, b, c, b / 2 + 1, d));  // b: N, c: nh
        } else if (!strcmp(kind, "grid")) {
            printf("%d\n", swk::slice_grid_cluster(a, d));
        } else if (!strcmp(kind, "spectrum")) {
            swk::SpectrumForm f{};
            const bool ok = swk::spectrum_form(a, b, c, 0, e, d, &f);  // e: zeros per image
            printf("%d %d %d %d %d %zu\n", ok, f.nsig, f.cluster, f.half, f.dense, f.smem);
        } else if (!strcmp(kind, "ramp")) {
            printf("%d\n", swk::ramp_pairs(a));
        } else if (!strcmp(kind, "best")) {
            printf("%d\n", swk::best_by_block(a, b, d));
        } else {
            return 3;
        }
    }
    return 0;
}
