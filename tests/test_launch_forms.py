"""The launch rules (sw_forms.h) on the host: tests/c_abi/launch_forms.cpp
prints their choices for the resident clusters that the runtime reports on a
GB300 (152 SMs) and for a part with fewer GPCs' worth of them.  No device."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# SMs, clusters of 1..8 CTAs at one CTA per SM, and at two
GB300 = [152, 152, 76, 46, 36, 28, 23, 15, 15, 304, 152, 97, 74, 58, 46, 38, 36]
SMALL = [92, 92, 46, 27, 21, 16, 13, 8, 8, 184, 92, 55, 43, 33, 26, 20, 19]
OPT_IN = 227 * 1024 - 512


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("forms") / "launch_forms")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I",
                    os.path.join(ROOT, "paper_2503_13756_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "c_abi", "launch_forms.cpp"), "-o", exe], check=True)

    def ask(device, queries):
        r = subprocess.run([exe, *map(str, device)], text=True, capture_output=True, check=True,
                           input="\n".join("%s %d %d %d %d" % q for q in queries))
        rows = [tuple(map(int, line.split())) for line in r.stdout.splitlines()]
        assert len(rows) == len(queries)
        return rows
    return ask


def _cap(device, per_sm, width):
    return device[8 * (per_sm - 1) + width]


@pytest.mark.parametrize("device", [GB300, SMALL], ids=["gb300", "small"])
def test_projector_clusters_are_resident_at_once(rules, device):
    for kind, per_sm in (("slice", 1), ("grid", 2)):
        count = range(1, 400)
        widths = [w for w, in rules(device, [(kind, nb, 96, 180, 0) for nb in count])]
        assert widths[0] == 8 and widths[-1] == 1
        for nb, w in zip(count, widths):
            assert w in (1, 2, 4, 8)
            assert w == 1 or nb <= _cap(device, per_sm, w), (kind, nb, w)
        assert sorted(widths, reverse=True) == widths


def _zeros(n, M):  # the FP16 split's rows of a template
    return n // 2 * (-(-2 * M // 64) * 64 - 2 * M) * 4


@pytest.mark.parametrize("device", [GB300, SMALL], ids=["gb300", "small"])
def test_spectrum_forms_fit_the_device(rules, device):
    queries = [("spectrum", nb, n, M, _zeros(n, M))
               for n in (4, 60, 64, 128, 256, 300, 360, 512, 600, 720, 1024)
               for M in (1, 33, 64, 96, 100, 128, 160, 192, 224, 256, 512, 1024)
               for nb in (1, 2, 8, 15, 16, 23, 24, 36, 46, 48, 74, 76, 80, 97, 152, 153, 310, 2000)]
    seen = set()
    for (_, nb, n, M, _), (ok, nsig, w, half, dense, smem) in zip(queries, rules(device, queries)):
        assert ok and nsig in (8, 16) and smem <= OPT_IN
        assert 1 <= w <= min(8, -(-M // (2 * nsig))) and (w > 1) + half + dense <= 1
        assert not dense or 4 * (smem + 1024 + 160) <= 228 * 1024  # 1 KB is the system's
        seen.add(w)
        if w > 1:
            sets = -(-nb // _cap(device, 2 if 2 * (smem + 1536) <= 228 * 1024 else 1, w))
            assert nb <= device[0] and sets <= 4, (nb, n, M, w)
    assert seen == set(range(1, 9))


def test_one_cluster_too_many_is_counted_as_a_second_set(rules):
    # of clusters of 8 with one CTA per SM, 15 are resident
    assert rules(GB300, [("slice", 15, 96, 180, 0), ("slice", 16, 96, 180, 0)]) == [(8,), (4,)]
    # 48 images of eight batches: 46 clusters of 3 fit (79 us), 76 of 2 (51 us; alone 65 us)
    assert [r[2] for r in rules(GB300, [("spectrum", 46, 360, 256, 0),
                                        ("spectrum", 48, 360, 256, 0)])] == [3, 2]


@pytest.mark.parametrize("N,nh,nb,width", [
    (64, 4, 2, 1), (64, 4, 20, 1), (64, 4, 46, 1), (64, 30, 36, 1),  # 9..13 us alone
    (96, 30, 20, 4), (96, 30, 46, 1), (32, 180, 20, 4), (32, 180, 46, 1), (96, 90, 20, 4), (96, 90, 46, 2), (192, 4, 2, 8),
    (192, 180, 76, 2), (192, 180, 77, 1)])
def test_images_of_little_work_stay_on_their_cta(rules, N, nh, nb, width):
    assert rules(GB300, [("slice", nb, N, nh, 0)]) == [(width,)]


# (n, M, images): us plain and in half batches, GB300
HALF = [((512, 256, 160), 164, 147), ((480, 64, 1000), 170, 123), ((500, 100, 310), 250, 184),
        ((360, 100, 420), 147, 133), ((360, 64, 420), 47, 45), ((900, 100, 160), 295, 266),
        ((1000, 4, 2000), 944, 575), ((320, 4, 600), 98, 88), ((1000, 33, 1000), 829, 629)]
PLAIN = [((360, 256, 420), 145, 156), ((320, 192, 600), 121, 147), ((600, 64, 600), 90, 139),
         ((768, 64, 600), 104, 223), ((720, 128, 420), 154, 274), ((1024, 64, 600), 188, 340),
         ((900, 64, 420), 133, 178), ((640, 192, 310), 203, 254), ((360, 256, 200), 92, 116)]


@pytest.mark.parametrize("size,plain,half", HALF + PLAIN)
def test_half_batches_where_they_are_faster(rules, size, plain, half):
    n, M, nb = size
    ok, _, w, got, _, smem = rules(GB300, [("spectrum", nb, n, M, _zeros(n, M))])[0]
    assert ok and w == 1 and smem <= OPT_IN
    assert got == (half < plain)


# (n, M, images): us at three and at four CTAs per SM, GB300
@pytest.mark.parametrize("size,three,four", [
    ((32, 1024, 600), 141, 106), ((8, 1024, 600), 88, 59), ((64, 512, 600), 90, 78),
    ((128, 33, 600), 63, 59), ((32, 1024, 420), 90, 90), ((128, 33, 420), 49, 49),
    ((216, 33, 600), 100, 100), ((256, 128, 1000), 96, 100)])
def test_four_ctas_per_sm_where_they_are_faster(rules, size, three, four):
    n, M, nb = size
    assert rules(GB300, [("spectrum", nb, n, M, _zeros(n, M))])[0][4] == (four < three)


# bins: us of 1500 images at n = 360 in pairs of stages and in single stages, GB300
@pytest.mark.parametrize("B,pairs,single", [
    (20, 263, 163), (32, 312, 196), (64, 386, 257), (96, 511, 384), (120, 607, 482), (256, 665, 726), (384, 1435, 1530)])
def test_ramp_stages_in_pairs_where_they_are_faster(rules, B, pairs, single):
    assert rules(GB300, [("ramp", B, 0, 0, 0)]) == [(pairs < single,)]


# (queries, templates): us with a block and with a warp per query, GB300
@pytest.mark.parametrize("Nq,Nt,block,warp", [
    (600, 129, 8, 4), (4000, 129, 31, 10), (100, 256, 4, 6), (4000, 256, 31, 12),
    (150, 500, 6, 8), (1000, 500, 12, 8), (30, 1000, 6, 10), (2000, 1000, 27, 18),
    (4000, 1000, 51, 39), (600, 4000, 22, 39)])
def test_best_template_by_block_where_it_is_faster(rules, Nq, Nt, block, warp):
    assert rules(GB300, [("best", Nq, Nt, 0, 0)]) == [(block < warp,)]
