"""The kernel that a call takes by default (``csrc/weo_route.h``), compiled alone.

``MEASURED`` has us per M_eo on one GB300 of every kernel the rules choose between: the
chosen one is at most 3 % slower than the fastest, so that no rule sends a size to a
kernel which its own measurement shows to be the slower one.
"""

import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2303_08609_gb300", "csrc")

# bits, link reals, V/2, right-hand sides: one site per thread, split, tiles
MEASURED = """
16 12 65536 2 26.75 23.47 32.60
16 12 65536 8 84.54 83.24 78.02
16 12 65536 9 93.09 92.76 96.91
16 12 65536 10 101.26 102.23 100.38
16 12 65536 12 119.07 121.37 109.45
16 12 65536 13 127.97 130.99 128.15
16 12 331776 2 106.94 106.45 147.34
16 12 331776 3 151.26 155.21 178.55
16 12 331776 4 196.17 204.05 195.93
16 12 331776 5 240.97 252.99 275.93
16 12 331776 6 285.53 301.80 291.99
16 12 331776 7 329.99 350.66 322.16
16 12 331776 9 419.06 448.34 411.90
16 12 331776 12 552.59 594.85 479.49
16 12 32768 16 83.81 83.04 84.80
16 12 131072 4 85.48 84.15 83.03
16 12 131072 6 119.96 122.10 122.34
16 12 262144 3 121.88 123.40 999
16 12 331776 1 62.83 56.46 999
16 12 589824 1 101.44 96.73 999
16 12 589824 2 179.20 185.00 999
16 12 1048576 1 168.36 165.59 999
16 12 1048576 2 306.75 323.17 999
16 12 5308416 1 788 817 9999
16 18 65536 5 60.58 51.62 64.22
16 18 65536 8 84.77 79.51 78.60
16 18 65536 9 91.29 88.52 97.70
16 18 65536 10 102.26 97.37 101.31
16 18 65536 12 120.21 115.42 110.08
16 18 65536 13 126.52 124.29 129.00
16 18 331776 3 155.01 150.45 180.10
16 18 331776 4 197.25 196.54 197.51
16 18 331776 5 239.86 242.94 277.96
16 18 331776 6 282.79 289.23 294.00
16 18 331776 7 325.61 335.56 324.19
16 18 331776 9 411.34 428.30 414.44
16 18 331776 10 454.24 474.72 434.17
16 18 331776 13 581.70 613.78 550.33
16 18 32768 16 83.37 79.13 85.40
16 18 131072 4 87.80 80.72 83.98
16 18 131072 6 123.35 116.78 123.36
16 18 5308416 1 867 851 9999
32 18 65536 4 59.24 50.35 51.65
32 18 65536 8 108.05 94.58 84.58
32 18 65536 9 115.49 104.52 105.11
32 18 65536 13 161.24 146.78 137.32
32 18 331776 3 207.14 188.25 192.44
32 18 331776 4 261.78 243.11 215.43
32 18 331776 5 317.00 297.25 295.06
32 18 331776 6 373.46 351.83 314.36
32 18 331776 9 537.62 516.52 440.47
32 18 32768 16 104.79 92.39 93.07
32 18 131072 4 113.47 98.47 92.01
32 18 131072 6 160.84 141.21 130.85
32 12 65536 8 99.90 86.62 82.58
32 12 65536 9 112.56 96.58 103.39
32 12 65536 10 118.24 106.51 106.37
32 12 65536 13 151.20 136.36 135.87
32 12 331776 4 245.61 220.77 208.29
32 12 331776 5 302.01 271.99 289.95
32 12 331776 6 355.33 323.43 308.65
32 12 331776 9 523.17 477.03 436.03
32 12 32768 16 97.32 85.83 91.81
32 12 131072 6 148.10 128.11 127.69
16 18 589824 2 183.10 179.44 257.54
16 18 589824 3 260.89 261.01 311.33
16 18 589824 4 337.97 343.13 340.26
16 18 589824 6 489.93 507.57 511.31
16 18 589824 7 566.02 589.95 569.34
32 18 589824 2 254.50 232.40 280.25
32 18 589824 3 354.08 329.01 329.78
32 18 589824 4 452.50 425.48 369.84
32 18 589824 6 647.89 621.08 540.04
32 18 589824 7 748.85 716.73 591.98
32 12 589824 2 233.71 205.02 269.16
32 12 589824 3 329.60 295.76 321.27
32 12 589824 4 426.32 387.66 358.86
32 12 589824 6 621.12 568.97 532.02
32 12 589824 7 725.83 660.63 585.54
16 12 589824 2 176.91 183.81 254.68
16 12 589824 3 256.87 270.69 308.85
16 12 589824 4 335.85 357.34 337.59
16 12 589824 6 495.15 530.73 508.27
16 12 589824 7 575.28 617.81 566.84
16 18 1048576 2 315.93 311.52 450.40
16 18 1048576 3 451.45 454.95 543.68
16 18 1048576 4 586.97 599.94 588.95
16 18 1048576 6 860.57 890.66 889.12
16 18 1048576 7 997.22 1035.94 996.89
32 18 1048576 2 439.51 409.29 478.49
32 18 1048576 3 612.72 579.34 563.13
32 18 1048576 4 781.71 749.34 629.44
32 18 1048576 6 1140.83 1096.95 940.11
32 18 1048576 7 1333.53 1276.48 1042.71
32 12 1048576 2 400.95 360.00 460.55
32 12 1048576 3 574.80 519.64 551.05
32 12 1048576 4 756.60 679.85 612.32
32 12 1048576 6 1114.07 1001.74 922.55
32 12 1048576 7 1297.27 1170.31 1025.51
16 12 1048576 2 304.94 322.00 444.69
16 12 1048576 3 447.00 476.24 539.47
16 12 1048576 4 587.93 629.98 584.45
16 12 1048576 6 872.43 937.46 881.55
16 12 1048576 7 1014.68 1092.77 991.35
16 18 5308416 2 1563.05 1580.24 2296.16
16 18 5308416 3 2284.06 2337.27 2797.42
32 18 5308416 2 2281.02 2099.01 2574.38
32 12 5308416 3 3065.02 2756.86 3018.95
16 12 1280000 1 200.21 199.88 9999
16 12 2048000 1 313.86 316.99 9999
"""

# FP64: link reals, V/2, right-hand sides: rows (16-site CTAs), pairs (32 sites)
MEASURED_F64 = """
18 256 1 11.36 17.46
18 256 4 11.57 18.15
18 256 12 18.93 18.43
18 2048 1 15.23 18.32
18 2048 2 22.24 18.60
18 2048 3 27.97 32.79
18 2048 4 34.95 32.88
18 2048 12 87.63 89.99
18 3072 1 18.96 18.44
18 3072 2 28.45 32.72
18 3072 3 34.98 32.98
18 3072 4 49.48 47.50
18 3072 12 125.76 119.44
18 4096 1 22.60 18.65
18 4096 2 34.97 32.90
18 4096 3 49.47 47.49
18 4096 4 57.50 62.05
18 4608 1 22.80 18.75
18 4608 4 65.28 62.28
18 7560 1 35.20 33.19
18 7560 2 57.57 62.26
18 7560 3 80.29 76.11
18 7560 4 103.36 105.05
18 7560 12 293.47 278.71
12 256 1 14.77 21.13
12 256 12 24.72 21.67
12 2048 1 19.87 21.52
12 2048 2 30.00 21.89
12 2048 3 37.36 39.63
12 2048 4 46.56 39.68
12 2048 12 121.42 109.13
12 3072 1 24.76 21.68
12 3072 2 37.85 39.65
12 3072 3 46.59 39.78
12 4096 1 30.03 21.88
12 4096 4 78.79 75.18
12 4608 4 89.42 75.36
12 7560 1 46.55 39.90
12 7560 2 78.74 75.52
12 7560 12 411.68 338.47
"""


@pytest.fixture(scope="module")
def route(tmp_path_factory):
    """(bits, reals, V/2, nrhs) -> 0 one site, 1 split (bits 64: 4 its rows kernel), 2 tiles"""
    gxx = shutil.which("g++") or pytest.skip("no g++")
    d = tmp_path_factory.mktemp("route")
    src = d / "route.cc"
    src.write_text('#include <cstdio>\n#include "weo_route.h"\nint main() { int b, l, n; long long v;\n'
                   'while (scanf("%d %d %lld %d", &b, &l, &v, &n) == 4)\n'
                   'printf("%d\\n", b == 64 && weo::rows_pay(l == 12, v, n) ? 4 :\n'
                   '       (int)weo::default_route(b == 64, b == 16, l == 12, v, n)); }\n')
    subprocess.run([gxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(d / "route")], check=True)

    def ask(rows):
        text = "\n".join(" ".join(map(str, r)) for r in rows)
        return list(map(int, subprocess.run([str(d / "route")], input=text, capture_output=True, text=True,
                                            check=True).stdout.split()))

    return ask


def test_the_chosen_kernel_is_the_measured_one(route):
    rows = [line.split() for line in MEASURED.split("\n") if line]
    for r, got in zip(rows, route([r[:4] for r in rows])):
        us = list(map(float, r[4:]))
        assert us[got] <= 1.03 * min(us), r


def test_rows_and_pairs_are_the_measured_ones(route):
    rows = [line.split() for line in MEASURED_F64.split("\n") if line]
    for r, got in zip(rows, route([["64"] + r[:3] for r in rows])):
        us = {4: float(r[3]), 1: float(r[4])}
        assert us[got] <= 1.03 * min(us.values()), r


def test_site_blocks_leave_other_lattices_alone(tmp_path):
    """The setting holds from Lx = 16 to 64; elsewhere the default kernel stays."""
    gxx = shutil.which("g++") or pytest.skip("no g++")
    (tmp_path / "b.cc").write_text('#include "weo_route.h"\nint main(int n, char **v) { for (int l = 1; l < 100; ++l)\n'
                                   'if (weo::site_blocks_apply(true, l) != (2 * l >= 16 && 2 * l <= 64) ||\n'
                                   'weo::site_blocks_apply(false, l)) return 1; return 0; }\n')
    subprocess.run([gxx, "-std=c++17", "-I", CSRC, str(tmp_path / "b.cc"), "-o", str(tmp_path / "b")], check=True)
    assert subprocess.run([str(tmp_path / "b")]).returncode == 0
    with open(os.path.join(CSRC, "weo_launch.cuh")) as f:
        assert f.read().count("cfg.blocked") == 1  # only through the rule


def test_tuner_times_thread_counts_where_they_matter(tmp_path):
    """12-real 16-bit links at V/2 = 5308416 (48^3 x 96) run one site per thread."""
    gxx = shutil.which("g++") or pytest.skip("no g++")
    (tmp_path / "t.cc").write_text('#include "weo_route.h"\nint main() { using weo::threads_matter;\n'
                                   'return !(threads_matter(false, true, true, 5308416, 1) && threads_matter(false, true, true, 331776, 3)\n'
                                   '&& !threads_matter(false, true, true, 331776, 1) && !threads_matter(false, false, true, 5308416, 1)\n'
                                   '&& !threads_matter(true, false, false, 331776, 1) && !threads_matter(false, true, false, 331776, 12)); }\n')
    subprocess.run([gxx, "-std=c++17", "-I", CSRC, str(tmp_path / "t.cc"), "-o", str(tmp_path / "t")], check=True)
    assert subprocess.run([str(tmp_path / "t")]).returncode == 0
    with open(os.path.join(CSRC, "tune.cu")) as f:
        assert "threads_matter(" in f.read()


def test_offsets_of_the_split_kernels(route):
    """Beyond 2^28 sites, where 32-bit offsets end, nothing takes them."""
    rows = [(b, l, v, n) for b in (64, 32, 16) for l in (18, 12) for v in (2 ** 28 + 1, 2 ** 31 - 1) for n in (1, 2, 3, 5, 8)]
    assert 1 not in route(rows)


@pytest.mark.gpu
@pytest.mark.parametrize("fmt", [18, 12])
@pytest.mark.parametrize("dims", [(8, 8, 8, 8), (8, 8, 8, 16), (6, 10, 8, 14)])
def test_fp64_rows_and_pairs_agree(dims, fmt):
    """Counts that alternate between the two kernels, ragged against both CTA sizes."""
    import torch

    import paper_2303_08609_gb300 as weo

    g = torch.Generator(device="cuda").manual_seed(1102)
    V, n = int(np.prod(dims)), 7
    U = 0.4 * torch.randn(4, V, 3, 3, dtype=torch.complex128, device="cuda", generator=g)
    x = torch.randn(n, 4, 3, V // 2, dtype=torch.complex128, device="cuda", generator=g)
    with weo.WilsonEO(dims, 0.13, U, prec="f64", linkfmt=fmt) as op:
        for dag in (False, True):
            one = torch.stack([op.apply(x[r].contiguous(), dag=dag) for r in range(n)])
            for k in range(2, n + 1):
                assert torch.equal(op.apply(x[:k].contiguous(), dag=dag), one[:k])


@pytest.mark.gpu
@pytest.mark.parametrize("prec,fmt,counts", [("f16", 12, (2, 3, 4, 5, 6, 7)), ("bf16", 18, (3, 5, 6, 7)),
                                             ("f32", 18, (3, 4, 5)), ("f32", 12, (4, 5))])
def test_right_hand_sides_on_both_sides_of_the_rules(prec, fmt, counts):
    """V/2 = 331776, where these counts cross the rules: each right-hand side is bitwise
    the single one (split for FP32 and 18-real links; 12-real 16-bit ones too)."""
    import torch

    import paper_2303_08609_gb300 as weo

    dims, n = (24, 24, 24, 48), max(counts)
    g = torch.Generator(device="cuda").manual_seed(1101)
    V = int(np.prod(dims))
    # any links do: the kernels are compared with one another
    U = 0.4 * torch.randn(4, V, 3, 3, dtype=torch.complex64, device="cuda", generator=g)
    x = torch.randn(n, 4, 3, V // 2, dtype=torch.complex64, device="cuda", generator=g)
    with weo.WilsonEO(dims, 0.13, U, prec=prec, linkfmt=fmt) as op:
        for dag in (False, True):
            one = torch.stack([op.apply(x[r].contiguous(), dag=dag) for r in range(n)])
            for k in counts:
                assert torch.equal(op.apply(x[:k].contiguous(), dag=dag), one[:k])
