"""The rules that choose launch shapes (csrc/lf_march2d.cuh, csrc/lf_cvt.h),
compiled for the host."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.join(os.path.dirname(__file__), "..")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

PROGRAM = r"""
#include "lf_march2d.cuh"
#include "lf_cvt.h"
#include <algorithm>
#include <chrono>
#include <cstdio>
#include <cstring>
using namespace lf;

static double us_per_call(int nx, int ny, bool iso)
{
    double best = 1e9;
    for (int batch = 0; batch < 20; ++batch) {
        const auto t = std::chrono::steady_clock::now();
        volatile int sink = 0;
        for (int i = 0; i < 500; ++i) sink = sink + march::pair_shape(nx, ny, 0, iso, true, 152).rows;
        best = std::min(best, std::chrono::duration<double>(std::chrono::steady_clock::now() - t).count() / 500 * 1e6);
    }
    return best;
}

int main()
{
    char what[16];
    int a[6];
    while (std::scanf("%15s %d %d %d %d %d %d", what, a, a + 1, a + 2, a + 3, a + 4, a + 5) == 7) {
        if (!std::strcmp(what, "time")) std::printf("%f\n", us_per_call(a[0], a[1], a[2] != 0));
        if (!std::strcmp(what, "convert")) std::printf("%u\n", convert_threads(a[0], a[1], a[2], a[3]));
        if (!std::strcmp(what, "pair")) {
            const march::PairShape c = march::pair_shape(a[0], a[1], a[2], a[3] != 0, a[4] != 0, 152);
            std::printf("%d %d\n", c.narrow, c.rows);
        }
        if (!std::strcmp(what, "spread")) std::printf("%d\n", march::spread(a[0], a[1], a[2], a[3], a[4], a[5]));
    }
}
"""


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("needs nvcc")
    d = tmp_path_factory.mktemp("shape")
    (d / "p.cu").write_text(PROGRAM)
    subprocess.run([NVCC, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_1102_3094_gb300", "csrc"),
                    str(d / "p.cu"), "-o", str(d / "p")], check=True)

    def run(*queries):
        text = "".join(" ".join(map(str, list(q) + [0] * (7 - len(q)))) + "\n" for q in queries)
        out = subprocess.run([str(d / "p")], input=text, capture_output=True, text=True, check=True).stdout
        return [[float(v) for v in line.split()] for line in out.splitlines()]

    return run


@pytest.mark.parametrize("element_bytes,threads,most,per_sm,want", [
    (4, 128, 3, 1, 1), (4, 128, 3, 2, 2), (4, 128, 3, 3, 0), (4, 128, 3, 4, 0), (4, 64, 6, 5, 5), (4, 64, 6, 6, 0),
    # FP64: two rounds of two; more rounds, or 64 threads, take what fits
    (8, 128, 3, 1, 1), (8, 128, 3, 2, 2), (8, 128, 3, 3, 0), (8, 128, 3, 4, 2), (8, 128, 3, 5, 0), (8, 128, 3, 6, 0),
    (8, 64, 4, 2, 2), (8, 64, 4, 3, 3), (8, 64, 4, 4, 0), (8, 64, 4, 8, 0)])
def test_spread_of_a_march(ask, element_bytes, threads, most, per_sm, want):
    # the last SM's share may be short
    for ctas in (152 * per_sm, 152 * (per_sm - 1) + 1):
        assert ask(("spread", element_bytes, threads, most, ctas, 1, 152)) == [[want]]


@pytest.mark.parametrize("nx,ny", [(256, 256), (1024, 1024), (2999, 1777), (4096, 4096), (32, 100000)])
def test_a_shape_is_cheap_to_choose(ask, nx, ny):
    """lf_step chooses it for every step: well under the launch itself (a few microseconds)."""
    for iso in (0, 1):
        assert ask(("time", nx, ny, iso))[0][0] < 2.0


@pytest.mark.parametrize("nx,ny", [(700, 611), (1024, 1024), (2048, 512), (512, 2048), (1400, 1300), (1800, 1900), (2048, 2048),
                                   (3000, 1500), (2500, 2400), (3000, 3000), (300, 5000)])
def test_compact_march_without_hydrodynamics_fills_the_schedulers(ask, nx, ny):
    """Measured best at every one of these: lanes so short that three warps per scheduler hold the lattice."""
    (narrow, rows), = ask(("pair", nx, ny, 0, 0, 0))
    strips, places = -(-nx // (56 if narrow else 120)), 152 * (2 if narrow else 1)
    ctas = strips * -(-ny // int(2 * rows))
    assert 2 * places < ctas <= 3 * places


@pytest.mark.parametrize("groups,planes,want", [(1, 1, 32), (1024, 1, 32), (1024, 9, 32), (8192, 9, 32), (16384, 9, 64),
                                                (34304, 9, 128), (69376, 9, 256), (311296, 1, 256), (310784, 1, 128), (1 << 29, 1, 256)])
def test_a_small_conversion_is_spread_over_the_sms(ask, groups, planes, want):
    """Two groups per thread and 152 SMs: the largest block that gives every SM four, 32 threads at least."""
    assert ask(("convert", groups, 2, planes, 152)) == [[want]]
