"""CPU: the kernels' index arithmetic on lattices with a side or a plane close to 2^31 sites, compiled
for the host with signed overflow trapped, against 64-bit divisions."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "lf2_arith.cuh"
using namespace lf2;
static void fail(const char *what, long long at) { printf("%s at %lld\n", what, at); exit(1); }
static void walk(int nx, int ny, int nz, long long stride, long long first, int steps) {
    const Geom g{nx, ny, nz, (long long)nx * ny * nz};
    const Stride3 d = make_stride3(stride, g);
    SiteWalk w(first, g);
    for (int k = 0; k < steps && w.s < g.sites; ++k, w.advance(d, g)) {
        const long long s = first + k * stride, r = s / nx;
        if (w.s != s || w.x != s % nx || w.y != r % ny || w.z != r / ny) fail("walk", s);
    }
}
static void plane(int nx, int ny) {
    const Geom g{nx, ny, 1, (long long)nx * ny};
    const long long p = (long long)nx * ny;
    const long long at[] = {0, 1, nx - 1, nx, 2LL * nx - 1, p / 2, p - nx, p - 2, p - 1};
    for (long long i : at) {
        if (i < 0 || i >= p) continue;
        const PlaneNbr n((int)i, g);
        const long long y = i / nx, x = i % nx;
        if (n.xm != y * nx + (x + nx - 1) % nx || n.xp != y * nx + (x + 1) % nx ||
            n.ym != (y + ny - 1) % ny * nx + x || n.yp != (y + 1) % ny * nx + x)
            fail("plane", i);
    }
}
int main() {
    const int big = 2147483647;
    for (long long stride : {256LL, 152LL * 4 * 256, 152LL * 16 * 256, 155189LL})
        for (int side : {big, big - 1, big - 300, big - 100000, 1 << 30})
            for (long long first : {0LL, 255LL, stride - 1}) {
                walk(side, 3, 2, stride, first, 200000);
                walk(1, side, 2, stride, first, 200000);
                walk(3, side, 1, stride, first, 200000);
                walk(1, 1, side, stride, first, 200000);
                walk(5, 1, side / 5, stride, first, 200000);
            }
    for (int s = 1; s < 12; ++s) walk(s, 13 - s, 7, 17, s, 100), plane(s, 13 - s), plane(1, s);
    plane(1000, 2147483), plane(65536, 32767), plane(big - 256, 1), plane(1, big - 256), plane(1 << 20, 2047);
    puts("ok");
}
"""


def test_coordinates_and_neighbours_near_2_to_the_31(tmp_path):
    from paper_1508_05610_gb300 import build
    src, exe = tmp_path / "geometry.cu", tmp_path / "geometry"
    src.write_text(SOURCE)
    cmd = [build._nvcc(), *build.ARCH, "-std=c++17", "-O1", "-I", build.CSRC, "-o", str(exe), str(src)]
    trap = ["-Xcompiler", "-fsanitize=signed-integer-overflow,-fsanitize-undefined-trap-on-error"]
    r = subprocess.run(cmd + trap, capture_output=True, text=True)
    if r.returncode != 0:
        pytest.skip("the host compiler cannot trap signed overflow: " + r.stderr[-200:])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", (r.returncode, r.stdout[-200:])
