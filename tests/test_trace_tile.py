"""The tile of pixels that a warp of the channel-map trace follows: whatever
the image's shape, at most a quarter of the lanes more than the best tile
needs go without a ray (so a strip one pixel wide or high fills them), square
images keep 8 x 4, and a tile's lanes are its 32 pixels, each once."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = """
#include <cstdio>
#include <cstdlib>
#include "trace_tile.cuh"
using namespace krl;
int main(int argc, char** argv)
{
    for (int b = 0; b <= 5; ++b) {
        unsigned seen = 0;
        for (int lane = 0; lane < 32; ++lane) {
            int x, y;
            trace_tile_place(lane, b, &x, &y);
            if (x < 0 || x >= 1 << b || y < 0 || y >= 32 >> b) return 1;
            seen |= 1u << (y * (1 << b) + x);
        }
        if (seen != 0xffffffffu) return 2;
    }
    for (int k = 1; k + 1 < argc; k += 2) {
        const long long x = atoll(argv[k]), y = atoll(argv[k + 1]);
        const int b = trace_tile_bits(x, y);
        printf("%d %lld\\n", b, trace_tiles_x(x, b) * trace_tiles_y(y, b));
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def tiles(tmp_path_factory):
    d = tmp_path_factory.mktemp("tile")
    (d / "t.cpp").write_text(SOURCE)
    inc = os.path.join(ROOT, "paper_2608_09340_gb300", "csrc")
    subprocess.check_call(["g++", "-std=c++17", "-I", inc, str(d / "t.cpp"), "-o", str(d / "t")])

    def ask(sizes):
        args = [str(v) for s in sizes for v in s]
        out = subprocess.check_output([str(d / "t"), *args], text=True)
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return ask


def test_lanes_have_rays(tiles):
    sides = [1, 2, 3, 4, 5, 7, 8, 9, 12, 17, 31, 100, 1000, 65536, 2 ** 31 - 1]
    sizes = [(x, y) for x in sides for y in sides]
    best = lambda x, y: min(-(-x // w) * -(-y // (32 // w)) for w in (1, 2, 4, 8, 16, 32))
    for (x, y), (b, n) in zip(sizes, tiles(sizes)):
        assert -(-x // 2 ** b) * -(-y // (32 >> b)) == n
        assert 4 * n <= 5 * best(x, y), (x, y, b)
        if max(x, y) >= 1000:               # no strip leaves more than 2 lanes of 5 idle
            assert x * y >= 0.6 * 32 * n, (x, y, b)


def test_square_images_keep_the_square_tile(tiles):
    assert all(b == 3 for b, _ in tiles([(n, n) for n in (8, 64, 100, 128, 200, 512, 700, 1024)]))


def test_strips_follow_the_image(tiles):
    assert [b for b, _ in tiles([(1, 5000), (5000, 1), (2, 5000), (5000, 2)])] == [0, 5, 1, 4]
