// The pixels that a warp of k_trace_cube follows: a tile of 32, 2^b wide and
// 2^(5-b) high. Host and device (constexpr), no CUDA headers.
#pragma once

namespace krl {

constexpr long long trace_tiles_x(long long npix_x, int b) { return (npix_x + (1 << b) - 1) >> b; }
constexpr long long trace_tiles_y(long long npix_y, int b) { return (npix_y + (32 >> b) - 1) / (32 >> b); }

// The squarest tile, 8 x 4 first, that needs at most a quarter more tiles
// than the best one: neighbouring lanes share cells most in a square tile,
// but 8 x 4 leaves 28 of 32 lanes without a ray in an image one pixel wide,
// 24 in one a pixel high. Measured through 128^3 cells, 64 channels, us per
// call, 8 x 4 / this rule: 1 x 65536 pixels 5786 / 1028, 65536 x 1 2538 / 882,
// 2 x 40000 3679 / 1180, 9 x 8000 1671 / 1179, 17 x 6000 1847 / 1610.
constexpr int trace_tile_bits(long long npix_x, long long npix_y)
{
    const int order[6] = {3, 2, 4, 1, 5, 0};
    long long fewest = 0;
    for (int b : order) {
        const long long t = trace_tiles_x(npix_x, b) * trace_tiles_y(npix_y, b);
        if (fewest == 0 || t < fewest) fewest = t;
    }
    for (int b : order)
        if (4 * trace_tiles_x(npix_x, b) * trace_tiles_y(npix_y, b) <= 5 * fewest) return b;
    return 3;
}

// The lane's place in the tile, in Z order: its bits go to x and y in turn
// while both have room, so that 4 or 8 lanes next to one another are 2 x 2 or
// 4 x 2 pixels.
constexpr void trace_tile_place(int lane, int b, int* x, int* y)
{
    int xb = 0, yb = 0;
    *x = *y = 0;
    for (int k = 0; k < 5; ++k) {
        const int bit = lane >> k & 1;
        if (xb < b && (xb <= yb || yb == 5 - b)) *x |= bit << xb++;
        else *y |= bit << yb++;
    }
}

}  // namespace krl
