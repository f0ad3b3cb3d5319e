// tile.h -- the order in which the planned queue walks over an image's pixels.
// Plain C++, so that a host program can check its arithmetic at sizes whose
// rays would fill a device.
#pragma once

#ifdef __CUDACC__
#define GRAY_TILE_FN __host__ __device__ __forceinline__
#else
#define GRAY_TILE_FN inline
#endif

namespace gray {

struct Pixel {
    unsigned row, col;
};

// The p-th pixel of an nx x ny image: strips of four rows, column by column
// (the last strip holds the rows that are left); `by_row` walks row by row.
// A strip is never higher than the image, so high * nx <= nx * ny, which a
// buffer bounds by 2^31 - 1: the products fit 32 bits.
GRAY_TILE_FN Pixel tile_pixel(unsigned p, unsigned nx, unsigned ny, bool by_row)
{
    const unsigned high = by_row ? 1u : ny < 4u ? ny : 4u;
    const unsigned strip = p / (high * nx), q = p - strip * high * nx;
    const unsigned left = ny - high * strip, rows = left < high ? left : high;
    const unsigned col = rows == 4 ? q >> 2 : q / rows;
    return Pixel{high * strip + (q - col * rows), col};
}

} // namespace gray
