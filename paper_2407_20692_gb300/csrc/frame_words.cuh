// The 32-bit words of a bit-packed frame that span a region.  Plain integer arithmetic,
// for the host and the device.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define CPI_HD __host__ __device__ __forceinline__
#else
#define CPI_HD inline
#endif

namespace cpi {

CPI_HD int64_t floor_div(int64_t a, int64_t b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

// First and last frame word of the region.
template <typename Frames>
CPI_HD int64_t region_first_word(const Frames& d) {
    return ((int64_t)d.y0 * d.row_stride + d.x0) >> 5;
}
template <typename Frames>
CPI_HD int64_t region_last_word(const Frames& d) {
    return ((int64_t)(d.y0 + d.height - 1) * d.row_stride + d.x0 + d.width - 1) >> 5;
}

// Frame words that end up to the region's last byte, and the bytes of it behind them
// (0 to 3): the last frame of a buffer may end with that byte.
template <typename Frames>
CPI_HD int64_t region_whole_words(const Frames& d) {
    const int64_t last = (int64_t)(d.y0 + d.height - 1) * d.row_stride + d.x0 + d.width - 1;
    return ((last >> 3) + 1) >> 2;
}
template <typename Frames>
CPI_HD int region_rest_bytes(const Frames& d) {
    const int64_t last = (int64_t)(d.y0 + d.height - 1) * d.row_stride + d.x0 + d.width - 1;
    return (int)(((last >> 3) + 1) & 3);
}

// Whether the word path pays for a pair of regions: it copies every word from a region's
// first pixel to its last, the bit-wise path the bytes of the pixels themselves.  Per
// frame a word costs about 0.8 ps there (what lies between the rows is read from HBM
// too) and a pixel 0.17 ps, and a pixel 0.85 ps on the bit-wise path: one word per pixel
// is where the two meet.  Ingest of 20000 frames, two equal regions (height x width, row
// length in pixels), word path against bit-wise, us: 16x16, 512: 18.5 / 17.1; 64x16, 512:
// 56 / 70; 64x8, 512: 54 / 37; 16x31, 512: 18.9 / 26; 16x31, 2048: 49 / 26; 64x31, 2048:
// 181 / 112; 16x50, 8192: 159 / 41; 64x8, 128: 25 / 26; 128x100, 256: 130 / 489.
template <typename Frames>
CPI_HD bool words_pay(const Frames& a, const Frames& b) {
    const int64_t words = region_last_word(a) - region_first_word(a) + region_last_word(b) - region_first_word(b) + 2;
    return words <= (int64_t)a.height * a.width + (int64_t)b.height * b.width;
}

}  // namespace cpi
