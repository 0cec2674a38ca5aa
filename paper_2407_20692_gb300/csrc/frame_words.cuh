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

}  // namespace cpi
