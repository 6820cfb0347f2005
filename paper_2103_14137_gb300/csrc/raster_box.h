// Which pixel centres of a face a projected triangle is tested at (raster.cu).
// Plain C++ besides the qualifiers: the tests compile it without CUDA.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define UVC_HD __host__ __device__ __forceinline__
#else
#define UVC_HD inline
#endif

namespace uvc {

struct PixelRange {
    int first, last;   // first > last: none
};

// lo, hi: the projection's extent along one edge of the face, within [-1, 1]; the
// centres (2 p + 1) / R - 1 inside it, widened.  The projection and the ray test
// move a vertex by less than 2^-20 of its distance over its depth, so 1/32 of a
// pixel covers up to R = 4096 where no depth is below 1/16 of the distances
// (`deep`).  Other triangles (next to the source's own plane) get the next centre
// outwards and one more, and no more: of a triangle whose plane holds the source the
// test hits pixels anywhere.
UVC_HD PixelRange pixel_range(float lo, float hi, int R, bool deep) {
    const float h = 0.5f * R, a = (lo + 1.f) * h - 0.5f, b = (hi + 1.f) * h - 0.5f;
    const int first = deep ? (int)ceilf(a - 0.03125f) : (int)floorf(a) - 1;
    const int last = deep ? (int)floorf(b + 0.03125f) : (int)ceilf(b) + 1;
    return PixelRange{first < 0 ? 0 : first, last > R - 1 ? R - 1 : last};
}

}  // namespace uvc
