// Visibility-cube estimator of the paper (Sec. IV-C, Fig. 2) as a CUDA
// software rasteriser: around every source point a cube of six R x R faces
// holds, per pixel, the nearest triangle along the ray through the pixel
// centre (a depth test); each pixel's power w_m P Omega_pixel / (4 pi) is
// added to its triangle when the ray meets the triangle's front side, and the
// flux over the triangle's area is its mean irradiance.
//
// The graphics pipeline of the paper (geometry shader, framebuffer, pixel
// blending) becomes, over a batch of cubes with faces cut into tiles of
// 64 x 64 pixels:
//   setup    per (cube, triangle), the six faces in turn: the triangle clipped
//            to the face's near plane and projected; the box of pixels whose
//            centres it can hold, counted into the tiles that it meets
//   plan     a place in the list for every tile's triangles, in any order, and
//            where it is much, the tile's work cut into units
//   fill     the triangles of every tile, in any order
//   tile     blocks take units as they finish: a warp tests 32 pixels of a
//            triangle's box at a time (watertight ray/triangle test through the
//            pixel centre), the nearest (depth bits, triangle id) per pixel kept
//            in shared memory; then each pixel's power (a precomputed table, like
//            the paper's emission texture E) is added to its triangle's flux in
//            2^-40 W fixed point (integer atomics: no order matters)
//   deep     the same for the tiles of several units, whose nearest went to
//            global memory instead
// and a finish pass divides by the triangle areas.
//
// One block per tile left the chip idle where there are few tiles, and lists of two
// entries a triangle sent most tiles through all boxes of their face where a
// triangle meets many.  Microseconds of a call on a ward (49,066 triangles), as it
// was with the depth buffer in memory | one block per tile | now: one cube at R = 64
// 101 | 958 | 71, at R = 512 211 | 338 | 137, at R = 4,096 6,130 | 34,080 | 2,400; 40
// cubes at R = 64 1,695 | 1,994 | 400, at R = 512 6,297 | 1,891 | 1,642.
#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <vector>

#include "raster_box.h"
#include "uvc_internal.cuh"

namespace uvc {
namespace {

constexpr float kFixOne = 1099511627776.0f;          // 2^40
constexpr float kFixInv = 1.0f / 1099511627776.0f;   // 2^-40
constexpr int kTile = 64;                            // pixels along a tile's edge
constexpr int kTilePix = kTile * kTile;
constexpr int kTileThreads = 256, kTileWarps = kTileThreads / 32, kTileBlocks = 6;   // blocks per SM
// A tile of more triangles, or of boxes of more pixels, than a unit is cut.  A unit
// is a quarter of an SM's share, but no smaller than these: cut tiles pay for
// clearing and merging their depths (with eighths 40 cubes of a room of 988
// triangles at R = 128 took 236 us, with quarters 210).  Past the largest a tile's
// other costs no longer show.
constexpr int kUnitsPerSm = 4;
constexpr int kUnitMin = 8, kUnitMax = 1024;         // triangles
constexpr int kAreaStep = 16, kUnitMinArea = 4096 / kAreaStep;   // pixels of the boxes, in steps
// Boxes are gone through in pieces of this many pixels, each by one warp: where a
// tile has fewer triangles than the block warps, or one that covers it all, a warp
// took up to 128 dependent rounds while others had nothing.
constexpr int kPiece = kTilePix / kTileWarps;
constexpr unsigned kNoBox = 0x00ffu;                 // x0 = 255 > x1 = 0
constexpr int kMaxSlots = 4096, kMaxUnits = 65536;   // tiles of several units, and those (more: one unit, whatever its size)
constexpr int kTileUnits = 256;                      // units of a tile, and of one whose triangles did not fit the list
constexpr int kBoxUnits = 8;

struct RasterUnit {
    int tile;            // -1: none
    unsigned lo, hi;     // of the tile's triangles, or of all boxes of its face
    int slot;
};

struct RasterCounters {
    unsigned long long listed;   // list entries given out
    unsigned units, slots, taken;
};

struct RasterBatch {
    const float4* tri;        // sorted triangles (v0.w = original id)
    int nt, R, C, K, tn;      // tn: tiles along a face's edge
    int T, unit, unit_area;   // tiles of the batch; triangles and pixel steps per unit
    const float* cand;        // candidates of this batch
    LampDev L;
    uint2* box;                   // [C][6][nt] x0 | x1 << 16, y0 | y1 << 16 (x0 > x1: empty)
    RasterCounters* n;
    unsigned* count;              // [T] triangles per tile (T = C x 6 x tn x tn)
    unsigned* area;               // [T] pixels of their boxes in the tile, in steps (may wrap: only the cutting rests on it)
    unsigned* cursor;             // [T] triangles filled in
    unsigned long long* first;    // [T] place of the tile's triangles in the list
    int* slot;                    // [T] place of the tile's depths in `deep`, -1: has one unit
    int* slot_tile;               // [slots] its tile
    RasterUnit* units;            // of the tiles that have several
    int* list;                    // the tiles' triangles (sorted positions), as far as they fit
    int64_t list_cap;
    unsigned long long* deep;     // [slots][kTilePix] depths of the tiles of several units
    int slot_cap;
    unsigned long long* F;        // [C / K][nt] flux, 2^-40 W units, by original id
    const float* e_unit;          // [R][R] Omega_pixel / (4 pi)
    const float* tri_normal;      // [nt][3] by original id
};

__device__ __forceinline__ float comp(float x, float y, float z, int k) { return k == 0 ? x : (k == 1 ? y : z); }

// Pixel-centre coordinate of pixel p on a face: fl32(fl32(2p + 1) / R) - 1.
__device__ __forceinline__ float pix_center(int p, int R) {
    return __fsub_rn(__fdiv_rn((float)(2 * p + 1), (float)R), 1.f);
}

// The source point of cube c.
__device__ __forceinline__ float3 cube_source(const RasterBatch& B, int c) {
    const int ci = c / B.K, m = c % B.K;
    return make_float3(B.cand[3 * ci] + B.L.ox[m], B.cand[3 * ci + 1] + B.L.oy[m], B.cand[3 * ci + 2] + B.L.oz[m]);
}

__device__ __forceinline__ unsigned pack_box(int x0, int x1, int y0, int y1) {   // within a tile
    return (unsigned)(x0 | x1 << 8 | y0 << 16 | y1 << 24);
}
__device__ __forceinline__ int box_pixels(unsigned b) {
    return ((int)(b >> 8 & 0xffu) - (int)(b & 0xffu) + 1) * ((int)(b >> 24) - (int)(b >> 16 & 0xffu) + 1);
}
__device__ __forceinline__ unsigned box_in_tile(uint2 bx, int px0, int py0) {
    const int x0 = max((int)(bx.x & 0xffffu) - px0, 0), x1 = min((int)(bx.x >> 16) - px0, kTile - 1);
    const int y0 = max((int)(bx.y & 0xffffu) - py0, 0), y1 = min((int)(bx.y >> 16) - py0, kTile - 1);
    return x0 <= x1 && y0 <= y1 ? pack_box(x0, x1, y0, y1) : kNoBox;
}

// The tiles that the lanes' boxes meet (x0 > x1: none), all lanes' shared out over
// the warp: a thread by itself took 5.8 ms for faces of 4,096 tiles that a triangle
// covers.  f(in, tile, lane of the box, the tile's first pixel) for every lane at
// once; `in`: this lane has a tile.
template <class F>
__device__ __forceinline__ void each_tile(const RasterBatch& B, uint2 bx, int face, F f) {
    const int lane = threadIdx.x & 31;
    const int tx0 = (bx.x & 0xffffu) / kTile, tx1 = (bx.x >> 16) / kTile, ty0 = (bx.y & 0xffffu) / kTile, ty1 = (bx.y >> 16) / kTile;
    const int w = tx1 - tx0 + 1, n = (bx.x & 0xffffu) <= (bx.x >> 16) ? w * (ty1 - ty0 + 1) : 0;
    int inc = n;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    const int total = __shfl_sync(0xffffffffu, inc, 31);
    for (int g0 = 0; g0 < total; g0 += 32) {
        const int g = g0 + lane;
        int src = 0;   // the first lane whose running sum passes g
        for (int o = 16; o > 0; o >>= 1)
            if (__shfl_sync(0xffffffffu, inc, src + o - 1) <= g) src += o;
        src = min(src, 31);
        const int q = g - __shfl_sync(0xffffffffu, inc - n, src), ws = __shfl_sync(0xffffffffu, w, src);
        const int x = __shfl_sync(0xffffffffu, tx0, src) + q % ws, y = __shfl_sync(0xffffffffu, ty0, src) + q / ws;
        f(g < total, (face * B.tn + y) * B.tn + x, src, x * kTile, y * kTile);
    }
}

__global__ void __launch_bounds__(256) k_rs_setup(RasterBatch B, float near_eps) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int c = blockIdx.y;
    const bool mine = k < B.nt;
    const size_t at = mine ? 3 * (size_t)k : 0;
    const float3 o = cube_source(B, c);
    const float4 p0 = __ldg(&B.tri[at]), p1 = __ldg(&B.tri[at + 1]), p2 = __ldg(&B.tri[at + 2]);
    const float rx[3] = {p0.x - o.x, p1.x - o.x, p2.x - o.x}, ry[3] = {p0.y - o.y, p1.y - o.y, p2.y - o.y},
                rz[3] = {p0.z - o.z, p1.z - o.z, p2.z - o.z};
    float reach = 0.f;   // largest coordinate, for the width of the box
#pragma unroll
    for (int q = 0; q < 3; ++q) reach = fmaxf(reach, fmaxf(fabsf(rx[q]), fmaxf(fabsf(ry[q]), fabsf(rz[q]))));
    const int faces = 6 / (int)gridDim.z;   // of this block: one where there are few warps, else all six
    for (int f = (int)blockIdx.z * faces; f < ((int)blockIdx.z + 1) * faces; ++f) {
        const int a = f >> 1, b1 = (a + 1) % 3, b2 = (a + 2) % 3;
        const float s = (f & 1) ? -1.f : 1.f;
        float w[3], u[3], v[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            w[q] = s * comp(rx[q], ry[q], rz[q], a);
            u[q] = comp(rx[q], ry[q], rz[q], b1);
            v[q] = comp(rx[q], ry[q], rz[q], b2);
        }
        float umin = 3e38f, umax = -3e38f, vmin = 3e38f, vmax = -3e38f;
        auto corner = [&](float cu, float cv, float cw) {
            const float pu = cu / cw, pv = cv / cw;
            umin = fminf(umin, pu); umax = fmaxf(umax, pu);
            vmin = fminf(vmin, pv); vmax = fmaxf(vmax, pv);
        };
        // clip the triangle to w >= near_eps (Sutherland-Hodgman, one plane)
        const float wlo = fminf(w[0], fminf(w[1], w[2])), whi = fmaxf(w[0], fmaxf(w[1], w[2]));
        uint2 bx = make_uint2(1u, 1u);
        if (mine && whi >= near_eps) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int r = (q + 1) % 3;
                const bool in_q = w[q] >= near_eps, in_r = w[r] >= near_eps;
                if (in_q) corner(u[q], v[q], w[q]);
                if (in_q != in_r) {
                    const float t = (near_eps - w[q]) / (w[r] - w[q]);
                    corner(u[q] + t * (u[r] - u[q]), v[q] + t * (v[r] - v[q]), near_eps);
                }
            }
            if (umax >= -1.f && umin <= 1.f && vmax >= -1.f && vmin <= 1.f) {
                umin = fmaxf(umin, -1.f); umax = fminf(umax, 1.f);
                vmin = fmaxf(vmin, -1.f); vmax = fminf(vmax, 1.f);
                const bool deep = wlo * 16.f >= reach;
                const PixelRange x = pixel_range(umin, umax, B.R, deep), y = pixel_range(vmin, vmax, B.R, deep);
                if (x.last >= x.first && y.last >= y.first)
                    bx = make_uint2((unsigned)x.first | ((unsigned)x.last << 16), (unsigned)y.first | ((unsigned)y.last << 16));
            }
        }
        const int face = c * 6 + f;
        if (mine) B.box[(int64_t)face * B.nt + k] = bx;
        each_tile(B, bx, face, [&](bool in, int t, int src, int px0, int py0) {
            const uint2 b = make_uint2(__shfl_sync(0xffffffffu, bx.x, src), __shfl_sync(0xffffffffu, bx.y, src));
            const unsigned group = __match_any_sync(0xffffffffu, in ? t : -1);
            const unsigned steps = __reduce_add_sync(group, (unsigned)((box_pixels(box_in_tile(b, px0, py0)) + kAreaStep - 1) / kAreaStep));
            if (in && (threadIdx.x & 31) == __ffs(group) - 1) {   // one addition for the lanes that share t
                atomicAdd(B.count + t, (unsigned)__popc(group));
                atomicAdd(B.area + t, steps);
            }
        });
    }
}

// One thread per tile: its place in the list and, where its work is to be cut, its
// units.
__global__ void __launch_bounds__(256) k_rs_plan(RasterBatch B) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const unsigned cnt = t < B.T ? B.count[t] : 0u;
    unsigned long long inc = cnt;   // one addition per warp
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    unsigned long long first = 0ull;
    if (lane == 31 && inc > 0ull) first = atomicAdd(&B.n->listed, inc);
    first = __shfl_sync(0xffffffffu, first, 31) + inc - cnt;
    if (!cnt) return;
    const bool listed = first + cnt <= (unsigned long long)B.list_cap;
    const unsigned all = listed ? cnt : (unsigned)B.nt;
    unsigned units = kBoxUnits;
    if (listed) units = max((cnt + B.unit - 1) / B.unit, (B.area[t] + B.unit_area - 1) / B.unit_area);
    units = min(units, min(all, (unsigned)kTileUnits));
    int slot = -1;
    if (units > 1u) {
        slot = (int)min(atomicAdd(&B.n->slots, 1u), (unsigned)B.slot_cap);
        if (slot == B.slot_cap) slot = -1;
    }
    if (slot >= 0) {
        const unsigned per = (all + units - 1) / units, at = atomicAdd(&B.n->units, units);
        const bool fits = at <= kMaxUnits - units;
        for (unsigned u = 0; u < units && at + u < (unsigned)kMaxUnits; ++u)
            B.units[at + u] = RasterUnit{fits ? t : -1, min(all, u * per), min(all, (u + 1) * per), slot};
        B.slot_tile[slot] = fits ? t : -1;
        if (!fits) slot = -1;
    }
    B.first[t] = listed ? first : ~0ull;
    B.slot[t] = slot;
}

// Blocks of the last row clear the depths of the tiles of several units.
__global__ void __launch_bounds__(256) k_rs_fill(RasterBatch B) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if ((int)blockIdx.y == B.C) {
        const int64_t n = blockIdx.z == 0 ? (int64_t)min(B.n->slots, (unsigned)B.slot_cap) * kTilePix : 0;
        for (int64_t q = k; q < n; q += (int64_t)gridDim.x * blockDim.x) B.deep[q] = ~0ull;
        return;
    }
    const int k0 = k - (int)(threadIdx.x & 31);
    if (k0 >= B.nt) return;   // whole warps
    const int faces = 6 / (int)gridDim.z;
    for (int f = (int)blockIdx.z * faces; f < ((int)blockIdx.z + 1) * faces; ++f) {
        const int face = (int)blockIdx.y * 6 + f;
        const uint2 bx = k < B.nt ? B.box[(int64_t)face * B.nt + k] : make_uint2(1u, 1u);
        each_tile(B, bx, face, [&](bool in, int t, int src, int, int) {
            const unsigned long long first = in ? B.first[t] : ~0ull;
            const unsigned group = __match_any_sync(0xffffffffu, in ? t : -1);
            const int lane = threadIdx.x & 31, lead = __ffs(group) - 1;
            unsigned at = 0u;
            if (in && lane == lead) at = atomicAdd(B.cursor + t, (unsigned)__popc(group));
            at = __shfl_sync(0xffffffffu, at, lead) + __popc(group & ((1u << lane) - 1u));
            if (first != ~0ull) B.list[first + at] = k0 + src;
        });
    }
}

// Adds the lanes' pixels (lx, ly of tile `tile`, depth and triangle `key`) to their
// triangles' flux.  Neighbouring pixels mostly see the same triangle: the lanes
// that add to the same triangle sum their fixed-point powers first (lanes grouped
// with __match_any_sync, the lowest lane adds for the group).  Every lane calls it;
// part: 32 values of the warp's own.
__device__ __forceinline__ void add_pixels(const RasterBatch& B, int tile, int q, unsigned long long key, unsigned long long* part) {
    const int px = tile % B.tn * kTile + q % kTile, py = tile / B.tn % B.tn * kTile + q / kTile;
    const int face = tile / (B.tn * B.tn), c = face / 6, f = face % 6, a = f >> 1, ci = c / B.K, m = c % B.K;
    const int lane = threadIdx.x & 31;
    const float s = f & 1 ? -1.f : 1.f;
    int own = -1;                         // the triangle that the lane adds to
    unsigned long long val = 0;
    if (key != ~0ull && px < B.R && py < B.R) {
        const int id = (int)(key & 0xffffffffull);
        const float* nrm = B.tri_normal + 3 * (size_t)id;
        const float u = pix_center(px, B.R), v = pix_center(py, B.R);
        const float d0 = a == 0 ? s : (a == 1 ? v : u), d1 = a == 0 ? u : (a == 1 ? s : v), d2 = a == 0 ? v : (a == 1 ? u : s);
        const float dn = d0 * nrm[0] + d1 * nrm[1] + d2 * nrm[2];
        if (dn < 0.f) {                   // front side; the back side absorbs
            const float pw = __fmul_rn(B.L.pw[m], B.e_unit[(int64_t)py * B.R + px]);
            val = __float2ull_rn(__fmul_rn(pw, kFixOne));
            own = id;
        }
    }
    const unsigned group = __match_any_sync(0xffffffffu, own);
    part[lane] = val;
    __syncwarp();
    if (own >= 0 && lane == __ffs(group) - 1) {
        unsigned long long sum = 0;
        for (unsigned g = group; g; g &= g - 1) sum += part[__ffs(g) - 1];
        atomicAdd(&B.F[(int64_t)ci * B.nt + own], sum);
    }
    __syncwarp();
}

// Units of tiles, and the tiles that are one.  256 triangles of the unit at a time:
// a thread each clips their boxes to the tile, then a warp takes a triangle (or a
// piece of a large box); its lanes go through the pixels, 32 at a time, and test
// the ray through each pixel centre (watertight, Woop, Benthin and Wald, JCGT 2013).  The face's axis a
// holds the largest component of the ray (+-1; |u|, |v| < 1 at pixel centres), so
// the shear divides by +-1, which is exact, and everything but the shear is the
// same for all of a triangle's pixels.  Tiles whose triangles did not fit the list
// look through all boxes of their face instead.
__global__ void __launch_bounds__(kTileThreads, kTileBlocks) k_rs_tile(RasterBatch B) {
    __shared__ unsigned long long near[kTilePix];
    __shared__ float cu[kTile], cv[kTile];
    __shared__ unsigned long long part[kTileWarps][32];
    __shared__ unsigned next_unit;
    uint2* entry = reinterpret_cast<uint2*>(part);   // triangles and their boxes in the tile
    static_assert(sizeof(part) == sizeof(uint2) * kTileThreads, "an entry per thread");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned units = min(B.n->units, (unsigned)kMaxUnits);
    for (unsigned u = blockIdx.x; u < units + B.T;) {   // the units, then the tiles that are one
        unsigned after = 0u;
        if (threadIdx.x == 0) after = gridDim.x + atomicAdd(&B.n->taken, 1u);
        RasterUnit U;
        if (u < units) {
            U = B.units[u];
        } else {
            U.tile = (int)(u - units);
            U.slot = -1;
            U.lo = 0u;
            U.hi = B.count[U.tile];
            if (U.hi > 0u && B.slot[U.tile] >= 0) U.hi = 0u;
        }
        const unsigned long long first = U.tile >= 0 && U.hi > U.lo ? B.first[U.tile] : 0ull;
        const bool listed = first != ~0ull;
        if (u >= units && !listed) U.hi = (unsigned)B.nt;
        if (U.tile < 0 || U.hi <= U.lo) {   // nothing here
            if (threadIdx.x == 0) next_unit = after;
            __syncthreads();
            u = next_unit;
            __syncthreads();
            continue;
        }
        const int tx = U.tile % B.tn, ty = U.tile / B.tn % B.tn, face = U.tile / (B.tn * B.tn);
        const int c = face / 6, f = face % 6, a = f >> 1;
        const bool pos = !(f & 1);
        const int px0 = tx * kTile, py0 = ty * kTile;
        for (int q = threadIdx.x; q < kTilePix; q += kTileThreads) near[q] = ~0ull;
        if (threadIdx.x < kTile) cu[threadIdx.x] = pix_center(px0 + threadIdx.x, B.R);
        else if (threadIdx.x < 2 * kTile) cv[threadIdx.x - kTile] = pix_center(py0 + threadIdx.x - kTile, B.R);
        const float3 o = cube_source(B, c);
        const float s = pos ? 1.f : -1.f;
        const int64_t n = (int64_t)U.hi - U.lo;
        for (int64_t j0 = 0; j0 < n; j0 += kTileThreads) {   // a triangle and its box in the tile per thread
            const int m = (int)min((int64_t)kTileThreads, n - j0);
            uint2 e = make_uint2(0u, kNoBox);
            if ((int)threadIdx.x < m) {
                const int64_t i = U.lo + j0 + threadIdx.x;
                const int k = listed ? __ldg(&B.list[first + i]) : (int)i;
                e = make_uint2((unsigned)k, box_in_tile(__ldg(&B.box[(int64_t)face * B.nt + k]), px0, py0));
            }
            entry[threadIdx.x] = e;
            __syncthreads();
            for (int j = 0; j < m; j += 32) {
                const uint2 own = entry[j + lane];
                const int pieces = (box_pixels(own.y) + kPiece - 1) / kPiece;   // none for kNoBox
                for (unsigned todo = __ballot_sync(0xffffffffu, ((warp - lane) & (kTileWarps - 1)) < pieces); todo; todo &= todo - 1) {
                    const int src = __ffs(todo) - 1, k = (int)__shfl_sync(0xffffffffu, own.x, src);
                    const unsigned box = __shfl_sync(0xffffffffu, own.y, src);
                    const int x0 = box & 0xffu, x1 = box >> 8 & 0xffu, y0 = box >> 16 & 0xffu;
                    const float4 A4 = __ldg(&B.tri[3 * (size_t)k]), B4 = __ldg(&B.tri[3 * (size_t)k + 1]), C4 = __ldg(&B.tri[3 * (size_t)k + 2]);
                    // relative vertices: along the axis, and across it in the order of the ray's winding
                    auto along = [&](float4 p) { return a == 0 ? __fsub_rn(p.x, o.x) : (a == 1 ? __fsub_rn(p.y, o.y) : __fsub_rn(p.z, o.z)); };
                    auto first_of = [&](float4 p) { return a == 0 ? __fsub_rn(p.y, o.y) : (a == 1 ? __fsub_rn(p.z, o.z) : __fsub_rn(p.x, o.x)); };
                    auto second_of = [&](float4 p) { return a == 0 ? __fsub_rn(p.z, o.z) : (a == 1 ? __fsub_rn(p.x, o.x) : __fsub_rn(p.y, o.y)); };
                    const float akz = along(A4), bkz = along(B4), ckz = along(C4);
                    const float Ax = pos ? first_of(A4) : second_of(A4), Ay = pos ? second_of(A4) : first_of(A4);
                    const float Bx = pos ? first_of(B4) : second_of(B4), By = pos ? second_of(B4) : first_of(B4);
                    const float Cx = pos ? first_of(C4) : second_of(C4), Cy = pos ? second_of(C4) : first_of(C4);
                    const float za = __fmul_rn(s, akz), zb = __fmul_rn(s, bkz), zc = __fmul_rn(s, ckz);
                    const unsigned id = (unsigned)__float_as_int(A4.w);
                    const int w = x1 - x0 + 1, cnt = box_pixels(box);   // at most 4096: the float quotient below is exact
                    const float rw = 1.f / (float)w;
                    const int from = ((warp - src) & (kTileWarps - 1)) * kPiece, stop = min(cnt, from + kPiece);
                    for (int g = from + lane; g < stop; g += 32) {
                        const int row = (int)(((float)g + 0.5f) * rw), lx = x0 + g - row * w, ly = y0 + row;
                        const float sx = pos ? cu[lx] : -cv[ly], sy = pos ? cv[ly] : -cu[lx];
                        const float ax = __fmaf_rn(-sx, akz, Ax), ay = __fmaf_rn(-sy, akz, Ay);
                        const float bx_ = __fmaf_rn(-sx, bkz, Bx), by = __fmaf_rn(-sy, bkz, By);
                        const float cx = __fmaf_rn(-sx, ckz, Cx), cy = __fmaf_rn(-sy, ckz, Cy);
                        const float U = __fsub_rn(__fmul_rn(cx, by), __fmul_rn(cy, bx_));
                        const float V = __fsub_rn(__fmul_rn(ax, cy), __fmul_rn(ay, cx));
                        const float W = __fsub_rn(__fmul_rn(bx_, ay), __fmul_rn(by, ax));
                        if ((U < 0.f || V < 0.f || W < 0.f) && (U > 0.f || V > 0.f || W > 0.f)) continue;
                        const float det = U + V + W;
                        if (det == 0.f) continue;
                        const float T = U * za + V * zb + W * zc;
                        const float t = __fdiv_rn(T, det);
                        if (!(t > 0.f)) continue;
                        const unsigned long long key = ((unsigned long long)__float_as_uint(t) << 32) | id;
                        unsigned long long* at = &near[ly * kTile + lx];
                        if (key < *reinterpret_cast<volatile unsigned long long*>(at)) atomicMin(at, key);
                    }
                }
            }
            __syncthreads();
        }
        if (U.slot >= 0) {
            unsigned long long* deep = B.deep + (int64_t)U.slot * kTilePix;
            for (int q = threadIdx.x; q < kTilePix; q += kTileThreads)
                if (near[q] != ~0ull) atomicMin(deep + q, near[q]);
        } else {
            for (int q = threadIdx.x; q < kTilePix; q += kTileThreads) add_pixels(B, U.tile, q, near[q], part[warp]);
        }
        if (threadIdx.x == 0) next_unit = after;
        __syncthreads();   // the shared arrays are free
        u = next_unit;
    }
}

// The pixels of the tiles of several units.
__global__ void __launch_bounds__(kTileThreads) k_rs_deep(RasterBatch B) {
    __shared__ unsigned long long part[kTileWarps][32];
    const int64_t n = (int64_t)min(B.n->slots, (unsigned)B.slot_cap) * kTilePix;
    for (int64_t q = (int64_t)blockIdx.x * kTileThreads + threadIdx.x; q < n; q += (int64_t)gridDim.x * kTileThreads)
        add_pixels(B, max(B.slot_tile[q / kTilePix], 0), (int)(q % kTilePix), B.deep[q], part[threadIdx.x >> 5]);
}

__global__ void k_rs_finish(RasterBatch B, int nb, float* __restrict__ A, int64_t lda) {
    const int64_t n = (int64_t)nb * B.nt;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(q / B.nt), k = (int)(q % B.nt);
        const float4 a = B.tri[3 * (size_t)k], b = B.tri[3 * (size_t)k + 1], c = B.tri[3 * (size_t)k + 2];
        const int id = __float_as_int(a.w);
        const float ex = b.x - a.x, ey = b.y - a.y, ez = b.z - a.z, fx = c.x - a.x, fy = c.y - a.y, fz = c.z - a.z;
        const float cx = ey * fz - ez * fy, cy = ez * fx - ex * fz, cz = ex * fy - ey * fx;
        const float area = 0.5f * sqrtf(cx * cx + cy * cy + cz * cz);
        const float flux = __fmul_rn(__ull2float_rn(B.F[(size_t)i * B.nt + id]), kFixInv);
        A[(size_t)i * lda + id] = area > 0.f ? flux / area : 0.f;
    }
}

// Omega_pixel / (4 pi) for one face (all faces are alike), from the closed
// form of the solid angle of a rectangle on the unit-distance plane:
// Omega = G(u1,v1) - G(u0,v1) - G(u1,v0) + G(u0,v0), G = atan(u v / sqrt(1 + u^2 + v^2)).
const std::vector<float>& pixel_table(int R) {
    static std::mutex mu;
    static std::map<int, std::vector<float>> cache;
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache.find(R);
    if (it != cache.end()) return it->second;
    std::vector<float> t((size_t)R * R);
    auto G = [](double u, double v) { return std::atan(u * v / std::sqrt(1.0 + u * u + v * v)); };
    for (int py = 0; py < R; ++py) {
        const double v0 = 2.0 * py / R - 1.0, v1 = 2.0 * (py + 1) / R - 1.0;
        for (int px = 0; px < R; ++px) {
            const double u0 = 2.0 * px / R - 1.0, u1 = 2.0 * (px + 1) / R - 1.0;
            t[(size_t)py * R + px] = (float)((G(u1, v1) - G(u0, v1) - G(u1, v0) + G(u0, v0)) / (4.0 * M_PI));
        }
    }
    return cache.emplace(R, std::move(t)).first->second;
}

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

int tiles_per_edge(int R) { return (R + kTile - 1) / kTile; }

// List entries of C cubes, twice what the tiles are expected to hold: if every
// triangle covers its share of the faces' pixels twice over, its box has edges of
// e = sqrt(12 R^2 / nt) pixels and meets (1 + e / kTile)^2 tiles (and one or two
// faces).  Tiles past the end look through their face's boxes.
int64_t list_entries(int64_t C, int64_t nt, int R) {
    const double e = std::sqrt(12.0 * R * R / (double)std::max<int64_t>(nt, 1)), tiles = 1.0 + e / kTile;
    const int64_t tn = tiles_per_edge(R), all = 6 * tn * tn;
    return C * nt * std::min<int64_t>(all, (int64_t)std::ceil(2.0 * tiles * tiles));
}

// Workspace layout for nb candidates per batch.  What is cleared before a batch
// (F, the counters, count, area, cursor) lies together.
struct RasterLayout {
    int64_t C, T, list;
    size_t box, units, first, slot, slot_tile, deep, e_unit, clear, F, counters, per_tile, bytes;   // byte offsets
    RasterLayout(int64_t nt, int K, int R, int64_t nb) {
        const int64_t tn = tiles_per_edge(R);
        C = nb * K;
        T = C * 6 * tn * tn;
        list = list_entries(C, nt, R);
        size_t at = align256(sizeof(int) * (size_t)list);   // the list comes first
        auto take = [&](size_t n) { const size_t q = at; at += align256(n); return q; };
        box = take(sizeof(uint2) * (size_t)(C * 6 * nt));
        units = take(sizeof(RasterUnit) * (size_t)kMaxUnits);
        first = take(sizeof(unsigned long long) * (size_t)T);
        slot = take(sizeof(int) * (size_t)T);
        slot_tile = take(sizeof(int) * (size_t)std::min<int64_t>(T, kMaxSlots));
        deep = take(sizeof(unsigned long long) * kTilePix * (size_t)std::min<int64_t>(T, kMaxSlots));
        e_unit = take(sizeof(float) * (size_t)R * R);
        clear = F = take(sizeof(unsigned long long) * (size_t)(nb * nt));
        counters = take(sizeof(RasterCounters));
        per_tile = take(3 * sizeof(unsigned) * (size_t)T);
        bytes = at + 256;
    }
};

// Candidates of one batch: gridDim.y holds the cubes and a row more, tiles are
// counted in 31 bits.
int64_t max_candidates(int K, int R) {
    const int64_t tn = tiles_per_edge(R);
    return std::max<int64_t>(1, std::min<int64_t>(65534, ((int64_t(1) << 31) - 1) / (6 * tn * tn)) / K);
}

size_t raster_bytes(int64_t nt, int K, int R, int64_t nb) { return RasterLayout(nt, K, R, nb).bytes; }

}  // namespace

size_t raster_workspace_bytes(int64_t nt, int K, int R, int64_t cand_per_batch) {
    return raster_bytes(nt, K, R, cand_per_batch);
}

int irradiance_raster(const uvc_scene* sc, const float* tri_normal, const float* cand, int64_t nc, const LampDev& L,
                      int R, float* A, int64_t lda, void* work, size_t bytes, cudaStream_t stream) {
    if (nc == 0 || sc->nt == 0) return UVC_OK;
    const int64_t nt = sc->nt;
    int64_t nb = 1;
    if (raster_bytes(nt, L.K, R, 1) > bytes) return UVC_E_INVAL;
    // the largest batch that fits (the bytes grow with nb)
    for (int64_t hi = std::min<int64_t>(nc, max_candidates(L.K, R)) + 1; hi - nb > 1;) {
        const int64_t mid = (nb + hi) / 2;
        if (raster_bytes(nt, L.K, R, mid) <= bytes) nb = mid;
        else hi = mid;
    }
    const std::vector<float>& table = pixel_table(R);
    char* p = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(work) + 255) & ~uintptr_t(255));
    const int tn = tiles_per_edge(R);
    const RasterLayout at(nt, L.K, R, nb);
    float* e_unit = reinterpret_cast<float*>(p + at.e_unit);
    cudaError_t err = cudaMemcpyAsync(e_unit, table.data(), sizeof(float) * table.size(), cudaMemcpyHostToDevice,
                                      stream);
    if (err != cudaSuccess) return status_from_cuda(err);
    const float near_eps = 1e-6f * fmaxf(sc->diameter, 1e-30f);
    const int sms = sm_count(), grid = sms * 8;
    RasterBatch B;
    B.tri = sc->tri;
    B.nt = (int)nt;
    B.R = R;
    B.K = L.K;
    B.tn = tn;
    B.L = L;
    B.list = reinterpret_cast<int*>(p);
    B.list_cap = at.list;
    B.box = reinterpret_cast<uint2*>(p + at.box);
    B.units = reinterpret_cast<RasterUnit*>(p + at.units);
    B.first = reinterpret_cast<unsigned long long*>(p + at.first);
    B.slot = reinterpret_cast<int*>(p + at.slot);
    B.slot_tile = reinterpret_cast<int*>(p + at.slot_tile);
    B.deep = reinterpret_cast<unsigned long long*>(p + at.deep);
    B.slot_cap = (int)std::min<int64_t>(at.T, kMaxSlots);
    B.F = reinterpret_cast<unsigned long long*>(p + at.F);
    B.n = reinterpret_cast<RasterCounters*>(p + at.counters);
    B.count = reinterpret_cast<unsigned*>(p + at.per_tile);
    B.e_unit = e_unit;
    B.tri_normal = tri_normal;
    for (int64_t i0 = 0; i0 < nc; i0 += nb) {
        const int64_t n = std::min<int64_t>(nb, nc - i0);
        B.C = (int)(n * L.K);
        B.T = B.C * 6 * tn * tn;
        B.cand = cand + 3 * i0;
        B.area = B.count + B.T;
        B.cursor = B.area + B.T;
        // an SM's share over kUnitsPerSm, for as many triangles per tile as expected
        // and three layers of boxes
        const int64_t goal = (int64_t)sms * kUnitsPerSm, layers = 3 * (int64_t)B.T * (kTilePix / kAreaStep);
        B.unit = (int)std::min<int64_t>(kUnitMax, std::max<int64_t>(kUnitMin, list_entries(B.C, nt, R) / 2 / goal));
        B.unit_area = (int)std::min<int64_t>(INT32_MAX, std::max<int64_t>(kUnitMinArea, layers / goal));
        const unsigned rows = (unsigned)((nt + 255) / 256);   // k_rs_fill: enough blocks to clear depths, too
        cudaMemsetAsync(p + at.clear, 0, (size_t)((char*)(B.cursor + B.T) - (p + at.clear)), stream);
        const unsigned split = (int64_t)rows * B.C < 4 * sms ? 6 : 1;   // a block per face
        k_rs_setup<<<dim3(rows, (unsigned)B.C, split), 256, 0, stream>>>(B, near_eps);
        k_rs_plan<<<(B.T + 255) / 256, 256, 0, stream>>>(B);
        k_rs_fill<<<dim3(std::max(rows, 32u), (unsigned)B.C + 1, split), 256, 0, stream>>>(B);
        k_rs_tile<<<kTileBlocks * sms, kTileThreads, 0, stream>>>(B);
        k_rs_deep<<<grid, kTileThreads, 0, stream>>>(B);
        k_rs_finish<<<grid, 256, 0, stream>>>(B, (int)n, A + (size_t)i0 * lda, lda);
    }
    return status_from_cuda(cudaGetLastError());
}

}  // namespace uvc
