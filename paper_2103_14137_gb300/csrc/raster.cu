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
//   scan     exclusive prefix sum of the tiles' counts
//   fill     the triangles of every tile, in any order
//   tile     one block per tile: a warp takes a triangle at a time and tests 32
//            pixels of its box (watertight ray/triangle test through the pixel
//            centre), the nearest (depth bits, triangle id) per pixel kept in
//            shared memory; then each pixel's power (a precomputed table, like
//            the paper's emission texture E) is added to its triangle's flux
//            in 2^-40 W fixed point (integer atomics: neither the fill's order
//            nor the threads' matters)
// and a finish pass divides by the triangle areas.
//
// The first form searched the triangle of every fragment in one flat index
// space (a binary search and three 64-bit divisions each) and kept the depth
// buffer in memory, 2 MB a face: 5.3 ms of fragments and 0.8 ms of resolving a
// five-candidate, K = 8, R = 512 batch on a 49,066-triangle ward.
#include <cmath>
#include <map>
#include <mutex>
#include <vector>

#include "uvc_internal.cuh"

namespace uvc {
namespace {

constexpr float kFixOne = 1099511627776.0f;          // 2^40
constexpr float kFixInv = 1.0f / 1099511627776.0f;   // 2^-40
constexpr int kScanBlock = 1024, kScanPer = 4;       // 4096 elements per scan block
constexpr int kTile = 64;                            // pixels along a tile's edge
constexpr int kTileThreads = 256;

struct RasterBatch {
    const float4* tri;        // sorted triangles (v0.w = original id)
    int nt, R, C, K, tn;      // tn: tiles along a face's edge
    const float* cand;        // candidates of this batch
    LampDev L;
    uint2* box;                   // [C][6][nt] x0 | x1 << 16, y0 | y1 << 16 (x0 > x1: empty)
    unsigned long long* toff;     // [C][6][tn][tn] + 1 triangles per tile, then their exclusive prefix sum
    unsigned* cursor;             // [C][6][tn][tn] triangles filled in
    int* list;                    // the tiles' triangles (sorted positions), as far as they fit
    int64_t list_cap;
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

// Tiles met by a box: a count each.
template <class F>
__device__ __forceinline__ void each_tile(const RasterBatch& B, uint2 bx, int64_t face, F f) {
    const int x0 = bx.x & 0xffffu, x1 = bx.x >> 16, y0 = bx.y & 0xffffu, y1 = bx.y >> 16;
    for (int ty = y0 / kTile; ty <= y1 / kTile; ++ty)
        for (int tx = x0 / kTile; tx <= x1 / kTile; ++tx) f((face * B.tn + ty) * B.tn + tx);
}

__global__ void __launch_bounds__(256) k_rs_setup(RasterBatch B, float near_eps) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int c = blockIdx.y;
    if (k >= B.nt) return;
    const float3 o = cube_source(B, c);
    const float4 p0 = __ldg(&B.tri[3 * (size_t)k]), p1 = __ldg(&B.tri[3 * (size_t)k + 1]), p2 = __ldg(&B.tri[3 * (size_t)k + 2]);
    const float rx[3] = {p0.x - o.x, p1.x - o.x, p2.x - o.x}, ry[3] = {p0.y - o.y, p1.y - o.y, p2.y - o.y},
                rz[3] = {p0.z - o.z, p1.z - o.z, p2.z - o.z};
    float reach = 0.f;   // largest coordinate, for the width of the box
#pragma unroll
    for (int q = 0; q < 3; ++q) reach = fmaxf(reach, fmaxf(fabsf(rx[q]), fmaxf(fabsf(ry[q]), fabsf(rz[q]))));
#pragma unroll
    for (int f = 0; f < 6; ++f) {
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
        if (whi >= near_eps) {
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
                const float h = 0.5f * B.R;
                // pixel centres (2p + 1) / R - 1 inside [min, max], widened: the
                // projection and the ray test move a vertex by less than 2^-20 of
                // its distance over its depth, so 1/32 of a pixel covers up to
                // R = 4096 where no depth is below 1/16 of the distances; other
                // triangles (next to the source's own plane) get two pixels
                const float e = wlo * 16.f >= reach ? 0.03125f : 2.f;
                const int x0 = max(0, (int)ceilf((umin + 1.f) * h - 0.5f - e));
                const int x1 = min(B.R - 1, (int)floorf((umax + 1.f) * h - 0.5f + e));
                const int y0 = max(0, (int)ceilf((vmin + 1.f) * h - 0.5f - e));
                const int y1 = min(B.R - 1, (int)floorf((vmax + 1.f) * h - 0.5f + e));
                if (x1 >= x0 && y1 >= y0) bx = make_uint2((unsigned)x0 | ((unsigned)x1 << 16), (unsigned)y0 | ((unsigned)y1 << 16));
            }
        }
        const int64_t face = (int64_t)c * 6 + f;
        B.box[face * B.nt + k] = bx;
        if ((bx.x & 0xffffu) <= (bx.x >> 16)) each_tile(B, bx, face, [&](int64_t t) { atomicAdd(&B.toff[t], 1ull); });
    }
}

__global__ void __launch_bounds__(256) k_rs_fill(RasterBatch B) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= B.nt) return;
    for (int f = 0; f < 6; ++f) {
        const int64_t face = (int64_t)blockIdx.y * 6 + f;
        const uint2 bx = B.box[face * B.nt + k];
        if ((bx.x & 0xffffu) > (bx.x >> 16)) continue;
        each_tile(B, bx, face, [&](int64_t t) {
            const unsigned long long at = B.toff[t] + atomicAdd(&B.cursor[t], 1u);
            if (at < (unsigned long long)B.list_cap) B.list[at] = k;
        });
    }
}

// Exclusive scan of n uint64 values in place (three passes).
__global__ void k_scan_blocks(unsigned long long* x, int64_t n, unsigned long long* sums) {
    __shared__ unsigned long long warp_tot[kScanBlock / 32];
    const int64_t base = (int64_t)blockIdx.x * kScanBlock * kScanPer + (int64_t)threadIdx.x * kScanPer;
    unsigned long long v[kScanPer], run = 0;
    for (int q = 0; q < kScanPer; ++q) {
        v[q] = base + q < n ? x[base + q] : 0ull;
        run += v[q];
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned long long inc = run;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) warp_tot[w] = inc;
    __syncthreads();
    if (w == 0) {
        unsigned long long t = lane < kScanBlock / 32 ? warp_tot[lane] : 0ull;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        if (lane < kScanBlock / 32) warp_tot[lane] = t;   // inclusive
    }
    __syncthreads();
    unsigned long long pre = (w > 0 ? warp_tot[w - 1] : 0ull) + inc - run;
    for (int q = 0; q < kScanPer; ++q) {
        if (base + q < n) x[base + q] = pre;
        pre += v[q];
    }
    if (threadIdx.x == kScanBlock - 1) sums[blockIdx.x] = warp_tot[kScanBlock / 32 - 1];
}

__global__ void k_scan_sums(unsigned long long* sums, int nb, unsigned long long* total) {
    // one warp, chunks of 32 with a running carry
    const int lane = threadIdx.x;
    unsigned long long carry = 0;
    for (int b0 = 0; b0 < nb; b0 += 32) {
        const unsigned long long v = b0 + lane < nb ? sums[b0 + lane] : 0ull;
        unsigned long long inc = v;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (b0 + lane < nb) sums[b0 + lane] = carry + inc - v;
        carry += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) *total = carry;
}

__global__ void k_scan_add(unsigned long long* x, int64_t n, const unsigned long long* sums) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] += sums[i / (kScanBlock * kScanPer)];
}

// One tile of one face.  A warp takes one triangle at a time; its lanes go
// through the pixels of the triangle's box within the tile, 32 at a time, and
// test the ray through each pixel centre (watertight, Woop, Benthin and Wald,
// JCGT 2013).  The face's axis a holds the largest component of the ray (+-1;
// |u|, |v| < 1 at pixel centres), so the shear divides by +-1, which is exact,
// and everything but the shear is the same for all of a triangle's pixels.
// Tiles whose triangles did not fit the list look through all boxes of their
// face instead.
__global__ void __launch_bounds__(kTileThreads) k_rs_tile(RasterBatch B) {
    __shared__ unsigned long long keys[kTile * kTile];
    __shared__ float cu[kTile], cv[kTile];
    __shared__ unsigned long long part[kTileThreads / 32][32];
    const int64_t tile = blockIdx.x;
    const int tx = (int)(tile % B.tn), ty = (int)(tile / B.tn % B.tn), face = (int)(tile / (B.tn * B.tn));
    const int c = face / 6, f = face % 6, a = f >> 1;
    const bool pos = !(f & 1);
    const int px0 = tx * kTile, py0 = ty * kTile, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned long long first = B.toff[tile], last = B.toff[tile + 1];
    if (first == last) return;
    for (int q = threadIdx.x; q < kTile * kTile; q += kTileThreads) keys[q] = ~0ull;
    if (threadIdx.x < kTile) cu[threadIdx.x] = pix_center(px0 + threadIdx.x, B.R);
    else if (threadIdx.x < 2 * kTile) cv[threadIdx.x - kTile] = pix_center(py0 + threadIdx.x - kTile, B.R);
    __syncthreads();
    const float3 o = cube_source(B, c);
    const float s = pos ? 1.f : -1.f;
    const bool listed = last <= (unsigned long long)B.list_cap;
    const int64_t n = listed ? (int64_t)(last - first) : B.nt;
    for (int64_t i = warp; i < n; i += kTileThreads / 32) {
        const int k = listed ? __ldg(&B.list[first + i]) : (int)i;
        const uint2 bx = __ldg(&B.box[(int64_t)face * B.nt + k]);
        const int x0 = max((int)(bx.x & 0xffffu), px0), x1 = min((int)(bx.x >> 16), px0 + kTile - 1);
        const int y0 = max((int)(bx.y & 0xffffu), py0), y1 = min((int)(bx.y >> 16), py0 + kTile - 1);
        if (x1 < x0 || y1 < y0) continue;
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
        const int w = x1 - x0 + 1, cnt = w * (y1 - y0 + 1);   // at most 4096: the float quotient below is exact
        const float rw = 1.f / (float)w;
        for (int g = lane; g < cnt; g += 32) {
            const int row = (int)(((float)g + 0.5f) * rw), lx = x0 - px0 + g - row * w, ly = y0 - py0 + row;
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
            unsigned long long* at = &keys[ly * kTile + lx];
            if (key < *reinterpret_cast<volatile unsigned long long*>(at)) atomicMin(at, key);
        }
    }
    __syncthreads();
    // Neighbouring pixels mostly see the same triangle: the lanes of a warp that
    // add to the same triangle sum their fixed-point powers first (lanes grouped
    // with __match_any_sync, the lowest lane adds for the group).
    const int ci = c / B.K, m = c % B.K;
    for (int q = threadIdx.x; q < kTile * kTile; q += kTileThreads) {
        const int lx = q % kTile, ly = q / kTile;
        const unsigned long long key = keys[q];
        int slot = -1;                        // the triangle that the lane adds to
        unsigned long long val = 0;
        if (key != ~0ull && px0 + lx < B.R && py0 + ly < B.R) {
            const int id = (int)(key & 0xffffffffull);
            const float* nrm = B.tri_normal + 3 * (size_t)id;
            const float u = cu[lx], v = cv[ly];
            const float d0 = a == 0 ? s : (a == 1 ? v : u), d1 = a == 0 ? u : (a == 1 ? s : v), d2 = a == 0 ? v : (a == 1 ? u : s);
            const float dn = d0 * nrm[0] + d1 * nrm[1] + d2 * nrm[2];
            if (dn < 0.f) {                   // front side; the back side absorbs
                const float pw = __fmul_rn(B.L.pw[m], B.e_unit[(int64_t)(py0 + ly) * B.R + px0 + lx]);
                val = __float2ull_rn(__fmul_rn(pw, kFixOne));
                slot = id;
            }
        }
        const unsigned group = __match_any_sync(0xffffffffu, slot);
        part[warp][lane] = val;
        __syncwarp();
        if (slot >= 0 && lane == __ffs(group) - 1) {
            unsigned long long sum = 0;
            for (unsigned g = group; g; g &= g - 1) sum += part[warp][__ffs(g) - 1];
            atomicAdd(&B.F[(int64_t)ci * B.nt + slot], sum);
        }
        __syncwarp();
    }
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

// List entries of C cubes: two per (face, triangle) on average; a triangle
// meets one face or two in earnest, so this leaves room for meshes of large
// ones, and tiles past the end look through their face's boxes.
int64_t list_entries(int64_t C, int64_t nt) { return 2 * C * nt; }

// Workspace layout for nb candidates per batch.
size_t raster_bytes(int64_t nt, int K, int R, int64_t nb) {
    const int64_t C = nb * K, E = C * 6 * nt, T = C * 6 * tiles_per_edge(R) * tiles_per_edge(R);
    const int64_t nblk = (T + kScanBlock * kScanPer - 1) / (kScanBlock * kScanPer);
    return align256(sizeof(uint2) * (size_t)E) + align256(sizeof(int) * (size_t)list_entries(C, nt)) +
           align256(sizeof(unsigned long long) * (size_t)(T + 1)) + align256(sizeof(unsigned) * (size_t)T) +
           align256(sizeof(unsigned long long) * (size_t)(nb * nt)) + align256(sizeof(float) * (size_t)R * R) +
           align256(sizeof(unsigned long long) * (size_t)(nblk + 1)) + 256;
}

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
    // the largest batch that fits (the bytes grow with nb; gridDim.y holds the cubes)
    for (int64_t hi = std::min<int64_t>(nc, 65535 / L.K) + 1; hi - nb > 1;) {
        const int64_t mid = (nb + hi) / 2;
        if (raster_bytes(nt, L.K, R, mid) <= bytes) nb = mid;
        else hi = mid;
    }
    const std::vector<float>& table = pixel_table(R);
    char* p = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(work) + 255) & ~uintptr_t(255));
    auto take = [&](size_t n) { char* q = p; p += align256(n); return q; };
    const int tn = tiles_per_edge(R);
    const int64_t Cmax = nb * L.K, Tmax = Cmax * 6 * tn * tn;
    RasterBatch B;
    B.tri = sc->tri;
    B.nt = (int)nt;
    B.R = R;
    B.K = L.K;
    B.tn = tn;
    B.L = L;
    B.box = reinterpret_cast<uint2*>(take(sizeof(uint2) * (size_t)(Cmax * 6 * nt)));
    B.list_cap = list_entries(Cmax, nt);
    B.list = reinterpret_cast<int*>(take(sizeof(int) * (size_t)B.list_cap));
    B.toff = reinterpret_cast<unsigned long long*>(take(sizeof(unsigned long long) * (size_t)(Tmax + 1)));
    B.cursor = reinterpret_cast<unsigned*>(take(sizeof(unsigned) * (size_t)Tmax));
    B.F = reinterpret_cast<unsigned long long*>(take(sizeof(unsigned long long) * (size_t)(nb * nt)));
    float* e_unit = reinterpret_cast<float*>(take(sizeof(float) * (size_t)R * R));
    unsigned long long* sums = reinterpret_cast<unsigned long long*>(p);
    B.e_unit = e_unit;
    B.tri_normal = tri_normal;
    cudaError_t err = cudaMemcpyAsync(e_unit, table.data(), sizeof(float) * table.size(), cudaMemcpyHostToDevice,
                                      stream);
    if (err != cudaSuccess) return status_from_cuda(err);
    const float near_eps = 1e-6f * fmaxf(sc->diameter, 1e-30f);
    const int grid = sm_count() * 8;
    for (int64_t i0 = 0; i0 < nc; i0 += nb) {
        const int64_t n = std::min<int64_t>(nb, nc - i0);
        B.C = (int)(n * L.K);
        B.cand = cand + 3 * i0;
        const int64_t T = (int64_t)B.C * 6 * tn * tn;
        const dim3 per_tri((unsigned)((nt + 255) / 256), (unsigned)B.C);
        cudaMemsetAsync(B.toff, 0, sizeof(unsigned long long) * (size_t)(T + 1), stream);
        cudaMemsetAsync(B.cursor, 0, sizeof(unsigned) * (size_t)T, stream);
        cudaMemsetAsync(B.F, 0, sizeof(unsigned long long) * (size_t)(n * nt), stream);
        k_rs_setup<<<per_tri, 256, 0, stream>>>(B, near_eps);
        const int64_t nblk = (T + kScanBlock * kScanPer - 1) / (kScanBlock * kScanPer);
        k_scan_blocks<<<(int)nblk, kScanBlock, 0, stream>>>(B.toff, T, sums);
        k_scan_sums<<<1, 32, 0, stream>>>(sums, (int)nblk, B.toff + T);
        k_scan_add<<<(int)((T + 255) / 256), 256, 0, stream>>>(B.toff, T, sums);
        k_rs_fill<<<per_tri, 256, 0, stream>>>(B);
        k_rs_tile<<<(unsigned)T, kTileThreads, 0, stream>>>(B);
        k_rs_finish<<<grid, 256, 0, stream>>>(B, (int)n, A + (size_t)i0 * lda, lda);
    }
    return status_from_cuda(cudaGetLastError());
}

}  // namespace uvc
