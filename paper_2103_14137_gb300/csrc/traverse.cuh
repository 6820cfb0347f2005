// Device code of the segment queries shared by the single-matrix, streamed
// and batched kernels: scene view, ray set-up, watertight segment/triangle
// test, four-wide packet traversal, and one irradiance entry (paper Sec.
// IV-C, Eq. (7) with its visibility rule).  See irradiance.cu for the design.
#pragma once

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "uvc_internal.cuh"

namespace uvc {
namespace {

// Resident blocks per SM the traversal kernels are compiled for (register cap
// 65536 / (256 * this)); tuning constants, measured on the ward workload.
#ifndef UVC_IRR_MIN_BLOCKS
#define UVC_IRR_MIN_BLOCKS 3
#endif
#ifndef UVC_STREAMED_MIN_BLOCKS
#define UVC_STREAMED_MIN_BLOCKS 3
#endif

constexpr unsigned kFull = 0xffffffffu;
// 1 + 2^-20: widening of the far slab distance; covers the relative rounding
// of (b - o) * (1/d) (three roundings) with a wide margin.
constexpr float kFarScale = 1.0f + 9.5367431640625e-07f;

// Checked build (UVC_CHECKED): every node, leaf and cached-triangle index of the
// traversals is tested against its array before it is used; an index out of
// range sets UVC_E_BOUNDS in the scene's status word and the access is
// skipped (the search ends for the lanes concerned, whose entries become NaN).
// The normal build compiles no checks.
#ifdef UVC_CHECKED
constexpr bool kChecked = true;
#else
constexpr bool kChecked = false;
#endif
__device__ __forceinline__ bool out_of_range(int* status, int idx, int n) {
    if (!kChecked || (idx >= 0 && idx < n)) return false;
    atomicCAS(status, 0, UVC_E_BOUNDS);
    return true;
}

struct SceneView {
    const float4* __restrict__ tri;
    const Node4* __restrict__ nodes4;
    const float4* __restrict__ ps;
    const float4* __restrict__ pn;
    const int2* __restrict__ pe;
    const float4* __restrict__ plates;   // [kMaxPlates][2], then the patch flag words
    int nt, np;
    uint16_t nplate;      // plates in use; kLooseBit set when triangles lie outside them
    uint16_t stack_cap;
    int visit_cap;
    float cut_eps;   // absolute slack (metres) subtracted from a patch's clearance
    float plate_eps;   // widening of a plate's box
    int* status;
};

constexpr int kLooseBit = 1 << 15;
static_assert(kMaxPlates < kLooseBit, "plates and their flag in 16 bits");
// Root reference: node 0, or the only triangle.
__device__ __forceinline__ int root_of(const SceneView& S) { return S.nt == 1 ? ~0 : 0; }

SceneView view_of(const uvc_scene* sc) {
    SceneView v;
    v.tri = sc->tri;
    v.nodes4 = sc->nodes4;
    v.ps = sc->patch_s;
    v.pn = sc->patch_n;
    v.pe = sc->patch_excl;
    v.nt = (int)sc->nt;
    v.np = (int)sc->np;
    // a scene with lowered limits searches the hierarchy for everything
    const bool plates = sc->nplate > 0 && sc->limit_stack <= 0 && sc->limit_visits <= 0;
    v.plates = sc->plates;
    v.nplate = (uint16_t)(plates ? (sc->nplate | (sc->nloose > 0 ? kLooseBit : 0)) : 0);
    // at most 3 pushes per four-wide level; a stack of 2^16 would not fit a block's
    // shared memory, its launch is refused
    v.stack_cap = (uint16_t)std::min(3 * ((int64_t)sc->depth4 + 1) + 1, (int64_t)65535);
    v.visit_cap = (int)sc->nt + 64;
    if (sc->limit_stack > 0 && sc->limit_stack < v.stack_cap) v.stack_cap = (uint16_t)sc->limit_stack;
    if (sc->limit_visits > 0 && sc->limit_visits < v.visit_cap) v.visit_cap = sc->limit_visits;
    v.cut_eps = 1e-5f * sc->diameter;
    // the box tests round absolute coordinates, by up to 2^-22 of them in all: in a
    // scene far from the origin that is more than cut_eps
    v.plate_eps = v.cut_eps + 4.76837158203125e-07f * sc->coord_bound;   // 2^-21
    v.status = sc->status;
    return v;
}

struct Ray {
    float ox, oy, oz;   // segment start (the source point, warp-uniform)
    float dx, dy, dz;   // segment vector: end = start + d
    float ix, iy, iz;   // 1/d with zero components replaced by +-1e-30
    float sx, sy, sz;   // shear constants of the watertight test
    float tend;         // box tests stop at this segment parameter (<= 1), see clearance
    int kx, ky, kz;     // axis permutation of the watertight test
    int ex0, ex1;       // triangles that never occlude this segment
};

__device__ __forceinline__ float pick(float x, float y, float z, int k) { return k == 0 ? x : (k == 1 ? y : z); }

__device__ __forceinline__ float safe_rcp(float d) {
    float a = fabsf(d) < 1e-30f ? copysignf(1e-30f, d) : d;
    return __frcp_rn(a);
}

__device__ __forceinline__ void setup_ray(Ray& r) {
    r.ix = safe_rcp(r.dx);
    r.iy = safe_rcp(r.dy);
    r.iz = safe_rcp(r.dz);
    float ax = fabsf(r.dx), ay = fabsf(r.dy), az = fabsf(r.dz);
    int kz = ax > ay ? (ax > az ? 0 : 2) : (ay > az ? 1 : 2);
    int kx = kz == 2 ? 0 : kz + 1;
    int ky = kx == 2 ? 0 : kx + 1;
    float dkz = pick(r.dx, r.dy, r.dz, kz);
    if (dkz < 0.f) { int t = kx; kx = ky; ky = t; }
    r.kx = kx; r.ky = ky; r.kz = kz;
    r.sz = __frcp_rn(dkz);   // the shear constants need no particular rounding, only one value per segment
    r.sx = __fmul_rn(pick(r.dx, r.dy, r.dz, kx), r.sz);
    r.sy = __fmul_rn(pick(r.dx, r.dy, r.dz, ky), r.sz);
}

__device__ __forceinline__ float max3f(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float min3f(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Watertight segment/triangle test: hit iff the segment's line passes through
// the closed triangle (all edge functions of one sign, non-degenerate) and
// the parameter tau = T/det lies in the open interval (0, 1).  The segment is
// given by its start (ox, oy, oz) and the shear constants of setup_ray.
__device__ __forceinline__ bool seg_tri_k(float ox, float oy, float oz, int kx, int ky, int kz, float sx, float sy,
                                          float sz, float4 a, float4 b, float4 c) {
    float Ax = __fsub_rn(a.x, ox), Ay = __fsub_rn(a.y, oy), Az = __fsub_rn(a.z, oz);
    float Bx = __fsub_rn(b.x, ox), By = __fsub_rn(b.y, oy), Bz = __fsub_rn(b.z, oz);
    float Cx = __fsub_rn(c.x, ox), Cy = __fsub_rn(c.y, oy), Cz = __fsub_rn(c.z, oz);
    float akz = pick(Ax, Ay, Az, kz), bkz = pick(Bx, By, Bz, kz), ckz = pick(Cx, Cy, Cz, kz);
    float ax = __fmaf_rn(-sx, akz, pick(Ax, Ay, Az, kx));
    float ay = __fmaf_rn(-sy, akz, pick(Ax, Ay, Az, ky));
    float bx = __fmaf_rn(-sx, bkz, pick(Bx, By, Bz, kx));
    float by = __fmaf_rn(-sy, bkz, pick(Bx, By, Bz, ky));
    float cx = __fmaf_rn(-sx, ckz, pick(Cx, Cy, Cz, kx));
    float cy = __fmaf_rn(-sy, ckz, pick(Cx, Cy, Cz, ky));
    float U = __fsub_rn(__fmul_rn(cx, by), __fmul_rn(cy, bx));
    float V = __fsub_rn(__fmul_rn(ax, cy), __fmul_rn(ay, cx));
    float W = __fsub_rn(__fmul_rn(bx, ay), __fmul_rn(by, ax));
    if ((U < 0.f || V < 0.f || W < 0.f) && (U > 0.f || V > 0.f || W > 0.f)) return false;
    float det = U + V + W;
    if (det == 0.f) return false;
    float T = U * __fmul_rn(sz, akz) + V * __fmul_rn(sz, bkz) + W * __fmul_rn(sz, ckz);
    // tau = T / det in (0, 1), compared without dividing
    unsigned sgn = __float_as_uint(det) & 0x80000000u;
    float Ts = __uint_as_float(__float_as_uint(T) ^ sgn);
    float ds = __uint_as_float(__float_as_uint(det) ^ sgn);
    return Ts > 0.f && Ts < ds;
}

__device__ __forceinline__ bool seg_tri(const Ray& r, float4 a, float4 b, float4 c) {
    return seg_tri_k(r.ox, r.oy, r.oz, r.kx, r.ky, r.kz, r.sx, r.sy, r.sz, a, b, c);
}

__device__ __forceinline__ uint32_t test_leaf(const SceneView& S, int k, const Ray& r, uint32_t mask, int lane) {
    const float4* t = S.tri + 3 * (size_t)k;
    float4 a = __ldg(t), b = __ldg(t + 1), c = __ldg(t + 2);
    int id = __float_as_int(a.w);
    bool hit = ((mask >> lane) & 1u) && id != r.ex0 && id != r.ex1 && seg_tri(r, a, b, c);
    return __ballot_sync(kFull, hit);
}

// Traversal counters of the instrumented variant (one launch, outside timing):
// [0] warp node visits, [1] warp leaf tests, [2] warp traversals,
// [3] lane segment box tests (alive lanes x 4 per node), [4] lane triangle
// tests (one segment against one triangle), [5] facing segments, [6] lane
// wedge box tests, [7] lane wedge plane tests (see the wedge traversal).
constexpr int kNumCounters = 8;

// Both boxes of a child pair (packed FP32x2).  Each lane loads, per axis, the
// pair of planes its segment meets first (near) and last (far): the near
// planes are the lower bounds when the direction component is positive, the
// upper bounds when it is negative (the sign of 1/d is that of d, zero
// components included), so no per-axis minimum or maximum is needed:
// t = (b - o) * (1/d), t_near = max(0, near values), t_far = min(tend, far
// values), and a child is entered when t_near <= t_far * (1 + 2^-20)
// (conservative).  tend < 1 skips the part of the segment next to the patch
// point that lies within the patch's clearance: no triangle there can
// occlude it (k_clearance).
__device__ __forceinline__ void pair_hits(const Ray& r, float2 nox, float2 noy, float2 noz, float2 ix, float2 iy,
                                          float2 iz, float2 nx, float2 fx, float2 ny, float2 fy, float2 nz,
                                          float2 fz, bool& h0, bool& h1) {
    const float2 tnx = __fmul2_rn(__fadd2_rn(nx, nox), ix), tfx = __fmul2_rn(__fadd2_rn(fx, nox), ix);
    const float2 tny = __fmul2_rn(__fadd2_rn(ny, noy), iy), tfy = __fmul2_rn(__fadd2_rn(fy, noy), iy);
    const float2 tnz = __fmul2_rn(__fadd2_rn(nz, noz), iz), tfz = __fmul2_rn(__fadd2_rn(fz, noz), iz);
    const float tn0 = max3f(tnx.x, tny.x, fmaxf(tnz.x, 0.f));
    const float tf0 = min3f(tfx.x, tfy.x, fminf(tfz.x, r.tend));
    const float tn1 = max3f(tnx.y, tny.y, fmaxf(tnz.y, 0.f));
    const float tf1 = min3f(tfx.y, tfy.y, fminf(tfz.y, r.tend));
    h0 = tn0 <= tf0 * kFarScale;
    h1 = tn1 <= tf1 * kFarScale;
}

__device__ __forceinline__ float2 ldg2(const char* p) { return __ldg(reinterpret_cast<const float2*>(p)); }

__device__ __forceinline__ int pick4(int4 v, int c) { return c == 0 ? v.x : (c == 1 ? v.y : (c == 2 ? v.z : v.w)); }

// Packet traversal of the four-wide tree from `node` with the lanes `alive`:
// returns the lanes found occluded; `failed` gets lanes whose search hit the
// visit cap; `hit_tri` receives the occluding leaf of each occluded lane.
// Children are entered in slot order (with the occluder cache in front, the
// order of children hardly changes the work).
// `all`: ~0 = the whole tree, 0 = only the subtrees that hold loose triangles.
template <bool COUNT>
__device__ __forceinline__ uint32_t traverse4(const SceneView& S, const Ray& r, uint32_t alive, unsigned all, int* stack,
                                           int lane, uint32_t& failed, unsigned long long* ctr, int& hit_tri) {
    const float2 nox = make_float2(-r.ox, -r.ox), noy = make_float2(-r.oy, -r.oy), noz = make_float2(-r.oz, -r.oz);
    const float2 ix = make_float2(r.ix, r.ix), iy = make_float2(r.iy, r.iy), iz = make_float2(r.iz, r.iz);
    // byte offset of the near pair inside an axis record (lo pair at 0, hi pair at 8)
    const int onx = (int)(__float_as_uint(r.dx) >> 31) * 8, ony = (int)(__float_as_uint(r.dy) >> 31) * 8,
              onz = (int)(__float_as_uint(r.dz) >> 31) * 8;
    uint32_t occl = 0;
    int top = 0, node = 0, visits = 0;
    unsigned long long c_leaf = 0, c_box = 0, c_tri = 0;
    while (true) {
        if (++visits > S.visit_cap) {
            failed = alive;
            if (lane == 0) atomicCAS(S.status, 0, UVC_E_TIMEOUT);
            break;
        }
        if (out_of_range(S.status, node, S.nt - 1)) {
            failed = alive;
            break;
        }
        const Node4* nd = S.nodes4 + node;
        const char* b = reinterpret_cast<const char*>(nd);
        const char *bnx = b + onx, *bfx = b + (8 - onx), *bny = b + 16 + ony, *bfy = b + 16 + (8 - ony);
        const char *bnz = b + 32 + onz, *bfz = b + 32 + (8 - onz);
        const int4 rr = __ldg(&nd->r);
        const int4 mm = __ldg(&nd->m);
        bool h0, h1, h2, h3;
        pair_hits(r, nox, noy, noz, ix, iy, iz, ldg2(bnx), ldg2(bfx), ldg2(bny), ldg2(bfy), ldg2(bnz), ldg2(bfz), h0, h1);
        pair_hits(r, nox, noy, noz, ix, iy, iz, ldg2(bnx + 48), ldg2(bfx + 48), ldg2(bny + 48), ldg2(bfy + 48),
                  ldg2(bnz + 48), ldg2(bfz + 48), h2, h3);
        if (COUNT) c_box += 4 * __popc(alive);
        // which children any searching lane enters (one warp OR-reduction)
        const unsigned nib = ((alive >> lane) & 1u) ? (unsigned)h0 | ((unsigned)h1 << 1) | ((unsigned)h2 << 2) |
                                                          ((unsigned)h3 << 3)
                                                    : 0u;
        const unsigned hit = __reduce_or_sync(kFull, nib) & ((unsigned)mm.z | all);
        unsigned leaves = hit & (unsigned)mm.x;
        while (leaves) {                   // leaf children: test their triangle
            const int c = __ffs(leaves) - 1;
            leaves &= leaves - 1;
            const uint32_t m = __ballot_sync(kFull, (nib >> c) & 1u) & alive;
            if (!m) continue;
            const int leaf = ~pick4(rr, c);
            if (out_of_range(S.status, leaf, S.nt)) {
                failed = alive;
                alive = 0;
                break;
            }
            if (COUNT) { ++c_leaf; c_tri += __popc(m); }
            const uint32_t h = test_leaf(S, leaf, r, m, lane);
            if ((h >> lane) & 1u) hit_tri = leaf;
            occl |= h;
            alive &= ~h;
        }
        if (!alive) break;
        unsigned inner = hit & (unsigned)mm.y;
        if ((leaves = hit & (unsigned)mm.x) != 0 && inner) {
            // lanes that just became occluded may have been the only ones wanting a child
            const unsigned nib2 = ((alive >> lane) & 1u) ? nib : 0u;
            inner &= __reduce_or_sync(kFull, nib2);
        }
        if (inner) {
            const int first = __ffs(inner) - 1;
            if (top + 3 > S.stack_cap) {
                failed = alive;
                if (lane == 0) atomicCAS(S.status, 0, UVC_E_STACK);
                break;
            }
            // push the others, highest slot first (branch-free)
            const unsigned rest = inner & (inner - 1);
            stack[top] = rr.w; top += (rest >> 3) & 1u;
            stack[top] = rr.z; top += (rest >> 2) & 1u;
            stack[top] = rr.y; top += (rest >> 1) & 1u;
            node = pick4(rr, first);
        } else {
            if (top == 0) break;
            node = stack[--top];
        }
    }
    if (COUNT && lane == 0) {
        atomicAdd(&ctr[0], (unsigned long long)visits);
        atomicAdd(&ctr[1], c_leaf);
        atomicAdd(&ctr[2], 1ull);
        atomicAdd(&ctr[3], c_box);
        atomicAdd(&ctr[4], c_tri);
    }
    return occl;
}

// Packet occlusion query for the lanes `alive`.
template <bool COUNT>
__device__ uint32_t warp_occluded(const SceneView& S, const Ray& r, uint32_t alive, unsigned all, int* stack, int lane,
                                  uint32_t& failed, unsigned long long* ctr, int& hit_tri) {
    failed = 0;
    if (COUNT && lane == 0) atomicAdd(&ctr[5], (unsigned long long)__popc(alive));
    if (S.nt == 0 || alive == 0) return 0;
    if (root_of(S) < 0) {
        if (COUNT && lane == 0) {
            atomicAdd(&ctr[1], 1ull);
            atomicAdd(&ctr[2], 1ull);
            atomicAdd(&ctr[4], (unsigned long long)__popc(alive));
        }
        const uint32_t h = test_leaf(S, ~root_of(S), r, alive, lane);
        if ((h >> lane) & 1u) hit_tri = ~root_of(S);
        return h;
    }
    return traverse4<COUNT>(S, r, alive, all, stack, lane, failed, ctr, hit_tri);
}

// Eq. (7) for one facing source: pw nv / d^3 from the squared distance d2.
// d^-3 = r^3 (1 + 1.5 e) with r the approximate reciprocal square root of d2
// (relative error 2^-22) and e = 1 - d2 r^2: the next term, 1.9 e^2, is below
// 2^-43.  Five roundings, as with a rounded square root and division (and half
// of the one of r^2, which e cancels in part), but no slow path to branch to
// and half the instructions.  Distances whose cube leaves FP32 take the plain
// form.
constexpr float kTermMin = 1e-24f, kTermMax = 1e24f;
__device__ __forceinline__ float rsqrt_approx(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float source_term(float pw, float nv, float d2) {
    if (!(d2 >= kTermMin && d2 <= kTermMax)) return __fmul_rn(pw, __fdiv_rn(nv, __fmul_rn(d2, sqrtf(d2))));
    const float r = rsqrt_approx(d2), r2 = __fmul_rn(r, r), r3 = __fmul_rn(r2, r);
    const float f = __fmaf_rn(d2, r2, -1.f);
    const float w = __fmaf_rn(__fmul_rn(f, -1.5f), r3, r3);
    return __fmul_rn(pw, __fmul_rn(nv, w));
}

// One source's terms for the patch point s (normal n): v = o - s as the
// rounded difference h plus its exact error (TwoSum), <n, v> with an
// error-free dot product (TwoProduct + TwoSum) rounded once, and |h|^2.  Both
// traversal paths call this, so their Eq. (7) terms agree bit for bit.
__device__ __forceinline__ void source_terms(float ox, float oy, float oz, float4 s4, float4 n4, float& hx, float& hy,
                                             float& hz, float& nv, float& d2) {
    hx = __fsub_rn(ox, s4.x);
    hy = __fsub_rn(oy, s4.y);
    hz = __fsub_rn(oz, s4.z);
    const float qx = __fsub_rn(hx, ox), qy = __fsub_rn(hy, oy), qz = __fsub_rn(hz, oz);
    const float lx = __fadd_rn(__fsub_rn(ox, __fsub_rn(hx, qx)), __fsub_rn(-s4.x, qx));
    const float ly = __fadd_rn(__fsub_rn(oy, __fsub_rn(hy, qy)), __fsub_rn(-s4.y, qy));
    const float lz = __fadd_rn(__fsub_rn(oz, __fsub_rn(hz, qz)), __fsub_rn(-s4.z, qz));
    const float p = __fmul_rn(n4.x, hx);
    float err = __fmaf_rn(n4.x, hx, -p);
    err = __fmaf_rn(n4.x, lx, err);
    float acc = p;
    {
        const float p2 = __fmul_rn(n4.y, hy);
        const float e2 = __fmaf_rn(n4.y, hy, -p2);
        const float s = __fadd_rn(acc, p2);
        const float z = __fsub_rn(s, acc);
        const float q = __fadd_rn(__fsub_rn(acc, __fsub_rn(s, z)), __fsub_rn(p2, z));
        acc = s;
        err = __fadd_rn(err, __fadd_rn(q, e2));
        err = __fmaf_rn(n4.y, ly, err);
    }
    {
        const float p3 = __fmul_rn(n4.z, hz);
        const float e3 = __fmaf_rn(n4.z, hz, -p3);
        const float s = __fadd_rn(acc, p3);
        const float z = __fsub_rn(s, acc);
        const float q = __fadd_rn(__fsub_rn(acc, __fsub_rn(s, z)), __fsub_rn(p3, z));
        acc = s;
        err = __fadd_rn(err, __fadd_rn(q, e3));
        err = __fmaf_rn(n4.z, lz, err);
    }
    nv = __fadd_rn(acc, err);
    d2 = __fmaf_rn(hx, hx, __fmaf_rn(hy, hy, __fmul_rn(hz, hz)));
}

// The patch of one lane: sample point, normal, excluded triangles.
struct PatchLane {
    float4 s, n;   // n.w = clearance (metres)
    int2 ex;
    bool valid;
};

__device__ __forceinline__ PatchLane load_patch(const SceneView& S, int j) {
    PatchLane P;
    P.valid = j < S.np;
    P.s = make_float4(0.f, 0.f, 0.f, 0.f);
    P.n = P.s;
    P.ex = make_int2(-1, -1);
    if (P.valid) {
        P.s = __ldg(&S.ps[j]);
        P.n = __ldg(&S.pn[j]);
        P.ex = __ldg(&S.pe[j]);
    }
    return P;
}

// ---------------------------------------------------------------------------
// Plates: segments decided at whole rectangles before any search
// ---------------------------------------------------------------------------
// A plate (plates.cu) is a flat, axis-aligned rectangle that triangles of the
// mesh tile completely.  One test per (lane, plate) decides all the segments
// from a vertical column of sources to the lane's point:
//   blocked   the segment crosses the plate's plane well inside the rectangle,
//             with both ends well off the plane: the tiling has no gaps and
//             the watertight test none either (neighbours evaluate a shared
//             edge to opposite values, rounding included), so one of the
//             plate's triangles hits
//   clear     the wedge box test misses the rectangle's box (a search would
//             enter no box inside it), or the segment stays well on one side
//             of the plane, or crosses it well outside: none of them hits
//   open      anything nearer to a border or an end; only these segments go
//             on to the search
// so every visibility bit is the search's own.  "Well": with u = 2^-24 and R the
// distance of a triangle's vertices from the source, the test's roundings move
// the triangle, seen along the segment, by at most 6 u R per coordinate
// (differences u, shear 4 u, product u), 2^-20.9 R in all.  R is at most the
// longest segment plus the plate's longest triangle edge for the triangles
// near a crossing; the margin is 2^-19 of that sum, divided by the segment's
// cosine with the plane's normal within the plane.  Off the plane the ends must
// be by 2^-19 of that sum plus 2^-16 of the edge: the rounding of a triangle's
// barycentric coordinates (2 u edge^2 each over its projected area, at least
// edge^2 / 32 times the cosine: 192 u / cosine in all) moves a hit by that part
// of its edge along the segment, 192 u of it along the normal.  All coordinates
// are differences from the source's foot or the point; a rectangle's middle and
// half width from those carry 3 u of its far side, for which 2^-21 of it is added
// to the margin.  NaN and infinities fail the comparisons and stay open.
//
// Which plates the packet's wedges can reach is found 32 at a time, a plate
// per lane, against the packet's shaft: the hull's box, the two vertical
// planes through the column that hold all points, and the two slanted planes
// below and above.  The rectangles are widened by twice the box tests' own
// widening, so the shaft misses no box test that would hit.  The box tests here
// are widened by more than the search's (SceneView::plate_eps).
// Measured on a ward (49,066 triangles in 66 plates, 98,132 x 2,000 pairs,
// K = 8): matrix 55.4 -> 10.5 ms, 7.45 with the set-up by surface and the lamp's
// ends tested first (ENDS: set-up 2.3 ms, shaft 0.7, cull 1.2, 1.2 rectangles hit
// a packet 2.4, hierarchy 0.8); on a floor of rooms (531,284 triangles) the
// streamed fluence 52.3 -> 5.0 ms, 2.6 with its weighting.
__device__ __forceinline__ float redux_min(float x) {
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float redux_max(float x) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// The horizontal slab constants of the wedge box tests (see WedgeLane).
struct Slabs {
    float igx, igy, oxn, oxf, oyn, oyf;
};

__device__ __forceinline__ Slabs slabs_of(float cx, float cy, float gx, float gy, float delta) {
    Slabs b;
    const float sgx = (__float_as_uint(gx) >> 31) ? -delta : delta;
    const float sgy = (__float_as_uint(gy) >> 31) ? -delta : delta;
    b.igx = safe_rcp(gx);
    b.igy = safe_rcp(gy);
    b.oxn = __fmul_rn(-(cx + sgx), b.igx);
    b.oxf = __fmul_rn(-(cx - sgx), b.igx);
    b.oyn = __fmul_rn(-(cy + sgy), b.igy);
    b.oyf = __fmul_rn(-(cy - sgy), b.igy);
    return b;
}

// What the plates need to know of the lane's point.  A point exactly in a
// plate's plane, with no other triangle of that plane (excluded ones aside)
// nearer than `gap`: a segment from the free side meets the plane in the point
// only.  The test's roundings along the normal scale with the source's height
// over the plane here, as the point and the vertices share that coordinate:
// seen in the plane they move a triangle by at most 6 u (dmax + edge) whatever
// the angle.  A point outside a triangle by more lies outside the moved one, and
// past one of its edges by 1/64 of that or more (angles of 1/32 at least), which
// the products' rounding (2 u edge) cannot hide: clear from 2^-20 dmax + 2^-16
// edge on.
struct PlateLane {
    bool flagged;    // takes no plate for an occluder (plates.cu: k_plate_patches)
    int own_axis;    // axis of the point's own plane, -1 = none
    float own;       // its coordinate
    float gap;       // metres
    int plate;       // the only plate that the gap holds for, -1 = all of the plane
};

__device__ __forceinline__ PlateLane no_plate_lane() { return PlateLane{false, -1, 0.f, 0.f, -1}; }

// The sources q < K of a column stand at (cx, cy, zsrc(q)); `want` holds the
// lane's sources that need a search, zlo and zhi their extreme heights, g and
// sz the lane's point (from c, horizontally; height), lend the largest
// parameter a search would look at, dmax the longest segment.  Takes the
// blocked sources out of `want` and returns the open ones among the rest (the
// others are clear of every plate).  Every lane of the warp calls it.
// UVC_PLATE_LOOP: a file whose kernel leaves the instruction cache (the area mean)
// defines it to keep the loops over the sources rolled.
#ifndef UVC_PLATE_LOOP
#define UVC_PLATE_LOOP
#endif
template <bool ENDS, class Z>
__device__ __forceinline__ uint32_t plates_decide(const SceneView& S, Z zsrc, int K, float cx, float cy, float sz,
                                                  float gx, float gy, float zlo, float zhi, float lend, float dmax,
                                                  const Slabs& sl, const PlateLane& pl, int lane, uint32_t& want) {
    const float kBig = 3.0e38f, kWide = 4.76837158203125e-07f;   // 2^-21: the rounding of a rectangle's middle and half width
    const bool a0 = want != 0u;
    const float delta = S.plate_eps, diag = S.cut_eps * 1e5f;
    // far outside the scene (or infinite, or NaN) the widening no longer covers the rounding of the shaft
    if (__any_sync(kFull, a0 && !(dmax < 32.f * diag))) return want;
    // the packet's shaft, relative to the column's foot in x and y
    const float tx = lend * gx, ty = lend * gy;
    const float tl = fmaf(lend, sz - zlo, zlo), th = fmaf(lend, sz - zhi, zhi);
    const float x0 = redux_min(a0 ? tx : kBig), x1 = redux_max(a0 ? tx : -kBig);
    const float y0 = redux_min(a0 ? ty : kBig), y1 = redux_max(a0 ? ty : -kBig);
    const float z0 = redux_min(a0 ? zlo : kBig), z1 = redux_max(a0 ? zhi : -kBig);
    const float zb = redux_min(a0 ? fminf(tl, zlo) : kBig), zt = redux_max(a0 ? fmaxf(th, zhi) : -kBig);
    const float ux = x0 + x1, uy = y0 + y1;
    const float along = tx * ux + ty * uy;
    const bool cone = redux_min(a0 ? along : kBig) > 0.f;
    const float r = rcp_approx(along), slope = (ux * ty - uy * tx) * r;
    const float s0 = redux_min(a0 ? slope : kBig), s1 = redux_max(a0 ? slope : -kBig);
    const float q0 = redux_min(a0 ? (tl - z0) * r : kBig), q1 = redux_max(a0 ? (th - z1) * r : -kBig);
    const float hx0 = fminf(x0, 0.f), hx1 = fmaxf(x1, 0.f), hy0 = fminf(y0, 0.f), hy1 = fmaxf(y1, 0.f);
    const float ax1 = -uy - s1 * ux, ay1 = ux - s1 * uy;   // outside the far side plane: ax1 x + ay1 y > 0
    const float ax0 = uy + s0 * ux, ay0 = s0 * uy - ux;
    const float bx0 = q0 * ux, by0 = q0 * uy, bx1 = -q1 * ux, by1 = -q1 * uy;
    const float e = 2.f * delta;
    const int n = S.nplate & ~kLooseBit;
    uint32_t open = 0u;
    for (int base = 0; base < n; base += 32) {
        bool in = false;
        if (base + lane < n) {
            const float4 lo = __ldg(&S.plates[2 * (base + lane)]), hi = __ldg(&S.plates[2 * (base + lane) + 1]);
            const float lx = lo.x - cx - e, ux_ = hi.x - cx + e, ly = lo.y - cy - e, uy_ = hi.y - cy + e;
            const float lz = lo.z - e, uz = hi.z + e;
            in = lx <= hx1 && ux_ >= hx0 && ly <= hy1 && uy_ >= hy0 && lz <= zt && uz >= zb;
            if (cone && in) {
                const float f1 = ax1 * (ax1 > 0.f ? lx : ux_) + ay1 * (ay1 > 0.f ? ly : uy_);
                const float f0 = ax0 * (ax0 > 0.f ? lx : ux_) + ay0 * (ay0 > 0.f ? ly : uy_);
                const float g0 = z0 + bx0 * (bx0 > 0.f ? lx : ux_) + by0 * (by0 > 0.f ? ly : uy_) - uz;
                const float g1 = lz - z1 + bx1 * (bx1 > 0.f ? lx : ux_) + by1 * (by1 > 0.f ? ly : uy_);
                in = !(f1 > 0.f || f0 > 0.f || g0 > 0.f || g1 > 0.f);
            }
        }
        for (uint32_t hits = __ballot_sync(kFull, in); hits; hits &= hits - 1) {
            const int p = base + __ffs(hits) - 1;
            const float4 lo = __ldg(&S.plates[2 * p]), hi = __ldg(&S.plates[2 * p + 1]);
            const int axis = __float_as_int(lo.w);
            const float reach = dmax + hi.w;
            const float far_off = reach * 1.9073486328125e-06f + hi.w * 1.52587890625e-05f;   // 2^-19, 2^-16
            const float near_in = reach * 1.9073486328125e-06f;   // 2^-19
            if (want) {
                // the wedge box test (wedge_pair_hits) on the rectangle's box
                const bool nx = __float_as_uint(gx) >> 31, ny = __float_as_uint(gy) >> 31;
                const float a = max3f(fmaf(nx ? hi.x : lo.x, sl.igx, sl.oxn), fmaf(ny ? hi.y : lo.y, sl.igy, sl.oyn), 0.f);
                const float b = min3f(fmaf(nx ? lo.x : hi.x, sl.igx, sl.oxf), fmaf(ny ? lo.y : hi.y, sl.igy, sl.oyf), lend);
                const float wl = fminf(fmaf(a, sz - zlo, zlo), fmaf(b, sz - zlo, zlo)) - delta;
                const float wh = fmaxf(fmaf(a, sz - zhi, zhi), fmaf(b, sz - zhi, zhi)) + delta;
                if (a <= b && hi.z >= wl && lo.z <= wh) {
                    uint32_t blocked = 0u, clear = 0u;
                    if (axis == pl.own_axis && pl.own == (axis == 0 ? lo.x : (axis == 1 ? lo.y : lo.z)) &&
                        (pl.plate < 0 || pl.plate == p)) {
                        const float h = axis == 0 ? fabsf(cx - lo.x) : (axis == 1 ? fabsf(cy - lo.y) : fmaxf(zlo - lo.z, lo.z - zhi));
                        if (pl.gap > 9.5367431640625e-07f * dmax + 1.52587890625e-05f * hi.w && h > 1e-6f * reach)
                            clear = want;   // 2^-20, 2^-16
                    } else if (axis != 2) {
                        const bool isx = axis == 0;
                        const float ho = isx ? cx - lo.x : cy - lo.y, ga = isx ? gx : gy, ig = isx ? sl.igx : sl.igy;
                        const float gb = isx ? gy : gx, hs = ho + ga;
                        const float lb = isx ? lo.y - cy : lo.x - cx, ub = isx ? hi.y - cy : hi.x - cx;
                        if (fminf(fabsf(ho), fabsf(hs)) >= far_off) {
                            const float lam = -ho * ig, mid = 0.5f * (lb + ub), half = 0.5f * (ub - lb);
                            const float m0 = near_in * dmax * fabsf(ig), m = fmaf(fabsf(mid) + half, kWide, m0);
                            const float t = fabsf(fmaf(lam, gb, -mid)) - half;
                            if (ho * hs > 0.f || t > m) {
                                clear = want;
                            } else {
                                const bool inside = t < -m;
                                const float lz = lo.z - sz, uz = hi.z - sz, mu = 1.f - lam;
                                const float mz = 0.5f * (lz + uz), hz = 0.5f * (uz - lz);
                                const float w = fmaf(fabsf(mz) + hz, kWide, m0);
                                const float e0 = fmaf(mu, zlo - sz, -mz), e1 = fmaf(mu, zhi - sz, -mz);
                                if (ENDS && fmaxf(-e1, e0) - hz > w) clear = want;
                                else if (ENDS && inside && fmaxf(-e0, e1) - hz < -w) blocked = want;
                                else UVC_PLATE_LOOP for (int q = 0; q < K; ++q) {
                                    const float tz = fabsf(fmaf(mu, zsrc(q) - sz, -mz)) - hz;
                                    if (tz > w) clear |= 1u << q;
                                    else if (inside && tz < -w) blocked |= 1u << q;
                                }
                            }
                        }
                    } else {
                        const float hs = sz - lo.z;
                        const float lx = lo.x - cx, ux_ = hi.x - cx, ly = lo.y - cy, uy_ = hi.y - cy;
                        const float xc = 0.5f * (lx + ux_), hx = 0.5f * (ux_ - lx), yc = 0.5f * (ly + uy_), hy = 0.5f * (uy_ - ly);
                        const float wide = fmaxf(fabsf(xc) + hx, fabsf(yc) + hy) * kWide;
                        if (fabsf(hs) >= far_off) {
                            bool done = false;
                            if (ENDS) {   // both ends of the lamp on one side; the crossing points lie on a line between theirs
                                const float h0 = zlo - lo.z, h1 = zhi - lo.z;
                                const bool off = fminf(fabsf(h0), fabsf(h1)) >= far_off;
                                if (fminf(h0 * hs, h1 * hs) > 0.f) {
                                    done = off;
                                    if (off) clear = want;
                                } else if (off && fmaxf(h0 * hs, h1 * hs) < 0.f) {
                                    const float i0 = rcp_approx(h0 - hs), i1 = rcp_approx(h1 - hs);
                                    const float m = fmaf(near_in * dmax, fmaxf(fabsf(i0), fabsf(i1)), wide);
                                    const float xa = fmaf(h0 * i0, gx, -xc), xb = fmaf(h1 * i1, gx, -xc);
                                    const float ya = fmaf(h0 * i0, gy, -yc), yb = fmaf(h1 * i1, gy, -yc);
                                    const float away = fmaxf(fmaxf(fminf(xa, xb), -fmaxf(xa, xb)) - hx,
                                                             fmaxf(fminf(ya, yb), -fmaxf(ya, yb)) - hy);
                                    const float in_ = fmaxf(fmaxf(fabsf(xa), fabsf(xb)) - hx, fmaxf(fabsf(ya), fabsf(yb)) - hy);
                                    done = away > m || in_ < -m;
                                    if (away > m) clear = want;
                                    else if (in_ < -m) blocked = want;
                                }
                            }
                            if (!done)
                                UVC_PLATE_LOOP for (int q = 0; q < K; ++q) {
                                    const float hm = zsrc(q) - lo.z, dz = hm - hs;
                                    if (fabsf(hm) >= far_off) {
                                        const float ig = rcp_approx(dz), lam = hm * ig;
                                        const float m = fmaf(near_in * dmax, fabsf(ig), wide);
                                        const float t = fmaxf(fabsf(fmaf(lam, gx, -xc)) - hx, fabsf(fmaf(lam, gy, -yc)) - hy);
                                        if (hm * hs > 0.f || t > m) clear |= 1u << q;
                                        else if (t < -m) blocked |= 1u << q;
                                    }
                                }
                        }
                    }
                    if (pl.flagged) blocked = 0u;
                    open |= want & ~(blocked | clear);
                    want &= ~blocked;
                }
            }
            if (!__any_sync(kFull, want != 0u)) return 0u;
        }
    }
    return open & want;
}

// The lane's patch (its flag bit: plates.cu, k_plate_patches).  A patch on an
// axis plane that has a clearance has no triangle of that plane but its own
// within 2^-14 of the scene's diagonal, nor within the clearance if that is less:
// the search for it looks at nothing farther away (build_bvh.cu: k_clearance).
__device__ __forceinline__ PlateLane plate_lane(const SceneView& S, int jb, int lane, const PatchLane& P) {
    PlateLane pl;
    pl.flagged = (__ldg(reinterpret_cast<const uint32_t*>(S.plates + 2 * kMaxPlates) + jb) >> lane) & 1u;
    const bool x = fabsf(P.n.x) == 1.f, y = fabsf(P.n.y) == 1.f, z = fabsf(P.n.z) == 1.f;
    const bool unit = (x && P.n.y == 0.f && P.n.z == 0.f) || (y && P.n.x == 0.f && P.n.z == 0.f) ||
                      (z && P.n.x == 0.f && P.n.y == 0.f);
    pl.own_axis = unit && P.n.w > 0.f ? (x ? 0 : (y ? 1 : 2)) : -1;
    pl.own = x ? P.s.x : (y ? P.s.y : P.s.z);
    pl.gap = fminf(S.cut_eps * 6.f, P.n.w);   // 1e5 2^-14 = 6.1
    pl.plate = -1;
    return pl;
}

// Irradiance of candidate i at this lane's patch (lanes beyond np give 0).
// Writes the K visibility words when vis != nullptr.  Returns NaN for a lane
// whose search failed (and records UVC_E_TIMEOUT / UVC_E_STACK).
// Each source's segments are decided at the plates where that can be done (a
// column of one source); the rest take the packet search: all of them through
// the subtrees that hold loose triangles, the open ones through the whole tree.
// `cache` is the lane's last occluding triangle (sorted index, -1 = none): it
// is tested first, and a hit settles the segment without a traversal (the
// same predicate the traversal would apply to that triangle).
template <bool COUNT, bool PLATES>
__device__ __forceinline__ float irradiance_entry(const SceneView& S, const float* __restrict__ cand, int nc,
                                                  const LampDev& L, int i, int jb, int lane, int* stack,
                                                  uint32_t* __restrict__ vis, int nwords, const PatchLane& P,
                                                  int& cache, unsigned long long* ctr = nullptr) {
    const float4 s4 = P.s, n4 = P.n;
    const float cx = __ldg(&cand[3 * (size_t)i]), cy = __ldg(&cand[3 * (size_t)i + 1]),
                cz = __ldg(&cand[3 * (size_t)i + 2]);
    const bool plates = PLATES && S.nplate != 0 && L.plates;
    const PlateLane pl = plates ? plate_lane(S, jb, lane, P) : no_plate_lane();
    float E = 0.f;
    bool bad = false;
    for (int m = 0; m < L.K; ++m) {
        const float ox = __fadd_rn(cx, L.ox[m]), oy = __fadd_rn(cy, L.oy[m]), oz = __fadd_rn(cz, L.oz[m]);
        float hx, hy, hz, nv, d2;
        source_terms(ox, oy, oz, s4, n4, hx, hy, hz, nv, d2);
        const float d = sqrtf(d2);
        const bool facing = P.valid && nv > 0.f && d2 > 0.f;
        // the last `cut` metres before the patch point need no box tests; a
        // segment shorter than the cut meets no triangle at all
        const float cut = __fmaf_rn(0.99f, P.n.w, -S.cut_eps);
        const float tend = cut > 0.f ? 1.f - cut * __frcp_rn(d) : 1.f;
        const uint32_t facing_mask = __ballot_sync(kFull, facing);
        uint32_t want = facing && !(tend <= 0.f) ? 1u : 0u, open = want, found = 0u, failed = 0u;
        const uint32_t before = want;
        if (plates && __any_sync(kFull, want))
            open = plates_decide<false>(S, [&](int) { return oz; }, 1, ox, oy, s4.z, -hx, -hy, oz, oz,
                                 tend, d, slabs_of(ox, oy, -hx, -hy, S.plate_eps), pl, lane, want);
        for (int whole = plates && (S.nplate & kLooseBit) ? 0 : 1; whole < 2; ++whole) {
            const uint32_t search = __ballot_sync(kFull, want && (whole ? open : !open));
            if (!search) continue;
            Ray r;
            r.ox = ox; r.oy = oy; r.oz = oz;
            r.dx = -hx; r.dy = -hy; r.dz = -hz;
            r.ex0 = P.ex.x; r.ex1 = P.ex.y;
            setup_ray(r);
            r.tend = tend;
            bool cached_hit = false;
            if (((search >> lane) & 1u) && cache >= 0 && !out_of_range(S.status, cache, S.nt)) {
                const float4* t = S.tri + 3 * (size_t)cache;
                cached_hit = seg_tri(r, __ldg(t), __ldg(t + 1), __ldg(t + 2));
            }
            const uint32_t cached_mask = __ballot_sync(kFull, cached_hit);
            uint32_t fail_now;
            int hit_tri = -1;
            found |= cached_mask | warp_occluded<COUNT>(S, r, search & ~cached_mask, whole ? ~0u : 0u, stack, lane,
                                                        fail_now, ctr, hit_tri);
            failed |= fail_now;
            if (hit_tri >= 0) cache = hit_tri;
        }
        const uint32_t occl = __ballot_sync(kFull, before && !want) | found;
        const uint32_t visible = facing_mask & ~occl & ~failed;
        if (vis && lane == 0) vis[((size_t)m * nc + i) * nwords + jb] = visible;
        if ((failed >> lane) & 1u) bad = true;
        if ((visible >> lane) & 1u) {
            E = __fadd_rn(E, source_term(L.pw[m], nv, d2));
        }
    }
    return bad ? __int_as_float(0x7fffffff) : E;
}

// ---------------------------------------------------------------------------
// Wedge traversal for vertical line lamps
// ---------------------------------------------------------------------------
// When every source offset is vertical (x = y = 0), the sources of candidate
// c are o_m = (c.x, c.y, fl32(c.z + off_m.z)), all on the vertical line
// through c, and the segments from them to a patch point s lie in one
// triangle, the wedge conv(o_lo, o_hi, s) (o_lo, o_hi: the lowest and highest
// source still searching).  One packet traversal of the wedges replaces the K
// segment traversals: a child box is entered when it meets the lane's wedge,
// widened by delta, and every triangle reached is tested, with the same
// watertight segment test, against each source still searching that can meet
// it: none if the triangle lies entirely on one side of the wedge's vertical
// plane (farther than delta), else those in its lamp-height interval
// (lamp_interval).  A source stops at its first hit, a lane when all its
// sources have stopped, and the wedge narrows as its outer sources stop.
//
// Every triangle that a source's own segment traversal would reach is reached
// here (each segment lies inside the wedge, and delta = 1e-5 D exceeds the
// segment box test's widening), so each source gets the result of its own
// traversal; the only exception would be a triangle hit inside the patch's
// clearance, which only a triangle in the patch's own plane touching the
// patch point can be (a grazing pair).
//
// Coordinates: the horizontal part g of every segment of the lane is the same
// (the ray direction's x and y, rounded once in the set-up), so the point at
// segment parameter tau lies above c.xy + tau g whatever the source, and
// lambda = tau is a common parameter.  At lambda the wedge spans
//   zlow(lambda)  = z_lo + lambda (s.z - z_lo)  to
//   zhigh(lambda) = z_hi + lambda (s.z - z_hi).
// A box (widened by delta) meets the wedge iff its x and y slabs leave a
// lambda interval [a, b] inside [0, lambda_end] with z1 >= min(zlow(a),
// zlow(b)) and z0 <= max(zhigh(a), zhigh(b)) (both bounds are linear in
// lambda).  lambda_end is the largest clearance cut (tend) of the lane's
// searching sources.

struct WedgeLane {
    float2 oxn, oxf, oyn, oyf;   // -(c.x + delta sgn g.x) / g.x, -(c.x - delta sgn g.x) / g.x, same in y
    float2 igx, igy;             // 1/g.x, 1/g.y (as safe_rcp)
    float2 zl, zh, sl, sh;       // z_lo - delta, z_hi + delta, s.z - z_lo, s.z - z_hi
    float lend;                  // lambda_end
    float ig2;                   // 1 / |g|^2
    float mz;                    // delta * (longest segment) / |g|: margin of lamp_interval before 1/(1 - lambda)
    int onx, ony;                // byte offsets of the near planes in an axis record
};

__device__ __forceinline__ float2 dup2(float v) { return make_float2(v, v); }

// z range of the searching sources `want` (bit m = source m).
__device__ __forceinline__ void wedge_z(WedgeLane& w, uint32_t want, float cz, const LampDev& L, float sz,
                                        float delta) {
    float zlo = 3.0e38f, zhi = -3.0e38f;
    for (uint32_t b = want; b; b &= b - 1) {
        const float oz = __fadd_rn(cz, L.oz[__ffs(b) - 1]);
        zlo = fminf(zlo, oz);
        zhi = fmaxf(zhi, oz);
    }
    w.zl = dup2(zlo - delta);
    w.zh = dup2(zhi + delta);
    w.sl = dup2(sz - zlo);
    w.sh = dup2(sz - zhi);
}

// The sources of `want` whose segment can meet triangle (a, b, c).  Project
// the triangle orthogonally onto the wedge's vertical plane (the projection
// holds every point where the triangle meets the plane, and a segment that
// passes within e of the triangle passes within e of the projection) and then
// centrally from s onto the lamp line: a segment from height z meets the
// projection iff z lies in the image, which is the interval spanned by the
// images z_s + (z_V - z_s) / (1 - lambda_V) of the three vertices while all
// lambda_V < 1.  The interval is widened by mz / (1 - lambda_max): a
// displacement e of a segment at parameter lambda moves its lamp end by at
// most e |d| / (|g| (1 - lambda)), and mz = delta |d|max / |g| with delta
// far above the rounding of the segment test and of this projection.  A
// triangle reaching lambda >= 1 - 2^-10 (next to s or beyond) keeps every
// source, as does a degenerate g (NaN comparisons fail).
__device__ __forceinline__ uint32_t lamp_interval(float ig2, float mz, uint32_t want, float4 a, float4 b, float4 c,
                                                  float cx, float cy, float cz, float sz, float gx, float gy,
                                                  const LampDev& L) {
    const float la = __fmul_rn(__fmaf_rn(__fsub_rn(a.x, cx), gx, __fmul_rn(__fsub_rn(a.y, cy), gy)), ig2);
    const float lb = __fmul_rn(__fmaf_rn(__fsub_rn(b.x, cx), gx, __fmul_rn(__fsub_rn(b.y, cy), gy)), ig2);
    const float lc = __fmul_rn(__fmaf_rn(__fsub_rn(c.x, cx), gx, __fmul_rn(__fsub_rn(c.y, cy), gy)), ig2);
    const float lmax = max3f(la, lb, lc);
    if (!(lmax < 0.9990234375f)) return want;
    const float za = __fmaf_rn(__fsub_rn(a.z, sz), rcp_approx(__fsub_rn(1.f, la)), sz);
    const float zb = __fmaf_rn(__fsub_rn(b.z, sz), rcp_approx(__fsub_rn(1.f, lb)), sz);
    const float zc = __fmaf_rn(__fsub_rn(c.z, sz), rcp_approx(__fsub_rn(1.f, lc)), sz);
    const float m = __fmul_rn(mz, rcp_approx(__fsub_rn(1.f, lmax)));
    const float z0 = __fsub_rn(min3f(za, zb, zc), m), z1 = __fadd_rn(max3f(za, zb, zc), m);
    if (L.wuniform) {
        // source q sits at fl32(cz + off_q), off_q within dz/64 of wz0 + q dz:
        // every q with a height in [z0, z1] lies in [ceil(t0 - 1/32), floor(t1 + 1/32)]
        const float t0 = fminf(fmaxf((z0 - cz - L.wz0) * L.wrdz, -4.f), 40.f);
        const float t1 = fminf(fmaxf((z1 - cz - L.wz0) * L.wrdz, -4.f), 40.f);
        const int qlo = max(0, (int)ceilf(t0 - 0.03125f)), qhi = min(L.K - 1, (int)floorf(t1 + 0.03125f));
        if (qhi < qlo) return 0u;
        return want & ((2u << qhi) - 1u) & ~((1u << qlo) - 1u);
    }
    uint32_t in = 0;
    for (uint32_t bits = want; bits; bits &= bits - 1) {
        const int q = __ffs(bits) - 1;
        const float oz = __fadd_rn(cz, L.oz[q]);
        if (oz >= z0 && oz <= z1) in |= 1u << q;
    }
    return in;
}

// The slab parameters lambda = (x - X) / g come as one FMA, x (1/g) + (-X / g),
// with -X / g rounded once per lane: the rounding moves a plane by about
// 2^-24 of the coordinates, far inside the delta the boxes are widened by.
__device__ __forceinline__ void wedge_pair_hits(const WedgeLane& w, float2 nx, float2 fx, float2 ny, float2 fy,
                                                float2 z0, float2 z1, bool& h0, bool& h1) {
    const float2 lnx = __ffma2_rn(nx, w.igx, w.oxn), lfx = __ffma2_rn(fx, w.igx, w.oxf);
    const float2 lny = __ffma2_rn(ny, w.igy, w.oyn), lfy = __ffma2_rn(fy, w.igy, w.oyf);
    const float2 a = make_float2(max3f(lnx.x, lny.x, 0.f), max3f(lnx.y, lny.y, 0.f));
    const float2 b = make_float2(min3f(lfx.x, lfy.x, w.lend), min3f(lfx.y, lfy.y, w.lend));
    const float2 la = __ffma2_rn(a, w.sl, w.zl), lb = __ffma2_rn(b, w.sl, w.zl);
    const float2 ha = __ffma2_rn(a, w.sh, w.zh), hb = __ffma2_rn(b, w.sh, w.zh);
    h0 = a.x <= b.x && z1.x >= fminf(la.x, lb.x) && z0.x <= fmaxf(ha.x, hb.x);
    h1 = a.y <= b.y && z1.y >= fminf(la.y, lb.y) && z0.y <= fmaxf(ha.y, hb.y);
}

// Per (source, lane) data of the wedge path, in shared memory (one warp's
// slice): shear constants and axis permutation of the source's segment, and
// its Eq. (7) term w_m P <n, v> / (4 pi |v|^3); and the warp's queue of leaf
// tests (see wedge_traverse): a ring of items (lane << 27 | leaf), and per
// lane the sources found occluded by the last batch and the leaf that did it.
// The packed items need leaf indices below 2^27 (kWedgeMaxTris); larger
// scenes take the per-source traversal.
// The queue is worked off, up to 32 items at a time, once kLeafFlush items
// wait (a tuning constant: fewer waiting items stop lanes sooner, more keep
// the batches fuller; on the ward 16: 76.7, 24: 75.9, 32: 77.1, 48: 80.4 ms
// per matrix).
#ifndef UVC_LEAF_FLUSH
#define UVC_LEAF_FLUSH 24
#endif
constexpr int kLeafQueue = 256;       // ring entries per warp (< kLeafFlush waiting + at most 4 x 32 new)
constexpr int kLeafBatch = 32;        // items per batch: one per lane
constexpr int kLeafFlush = UVC_LEAF_FLUSH;
static_assert(kLeafFlush - 1 + 4 * 32 <= kLeafQueue && (kLeafQueue & (kLeafQueue - 1)) == 0,
              "the ring holds the waiting items plus one node's");
constexpr uint32_t kOobBit = 0x80000000u;   // checked build: a leaf index out of range (sources use bits 0..15)
constexpr int kItemLeafBits = 27;
constexpr uint32_t kItemLeafMask = (1u << kItemLeafBits) - 1u;
struct WedgeSmem {
    float4* shear;            // [K][32]: (sx, sy, sz, kx | ky << 2 | kz << 4)
    float* term;              // [K][32]
    uint32_t* qitem;          // [kLeafQueue]: lane << 27 | leaf
    uint32_t* occ;            // [32]
    int* qhit;                // [32]
    char* base;               // where the arrays of all the block's warps start, and the K they are laid out for
    int base_k;
};

// Shared memory of a block of the traversal kernels: the warps' stacks
// (16-byte aligned size), then kernel-specific staging, then the wedge arrays
// of all warps (shear of every warp, then term of every warp).
__host__ __device__ inline size_t stack_smem_bytes(int stack_cap) {
    return ((size_t)kWarpsPerBlock * stack_cap * sizeof(int) + 15) & ~size_t(15);
}
constexpr size_t kWedgeQueueBytes = kLeafQueue * sizeof(uint32_t) + 32 * (sizeof(uint32_t) + sizeof(int));
inline size_t wedge_smem_bytes(int K) {
    return (size_t)kWarpsPerBlock * (K * 32 * (sizeof(float4) + sizeof(float)) + kWedgeQueueBytes);
}

__device__ __forceinline__ WedgeSmem wedge_smem(char* base, int K, int warp) {
    WedgeSmem w;
    w.base = base;
    w.base_k = K;
    const size_t per_src = (size_t)kWarpsPerBlock * K * 32;
    w.shear = reinterpret_cast<float4*>(base) + (size_t)warp * K * 32;
    w.term = reinterpret_cast<float*>(base + per_src * sizeof(float4)) + (size_t)warp * K * 32;
    char* q = base + per_src * (sizeof(float4) + sizeof(float));   // 4-byte aligned
    w.qitem = reinterpret_cast<uint32_t*>(q) + (size_t)warp * kLeafQueue;
    q += (size_t)kWarpsPerBlock * kLeafQueue * sizeof(uint32_t);
    w.occ = reinterpret_cast<uint32_t*>(q) + (size_t)warp * 32;
    q += (size_t)kWarpsPerBlock * 32 * sizeof(uint32_t);
    w.qhit = reinterpret_cast<int*>(q) + (size_t)warp * 32;
    return w;
}

// One batch of queued leaf tests: lane k of the warp takes item head + k
// (k < n), a leaf wanted by some lane `own` of the warp, and tests it with
// own's wedge (the plane and lamp-height filters) and own's searching
// sources (the watertight segment test with own's shear constants), as own
// would have done itself; the sources found occluded are OR-ed into own's
// word, which own folds into `want` after the batch (narrowing its wedge).
// Items whose lane has stopped are skipped.  Every lane of the warp calls it.
template <bool COUNT>
__device__ __forceinline__ void wedge_leaf_batch(const SceneView& S, const LampDev& L, WedgeLane& w, uint32_t& want,
                                                 int lane, const WedgeSmem& ws, int head, int n, float cx, float cy,
                                                 float cz, float sz, float gx, float gy, float mh, int ex0, int ex1,
                                                 unsigned& c_leaf, unsigned& c_tri, int& hit_tri, bool& oob) {
    const bool has = lane < n;
    const uint32_t item = has ? ws.qitem[(head + lane) & (kLeafQueue - 1)] : (uint32_t)lane << kItemLeafBits;
    const int own = (int)(item >> kItemLeafBits);
    const int leaf = (int)(item & kItemLeafMask);
    const uint32_t owant = __shfl_sync(kFull, want, own);
    const float osz = __shfl_sync(kFull, sz, own);
    const float ogx = __shfl_sync(kFull, gx, own);
    const float ogy = __shfl_sync(kFull, gy, own);
    const float omh = __shfl_sync(kFull, mh, own);
    const float oig2 = __shfl_sync(kFull, w.ig2, own);
    const float omz = __shfl_sync(kFull, w.mz, own);
    const int oex0 = __shfl_sync(kFull, ex0, own);
    const int oex1 = __shfl_sync(kFull, ex1, own);
    if (has && owant) {
        uint32_t occl = 0;
        if (out_of_range(S.status, leaf, S.nt)) {
            occl = kOobBit;
        } else {
            const float4* t = S.tri + 3 * (size_t)leaf;
            const float4 ta = __ldg(t), tb = __ldg(t + 1), tc = __ldg(t + 2);
            const int id = __float_as_int(ta.w);
            if (COUNT) ++c_leaf;
            if (id != oex0 && id != oex1) {
                // triangle entirely on one side of the wedge's vertical plane,
                // farther than delta: no segment of the lane can meet it
                const float qa = __fmaf_rn(__fsub_rn(ta.x, cx), -ogy, __fmul_rn(__fsub_rn(ta.y, cy), ogx));
                const float qb = __fmaf_rn(__fsub_rn(tb.x, cx), -ogy, __fmul_rn(__fsub_rn(tb.y, cy), ogx));
                const float qc = __fmaf_rn(__fsub_rn(tc.x, cx), -ogy, __fmul_rn(__fsub_rn(tc.y, cy), ogx));
                const bool beside = (qa > omh && qb > omh && qc > omh) || (qa < -omh && qb < -omh && qc < -omh);
                if (!beside) {
                    const uint32_t test = owant & lamp_interval(oig2, omz, owant, ta, tb, tc, cx, cy, cz, osz, ogx,
                                                                ogy, L);
                    for (uint32_t bits = test; bits; bits &= bits - 1) {
                        const int q = __ffs(bits) - 1;
                        const float4 sh = ws.shear[q * 32 + own];
                        const int kb = __float_as_int(sh.w);
                        if (COUNT) ++c_tri;
                        if (seg_tri_k(cx, cy, __fadd_rn(cz, L.oz[q]), kb & 3, (kb >> 2) & 3, (kb >> 4) & 3, sh.x,
                                      sh.y, sh.z, ta, tb, tc))
                            occl |= 1u << q;
                    }
                }
            }
        }
        if (occl) {
            atomicOr(&ws.occ[own], occl);
            atomicMax(&ws.qhit[own], leaf);   // the lane caches the highest such leaf (deterministic)
        }
    }
    __syncwarp();
    const uint32_t o = ws.occ[lane];
    if (o) {
        ws.occ[lane] = 0u;
        if (kChecked && (o & kOobBit)) {
            oob = true;
            want = 0u;
        }
        const uint32_t nw = want & ~o;
        if (nw != want) {
            want = nw;
            hit_tri = ws.qhit[lane];
            if (want) wedge_z(w, want, cz, L, sz, S.cut_eps);
        }
        ws.qhit[lane] = -1;
    }
    __syncwarp();
}

// Lane-level wedge search.  `want` holds the lane's searching sources and
// loses the bit of each source found occluded; `hit_tri` gets the last
// occluding leaf.
//
// The leaf children a lane's wedge enters are not tested at once: they go to
// the warp's queue (shared memory), and whenever 32 items wait the whole warp
// works off 32 of them, one per lane, whichever lane wanted them.  Lanes want
// leaves unevenly (a few lanes near dense geometry, the rest none), so testing
// them where they arise would leave most lanes idle; the queue keeps the leaf
// tests nearly fully occupied at the price of narrowing a lane's wedge (and
// stopping it) up to a batch later.  The sources a lane finds occluded are
// those of its own search: every leaf its wedge enters while a source is
// still searching is tested against that source.
template <bool COUNT>
__device__ __forceinline__ void wedge_traverse(const SceneView& S, const LampDev& L, WedgeLane& w, uint32_t& want,
                                               uint32_t alive, unsigned all, int* stack, int lane,
                                               const WedgeSmem& ws, float cx, float cy, float cz, float sz, float gx,
                                               float gy, float mh, int ex0,
                                               int ex1, uint32_t& failed, unsigned long long* ctr, int& hit_tri) {
    int top = 0, node = 0, visits = 0, head = 0, tail = 0;
    unsigned long long c_box = 0;
    unsigned c_leaf = 0, c_tri = 0;
    bool oob = false;   // checked build: this lane met an index out of range
    ws.occ[lane] = 0u;
    ws.qhit[lane] = -1;
    __syncwarp();
    while (true) {
        if (++visits > S.visit_cap) {
            failed = alive;
            if (lane == 0) atomicCAS(S.status, 0, UVC_E_TIMEOUT);
            break;
        }
        if (out_of_range(S.status, node, S.nt - 1)) {
            failed = alive;
            break;
        }
        const Node4* nd = S.nodes4 + node;
        const int4 rr = __ldg(&nd->r);
        const int4 mm = __ldg(&nd->m);
        bool h0, h1, h2, h3;
        {
            const char* b = reinterpret_cast<const char*>(nd);
            const char *bnx = b + w.onx, *bfx = b + (8 - w.onx), *bny = b + 16 + w.ony, *bfy = b + 16 + (8 - w.ony);
            const char* bz = b + 32;
            wedge_pair_hits(w, ldg2(bnx), ldg2(bfx), ldg2(bny), ldg2(bfy), ldg2(bz), ldg2(bz + 8), h0, h1);
            wedge_pair_hits(w, ldg2(bnx + 48), ldg2(bfx + 48), ldg2(bny + 48), ldg2(bfy + 48), ldg2(bz + 48),
                            ldg2(bz + 56), h2, h3);
        }
        if (COUNT) c_box += 4 * __popc(alive);
        const unsigned nib = ((alive >> lane) & 1u) ? (unsigned)h0 | ((unsigned)h1 << 1) | ((unsigned)h2 << 2) |
                                                          ((unsigned)h3 << 3)
                                                    : 0u;
        const unsigned hit = __reduce_or_sync(kFull, nib) & ((unsigned)mm.z | all);
        if (hit & (unsigned)mm.x) {
            // queue the lane's leaf children (prefix sum of the counts, at most 4 each)
            const unsigned mine = nib & hit & (unsigned)mm.x;
            const unsigned cnt = __popc(mine), lt = (1u << lane) - 1u;
            const unsigned b0 = __ballot_sync(kFull, cnt & 1u), b1 = __ballot_sync(kFull, cnt & 2u),
                           b2 = __ballot_sync(kFull, cnt & 4u);
            int pos = tail + __popc(b0 & lt) + 2 * __popc(b1 & lt) + 4 * __popc(b2 & lt);
            tail += __popc(b0) + 2 * __popc(b1) + 4 * __popc(b2);
            for (unsigned m = mine; m; m &= m - 1) {
                ws.qitem[pos & (kLeafQueue - 1)] = ((uint32_t)lane << kItemLeafBits) | (uint32_t)~pick4(rr, __ffs(m) - 1);
                ++pos;
            }
            __syncwarp();
            if (tail - head >= kLeafFlush) {
                do {
                    const int n = min(kLeafBatch, tail - head);
                    wedge_leaf_batch<COUNT>(S, L, w, want, lane, ws, head, n, cx, cy, cz, sz, gx, gy, mh, ex0, ex1,
                                            c_leaf, c_tri, hit_tri, oob);
                    head += n;
                } while (tail - head >= kLeafFlush);
                if (kChecked) failed |= __ballot_sync(kFull, oob);
                alive &= __ballot_sync(kFull, want != 0u);
                if (!alive) break;
            }
        }
        unsigned inner = hit & (unsigned)mm.y;
        if (inner) {
            const int first = __ffs(inner) - 1;
            if (top + 3 > S.stack_cap) {
                failed = alive;
                if (lane == 0) atomicCAS(S.status, 0, UVC_E_STACK);
                break;
            }
            const unsigned rest = inner & (inner - 1);
            stack[top] = rr.w; top += (rest >> 3) & 1u;
            stack[top] = rr.z; top += (rest >> 2) & 1u;
            stack[top] = rr.y; top += (rest >> 1) & 1u;
            node = pick4(rr, first);
        } else {
            if (top == 0) break;
            node = stack[--top];
        }
    }
    if (tail > head) {   // the leaves still queued when the traversal ends
        wedge_leaf_batch<COUNT>(S, L, w, want, lane, ws, head, tail - head, cx, cy, cz, sz, gx, gy, mh, ex0, ex1,
                                c_leaf, c_tri, hit_tri, oob);
        if (kChecked) failed |= __ballot_sync(kFull, oob);
    }
    if (COUNT && lane == 0) {
        atomicAdd(&ctr[0], (unsigned long long)visits);
        atomicAdd(&ctr[2], 1ull);
        atomicAdd(&ctr[6], c_box);
    }
    if (COUNT) {   // leaf loads (each with its plane test) and triangle tests, by the lanes that made them
        const unsigned nleaf = __reduce_add_sync(kFull, c_leaf);
        const unsigned ntri = __reduce_add_sync(kFull, c_tri);
        if (lane == 0) {
            atomicAdd(&ctr[1], (unsigned long long)nleaf);
            atomicAdd(&ctr[7], (unsigned long long)nleaf);
            atomicAdd(&ctr[4], (unsigned long long)ntri);
        }
    }
}

// a - b, rounded once, for both halves (m1 = -1, -1).
__device__ __forceinline__ float2 sub2(float2 a, float2 b, float2 m1) { return __ffma2_rn(b, m1, a); }

// Set-up of the segments from candidate c's sources to the lane's patch point:
// the arithmetic of source_terms and source_term, bit for bit, with what a
// vertical lamp's sources share computed once and two sources at a time in
// packed FP32x2 (one scalar source at a time took 2.9 ms of a 10.5 ms ward
// matrix).  Their Eq. (7) terms (0 where the source does not face) go to
// shared memory, and their sum in source order to `sum`.  Returns the facing
// sources and, in `want`, those that need a search (facing, longer than the
// clearance cut), with the largest cut parameter `lend`, the longest such
// segment `dmax` and the common horizontal direction (gx, gy).
// MODES: separate passes for horizontal and vertical normals (the walls, floors
// and ceilings of rooms: ward matrix 8.6 -> 8.1 ms, 7.5 with the whole-lamp form).
template <bool MODES>
__device__ __forceinline__ uint32_t wedge_setup_patch(const SceneView& S, const LampDev& L, float cx, float cy,
                                                      float cz, const PatchLane& P, int lane, const WedgeSmem& ws,
                                                      uint32_t& want, float& lend, float& dmax, float& gx,
                                                      float& gy, float& sum) {
    const float4 s4 = P.s, n4 = P.n;
    const float hx = __fsub_rn(cx, s4.x), hy = __fsub_rn(cy, s4.y);
    const float qx = __fsub_rn(hx, cx), qy = __fsub_rn(hy, cy);
    const float lx = __fadd_rn(__fsub_rn(cx, __fsub_rn(hx, qx)), __fsub_rn(-s4.x, qx));
    const float ly = __fadd_rn(__fsub_rn(cy, __fsub_rn(hy, qy)), __fsub_rn(-s4.y, qy));
    float acc0 = __fmul_rn(n4.x, hx);
    float err0 = __fmaf_rn(n4.x, lx, __fmaf_rn(n4.x, hx, -acc0));
    {
        const float p2 = __fmul_rn(n4.y, hy);
        const float e2 = __fmaf_rn(n4.y, hy, -p2);
        const float s = __fadd_rn(acc0, p2);
        const float z = __fsub_rn(s, acc0);
        const float q = __fadd_rn(__fsub_rn(acc0, __fsub_rn(s, z)), __fsub_rn(p2, z));
        acc0 = s;
        err0 = __fadd_rn(err0, __fadd_rn(q, e2));
        err0 = __fmaf_rn(n4.y, ly, err0);
    }
    const float2 m1 = make_float2(-1.f, -1.f), acc = make_float2(acc0, acc0), err = make_float2(err0, err0);
    const float2 nz = make_float2(n4.z, n4.z), nzn = make_float2(-n4.z, -n4.z), sz = make_float2(s4.z, s4.z);
    const float2 szn = make_float2(-s4.z, -s4.z), c2 = make_float2(cz, cz);
    const float2 hx2 = make_float2(hx, hx), hy2 = make_float2(hy, hy);
    uint32_t facing = 0;
    float far2 = 0.f;
    sum = 0.f;
    // One pass over the pairs of sources.  VERTICAL: for vertical normals, where
    // <n, v> is n.z times the rounded height difference (the rounded sum of a
    // rounded difference and its error is that difference): what the general
    // form gives.
    auto pass = [&](auto vertical) {
        constexpr bool VERTICAL = decltype(vertical)::value;
        for (int m = 0; m < L.K; m += 2) {
            const int k = min(m + 1, L.K - 1);   // an odd lamp's last source twice; its second half is dropped
            const float2 oz = __fadd2_rn(c2, make_float2(L.oz[m], L.oz[k]));
            const float2 hz = sub2(oz, sz, m1);
            float2 nv;
            if constexpr (VERTICAL) {
                nv = __fmul2_rn(nz, hz);
            } else {
                const float2 qz = sub2(hz, oz, m1);
                const float2 lz = __fadd2_rn(sub2(oz, sub2(hz, qz, m1), m1), sub2(szn, qz, m1));
                const float2 pn = __fmul2_rn(nzn, hz), e3 = __ffma2_rn(nz, hz, pn);   // pn = -(n.z h.z)
                const float2 s = sub2(acc, pn, m1), z = sub2(s, acc, m1);
                const float2 q = sub2(sub2(acc, sub2(s, z, m1), m1), __fadd2_rn(pn, z), m1);
                nv = __fadd2_rn(s, __ffma2_rn(nz, lz, __fadd2_rn(err, __fadd2_rn(q, e3))));
            }
            const float2 d2 = __ffma2_rn(hx2, hx2, __ffma2_rn(hy2, hy2, __fmul2_rn(hz, hz)));
            const float2 r = make_float2(rsqrt_approx(d2.x), rsqrt_approx(d2.y));
            const float2 r2 = __fmul2_rn(r, r), r3 = __fmul2_rn(r2, r), f = __ffma2_rn(d2, r2, m1);
            const float2 w = __ffma2_rn(__fmul2_rn(f, make_float2(-1.5f, -1.5f)), r3, r3);
            float2 t = __fmul2_rn(make_float2(L.pw[m], L.pw[k]), __fmul2_rn(nv, w));
            bool f0 = nv.x > 0.f, f1 = nv.y > 0.f && k > m;
            if (!(fminf(d2.x, d2.y) >= kTermMin && fmaxf(d2.x, d2.y) <= kTermMax)) {
                f0 = f0 && d2.x > 0.f;
                f1 = f1 && d2.y > 0.f;
                t = make_float2(source_term(L.pw[m], nv.x, d2.x), source_term(L.pw[k], nv.y, d2.y));
            }
            t.x = f0 ? t.x : 0.f;
            t.y = f1 ? t.y : 0.f;
            ws.term[m * 32 + lane] = t.x;
            if (k > m) ws.term[k * 32 + lane] = t.y;
            sum = __fadd_rn(__fadd_rn(sum, t.x), t.y);
            far2 = fmaxf(far2, fmaxf(f0 ? d2.x : 0.f, f1 ? d2.y : 0.f));
            facing |= ((uint32_t)f0 << m) | ((uint32_t)f1 << k);
        }
    };
    if constexpr (MODES) {
        // Horizontal normals (n.z = 0), where <n, v> is the same for all sources,
        // and vertical ones whose lamp is all above or all below: every source
        // faces or none does, and distances are extreme at the lamp's ends (each
        // step of d2 is monotonic under rounding).
        const bool hor = n4.z == 0.f, ver = n4.x == 0.f && n4.y == 0.f && fabsf(n4.z) == 1.f;
        const float hl = __fsub_rn(__fadd_rn(cz, L.zmin), s4.z), hh = __fsub_rn(__fadd_rn(cz, L.zmax), s4.z);
        const float he = fmaxf(-hl, hh), hm = fmaxf(fmaxf(hl, -hh), 0.f);   // largest and least distance in z
        const float dmin = __fmaf_rn(hx, hx, __fmaf_rn(hy, hy, __fmul_rn(hm, hm)));
        const float n0 = hor ? __fadd_rn(acc0, err0) : 0.f, n1 = hor ? 0.f : n4.z;
        const bool up = __fmaf_rn(n1, hl, n0) > 0.f, down = __fmaf_rn(n1, hh, n0) > 0.f;
        far2 = __fmaf_rn(hx, hx, __fmaf_rn(hy, hy, __fmul_rn(he, he)));
        const bool ordinary = dmin >= kTermMin && far2 <= kTermMax;
        const bool simple = __all_sync(kFull, !P.valid || ((hor || ver) && up == down && ordinary));
        if (simple) {
            const bool face = P.valid && up;
            if (__any_sync(kFull, face)) {
                const float2 b = dup2(n0), nzs = dup2(n1);
                for (int m = 0; m < L.K; m += 2) {
                    const float2 hz = sub2(__fadd2_rn(c2, *reinterpret_cast<const float2*>(&L.oz[m])), sz, m1);
                    const float2 nv = __ffma2_rn(nzs, hz, b);
                    const float2 d2 = __ffma2_rn(hx2, hx2, __ffma2_rn(hy2, hy2, __fmul2_rn(hz, hz)));
                    const float2 r = make_float2(rsqrt_approx(d2.x), rsqrt_approx(d2.y));
                    const float2 r2 = __fmul2_rn(r, r), r3 = __fmul2_rn(r2, r), f = __ffma2_rn(d2, r2, m1);
                    const float2 w = __ffma2_rn(__fmul2_rn(f, make_float2(-1.5f, -1.5f)), r3, r3);
                    const float2 t = __fmul2_rn(*reinterpret_cast<const float2*>(&L.pw[m]), __fmul2_rn(nv, w));
                    ws.term[m * 32 + lane] = t.x;
                    if (m + 1 < L.K) ws.term[(m + 1) * 32 + lane] = t.y;
                    sum = __fadd_rn(__fadd_rn(sum, t.x), t.y);   // an odd lamp's extra half adds 0
                }
            }
            sum = face ? sum : 0.f;
            facing = face ? (1u << L.K) - 1u : 0u;
        } else {
            far2 = 0.f;
            if (__all_sync(kFull, ver || !P.valid)) pass(std::true_type());
            else pass(std::false_type());
        }
    } else {
        pass(std::false_type());
    }
    if (!P.valid) facing = 0u;
    gx = -hx;
    gy = -hy;
    dmax = facing ? sqrtf(far2) : 0.f;
    want = facing;
    // a segment shorter than the cut meets no triangle at all; the lamp's
    // distance tells most lanes that none of theirs is
    const float cut = __fmaf_rn(0.99f, P.n.w, -S.cut_eps);
    if (cut > 0.f && facing) {
        const float dz = fmaxf(fmaxf(cz + L.zmin - s4.z, s4.z - (cz + L.zmax)), 0.f);
        if (!(hx * hx + hy * hy + dz * dz > 1.003f * cut * cut)) {
            dmax = 0.f;
            for (uint32_t b = facing; b; b &= b - 1) {
                const int m = __ffs(b) - 1;
                const float hz = __fsub_rn(__fadd_rn(cz, L.oz[m]), s4.z);
                const float d = sqrtf(__fmaf_rn(hx, hx, __fmaf_rn(hy, hy, __fmul_rn(hz, hz))));
                if (1.f - cut * __frcp_rn(d) > 0.f) dmax = fmaxf(dmax, d);
                else want &= ~(1u << m);
            }
        }
    }
    lend = !want ? 0.f : (cut > 0.f ? 1.f - cut * __frcp_rn(dmax) : 1.f);   // rises with d: the longest segment's
    return facing;
}

// As wedge_setup_patch, for the segments from the sources in `want` to point p
// (direction p - o rounded once, as a plain segment query; no clearance cut).
__device__ __forceinline__ void wedge_setup_point(const LampDev& L, float cx, float cy, float cz, float3 p,
                                                  uint32_t want, float& dmax, float& gx, float& gy) {
    dmax = 0.f;
    gx = __fsub_rn(p.x, cx);
    gy = __fsub_rn(p.y, cy);
    for (uint32_t bits = want; bits; bits &= bits - 1) {
        const float dz = __fsub_rn(p.z, __fadd_rn(cz, L.oz[__ffs(bits) - 1]));
        dmax = fmaxf(dmax, sqrtf(__fmaf_rn(gx, gx, __fmaf_rn(gy, gy, __fmul_rn(dz, dz)))));
    }
}

// Shear constants of the segments from the sources in `set` to the point
// (gx, gy from c, height sz), to shared memory.
__device__ __forceinline__ void wedge_shear(const LampDev& L, float cz, float sz, float gx, float gy, uint32_t set,
                                            int lane, const WedgeSmem& ws) {
    for (uint32_t bits = set; bits; bits &= bits - 1) {
        const int m = __ffs(bits) - 1;
        Ray r;
        r.dx = gx; r.dy = gy;
        r.dz = __fsub_rn(sz, __fadd_rn(cz, L.oz[m]));
        setup_ray(r);
        ws.shear[m * 32 + lane] = make_float4(r.sx, r.sy, r.sz, __int_as_float(r.kx | (r.ky << 2) | (r.kz << 4)));
    }
}

// What the plates leave of a search: one wedge search of the subtrees with
// loose triangles for the sources in `want` that are not open, and one of the
// whole tree for the open ones (for all where plates are not used).  A wedge
// search tests the lane's cached occluder, then walks the tree.  Returns the
// sources left unoccluded; `failed` gets the lanes whose search hit the visit
// cap or the stack limit.
template <bool COUNT>
__device__ __forceinline__ uint32_t wedge_rest(const SceneView& S, const LampDev& L, bool plates, float cx, float cy,
                                               float cz, float sz, float gx, float gy, uint32_t want, uint32_t open,
                                               float lend, float dmax, int2 ex, int lane, int* stack,
                                               const WedgeSmem& ws, const Slabs& sl, int& cache, uint32_t& failed,
                                               unsigned long long* ctr) {
    const float delta = S.cut_eps;
    for (int whole = plates && (S.nplate & kLooseBit) ? 0 : 1; whole < 2; ++whole) {
        uint32_t set = want & (whole ? open : ~open);
        if (!__any_sync(kFull, set != 0u)) continue;
        wedge_shear(L, cz, sz, gx, gy, set, lane, ws);
        WedgeLane w;
        const float g2 = __fmaf_rn(gx, gx, __fmul_rn(gy, gy));
        const float gn = sqrtf(g2);
        const float mh = delta * gn;   // plane margin (the plane's normal (-g.y, g.x) is not normalised)
        w.ig2 = 1.f / g2;
        w.mz = delta * dmax / gn;
        const uint32_t set0 = set;
        // the lane's last occluder first, against the searching sources it can reach
        if (set && cache >= 0 && !out_of_range(S.status, cache, S.nt)) {
            const float4* t = S.tri + 3 * (size_t)cache;
            const float4 ta = __ldg(t), tb = __ldg(t + 1), tc = __ldg(t + 2);
            const float qa = __fmaf_rn(__fsub_rn(ta.x, cx), -gy, __fmul_rn(__fsub_rn(ta.y, cy), gx));
            const float qb = __fmaf_rn(__fsub_rn(tb.x, cx), -gy, __fmul_rn(__fsub_rn(tb.y, cy), gx));
            const float qc = __fmaf_rn(__fsub_rn(tc.x, cx), -gy, __fmul_rn(__fsub_rn(tc.y, cy), gx));
            const bool beside = (qa > mh && qb > mh && qc > mh) || (qa < -mh && qb < -mh && qc < -mh);
            const uint32_t test = beside ? 0u : lamp_interval(w.ig2, w.mz, set, ta, tb, tc, cx, cy, cz, sz, gx, gy, L);
            for (uint32_t bits = test; bits; bits &= bits - 1) {
                const int q = __ffs(bits) - 1;
                const float4 sh = ws.shear[q * 32 + lane];
                const int kb = __float_as_int(sh.w);
                if (seg_tri_k(cx, cy, __fadd_rn(cz, L.oz[q]), kb & 3, (kb >> 2) & 3, (kb >> 4) & 3, sh.x, sh.y, sh.z,
                              ta, tb, tc))
                    set &= ~(1u << q);
            }
        }
        if (COUNT) {   // segments that need a search
            const unsigned nseg = __reduce_add_sync(kFull, (unsigned)__popc(set));
            if (lane == 0) atomicAdd(&ctr[5], (unsigned long long)nseg);
        }
        int hit_tri = -1;
        const uint32_t alive = __ballot_sync(kFull, set != 0u);
        if (alive) {
            if (root_of(S) < 0) {   // a single triangle: test it directly
                const float4* t = S.tri;
                const float4 ta = __ldg(t), tb = __ldg(t + 1), tc = __ldg(t + 2);
                const int id = __float_as_int(ta.w);
                if (id != ex.x && id != ex.y) {
                    for (uint32_t bits = set; bits; bits &= bits - 1) {
                        const int q = __ffs(bits) - 1;
                        const float4 sh = ws.shear[q * 32 + lane];
                        const int kb = __float_as_int(sh.w);
                        if (seg_tri_k(cx, cy, __fadd_rn(cz, L.oz[q]), kb & 3, (kb >> 2) & 3, (kb >> 4) & 3, sh.x, sh.y,
                                      sh.z, ta, tb, tc)) {
                            set &= ~(1u << q);
                            hit_tri = 0;
                        }
                    }
                }
            } else {
                w.oxn = dup2(sl.oxn);
                w.oxf = dup2(sl.oxf);
                w.oyn = dup2(sl.oyn);
                w.oyf = dup2(sl.oyf);
                w.igx = dup2(sl.igx);
                w.igy = dup2(sl.igy);
                w.lend = lend;
                w.onx = (int)(__float_as_uint(gx) >> 31) * 8;
                w.ony = (int)(__float_as_uint(gy) >> 31) * 8;
                if (set) wedge_z(w, set, cz, L, sz, delta);
                uint32_t fail_now = 0u;
                wedge_traverse<COUNT>(S, L, w, set, alive, whole ? ~0u : 0u, stack, lane, ws, cx, cy, cz, sz, gx, gy,
                                      mh, ex.x, ex.y, fail_now, ctr, hit_tri);
                failed |= fail_now;
            }
        }
        want &= ~(set0 & ~set);
        if (hit_tri >= 0) cache = hit_tri;
    }
    return want;
}

// wedge_rest as a call, for kernels that hold much else in registers (the
// batch's job records, the area mean's patches and gaps): on a room of plates a
// packet in a hundred gets there.  Measured with 128 registers (two blocks per SM):
// batched rooms 3.09 -> 2.71 ms, area mean 4.08 -> 3.56 ms; inlined at two blocks
// 3.07 and 3.83.  The streamed kernel: 2.67 against 2.84 ms inlined at three
// blocks.  The plain kernel is faster with it inlined at three blocks (ward matrix
// 8.1 against 8.6 ms).
constexpr int kCallMinBlocks = 2;
struct WedgeRest {
    uint32_t want, failed;
    int cache;
};
__device__ __noinline__ WedgeRest wedge_rest_call(const SceneView& S, const LampDev& L, bool plates, float cx, float cy,
                                                  float cz, float sz, float gx, float gy, uint32_t want, uint32_t open,
                                                  float lend, float dmax, int ex0, int ex1, int* stack, char* base,
                                                  int base_k, int cache) {
    WedgeRest r;
    r.failed = 0u;
    r.cache = cache;
    r.want = wedge_rest<false>(S, L, plates, cx, cy, cz, sz, gx, gy, want, open, lend, dmax, make_int2(ex0, ex1),
                               threadIdx.x & 31, stack, wedge_smem(base, base_k, threadIdx.x >> 5),
                               slabs_of(cx, cy, gx, gy, S.cut_eps), r.cache, r.failed, nullptr);
    return r;
}

// The search from the lamp line of candidate c to the lane's point (height sz,
// horizontal direction (gx, gy) from c) for the sources in `want`: the plates
// first, then the hierarchy for what they leave.  Returns the sources found
// occluded; `failed` as in wedge_rest.  PLATES: compiled with the plate tests
// (scenes without plates take kernels without them: their registers cost a
// tilted room 4 to 20 %).  CALL: wedge_rest is called, not inlined.
template <bool COUNT, bool PLATES, bool ENDS, bool CALL>
__device__ __forceinline__ uint32_t wedge_search(const SceneView& S, const LampDev& L, float cx, float cy, float cz,
                                                 float sz, float gx, float gy, uint32_t want, float lend, float dmax,
                                                 int2 ex, const PlateLane& pl, int lane, int* stack, const WedgeSmem& ws,
                                                 int& cache, uint32_t& failed, unsigned long long* ctr) {
    failed = 0;
    if (S.nt == 0 || !__any_sync(kFull, want != 0u)) return 0u;
    const uint32_t before = want;
    const bool plates = PLATES && S.nplate != 0 && L.plates;
    const Slabs sl = slabs_of(cx, cy, gx, gy, plates ? S.plate_eps : S.cut_eps);
    uint32_t open = want;
    if (plates) {
        float zlo = __fadd_rn(cz, L.zmin), zhi = __fadd_rn(cz, L.zmax);
        if (__any_sync(kFull, want != 0u && want != (1u << L.K) - 1u) && want) {
            zlo = 3.0e38f;
            zhi = -3.0e38f;
            for (uint32_t b = want; b; b &= b - 1) {
                const float oz = __fadd_rn(cz, L.oz[__ffs(b) - 1]);
                zlo = fminf(zlo, oz);
                zhi = fmaxf(zhi, oz);
            }
        }
        open = plates_decide<ENDS>(S, [&](int q) { return __fadd_rn(cz, L.oz[q]); }, L.K, cx, cy, sz, gx, gy, zlo, zhi, lend,
                             dmax, sl, pl, lane, want);
    }
    if (CALL) {
        if (__any_sync(kFull, (want & (!plates || (S.nplate & kLooseBit) ? ~0u : open)) != 0u)) {
            const WedgeRest r = wedge_rest_call(S, L, plates, cx, cy, cz, sz, gx, gy, want, open, lend, dmax, ex.x, ex.y,
                                                stack, ws.base, ws.base_k, cache);
            want = r.want;
            failed = r.failed;
            cache = r.cache;
        }
    } else {
        want = wedge_rest<COUNT>(S, L, plates, cx, cy, cz, sz, gx, gy, want, open, lend, dmax, ex, lane, stack, ws, sl,
                                 cache, failed, ctr);
    }
    return before & ~want;
}

// Irradiance of candidate i at this lane's patch for a vertical line lamp
// (L.wedge): the same entry as irradiance_entry, with one search per candidate
// instead of one per source.
template <bool COUNT, bool PLATES, bool MODES, bool CALL>
__device__ __forceinline__ float irradiance_wedge(const SceneView& S, const float* __restrict__ cand, int nc,
                                                  const LampDev& L, int i, int jb, int lane, int* stack,
                                                  const WedgeSmem& ws, uint32_t* __restrict__ vis, int nwords,
                                                  const PatchLane& P, int& cache, unsigned long long* ctr = nullptr) {
    const float cx = __ldg(&cand[3 * (size_t)i]), cy = __ldg(&cand[3 * (size_t)i + 1]),
                cz = __ldg(&cand[3 * (size_t)i + 2]);
    uint32_t want;
    float lend, dmax, gx, gy;
    float E;
    const uint32_t facing = wedge_setup_patch<MODES>(S, L, cx, cy, cz, P, lane, ws, want, lend, dmax, gx, gy, E);
    uint32_t failed;
    const PlateLane pl = PLATES && S.nplate != 0 ? plate_lane(S, jb, lane, P) : no_plate_lane();
    const uint32_t occl = wedge_search<COUNT, PLATES, MODES, CALL>(S, L, cx, cy, cz, P.s.z, gx, gy, want, lend, dmax, P.ex, pl, lane,
                                              stack, ws, cache, failed, ctr);
    const bool bad = (failed >> lane) & 1u;
    const uint32_t visible = bad ? 0u : (facing & ~occl);
    if (!__all_sync(kFull, visible == facing)) {   // some source is hidden: the sum of the others
        E = 0.f;
        for (int m = 0; m < L.K; ++m)
            if ((visible >> m) & 1u) E = __fadd_rn(E, ws.term[m * 32 + lane]);
    }
    if (vis) {   // lane m keeps source m's word (K <= 16), and the words leave in one store
        uint32_t word = __ballot_sync(kFull, P.valid);
        if (!__all_sync(kFull, !P.valid || visible == (1u << L.K) - 1u))
            for (int m = 0; m < L.K; ++m) {
                const uint32_t b = __ballot_sync(kFull, (visible >> m) & 1u);
                if (lane == m) word = b;
            }
        if (lane < L.K) vis[((size_t)lane * nc + i) * nwords + jb] = word;
    }
    return bad ? __int_as_float(0x7fffffff) : E;
}

}  // namespace
}  // namespace uvc
