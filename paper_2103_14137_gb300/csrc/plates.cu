// Plates: the flat, axis-aligned rectangles that the mesh tiles completely
// (walls, floors, the faces of furniture), found when a scene is built.  A
// room's few dozen plates hold most of its triangles, and one test decides
// what a segment does at a whole plate, so the searches try the plates first
// (traverse.cuh) and enter the hierarchy only for what they leave open.
//
// A plate is a set of triangles, connected by shared edges, that
//   - lie in one plane x = p, y = p or z = p, exactly (vertex coordinates are
//     compared, not rounded), and are wound the same way round in it,
//   - share every edge with exactly one other of them, run the other way
//     round, except for edges on the border of their common bounding rectangle.
// Then they cover the rectangle: added up as oriented areas, their boundary is
// what the unshared edges leave, all of it on the border, so every point inside
// is covered equally often, and at least once as no triangle has zero area.
// Sets whose triangles' areas add up to more than the rectangle's (covered more
// than once) are given up too: one triangle's place then holds no other.
// Triangles thinner than 1 : 64 (twice the area against the longest edge
// squared below 1/32) stay out: the searches' margins assume that the
// intersection test's rounding moves a hit by far less than a triangle.
//
//   edges    each directed edge into a hash table over (plane, winding, end
//            points); the second arrival is the mate: both triangles join
//            one set (lock-free union-find, smaller index as root)
//   stats    per set: bounding rectangle and triangle count
//   check    unshared edges must lie on their set's border
//   select   sets that pass and hold at least kPlateMinTris triangles
//   order    the larger plates first, those on the bounds last
//   mark     triangles outside every plate mark their ancestors in the
//            hierarchy, so that a search may skip subtrees of plates only
//            (none where there are no plates)
// All of it is linear in the triangles and latency-bound on rooms.
#include "uvc_internal.cuh"

namespace uvc {
namespace {

constexpr int kPlateMinTris = 4;     // smaller sets stay in the hierarchy
constexpr int kMaxProbes = 256;      // slots tried for an edge before its set is given up

__device__ __forceinline__ float axis_of(const float4& v, int a) { return a == 0 ? v.x : (a == 1 ? v.y : v.z); }

// A triangle's place in its plane: axis (-1: not flat or too thin), plane
// coordinate, winding, and the vertices' two other coordinates.
struct Flat {
    int axis;
    int ccw;
    float p;
    float u[3], v[3];
    float longest;   // squared length of the longest edge
    float area2;     // twice the area
};

__device__ __forceinline__ Flat flat_of(const float4* __restrict__ tri, int k) {
    const float4 a = tri[3 * (size_t)k], b = tri[3 * (size_t)k + 1], c = tri[3 * (size_t)k + 2];
    Flat f;
    f.axis = (a.x == b.x && a.x == c.x) ? 0 : (a.y == b.y && a.y == c.y) ? 1 : (a.z == b.z && a.z == c.z) ? 2 : -1;
    f.ccw = 0;
    if (f.axis < 0) return f;
    const int i = f.axis == 2 ? 0 : f.axis + 1, j = i == 2 ? 0 : i + 1;
    // + 0: the two zeros become one
    f.p = axis_of(a, f.axis) + 0.f;
    f.u[0] = axis_of(a, i) + 0.f; f.u[1] = axis_of(b, i) + 0.f; f.u[2] = axis_of(c, i) + 0.f;
    f.v[0] = axis_of(a, j) + 0.f; f.v[1] = axis_of(b, j) + 0.f; f.v[2] = axis_of(c, j) + 0.f;
    const float e1u = f.u[1] - f.u[0], e1v = f.v[1] - f.v[0], e2u = f.u[2] - f.u[0], e2v = f.v[2] - f.v[0];
    const float e3u = e2u - e1u, e3v = e2v - e1v;
    const float area2 = e1u * e2v - e1v * e2u;
    f.longest = fmaxf(e1u * e1u + e1v * e1v, fmaxf(e2u * e2u + e2v * e2v, e3u * e3u + e3v * e3v));
    if (!(fabsf(area2) * 32.f >= f.longest) || !(f.longest > 0.f)) f.axis = -1;
    f.ccw = area2 > 0.f;
    f.area2 = fabsf(area2);
    return f;
}

// Edge e of a flat triangle, from vertex e to vertex e + 1, with its end
// points in ascending order (`up`: that is its own direction).
struct Edge {
    float u0, v0, u1, v1;
    bool up;
};

__device__ __forceinline__ Edge edge_of(const Flat& f, int e) {
    const int n = e == 2 ? 0 : e + 1;
    const float au = f.u[e], av = f.v[e], bu = f.u[n], bv = f.v[n];
    Edge g;
    g.up = au < bu || (au == bu && av < bv);
    g.u0 = g.up ? au : bu; g.v0 = g.up ? av : bv;
    g.u1 = g.up ? bu : au; g.v1 = g.up ? bv : av;
    return g;
}

__device__ __forceinline__ uint32_t mix(uint32_t h, uint32_t x) {   // Murmur3's 32-bit block step (Appleby)
    x *= 0xcc9e2d51u;
    x = __funnelshift_l(x, x, 15);
    h ^= x * 0x1b873593u;
    return __funnelshift_l(h, h, 13) * 5u + 0xe6546b64u;
}

__device__ __forceinline__ uint32_t edge_hash(const Flat& f, const Edge& g) {
    uint32_t h = mix((uint32_t)(f.axis * 2 + f.ccw), __float_as_uint(f.p));
    h = mix(h, __float_as_uint(g.u0));
    h = mix(h, __float_as_uint(g.v0));
    h = mix(h, __float_as_uint(g.u1));
    h = mix(h, __float_as_uint(g.v1));
    h ^= h >> 16;
    h *= 0x85ebca6bu;
    return h ^ (h >> 13);
}

// Root of x's set.  Parents only ever move to smaller indices, so the walk
// ends; halving the path keeps it short.  Read through L1: an old parent is an
// ancestor all the same, and an old root is found out by the exchange in set_join
// (the floor of a floor of rooms is one set of some 80,000 triangles; with all of
// them reading its root from one L2 line k_plate_edges took 427 us there, now 294).
__device__ __forceinline__ int parent_of(const int* parent, int x) {
    int q;
    asm volatile("ld.global.ca.s32 %0, [%1];" : "=r"(q) : "l"(parent + x) : "memory");
    return q;
}

__device__ __forceinline__ int set_root(int* parent, int x) {
    int q = parent_of(parent, x);
    while (q != x) {
        const int g = parent_of(parent, q);
        if (g != q) parent[x] = g;
        x = q;
        q = g;
    }
    return x;
}

__device__ __forceinline__ void set_join(int* parent, int a, int b) {
    a = set_root(parent, a);
    b = set_root(parent, b);
    while (a != b) {   // each failed exchange gives a parent below a
        if (a < b) { const int t = a; a = b; b = t; }
        const int now = atomicCAS(&parent[a], a, b);
        if (now == a) return;
        a = set_root(parent, now);
    }
}

__global__ void k_plate_init(const float4* __restrict__ tri, int nt, int* __restrict__ parent,
                             unsigned* __restrict__ state) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nt) return;
    parent[k] = flat_of(tri, k).axis >= 0 ? k : -1;
    state[k] = 0u;
}

// state: bit e = edge e has its mate, kStateBad = an edge is shared wrongly, bit
// 4 + e = edge e is in the table and has been taken by a mate
constexpr unsigned kStateBad = 8u, kStateTaken = 16u;

__global__ void k_plate_edges(const float4* __restrict__ tri, int nt, int* __restrict__ table, uint32_t mask,
                              int* __restrict__ parent, unsigned* __restrict__ state) {
    const int id = blockIdx.x * blockDim.x + threadIdx.x;   // 4 k + e
    const int k = id >> 2, e = id & 3;
    if (k >= nt || e == 3 || parent_of(parent, k) < 0) return;
    const Flat f = flat_of(tri, k);
    const Edge g = edge_of(f, e);
    uint32_t h = edge_hash(f, g) & mask;
    for (int probe = 0; probe < kMaxProbes; ++probe, h = (h + 1) & mask) {
        int own = *reinterpret_cast<volatile int*>(table + h);
        if (own == -1) own = atomicCAS(table + h, -1, id);
        if (own == -1) return;   // first of its kind
        const Flat o = flat_of(tri, own >> 2);
        if (o.axis != f.axis || o.ccw != f.ccw || o.p != f.p) continue;
        const Edge q = edge_of(o, own & 3);
        if (q.u0 != g.u0 || q.v0 != g.v0 || q.u1 != g.u1 || q.v1 != g.v1) continue;
        const unsigned taken = kStateTaken << (own & 3);
        if (q.up != g.up && !(atomicOr(&state[own >> 2], taken) & taken)) {
            atomicOr(&state[k], 1u << e);
            atomicOr(&state[own >> 2], 1u << (own & 3));
            set_join(parent, k, own >> 2);
        } else {   // the same way round twice, or a third triangle
            atomicOr(&state[k], kStateBad);
            atomicOr(&state[own >> 2], kStateBad);
        }
        return;
    }
    atomicOr(&state[k], kStateBad);   // not placed
}

__device__ __forceinline__ unsigned ordered(float f) {
    const unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float unordered(unsigned u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// Per set (at its root): bounding rectangle, triangle count, kStateBad, longest
// edge (squared, as the bits of a positive float), twice the area (only looked
// at to tell one covering from two).  The
// triangles are in Morton order, so a warp holds few sets and adds each once.
__global__ void k_plate_stats(const float4* __restrict__ tri, int nt, int* __restrict__ parent,
                              const unsigned* __restrict__ state, uint2* __restrict__ lo, uint2* __restrict__ hi,
                              int2* __restrict__ cnt_bad, unsigned* __restrict__ len, float* __restrict__ area2) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned edge = 0u;
    float twice = 0.f;
    int root = -1;
    unsigned lu = ~0u, lv = ~0u, hu = 0u, hv = 0u;
    bool bad = false;
    if (k < nt && parent[k] >= 0) {
        root = set_root(parent, k);
        const Flat f = flat_of(tri, k);
        lu = ordered(fminf(f.u[0], fminf(f.u[1], f.u[2])));
        lv = ordered(fminf(f.v[0], fminf(f.v[1], f.v[2])));
        hu = ordered(fmaxf(f.u[0], fmaxf(f.u[1], f.u[2])));
        hv = ordered(fmaxf(f.v[0], fmaxf(f.v[1], f.v[2])));
        bad = (state[k] & kStateBad) != 0u;
        edge = __float_as_uint(f.longest);
        twice = f.area2;
    }
    unsigned todo = __ballot_sync(0xffffffffu, root >= 0);
    const int lane = threadIdx.x & 31;
    while (todo) {
        const int lead = __ffs(todo) - 1;
        const int r = __shfl_sync(0xffffffffu, root, lead);
        const bool in = root == r;
        const unsigned grp = __ballot_sync(0xffffffffu, in);
        const unsigned a = __reduce_min_sync(0xffffffffu, in ? lu : ~0u), b = __reduce_min_sync(0xffffffffu, in ? lv : ~0u);
        const unsigned c = __reduce_max_sync(0xffffffffu, in ? hu : 0u), d = __reduce_max_sync(0xffffffffu, in ? hv : 0u);
        const unsigned l = __reduce_max_sync(0xffffffffu, in ? edge : 0u);
        float sum = in ? twice : 0.f;
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        const bool any_bad = __any_sync(0xffffffffu, in && bad);
        if (lane == lead) {
            atomicMin(&lo[r].x, a);
            atomicMin(&lo[r].y, b);
            atomicMax(&hi[r].x, c);
            atomicMax(&hi[r].y, d);
            atomicMax(&len[r], l);
            atomicAdd(&area2[r], sum);
            atomicAdd(&cnt_bad[r].x, __popc(grp));
            if (any_bad) atomicOr(&cnt_bad[r].y, 1);
        }
        todo &= ~grp;
    }
}

__global__ void k_plate_check(const float4* __restrict__ tri, int nt, int* __restrict__ parent,
                              const unsigned* __restrict__ state, const uint2* __restrict__ lo,
                              const uint2* __restrict__ hi, int2* __restrict__ cnt_bad) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nt || parent[k] < 0 || (state[k] & 7u) == 7u) return;
    const int root = set_root(parent, k);
    const Flat f = flat_of(tri, k);
    const float ul = unordered(lo[root].x), vl = unordered(lo[root].y), uh = unordered(hi[root].x),
                vh = unordered(hi[root].y);
    for (int e = 0; e < 3; ++e) {
        if ((state[k] >> e) & 1u) continue;
        const Edge g = edge_of(f, e);
        const bool border = (g.u0 == ul && g.u1 == ul) || (g.u0 == uh && g.u1 == uh) || (g.v0 == vl && g.v1 == vl) ||
                            (g.v0 == vh && g.v1 == vh);
        if (!border) {
            atomicOr(&cnt_bad[root].y, 1);
            return;
        }
    }
}

// The plates, in any order; their number may pass kMaxPlates, and the scene
// then goes without.  plate_id: per root, or -1.
// box: the scene's bounds; inner: triangles of the plates inside them.
__global__ void k_plate_select(const float4* __restrict__ tri, int nt, const int* __restrict__ parent,
                               const uint2* __restrict__ lo, const uint2* __restrict__ hi,
                               const int2* __restrict__ cnt_bad, const unsigned* __restrict__ len,
                               const float* __restrict__ area2, float4* __restrict__ plates, int* __restrict__ plate_id,
                               const unsigned* __restrict__ box, int* __restrict__ nplate, int* __restrict__ inner) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nt) return;
    int id = -1;
    if (parent[k] == k && cnt_bad[k].x >= kPlateMinTris && !cnt_bad[k].y &&
        area2[k] < 3.f * (unordered(hi[k].x) - unordered(lo[k].x)) * (unordered(hi[k].y) - unordered(lo[k].y))) {
        id = atomicAdd(nplate, 1);
        if (id < kMaxPlates) {
            const Flat f = flat_of(tri, k);
            if (f.p > unordered(box[f.axis]) && f.p < unordered(box[3 + f.axis])) atomicAdd(inner, cnt_bad[k].x);
            const int i = f.axis == 2 ? 0 : f.axis + 1, j = i == 2 ? 0 : i + 1;
            float a[3], b[3];
            a[f.axis] = b[f.axis] = f.p;
            a[i] = unordered(lo[k].x); a[j] = unordered(lo[k].y);
            b[i] = unordered(hi[k].x); b[j] = unordered(hi[k].y);
            plates[2 * id] = make_float4(a[0], a[1], a[2], __int_as_float(f.axis));
            plates[2 * id + 1] = make_float4(b[0], b[1], b[2], sqrtf(__uint_as_float(len[k])));
        } else {
            id = -1;
        }
    }
    plate_id[k] = id;
}

// Orders the plates: the larger ones first, which block more and so end a
// search earlier, those on the sides of the scene's bounds, which block
// nothing, last.  No result depends on the order.  place_of: new place by the
// old.  One block counts the larger ones of each.
__global__ void __launch_bounds__(kMaxPlates) k_plate_order(float4* __restrict__ plates, const int* __restrict__ nplate,
                                                            const unsigned* __restrict__ box, int* __restrict__ place_of) {
    __shared__ float key[kMaxPlates];
    const int n = *nplate, p = threadIdx.x;
    if (n > kMaxPlates) {
        place_of[p] = -1;
        return;
    }
    float4 lo, hi;
    if (p < n) {
        lo = plates[2 * p];
        hi = plates[2 * p + 1];
        const int a = __float_as_int(lo.w);
        const float at = axis_of(lo, a), x = hi.x - lo.x, y = hi.y - lo.y, z = hi.z - lo.z;
        const bool inner = at > unordered(box[a]) && at < unordered(box[3 + a]);
        key[p] = inner ? (a == 0 ? y * z : (a == 1 ? x * z : x * y)) : -1.f;
    }
    __syncthreads();
    if (p < n) {
        const float mine = key[p];
        int rank = 0;
        for (int q = 0; q < n; ++q) rank += key[q] > mine || (key[q] == mine && q < p);
        place_of[p] = rank;
        plates[2 * rank] = lo;
        plates[2 * rank + 1] = hi;
    }
}

// place: each triangle's sorted position and plate (-1 = none) by its input
// index.  A triangle of no plate (loose) marks its leaf and every node above it.
__global__ void k_plate_mark(const float4* __restrict__ tri, int nt, int* __restrict__ parent,
                             const int* __restrict__ plate_id, const int* __restrict__ place_of,
                             const int* __restrict__ parent_leaf,
                             const int* __restrict__ parent_int, int2* __restrict__ place,
                             int* __restrict__ leaf_loose, int* __restrict__ node_loose, const int* __restrict__ nplate,
                             int* __restrict__ nloose) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (*nplate == 0) {   // nothing to look up or to skip: no marks, and the places are not read
        if (k < nt) leaf_loose[k] = 0;
        return;
    }
    int plate = 0;
    if (k < nt) {
        plate = parent[k] >= 0 ? plate_id[set_root(parent, k)] : -1;
        if (plate >= 0) plate = place_of[plate];
        place[__float_as_int(tri[3 * (size_t)k].w)] = make_int2(k, plate);
        leaf_loose[k] = plate < 0;
        if (plate < 0 && nt > 1)
            for (int p = parent_leaf[k]; p >= 0 && !*reinterpret_cast<volatile int*>(&node_loose[p]); p = parent_int[p])
                node_loose[p] = 1;
    }
    const unsigned out = __ballot_sync(0xffffffffu, k < nt && plate < 0);
    if (out && (threadIdx.x & 31) == 0) atomicAdd(nloose, __popc(out));
}

// Bit j of the flag words: patch j excludes a triangle of a plate that it does
// not itself lie in; such a patch takes no plate for an occluder (the search
// decides, which knows the excluded triangles).
__global__ void k_plate_patches(const float4* __restrict__ ps, const int2* __restrict__ pe, int np, int nt,
                                const int2* __restrict__ place, const float4* __restrict__ plates,
                                const int* __restrict__ nplate, uint32_t* __restrict__ flags) {
    if (*nplate == 0) return;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    bool flag = false;
    if (j < np) {
        const float4 s = ps[j];
        const int ex[2] = {pe[j].x, pe[j].y};
        for (int q = 0; q < 2; ++q) {
            const int id = ex[q] >= 0 && ex[q] < nt ? place[ex[q]].y : -1;
            if (id < 0) continue;
            const float4 lo = plates[2 * id];
            const int a = __float_as_int(lo.w);
            if (axis_of(s, a) != axis_of(lo, a)) flag = true;
        }
    }
    const uint32_t word = __ballot_sync(0xffffffffu, flag);
    if ((threadIdx.x & 31) == 0 && j < np) flags[j >> 5] = word;
}

int grid(int64_t n) { return (int)((n + 255) / 256); }

uint32_t table_slots(int64_t nt) {   // a power of two, at least 4 per triangle (of at most 3 edges)
    uint32_t n = 64;
    while ((int64_t)n < 4 * nt) n *= 2;
    return n;
}

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

// Bytes of find_plates' workspace.
size_t plates_work_bytes(int64_t nt) {
    return align256(sizeof(int) * (size_t)table_slots(nt)) + 5 * align256(sizeof(int) * (size_t)nt) +
           3 * align256(sizeof(int2) * (size_t)nt) + align256(sizeof(int) * kMaxPlates);
}

// Enqueues the search for the scene's plates (see above): sc->plates and the
// patch flags, counts[0] = plates found (may pass kMaxPlates), counts[1] =
// loose triangles, counts[2] = triangles of plates inside the scene's bounds
// (all zeroed by the caller), and the loose marks of leaves and binary nodes
// (node_loose zeroed by the caller).  box: the triangles' bounds, lo and hi, as
// ordered integers.
void find_plates(uvc_scene* sc, const int* parent_leaf, const int* parent_int, int* leaf_loose, int* node_loose,
                 const unsigned* box, int* counts, void* work, cudaStream_t stream) {
    const int nt = (int)sc->nt, np = (int)sc->np;
    const uint32_t slots = table_slots(nt);
    char* p = static_cast<char*>(work);
    auto take = [&](size_t n) { char* q = p; p += align256(n); return q; };
    int* table = reinterpret_cast<int*>(take(sizeof(int) * (size_t)slots));
    int* parent = reinterpret_cast<int*>(take(sizeof(int) * (size_t)nt));
    unsigned* state = reinterpret_cast<unsigned*>(take(sizeof(int) * (size_t)nt));
    int* plate_id = reinterpret_cast<int*>(take(sizeof(int) * (size_t)nt));
    uint2* lo = reinterpret_cast<uint2*>(take(sizeof(uint2) * (size_t)nt));
    uint2* hi = reinterpret_cast<uint2*>(take(sizeof(uint2) * (size_t)nt));
    int2* cnt_bad = reinterpret_cast<int2*>(take(sizeof(int2) * (size_t)nt));
    unsigned* len = reinterpret_cast<unsigned*>(take(sizeof(unsigned) * (size_t)nt));
    float* area2 = reinterpret_cast<float*>(take(sizeof(float) * (size_t)nt));
    int* place_of = reinterpret_cast<int*>(take(sizeof(int) * kMaxPlates));
    cudaMemsetAsync(table, 0xff, sizeof(int) * (size_t)slots, stream);
    cudaMemsetAsync(lo, 0xff, sizeof(uint2) * (size_t)nt, stream);
    cudaMemsetAsync(hi, 0, (char*)(area2 + nt) - (char*)hi, stream);   // hi, cnt_bad, len, area2
    k_plate_init<<<grid(nt), 256, 0, stream>>>(sc->tri, nt, parent, state);
    k_plate_edges<<<grid(4 * (int64_t)nt), 256, 0, stream>>>(sc->tri, nt, table, slots - 1, parent, state);
    k_plate_stats<<<grid(nt), 256, 0, stream>>>(sc->tri, nt, parent, state, lo, hi, cnt_bad, len, area2);
    k_plate_check<<<grid(nt), 256, 0, stream>>>(sc->tri, nt, parent, state, lo, hi, cnt_bad);
    k_plate_select<<<grid(nt), 256, 0, stream>>>(sc->tri, nt, parent, lo, hi, cnt_bad, len, area2, sc->plates, plate_id,
                                                 box, counts, counts + 2);
    k_plate_order<<<1, kMaxPlates, 0, stream>>>(sc->plates, counts, box, place_of);
    k_plate_mark<<<grid(nt), 256, 0, stream>>>(sc->tri, nt, parent, plate_id, place_of, parent_leaf, parent_int, sc->tri_place,
                                               leaf_loose, node_loose, counts, counts + 1);
    if (np > 0)
        k_plate_patches<<<grid(np), 256, 0, stream>>>(sc->patch_s, sc->patch_excl, np, nt, sc->tri_place, sc->plates, counts,
                                                      reinterpret_cast<uint32_t*>(sc->plates + 2 * kMaxPlates));
}

}  // namespace uvc
