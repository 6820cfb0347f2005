// Candidate features for the learned candidate proposal: per candidate lamp
// position c, the area-weighted histogram of distances from c to the patch
// points (64 log-spaced bins, 0.1 m to 25 m), the distance from c to the
// nearest triangle, and c's height.  No visibility is involved: the features
// cost one pass over the patches per candidate, a small fraction of the
// occlusion-tested matrix they help to avoid.
#include <cmath>

#include "uvc_internal.cuh"

namespace uvc {
namespace {

constexpr int kBins = 64;
// Probe-column kernels (k_col_max, k_mark_best, k_probe_lost): a block covers W
// columns x SL row slices, thread (slice, column) scans rows slice, slice + SL,
// ..., and the slices are combined by shuffles and in shared memory.  The shape
// follows the number of columns: up to a block of 8 per SM (a probe's few hundred)
// 128 slices keep the chain of rows short, up to eight such blocks 32 do, and wide
// matrices read 128 bytes a row.  Marks of 511 x 2,000, 5,000 x 2,000 and 60,000 x
// 2,000 (columns x rows), whole calls in us: 32 columns x 8 slices 42 / 43 / 117, 8
// x 128 for all 39 / 60 / 389, by this rule 37 / 37 / 120.
template <int W, int SL>
struct Columns {
    static constexpr int kW = W, kSlices = SL, kThreads = W * SL, kWarps = W * SL / 32;
    static_assert(W <= 32 && 32 % W == 0 && W * SL <= 1024, "columns of a block");
    __device__ static int column() { return (int)threadIdx.x % W; }
    __device__ static int slice() { return (int)threadIdx.x / W; }
    __device__ static int j() { return (int)blockIdx.x * W + column(); }
    // f(row, A[row][j]) for this slice's rows in order, kAhead loads at a time (rows
    // past the end give 0); ends after a batch of which f returned true for one.
    static constexpr int kAhead = W == 32 ? 4 : 8;
    template <class F>
    __device__ static void rows_until(const float* __restrict__ A, int nc, int64_t lda, int j, F f) {
        const float* p = A + (int64_t)slice() * lda + j;
        const int64_t step = (int64_t)SL * lda;
        bool done = false;
        for (int64_t i = slice(); i < nc && !done; i += kAhead * SL, p += kAhead * step) {
            float v[kAhead];
            const bool whole = i + (kAhead - 1) * SL < nc;
#pragma unroll
            for (int u = 0; u < kAhead; ++u) v[u] = whole || i + u * SL < nc ? __ldg(p + u * step) : 0.f;
#pragma unroll
            for (int u = 0; u < kAhead; ++u) done |= f((int)i + u * SL, v[u]);
        }
    }
    // All rows.  Wide matrices fill the chip with rows in flight as they are: a plain
    // loop (marks of 60,000 x 2,000 in 120 us, by batches of 8 152, of 4 136).
    template <class F>
    __device__ static void rows(const float* __restrict__ A, int nc, int64_t lda, int j, F f) {
        if constexpr (W == 32)
            for (int i = slice(); i < nc; i += SL) f(i, A[(int64_t)i * lda + j]);
        else
            rows_until(A, nc, lda, j, [&](int i, float v) { f(i, v); return false; });
    }
    // v of this column's slices put together by `op`, in its slice-0 thread
    template <class T, class Op>
    __device__ static T combine(T v, T (*part)[W], Op op) {
        for (int o = W; o < 32; o <<= 1) {
            T other = v;
            constexpr int kWords = sizeof(T) / 4;
            int* w = reinterpret_cast<int*>(&other);
#pragma unroll
            for (int q = 0; q < kWords; ++q) w[q] = __shfl_down_sync(0xffffffffu, w[q], o);
            v = op(v, other);
        }
        const int warp = (int)threadIdx.x >> 5;
        if (((int)threadIdx.x & 31) < W) part[warp][column()] = v;
        __syncthreads();
        if (slice() == 0)
            for (int q = 1; q < kWarps; ++q) v = op(v, part[q][column()]);
        return v;
    }
};
// f(shape) with the shape for np columns.
template <class F>
void with_columns(int64_t np, F f) {
    const int64_t sms = sm_count();
    if (np <= 8 * sms) f(Columns<8, 128>());
    else if (np <= 64 * sms) f(Columns<8, 32>());
    else f(Columns<32, 8>());
}

constexpr int kHistThreads = 256;

struct Edges {
    float e[kBins - 1];   // squared bin edges
};

// One block per candidate; each thread keeps its own 64 slots in shared
// memory (no atomics), the slots are then added in a fixed order.  The bin of
// a squared distance follows from its logarithm (the edges are log-spaced): the
// approximate one decides away from the edges, within kEdgeZone of one the exact
// edge does, so every patch falls where a search through the edges would put
// it.  That search, six dependent loads a pair, took 1.01 ms of 2,000 ward
// candidates x 98,132 patches.
constexpr float kEdgeZone = 1e-3f;   // in bins; the logarithm is good to 1e-5 of one
__global__ void __launch_bounds__(kHistThreads) k_feat_hist(const float4* __restrict__ ps, int np,
                                                             const float* __restrict__ area_total,
                                                             const float* __restrict__ cand, Edges E,
                                                             float bins_per_log2, float bin0,
                                                             float* __restrict__ feat, int64_t ldf) {
    extern __shared__ __align__(16) float slot[];   // [kBins][kHistThreads]
    __shared__ float edge[kBins + 1];   // lower edges (0 first, then E, infinity last)
    const int i = blockIdx.x;
    const int t = threadIdx.x;
    for (int b = t; b <= kBins; b += blockDim.x) edge[b] = b == 0 ? 0.f : (b == kBins ? __int_as_float(0x7f800000) : E.e[b - 1]);
    for (int b = 0; b < kBins; ++b) slot[b * kHistThreads + t] = 0.f;
    __syncthreads();
    const float cx = cand[3 * (size_t)i], cy = cand[3 * (size_t)i + 1], cz = cand[3 * (size_t)i + 2];
#pragma unroll 4
    for (int j = t; j < np; j += kHistThreads) {
        const float4 s = __ldg(&ps[j]);
        const float dx = s.x - cx, dy = s.y - cy, dz = s.z - cz;
        const float d2 = dx * dx + dy * dy + dz * dz;
        float lg;
        asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(lg) : "f"(d2));
        const float x = fminf(fmaxf(fmaf(lg, bins_per_log2, bin0), 0.f), (float)kBins - 0.5f);   // NaN: bin 0
        const float r = (x + 12582912.f) - 12582912.f;   // nearest edge (1.5 2^23: rounds to integers)
        int b = (int)r;
        if (x < r) --b;
        if (fabsf(x - r) < kEdgeZone) {
            const int n = (int)r;
            b = d2 >= edge[n] || n == 0 ? n : n - 1;
        }
        slot[b * kHistThreads + t] += s.w;
    }
    __syncthreads();
    const float tot = *area_total;
    if (t < kBins) {   // in thread order, four slots a load
        float sum = 0.f;
        const float4* q = reinterpret_cast<const float4*>(slot + t * kHistThreads);
#pragma unroll 8
        for (int k = 0; k < kHistThreads / 4; ++k) {
            const float4 v = q[k];
            sum += v.x;
            sum += v.y;
            sum += v.z;
            sum += v.w;
        }
        feat[i * ldf + t] = tot > 0.f ? sum / tot : 0.f;
    }
}

// Squared distance from p to triangle abc: the closest point is a vertex, a
// point of an edge or an interior point, decided by the signs of the
// barycentric-style dot products (Voronoi regions of the triangle).
__device__ float point_tri_dist2(float3 p, float3 a, float3 b, float3 c) {
    const float3 ab = make_float3(b.x - a.x, b.y - a.y, b.z - a.z), ac = make_float3(c.x - a.x, c.y - a.y, c.z - a.z);
    const float3 ap = make_float3(p.x - a.x, p.y - a.y, p.z - a.z);
    auto dot = [](float3 u, float3 v) { return u.x * v.x + u.y * v.y + u.z * v.z; };
    auto d2of = [&](float3 q) {
        const float x = p.x - q.x, y = p.y - q.y, z = p.z - q.z;
        return x * x + y * y + z * z;
    };
    const float d1 = dot(ab, ap), d2 = dot(ac, ap);
    if (d1 <= 0.f && d2 <= 0.f) return d2of(a);
    const float3 bp = make_float3(p.x - b.x, p.y - b.y, p.z - b.z);
    const float d3 = dot(ab, bp), d4 = dot(ac, bp);
    if (d3 >= 0.f && d4 <= d3) return d2of(b);
    const float3 cp = make_float3(p.x - c.x, p.y - c.y, p.z - c.z);
    const float d5 = dot(ab, cp), d6 = dot(ac, cp);
    if (d6 >= 0.f && d5 <= d6) return d2of(c);
    const float vc = d1 * d4 - d3 * d2;
    if (vc <= 0.f && d1 >= 0.f && d3 <= 0.f) {
        const float v = d1 / (d1 - d3);
        return d2of(make_float3(a.x + v * ab.x, a.y + v * ab.y, a.z + v * ab.z));
    }
    const float vb = d5 * d2 - d1 * d6;
    if (vb <= 0.f && d2 >= 0.f && d6 <= 0.f) {
        const float w = d2 / (d2 - d6);
        return d2of(make_float3(a.x + w * ac.x, a.y + w * ac.y, a.z + w * ac.z));
    }
    const float va = d3 * d6 - d5 * d4;
    if (va <= 0.f && (d4 - d3) >= 0.f && (d5 - d6) >= 0.f) {
        const float w = (d4 - d3) / ((d4 - d3) + (d5 - d6));
        return d2of(make_float3(b.x + w * (c.x - b.x), b.y + w * (c.y - b.y), b.z + w * (c.z - b.z)));
    }
    const float den = 1.f / (va + vb + vc);
    const float v = vb * den, w = vc * den;
    return d2of(make_float3(a.x + ab.x * v + ac.x * w, a.y + ab.y * v + ac.y * w, a.z + ab.z * v + ac.z * w));
}

__device__ __forceinline__ float box_d2(float3 p, float lx, float ly, float lz, float hx, float hy, float hz) {
    const float dx = fmaxf(fmaxf(lx - p.x, p.x - hx), 0.f);
    const float dy = fmaxf(fmaxf(ly - p.y, p.y - hy), 0.f);
    const float dz = fmaxf(fmaxf(lz - p.z, p.z - hz), 0.f);
    return dx * dx + dy * dy + dz * dz;
}

// Nearest triangle, one warp per candidate: up to 8 nodes of the four-wide tree
// leave the warp's list at a time, each lane takes one child of one of them,
// triangles are measured where they turn up, and children no nearer than the
// best so far are dropped (before they are listed and when they are taken).  A
// thread per candidate walked the binary tree through some sixty dependent
// loads: 73 us for 2,000 candidates, with 63 warps on the chip; now 26 us.
// A list that would overflow sends the candidate through that walk.
constexpr int kClearWarps = 4, kClearList = 256;

__device__ float nearest_walk(const Node* __restrict__ nodes, const float4* __restrict__ tri, int nt, float3 p) {
    float best = 3.0e38f;
    int stack[128];
    int top = 0;
    if (nt > 1) stack[top++] = 0;
    else if (nt == 1) stack[top++] = ~0;
    int guard = 0;
    while (top > 0 && ++guard < 4 * nt + 64) {
        const int ref = stack[--top];
        if (ref < 0) {
            const int k = ~ref;
            const float4 a = tri[3 * k], b = tri[3 * k + 1], c = tri[3 * k + 2];
            best = fminf(best, point_tri_dist2(p, make_float3(a.x, a.y, a.z), make_float3(b.x, b.y, b.z),
                                               make_float3(c.x, c.y, c.z)));
            continue;
        }
        const Node nd = nodes[ref];
        const float dL = box_d2(p, nd.x.x, nd.y.x, nd.z.x, nd.x.z, nd.y.z, nd.z.z);
        const float dR = box_d2(p, nd.x.y, nd.y.y, nd.z.y, nd.x.w, nd.y.w, nd.z.w);
        // never taken: the stack holds at most one pending sibling per level plus
        // the two children just pushed, and candidate_features refuses trees
        // deeper than 126
        if (top + 2 > 128) break;
        const bool lfirst = dL <= dR;
        if ((lfirst ? dR : dL) < best) stack[top++] = lfirst ? nd.r.y : nd.r.x;
        if ((lfirst ? dL : dR) < best) stack[top++] = lfirst ? nd.r.x : nd.r.y;
    }
    return best;
}

__global__ void __launch_bounds__(32 * kClearWarps) k_feat_clear(const Node4* __restrict__ nodes4,
                                                                 const Node* __restrict__ nodes,
                                                                 const float4* __restrict__ tri, int nt,
                                                                 const float* __restrict__ cand, int nc,
                                                                 float* __restrict__ feat, int64_t ldf) {
    __shared__ int list[kClearWarps][kClearList];
    __shared__ float dist[kClearWarps][kClearList];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = blockIdx.x * kClearWarps + warp;
    if (i >= nc) return;
    const float3 p = make_float3(cand[3 * (size_t)i], cand[3 * (size_t)i + 1], cand[3 * (size_t)i + 2]);
    float best = 3.0e38f;   // the same in every lane
    bool over = nt < 2;
    int top = over ? 0 : 1;
    if (lane == 0) {
        list[warp][0] = 0;
        dist[warp][0] = 0.f;
    }
    __syncwarp();
    for (int guard = 0; top > 0 && guard < 4 * nt + 64; ++guard) {
        const int n = min(min(8, top), (kClearList - top) / 3);
        if (n < 1) {
            over = true;
            break;
        }
        const int slot = lane >> 2, c = lane & 3;
        int ref = kEmptyChild;
        float d = 3.0e38f;
        if (slot < n && dist[warp][top - 1 - slot] < best) {
            const Node4* nd = nodes4 + list[warp][top - 1 - slot];
            ref = __ldg(reinterpret_cast<const int*>(&nd->r) + c);
            const float* q = reinterpret_cast<const float*>(nd) + (c >> 1) * 12 + (c & 1);
            d = box_d2(p, __ldg(q), __ldg(q + 4), __ldg(q + 8), __ldg(q + 2), __ldg(q + 6), __ldg(q + 10));
        }
        __syncwarp();   // the popped entries are read
        top -= n;
        float t = 3.0e38f;
        if (ref < 0 && d < best) {
            const float4 a = __ldg(&tri[3 * (size_t)~ref]), b = __ldg(&tri[3 * (size_t)~ref + 1]), e = __ldg(&tri[3 * (size_t)~ref + 2]);
            t = point_tri_dist2(p, make_float3(a.x, a.y, a.z), make_float3(b.x, b.y, b.z), make_float3(e.x, e.y, e.z));
        }
        // distances are not negative: their bits order them (NaN from a NaN candidate stays out)
        best = fminf(best, __uint_as_float(__reduce_min_sync(0xffffffffu, t >= 0.f ? __float_as_uint(t) : 0x7f61b1e6u)));
        // the nearest of the new children goes on top
        const bool in = ref >= 0 && ref != kEmptyChild && d < best;
        const unsigned m = __ballot_sync(0xffffffffu, in);
        const unsigned near = __reduce_min_sync(0xffffffffu, in ? __float_as_uint(d) : 0xffffffffu);
        const unsigned w = __ballot_sync(0xffffffffu, in && __float_as_uint(d) == near);
        const int win = __ffs(w) - 1, cnt = __popc(m);
        if (in) {
            int at = __popc(m & ((1u << lane) - 1u));
            if (lane == win) at = cnt - 1;
            else if (lane > win) --at;
            list[warp][top + at] = ref;
            dist[warp][top + at] = d;
        }
        top += cnt;
        __syncwarp();
    }
    if (lane == 0) {
        if (over) best = nearest_walk(nodes, tri, nt, p);
        feat[i * ldf + kBins] = nt > 0 ? sqrtf(best) : 3.0e38f;
        feat[i * ldf + kBins + 1] = p.z;
    }
}

constexpr int kSelectMax = 16384;
constexpr int kSelectThreads = 1024;

// Order-preserving map of a float score to an unsigned key (NaN lowest).
__device__ __forceinline__ uint32_t score_key(float v) {
    if (v != v) return 0u;
    const uint32_t u = __float_as_uint(v);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// The k best of n scores (higher first, ties to the lower index), written in
// ascending index order.  The k-th largest key is found by four passes over
// its bytes (a histogram of the keys that share the bytes found so far, its
// suffix sums by one warp); the scores above it are all taken, those equal to it
// in index order as far as they are needed, and a block-wide scan writes them.
// (A bitonic sort of all keys took 25 us for 2,000 scores, this 9 us.)
__global__ void __launch_bounds__(kSelectThreads) k_select_top(const float* __restrict__ score, int n, int k,
                                                                const float* __restrict__ cand,
                                                                float* __restrict__ out_cand,
                                                                int32_t* __restrict__ out_idx) {
    extern __shared__ uint32_t key[];   // [n], then flags [n] as bytes
    __shared__ int warp_tot[kSelectThreads / 32];
    __shared__ unsigned hist[256];
    __shared__ uint32_t sh_prefix;
    __shared__ int sh_want;
    unsigned char* flag = reinterpret_cast<unsigned char*>(key + n);
    const int t = threadIdx.x;
    for (int i = t; i < n; i += blockDim.x) key[i] = score_key(score[i]);
    uint32_t prefix = 0u;
    int want = k;   // keys still to be taken among those that share the prefix
    for (int shift = 24; shift >= 0; shift -= 8) {
        if (t < 256) hist[t] = 0u;
        __syncthreads();
        for (int i = t; i < n; i += blockDim.x) {
            const uint32_t v = key[i];
            if (shift == 24 || (v >> (shift + 8)) == prefix) atomicAdd(&hist[(v >> shift) & 255u], 1u);
        }
        __syncthreads();
        if (t < 32) {   // lane l: bytes 255 - 8 l down to 248 - 8 l
            unsigned c[8], sum = 0u;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                c[q] = hist[255 - 8 * t - q];
                sum += c[q];
            }
            unsigned inc = sum;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned v = __shfl_up_sync(0xffffffffu, inc, o);
                if (t >= o) inc += v;
            }
            unsigned above = inc - sum;   // keys with a larger byte than this lane's
            if (above < (unsigned)want && inc >= (unsigned)want)
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    if (above < (unsigned)want && above + c[q] >= (unsigned)want) {
                        sh_prefix = (prefix << 8) | (uint32_t)(255 - 8 * t - q);
                        sh_want = want - (int)above;
                    }
                    above += c[q];
                }
        }
        __syncthreads();
        prefix = sh_prefix;
        want = sh_want;
    }
    // each thread's run of consecutive indices: how many equal keys come before it
    {
        const int per = (n + blockDim.x - 1) / blockDim.x, lo = min(n, t * per), hi = min(n, lo + per);
        int eq = 0;
        for (int i = lo; i < hi; ++i) eq += key[i] == prefix;
        int inc = eq;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if ((t & 31) >= o) inc += v;
        }
        if ((t & 31) == 31) warp_tot[t >> 5] = inc;
        __syncthreads();
        int before = inc - eq;
        for (int q = 0; q < (t >> 5); ++q) before += warp_tot[q];
        for (int i = lo; i < hi; ++i) {
            flag[i] = key[i] > prefix || (key[i] == prefix && before < want);
            before += key[i] == prefix;
        }
        __syncthreads();
    }
    // each thread owns a run of consecutive indices
    const int per = (n + blockDim.x - 1) / blockDim.x;
    const int lo = min(n, t * per), hi = min(n, lo + per);
    int cnt = 0;
    for (int i = lo; i < hi; ++i) cnt += flag[i];
    const int lane = t & 31, w = t >> 5;
    int inc = cnt;
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    if (lane == 31) warp_tot[w] = inc;
    __syncthreads();
    int base = 0;
    for (int q = 0; q < w; ++q) base += warp_tot[q];
    int pos = base + inc - cnt;
    for (int i = lo; i < hi; ++i)
        if (flag[i]) {
            if (out_idx) out_idx[pos] = i;
            if (out_cand) {
                out_cand[3 * (size_t)pos] = cand[3 * (size_t)i];
                out_cand[3 * (size_t)pos + 1] = cand[3 * (size_t)i + 1];
                out_cand[3 * (size_t)pos + 2] = cand[3 * (size_t)i + 2];
            }
            ++pos;
        }
}

// Per probe patch j: its area if some candidate lights it (A[i][j] > 0) but
// none of the selected ones does, else 0.  Four rows at a time until one is lit.
template <class C>
__global__ void __launch_bounds__(C::kThreads) k_probe_lost(const float* __restrict__ A, int nc, int64_t lda, int np,
                                                            const int32_t* __restrict__ idx, int k,
                                                            const float* __restrict__ area, float* __restrict__ lost) {
    __shared__ int part[C::kWarps][C::kW];
    const int j = C::j(), sl = C::slice();
    bool full = false, red = false;
    if (j < np) {
        C::rows_until(A, nc, lda, j, [&](int, float v) { return full |= v > 0.f; });
        for (int r = sl; r < k && !red; r += 4 * C::kSlices) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = r + u * C::kSlices < k ? idx[r + u * C::kSlices] : -1;
                if (i >= 0 && i < nc) red |= A[(int64_t)i * lda + j] > 0.f;   // rows out of range are ignored
            }
        }
    }
    const int m = C::combine((int)full | (int)red << 1, part, [](int x, int y) { return x | y; });
    if (sl == 0 && j < np) lost[j] = m == 1 ? area[j] : 0.f;
}

// out = sum(lost) / sum(area), compensated sums in a fixed order (one block).
__global__ void k_probe_total(const float* __restrict__ lost, const float* __restrict__ area, int np,
                              float* __restrict__ out) {
    __shared__ float sl[256], sa[256];
    float l = 0.f, cl = 0.f, a = 0.f, ca = 0.f;
    for (int j = threadIdx.x; j < np; j += 256) {
        const float yl = lost[j] - cl, tl = l + yl;
        cl = (tl - l) - yl;
        l = tl;
        const float ya = area[j] - ca, ta = a + ya;
        ca = (ta - a) - ya;
        a = ta;
    }
    sl[threadIdx.x] = l;
    sa[threadIdx.x] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        float L = 0.f, cL = 0.f, S = 0.f, cS = 0.f;
        for (int q = 0; q < 256; ++q) {
            const float yl = sl[q] - cL, tl = L + yl;
            cL = (tl - L) - yl;
            L = tl;
            const float ya = sa[q] - cS, ta = S + ya;
            cS = (ta - S) - ya;
            S = ta;
        }
        *out = S > 0.f ? L / S : 0.f;
    }
}

constexpr int kHardBins = 8, kEffBins = 6, kProbeFeat = kHardBins * kEffBins;
constexpr int kProbeWarps = 4;

// E*_j = max_i A[i][j].
template <class C>
__global__ void __launch_bounds__(C::kThreads) k_col_max(const float* __restrict__ A, int nc, int64_t lda, int np,
                                                         float* __restrict__ emax) {
    __shared__ float part[C::kWarps][C::kW];
    const int j = C::j();
    float m = 0.f;
    if (j < np) C::rows(A, nc, lda, j, [&](int, float v) { m = fmaxf(m, v); });
    m = C::combine(m, part, [](float x, float y) { return fmaxf(x, y); });
    if (C::slice() == 0 && j < np) emax[j] = m;
}

// Lit-area-weighted mean of E* (compensated sums, fixed order, one block),
// then each lit patch's hardness bin floor(log2(E*_j / mean)) + 4 clamped to
// [0, 7] (-1 for an unlit patch); stats = (sum a E*, sum a) over lit patches.
__global__ void k_probe_bins(const float* __restrict__ emax, const float* __restrict__ area, int np,
                             float* __restrict__ stats, signed char* __restrict__ hb) {
    __shared__ float s0[256], s1[256];
    __shared__ float mean_sh;
    float a0 = 0.f, c0 = 0.f, a1 = 0.f, c1 = 0.f;
    for (int j = threadIdx.x; j < np; j += 256) {
        const float e = emax[j];
        if (!(e > 0.f)) continue;
        const float y0 = area[j] * e - c0, t0 = a0 + y0;
        c0 = (t0 - a0) - y0;
        a0 = t0;
        const float y1 = area[j] - c1, t1 = a1 + y1;
        c1 = (t1 - a1) - y1;
        a1 = t1;
    }
    s0[threadIdx.x] = a0;
    s1[threadIdx.x] = a1;
    __syncthreads();
    if (threadIdx.x == 0) {
        float A0 = 0.f, C0 = 0.f, A1 = 0.f, C1 = 0.f;
        for (int q = 0; q < 256; ++q) {
            const float y0 = s0[q] - C0, t0 = A0 + y0;
            C0 = (t0 - A0) - y0;
            A0 = t0;
            const float y1 = s1[q] - C1, t1 = A1 + y1;
            C1 = (t1 - A1) - y1;
            A1 = t1;
        }
        stats[0] = A0;
        stats[1] = A1;
        mean_sh = A1 > 0.f ? A0 / A1 : 0.f;
    }
    __syncthreads();
    const float mean = mean_sh;
    for (int j = threadIdx.x; j < np; j += 256) {
        const float e = emax[j];
        if (!(e > 0.f) || !(mean > 0.f)) {
            hb[j] = -1;
            continue;
        }
        int ex;
        frexpf(e / mean, &ex);   // e / mean = f 2^ex, f in [0.5, 1): floor(log2) = ex - 1
        hb[j] = (signed char)min(kHardBins - 1, max(0, ex - 1 + 4));
    }
}

// One warp per candidate: area of the lit probe patches by (hardness bin,
// efficiency bin of A[i][j] / E*_j), over the lit area.  Per-lane slots in
// shared memory, lanes added in a fixed order.
__global__ void __launch_bounds__(kProbeWarps * 32) k_probe_feat(const float* __restrict__ A, int nc, int64_t lda,
                                                                  int np, const float* __restrict__ emax,
                                                                  const signed char* __restrict__ hb,
                                                                  const float* __restrict__ area,
                                                                  const float* __restrict__ stats,
                                                                  float* __restrict__ feat, int64_t ldf) {
    __shared__ float slot[kProbeWarps][kProbeFeat][32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * kProbeWarps + w;
    if (i >= nc) return;
    for (int b = 0; b < kProbeFeat; ++b) slot[w][b][lane] = 0.f;
    const float* row = A + (int64_t)i * lda;
    for (int j = lane; j < np; j += 32) {
        const int h = hb[j];
        if (h < 0) continue;
        const float e = row[j] / emax[j];
        const int eb = e < 0.5f ? 0 : e < 0.7f ? 1 : e < 0.8f ? 2 : e < 0.9f ? 3 : e < 0.95f ? 4 : 5;
        slot[w][h * kEffBins + eb][lane] += area[j];
    }
    __syncwarp();
    const float lit = stats[1];
    for (int b = lane; b < kProbeFeat; b += 32) {
        float sum = 0.f;
        for (int q = 0; q < 32; ++q) sum += slot[w][b][q];
        feat[(int64_t)i * ldf + b] = lit > 0.f ? sum / lit : 0.f;
    }
}

// For each lit probe patch j, score[argmax_i A[i][j]] = value (the lowest
// index among equal maxima); with rare > 0, also every candidate that lights
// a patch lit by at most `rare` candidates.  Several patches may write the
// same candidate with the same value.
struct Best {
    float v;
    int i, lit;   // row of the maximum (-1: none above 0), rows above 0
};
template <class C>
__global__ void __launch_bounds__(C::kThreads) k_mark_best(const float* __restrict__ A, int nc, int64_t lda, int np,
                                                           float* __restrict__ score, float value, int rare) {
    __shared__ Best part[C::kWarps][C::kW];
    __shared__ int lit[C::kW];
    const int j = C::j(), sl = C::slice();
    Best b{0.f, -1, 0};
    if (j < np)
        C::rows(A, nc, lda, j, [&](int i, float v) {
            b.lit += v > 0.f;
            if (v > b.v) {        // rows ascend within a slice: the first maximum is kept
                b.v = v;
                b.i = i;
            }
        });
    b = C::combine(b, part, [](Best x, Best y) {
        const bool other = y.i >= 0 && (y.v > x.v || (y.v == x.v && (x.i < 0 || y.i < x.i)));
        return Best{other ? y.v : x.v, other ? y.i : x.i, x.lit + y.lit};
    });
    if (sl == 0) {
        lit[C::column()] = b.lit;
        if (j < np && b.i >= 0) score[b.i] = value;
    }
    if (rare <= 0) return;
    __syncthreads();
    const int total = lit[C::column()];
    if (j < np && total > 0 && total <= rare)
        for (int i = sl; i < nc; i += C::kSlices)
            if (A[(int64_t)i * lda + j] > 0.f) score[i] = value;
}

// score[winner of each group of `group` consecutive candidates] += bonus;
// the winner is the highest score of the group (lowest index among equals,
// NaN lowest).  One thread per group.
__global__ void k_group_boost(float* __restrict__ score, int n, int group, float bonus) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    const int i0 = g * group;
    if (i0 >= n) return;
    const int i1 = min(n, i0 + group);
    int best = i0;
    uint32_t bk = score_key(score[i0]);
    for (int i = i0 + 1; i < i1; ++i) {
        const uint32_t k = score_key(score[i]);
        if (k > bk) {
            bk = k;
            best = i;
        }
    }
    score[best] = score[best] + bonus;
}

}  // namespace

int group_boost(float* score, int64_t n, int group, float bonus, cudaStream_t stream) {
    const int64_t ng = (n + group - 1) / group;
    if (ng > 0) k_group_boost<<<(int)((ng + 255) / 256), 256, 0, stream>>>(score, (int)n, group, bonus);
    return status_from_cuda(cudaGetLastError());
}

int mark_best(const float* A, int64_t nc, int64_t lda, int64_t np, float* score, float value, int rare,
              cudaStream_t stream) {
    if (np > 0 && nc > 0) {
        with_columns(np, [&](auto shape) {
            using C = decltype(shape);
            k_mark_best<C><<<(int)((np + C::kW - 1) / C::kW), C::kThreads, 0, stream>>>(A, (int)nc, lda, (int)np, score, value, rare);
        });
    }
    return status_from_cuda(cudaGetLastError());
}

int probe_features(const float* A, int64_t nc, int64_t lda, int64_t np, const float* area, float* work,
                   float* feat, int64_t ldf, cudaStream_t stream) {
    if (nc == 0) return UVC_OK;
    float* emax = work;
    float* stats = work + np;
    signed char* hb = reinterpret_cast<signed char*>(work + np + 4);
    if (np > 0) {
        with_columns(np, [&](auto shape) {
            using C = decltype(shape);
            k_col_max<C><<<(int)((np + C::kW - 1) / C::kW), C::kThreads, 0, stream>>>(A, (int)nc, lda, (int)np, emax);
        });
    }
    k_probe_bins<<<1, 256, 0, stream>>>(emax, area, (int)np, stats, hb);
    k_probe_feat<<<(int)((nc + kProbeWarps - 1) / kProbeWarps), kProbeWarps * 32, 0, stream>>>(
        A, (int)nc, lda, (int)np, emax, hb, area, stats, feat, ldf);
    return status_from_cuda(cudaGetLastError());
}

int probe_lost(const float* A, int64_t nc, int64_t lda, int64_t np, const int32_t* idx, int64_t k,
               const float* area, float* lost, float* out, cudaStream_t stream) {
    if (np > 0) {
        with_columns(np, [&](auto shape) {
            using C = decltype(shape);
            k_probe_lost<C><<<(int)((np + C::kW - 1) / C::kW), C::kThreads, 0, stream>>>(A, (int)nc, lda, (int)np, idx, (int)k, area, lost);
        });
    }
    k_probe_total<<<1, 256, 0, stream>>>(lost, area, (int)np, out);
    return status_from_cuda(cudaGetLastError());
}

int select_top(const float* score, int64_t n, int64_t k, const float* cand, float* out_cand, int32_t* out_idx,
               cudaStream_t stream) {
    if (n < 0 || n > kSelectMax || k < 0 || k > n) return UVC_E_INVAL;
    if (k == 0) return UVC_OK;
    const size_t smem = (sizeof(uint32_t) + 1) * (size_t)n;
    static const cudaError_t attr =
        cudaFuncSetAttribute(k_select_top, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)((sizeof(uint32_t) + 1) * kSelectMax));
    if (attr != cudaSuccess) return status_from_cuda(attr);
    k_select_top<<<1, kSelectThreads, smem, stream>>>(score, (int)n, (int)k, cand, out_cand, out_idx);
    return status_from_cuda(cudaGetLastError());
}

int candidate_features(const uvc_scene* sc, const float* cand, int64_t nc, float* feat, int64_t ldf,
                       cudaStream_t stream) {
    if (nc == 0) return UVC_OK;
    if (sc->depth > 126) return UVC_E_STACK;   // k_feat_clear's fixed stack of 128 entries
    Edges E;
    for (int b = 1; b < kBins; ++b) {
        const double e = 0.1 * std::pow(250.0, (double)b / kBins);
        E.e[b - 1] = (float)(e * e);
    }
    static const cudaError_t attr = cudaFuncSetAttribute(k_feat_hist, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                         (int)(sizeof(float) * kBins * kHistThreads));
    if (attr != cudaSuccess) return status_from_cuda(attr);
    k_feat_hist<<<(int)nc, kHistThreads, sizeof(float) * kBins * kHistThreads, stream>>>(
        sc->patch_s, (int)sc->np, sc->area_total, cand, E, (float)(kBins / (2.0 * std::log2(250.0))),
        (float)(-2.0 * std::log2(0.1) * kBins / (2.0 * std::log2(250.0))), feat, ldf);
    k_feat_clear<<<(int)((nc + kClearWarps - 1) / kClearWarps), 32 * kClearWarps, 0, stream>>>(
        sc->nodes4, sc->nodes, sc->tri, (int)sc->nt, cand, (int)nc, feat, ldf);
    return status_from_cuda(cudaGetLastError());
}

}  // namespace uvc
