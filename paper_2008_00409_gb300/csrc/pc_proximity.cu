// Proximity query feeding the one-sided thickness contact model: every (vertex p,
// triangle t) pair whose distance at the current positions is below the contact
// thickness delta, t touching neither p nor a mesh-edge neighbour of p, with the
// barycentric weights of the point of t closest to p. It is the proximity step in front
// of the implicit integrator (Sec. 2.5, Eq. 3); the paper's own collision handling
// (spatial hashing, continuous collision detection, Sec. 4) is not reproduced.
//
// Uniform grid, rebuilt per call: the cell size is the largest triangle bounding box
// grown by delta (so every grown box covers at most 2 x 2 x 2 cells); each triangle is
// listed under every cell its grown box overlaps, the list is put in cell order by the
// stable radix sort (triangles of a cell stay in index order), and each vertex tests the
// triangles listed under its own cell: a vertex within delta of a triangle lies in that
// triangle's grown box, hence in one of its cells. A pass over the vertices counts each
// one's pairs and remembers the first PX_HITS of them, a scan gives their places, and a
// second pass writes them: ordered by vertex, then by triangle, without atomics.
//
// Cells are numbered inside the boxes' own extent, so that the sort needs the bits of that
// many cells (17 for three 301 x 301 sheets: 3 passes) and not of 3 packed 21-bit
// coordinates (8 passes, 400 of the query's 1,130 us), and a vertex finds its cell's list
// in a table instead of by binary search. A vertex meets about 55 triangles in its cell;
// the grown box of each (32 bytes, kept per triangle) rejects most before the ring and the
// distance are looked at, and only the first pass looks (both did: 320 us each; the whole query
// now takes 442 us). Bound by the latency of those gathers: a thread tests the boxes of up to
// 32 triangles, PX_BATCH in flight, before it looks at any of those it is left with (triangle
// by triangle, with the lanes' hits at different places of their lists: 500 us).
//
// The region of the closest point (Voronoi classification of a point against a
// triangle, Ericson 2005, Sec. 5.1.5) and the test d^2 < delta^2 are decided in FP32
// with one rounding per operation in a fixed order (the _rn intrinsics keep the compiler
// from contracting into fused multiply-adds), so the pairs are reproducible bit for bit.
#include <algorithm>
#include <cstring>

#include "pc_internal.cuh"

#define PX_CELLS_PER_TRI 8
#define PX_COORD_BIAS (1 << 20)  // cell coordinates must lie in [-2^20, 2^20)
#define PX_HITS 16               // pairs of a vertex remembered from the counting pass

// The numbered cells: first coordinates, extents (nx, ny), and how many there are.
struct PxGrid {
    int x0, y0, z0;
    int64_t nx, ny;
    uint64_t n;  // up to 2^63
};

__device__ __forceinline__ float3 px_ld(const float *x, int i)
{
    return make_float3(x[3ll * i], x[3ll * i + 1], x[3ll * i + 2]);
}
__device__ __forceinline__ float3 px_sub(float3 a, float3 b)
{
    return make_float3(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y), __fsub_rn(a.z, b.z));
}
__device__ __forceinline__ float px_dot(float3 u, float3 v)
{
    return __fadd_rn(__fadd_rn(__fmul_rn(u.x, v.x), __fmul_rn(u.y, v.y)), __fmul_rn(u.z, v.z));
}

// Weights (wa, wb, wc) of the point of (a, b, c) closest to p; returns the squared
// distance. Regions in priority order: vertex a, vertex b, edge ab, vertex c, edge ac,
// edge bc, a degenerate triangle (treated as vertex a), the face.
__device__ float px_closest(float3 p, float3 a, float3 b, float3 c, float &wa, float &wb, float &wc)
{
    const float3 ab = px_sub(b, a), ac = px_sub(c, a), ap = px_sub(p, a);
    const float d1 = px_dot(ab, ap), d2 = px_dot(ac, ap);
    const float3 bp = px_sub(p, b);
    const float d3 = px_dot(ab, bp), d4 = px_dot(ac, bp);
    const float3 cp = px_sub(p, c);
    const float d5 = px_dot(ab, cp), d6 = px_dot(ac, cp);
    const float vc = __fsub_rn(__fmul_rn(d1, d4), __fmul_rn(d3, d2));
    const float vb = __fsub_rn(__fmul_rn(d5, d2), __fmul_rn(d1, d6));
    const float va = __fsub_rn(__fmul_rn(d3, d6), __fmul_rn(d5, d4));
    const float e43 = __fsub_rn(d4, d3), e56 = __fsub_rn(d5, d6);
    const float s = __fadd_rn(__fadd_rn(va, vb), vc);
    if (d1 <= 0.f && d2 <= 0.f) { wb = 0.f; wc = 0.f; }
    else if (d3 >= 0.f && d4 <= d3) { wb = 1.f; wc = 0.f; }
    else if (vc <= 0.f && d1 >= 0.f && d3 <= 0.f) { wb = __fdiv_rn(d1, __fsub_rn(d1, d3)); wc = 0.f; }
    else if (d6 >= 0.f && d5 <= d6) { wb = 0.f; wc = 1.f; }
    else if (vb <= 0.f && d2 >= 0.f && d6 <= 0.f) { wb = 0.f; wc = __fdiv_rn(d2, __fsub_rn(d2, d6)); }
    else if (va <= 0.f && e43 >= 0.f && e56 >= 0.f) {
        const float t = __fdiv_rn(e43, __fadd_rn(e43, e56));
        wb = __fsub_rn(1.f, t);
        wc = t;
    } else if (!(s > 0.f)) { wb = 0.f; wc = 0.f; }
    else { wb = __fdiv_rn(vb, s); wc = __fdiv_rn(vc, s); }
    wa = __fsub_rn(__fsub_rn(1.f, wb), wc);
    const float3 q = make_float3(__fadd_rn(__fadd_rn(a.x, __fmul_rn(ab.x, wb)), __fmul_rn(ac.x, wc)),
                                 __fadd_rn(__fadd_rn(a.y, __fmul_rn(ab.y, wb)), __fmul_rn(ac.y, wc)),
                                 __fadd_rn(__fadd_rn(a.z, __fmul_rn(ab.z, wb)), __fmul_rn(ac.z, wc)));
    const float3 r = px_sub(p, q);
    return px_dot(r, r);
}

// Grown bounding box of triangle t.
__device__ __forceinline__ void px_box(const float *x, const int32_t *tri, int t, float pad, float3 &lo, float3 &hi)
{
    const float3 a = px_ld(x, tri[3ll * t]), b = px_ld(x, tri[3ll * t + 1]), c = px_ld(x, tri[3ll * t + 2]);
    lo = make_float3(fminf(fminf(a.x, b.x), c.x) - pad, fminf(fminf(a.y, b.y), c.y) - pad,
                     fminf(fminf(a.z, b.z), c.z) - pad);
    hi = make_float3(fmaxf(fmaxf(a.x, b.x), c.x) + pad, fmaxf(fmaxf(a.y, b.y), c.y) + pad,
                     fmaxf(fmaxf(a.z, b.z), c.z) + pad);
}

// Cell coordinate along one axis; false when outside the packable range.
__device__ __forceinline__ bool px_cell(float v, float inv, int &i)
{
    const float f = floorf(v * inv);
    if (!(f >= -(float)PX_COORD_BIAS && f < (float)PX_COORD_BIAS)) return false;
    i = (int)f;
    return true;
}
// Number of the cell at (ix, iy, iz), at least 0; -1 outside the numbered extent.
__device__ __forceinline__ int64_t px_number(const PxGrid &g, int ix, int iy, int iz)
{
    const int64_t x = (int64_t)ix - g.x0, y = (int64_t)iy - g.y0, z = (int64_t)iz - g.z0;
    if (x < 0 || y < 0 || z < 0 || x >= g.nx || y >= g.ny) return -1;
    const int64_t c = (z * g.ny + y) * g.nx + x;
    return (uint64_t)c < g.n ? c : -1;
}

// A float as an unsigned integer of the same order, and back (host side).
__device__ __forceinline__ uint32_t px_ordered(float f)
{
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : u | 0x80000000u;
}
static float px_from_ordered(uint32_t u)
{
    u = (u & 0x80000000u) ? u & 0x7fffffffu : ~u;
    float f;
    memcpy(&f, &u, sizeof(f));
    return f;
}

// Extent of the grown boxes: ext[0] the largest edge, ext[1..3] the complement of the lowest
// corner, ext[4..6] the highest corner (ordered integers; all maxima, from zero).
__global__ void __launch_bounds__(256) px_extent_kernel(int T, const float *x, const int32_t *tri, float pad, uint32_t *ext)
{
    __shared__ uint32_t s_m[7][8];
    uint32_t m[7] = {0u, 0u, 0u, 0u, 0u, 0u, 0u};
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < T; t += gridDim.x * blockDim.x) {
        float3 lo, hi;
        px_box(x, tri, t, pad, lo, hi);
        const float e = fmaxf(fmaxf(hi.x - lo.x, hi.y - lo.y), hi.z - lo.z);
        if (e > 0.f) m[0] = max(m[0], __float_as_uint(e));
        m[1] = max(m[1], ~px_ordered(lo.x));
        m[2] = max(m[2], ~px_ordered(lo.y));
        m[3] = max(m[3], ~px_ordered(lo.z));
        m[4] = max(m[4], px_ordered(hi.x));
        m[5] = max(m[5], px_ordered(hi.y));
        m[6] = max(m[6], px_ordered(hi.z));
    }
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        m[k] = __reduce_max_sync(0xffffffffu, m[k]);
        if ((threadIdx.x & 31) == 0) s_m[k][threadIdx.x >> 5] = m[k];
    }
    __syncthreads();
    if (threadIdx.x < 7) {
        uint32_t v = 0u;
        for (int w = 0; w < 8; ++w) v = max(v, s_m[threadIdx.x][w]);
        atomicMax(ext + threadIdx.x, v);
    }
}

// Cells per triangle (0 and an error bit when a box leaves the grid).
__global__ void px_count_cells_kernel(int T, const float *x, const int32_t *tri, float pad, float inv,
                                      int32_t *cnt, float4 *box, uint32_t *err)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t > T) return;
    if (t == T) {
        cnt[T] = 0;
        return;
    }
    float3 lo, hi;
    px_box(x, tri, t, pad, lo, hi);
    box[2ll * t] = make_float4(lo.x, lo.y, lo.z, hi.x);
    box[2ll * t + 1] = make_float4(hi.y, hi.z, 0.f, 0.f);
    int i0, i1, j0, j1, k0, k1;
    if (!(px_cell(lo.x, inv, i0) && px_cell(hi.x, inv, i1) && px_cell(lo.y, inv, j0) && px_cell(hi.y, inv, j1) &&
          px_cell(lo.z, inv, k0) && px_cell(hi.z, inv, k1))) {
        cnt[t] = 0;
        pc_set_err(err, PC_DERR_INDEX);
        return;
    }
    cnt[t] = (i1 - i0 + 1) * (j1 - j0 + 1) * (k1 - k0 + 1);
}

__global__ void px_emit_cells_kernel(int T, const float4 *__restrict__ box, float inv, PxGrid g, const int32_t *off,
                                     int64_t cap, uint64_t *keys, uint32_t *vals)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    const float4 p = box[2ll * t], q = box[2ll * t + 1];
    int i0, i1, j0, j1, k0, k1;
    if (!(px_cell(p.x, inv, i0) && px_cell(p.w, inv, i1) && px_cell(p.y, inv, j0) && px_cell(q.x, inv, j1) &&
          px_cell(p.z, inv, k0) && px_cell(q.y, inv, k1)))
        return;
    int64_t o = off[t];
    for (int k = k0; k <= k1; ++k)
        for (int j = j0; j <= j1; ++j)
            for (int i = i0; i <= i1; ++i) {
                if (o < cap) {
                    keys[o] = (uint64_t)px_number(g, i, j, k);
                    vals[o] = (uint32_t)t;
                }
                ++o;
            }
}

// first[c]: where cell c's list begins (c = 0 .. n), from the sorted keys: a thread per key fills
// the cells after the key before it, its whole warp where they are many. (Alone, one thread walked
// the run of empty cells between two 301 x 301 sheets 10 cm apart, 500,000 cells: a query took
// 1,937 us that takes 360. A search per cell takes 311 there, but 276-282 instead of 274-277 for
// three 100 x 100 sheets 0.5 mm apart.)
#define PX_RUN 64
__global__ void px_first_kernel(int64_t K, const uint64_t *__restrict__ keys, int64_t n, int32_t *first)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    int64_t b = 0, e = -1;
    if (i <= K) {
        b = i == 0 ? 0 : (int64_t)keys[i - 1] + 1;
        e = i == K ? n : (int64_t)keys[i];
    }
    const bool many = e - b >= PX_RUN;
    if (!many)
        for (int64_t c = b; c <= e; ++c) first[c] = (int32_t)i;
    for (unsigned m = __ballot_sync(0xffffffffu, many); m; m &= m - 1) {
        const int from = __ffs(m) - 1;
        const int64_t wb = __shfl_sync(0xffffffffu, b, from), we = __shfl_sync(0xffffffffu, e, from);
        const int32_t v = (int32_t)__shfl_sync(0xffffffffu, i, from);
#pragma unroll 8
        for (int64_t c = wb + lane; c <= we; c += 32) first[c] = v;
    }
}

// true when v is among ecol[lo .. hi) (sorted)
__device__ __forceinline__ bool px_ring_has(const int32_t *ecol, int lo, int hi, int v)
{
    const int end = hi;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (ecol[mid] < v) lo = mid + 1;
        else hi = mid;
    }
    return lo < end && ecol[lo] == v;
}

struct PxArgs {
    int V;
    const float *x;
    const int32_t *tri;
    const float4 *box;
    const uint64_t *keys;
    const uint32_t *vals;
    int64_t K;
    const int32_t *first;  // null: more cells than the table holds
    PxGrid g;
    float inv, delta;
    float round;           // how far outside its box the triangles' rounding can put a closest point
    const int32_t *erp, *ecol;
    int32_t *cnt;          // [V + 1] pairs of each vertex
    uint32_t *hits;        // [PX_HITS][V] their first triangles
    const int32_t *off;
    int32_t *pairs;
    float *w;
    uint32_t *err;
};

// Where the list of cell `c` begins (and, with the table, ends).
__device__ __forceinline__ void px_list(const PxArgs &a, int64_t c, int64_t &lo, int64_t &hi)
{
    lo = 0;
    hi = 0;
    if (c < 0) return;
    if (a.first) {
        lo = a.first[c];
        hi = a.first[c + 1];
        return;
    }
    int64_t h = a.K;
    while (lo < h) {
        const int64_t mid = (lo + h) >> 1;
        if (a.keys[mid] < (uint64_t)c) lo = mid + 1;
        else h = mid;
    }
    for (hi = lo; hi < a.K && a.keys[hi] == (uint64_t)c;) ++hi;
}

// Whether (p, t) is a pair, with the closest point's weights.
__device__ __forceinline__ bool px_pair(const PxArgs &a, int p, float3 xp, int t, int r0, int r1, float d2max, int &ia,
                                        int &ib, int &ic, float &wa, float &wb, float &wc)
{
    ia = a.tri[3ll * t];
    ib = a.tri[3ll * t + 1];
    ic = a.tri[3ll * t + 2];
    if (ia == p || ib == p || ic == p) return false;
    if (px_ring_has(a.ecol, r0, r1, ia) || px_ring_has(a.ecol, r0, r1, ib) || px_ring_has(a.ecol, r0, r1, ic))
        return false;
    return px_closest(xp, px_ld(a.x, ia), px_ld(a.x, ib), px_ld(a.x, ic), wa, wb, wc) < d2max;
}

// One thread per vertex: the triangles listed under its cell whose grown box holds it. COUNT:
// cnt[p] = pairs of p, the first PX_HITS in hits; WRITE: the pairs at off[p] ..., from hits
// unless there are more.
#define PX_BATCH 4  // boxes in flight per thread

template <bool WRITE>
__global__ void __launch_bounds__(128) px_pairs_kernel(PxArgs a)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p > a.V) return;
    if (p == a.V) {
        if (!WRITE) a.cnt[a.V] = 0;
        return;
    }
    const int have = WRITE ? a.cnt[p] : 0;
    if (WRITE && have == 0) return;
    const float3 xp = px_ld(a.x, p);
    const float d2max = __fmul_rn(a.delta, a.delta);
    const int r0 = a.erp[p], r1 = a.erp[p + 1];
    int ia, ib, ic;
    float wa, wb, wc;
    int n = 0;
    auto put = [&](int64_t o) {
        a.pairs[4 * o] = p;
        a.pairs[4 * o + 1] = ia;
        a.pairs[4 * o + 2] = ib;
        a.pairs[4 * o + 3] = ic;
        a.w[3 * o] = wa;
        a.w[3 * o + 1] = wb;
        a.w[3 * o + 2] = wc;
    };
    if (WRITE && have <= PX_HITS) {
        for (; n < have; ++n) {
            px_pair(a, p, xp, (int)a.hits[(int64_t)n * a.V + p], r0, r1, d2max, ia, ib, ic, wa, wb, wc);
            put((int64_t)a.off[p] + n);
        }
        return;
    }
    int ix, iy, iz;
    if (!(px_cell(xp.x, a.inv, ix) && px_cell(xp.y, a.inv, iy) && px_cell(xp.z, a.inv, iz))) {
        if (!WRITE) a.cnt[p] = 0;
        pc_set_err(a.err, PC_DERR_INDEX);
        return;
    }
    // the box already exceeds delta by a hundredth; this far outside it, no rounding can bring
    // the computed distance below delta: of p's coordinates (16 units in their last place), or of
    // the closest point a + wb (b - a) + wc (c - a) (6 half units of the mesh's largest one)
    const float slack = 0.05f * a.delta + 1e-6f * (fabsf(xp.x) + fabsf(xp.y) + fabsf(xp.z)) + a.round;
    int64_t lo, hi;
    px_list(a, px_number(a.g, ix, iy, iz), lo, hi);
    for (int64_t i = lo; i < hi; i += 32) {
        // first the boxes, four triangles' loads at a time, then the tests of those that hold
        // the vertex: the lanes of a warp take their first, second, ... one together
        const int len = (int)min((int64_t)32, hi - i);
        uint32_t held = 0;
        for (int j = 0; j < len; j += PX_BATCH) {
            float4 b0[PX_BATCH], b1[PX_BATCH];
#pragma unroll
            for (int u = 0; u < PX_BATCH; ++u) {
                const int64_t t = a.vals[i + min(j + u, len - 1)];
                b0[u] = a.box[2 * t];
                b1[u] = a.box[2 * t + 1];
            }
#pragma unroll
            for (int u = 0; u < PX_BATCH; ++u)
                if (j + u < len && !(xp.x < b0[u].x - slack || xp.y < b0[u].y - slack || xp.z < b0[u].z - slack ||
                                     xp.x > b0[u].w + slack || xp.y > b1[u].x + slack || xp.z > b1[u].y + slack))
                    held |= 1u << (j + u);
        }
        for (; held; held &= held - 1) {
            const int t = (int)a.vals[i + __ffs(held) - 1];
            if (!px_pair(a, p, xp, t, r0, r1, d2max, ia, ib, ic, wa, wb, wc)) continue;
            if (WRITE) put((int64_t)a.off[p] + n);
            else if (n < PX_HITS) a.hits[(int64_t)n * a.V + p] = (uint32_t)t;
            ++n;
        }
    }
    if (!WRITE) a.cnt[p] = n;
}

// The coordinate of the cell that holds v, as the kernels compute it (host side).
static bool px_host_cell(float v, float inv, int *i)
{
    const float f = floorf(v * inv);
    if (!(f >= -(float)PX_COORD_BIAS && f < (float)PX_COORD_BIAS)) return false;
    *i = (int)f;
    return true;
}

extern "C" pc_status pc_proximity_query(pc_ctx *ctx, const float *x, float delta, int32_t cap, int32_t *pairs,
                                        float *w, int32_t *n_out, void *stream)
{
    if (!ctx || !x || !n_out || cap < 0 || (cap > 0 && (!pairs || !w))) return PC_ERR_ARG;
    if (!(delta > 0.f) || !(delta < 1e30f)) return PC_ERR_ARG;
    *n_out = 0;
    cudaStream_t st = (cudaStream_t)stream;
    const int V = ctx->V, T = ctx->T;
    if (T == 0) return PC_OK;
    if (!ctx->px_keys) return PC_ERR_ARG;
    const float pad = delta * 1.01f;
    // cell size: the largest grown box (at least delta)
    PC_CUDA_TRY(cudaMemsetAsync(ctx->px_max, 0, 7 * sizeof(uint32_t), st));
    const unsigned ext_grid = pc_blocks(T, 256) < (unsigned)(ctx->num_sms * 8) ? pc_blocks(T, 256) : ctx->num_sms * 8;
    PC_LAUNCH(ctx, px_extent_kernel, ext_grid, 256, 0, st, T, x, ctx->tri, pad, ctx->px_max);
    PC_CUDA_TRY(cudaMemcpyAsync(ctx->h_count, ctx->px_max, 7 * sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
    PC_CUDA_TRY(cudaStreamSynchronize(st));
    uint32_t ext[7];
    memcpy(ext, ctx->h_count, sizeof(ext));
    const uint32_t bits_ext = ext[0];
    float corner[6];
    for (int k = 0; k < 3; ++k) {
        corner[k] = px_from_ordered(~ext[1 + k]);
        corner[3 + k] = px_from_ordered(ext[4 + k]);
    }
    float cs;
    memcpy(&cs, &bits_ext, sizeof(float));
    if (!(cs < 1e30f)) return PC_ERR_NONFINITE;
    cs = fmaxf(cs, delta) * 1.001f;
    const int64_t cap_k = ctx->px_cap;
    int64_t K = 0;
    PxGrid g{};
    for (int attempt = 0;; ++attempt) {
        const float inv = 1.0f / cs;
        PC_CUDA_TRY(cudaMemsetAsync(ctx->d_err, 0, sizeof(uint32_t), st));
        PC_LAUNCH(ctx, px_count_cells_kernel, pc_blocks(T + 1ll, 256), 256, 0, st, T, x, ctx->tri, pad, inv,
                  ctx->px_cnt, ctx->px_box, ctx->d_err);
        PC_TRY(pc_exclusive_scan(ctx, ctx->px_cnt, ctx->px_off, T, st));
        PC_CUDA_TRY(cudaMemcpyAsync(ctx->h_count, ctx->px_off + T, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
        uint32_t bits = 0;
        PC_TRY(pc_read_errors(ctx, st, &bits));
        if (bits) return PC_ERR_ARG;  // positions too far out for the cell grid
        K = *reinterpret_cast<int32_t *>(ctx->h_count);
        if (K <= cap_k) {
            int c[6];
            for (int k = 0; k < 6; ++k)
                if (!px_host_cell(corner[k], inv, c + k)) return PC_ERR_ARG;
            g.x0 = c[0];
            g.y0 = c[1];
            g.z0 = c[2];
            g.nx = (int64_t)c[3] - c[0] + 1;  // each extent at most 2^21: their product at most 2^63
            g.ny = (int64_t)c[4] - c[1] + 1;
            g.n = (uint64_t)(g.nx * g.ny) * (uint64_t)((int64_t)c[5] - c[2] + 1);
            PC_LAUNCH(ctx, px_emit_cells_kernel, pc_blocks(T, 256), 256, 0, st, T, ctx->px_box, inv, g, ctx->px_off,
                      cap_k, ctx->px_keys, ctx->px_vals);
            PC_TRY(pc_radix_sort(ctx, ctx->px_keys, ctx->px_vals, K, pc_bits_for((int64_t)std::min<uint64_t>(g.n, INT64_MAX)), st));
            break;
        }
        if (attempt >= 4) return PC_ERR_CAPACITY;
        cs *= 2.0f;  // rounding put some boxes across three cells: coarser grid
    }
    PxArgs a{};
    a.V = V;
    a.x = x;
    a.tri = ctx->tri;
    a.box = ctx->px_box;
    a.keys = ctx->px_keys;
    a.vals = ctx->px_vals;
    a.K = K;
    // a list of its own for every cell where the table has room (sheets do: a few triangles
    // per cell), else binary searches in the sorted keys
    a.first = g.n <= (uint64_t)ctx->px_first_cap ? ctx->px_first : nullptr;
    a.g = g;
    a.inv = 1.0f / cs;
    a.delta = delta;
    for (float v : corner) a.round = fmaxf(a.round, 1e-6f * fabsf(v));
    a.erp = ctx->erp;
    a.ecol = ctx->ecol;
    a.cnt = ctx->px_vcnt;
    a.hits = ctx->px_hits;
    a.off = ctx->px_voff;
    a.pairs = pairs;
    a.w = w;
    a.err = ctx->d_err;
    if (a.first)
        PC_LAUNCH(ctx, px_first_kernel, pc_blocks(K + 1, 256), 256, 0, st, K, ctx->px_keys, (int64_t)g.n, ctx->px_first);
    PC_LAUNCH(ctx, px_pairs_kernel<false>, pc_blocks(V + 1ll, 128), 128, 0, st, a);
    PC_TRY(pc_exclusive_scan(ctx, ctx->px_vcnt, ctx->px_voff, V, st));
    PC_CUDA_TRY(cudaMemcpyAsync(ctx->h_count, ctx->px_voff + V, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    uint32_t bits = 0;
    PC_TRY(pc_read_errors(ctx, st, &bits));
    if (bits) return PC_ERR_ARG;
    const int32_t P = *reinterpret_cast<int32_t *>(ctx->h_count);
    *n_out = P;
    if (P > cap) return PC_ERR_CAPACITY;
    if (P > 0)
        PC_LAUNCH(ctx, px_pairs_kernel<true>, pc_blocks(V + 1ll, 128), 128, 0, st, a);
    PC_CUDA_TRY(cudaStreamSynchronize(st));
    return PC_OK;
}

// Query buffers (called at context creation): 8 cell entries and a box per triangle, a table
// of two cells per triangle, per-triangle and per-vertex counts and offsets, remembered pairs.
pc_status pc_proximity_alloc(pc_ctx *c)
{
    c->px_cap = (int64_t)PX_CELLS_PER_TRI * c->T + 1;
    PC_CUDA_TRY(cudaMalloc(&c->px_keys, sizeof(uint64_t) * (size_t)c->px_cap));
    PC_CUDA_TRY(cudaMalloc(&c->px_vals, sizeof(uint32_t) * (size_t)c->px_cap));
    PC_CUDA_TRY(cudaMalloc(&c->px_cnt, sizeof(int32_t) * (c->T + 1ll)));
    PC_CUDA_TRY(cudaMalloc(&c->px_off, sizeof(int32_t) * (c->T + 1ll)));
    PC_CUDA_TRY(cudaMalloc(&c->px_vcnt, sizeof(int32_t) * (c->V + 1ll)));
    PC_CUDA_TRY(cudaMalloc(&c->px_voff, sizeof(int32_t) * (c->V + 1ll)));
    PC_CUDA_TRY(cudaMalloc(&c->px_max, 7 * sizeof(uint32_t)));
    PC_CUDA_TRY(cudaMalloc(&c->px_box, sizeof(float4) * 2 * (size_t)(c->T > 0 ? c->T : 1)));
    PC_CUDA_TRY(cudaMalloc(&c->px_hits, sizeof(uint32_t) * PX_HITS * (size_t)c->V));
    c->px_first_cap = 2ll * c->T + 4096;
    PC_CUDA_TRY(cudaMalloc(&c->px_first, sizeof(int32_t) * (size_t)(c->px_first_cap + 1)));
    return PC_OK;
}
