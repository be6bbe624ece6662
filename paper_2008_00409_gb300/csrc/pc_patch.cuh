// Patch storage of the system for the difference-form products of the PCG, and the product.
//
// Rows are renumbered so that runs of R consecutive rows ("patches") are compact pieces of
// the mesh (pc_patch.cu), and each off-diagonal block is stored once where that is possible:
// a block (i, j) with both rows in one patch is kept by one of them only and used for both,
// y_i += B (p_j - p_i) and y_j += B^T (p_i - p_j); a block that leaves its patch is kept by
// both rows. On a cloth (12 off-diagonal blocks per row) a 128-row patch keeps about 7 blocks
// per row: about 310 bytes per row in all, instead of the 480 of the BSR rows. At 830,028
// rows (three 526 x 526 layers) a product takes 53 us, 73 from the BSR rows.
//
// The keeping row's thread forms both products from one read of the block and leaves the
// other row's share in the block's own place; the other row's thread adds it after a
// barrier. (Reading the kept block a second time, transposed, was built first: twice the
// shared-memory wavefronts, half of them bank conflicts, and 54 us per product at paper
// scale.) Each sum has a fixed order, so the product is deterministic.
//
// Record of a patch, every part 16-byte aligned (n_own kept blocks; a slice is 32 rows):
//   first   int32[2][R / 32 + 1]: where each slice's entries and shares begin, in columns of 32
//   halo    int32[n_halo]: rows (new numbers) outside the patch that its blocks name, sorted
//   ent     uint32[32 x columns]: kept block e of a slice's row l at 32 (first + e) + l:
//           no share << 31 | local column (R + halo position outside the patch) << 16 | slot
//   mir     uint16[32 x columns]: slots of the blocks that other rows keep for this row
//   va, vb  float4[n_own + 1] each, vc float[n_own + 1]: a block's entries 0..3, 4..7, 8
// Every row of a slice has as many entries as its longest (missing ones name the row's own p,
// so that they add exactly zero, with a neighbouring lane's block; missing shares the zero
// block in slot n_own), so the loops have no conditions;
// of two rows with a common block the one with fewer blocks that leave the patch keeps it,
// which evens the rows out. Kept blocks of a slice are numbered by their rank in the row,
// then by row: the lanes of a warp, one row each, read consecutive slots.
#pragma once

#include "pc_internal.cuh"
#include "pc_tma.cuh"

#define PT_ROWS 128                       // rows per patch of the streamed product
#define PT_RESIDENT_ROWS 480              // largest patch whose records and vectors can fit one SM's shared memory
#define PT_MAX_ROWS 1024                  // largest patch the records can describe
#define PT_SLICES (PT_MAX_ROWS / 32)
#define PT_MAX_OWN 64                     // most kept blocks of one row
#define PT_HALO_CAP 4096                  // most block columns outside the patch
#define PT_RED_SLOTS 4                    // doubles per CTA of the partials array
#define PT_NO_SHARE 0x80000000u           // the entry's block leaves the patch, or there is none
#define PT_WAIT_BUDGET (1ll << 31)        // cycles (about a second) before a wait gives up

struct PatchDesc {
    int64_t offset;                // bytes from the start of the store
    int32_t n_own, n_ent, n_mir;   // kept blocks; columns of 32 entries and of 32 shares
    int32_t n_halo;
    int32_t bytes;                 // record size
    int32_t pad;
};

// Byte offsets of a record's parts.
struct PatchLayout {
    int halo, ent, mir, va, vb, vc, bytes;
};
__host__ __device__ inline int pt_up16(int n) { return (n + 15) & ~15; }
__host__ __device__ inline int pt_header(int R) { return pt_up16(8 * (R / 32 + 1)); }
__host__ __device__ inline PatchLayout patch_layout(int R, const PatchDesc &d)
{
    PatchLayout l;
    l.halo = pt_header(R);
    l.ent = l.halo + pt_up16(4 * d.n_halo);
    l.mir = l.ent + 128 * d.n_ent;
    l.va = l.mir + 64 * d.n_mir;
    l.vb = l.va + 16 * (d.n_own + 1);
    l.vc = l.vb + 16 * (d.n_own + 1);
    l.bytes = l.vc + pt_up16(4 * (d.n_own + 1));
    return l;
}

// p of a patch's rows and halo in shared memory, one array per component (three 4-byte
// loads of neighbouring lanes take three wavefronts, one 16-byte load takes four).
struct PatchP {
    float *x;
    int n;  // stride between the components
    __device__ __forceinline__ void put(int i, float4 v) const
    {
        x[i] = v.x;
        x[n + i] = v.y;
        x[2 * n + i] = v.z;
    }
};

// W kept blocks of this lane's row (ent: the first, STEP columns apart), all loads before the
// first FMA; the other row's share goes to `share` at the block's slot (va's own place, or
// an array of its own where the record is kept).
template <int W, int STEP>
__device__ __forceinline__ void patch_keep(const uint32_t *ent, const float4 *va, const float4 *vb, const float *vc,
                                           float4 *share, const PatchP &ps, float4 pi, float &a0, float &a1, float &a2)
{
    uint32_t r[W];
    float4 A[W], B[W];
    float C[W], x[W], y[W], z[W];
#pragma unroll
    for (int w = 0; w < W; ++w) r[w] = ent[32 * STEP * w];
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const uint32_t s = r[w] & 0xffffu, c = (r[w] >> 16) & 0x7fffu;
        A[w] = va[s];
        B[w] = vb[s];
        C[w] = vc[s];
        x[w] = ps.x[c];
        y[w] = ps.x[ps.n + c];
        z[w] = ps.x[2 * ps.n + c];
    }
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const float dx = x[w] - pi.x, dy = y[w] - pi.y, dz = z[w] - pi.z;
        a0 = fmaf(A[w].x, dx, fmaf(A[w].y, dy, fmaf(A[w].z, dz, a0)));
        a1 = fmaf(A[w].w, dx, fmaf(B[w].x, dy, fmaf(B[w].y, dz, a1)));
        a2 = fmaf(B[w].z, dx, fmaf(B[w].w, dy, fmaf(C[w], dz, a2)));
        if (!(r[w] & PT_NO_SHARE))
            share[r[w] & 0xffffu] =
                make_float4(fmaf(A[w].x, dx, fmaf(A[w].w, dy, B[w].z * dz)),
                            fmaf(A[w].y, dx, fmaf(B[w].x, dy, B[w].w * dz)),
                            fmaf(A[w].z, dx, fmaf(B[w].y, dy, C[w] * dz)), 0.f);
    }
}

// The row's kept blocks part, part + SPLIT, ... (lane = row of the slice), W at a time.
template <int SPLIT, int W>
__device__ __forceinline__ void patch_row_keep(const unsigned char *rec, const PatchLayout &L, float4 *share,
                                               const PatchP &ps, int slice, float4 pi, int part, float &a0, float &a1,
                                               float &a2)
{
    static_assert(W == 2 || W == 4, "the tail below");
    const float4 *va = reinterpret_cast<const float4 *>(rec + L.va), *vb = reinterpret_cast<const float4 *>(rec + L.vb);
    const float *vc = reinterpret_cast<const float *>(rec + L.vc);
    const int32_t *first = reinterpret_cast<const int32_t *>(rec);
    const int c1 = first[slice + 1];
    int c = first[slice] + part;
    const uint32_t *ent = reinterpret_cast<const uint32_t *>(rec + L.ent) + 32 * c + (threadIdx.x & 31);
#pragma unroll 1
    for (; c + (W - 1) * SPLIT < c1; c += W * SPLIT, ent += 32 * W * SPLIT)
        patch_keep<W, SPLIT>(ent, va, vb, vc, share, ps, pi, a0, a1, a2);
    if (W == 4 && c + SPLIT < c1) {
        patch_keep<2, SPLIT>(ent, va, vb, vc, share, ps, pi, a0, a1, a2);
        c += 2 * SPLIT;
        ent += 64 * SPLIT;
    }
    if (c < c1) patch_keep<1, SPLIT>(ent, va, vb, vc, share, ps, pi, a0, a1, a2);
}

// The shares that other rows left for this row (after a barrier): B^T (p_i - p_j) each.
template <int SPLIT>
__device__ __forceinline__ void patch_row_shares(const unsigned char *rec, const PatchLayout &L, const float4 *share, int R,
                                                 int slice, int part, float &a0, float &a1, float &a2)
{
    const int32_t *first = reinterpret_cast<const int32_t *>(rec) + R / 32 + 1;
    const int c1 = first[slice + 1];
    int c = first[slice] + part;
    const uint16_t *mir = reinterpret_cast<const uint16_t *>(rec + L.mir) + 32 * c + (threadIdx.x & 31);
#pragma unroll 4
    for (; c < c1; c += SPLIT, mir += 32 * SPLIT) {
        const float4 m = share[*mir];
        a0 -= m.x;
        a1 -= m.y;
        a2 -= m.z;
    }
}

struct PatchArgs {
    int V, R, n;                // rows, rows per patch, patches
    const PatchDesc *desc;
    const unsigned char *store;
    int64_t keep;               // records below this offset are copied without the evict-first policy
    int rec_cap, halo_cap;      // largest record (rounded up) and halo: the shared memory's parts
    const float *dsc;           // [V] scalar difference diagonal or -1, new numbers
    const float *dres;          // difference diagonal, original numbers
    const int32_t *old_of;      // new number -> original
    const float4 *x4;           // p, new numbers
    float4 *y4;                 // q = A p
    double *partials;
    pc_scalars *sc;
    uint32_t *err;
};

// q = A p and this CTA's p.q partial (as spmv_kernel): persistent CTAs of one thread per
// patch row, as many per SM as the records leave room for; each copies a patch's record to
// shared memory (one bulk copy) and computes. While some CTAs of an SM wait for their
// copies the others compute, so a CTA needs no second stage; what does not need the record
// is fetched a patch ahead (the descriptor two): the rows' own p and scalar diagonal, and
// the p of the halo's first 2 x 128 rows, which wait in registers during the computation. The
// first record does not depend on the preceding kernel and is requested before the
// programmatic wait.
// Bound by shared-memory wavefronts and their latency at 16 warps per SM about as much as by
// HBM: 52.9 us at 830,028 rows, 290 MB, 5.5 TB/s (the BSR stream: 73 us, 439 MB). Patches of 64
// and 160 rows take 56.5 and 53.7 us: 128 keeps as many blocks inside as four CTAs of an SM
// have room for. The slowest SM needs a fifth more cycles than the average; handing out the
// last patches by ticket evened that out but needs a partial sum per patch to keep the order of
// p.q, which cost more than it gave (a whole step 629 -> 681 ms).
#define PT_AHEAD 2  // halo rows per thread fetched a patch ahead

struct PatchAhead {
    float4 pi, h[PT_AHEAD];
    float s;
};

// The record of patch `d` to shared memory (one thread).
__device__ __forceinline__ void patch_copy(const PatchArgs &a, const PatchDesc &d, unsigned char *s_rec, uint64_t *bar)
{
    mbar_arrive_expect_tx(bar, (uint32_t)d.bytes);
    if (d.offset < a.keep) bulk_g2s_keep(s_rec, a.store + d.offset, (uint32_t)d.bytes, bar);
    else bulk_g2s(s_rec, a.store + d.offset, (uint32_t)d.bytes, bar);
}

// The halo's first rows go to `idx` in shared memory without passing through registers
// (a thread reads back only what it asked for itself).
__device__ __forceinline__ void patch_ahead_index(const PatchArgs &a, const PatchDesc &d, int32_t *idx)
{
    const int32_t *halo = reinterpret_cast<const int32_t *>(a.store + d.offset + pt_header(PT_ROWS));
#pragma unroll
    for (int k = 0; k < PT_AHEAD; ++k) {
        const int i = threadIdx.x + k * PT_ROWS;
        if (i < d.n_halo)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(idx + i)), "l"(halo + i) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}
__device__ __forceinline__ void patch_ahead_load(const PatchArgs &a, int patch, int n_halo, const int32_t *idx,
                                                 PatchAhead &n)
{
    asm volatile("cp.async.wait_all;" ::: "memory");
    const int row = patch * PT_ROWS + threadIdx.x;
    n.pi = make_float4(0.f, 0.f, 0.f, 0.f);
    n.s = 0.f;
    if (row < a.V) {
        n.pi = a.x4[row];
        n.s = a.dsc[row];
    }
#pragma unroll
    for (int k = 0; k < PT_AHEAD; ++k)
        if (threadIdx.x + k * PT_ROWS < n_halo) n.h[k] = a.x4[idx[threadIdx.x + k * PT_ROWS]];
}

static __global__ void __launch_bounds__(PT_ROWS, 4) patch_spmv_kernel(PatchArgs a)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t bar;
    __shared__ int s_timeout, s_done;
    __shared__ int32_t s_idx[PT_AHEAD * PT_ROWS];
    unsigned char *s_rec = smem_raw;
    const PatchP ps{reinterpret_cast<float *>(smem_raw + a.rec_cap), PT_ROWS + a.halo_cap};
    const int t = threadIdx.x, G = gridDim.x, last = a.n - 1;
    if (t == 0) {
        mbar_init(&bar, 1);
        s_timeout = 0;
        mbar_fence_init();
    }
    __syncthreads();
    int patch = blockIdx.x;  // the grid has at most as many CTAs as there are patches
    PatchDesc d = a.desc[patch], nd = a.desc[min(patch + G, last)];
    if (t == 0) patch_copy(a, d, s_rec, &bar);
    patch_ahead_index(a, d, s_idx);
    pdl_wait();
    if (t == 0) s_done = a.sc->done;
    __syncthreads();
    const bool done = s_done != 0;
    PatchAhead cur;
    if (!done) patch_ahead_load(a, patch, d.n_halo, s_idx, cur);
    uint32_t ph = 0;
    float dot_acc = 0.f, dot_c = 0.f;
    bool ok = true;
    for (; patch < a.n; patch += G) {
        const int row = patch * PT_ROWS + t;
        const bool more = patch + G < a.n;
        const PatchDesc nd2 = a.desc[min(patch + 2 * G, last)];
        if (more) patch_ahead_index(a, nd, s_idx);
        ok = mbar_wait_bounded(&bar, ph, PT_WAIT_BUDGET);
        ph ^= 1u;
        if (!ok) s_timeout = 1;
        if (done) {  // the copies in flight have landed (or the wait has given up)
            asm volatile("cp.async.wait_all;" ::: "memory");
            return;
        }
        const PatchLayout L = patch_layout(PT_ROWS, d);
        ps.put(t, cur.pi);
#pragma unroll
        for (int k = 0; k < PT_AHEAD; ++k)
            if (t + k * PT_ROWS < d.n_halo) ps.put((k + 1) * PT_ROWS + t, cur.h[k]);
        if (ok) {  // a thread whose wait gave up reads nothing of the record
            const int32_t *halo = reinterpret_cast<const int32_t *>(s_rec + L.halo);
            for (int i = t + PT_AHEAD * PT_ROWS; i < d.n_halo; i += PT_ROWS) ps.put(PT_ROWS + i, a.x4[halo[i]]);
        }
        const float4 pi = cur.pi;
        const float s = cur.s;
        __syncthreads();
        if (s_timeout) break;
        float a0 = 0.f, a1 = 0.f, a2 = 0.f;
        float4 *share = reinterpret_cast<float4 *>(s_rec + L.va);
        patch_row_keep<1, 4>(s_rec, L, share, ps, t >> 5, pi, 0, a0, a1, a2);
        __syncthreads();
        patch_row_shares<1>(s_rec, L, share, PT_ROWS, t >> 5, 0, a0, a1, a2);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the shares precede the next copy
        __syncthreads();  // the record and ps are free
        if (t == 0 && more) patch_copy(a, nd, s_rec, &bar);
        // not before the computation: the indices, fetched from the record in DRAM, have
        // arrived by now, and the gathers overlap the record's copy
        if (more) patch_ahead_load(a, patch + G, nd.n_halo, s_idx, cur);
        if (row < a.V) {
            if (s > 0.f) {
                a0 = fmaf(s, pi.x, a0);
                a1 = fmaf(s, pi.y, a1);
                a2 = fmaf(s, pi.z, a2);
            } else {
                const float *D = a.dres + 9ll * a.old_of[row];
                a0 = fmaf(D[0], pi.x, fmaf(D[1], pi.y, fmaf(D[2], pi.z, a0)));
                a1 = fmaf(D[3], pi.x, fmaf(D[4], pi.y, fmaf(D[5], pi.z, a1)));
                a2 = fmaf(D[6], pi.x, fmaf(D[7], pi.y, fmaf(D[8], pi.z, a2)));
            }
            a.y4[row] = make_float4(a0, a1, a2, 0.f);
            const float term = fmaf(pi.x, a0, fmaf(pi.y, a1, pi.z * a2));
            const float yk = term - dot_c, tk = dot_acc + yk;
            dot_c = (tk - dot_acc) - yk;
            dot_acc = tk;
        }
        d = nd;
        nd = nd2;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (s_timeout && t == 0) {
        atomicOr(a.err, PC_DERR_TIMEOUT);
        a.sc->status = PC_ERR_TIMEOUT;
        a.sc->done = 1;
    }
    pdl_trigger();
    float hi[1] = {dot_acc}, lo[1] = {-dot_c};
    pc_block_sum_df(hi, lo, 1);
    if (t == 0) reinterpret_cast<float2 *>(a.partials)[(int64_t)blockIdx.x * PT_RED_SLOTS + 3] = make_float2(hi[0], lo[0]);
}
