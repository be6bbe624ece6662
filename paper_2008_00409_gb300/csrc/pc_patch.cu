// Row order and per-solve records of the patch storage (pc_patch.cuh).
//
// Order, once per context: vertices sorted by connected component of the mesh, then along
// the Morton curve of their rest positions; R consecutive ones form a patch, and inside a
// patch rows keep the order of their original numbers. The order only decides how much is
// shared within a patch: any matrix of the context's size is stored correctly with it.
//
// Records, once per solve: a counting pass over the patches (one CTA each, one thread per
// row), a scan of the record sizes, a filling pass. A block whose mirror image is not its
// transpose bit for bit, a row that keeps more than PT_MAX_OWN blocks, a column
// out of order, or a patch whose halo or store does not fit make the build report failure;
// the solve then streams the BSR rows.
#include <algorithm>

#include "pc_patch.cuh"

// ------------------------------------------------------------------------- order

__global__ void comp_init_kernel(int V, int32_t *lab)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < V) lab[i] = i;
}
// hook: the smallest label around a vertex becomes the parent of its own label's root
__global__ void comp_hook_kernel(int V, const int32_t *__restrict__ erp, const int32_t *__restrict__ ecol, int32_t *lab,
                                 int32_t *changed)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= V) return;
    const int own = lab[i];
    int m = own;
    for (int e = erp[i]; e < erp[i + 1]; ++e) m = min(m, lab[ecol[e]]);
    if (m < own) {
        atomicMin(lab + own, m);
        *changed = 1;
    }
}
__global__ void comp_compress_kernel(int V, int32_t *lab)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= V) return;
    int l = lab[i];
    while (lab[l] < l) l = lab[l];
    lab[i] = l;
}

__global__ void __launch_bounds__(1024) bbox_kernel(int V, const float *__restrict__ X, float *box)
{
    __shared__ float s[6][32];
    float lo[3] = {1e30f, 1e30f, 1e30f}, hi[3] = {-1e30f, -1e30f, -1e30f};
    for (int i = threadIdx.x; i < V; i += blockDim.x)
        for (int a = 0; a < 3; ++a) {
            lo[a] = fminf(lo[a], X[3ll * i + a]);
            hi[a] = fmaxf(hi[a], X[3ll * i + a]);
        }
    for (int a = 0; a < 3; ++a) {
        for (int o = 16; o > 0; o >>= 1) {
            lo[a] = fminf(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
            hi[a] = fmaxf(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
        }
        if ((threadIdx.x & 31) == 0) {
            s[a][threadIdx.x >> 5] = lo[a];
            s[3 + a][threadIdx.x >> 5] = hi[a];
        }
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        float v = s[threadIdx.x][0];
        for (int w = 1; w < 32; ++w) v = threadIdx.x < 3 ? fminf(v, s[threadIdx.x][w]) : fmaxf(v, s[threadIdx.x][w]);
        box[threadIdx.x] = v;
    }
}

__device__ __forceinline__ uint64_t spread3(uint32_t x)
{
    uint64_t r = 0;
    for (int b = 0; b < 16; ++b) r |= (uint64_t)((x >> b) & 1u) << (3 * b);
    return r;
}
__global__ void morton_kernel(int V, const float *__restrict__ X, const float *__restrict__ box, int axis_bits,
                              uint64_t *keys, uint32_t *vals)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= V) return;
    const float ext = fmaxf(box[3] - box[0], fmaxf(box[4] - box[1], box[5] - box[2]));
    const float top = (float)((1 << axis_bits) - 1);
    const float sc = ext > 0.f ? top / ext : 0.f;
    uint64_t k = 0;
    for (int a = 0; a < 3; ++a) {
        const float q = fminf(fmaxf((X[3ll * i + a] - box[a]) * sc, 0.f), top);
        k |= spread3((uint32_t)q) << a;
    }
    keys[i] = k;
    vals[i] = (uint32_t)i;
}
__global__ void comp_key_kernel(int V, const int32_t *__restrict__ lab, const uint32_t *__restrict__ vals, uint64_t *keys)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < V) keys[i] = (uint64_t)lab[vals[i]];
}
__global__ void patch_key_kernel(int V, int R, int bits, const uint32_t *__restrict__ vals, uint64_t *keys)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < V) keys[i] = ((uint64_t)(i / R) << bits) | vals[i];
}
__global__ void order_kernel(int V, const uint32_t *__restrict__ vals, int32_t *old_of, int32_t *new_of)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= V) return;
    old_of[i] = (int32_t)vals[i];
    new_of[vals[i]] = i;
}

// The largest record that a solve can use: all the shared memory a CTA can have where the
// record stays in it, a third of an SM's where it is streamed (three CTAs beside each other).
pc_status pc_patch_limit(const pc_ctx *c, bool resident, int *bytes)
{
    PC_CUDA_TRY(cudaDeviceGetAttribute(bytes, resident ? cudaDevAttrMaxSharedMemoryPerBlockOptin
                                                       : cudaDevAttrMaxSharedMemoryPerMultiprocessor, c->device));
    if (!resident) *bytes /= 3;
    return PC_OK;
}

pc_status pc_patch_alloc(pc_ctx *c, cudaStream_t st)
{
    const int V = c->V;
    // one patch per SM where that many rows' records can stay in shared memory (the resident
    // schedule), else the streamed product's patches
    const int per_sm = ((V + c->num_sms - 1) / c->num_sms + 31) / 32 * 32;
    c->pt_rows = per_sm <= PT_RESIDENT_ROWS ? per_sm : PT_ROWS;
    c->pt_n = (V + c->pt_rows - 1) / c->pt_rows;
    const bool resident = c->pt_n <= c->num_sms;
    // kept blocks at most all of them, entries 4 bytes each, twice that with the slices' padding;
    // and never more than records that the solves can use (pc_patch_limit), however many
    // contacts the context has room for
    int limit = 0;
    PC_TRY(pc_patch_limit(c, resident, &limit));
    c->pt_cap = std::min(48 * c->A_cap + (int64_t)c->pt_n * 1024, (int64_t)c->pt_n * pt_up16(limit));
    // the arrays, in one allocation (pc_destroy frees it through pt_old)
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t o = at;
        at += (bytes + 255) / 256 * 256;
        return o;
    };
    const size_t o_old = take(sizeof(int32_t) * (size_t)V), o_new = take(sizeof(int32_t) * (size_t)V);
    const size_t o_desc = take(sizeof(PatchDesc) * (size_t)c->pt_n), o_cnt = take((size_t)c->pt_n * c->pt_rows);
    const size_t o_named = take((size_t)V), o_size = take(sizeof(int32_t) * 2 * (c->pt_n + 1ll)), o_info = take(32);
    const size_t o_z = take(resident ? 4 * sizeof(uint64_t) * (size_t)V : 0);
    const size_t o_slots = take(resident ? sizeof(uint64_t) * (12 * (size_t)c->pt_n * c->pt_n + 1) : 0);
    const size_t o_store = take((size_t)c->pt_cap);
    // without room for it the context has no order (pt_store stays null: the solves stream the
    // BSR rows)
    unsigned char *base = nullptr;
    if (cudaMalloc(&base, at) != cudaSuccess) {
        (void)cudaGetLastError();
        return PC_OK;
    }
    c->pt_old = reinterpret_cast<int32_t *>(base + o_old);
    c->pt_new = reinterpret_cast<int32_t *>(base + o_new);
    c->pt_desc = base + o_desc;
    c->pt_cnt = base + o_cnt;
    c->pt_named = base + o_named;
    c->pt_size = reinterpret_cast<int32_t *>(base + o_size);
    c->pt_info = reinterpret_cast<int32_t *>(base + o_info);
    if (resident) {
        c->pt_z = reinterpret_cast<unsigned long long *>(base + o_z);
        c->pt_slots = reinterpret_cast<unsigned long long *>(base + o_slots);
    }
    // keys and values in the proximity query's lists (8 entries per triangle) where they have room
    const bool own = c->px_cap < V;
    uint64_t *keys = c->px_keys;
    uint32_t *vals = c->px_vals;
    if (own) {
        keys = nullptr;
        if (cudaMalloc(&keys, (sizeof(uint64_t) + sizeof(uint32_t)) * (size_t)V) != cudaSuccess) {
            (void)cudaGetLastError();
            return PC_OK;
        }
        vals = reinterpret_cast<uint32_t *>(keys + V);
    }
    float *box = reinterpret_cast<float *>(c->pt_info);
    int32_t *lab = c->pt_new, *changed = reinterpret_cast<int32_t *>(c->d_count);
    const unsigned g = pc_blocks(V, 256);
    // the curve's cells: eight times as fine, along each axis, as V vertices on a square
    const int axis = std::min(16, pc_bits_for(V) / 2 + 3);
    pc_status s = PC_OK;
    do {
        comp_init_kernel<<<g, 256, 0, st>>>(V, lab);
        for (int it = 0; it < 32; ++it) {  // each round at least halves the steps that are left; 32 never binds
            cudaMemsetAsync(changed, 0, sizeof(int32_t), st);
            for (int k = 0; k < 3; ++k) {
                if (k == 2) cudaMemsetAsync(changed, 0, sizeof(int32_t), st);  // the last pass decides
                comp_hook_kernel<<<g, 256, 0, st>>>(V, c->erp, c->ecol, lab, changed);
                comp_compress_kernel<<<g, 256, 0, st>>>(V, lab);
            }
            c->launches += 6;
            cudaMemcpyAsync(c->h_count, changed, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
            if (cudaStreamSynchronize(st) != cudaSuccess) { s = PC_ERR_CUDA; break; }
            if (*reinterpret_cast<int32_t *>(c->h_count) == 0) break;
        }
        if (s != PC_OK) break;
        bbox_kernel<<<1, 1024, 0, st>>>(V, c->rest, box);
        morton_kernel<<<g, 256, 0, st>>>(V, c->rest, box, axis, keys, vals);
        if ((s = pc_radix_sort(c, keys, vals, V, 3 * axis, st)) != PC_OK) break;
        comp_key_kernel<<<g, 256, 0, st>>>(V, lab, vals, keys);
        if ((s = pc_radix_sort(c, keys, vals, V, pc_bits_for(V), st)) != PC_OK) break;
        // within a patch by original number: the values' low bits first, then the patch
        patch_key_kernel<<<g, 256, 0, st>>>(V, c->pt_rows, pc_bits_for(V), vals, keys);
        if ((s = pc_radix_sort(c, keys, vals, V, pc_bits_for(V) + pc_bits_for(c->pt_n), st)) != PC_OK) break;
        order_kernel<<<g, 256, 0, st>>>(V, vals, c->pt_old, c->pt_new);
        c->launches += 6;
        if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) s = PC_ERR_CUDA;
    } while (0);
    if (own) cudaFree(keys);
    if (s == PC_OK) c->pt_store = base + o_store;
    return s;
}

// ------------------------------------------------------------------------- records

struct BuildArgs {
    int V, R;
    const int32_t *rp, *ci;
    const float *vals;
    const int32_t *new_of, *old_of;
    PatchDesc *desc;
    uint8_t *cnt, *named;   // kept blocks of each row; rows in some patch's halo
    int32_t *size, *at;     // record sizes and offsets, in 16-byte units
    int32_t *info;          // [0] no record (count), [1] largest record, [2] largest halo, [3] failure (fill), [4] most kept blocks, [5] all of them
    int64_t cap;            // bytes of the store
    unsigned char *store;
};

// The patch's block columns outside it, sorted and without repeats, in s_list; returns
// their number (-1: too many). n: entries of s_list, not sorted.
__device__ int halo_sort(int *s_list, int n)
{
    if (n > PT_HALO_CAP) return -1;
    int m = 32;
    while (m < n) m <<= 1;
    for (int i = n + threadIdx.x; i < m; i += blockDim.x) s_list[i] = 0x7fffffff;
    __syncthreads();
    for (int k = 2; k <= m; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < m; i += blockDim.x) {
                const int o = i ^ j;
                if (o > i) {
                    const int x = s_list[i], y = s_list[o];
                    if ((x > y) == ((i & k) == 0)) {
                        s_list[i] = y;
                        s_list[o] = x;
                    }
                }
            }
            __syncthreads();
        }
    // compact in place: every thread takes a run, counts its firsts, then writes them
    __shared__ int s_run[1024];
    const int per = (n + blockDim.x - 1) / blockDim.x, b = min((int)threadIdx.x * per, n), e = min(b + per, n);
    int c = 0;
    for (int i = b; i < e; ++i) c += i == 0 || s_list[i] != s_list[i - 1];
    s_run[threadIdx.x] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int s = 0;
        for (int i = 0; i < (int)blockDim.x; ++i) {
            const int v = s_run[i];
            s_run[i] = s;
            s += v;
        }
    }
    __syncthreads();
    const int prev = b > 0 && b < n ? s_list[b - 1] : -1;
    int keep[PT_HALO_CAP / 128 + 1];  // per <= PT_HALO_CAP / blockDim (>= 128)
    int o = s_run[threadIdx.x], kk = 0;
    int last = prev;
    for (int i = b; i < e; ++i) {
        const int v = s_list[i];
        if (i == 0 || v != last) keep[kk++] = v;
        last = v;
    }
    __syncthreads();
    for (int i = 0; i < kk; ++i) s_list[o + i] = keep[i];
    __shared__ int s_n;
    if (threadIdx.x == blockDim.x - 1) s_n = o + kk;
    __syncthreads();
    return s_n;
}

// Whether, of two rows a and b of one patch (local numbers) that share a block, a keeps it: the
// one with fewer blocks that leave the patch, so that rows keep about equally many; else by
// the parity of a + b.
__device__ __forceinline__ bool patch_keeps(const uint16_t *cross, int a, int b)
{
    if (cross[a] != cross[b]) return cross[a] < cross[b];
    return ((a + b) & 1) ? a > b : a < b;
}

// cross[t]: blocks of local row t whose column lies outside the patch; their columns go to
// s_list (*s_n of them, at most PT_HALO_CAP kept).
__device__ void patch_cross(const BuildArgs &a, int base, uint16_t *cross, int *s_list, int *s_n)
{
    for (int t = threadIdx.x; t < a.R; t += blockDim.x) {
        int x = 0;
        if (base + t < a.V) {
            const int r = a.old_of[base + t];
            for (int k = a.rp[r]; k < a.rp[r + 1]; ++k) {
                const int nc = a.new_of[a.ci[k]];
                if (nc < base || nc >= base + a.R) {
                    ++x;
                    const int p = atomicAdd(s_n, 1);
                    if (p < PT_HALO_CAP) s_list[p] = nc;
                }
            }
        }
        cross[t] = (uint16_t)min(x, 65535);
    }
    __syncthreads();
}

// Count: per row its kept blocks, per patch its record's size.
__global__ void patch_count_kernel(BuildArgs a)
{
    __shared__ int s_list[PT_HALO_CAP];
    __shared__ uint16_t s_cross[PT_MAX_ROWS];
    __shared__ int s_n, s_own, s_ent, s_mir, s_bad;
    const int patch = blockIdx.x, base = patch * a.R;
    if (threadIdx.x == 0) s_n = s_own = s_ent = s_mir = s_bad = 0;
    __syncthreads();
    patch_cross(a, base, s_cross, s_list, &s_n);
    for (int t = threadIdx.x; t < a.R; t += blockDim.x) {
        int own = s_cross[t], mir = 0;
        if (base + t < a.V) {
            const int r = a.old_of[base + t];
            int prev = -1;
            for (int k = a.rp[r]; k < a.rp[r + 1]; ++k) {
                const int c = a.ci[k];
                if (c <= prev) s_bad = 1;  // columns ascend (a mirrored block is looked up once)
                prev = c;
                const int lc = a.new_of[c] - base;
                if (c == r || lc < 0 || lc >= a.R) continue;
                if (patch_keeps(s_cross, t, lc)) ++own;
                else ++mir;
            }
            if (own > PT_MAX_OWN || mir > 65535) s_bad = 1;
        }
        a.cnt[base + t] = (uint8_t)min(own, 255);
        const int n = (int)__reduce_add_sync(0xffffffffu, (unsigned)own);
        const int we = (int)__reduce_max_sync(0xffffffffu, (unsigned)own);
        const int wm = (int)__reduce_max_sync(0xffffffffu, (unsigned)mir);
        if ((t & 31) == 0) {
            atomicAdd(&s_own, n);
            atomicAdd(&s_ent, we);
            atomicAdd(&s_mir, wm);
        }
    }
    __syncthreads();
    const int nh = halo_sort(s_list, s_n);
    for (int i = threadIdx.x; i < nh; i += blockDim.x) a.named[s_list[i]] = 1;
    if (threadIdx.x == 0) {
        PatchDesc d{};
        d.n_own = s_own;
        d.n_ent = s_ent;
        d.n_mir = s_mir;
        d.n_halo = max(nh, 0);
        const bool bad = s_bad || nh < 0 || s_own > 65534 || a.R + d.n_halo > 32767 || s_mir > 4096;
        d.bytes = bad ? 0 : patch_layout(a.R, d).bytes;
        a.desc[patch] = d;
        a.size[patch] = d.bytes / 16;
        if (bad) atomicOr(a.info, 1);
        atomicMax(a.info + 1, d.bytes);
        atomicMax(a.info + 2, d.n_halo);
        atomicMax(a.info + 4, d.n_own);
        atomicAdd(a.info + 5, d.n_own);
    }
}

__global__ void patch_fill_kernel(BuildArgs a)
{
    __shared__ int s_list[PT_HALO_CAP];
    __shared__ uint16_t s_cross[PT_MAX_ROWS];
    __shared__ unsigned s_mask[PT_SLICES][PT_MAX_OWN];   // rows of the slice with an e-th kept block
    __shared__ uint16_t s_at[PT_SLICES][PT_MAX_OWN + 1]; // and the slot of the first of them
    __shared__ int s_base[3][PT_SLICES + 1];             // first slot, entry column, share column of each slice
    __shared__ int s_n;
    const int patch = blockIdx.x, base = patch * a.R, lane = threadIdx.x & 31;
    const int slices = a.R / 32;
    PatchDesc d = a.desc[patch];
    d.offset = 16ll * a.at[patch];
    if (a.info[0] || d.offset + d.bytes > a.cap) {  // info[0] is final: this kernel reports in info[3]
        if (threadIdx.x == 0) atomicOr(a.info + 3, 1);
        return;
    }
    if (threadIdx.x == 0) {
        a.desc[patch].offset = d.offset;
        s_n = 0;
    }
    __syncthreads();
    unsigned char *rec = a.store + d.offset;
    const PatchLayout L = patch_layout(a.R, d);
    patch_cross(a, base, s_cross, s_list, &s_n);
    for (int t = threadIdx.x; t < a.R; t += blockDim.x) {
        const int nr = base + t, sl = t >> 5;
        const int co = a.cnt[nr];
        const int mo = (int)__reduce_max_sync(0xffffffffu, (unsigned)co);
        int at = 0;
        for (int e = 0; e < mo; ++e) {
            const unsigned m = __ballot_sync(0xffffffffu, e < co);
            if (lane == 0) {
                s_mask[sl][e] = m;
                s_at[sl][e] = (uint16_t)at;
            }
            at += __popc(m);
        }
        int mir = 0;
        if (nr < a.V) {
            const int r = a.old_of[nr];
            for (int k = a.rp[r]; k < a.rp[r + 1]; ++k) {
                const int c = a.ci[k], lc = a.new_of[c] - base;
                mir += c != r && lc >= 0 && lc < a.R && !patch_keeps(s_cross, t, lc);
            }
        }
        const int wm = (int)__reduce_max_sync(0xffffffffu, (unsigned)mir);
        if (lane == 0) {
            s_base[0][sl] = at;
            s_base[1][sl] = mo;
            s_base[2][sl] = wm;
        }
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        int s = 0;
        for (int i = 0; i <= slices; ++i) {
            const int v = i < slices ? s_base[threadIdx.x][i] : 0;
            s_base[threadIdx.x][i] = s;
            if (threadIdx.x > 0) reinterpret_cast<int32_t *>(rec)[(threadIdx.x - 1) * (slices + 1) + i] = s;
            s += v;
        }
    }
    __syncthreads();
    const int nh = halo_sort(s_list, s_n);
    for (int i = threadIdx.x; i < nh; i += blockDim.x) reinterpret_cast<int32_t *>(rec + L.halo)[i] = s_list[i];
    uint32_t *ent = reinterpret_cast<uint32_t *>(rec + L.ent);
    uint16_t *mir = reinterpret_cast<uint16_t *>(rec + L.mir);
    float4 *va = reinterpret_cast<float4 *>(rec + L.va), *vb = reinterpret_cast<float4 *>(rec + L.vb);
    float *vc = reinterpret_cast<float *>(rec + L.vc);
    if (threadIdx.x == 0) {
        va[d.n_own] = vb[d.n_own] = make_float4(0.f, 0.f, 0.f, 0.f);
        vc[d.n_own] = 0.f;
    }
    for (int t = threadIdx.x; t < a.R; t += blockDim.x) {
        const int nr = base + t, sl = t >> 5;
        const unsigned lt = (1u << lane) - 1u;
        const int r = nr < a.V ? a.old_of[nr] : 0;
        const int k0 = nr < a.V ? a.rp[r] : 0, k1 = nr < a.V ? a.rp[r + 1] : 0;
        uint32_t *o = ent + 32 * s_base[1][sl] + lane, *o_end = ent + 32 * s_base[1][sl + 1];
        uint16_t *m = mir + 32 * s_base[2][sl] + lane, *m_end = mir + 32 * s_base[2][sl + 1];
        int e = 0;
        for (int k = k0; k < k1; ++k) {
            const int c = a.ci[k];
            if (c == r) continue;
            const int nc = a.new_of[c];
            int lc = nc - base;
            const bool out = lc < 0 || lc >= a.R;
            const float *B = a.vals + 9ll * k;
            if (out || patch_keeps(s_cross, t, lc)) {
                const int s = s_base[0][sl] + s_at[sl][e] + __popc(s_mask[sl][e] & lt);
                ++e;
                if (out) {
                    int lo = 0, hi = nh;
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (s_list[mid] < nc) lo = mid + 1; else hi = mid;
                    }
                    lc = a.R + lo;
                }
                va[s] = make_float4(B[0], B[1], B[2], B[3]);
                vb[s] = make_float4(B[4], B[5], B[6], B[7]);
                vc[s] = B[8];
                *o = (out ? PT_NO_SHARE : 0u) | ((uint32_t)lc << 16) | (uint32_t)s;
                o += 32;
            } else {  // block (c, r), kept by row c: its place among that row's kept blocks
                const int ls = lc >> 5;
                int e2 = 0, q = a.rp[c];
                const int q1 = a.rp[c + 1];
                for (; q < q1 && a.ci[q] != r; ++q) {
                    const int l2 = a.new_of[a.ci[q]] - base;
                    e2 += l2 != lc && (l2 < 0 || l2 >= a.R || patch_keeps(s_cross, lc, l2));
                }
                bool same = q < q1;
                if (same) {
                    const float *T = a.vals + 9ll * q;
                    for (int i = 0; i < 3; ++i)
                        for (int j = 0; j < 3; ++j)
                            same = same && __float_as_uint(B[3 * i + j]) == __float_as_uint(T[3 * j + i]);
                }
                int s = d.n_own;
                if (!same) atomicOr(a.info + 3, 1);
                else s = s_base[0][ls] + s_at[ls][e2] + __popc(s_mask[ls][e2] & ((1u << (lc & 31)) - 1u));
                *m = (uint16_t)s;
                m += 32;
            }
        }
        // missing entries: own p (zero difference), the block of a lane of the same eight,
        // which one 16-byte shared-memory access serves together
        for (; o < o_end; o += 32, ++e) {
            const unsigned m8 = s_mask[sl][e] & (0xffu << (lane & 24)), all = s_mask[sl][e];
            const int from = __ffs(m8 ? m8 : all) - 1;
            *o = PT_NO_SHARE | ((uint32_t)t << 16) |
                 (uint32_t)(s_base[0][sl] + s_at[sl][e] + __popc(all & ((1u << from) - 1u)));
        }
        for (; m < m_end; m += 32) *m = (uint16_t)d.n_own;
    }
}

pc_status pc_patch_build(pc_ctx *c, const pc_bsr *A, const float *vals, PatchInfo *out, cudaStream_t st)
{
    out->ok = false;
    if (!c->pt_store || A->nnzb > c->A_cap) return PC_OK;
    BuildArgs a{};
    a.V = c->V;
    a.R = c->pt_rows;
    a.rp = A->row_ptr;
    a.ci = A->col_idx;
    a.vals = vals;
    a.new_of = c->pt_new;
    a.old_of = c->pt_old;
    a.desc = static_cast<PatchDesc *>(c->pt_desc);
    a.cnt = c->pt_cnt;
    a.named = c->pt_named;
    a.size = c->pt_size;
    a.at = c->pt_size + c->pt_n + 1;
    a.info = c->pt_info;
    a.cap = c->pt_cap;
    a.store = c->pt_store;
    const int threads = a.R < 128 ? 128 : a.R > 512 ? 512 : a.R;
    PC_CUDA_TRY(cudaMemsetAsync(c->pt_info, 0, sizeof(int32_t) * 6, st));
    PC_CUDA_TRY(cudaMemsetAsync(c->pt_named, 0, (size_t)c->V, st));
    PC_LAUNCH(c, patch_count_kernel, c->pt_n, threads, 0, st, a);
    PC_TRY(pc_exclusive_scan(c, a.size, a.at, c->pt_n, st));
    PC_LAUNCH(c, patch_fill_kernel, c->pt_n, threads, 0, st, a);
    PC_CUDA_TRY(cudaMemcpyAsync(c->h_count, c->pt_info, sizeof(int32_t) * 6, cudaMemcpyDeviceToHost, st));
    PC_CUDA_TRY(cudaStreamSynchronize(st));
    const int32_t *h = reinterpret_cast<const int32_t *>(c->h_count);
    out->ok = h[0] == 0 && h[3] == 0;
    out->max_bytes = h[1];
    out->max_halo = h[2];
    out->max_own = h[4];
    c->pt_kept = h[5];
    return PC_OK;
}
