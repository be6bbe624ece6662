// Row order and per-solve records of the patch storage (pc_patch.cuh).
//
// Order, once per context: vertices sorted by connected component of the mesh, then along
// the Morton curve of their rest positions; R consecutive ones form a patch, and inside a
// patch rows keep the order of their original numbers. The order only decides how much is
// shared within a patch: any matrix of the context's size is stored correctly with it.
//
// Records, once per solve: a counting pass over the patches (one CTA each), a scan of the
// record sizes, a filling pass. A block whose mirror image is not its transpose bit for bit, a
// row that keeps more than PT_MAX_OWN blocks, a column out of order, or a patch whose halo or
// record does not fit make the build report failure; the solve then streams the BSR rows.
// Contacts between sheets join different patches, so both rows keep their blocks: three sheets'
// records fit with up to 0.5 contacts per vertex where they are streamed (10 kept blocks per row),
// and with 0.1, 1 and 4 where they stay on SMs of 444, 198 and 81 rows.
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
    const size_t o_cross = take(2 * sizeof(uint16_t) * (size_t)c->pt_n * c->pt_rows);
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
    c->pt_cross = reinterpret_cast<uint16_t *>(base + o_cross);
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
    uint16_t *cross, *mirs; // blocks of each row that leave the patch; that another row keeps
    int32_t *size, *at;     // record sizes and offsets, in 16-byte units
    int32_t *info;          // [0] no record (count), [1] largest record, [2] largest halo, [3] failure (fill), [4] most kept blocks, [5] all of them
    int limit;              // bytes of the largest record that a solve can use
    int64_t cap;            // bytes of the store
    unsigned char *store;
};

// f(k, column, its new number) for the blocks k of row r, four columns in flight.
template <typename F>
__device__ __forceinline__ void patch_row(const BuildArgs &a, int r, F f)
{
    const int k1 = a.rp[r + 1];
    for (int k = a.rp[r]; k < k1; k += 4) {
        int c[4], n[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) c[u] = a.ci[min(k + u, k1 - 1)];
#pragma unroll
        for (int u = 0; u < 4; ++u) n[u] = a.new_of[c[u]];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (k + u < k1) f(k + u, c[u], n[u]);
    }
}

// The patch's block columns outside it, sorted and without repeats, in s_list; returns
// their number (-1: too many). n: entries of s_list, not sorted.
__device__ int halo_sort(int *s_list, int n)
{
    __shared__ int s_cnt[32];
    if (n > PT_HALO_CAP) return -1;
    int m = 32;
    while (m < n) m <<= 1;
    for (int i = n + threadIdx.x; i < m; i += blockDim.x) s_list[i] = 0x7fffffff;
    __syncthreads();
    for (int k = 2; k <= m; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int t = threadIdx.x; t < m / 2; t += blockDim.x) {
                const int i = 2 * t - (t & (j - 1)), o = i + j;
                const int x = s_list[i], y = s_list[o];
                if ((x > y) == ((i & k) == 0)) {
                    s_list[i] = y;
                    s_list[o] = x;
                }
            }
            __syncthreads();
        }
    // compact in place, a chunk of one value per thread at a time
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int kept = 0;
    for (int i0 = 0; i0 < n; i0 += blockDim.x) {
        const int i = i0 + threadIdx.x;
        const int v = i < n ? s_list[i] : 0;
        const bool first = i < n && (i == 0 || s_list[i - 1] != v);
        const unsigned b = __ballot_sync(0xffffffffu, first);
        if (lane == 0) s_cnt[warp] = __popc(b);
        __syncthreads();  // (and the chunk has been read)
        int at = kept;
        for (int w = 0; w < nw; ++w) {
            const int c = s_cnt[w];
            if (w < warp) at += c;
            kept += c;
        }
        if (first) s_list[at + __popc(b & ((1u << lane) - 1u))] = v;
        __syncthreads();
    }
    return kept;
}

// Whether, of two rows a and b of one patch (local numbers) that share a block, a keeps it: the
// one with fewer blocks that leave the patch, so that rows keep about equally many; else by
// the parity of a + b.
__device__ __forceinline__ bool patch_keeps(const uint16_t *cross, int a, int b)
{
    if (cross[a] != cross[b]) return cross[a] < cross[b];
    return ((a + b) & 1) ? a > b : a < b;
}

// Count: per row its kept blocks, per patch its record's size. A patch that no solve can use
// (dense contacts: more blocks than fit) is found before its halo is sorted.
__global__ void __launch_bounds__(1024) patch_count_kernel(BuildArgs a)
{
    extern __shared__ uint16_t s_cross[];  // [R]
    __shared__ int s_list[PT_HALO_CAP];
    __shared__ int s_n, s_own, s_ent, s_mir, s_bad;
    const int patch = blockIdx.x, base = patch * a.R;
    if (threadIdx.x == 0) s_n = s_own = s_ent = s_mir = s_bad = 0;
    __syncthreads();
    for (int t = threadIdx.x; t < a.R; t += blockDim.x) {
        int x = 0;
        if (base + t < a.V)
            patch_row(a, a.old_of[base + t], [&](int, int, int nc) {
                if (nc >= base && nc < base + a.R) return;
                ++x;
                const int p = atomicAdd(&s_n, 1);
                if (p < PT_HALO_CAP) s_list[p] = nc;
            });
        a.cross[base + t] = s_cross[t] = (uint16_t)min(x, 65535);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < a.R; t += blockDim.x) {
        int own = s_cross[t], mir = 0;
        if (base + t < a.V) {
            const int r = a.old_of[base + t];
            int prev = -1;
            patch_row(a, r, [&](int, int c, int nc) {
                if (c <= prev) s_bad = 1;  // columns ascend (a mirrored block is looked up once)
                prev = c;
                const int lc = nc - base;
                if (c == r || lc < 0 || lc >= a.R) return;
                if (patch_keeps(s_cross, t, lc)) ++own;
                else ++mir;
            });
            if (own > PT_MAX_OWN || mir > 65535) s_bad = 1;
        }
        a.cnt[base + t] = (uint8_t)min(own, 255);
        a.mirs[base + t] = (uint16_t)min(mir, 65535);
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
    PatchDesc d{};
    d.n_own = s_own;
    d.n_ent = s_ent;
    d.n_mir = s_mir;
    bool bad = s_bad || s_own > 65534 || s_mir > 4096 || patch_layout(a.R, d).bytes > a.limit;
    const int nh = bad ? -1 : halo_sort(s_list, s_n);
    for (int i = threadIdx.x; i < nh; i += blockDim.x) a.named[s_list[i]] = 1;
    if (threadIdx.x == 0) {
        d.n_halo = max(nh, 0);
        bad = bad || nh < 0 || a.R + d.n_halo > 32767;
        d.bytes = bad ? 0 : patch_layout(a.R, d).bytes;
        a.desc[patch] = d;
        a.size[patch] = d.bytes / 16;
        if (bad || d.bytes > a.limit) atomicOr(a.info, 1);
        atomicMax(a.info + 1, d.bytes);
        atomicMax(a.info + 2, d.n_halo);
        atomicMax(a.info + 4, d.n_own);
        atomicAdd(a.info + 5, d.n_own);
    }
}

// Fill, in three passes with the CTA's barrier between them: each row numbers its blocks (a kept
// one leaves its place in the matrix, its entry's place and its column in the slot it gets, a
// mirrored one the row that keeps it); each slot becomes the block and its entry; each mirrored
// block finds its slot among the keeping row's entries and is compared with it.
// Bound by the latency of the columns' and blocks' gathers. 271,803 rows with 5% contacts: 191 us,
// and 50 for 12,288 rows with dense ones (796 and 377 with a thread per row that copied each block,
// and looked for each mirrored one along the other row's columns).
__global__ void __launch_bounds__(1024) patch_fill_kernel(BuildArgs a)
{
    extern __shared__ unsigned char s_raw[];
    __shared__ int s_list[PT_HALO_CAP];
    __shared__ int s_base[3][PT_SLICES + 1];  // first slot, entry column, share column of each slice
    __shared__ int s_n;
    const int patch = blockIdx.x, base = patch * a.R, lane = threadIdx.x & 31;
    const int slices = a.R / 32;
    unsigned *s_mask = reinterpret_cast<unsigned *>(s_raw);                        // [slice][e]: rows with an e-th kept block
    uint16_t *s_at = reinterpret_cast<uint16_t *>(s_mask + slices * PT_MAX_OWN);   // and the slot of the first of them
    uint16_t *s_cross = s_at + slices * PT_MAX_OWN;                                // [R]
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
    unsigned char *rec = a.store + d.offset;
    const PatchLayout L = patch_layout(a.R, d);
    for (int t = threadIdx.x; t < a.R; t += blockDim.x) {
        const int sl = t >> 5, co = a.cnt[base + t];
        const int mo = (int)__reduce_max_sync(0xffffffffu, (unsigned)co);
        const int wm = (int)__reduce_max_sync(0xffffffffu, (unsigned)a.mirs[base + t]);
        s_cross[t] = a.cross[base + t];
        int at = 0;
        for (int e = 0; e < mo; ++e) {
            const unsigned m = __ballot_sync(0xffffffffu, e < co);
            if (lane == 0) {
                s_mask[sl * PT_MAX_OWN + e] = m;
                s_at[sl * PT_MAX_OWN + e] = (uint16_t)at;
            }
            at += __popc(m);
        }
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
        int o = 32 * s_base[1][sl] + lane, m = 32 * s_base[2][sl] + lane, e = 0;
        if (nr < a.V) {
            const int r = a.old_of[nr];
            patch_row(a, r, [&](int k, int c, int nc) {
                if (c == r) return;
                const int lc = nc - base;
                const bool out = lc < 0 || lc >= a.R;
                if (out || patch_keeps(s_cross, t, lc)) {
                    const int s = s_base[0][sl] + s_at[sl * PT_MAX_OWN + e] + __popc(s_mask[sl * PT_MAX_OWN + e] & lt);
                    ++e;
                    reinterpret_cast<int4 *>(va)[s] = make_int4(k, o, nc, 0);
                    o += 32;
                    if (out) {
                        const int p = atomicAdd(&s_n, 1);
                        if (p < PT_HALO_CAP) s_list[p] = nc;
                    }
                } else {
                    mir[m] = (uint16_t)lc;
                    m += 32;
                }
            });
        }
        // missing entries: own p (zero difference), the block of a lane of the same eight,
        // which one 16-byte shared-memory access serves together
        for (; o < 32 * s_base[1][sl + 1]; o += 32, ++e) {
            const unsigned all = s_mask[sl * PT_MAX_OWN + e], m8 = all & (0xffu << (lane & 24));
            const int from = __ffs(m8 ? m8 : all) - 1;
            ent[o] = PT_NO_SHARE | ((uint32_t)t << 16) |
                     (uint32_t)(s_base[0][sl] + s_at[sl * PT_MAX_OWN + e] + __popc(all & ((1u << from) - 1u)));
        }
        for (; m < 32 * s_base[2][sl + 1]; m += 32) mir[m] = (uint16_t)d.n_own;
    }
    __syncthreads();
    const int nh = halo_sort(s_list, s_n);
    for (int i = threadIdx.x; i < nh; i += blockDim.x) reinterpret_cast<int32_t *>(rec + L.halo)[i] = s_list[i];
    for (int s = threadIdx.x; s < d.n_own; s += blockDim.x) {
        const int4 w = reinterpret_cast<const int4 *>(va)[s];
        const float *B = a.vals + 9ll * w.x;
        float b[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) b[q] = B[q];
        int lc = w.z - base;
        const bool out = lc < 0 || lc >= a.R;
        if (out) {
            int lo = 0, hi = nh;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (s_list[mid] < w.z) lo = mid + 1; else hi = mid;
            }
            lc = a.R + lo;
        }
        va[s] = make_float4(b[0], b[1], b[2], b[3]);
        vb[s] = make_float4(b[4], b[5], b[6], b[7]);
        vc[s] = b[8];
        ent[w.y] = (out ? PT_NO_SHARE : 0u) | ((uint32_t)lc << 16) | (uint32_t)s;
    }
    __syncthreads();
    const int parts = max(1, (int)blockDim.x / a.R);
    for (int i = threadIdx.x; i < parts * a.R; i += blockDim.x) {
        const int part = i / a.R, t = i - part * a.R, nr = base + t;
        if (nr >= a.V) continue;
        const int r = a.old_of[nr], k0 = a.rp[r], k1 = a.rp[r + 1], n = a.mirs[nr];
        uint16_t *m = mir + 32 * s_base[2][t >> 5] + lane;
        for (int j = part; j < n; j += parts) {
            const int lc = m[32 * j], c = a.old_of[base + lc];
            int lo = k0, hi = k1;  // the block (r, c)
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (a.ci[mid] < c) lo = mid + 1; else hi = mid;
            }
            const float *B = a.vals + 9ll * lo;
            const uint32_t *o = ent + 32 * s_base[1][lc >> 5] + (lc & 31);
            uint32_t w = 0;
            const int ne = a.cnt[base + lc];
            int e = 0;
            for (; e < ne; ++e) {
                w = o[32 * e];
                if ((w >> 16) == (uint32_t)t) break;  // a shared entry (its top bit clear) of column t
            }
            const int s = w & 0xffffu;
            bool same = e < ne;
            if (same) {
                const float4 p = va[s], q = vb[s];
                const float T[9] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w, vc[s]};
#pragma unroll
                for (int x = 0; x < 3; ++x)
#pragma unroll
                    for (int y = 0; y < 3; ++y)
                        same = same && __float_as_uint(B[3 * x + y]) == __float_as_uint(T[3 * y + x]);
            }
            if (!same) atomicOr(a.info + 3, 1);
            m[32 * j] = (uint16_t)(same ? s : d.n_own);
        }
    }
}

// `limit`: bytes of the largest record that the solve can use.
pc_status pc_patch_build(pc_ctx *c, const pc_bsr *A, const float *vals, int limit, PatchInfo *out, cudaStream_t st)
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
    a.cross = c->pt_cross;
    a.mirs = c->pt_cross + (size_t)c->pt_n * c->pt_rows;
    a.named = c->pt_named;
    a.size = c->pt_size;
    a.at = c->pt_size + c->pt_n + 1;
    a.info = c->pt_info;
    a.limit = limit;
    a.cap = c->pt_cap;
    a.store = c->pt_store;
    // one CTA per SM and patch: as many threads as the rows can use. Else two per row: the passes
    // over slots and mirrored blocks share them (830,028 rows: 525 us; 596 with one, 679 with four)
    const int threads = c->pt_slots ? (a.R <= 256 ? 4 : 2) * a.R : 2 * PT_ROWS;
    const size_t fill_smem = a.R / 32 * PT_MAX_OWN * (sizeof(unsigned) + sizeof(uint16_t)) + sizeof(uint16_t) * a.R;
    PC_CUDA_TRY(cudaMemsetAsync(c->pt_info, 0, sizeof(int32_t) * 6, st));
    PC_CUDA_TRY(cudaMemsetAsync(c->pt_named, 0, (size_t)c->V, st));
    PC_LAUNCH(c, patch_count_kernel, c->pt_n, threads, sizeof(uint16_t) * a.R, st, a);
    PC_TRY(pc_exclusive_scan(c, a.size, a.at, c->pt_n, st));
    PC_LAUNCH(c, patch_fill_kernel, c->pt_n, threads, fill_smem, st, a);
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
