// PCG iterations of a system whose patch records (pc_patch.cuh) fit the GPU's shared memory:
// one cooperative launch runs iterations until the solve needs the host (it stopped, or a
// mixed-precision residual replacement is due), with the matrix, p and the halo's p in
// shared memory and x, r and the preconditioner in registers for the length of the launch.
//
// One CTA per patch, one patch per SM, SPLIT threads per row. An iteration is
//   q = A p from shared memory, p.q over all CTAs;  x += alpha p, r -= alpha q, z = M^-1 r,
//   z to global memory, r.z and r.r over all CTAs;  p = z + beta p, the halo's p from the
//   neighbours' z (their p is never exchanged),
// the iteration of the streamed schedule with its two grid-wide sums. A sum is also the
// barrier: every CTA publishes its partial sums as 64-bit pairs (float, epoch), and reads
// everyone's until the epochs match, so no counter is shared, and arrival, waiting and the
// values cost one store and one load of L2 latency. The z rows that other
// patches name carry their epoch in the same words, so neither side needs a fence (with
// fences, which drain the CTA's stores and drop its L1, an iteration took 14 us at 22,801
// rows). Slots alternate between two
// places: a CTA can publish its second next sum only after all have published the next
// one, which they do after reading this one; a z row is written again only after the next
// iteration's first sum, which a CTA joins after it has gathered its halo. Epochs only grow
// over a context's launches. Sums are double-float in a fixed order, so every CTA gets the
// same bits and takes the same decisions.
//
// Bound by the two sums (4,300 cycles each and more with 128 CTAs, most of it words on their
// way through L2) and, towards the largest systems, by the product's shared-memory reads:
// 7.0 us per iteration at 4,096 rows, 8.0 at 20,083, 9.9 at 22,801, 11.7 at 71,824, where two
// kernels per iteration take 10.0, 11.5, 12 and 16.7. So every system that fits takes this
// path; what does not fit (more than PT_RESIDENT_ROWS rows per SM, or a record too large) is streamed.
#pragma once

#include "pc_patch.cuh"

// The slots, 64-bit words: [parity][a single sum: 2 words, or two sums: 4][reader][writer].
// Every CTA has a mailbox of its own that all write and only it reads: one array that all
// CTAs read kept each read waiting for its L2 slice (2,900 cycles and more, against about
// 1,200 for a lone L2 access; with the CTAs' words packed side by side up to 7,000).
#define RES_WORDS(n) (2 * 6 * (size_t)(n) * (size_t)(n))

struct ResArgs {
    int V, R, n;                 // rows, rows per patch, patches (= CTAs)
    const PatchDesc *desc;
    const unsigned char *store;
    int rec_cap, share_cap, halo_cap;
    const float *dsc, *dres;
    const int32_t *old_of;
    const uint8_t *named;        // rows in some patch's halo
    const float *dinv;
    float *x;                    // increment, new numbers, packed
    float *r;
    float4 *p;                   // on entry and exit
    unsigned long long *z;       // [V][4] the exchange: z and its epoch
    double *x64;                 // FP64 accumulator, original numbers (mixed), or null
    double rr_last, refresh2;    // leave when rr <= rr_last * refresh2 at a check (mixed)
    int iter_last, refresh_every, check_every;
    unsigned long long *slots;   // RES_WORDS(n)
    unsigned *abort_flag;        // a wait of the launch that began at this epoch gave up
    unsigned epoch0;             // every epoch in slots and z is below this
    pc_scalars *sc;
    uint32_t *err;
    long long budget;
};

__device__ __forceinline__ unsigned long long res_word(float v, unsigned epoch)
{
    return ((unsigned long long)__float_as_uint(v) << 32) | epoch;
}

// Whether a wait should give up: looked at before the first read and then every 16th (every
// 256th also for another CTA's abort), so a budget of a few cycles makes every CTA give up.
__device__ __forceinline__ bool res_give_up(const ResArgs &a, unsigned tries, long long t0)
{
    if ((tries & 15u) != 0u) return false;
    if (clock64() - t0 > a.budget) {
        *(volatile unsigned *)a.abort_flag = a.epoch0;
        return true;
    }
    return (tries & 255u) == 240u && *(volatile unsigned *)a.abort_flag == a.epoch0;
}

// Sum K double-float pairs over the grid, in a fixed order; false (in every thread) when a
// wait gave up. hi/lo: this thread's terms in, the totals out, in every thread.
template <int K>
__device__ __forceinline__ bool res_sum(const ResArgs &a, unsigned epoch, float (&hi)[K], float (&lo)[K])
{
    __shared__ float2 s_w[K][32], s_g[K][32];
    __shared__ int s_bad;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nw = blockDim.x >> 5;
    unsigned long long *base = a.slots + ((size_t)((epoch >> 1) & 1u) * 6 + (K == 1 ? 0 : 2)) * a.n * a.n;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        pc_warp_sum_df(hi[k], lo[k]);
        if (lane == 0) s_w[k][warp] = make_float2(hi[k], lo[k]);
    }
    if (t == 0) s_bad = 0;
    __syncthreads();
    const int gw = min(nw, (a.n + 31) / 32);  // warps that write to and read from the others
    if (warp < gw) {
#pragma unroll
        for (int k = 0; k < K; ++k) {  // the CTA's total, in each of these warps
            float2 w = lane < nw ? s_w[k][lane] : make_float2(0.f, 0.f);
            pc_warp_sum_df(w.x, w.y);
            hi[k] = w.x;
            lo[k] = w.y;
        }
        for (int i = t; i < a.n; i += 32 * gw) {
            unsigned long long *s = base + ((size_t)i * a.n + blockIdx.x) * (2 * K);
#pragma unroll
            for (int k = 0; k < K; ++k)
                asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(s + 2 * k),
                             "l"(res_word(hi[k], epoch)), "l"(res_word(lo[k], epoch))
                             : "memory");
        }
    }
    float gh[K], gl[K];
#pragma unroll
    for (int k = 0; k < K; ++k) gh[k] = gl[k] = 0.f;
    const long long t0 = clock64();
    for (int i = warp < gw ? t : a.n; i < a.n; i += 32 * gw) {
        const unsigned long long *s = base + ((size_t)blockIdx.x * a.n + i) * (2 * K);
        for (unsigned tries = 0;; ++tries) {
            if (res_give_up(a, tries, t0)) {
                s_bad = 1;
                break;
            }
            unsigned long long w[2 * K];
            bool ready = true;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];"
                             : "=l"(w[2 * k]), "=l"(w[2 * k + 1])
                             : "l"(s + 2 * k)
                             : "memory");
                ready = ready && (unsigned)w[2 * k] == epoch && (unsigned)w[2 * k + 1] == epoch;
            }
            if (ready) {
#pragma unroll
                for (int k = 0; k < K; ++k)
                    pc_df_add(gh[k], gl[k], __uint_as_float((unsigned)(w[2 * k] >> 32)),
                              __uint_as_float((unsigned)(w[2 * k + 1] >> 32)));
                break;
            }
        }
    }
    if (warp < gw)
#pragma unroll
        for (int k = 0; k < K; ++k) {
            pc_warp_sum_df(gh[k], gl[k]);
            if (lane == 0) s_g[k][warp] = make_float2(gh[k], gl[k]);
        }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        hi[k] = lo[k] = 0.f;
        for (int w = 0; w < gw; ++w) pc_df_add(hi[k], lo[k], s_g[k][w].x, s_g[k][w].y);
    }
    return s_bad == 0;
}

// A z row: four 64-bit words, (x, epoch) (y, epoch) (z, epoch) and one unused.
__device__ __forceinline__ void res_put_z(unsigned long long *z, float x, float y, float w, unsigned epoch)
{
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(z), "l"(res_word(x, epoch)), "l"(res_word(y, epoch))
                 : "memory");
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(z + 2), "l"(res_word(w, epoch)) : "memory");
}
__device__ __forceinline__ bool res_get_z(const unsigned long long *z, unsigned epoch, float (&v)[3])
{
    unsigned long long w[3];
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w[0]), "=l"(w[1]) : "l"(z) : "memory");
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w[2]) : "l"(z + 2) : "memory");
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        v[k] = __uint_as_float((unsigned)(w[k] >> 32));
        ok = ok && (unsigned)w[k] == epoch;
    }
    return ok;
}

// z = M^-1 r with the row's preconditioner in registers.
template <bool BLOCK>
__device__ __forceinline__ void res_precond(const float *D, const float *r, float *z)
{
    if (BLOCK) {
        z[0] = D[0] * r[0] + D[1] * r[1] + D[2] * r[2];
        z[1] = D[3] * r[0] + D[4] * r[1] + D[5] * r[2];
        z[2] = D[6] * r[0] + D[7] * r[1] + D[8] * r[2];
    } else {
        z[0] = D[0] * r[0];
        z[1] = D[1] * r[1];
        z[2] = D[2] * r[2];
    }
}

// PROF: count cycles for pc_spmv_stats (as a flag of the launch it cost 1% of every iteration).
template <int SPLIT, bool BLOCK, bool PROF>
__global__ void __launch_bounds__(1024, 1) pcg_resident_kernel(ResArgs a)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t bar;
    __shared__ int s_fail, s_stop, s_iter;
    __shared__ float s_rz;
    __shared__ long long s_cycles[2];  // thread 0's, in products and in the launch
    unsigned char *rec = smem_raw;
    float4 *share = reinterpret_cast<float4 *>(smem_raw + a.rec_cap);
    const PatchP ps{reinterpret_cast<float *>(smem_raw + a.rec_cap + 16 * a.share_cap), a.R + a.halo_cap};
    float *parts = ps.x + 3 * ps.n;  // [SPLIT - 1][3][R]
    const int t = threadIdx.x, part = t / a.R, lr = t - part * a.R, slice = lr >> 5;
    const int row = blockIdx.x * a.R + lr;
    const bool mine = part == 0 && row < a.V;
    const PatchDesc d = a.desc[blockIdx.x];
    const PatchLayout L = patch_layout(a.R, d);
    const int32_t *halo = reinterpret_cast<const int32_t *>(rec + L.halo);
    if (t == 0) {
        s_fail = 0;
        if (PROF) {
            s_cycles[0] = 0;
            s_cycles[1] = -clock64();
        }
        mbar_init(&bar, 1);
        mbar_fence_init();
    }
    __syncthreads();
    if (t == 0) {
        mbar_arrive_expect_tx(&bar, (uint32_t)d.bytes);
        // a bulk copy counts its bytes on the barrier; parts of 64 KB keep each below its range
        for (int o = 0; o < d.bytes; o += 65536)
            bulk_g2s(rec + o, a.store + d.offset + o, (uint32_t)min(65536, d.bytes - o), &bar);
        share[d.n_own] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float x[3] = {0.f, 0.f, 0.f}, r[3] = {0.f, 0.f, 0.f}, Dm[BLOCK ? 9 : 3], s = 0.f;
    float4 pi = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row < a.V) pi = a.p[row];
    if (part == 0) {
#pragma unroll
        for (int k = 0; k < (BLOCK ? 9 : 3); ++k) Dm[k] = 0.f;
        if (row < a.V) {
            s = a.dsc[row];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                x[k] = a.x[3ll * row + k];
                r[k] = a.r[3ll * row + k];
            }
            if (BLOCK) {
#pragma unroll
                for (int k = 0; k < 9; ++k) Dm[k] = a.dinv[12ll * row + 4 * (k / 3) + k % 3];
            } else {
#pragma unroll
                for (int k = 0; k < 3; ++k) Dm[k] = a.dinv[3ll * row + k];
            }
        }
        ps.put(lr, pi);
    }
    if (t == 0) {
        s_rz = (float)a.sc->rz;
        s_iter = a.sc->iter;
        s_stop = a.sc->done != 0;
    }
    if (!mbar_wait_bounded(&bar, 0u, PT_WAIT_BUDGET)) s_fail = 1;
    __syncthreads();
    if (s_fail) {  // the record never came: nothing was written
        if (t == 0) {
            atomicOr(a.err, PC_DERR_TIMEOUT);
            *(volatile unsigned *)a.abort_flag = a.epoch0;
            a.sc->status = PC_ERR_TIMEOUT;
            a.sc->done = 1;
        }
        return;
    }
    const bool named = mine && a.named[row] != 0;  // other patches want the row's z
    float rz = s_rz;
    int iter = s_iter;
    bool stop = s_stop != 0;
    if (!stop)
        for (int i = t; i < d.n_halo; i += blockDim.x) ps.put(a.R + i, a.p[halo[i]]);
    __syncthreads();
    unsigned epoch = a.epoch0;
    float alpha = 0.f, beta = 0.f;
    bool timeout = false;
    while (!stop) {
        // ---- q = A p
        if (PROF && t == 0) s_cycles[0] -= clock64();
        float q[3] = {0.f, 0.f, 0.f};
        patch_row_keep<SPLIT, 2>(rec, L, share, ps, slice, pi, part, q[0], q[1], q[2]);
        __syncthreads();
        patch_row_shares<SPLIT>(rec, L, share, a.R, slice, part, q[0], q[1], q[2]);
        if (SPLIT > 1) {
            if (part > 0)
#pragma unroll
                for (int k = 0; k < 3; ++k) parts[((part - 1) * 3 + k) * a.R + lr] = q[k];
            __syncthreads();
            if (part == 0)
#pragma unroll
                for (int w = 0; w < SPLIT - 1; ++w)
#pragma unroll
                    for (int k = 0; k < 3; ++k) q[k] += parts[(w * 3 + k) * a.R + lr];
        }
        float hi[1] = {0.f}, lo[1] = {0.f};
        if (mine) {
            if (s > 0.f) {
                q[0] = fmaf(s, pi.x, q[0]);
                q[1] = fmaf(s, pi.y, q[1]);
                q[2] = fmaf(s, pi.z, q[2]);
            } else {
                const float *D = a.dres + 9ll * a.old_of[row];
                q[0] = fmaf(D[0], pi.x, fmaf(D[1], pi.y, fmaf(D[2], pi.z, q[0])));
                q[1] = fmaf(D[3], pi.x, fmaf(D[4], pi.y, fmaf(D[5], pi.z, q[1])));
                q[2] = fmaf(D[6], pi.x, fmaf(D[7], pi.y, fmaf(D[8], pi.z, q[2])));
            }
            hi[0] = fmaf(pi.x, q[0], fmaf(pi.y, q[1], pi.z * q[2]));
        }
        if (PROF && t == 0) s_cycles[0] += clock64();
        if (!res_sum<1>(a, ++epoch, hi, lo)) {
            timeout = true;
            break;
        }
        // ---- x, r, z
        const float pq = __fadd_rn(hi[0], lo[0]);
        alpha = rz / pq;
        const bool bad = !(pq > 0.f) || !isfinite(alpha);
        if (bad) alpha = 0.f;
        float z[3] = {0.f, 0.f, 0.f};
        float h2[2] = {0.f, 0.f}, l2[2] = {0.f, 0.f};
        if (mine) {
            x[0] = fmaf(alpha, pi.x, x[0]);
            x[1] = fmaf(alpha, pi.y, x[1]);
            x[2] = fmaf(alpha, pi.z, x[2]);
#pragma unroll
            for (int k = 0; k < 3; ++k) r[k] = fmaf(-alpha, q[k], r[k]);
            res_precond<BLOCK>(Dm, r, z);
            h2[0] = fmaf(r[0], z[0], fmaf(r[1], z[1], r[2] * z[2]));
            h2[1] = fmaf(r[0], r[0], fmaf(r[1], r[1], r[2] * r[2]));
            if (named) res_put_z(a.z + 4ll * row, z[0], z[1], z[2], epoch + 1);
        }
        if (!res_sum<2>(a, ++epoch, h2, l2)) {
            timeout = true;
            break;
        }
        const float rz_new = __fadd_rn(h2[0], l2[0]);
        beta = rz_new / rz;
        rz = rz_new;
        ++iter;
        const bool check = a.x64 && iter % a.check_every == 0;
        // FP64 belongs to one thread per CTA (its pipe is about 60 times slower than FP32's: in
        // every thread, these few operations took 8 us of an iteration), and its latency
        // hides behind the gathers below
        if (t == 0) {
            const double rr = pc_df_value(h2[1], l2[1]);
            int32_t status = PC_OK;
            bool ended = false;
            if (bad || !isfinite(h2[1]) || !isfinite(beta)) status = PC_ERR_NONFINITE;
            else if (rr <= a.sc->tol2) ended = true;
            else if (iter >= a.sc->max_iter) status = PC_ERR_NOT_CONVERGED;
            ended = ended || status != PC_OK;
            s_stop = ended || (check && (rr <= a.rr_last * a.refresh2 || iter - a.iter_last >= a.refresh_every));
            if (s_stop && blockIdx.x == 0) {
                a.sc->rz = pc_df_value(h2[0], l2[0]);
                a.sc->rr = rr;
                a.sc->pq = pc_df_value(hi[0], lo[0]);
                a.sc->alpha = (double)alpha;
                a.sc->beta = (double)beta;
                a.sc->iter = iter;
                if (status != PC_OK) atomicCAS(&a.sc->status, (int32_t)PC_OK, status);
                if (ended) a.sc->done = 1;
            }
        }
        // ---- p = z + beta p, own rows and halo (also in an iteration that stops the solve: a
        // residual replacement that resumes it corrects p from the old z to the replaced one)
        if (isfinite(beta)) {
            pi = make_float4(0.f, 0.f, 0.f, 0.f);
            if (part == 0) {
                const float px = ps.x[lr], py = ps.x[ps.n + lr], pz = ps.x[2 * ps.n + lr];
                pi = make_float4(fmaf(beta, px, z[0]), fmaf(beta, py, z[1]), fmaf(beta, pz, z[2]), 0.f);
                ps.put(lr, pi);
            }
            // the last threads first: the first ones have their own rows
            const long long t0 = clock64();
            for (int i = (int)blockDim.x - 1 - t; i < d.n_halo; i += blockDim.x) {
                float zh[3];
                for (unsigned tries = 0; !res_get_z(a.z + 4ll * halo[i], epoch, zh); ++tries)
                    if (res_give_up(a, tries + 1, t0)) {
                        s_fail = 1;
                        break;
                    }
                const int c = a.R + i;
                ps.put(c, make_float4(fmaf(beta, ps.x[c], zh[0]), fmaf(beta, ps.x[ps.n + c], zh[1]),
                                      fmaf(beta, ps.x[2 * ps.n + c], zh[2]), 0.f));
            }
        }
        if (check && mine) {
            // the FP32 increment never grows large (as in the streamed schedule's checks)
            const int64_t o = 3ll * a.old_of[row];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                a.x64[o + k] += (double)x[k];
                x[k] = 0.f;
            }
        }
        __syncthreads();
        if (s_fail) {
            timeout = true;
            break;
        }
        stop = s_stop != 0;
        if (part > 0 && row < a.V) pi = make_float4(ps.x[lr], ps.x[ps.n + lr], ps.x[2 * ps.n + lr], 0.f);
    }
    if (timeout) {
        if (t == 0) {
            atomicOr(a.err, PC_DERR_TIMEOUT);
            atomicExch(&a.sc->status, (int32_t)PC_ERR_TIMEOUT);
            a.sc->done = 1;
        }
        return;
    }
    if (epoch == a.epoch0) return;  // the solve had stopped before this launch
    if (PROF && t == 0) {
        atomicMax(&a.sc->prod_cycles, (unsigned long long)s_cycles[0]);
        if (blockIdx.x == 0) a.sc->all_cycles = (unsigned long long)(s_cycles[1] + clock64());
    }
    if (mine) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            a.x[3ll * row + k] = x[k];
            a.r[3ll * row + k] = r[k];
        }
        a.p[row] = pi;
    }
}
