// Value assembly (Sec. 3.2.2 "value filling", Eq. 2-3): element kernels evaluate every
// assembly element once (force and Hessian at x_t) into per-element records, and the
// right-hand side is Eq. 3's h f(x_t + h v_t) to first order, b = h (f(x_t) - h K v_t);
// a thread per off-diagonal block then sums the records on the block's own list, and one per row
// those incident to the row (diagonal and right-hand side), in a fixed order. No atomics: the
// result is deterministic and the matrix is bitwise symmetric.
//
// Precision: the membrane strain G = (F^T F - I)/2 cancels catastrophically in FP32 at
// cloth strains (1e-5..1e-3). It is formed instead as Dm^-T (Ds^T Ds - Dm^T Dm) Dm^-1 with
// the Gram difference of the current and rest edges evaluated in double-float (pairs of
// FP32 values, exact TwoSum / fma-based TwoProduct), so the strain keeps FP32 relative
// accuracy; everything else is plain FP32.
#include <float.h>

#include "pc_internal.cuh"

// ------------------------------------------------------------------------- double-float

struct dfl {
    float hi, lo;
};

__device__ __forceinline__ dfl two_sum(float a, float b)
{
    float s = __fadd_rn(a, b);
    float bb = __fsub_rn(s, a);
    float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}
__device__ __forceinline__ dfl quick_two_sum(float a, float b)
{
    float s = __fadd_rn(a, b);
    float e = __fsub_rn(b, __fsub_rn(s, a));
    return {s, e};
}
__device__ __forceinline__ dfl df_add(dfl a, dfl b)
{
    dfl s = two_sum(a.hi, b.hi);
    float lo = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
    return quick_two_sum(s.hi, lo);
}
__device__ __forceinline__ dfl df_mul(dfl a, dfl b)
{
    float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    return quick_two_sum(p, e);
}
__device__ __forceinline__ dfl df_dot3(const dfl *a, const dfl *b)
{
    return df_add(df_add(df_mul(a[0], b[0]), df_mul(a[1], b[1])), df_mul(a[2], b[2]));
}

// ------------------------------------------------------------------------- small helpers

__device__ __forceinline__ float3 ld3(const float *p, int i) { return make_float3(p[3 * i], p[3 * i + 1], p[3 * i + 2]); }
__device__ __forceinline__ float3 sub(float3 a, float3 b) { return make_float3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ float3 add(float3 a, float3 b) { return make_float3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ __forceinline__ float3 mul(float s, float3 a) { return make_float3(s * a.x, s * a.y, s * a.z); }
__device__ __forceinline__ float dot(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ float3 cross(float3 a, float3 b)
{
    return make_float3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}

// upper-triangular block index of (k, l), k <= l, in a 3-vertex element
__device__ __forceinline__ int tri_blk(int k, int l) { return k == 0 ? l : (k == 1 ? 2 + l : 5); }

// Positive part of a symmetric 2x2 matrix [a b; b c].
__device__ __forceinline__ void sym2_positive(float a, float b, float c, float &pa, float &pb, float &pc)
{
    float m = 0.5f * (a + c);
    float r = sqrtf(0.25f * (a - c) * (a - c) + b * b);
    float l1 = m + r, l2 = m - r;
    if (l2 >= 0.0f) { pa = a; pb = b; pc = c; return; }
    if (l1 <= 0.0f) { pa = pb = pc = 0.0f; return; }
    float v0, v1;
    if (fabsf(b) > 0.0f) {
        if (fabsf(l1 - a) > fabsf(l1 - c)) { v0 = b; v1 = l1 - a; } else { v0 = l1 - c; v1 = b; }
    } else if (a >= c) { v0 = 1.0f; v1 = 0.0f; } else { v0 = 0.0f; v1 = 1.0f; }
    float inv = rsqrtf(v0 * v0 + v1 * v1);
    v0 *= inv;
    v1 *= inv;
    pa = l1 * v0 * v0;
    pb = l1 * v0 * v1;
    pc = l1 * v1 * v1;
}

// ------------------------------------------------------------------------- membrane triangles

// Green strain G = Dm^-T (Gram(edges) - Gram(rest)) Dm^-1 / 2 from exact edge pairs.
__device__ __forceinline__ void strain_from_edges(const dfl *e1, const dfl *e2, const float *rg, const float *dmi,
                                                  float &G00, float &G01, float &G11)
{
    dfl g11 = df_dot3(e1, e1), g22 = df_dot3(e2, e2), g12 = df_dot3(e1, e2);
    float D11 = df_add(g11, {-rg[0], -rg[1]}).hi;
    float D22 = df_add(g22, {-rg[2], -rg[3]}).hi;
    float D12 = df_add(g12, {-rg[4], -rg[5]}).hi;
    // G = 1/2 Dm^-T D Dm^-1 with Dm^-1 = [[d0 d1] [d2 d3]]
    float d0 = dmi[0], d1 = dmi[1], d2 = dmi[2], d3 = dmi[3];
    // M = D Dm^-1
    float m00 = D11 * d0 + D12 * d2, m01 = D11 * d1 + D12 * d3;
    float m10 = D12 * d0 + D22 * d2, m11 = D12 * d1 + D22 * d3;
    G00 = 0.5f * (d0 * m00 + d2 * m10);
    G01 = 0.5f * (d0 * m01 + d2 * m11);
    G11 = 0.5f * (d1 * m01 + d3 * m11);
}

// One thread per triangle, everything at x_t. With F the deformation gradient, g_k the
// shape gradients, Fg_k = F g_k, S+ the clamped stress and c = h^2 A0 (h (h + beta) A0 with
// damping), the Hessian block (k, l) is
//   c (mu Fg_l Fg_k^T + lam Fg_k Fg_l^T + mu (g_k.g_l) F F^T + (g_k.S+ g_l) I),
// so the record holds those factors (32 floats: one 128-byte line) instead of the six
// upper blocks (54 floats), and the rows expand the block they need (tri_block below).
// Record, as eight float4: (c_0, c mu) (c_1, saa) (c_2, sab) (Fg_a, sbb) (Fg_b, gg00)
// (M00 M01 M02 gg01) (M11 M12 M22 gg02) (gg11 gg12 gg22 m), M = c mu F F^T, s = c g.S+ g.
// m is the vertex with the longest gradient and a < b are the other two: the gradients sum to
// zero, and the longest follows from the others without cancellation.
// c_k = h f_k - sum_l (h^2 H_kl) v_l is the element's share of b = h (f - h K v), the
// first-order form of h f(x_t + h v_t) (Eq. 2-3); since each Hessian row sums to zero,
// sum_l H_kl v_l is formed as sum_l H_kl (v_l - v_k).
// Eight consecutive triangles' records are interleaved, quad by quad (tri_quad): lanes that
// read the same quad of neighbouring triangles share a line (assembly at 830k rows: 1,095 us
// with each record a line of its own, 987 interleaved).
// Bound by DRAM (reads 56 B of rest data per triangle, writes 128 B): 1.65M triangles: 64 us
// (523 with 256-byte records stored a float at a time).
#define TE_THREADS 128

__host__ __device__ __forceinline__ int64_t tri_quad(uint32_t id, int quad)
{
    return (int64_t)(PC_TRI_STRIDE / 4) * (id & ~7u) + 8 * quad + (id & 7u);
}

struct TriFactors {
    float Fg[3][3];  // F g_k
    float M[6];      // c mu F F^T, upper: 00 01 02 11 12 22
    float gg[6];     // g_k . g_l, upper: 00 01 02 11 12 22
    float s[6];      // c g_k . S+ g_l, same order
    float cm, cl;    // c mu, c lam
};

// Entry (a, b) of the Hessian block (k, l), k <= l.
__device__ __forceinline__ float tri_entry(const TriFactors &R, int k, int l, int a, int b)
{
    const int m = a == 0 || b == 0 ? a + b : a + b + 1;
    float v = R.gg[tri_blk(k, l)] * R.M[m];
    v = fmaf(R.cm * R.Fg[l][a], R.Fg[k][b], v);
    v = fmaf(R.cl * R.Fg[k][a], R.Fg[l][b], v);
    return a == b ? v + R.s[tri_blk(k, l)] : v;
}

__global__ void __launch_bounds__(TE_THREADS) tri_eval_kernel(int T, const int32_t *__restrict__ tri,
                                                       const float *__restrict__ x, const float *__restrict__ v,
                                                       const float *__restrict__ dmi_all,
                                                       const float *__restrict__ area, const float *__restrict__ rgram,
                                                       float mu, float lam, float h, float hk,
                                                       float4 *__restrict__ out)
{
    const int t = blockIdx.x * TE_THREADS + threadIdx.x;
    if (t < T) {
        int i0 = tri[3 * t], i1 = tri[3 * t + 1], i2 = tri[3 * t + 2];
        const float4 dm = reinterpret_cast<const float4 *>(dmi_all)[t];
        const float dmi[4] = {dm.x, dm.y, dm.z, dm.w};
        float rg[6];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float2 r2 = reinterpret_cast<const float2 *>(rgram)[3ll * t + k];
            rg[2 * k] = r2.x;
            rg[2 * k + 1] = r2.y;
        }
        const float A0 = area[t];
        float x0[3], x1[3], x2[3], v0[3], d1[3], d2[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            x0[a] = x[3 * i0 + a]; x1[a] = x[3 * i1 + a]; x2[a] = x[3 * i2 + a];
            v0[a] = v[3 * i0 + a];
            d1[a] = v[3 * i1 + a] - v0[a];
            d2[a] = v[3 * i2 + a] - v0[a];
        }
        dfl e1[3], e2[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            e1[a] = two_sum(x1[a], -x0[a]);
            e2[a] = two_sum(x2[a], -x0[a]);
        }
        // shape-function gradients: g1 = row 0 of Dm^-1, g2 = row 1, g0 = -g1 - g2
        float g[3][2] = {{-dmi[0] - dmi[2], -dmi[1] - dmi[3]}, {dmi[0], dmi[1]}, {dmi[2], dmi[3]}};
        float G00, G01, G11;
        strain_from_edges(e1, e2, rg, dmi, G00, G01, G11);
        const float tr = G00 + G11;
        const float S00 = 2.0f * mu * G00 + lam * tr, S01 = 2.0f * mu * G01, S11 = 2.0f * mu * G11 + lam * tr;
        float F[3][2];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            F[a][0] = e1[a].hi * dmi[0] + e2[a].hi * dmi[2];
            F[a][1] = e1[a].hi * dmi[1] + e2[a].hi * dmi[3];
        }
        float f[3][3];  // forces at x_t
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float P0 = F[a][0] * S00 + F[a][1] * S01, P1 = F[a][0] * S01 + F[a][1] * S11;
            f[1][a] = -A0 * (P0 * g[1][0] + P1 * g[1][1]);
            f[2][a] = -A0 * (P0 * g[2][0] + P1 * g[2][1]);
            f[0][a] = -(f[1][a] + f[2][a]);
        }
        // Hessian factors at x_t (stress clamped to its positive part in the geometric term)
        float Sp00, Sp01, Sp11;
        sym2_positive(S00, S01, S11, Sp00, Sp01, Sp11);
        TriFactors R;
        const float c = hk * A0;
        R.cm = c * mu;
        R.cl = c * lam;
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int a = 0; a < 3; ++a) R.Fg[k][a] = F[a][0] * g[k][0] + F[a][1] * g[k][1];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = a; b < 3; ++b)
                R.M[a == 0 ? b : a + b + 1] = R.cm * (F[a][0] * F[b][0] + F[a][1] * F[b][1]);
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int l = k; l < 3; ++l) {
                R.gg[tri_blk(k, l)] = g[k][0] * g[l][0] + g[k][1] * g[l][1];
                R.s[tri_blk(k, l)] = c * (g[k][0] * (Sp00 * g[l][0] + Sp01 * g[l][1]) +
                                          g[k][1] * (Sp01 * g[l][0] + Sp11 * g[l][1]));
            }
        // right-hand-side shares c_k = h f_k - sum_{l != k} Hs_kl (v_l - v_k)
        float ck[3][3];
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int a = 0; a < 3; ++a) ck[k][a] = h * f[k][a];
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int l = k + 1; l < 3; ++l) {
                float d[3];  // v_l - v_k
#pragma unroll
                for (int a = 0; a < 3; ++a) d[a] = (l == 1 ? d1[a] : d2[a]) - (k == 1 ? d1[a] : 0.f);
#pragma unroll
                for (int a = 0; a < 3; ++a)
#pragma unroll
                    for (int b = 0; b < 3; ++b) {
                        const float e = tri_entry(R, k, l, a, b);
                        ck[k][a] = fmaf(-e, d[b], ck[k][a]);
                        ck[l][b] = fmaf(e, d[a], ck[l][b]);
                    }
            }
        const int m = R.gg[0] >= R.gg[3] && R.gg[0] >= R.gg[5] ? 0 : R.gg[3] >= R.gg[5] ? 1 : 2;
        float Fa[3], Fb[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            Fa[a] = m == 0 ? R.Fg[1][a] : R.Fg[0][a];
            Fb[a] = m == 2 ? R.Fg[1][a] : R.Fg[2][a];
        }
        float4 *o = out + tri_quad(t, 0);
        o[0] = make_float4(ck[0][0], ck[0][1], ck[0][2], R.cm);
        o[8] = make_float4(ck[1][0], ck[1][1], ck[1][2], m == 0 ? R.s[3] : R.s[0]);
        o[16] = make_float4(ck[2][0], ck[2][1], ck[2][2], m == 0 ? R.s[4] : m == 1 ? R.s[2] : R.s[1]);
        o[24] = make_float4(Fa[0], Fa[1], Fa[2], m == 2 ? R.s[3] : R.s[5]);
        o[32] = make_float4(Fb[0], Fb[1], Fb[2], R.gg[0]);
        o[40] = make_float4(R.M[0], R.M[1], R.M[2], R.gg[1]);
        o[48] = make_float4(R.M[3], R.M[4], R.M[5], R.gg[2]);
        o[56] = make_float4(R.gg[3], R.gg[4], R.gg[5], __int_as_float(m));
    }
}

// The factors of triangle record `id` (cl_cm = lam / mu).
__device__ __forceinline__ TriFactors tri_load(const float4 *__restrict__ buf, uint32_t id, float cl_cm)
{
    const float4 *r = buf + tri_quad(id, 0);
    const float cm = r[0].w, saa = r[8].w, sab = r[16].w;
    const float4 fa = r[24], fb = r[32], m0 = r[40], m1 = r[48], q = r[56];
    const int m = __float_as_int(q.w);
    const float Fa[3] = {fa.x, fa.y, fa.z}, Fb[3] = {fb.x, fb.y, fb.z}, sbb = fa.w;
    TriFactors R;
    R.cm = cm;
    R.cl = cl_cm * cm;
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const float Fm = -(Fa[e] + Fb[e]);
        R.Fg[0][e] = m == 0 ? Fm : Fa[e];
        R.Fg[1][e] = m == 0 ? Fa[e] : m == 1 ? Fm : Fb[e];
        R.Fg[2][e] = m == 2 ? Fm : Fb[e];
    }
    R.M[0] = m0.x; R.M[1] = m0.y; R.M[2] = m0.z;
    R.M[3] = m1.x; R.M[4] = m1.y; R.M[5] = m1.z;
    R.gg[0] = fb.w; R.gg[1] = m0.w; R.gg[2] = m1.w;
    R.gg[3] = q.x; R.gg[4] = q.y; R.gg[5] = q.z;
    const float sam = -(saa + sab), sbm = -(sab + sbb), smm = -(sam + sbm);
    R.s[0] = m == 0 ? smm : saa;
    R.s[1] = m == 2 ? sab : sam;                       // (0, 1): m, a | a, m | a, b
    R.s[2] = m == 1 ? sab : m == 0 ? sbm : sam;        // (0, 2): m, b | a, b | a, m
    R.s[3] = m == 0 ? saa : m == 1 ? smm : sbb;
    R.s[4] = m == 0 ? sab : sbm;                       // (1, 2): a, b | m, b | b, m
    R.s[5] = m == 2 ? smm : sbb;
    return R;
}

// ------------------------------------------------------------------------- bending hinges

// theta = atan2((n1 x n2).e, n1.n2) of a hinge given relative vectors a1 = x1-x3,
// a2 = x2-x3, a4 = x4-x3 (x1, x2 wings; x3, x4 edge) and its gradient
// (Bridson, Marino and Fedkiw 2003).
__device__ __forceinline__ float hinge_angle_grad(float3 a1, float3 a2, float3 a4, float3 *grad)
{
    float3 E = a4;
    float3 N1 = cross(a1, sub(a1, a4));            // (x1-x3) x (x1-x4)
    float3 N2 = cross(sub(a2, a4), a2);            // (x2-x4) x (x2-x3)
    float lE = sqrtf(dot(E, E));
    float n1sq = dot(N1, N1), n2sq = dot(N2, N2);
    float in1 = rsqrtf(n1sq), in2 = rsqrtf(n2sq);
    float3 c = cross(N1, N2);
    float s = dot(c, E) * (in1 * in2 / lE);
    float co = dot(N1, N2) * (in1 * in2);
    float theta = atan2f(s, co);
    float3 u1 = mul(lE / n1sq, N1), u2 = mul(lE / n2sq, N2);
    float s13 = dot(sub(a1, a4), E) / lE, s23 = dot(sub(a2, a4), E) / lE;
    float s14 = dot(a1, E) / lE, s24 = dot(a2, E) / lE;
    float3 u3 = add(mul(s13 / n1sq, N1), mul(s23 / n2sq, N2));
    float3 u4 = add(mul(-s14 / n1sq, N1), mul(-s24 / n2sq, N2));
    grad[0] = mul(-1.0f, u1);
    grad[1] = mul(-1.0f, u2);
    grad[2] = mul(-1.0f, u3);
    grad[3] = mul(-1.0f, u4);
    return theta;
}

// One thread per hinge, at x_t. With q_k = h sqrt(2 kb c_h) grad_k(theta) (h^2 -> h (h + beta)
// with damping) the Gauss-Newton Hessian block (k, l) is q_k q_l^T, and the right-hand-side
// contribution h f_k - q_k (q . v) is q_k times one scalar w, because f_k is parallel to
// grad_k too: h f_k = -h (2 kb c_h) (theta - theta_rest) grad_k. Record: four float4 (q_k, w),
// 64 bytes, instead of 12 contributions and 12 gradients. The gradient sums to zero over
// the four vertices, so q . v uses velocities relative to edge0. hb = h + beta, hk = h hb,
// ih = h / hk. Bound by DRAM (reads 24 B of rest data and writes 64 B per hinge); 2.48M hinges:
// 60 us (247 with 96-byte records).
__global__ void __launch_bounds__(128) hinge_eval_kernel(int H, const int32_t *__restrict__ hinge,
                                                         const float *__restrict__ x, const float *__restrict__ v,
                                                         const float *__restrict__ hcoef,
                                                         const float *__restrict__ hrest, float h, float hb, float hk,
                                                         float ih, float *__restrict__ out)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= H) return;
    const int4 hv = reinterpret_cast<const int4 *>(hinge)[i];
    const int vid[4] = {hv.x, hv.y, hv.z, hv.w};
    float3 X[4], W[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) { X[k] = ld3(x, vid[k]); W[k] = ld3(v, vid[k]); }
    const float kc = hcoef[i];
    float3 grad[4];
    // positions relative to edge0
    float3 a1 = sub(X[0], X[2]), a2 = sub(X[1], X[2]), a4 = sub(X[3], X[2]);
    float th = hinge_angle_grad(a1, a2, a4, grad);
    const float hkc = hk * kc;
    // (the force needs sc where its square, which only the Hessian has, leaves FP32's range)
    const float sc = hkc > 1e-30f ? sqrtf(hkc) : sqrtf(h * kc) * sqrtf(hb);
    float3 q[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) q[k] = mul(sc, grad[k]);
    float qv = dot(q[0], sub(W[0], W[2])) + dot(q[1], sub(W[1], W[2])) + dot(q[3], sub(W[3], W[2]));
    // h f_k = -h kc (theta - rest) grad_k = -(h / hk) sc (theta - rest) q_k
    const float w = -ih * sc * (th - hrest[i]) - qv;
    float4 *o = reinterpret_cast<float4 *>(out) + (int64_t)(PC_HINGE_STRIDE / 4) * i;
#pragma unroll
    for (int k = 0; k < 4; ++k) o[k] = make_float4(q[k].x, q[k].y, q[k].z, w);
}

// ------------------------------------------------------------------------- contacts

// One thread per pair (p; a, b, c). Record: right-hand-side contributions (12), unit
// normal n of (a, b, c) at x (3), weights (3), h^2 kc (1) (h (h + beta) kc with Rayleigh
// damping; 0 for an inactive thickness contact), 1 when one of the four vertices is pinned. With s = (1, -w_a, -w_b, -w_c) the
// Hessian block (k, l) is h^2 kc s_k s_l n n^T. The hold penalty is zero at x_t (d = d0)
// and linear in x, so its contribution h (f - h K v) is -h^2 kc (n . sum_l s_l v_l) s_k n;
// the thickness penalty adds its force at x_t, h kc (delta - d) s_k n.
__global__ void contact_eval_kernel(int P, const int32_t *__restrict__ pairs, const float *__restrict__ wts,
                                    const float *__restrict__ x, const float *__restrict__ v, float kc, float h,
                                    float hk, float thick, const uint8_t *__restrict__ pinned,
                                    float *__restrict__ out)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P) return;
    int vid[4] = {pairs[4 * i], pairs[4 * i + 1], pairs[4 * i + 2], pairs[4 * i + 3]};
    float w[3] = {wts[3 * i], wts[3 * i + 1], wts[3 * i + 2]};
    float3 xa = ld3(x, vid[1]);
    float3 n = cross(sub(ld3(x, vid[2]), xa), sub(ld3(x, vid[3]), xa));
    n = mul(rsqrtf(dot(n, n)), n);
    float s[4] = {1.0f, -w[0], -w[1], -w[2]};
    // one-sided thickness model: n turned towards p at x_t, force h kc (delta - d) at x_t
    // while d < delta, no stiffness otherwise; hold penalty (delta = 0): no force at x_t
    float kc_eff = kc, fd = 0.f;
    if (thick > 0.f) {
        float3 r = make_float3(0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 4; ++k) r = add(r, mul(s[k], ld3(x, vid[k])));
        float dt = dot(n, r);
        if (dt < 0.f) {
            n = mul(-1.0f, n);
            dt = -dt;
        }
        if (dt < thick) fd = h * kc * (thick - dt);
        else kc_eff = 0.f;
    }
    float3 rv = make_float3(0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 4; ++k) rv = add(rv, mul(s[k], ld3(v, vid[k])));
    float dd = dot(n, rv);  // n . sum_l s_l v_l
    float *o = out + (int64_t)PC_CONTACT_STRIDE * i;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float fk = (fd - hk * kc_eff * dd) * s[k];
        o[3 * k] = fk * n.x;
        o[3 * k + 1] = fk * n.y;
        o[3 * k + 2] = fk * n.z;
    }
    o[12] = n.x; o[13] = n.y; o[14] = n.z;
    o[15] = w[0]; o[16] = w[1]; o[17] = w[2];
    o[18] = hk * kc_eff;
    o[19] = pinned[vid[0]] || pinned[vid[1]] || pinned[vid[2]] || pinned[vid[3]] ? 1.0f : 0.0f;
}

// ------------------------------------------------------------------------- row reduction

#define RR_ROWS 32                     // rows per CTA
#define RR_FEW_ROWS 8                  // where there are too few rows to fill the GPU with such CTAs
#define RR_THREADS 128
#define RR_CTAS_PER_SM 9

// Contributions to one block (row, col), col != row, from the mesh's elements, in incidence
// order: the static list of (type, k, l, id) codes that pc_create made for the block
// (value_lists_kernel in pc_pattern.cu). Every product is rounded before it is added; block
// (col, row) has the same elements in the same order and the products commute, so A is
// bitwise symmetric.
__device__ __forceinline__ void add_static(const uint32_t *__restrict__ codes, int c0, int c1,
                                           const float4 *__restrict__ tri_buf, const float4 *__restrict__ hinge_buf,
                                           float cl_cm, float acc[9])
{
    for (int c = c0; c < c1; ++c) {
        const uint32_t code = codes[c];
        const int k = (int)((code >> 29) & 3u), l = (int)((code >> 27) & 3u);
        const uint32_t id = code & PC_CODE_ID;
        if (code & PC_CODE_HINGE) {
            const float4 qk = hinge_buf[4ll * id + k], ql = hinge_buf[4ll * id + l];
            const float a[3] = {qk.x, qk.y, qk.z}, b[3] = {ql.x, ql.y, ql.z};
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j) acc[3 * i + j] = __fadd_rn(acc[3 * i + j], __fmul_rn(a[i], b[j]));
        } else {
            const TriFactors R = tri_load(tri_buf, id, cl_cm);
            // the block of the vertex pair in its canonical order (lower local index first),
            // transposed for the other row
            const int lo = min(k, l), hi = max(k, l);
            float F0[3], F1[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                F0[a] = lo == 0 ? R.Fg[0][a] : R.Fg[1][a];
                F1[a] = hi == 1 ? R.Fg[1][a] : R.Fg[2][a];
            }
            const float gg = lo == 1 ? R.gg[4] : (hi == 1 ? R.gg[1] : R.gg[2]);
            const float s = lo == 1 ? R.s[4] : (hi == 1 ? R.s[1] : R.s[2]);
            float B[9];
            const float m[9] = {R.M[0], R.M[1], R.M[2], R.M[1], R.M[3], R.M[4], R.M[2], R.M[4], R.M[5]};
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    float v = __fmul_rn(gg, m[3 * a + b]);
                    v = fmaf(__fmul_rn(R.cm, F1[a]), F0[b], v);
                    v = fmaf(__fmul_rn(R.cl, F0[a]), F1[b], v);
                    B[3 * a + b] = a == b ? __fadd_rn(v, s) : v;
                }
            const bool tr = k > l;
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b) acc[3 * a + b] = __fadd_rn(acc[3 * a + b], tr ? B[3 * b + a] : B[3 * a + b]);
        }
    }
}

// Contributions of the row's contacts to block (row, col), in contact order. Every block of the row
// looks at all of them, so four are in flight (12,288 rows of 48 contacts and 28 blocks: the values
// 260 -> 218 us, 830k rows of 16 contacts 2,566 -> 2,354).
__device__ __forceinline__ void add_contacts(const uint32_t *__restrict__ cinc, int c0, int c1,
                                             const int32_t *__restrict__ pairs, const float *__restrict__ cont_buf,
                                             int col, float acc[9])
{
    for (int i = c0; i < c1; i += 4) {
        uint32_t ref[4];
        int l[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) ref[u] = cinc[min(i + u, c1 - 1)];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int32_t *pv = pairs + 4ll * pc_ref_id(ref[u]);
            const int v0 = pv[0], v1 = pv[1], v2 = pv[2], v3 = pv[3];
            l[u] = i + u >= c1 ? -1 : v0 == col ? 0 : v1 == col ? 1 : v2 == col ? 2 : v3 == col ? 3 : -1;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (l[u] < 0) continue;
            const int k = (int)pc_ref_local(ref[u]);
            const float *o = cont_buf + (int64_t)PC_CONTACT_STRIDE * pc_ref_id(ref[u]);
            const float sk = k == 0 ? 1.0f : -o[14 + k], sl = l[u] == 0 ? 1.0f : -o[14 + l[u]];
            const float cs = o[18] * (sk * sl);
            const float n[3] = {o[12], o[13], o[14]};
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b)
                    acc[3 * a + b] = __fadd_rn(acc[3 * a + b], __fmul_rn(cs, __fmul_rn(n[a], n[b])));
        }
    }
}

struct RowArgs {
    int V;
    const int32_t *rp, *ci;            // this step's pattern
    const int32_t *srp, *scol;         // static pattern
    const int32_t *lptr;               // [static blocks + 1] contributions of each static block
    const uint32_t *codes;
    const int32_t *vinc_ptr;
    const uint32_t *vinc;
    const int32_t *cinc_ptr;
    const uint32_t *cinc;
    const int32_t *pairs;
    const float4 *tri_buf;
    const float4 *hinge_buf;
    const float *cont_buf;
    const float *mass;
    const uint8_t *pinned, *pin_adj;   // pinned vertex; some static neighbour is pinned
    float gx, gy, gz, h, md, ha, cl_cm;
    const float *v;
    float *vals, *b, *dres;
};

// The unzeroed block at dynamic slot `slot` of `row` (column `col` != row).
__device__ __forceinline__ void row_block(const RowArgs &a, int row, int slot, int col, int s0, int s1, int t0, int t1,
                                          int n0, int n1, float acc[9])
{
#pragma unroll
    for (int q = 0; q < 9; ++q) acc[q] = 0.f;
    int ss = t0 + (slot - s0);  // static slot: the same place unless contacts added columns to the row
    if (s1 - s0 != t1 - t0) {
        int lo = t0, hi = t1;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (a.scol[mid] < col) lo = mid + 1; else hi = mid;
        }
        ss = lo < t1 && a.scol[lo] == col ? lo : -1;
    }
    if (ss >= 0) add_static(a.codes, a.lptr[ss], a.lptr[ss + 1], a.tri_buf, a.hinge_buf, a.cl_cm, acc);
    if (n1 > n0) add_contacts(a.cinc, n0, n1, a.pairs, a.cont_buf, col, acc);
}

// One CTA per 32 rows (ROWS). Warp 0 first forms the rows' diagonal blocks, right-hand sides and
// difference-form diagonals, one thread per row over the row's incident elements; the
// other blocks go one per thread, over the block's own contribution list, in chunks of 32
// handed out by a shared counter (warp 0 joins when its rows are done; which warp takes a
// chunk does not change any sum).
// Bound by L1 and L2: 44 B per block written (vals and its column read), about 5
// contributions of 64..128 B per block read through L1, a line looked up for nearly every
// lane. So L1 gets all of an SM's memory: blocks are written where they belong (a warp's 32
// blocks are 1,152 consecutive bytes), and 56 registers allow nine CTAs per SM. At 830k rows /
// 10.9M blocks, the whole assembly: 827 us; 987 with the blocks staged in shared memory for
// whole-line stores (879 unstaged at 64 registers, 891 at 40). Also slower: records copied to
// shared memory first, a thread per row that adds each element to its blocks in shared memory,
// CTAs of 256 threads (921). A warp per row that staged every expanded block, each lane
// comparing all of them with its column, took 2,825 us for this kernel alone.
// Fewer rows than fill the GPU with such CTAs once are latency, and longest where rows have many
// contacts: CTAs of 8 rows, and registers for four of a row's contacts in flight (12,288 rows of 48
// contacts 218 -> 167 us, 4,096 rows of 0.08 with the pattern 92.4 -> 87.4; 49,152 rows of 47 495 -> 400,
// but 271,803 rows of 12 665 -> 764).
template <int ROWS>
__global__ void __launch_bounds__(RR_THREADS, ROWS == RR_ROWS ? RR_CTAS_PER_SM : 6) row_reduce_kernel(RowArgs a)
{
    __shared__ int s_rp[ROWS + 1], s_sp[ROWS + 1], s_cp[ROWS + 1];
    __shared__ int s_next;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r0 = blockIdx.x * ROWS, nr = min(ROWS, a.V - r0);
    for (int i = threadIdx.x; i <= nr; i += blockDim.x) {
        s_rp[i] = a.rp[r0 + i];
        s_sp[i] = a.srp[r0 + i];
        s_cp[i] = a.cinc_ptr[r0 + i];
    }
    if (threadIdx.x == 0) s_next = 0;
    __syncthreads();
    const int b0 = s_rp[0], nblk = s_rp[nr] - b0;

    if (warp == 0 && lane < nr) {
        const int row = r0 + lane;
        const int s0 = s_rp[lane], s1 = s_rp[lane + 1], t0 = s_sp[lane], t1 = s_sp[lane + 1];
        const int n0 = s_cp[lane], n1 = s_cp[lane + 1];
        const float m = a.mass[row];
        const float mA = a.md * m;  // diagonal mass term (1 + h alpha) m of an unpinned row
        const bool prow = a.pinned[row] != 0;
        float f[3] = {0.f, 0.f, 0.f};
        float u[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // upper triangle 00 01 02 11 12 22
        const int i1 = a.vinc_ptr[row + 1];
        for (int i = a.vinc_ptr[row]; i < i1; ++i) {
            const uint32_t ref = a.vinc[i], k = pc_ref_local(ref), id = pc_ref_id(ref);
            if (pc_ref_type(ref) == PC_REF_HINGE) {
                const float4 q = a.hinge_buf[4ll * id + k];
                f[0] = fmaf(q.x, q.w, f[0]);
                f[1] = fmaf(q.y, q.w, f[1]);
                f[2] = fmaf(q.z, q.w, f[2]);
                u[0] = __fadd_rn(u[0], __fmul_rn(q.x, q.x));
                u[1] = __fadd_rn(u[1], __fmul_rn(q.x, q.y));
                u[2] = __fadd_rn(u[2], __fmul_rn(q.x, q.z));
                u[3] = __fadd_rn(u[3], __fmul_rn(q.y, q.y));
                u[4] = __fadd_rn(u[4], __fmul_rn(q.y, q.z));
                u[5] = __fadd_rn(u[5], __fmul_rn(q.z, q.z));
            } else {
                const float4 c = a.tri_buf[tri_quad(id, k)];
                f[0] += c.x;
                f[1] += c.y;
                f[2] += c.z;
                const TriFactors R = tri_load(a.tri_buf, id, a.cl_cm);
                float F[3];
#pragma unroll
                for (int e = 0; e < 3; ++e) F[e] = k == 0 ? R.Fg[0][e] : k == 1 ? R.Fg[1][e] : R.Fg[2][e];
                const float gg = k == 0 ? R.gg[0] : k == 1 ? R.gg[3] : R.gg[5];
                const float s = k == 0 ? R.s[0] : k == 1 ? R.s[3] : R.s[5];
                const float cf = R.cm + R.cl;
                u[0] += fmaf(cf * F[0], F[0], fmaf(gg, R.M[0], s));
                u[1] += fmaf(cf * F[0], F[1], gg * R.M[1]);
                u[2] += fmaf(cf * F[0], F[2], gg * R.M[2]);
                u[3] += fmaf(cf * F[1], F[1], fmaf(gg, R.M[3], s));
                u[4] += fmaf(cf * F[1], F[2], gg * R.M[4]);
                u[5] += fmaf(cf * F[2], F[2], fmaf(gg, R.M[5], s));
            }
        }
        bool adj = a.pin_adj[row] != 0;
        constexpr int W = ROWS == RR_ROWS ? 1 : 4;  // contacts in flight (registers)
        for (int i = n0; i < n1; i += W) {
            uint32_t ref[W];
            float4 p[W], q[W];  // (n, w_a) (w_b, w_c, scale, pinned)
            float g[W][3], sk[W];
#pragma unroll
            for (int w = 0; w < W; ++w) ref[w] = a.cinc[min(i + w, n1 - 1)];
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const float4 *o = reinterpret_cast<const float4 *>(a.cont_buf + (int64_t)PC_CONTACT_STRIDE * pc_ref_id(ref[w]));
                const int k = (int)pc_ref_local(ref[w]);
                p[w] = o[3];
                q[w] = o[4];
                const float *c = reinterpret_cast<const float *>(o) + 3 * k;
                g[w][0] = c[0];
                g[w][1] = c[1];
                g[w][2] = c[2];
                sk[w] = k == 0 ? 1.0f : k == 1 ? -p[w].w : k == 2 ? -q[w].x : -q[w].y;
            }
#pragma unroll
            for (int w = 0; w < W; ++w) {
                if (i + w >= n1) break;
                f[0] += g[w][0];
                f[1] += g[w][1];
                f[2] += g[w][2];
                const float cs = q[w].z * (sk[w] * sk[w]);
                const float n[3] = {p[w].x, p[w].y, p[w].z};
                u[0] = __fadd_rn(u[0], __fmul_rn(cs, __fmul_rn(n[0], n[0])));
                u[1] = __fadd_rn(u[1], __fmul_rn(cs, __fmul_rn(n[0], n[1])));
                u[2] = __fadd_rn(u[2], __fmul_rn(cs, __fmul_rn(n[0], n[2])));
                u[3] = __fadd_rn(u[3], __fmul_rn(cs, __fmul_rn(n[1], n[1])));
                u[4] = __fadd_rn(u[4], __fmul_rn(cs, __fmul_rn(n[1], n[2])));
                u[5] = __fadd_rn(u[5], __fmul_rn(cs, __fmul_rn(n[2], n[2])));
                adj |= q[w].w != 0.f;
            }
        }
        float B[9] = {u[0], u[1], u[2], u[1], u[3], u[4], u[2], u[4], u[5]};
        // the diagonal's slot; its list holds elements that meet the vertex twice (two
        // triangles on the same three vertices): none on an ordinary mesh
        int lo = s0, hi = s1;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (a.ci[mid] < row) lo = mid + 1; else hi = mid;
        }
        const int ds = lo;
        int sl = t0, sh = t1;
        if (s1 - s0 == t1 - t0) {
            sl = t0 + (ds - s0);
        } else {
            while (sl < sh) {
                const int mid = (sl + sh) >> 1;
                if (a.scol[mid] < row) sl = mid + 1; else sh = mid;
            }
        }
        if (a.lptr[sl + 1] > a.lptr[sl])
            add_static(a.codes, a.lptr[sl], a.lptr[sl + 1], a.tri_buf, a.hinge_buf, a.cl_cm, B);
        // difference-form diagonal: m I minus the unzeroed blocks toward pinned neighbours
        if (a.dres) {
            float D[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            if (adj && !prow)
                for (int slot = s0; slot < s1; ++slot) {
                    const int col = a.ci[slot];
                    if (col == row || !a.pinned[col]) continue;
                    float acc[9];
                    row_block(a, row, slot, col, s0, s1, t0, t1, n0, n1, acc);
#pragma unroll
                    for (int q = 0; q < 9; ++q) D[q] -= acc[q];
                }
            D[0] += prow ? m : mA;
            D[4] += prow ? m : mA;
            D[8] += prow ? m : mA;
#pragma unroll
            for (int q = 0; q < 9; ++q) a.dres[9ll * row + q] = D[q];
        }
        float *bb = a.b + 3ll * row;
        if (prow) {
            bb[0] = bb[1] = bb[2] = 0.f;
#pragma unroll
            for (int q = 0; q < 9; ++q) B[q] = 0.f;
            B[0] = B[4] = B[8] = m;
        } else {
            // gravity and the mass-damping force at v_t, both times h
            const float hm = a.h * m, ham = a.ha * m;
            bb[0] = f[0] + hm * a.gx - ham * a.v[3ll * row];
            bb[1] = f[1] + hm * a.gy - ham * a.v[3ll * row + 1];
            bb[2] = f[2] + hm * a.gz - ham * a.v[3ll * row + 2];
            B[0] += mA;
            B[4] += mA;
            B[8] += mA;
        }
        float *dst = a.vals + 9ll * ds;
#pragma unroll
        for (int q = 0; q < 9; ++q) dst[q] = B[q];
    }
    __syncwarp();

    for (;;) {
        int c = 0;
        if (lane == 0) c = atomicAdd(&s_next, 32);
        c = __shfl_sync(0xffffffffu, c, 0);
        if (c >= nblk) break;
        const int i = c + lane;
        if (i >= nblk) continue;
        const int slot = b0 + i;
        int r = 0;  // the row: last r with s_rp[r] <= slot
#pragma unroll
        for (int step = ROWS / 2; step > 0; step >>= 1)
            if (r + step < nr && s_rp[r + step] <= slot) r += step;
        const int row = r0 + r, col = a.ci[slot];
        if (col == row) continue;
        float acc[9];
        if (a.pinned[row] || a.pinned[col]) {
#pragma unroll
            for (int q = 0; q < 9; ++q) acc[q] = 0.f;
        } else {
            row_block(a, row, slot, col, s_rp[r], s_rp[r + 1], s_sp[r], s_sp[r + 1], s_cp[r], s_cp[r + 1], acc);
        }
        float *dst = a.vals + 9ll * slot;
#pragma unroll
        for (int q = 0; q < 9; ++q) dst[q] = acc[q];
    }
}

extern "C" pc_status pc_assemble_values(pc_ctx *ctx, const pc_bsr *A, const float *x, const float *v,
                                        const pc_contacts *contacts, float h, float *vals, float *b, float *dres,
                                        void *stream)
{
    if (!ctx || !A || !A->row_ptr || !A->col_idx || !x || !v || !vals || !b) return PC_ERR_ARG;
    int32_t P = contacts ? contacts->n : 0;
    if (P < 0 || P > ctx->max_contacts || (P > 0 && (!contacts->pairs || !contacts->w))) return PC_ERR_ARG;
    if (P != ctx->n_contacts) return PC_ERR_ARG;  // pattern was built for another contact set
    if (!(h > 0.0f)) return PC_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const int V = ctx->V, T = ctx->T, H = ctx->H;
    // Rayleigh damping: element Hessians enter A as h (h + beta) K, the mass as
    // (1 + h alpha) M (beta = alpha = 0: h^2 K and M)
    const float hb = h + ctx->mat.damp_stiff, hk = h * hb, ih = hk >= FLT_MIN ? h / hk : fminf(1.0f / hb, FLT_MAX);
    const float md = 1.0f + h * ctx->mat.damp_mass, ha = h * ctx->mat.damp_mass;
    if (T > 0)
        PC_LAUNCH(ctx, tri_eval_kernel, pc_blocks(T, TE_THREADS), TE_THREADS, 0, st, T, ctx->tri, x, v, ctx->tri_dmi, ctx->tri_area,
                  ctx->tri_rgram, ctx->mu, ctx->lam, h, hk, ctx->tri_buf);
    if (H > 0)
        PC_LAUNCH(ctx, hinge_eval_kernel, pc_blocks(H, 128), 128, 0, st, H, ctx->hinge, x, v, ctx->hcoef, ctx->hrest, h, hb,
                  hk, ih, ctx->hinge_buf);
    if (P > 0)
        PC_LAUNCH(ctx, contact_eval_kernel, pc_blocks(P, 128), 128, 0, st, P, contacts->pairs, contacts->w, x, v,
                  ctx->mat.k_contact, h, hk, ctx->mat.contact_thickness, ctx->pinned, ctx->cont_buf);
    RowArgs r{};
    r.V = V;
    r.rp = A->row_ptr;
    r.ci = A->col_idx;
    r.srp = ctx->srp;
    r.scol = ctx->scol;
    r.lptr = ctx->val_ptr;
    r.codes = ctx->val_codes;
    r.vinc_ptr = ctx->vinc_ptr;
    r.vinc = ctx->vinc;
    r.cinc_ptr = ctx->cinc_ptr;
    r.cinc = ctx->cinc;
    r.pairs = P > 0 ? contacts->pairs : nullptr;
    r.tri_buf = ctx->tri_buf;
    r.hinge_buf = reinterpret_cast<const float4 *>(ctx->hinge_buf);
    r.cont_buf = ctx->cont_buf;
    r.mass = ctx->mass;
    r.pinned = ctx->pinned;
    r.pin_adj = ctx->pin_adj;
    r.gx = ctx->mat.gravity[0];
    r.gy = ctx->mat.gravity[1];
    r.gz = ctx->mat.gravity[2];
    r.h = h;
    r.md = md;
    r.ha = ha;
    r.cl_cm = ctx->lam / ctx->mu;
    r.v = v;
    r.vals = vals;
    r.b = b;
    r.dres = dres;
    if (V < RR_ROWS * RR_CTAS_PER_SM * ctx->num_sms)
        PC_LAUNCH(ctx, row_reduce_kernel<RR_FEW_ROWS>, pc_blocks(V, RR_FEW_ROWS), RR_THREADS, 0, st, r);
    else
        PC_LAUNCH(ctx, row_reduce_kernel<RR_ROWS>, pc_blocks(V, RR_ROWS), RR_THREADS, 0, st, r);
    return PC_OK;
}
