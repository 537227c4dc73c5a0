// Cross-patch sum of FP32 plans (Section 2, Eq. eqnXforce2 with the order-1
// reconstruction of Eq. eqnGamma): every leaf target receives the cells of every
// patch other than its own (whose contribution is its FFT convolution), from the
// composite sources S_p (amr.cu). Force, mid-plane potential, off-plane force.
//
// Three ranges, by the distance between a target and a source cell of width H:
//
//  * Near cells (centre within SG_NEAR_R cell widths along both axes): the
//    closed forms of Section 2. Targets and cells lie on one lattice, so a
//    target's position inside the source lattice takes 4^g values when its cells
//    are 2^g times narrower than H (one when they are wider): the FP64 integrals
//    of the 12 x 12 cells around each position are tabulated when the plan is
//    built, each as an unevaluated sum of two FP32 numbers (48 bits), with G and
//    H multiplied in. A target then costs a product and a compensated sum per
//    cell and plane instead of two FP64 logarithms and a square root per corner:
//    the exact product (one FMA for its rounding error) is added by Knuth's
//    two-sum. FP64 units run at 1/64 of the FP32 rate here; the pair arithmetic is
//    five times cheaper than a DFMA and rounds at 2^-45. Pairs of levels more
//    than SG_NT_GMAX apart (4^g positions) or with too few targets to repay a
//    table keep the corner form in FP64 (k_near_corner).
//  * Middle cells (up to two clusters of 4 cells away): the expansion of each
//    cell's integrals about its centre through H^6 (force, potential) or 3 x 3
//    Gauss-Legendre nodes (off the plane), in FP32. Per unit G, with a, b =
//    (centre - target)/H, rho^2 = a^2 + b^2, w = 1/(a + i b), s = 1/rho^2, m =
//    sigma0, D = (deltax + i deltay) H:
//      Fx - i Fy = rho^-1 { m [w (1 + s/8 + 7 s^2/256) - 21 w^5/512 - 7 s conj(w)^3/1536]
//                 - D w^2/8 - conj(D) s/24
//                 + 7 conj(D) w^4/384 + D s (conj(w)^2 - 7 w^2)/384 - 7 conj(D) s^2/640 }
//      (from an operator series in d, d~ applied to 1/rho; truncation relative to
//      1/rho^2 at most 1.3e-7 per unit sigma0 and 1.02e-6 per unit slope times H
//      from 6 widths on)
//      Phi = -G H (m I0 + deltax H Ix + deltay H Iy), p = 1/rho:
//      I0 = p + p^3/24 + p^5 (-7/1920 + (7/96) a^2 b^2 p^4)
//      Ix = -a p^3/12 + (7/240) a p^5 - a p^7 (a^2/32 + 5 b^2/96)   (Iy: a <-> b)
//  * Far cells, in clusters. A cluster is a square of 4 2^k cells of a patch; its
//    density is carried by 8 x 8 charges on the Chebyshev points of the square,
//      q_nm = (1/a^2) integral of L_n(x) L_m(y) sigma,  a = half its width,
//    L the Lagrange polynomials: interpolation of the kernel in the source
//    coordinate (a black-box fast multipole method; barycentric Lagrange
//    treecode of Wang, Krasny & Tlupova 2020). It serves every kernel: a charge
//    acts as a point mass. With the target 4 a from the centre (maximum norm) the
//    interpolation errs by at most 3.3e-6 of a charge's own field (5.2e-7 rms over the
//    square; the potential 4.0e-7 and 4.6e-8), with the sign changing from charge to
//    charge; it falls as the eighth power of the distance (7e-9 at 8 a).
//    Charges of level 0 come from the cells (k_p2m), those of level k + 1 from
//    level k by the same interpolation (k_m2m).
//    Each block of up to 256 targets (16 x 16 cells) takes, per source patch, at
//    every level the clusters that are far enough whose parents are not: an index
//    rectangle minus an index rectangle, so no interaction lists are kept. Where
//    the cluster lies two block widths from the block's centre, its field is smooth
//    over the block: it is evaluated on 8 x 8 Chebyshev points of the block and
//    interpolated to the targets once at the end (same bound by symmetry), which
//    is a quarter of the evaluations; four groups of 64 threads share the
//    clusters. The clusters between act on the targets directly.
//    Clusters start at 4 cells (four charges a cell): a charge takes 8 cycles of the
//    special-function unit, a middle cell 62 operations, so that between 8 and 16
//    cells from a block a cluster costs half of its cells. From 8 cells on, six nested
//    256^2 levels took 3.74 ms and three off the plane 1.64; from 4 on, 3.23 and 1.32.
//
// The direct sum over all pairs that this replaces cost 17.3 ms (far) + 8.9 ms
// (near, FP64 pipe) on three nested 256^2 levels. Measured per solve: six nested
// 256^2 levels 121.5 -> 3.03 ms, three off the plane 50.4 -> 1.10 ms; error against
// FP64 4.4e-7 -> 1.4e-7 and 1.5e-7 -> 8e-8.
#include "common.cuh"
#include "kmath.cuh"

#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <utility>
#include <vector>

namespace {

enum { Q_FORCE = 0, Q_POT = 1, Q_OFF = 2 };
template <int Q> constexpr int q_out() { return Q == Q_POT ? 1 : (Q == Q_OFF ? 3 : 2); }
// kernel planes of a near table
template <int Q> constexpr int q_planes() { return Q == Q_POT ? 3 : (Q == Q_OFF ? 9 : 6); }

constexpr int CL = SG_CL_CELLS;        // cells per side of a level-0 cluster
constexpr int NP = 8;                  // Chebyshev points per axis
constexpr int NQ = NP * NP;            // charges of a cluster
static_assert(CL * CL <= NQ && NP * CL <= NQ && NQ == 64, "thread maps below");

// Chebyshev points cos((2 n + 1) pi / 16)
__device__ __forceinline__ constexpr float cheb(int n)
{
    return n == 0 ? 0.98078528040323044f : n == 1 ? 0.83146961230254524f : n == 2 ? 0.55557023301960222f
         : n == 3 ? 0.19509032201612827f : n == 4 ? -0.19509032201612827f : n == 5 ? -0.55557023301960222f
         : n == 6 ? -0.83146961230254524f : -0.98078528040323044f;
}
__device__ const float cheb_points[NP] = {0.98078528040323044f, 0.83146961230254524f, 0.55557023301960222f,
                                          0.19509032201612827f, -0.19509032201612827f, -0.55557023301960222f,
                                          -0.83146961230254524f, -0.98078528040323044f};

// (hi, lo) += v: two-sum (the rounding error of hi + v, exactly, into lo)
__device__ __forceinline__ void add2(float &hi, float &lo, float v)
{
    const float t = __fadd_rn(hi, v);
    const float z = __fsub_rn(t, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, z)), __fsub_rn(v, z)));
    hi = t;
}

// (hi, lo) += s k, k = (kh, kl) a two-part FP32 number: the product's rounding
// error from one FMA
__device__ __forceinline__ void mac2(float &hi, float &lo, float s, float2 k)
{
    const float p = __fmul_rn(s, k.x);
    const float e = __fmaf_rn(s, k.y, __fmaf_rn(s, k.x, -p));
    add2(hi, lo, p);
    lo = __fadd_rn(lo, e);
}

__device__ __forceinline__ int floor_div(int64_t a, int64_t b)
{
    return (int)(a >= 0 ? a / b : -((-a + b - 1) / b));
}

// ------------------------------------------------------------ charges --

// Charges of the level-0 clusters from their cells: with A_n[i] the integral of
// L_n over cell i (cluster coordinate in [-1, 1]) and B_n[i] that of L_n times
// the distance from the cell's centre,
//   q_nm = sum_j [ sum_i (sigma A_n[i] + deltax a B_n[i]) ] A_m[j] + [ sum_i deltay a A_n[i] ] B_m[j].
// 64 threads per cluster (four clusters per CTA), one charge each; bound by
// latency (3.5 k FMAs and 192 bytes per cluster). Clears the targets' sums as well.
__global__ void __launch_bounds__(256) k_p2m(const int4 *__restrict__ desc, int ncl, const sg_patch_dev *__restrict__ pd,
                                             const float *__restrict__ sigma, const float *__restrict__ dx,
                                             const float *__restrict__ dy, double lambda,
                                             const float *__restrict__ mat, float *__restrict__ charges,
                                             double *__restrict__ sums, int64_t nsums)
{
    sg_dep_trigger();
    sg_dep_wait();  // the composite sources (and the reader of the previous solve's sums)
    for (int64_t e = blockIdx.x * 256LL + threadIdx.x; e < nsums; e += gridDim.x * 256LL) sums[e] = 0.0;
    __shared__ float f[4][3][CL * CL];
    __shared__ float T[4][2][NP * CL];
    const int g = threadIdx.x >> 6, t = threadIdx.x & 63;
    const int c = blockIdx.x * 4 + g;
    const float *A = mat, *B = mat + NP * CL;  // [n][i]
    const bool live = c < ncl;
    if (live) {
        const int4 d = desc[c];
        const sg_patch_dev &p = pd[d.x];
        const int i = d.y * CL + t % CL, j = d.z * CL + t / CL;
        float s = 0.f, x = 0.f, y = 0.f;
        if (t < CL * CL && i < p.nx && j < p.ny) {
            const int64_t o = p.cell_off + (int64_t)j * p.nx + i;
            const double a = (double)(CL / 2) * p.step * lambda;  // half the cluster's width
            s = sigma[o];
            x = (float)((double)dx[o] * a);
            y = (float)((double)dy[o] * a);
        }
        if (t < CL * CL) {
            f[g][0][t] = s;
            f[g][1][t] = x;
            f[g][2][t] = y;
        }
    }
    __syncthreads();
    if (live && t < NP * CL) {  // t = n CL + j
        const int n = t / CL, j = t % CL;
        float t1 = 0.f, t2 = 0.f;
#pragma unroll
        for (int i = 0; i < CL; ++i) {
            const float An = __ldg(&A[n * CL + i]);
            t1 = fmaf(f[g][0][j * CL + i], An, t1);
            t1 = fmaf(f[g][1][j * CL + i], __ldg(&B[n * CL + i]), t1);
            t2 = fmaf(f[g][2][j * CL + i], An, t2);
        }
        T[g][0][t] = t1;
        T[g][1][t] = t2;
    }
    __syncthreads();
    if (live) {  // t = m * 8 + n
        const int m = t >> 3, n = t & 7;
        float q = 0.f;
#pragma unroll
        for (int j = 0; j < CL; ++j) {
            q = fmaf(T[g][0][n * CL + j], __ldg(&A[m * CL + j]), q);
            q = fmaf(T[g][1][n * CL + j], __ldg(&B[m * CL + j]), q);
        }
        charges[(int64_t)c * NQ + t] = q;
    }
}

// Charges of the clusters of one level from their up to four children: the
// children's charges interpolated onto the parent's points (C_h[n'][n] =
// L_n at child point n' of half h), times (child width / parent width)^2 = 1/4.
__global__ void __launch_bounds__(256) k_m2m(const int4 *__restrict__ desc, int first, int ncl,
                                             const sg_cl_patch *__restrict__ cp, const int *__restrict__ slot,
                                             const float *__restrict__ mat, float *__restrict__ charges)
{
    sg_dep_trigger();
    sg_dep_wait();  // the level below
    __shared__ float ch[4][4][NQ];
    __shared__ float T[4][2][NQ];
    const int g = threadIdx.x >> 6, t = threadIdx.x & 63;
    const int e = blockIdx.x * 4 + g;
    const bool live = e < ncl;
    const float *Cm = mat + 2 * NP * CL;  // [h][n'][n]
    const int c = first + (live ? e : 0);
    const int4 d = desc[c];
    const sg_cl_patch &p = cp[d.x];
    const int k = d.w - 1;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int cx = 2 * d.y + (q & 1), cy = 2 * d.z + (q >> 1);
        float v = 0.f;
        if (live && cx < p.nx[k] && cy < p.ny[k]) {
            const int s = slot[p.off[k] + cy * p.nx[k] + cx];
            if (s >= 0) v = charges[(int64_t)s * NQ + t];
        }
        ch[g][q][t] = v;
    }
    __syncthreads();
    const int r = t >> 3, n = t & 7;
#pragma unroll
    for (int h = 0; h < 2; ++h) {  // h: lower, upper children; t = m' * 8 + n
        float s = 0.f;
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            s = fmaf(ch[g][2 * h][r * NP + u], __ldg(&Cm[u * NP + n]), s);
            s = fmaf(ch[g][2 * h + 1][r * NP + u], __ldg(&Cm[NQ + u * NP + n]), s);
        }
        T[g][h][t] = s;
    }
    __syncthreads();
    float s = 0.f;  // t = m * 8 + n
#pragma unroll
    for (int u = 0; u < NP; ++u) {
        s = fmaf(T[g][0][u * NP + n], __ldg(&Cm[u * NP + r]), s);
        s = fmaf(T[g][1][u * NP + n], __ldg(&Cm[NQ + u * NP + r]), s);
    }
    if (live) charges[(int64_t)c * NQ + t] = 0.25f * s;
}

// --------------------------------------------------------- middle cells --

// Contribution Q = (Fx - i Fy) / G of one cell, accumulated into (qr, qi). (a,
// b): centre minus target in cell widths; c = (m, d_x, d_y) with d = D / 8. In
// real form with s = 1/rho^2, ir3 = rho^-3, ir5 = rho^-5, c2 = a^2 - b^2, ab2 =
// 2 a b the terms through H^4 are
//   Re Q = m (1 + s/8) ir3 a - d_x (ir5 c2 + ir3/3) - d_y ir5 ab2
//   Im Q = -m (1 + s/8) ir3 b + d_y (ir3/3 - ir5 c2) + d_x ir5 ab2;
// the H^6 terms are added in complex form.
__device__ __forceinline__ void cell_far(float a, float b, const float4 c, float &qr, float &qi)
{
    const float b2 = b * b, tb = 2.f * b;
    const float r2 = fmaf(a, a, b2);
    const float c2 = fmaf(a, a, -b2);
    const float ab2 = a * tb;
    const float ir = rsqrtf(r2);
    const float s = ir * ir;
    const float ir3 = ir * s, ir5 = ir3 * s;
    const float poly = fmaf(s, fmaf(s, 7.f / 256.f, 0.125f), 1.f);
    const float g = c.x * poly * ir3;
    const float u3 = ir3 * (1.f / 3.f);
    const float e1 = fmaf(ir5, c2, u3), e2 = fmaf(-ir5, c2, u3), f = ir5 * ab2;
    qr = fmaf(g, a, qr);
    qr = fmaf(-c.y, e1, qr);
    qr = fmaf(-c.z, f, qr);
    qi = fmaf(-g, b, qi);
    qi = fmaf(c.z, e2, qi);
    qi = fmaf(c.y, f, qi);
    // w = (a - i b) s, w^2 = (c2 - i ab2) s^2
    const float wr = a * s, wi = -b * s;
    const float ss = s * s;
    const float w2r = c2 * ss, w2i = -ab2 * ss;
    const float w3r = fmaf(w2r, wr, -w2i * wi), w3i = fmaf(w2r, wi, w2i * wr);
    const float w4r = fmaf(w2r, w2r, -w2i * w2i), w4i = 2.f * w2r * w2i;
    const float w5r = fmaf(w4r, wr, -w4i * wi), w5i = fmaf(w4r, wi, w4i * wr);
    // - m (21/512) w^5 - m s (7/1536) conj(w^3)
    const float m1 = c.x * (21.f / 512.f), m2 = c.x * s * (7.f / 1536.f);
    float pr = -m1 * w5r, pi = -m1 * w5i;
    pr = fmaf(-m2, w3r, pr);
    pi = fmaf(m2, w3i, pi);
    // + 7 conj(D) w^4 / 384 = (7/48) conj(d) w^4
    const float e7 = 7.f / 48.f;
    pr = fmaf(e7, fmaf(c.y, w4r, c.z * w4i), pr);
    pi = fmaf(e7, fmaf(c.y, w4i, -c.z * w4r), pi);
    // + D s (conj(w^2) - 7 w^2) / 384 = (s/48) d (-6 w2r - 8 i w2i)
    const float ur = s * (-6.f / 48.f) * w2r, ui = s * (-8.f / 48.f) * w2i;
    pr = fmaf(c.y, ur, pr);
    pr = fmaf(-c.z, ui, pr);
    pi = fmaf(c.y, ui, pi);
    pi = fmaf(c.z, ur, pi);
    // - 7 conj(D) s^2 / 640 = -(7/80) conj(d) s^2
    const float s2 = ss * (7.f / 80.f);
    pr = fmaf(-c.y, s2, pr);
    pi = fmaf(c.z, s2, pi);
    qr = fmaf(ir, pr, qr);
    qi = fmaf(ir, pi, qi);
}

// One cell's potential per unit (-G H): c = (m, deltax H / 8, deltay H / 8).
__device__ __forceinline__ float cell_far_pot(float a, float b, const float4 c)
{
    const float b2 = b * b;
    const float r2 = fmaf(a, a, b2);
    const float p = rsqrtf(r2);
    const float s = p * p;
    const float p3 = p * s;
    float i0 = fmaf(p3, 1.f / 24.f, p);
    float kx = p3 * (-8.f / 12.f);
    const float p5 = p3 * s, p7 = p5 * s;
    const float ab = a * b;
    i0 = fmaf(p5, fmaf(ab * ab * s * s, 7.f / 96.f, -7.f / 1920.f), i0);
    kx = fmaf(p5, 8.f * 7.f / 240.f, kx);
    float ky = kx;
    kx = fmaf(-8.f * p7, fmaf(a, a * (1.f / 32.f), b2 * (5.f / 96.f)), kx);
    ky = fmaf(-8.f * p7, fmaf(b2, 1.f / 32.f, a * a * (5.f / 96.f)), ky);
    return fmaf(c.x, i0, fmaf(c.y * a, kx, c.z * b * ky));
}

// Off the plane: 3 x 3 Gauss-Legendre nodes of (m + deltax H xi + deltay H eta)
// (a + xi, b + eta, -zeta) / R^3 over the unit cell (relative error below 3e-7
// from SG_NEAR_R cell widths on).
__device__ __forceinline__ void cell_far_z(float a, float b, float zeta2, float4 c, float &qx, float &qy, float &qz)
{
    constexpr float X3 = 0.387298334620742f, W3a = 5.f / 18.f, W3b = 8.f / 18.f;  // on [-1/2, 1/2], weights sum to 1
    float sx = 0.f, sy = 0.f, s0 = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float xi = i == 0 ? -X3 : (i == 1 ? 0.f : X3);
        const float wi = i == 1 ? W3b : W3a;
        const float da = a + xi;
        const float da2z = fmaf(da, da, zeta2);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float eta = j == 0 ? -X3 : (j == 1 ? 0.f : X3);
            const float wj = j == 1 ? W3b : W3a;
            const float db = b + eta;
            const float ir = rsqrtf(fmaf(db, db, da2z));
            const float w = wi * wj * fmaf(8.f * c.y, xi, fmaf(8.f * c.z, eta, c.x)) * (ir * ir * ir);
            sx = fmaf(w, da, sx);
            sy = fmaf(w, db, sy);
            s0 += w;
        }
    }
    qx += sx;
    qy += sy;
    qz += s0;  // times -zeta by the caller
}

// ------------------------------------------------------------- far field --

// Field of one cluster's charges at a point: (X0, Y0) = cluster centre minus
// point, zeta2 = (z / a)^2, in units of a, half the cluster's width. Force:
// sums of q d / R^3 (off the plane also of q / R^3); potential: of q / R. Six
// FP32 operations and one reciprocal square root per charge: bound by the
// special-function unit (16 per clock and SM).
template <int Q>
__device__ __forceinline__ void cluster_field(const float4 *__restrict__ q, float X0, float Y0, float zeta2,
                                              float (&out)[q_out<Q>()])
{
    float a[NP], a2[NP];
#pragma unroll
    for (int n = 0; n < NP; ++n) {
        a[n] = X0 + cheb(n);
        a2[n] = a[n] * a[n];
        if (Q == Q_OFF) a2[n] += zeta2;
    }
#pragma unroll
    for (int o = 0; o < q_out<Q>(); ++o) out[o] = 0.f;
#pragma unroll
    for (int m = 0; m < NP; ++m) {
        const float b = Y0 + cheb(m), b2 = b * b;
        const float4 q0 = __ldg(&q[2 * m]), q1 = __ldg(&q[2 * m + 1]);
        const float qq[NP] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
        float w = 0.f;
#pragma unroll
        for (int n = 0; n < NP; ++n) {
            const float ir = rsqrtf(a2[n] + b2);
            if constexpr (Q == Q_POT) {
                w = fmaf(qq[n], ir, w);
            } else {
                const float v = qq[n] * ir * (ir * ir);
                out[0] = fmaf(v, a[n], out[0]);
                w += v;
            }
        }
        if constexpr (Q == Q_POT) {
            out[0] += w;
        } else {
            out[1] = fmaf(w, b, out[1]);
            if constexpr (Q == Q_OFF) out[2] += w;
        }
    }
}

struct far_args {
    const sg_target_block *blocks;
    int nblocks;
    const int4 *targets;
    const sg_patch_dev *pd;
    const sg_cl_patch *cp;
    const int *slot;
    const float *charges;
    int npatches;
    const float *sigma, *dx, *dy;   // composite sources
    double lambda;                  // lattice unit
    double G;                       // over 2^sum_exponent
    double zl;                      // height in lattice units
    int ctas;                       // CTAs of the middle and far field; the near field's follow
    int ntargets;
    const int *keys;                // near tables
    const float2 *tab;
    double *sums;                   // near + far per target, q_out components, cleared by k_p2m
};

// Middle and far field of one target block per CTA. CTAs take blocks from the last to the
// first (the finest patches, with the most coarser cells near them, first).
// Bound by FP32 issue (middle cells: 62 operations each) and the special-function
// unit (clusters). Middle cells smooth over the block go on its points as well: 2.7 ms
// for six nested 256^2 levels against 3.8 with every middle cell on the targets, 1.25
// against 1.49 for three off the plane (with clusters of 8 cells; 4 save 0.5 and 0.3).
template <int Q>
__device__ __forceinline__ void far_field(const far_args &A)
{
    constexpr int NO = q_out<Q>();
    __shared__ float4 mc[256];
    __shared__ float2 mp[256];
    __shared__ float nodes[4][NQ][NO][2];
    __shared__ double base[NO];
    __shared__ float diff[NQ][NO];
    const int tid = threadIdx.x;
    const int grp = tid >> 6, node = tid & 63;
    for (int item = blockIdx.x; item < A.nblocks; item += A.ctas) {
        const sg_target_block blk = A.blocks[A.nblocks - 1 - item];
        const bool active = tid < blk.count;
        const int4 tg = A.targets[blk.first + (active ? tid : 0)];
        // the block as a square in twice the lattice coordinates: centre C, width b2 (of target positions)
        const int Cx = blk.tx0 + blk.tx1, Cy = blk.ty0 + blk.ty1;
        const int b2 = max(blk.tx1 - blk.tx0, blk.ty1 - blk.ty0);
        const float hb = 0.5f * (float)b2;
        // this thread's target and its block point, lattice units from the centre
        const float tx = 0.5f * (float)(2 * tg.x - Cx), ty = 0.5f * (float)(2 * tg.y - Cy);
        const float px = hb * cheb_points[node & 7], py = hb * cheb_points[node >> 3];
        float th[NO], tl[NO], nh[NO], nl[NO];  // sums at the target and at the point, two-part
#pragma unroll
        for (int o = 0; o < NO; ++o) th[o] = tl[o] = nh[o] = nl[o] = 0.f;
        for (int q = 0; q < A.npatches; ++q) {
            if (q == blk.patch) continue;
            const sg_patch_dev &p = A.pd[q];
            const sg_cl_patch &cp = A.cp[q];
            const int ox2 = 2 * p.ox - Cx, oy2 = 2 * p.oy - Cy;  // patch corner from the centre, doubled
            // near clusters of the level above (the whole grid's parent to begin with)
            int pi0 = 0, pi1 = 0, pj0 = 0, pj1 = 0;
            for (int k = cp.nlev - 1; k >= 0; --k) {
                const int nx = cp.nx[k], ny = cp.ny[k];
                const int W = (CL * p.step) << k;  // the cluster's width (lattice units)
                const int ca = 2 * pi0, cb = min(nx - 1, 2 * pi1 + 1), ra = 2 * pj0, rb = min(ny - 1, 2 * pj1 + 1);
                // clusters nearer than 4 a = 2 W: 2 (centre) = o2 + (2 i + 1) W in (-b2 - 4 W, b2 + 4 W)
                const int ni0 = max(ca, floor_div(-b2 - 5 * (int64_t)W - ox2, 2 * (int64_t)W) + 1);
                const int ni1 = min(cb, -floor_div(-(b2 + 3 * (int64_t)W - ox2), 2 * (int64_t)W) - 1);
                const int nj0 = max(ra, floor_div(-b2 - 5 * (int64_t)W - oy2, 2 * (int64_t)W) + 1);
                const int nj1 = min(rb, -floor_div(-(b2 + 3 * (int64_t)W - oy2), 2 * (int64_t)W) - 1);
                const bool some = ni0 <= ni1 && nj0 <= nj1;
                // clusters nearer than 2 b2 + W/2, whose field is not smooth over the block
                const int M2 = max(4 * b2 + W, b2 + 4 * W);
                const int mi0 = max(ca, floor_div(-(int64_t)M2 - ox2 - W, 2 * (int64_t)W) + 1);
                const int mi1 = min(cb, -floor_div(-((int64_t)M2 - ox2 - W), 2 * (int64_t)W) - 1);
                const int mj0 = max(ra, floor_div(-(int64_t)M2 - oy2 - W, 2 * (int64_t)W) + 1);
                const int mj1 = min(rb, -floor_div(-((int64_t)M2 - oy2 - W), 2 * (int64_t)W) - 1);
                const bool mid = mi0 <= mi1 && mj0 <= mj1;
                const float inv = 2.f / (float)W;
                const float zeta = Q == Q_OFF ? (float)(2.0 * A.zl / (double)W) : 0.f;
                const int *sl = A.slot + cp.off[k];
                // two passes: the others on the block's points, a quarter per group; those on the targets
                for (int pass = 0; pass < 2; ++pass) {
                    const bool outer = pass == 0;
                    if (!outer && (W >= b2 || !mid || (tid & ~31) >= blk.count)) continue;
                    const int x0 = outer ? ca : mi0, x1 = outer ? cb : mi1, y1 = outer ? rb : mj1;
                    const bool hole = outer ? mid : some;
                    const int hx0 = outer ? mi0 : ni0, hx1 = outer ? mi1 : ni1;
                    const int hy0 = outer ? mj0 : nj0, hy1 = outer ? mj1 : nj1;
                    const int w = x1 - x0 + 1, de = outer ? 4 : 1;
                    const float ux = (outer ? px : tx) * inv, uy = (outer ? py : ty) * inv;
                    int i = x0 + (outer ? grp : 0), jj = outer ? ra : mj0;
                    for (;; i += de) {
                        while (i > x1) {
                            i -= w;
                            ++jj;
                        }
                        if (jj > y1) break;
                        if (hole && i >= hx0 && i <= hx1 && jj >= hy0 && jj <= hy1) continue;
                        const int s = __ldg(&sl[jj * nx + i]);
                        if (s < 0) continue;
                        const float X0 = (float)(ox2 + (2 * i + 1) * W) / (float)W - ux;
                        const float Y0 = (float)(oy2 + (2 * jj + 1) * W) / (float)W - uy;
                        float v[NO];
                        cluster_field<Q>(reinterpret_cast<const float4 *>(A.charges + (int64_t)s * NQ), X0, Y0, zeta * zeta, v);
                        if constexpr (Q == Q_POT) v[0] *= 0.5f * (float)W;  // q / R in lattice units
                        if constexpr (Q == Q_OFF) v[2] *= -zeta;
#pragma unroll
                        for (int o = 0; o < NO; ++o) {
                            if (outer) add2(nh[o], nl[o], v[o]);
                            else add2(th[o], tl[o], v[o]);
                        }
                    }
                }
                pi0 = ni0;
                pi1 = ni1;
                pj0 = nj0;
                pj1 = nj1;
                if (!some) break;
            }
            if (pi0 > pi1 || pj0 > pj1) continue;
            // the cells of the near level-0 clusters, in two passes: those whose field is
            // smooth over the block (two block widths from its centre, and no target's near
            // cell) on the block's points, a quarter per group of threads; the others on the targets
            const int L = p.step;
            const int i0 = CL * pi0, i1 = min(p.nx, CL * (pi1 + 1)) - 1, j0 = CL * pj0, j1 = min(p.ny, CL * (pj1 + 1)) - 1;
            const int M2 = max(4 * b2 + L, 2 * SG_NEAR_R * L + b2);  // twice the distance, doubled
            const int ii0 = max(i0, floor_div(-(int64_t)M2 - ox2 - L, 2 * L) + 1), ii1 = min(i1, -floor_div(-((int64_t)M2 - ox2 - L), 2 * L) - 1);
            const int ij0 = max(j0, floor_div(-(int64_t)M2 - oy2 - L, 2 * L) + 1), ij1 = min(j1, -floor_div(-((int64_t)M2 - oy2 - L), 2 * L) - 1);
            const bool inner = ii0 <= ii1 && ij0 <= ij1;
            const float invL = 1.f / (float)L;  // a power of two: exact
            const double h8 = L * A.lambda * 0.125;
            const float zeta = Q == Q_OFF ? (float)(A.zl / (double)L) : 0.f;
            for (int pass = 0; pass < 2; ++pass) {
                const bool outer = pass == 0;
                if (outer && inner && ii0 == i0 && ii1 == i1 && ij0 == j0 && ij1 == j1) continue;
                if (!outer && !inner) continue;
                const int a0 = outer ? i0 : ii0, b0 = outer ? j0 : ij0;
                const int w = (outer ? i1 : ii1) - a0 + 1, total = w * ((outer ? j1 : ij1) - b0 + 1);
                const float ux = (outer ? px : tx) * invL, uy = (outer ? py : ty) * invL;
                for (int e0 = 0; e0 < total; e0 += 256) {
                    const int e = e0 + tid;
                    __syncthreads();  // the previous cells have been used
                    if (e < total) {
                        const int jr = e / w, i = a0 + e - jr * w, j = b0 + jr;
                        const int64_t o = p.cell_off + (int64_t)j * p.nx + i;
                        float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (!(outer && inner && i >= ii0 && i <= ii1 && j >= ij0 && j <= ij1))
                            c = make_float4(A.sigma[o], (float)((double)A.dx[o] * h8), (float)((double)A.dy[o] * h8), 0.f);
                        mc[tid] = c;
                        mp[tid] = make_float2(0.5f * (float)(ox2 + (2 * i + 1) * L) * invL,
                                              0.5f * (float)(oy2 + (2 * j + 1) * L) * invL);
                    }
                    __syncthreads();
                    if (!outer && (tid & ~31) >= blk.count) continue;  // no target in this warp
                    const int nc = min(256, total - e0), dc = outer ? 4 : 1;
                    float s[NO];
#pragma unroll
                    for (int o = 0; o < NO; ++o) s[o] = 0.f;
                    for (int c = outer ? grp : 0; c < nc; c += dc) {
                        const float4 cc = mc[c];
                        if (cc.x == 0.f && cc.y == 0.f && cc.z == 0.f) continue;  // no density (the same in the warp)
                        const float a = mp[c].x - ux, b = mp[c].y - uy;  // at targets exact: half-cell multiples
                        const bool nearc = fabsf(a) < (float)SG_NEAR_R && fabsf(b) < (float)SG_NEAR_R;
                        float t[NO];
#pragma unroll
                        for (int o = 0; o < NO; ++o) t[o] = s[o];
                        if constexpr (Q == Q_FORCE) cell_far(a, b, cc, t[0], t[1]);
                        else if constexpr (Q == Q_POT) t[0] += cell_far_pot(a, b, cc);
                        else cell_far_z(a, b, zeta * zeta, cc, t[0], t[1], t[2]);
#pragma unroll
                        for (int o = 0; o < NO; ++o) s[o] = nearc ? s[o] : t[o];
                    }
                    if constexpr (Q == Q_FORCE) s[1] = -s[1];    // Q = Fx - i Fy
                    if constexpr (Q == Q_POT) s[0] *= (float)L;  // per lattice unit
                    if constexpr (Q == Q_OFF) s[2] *= -zeta;
#pragma unroll
                    for (int o = 0; o < NO; ++o) {
                        if (outer) add2(nh[o], nl[o], s[o]);
                        else add2(th[o], tl[o], s[o]);
                    }
                }
            }
        }
        // the field at the block's points, then its interpolation to the targets:
        // the value at point 0 in FP64 plus the interpolated differences from it
        // (small where the field is smooth), since the weights sum to one
        __syncthreads();
#pragma unroll
        for (int o = 0; o < NO; ++o) {
            nodes[grp][node][o][0] = nh[o];
            nodes[grp][node][o][1] = nl[o];
        }
        __syncthreads();
        double v[NO];
        if (grp == 0) {
#pragma unroll
            for (int o = 0; o < NO; ++o) {
                v[o] = 0.0;
                for (int u = 0; u < 4; ++u) v[o] += (double)nodes[u][node][o][0] + (double)nodes[u][node][o][1];
                if (node == 0) base[o] = v[o];
            }
        }
        __syncthreads();
        if (grp == 0) {
#pragma unroll
            for (int o = 0; o < NO; ++o) diff[node][o] = (float)(v[o] - base[o]);
        }
        __syncthreads();
        if (active) {
            // Lagrange weights at the target (b2 = 0: one position, on the coincident points)
            const float x = b2 > 0 ? tx / hb : 0.f, y = b2 > 0 ? ty / hb : 0.f;
            float lx[NP], ly[NP];
#pragma unroll
            for (int n = 0; n < NP; ++n) {
                float u = 1.f, v1 = 1.f, d = 1.f;
#pragma unroll
                for (int r = 0; r < NP; ++r) {
                    if (r == n) continue;
                    u *= x - cheb(r);
                    v1 *= y - cheb(r);
                    d *= cheb(n) - cheb(r);
                }
                lx[n] = u * (1.f / d);
                ly[n] = v1 * (1.f / d);
            }
            float f[NO];
#pragma unroll
            for (int o = 0; o < NO; ++o) f[o] = 0.f;
#pragma unroll
            for (int m = 0; m < NP; ++m) {
                float r[NO];
#pragma unroll
                for (int o = 0; o < NO; ++o) r[o] = 0.f;
#pragma unroll
                for (int n = 0; n < NP; ++n)
#pragma unroll
                    for (int o = 0; o < NO; ++o) r[o] = fmaf(lx[n], diff[m * NP + n][o], r[o]);
#pragma unroll
                for (int o = 0; o < NO; ++o) f[o] = fmaf(ly[m], r[o], f[o]);
            }
            const double scale = Q == Q_POT ? -A.G * A.lambda : A.G;
#pragma unroll
            for (int o = 0; o < NO; ++o) {
                const double far = base[o] + (double)f[o] + ((double)th[o] + (double)tl[o]);
                atomicAdd(&A.sums[(int64_t)(blk.first + tid) * NO + o], scale * far);
            }
        }
        __syncthreads();  // base and diff have been read
    }
}

// ------------------------------------------------------------ near field --

constexpr int NEAR_BOX = 2 * SG_NEAR_R;              // cells per side of a table
constexpr int NEAR_CELLS = NEAR_BOX * NEAR_BOX;

// First cell of a table's box from the cell that holds the target (frac, the
// target's position in that cell): cells with |centre - target| < SG_NEAR_R.
__host__ __device__ __forceinline__ int near_first(int f, int g)
{
    // frac = (f + 1/2) / 2^g (g >= 0) or 0 (g < 0: on the cell's lower corner)
    return g >= 0 && 2 * f + 1 > (1 << g) ? -SG_NEAR_R + 1 : -SG_NEAR_R;
}

// The tables to build: key k holds the classes first[k] .. first[k + 1] for cells
// of width H[k] and ratio exponent g[k].
struct near_list {
    int n;
    int first[SG_NT_STEPS * SG_NT_KEYS + 1];
    int g[SG_NT_STEPS * SG_NT_KEYS];
    double H[SG_NT_STEPS * SG_NT_KEYS];
};

// Near tables, every key in one launch (the smallest have 144 entries, whose FP64
// latency alone is 0.1 ms: one launch per key added 2.7 ms to a plan of six levels):
// the closed-form integrals of the 12 x 12 cells around each position (fx, fy),
// scaled, in two FP32 parts, [plane][cell]; zero outside the near box and where
// the integral diverges (a target on a corner or inside an edge of a cell: never a
// leaf target with a cell that carries density).
template <int Q>
__global__ void k_near_table(float2 *__restrict__ out, near_list L, double G, double z)  // G: over 2^sum_exponent
{
    const int64_t total = (int64_t)L.first[L.n] * NEAR_CELLS;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int cls = (int)(e / NEAR_CELLS), c = (int)(e % NEAR_CELLS);
        int k0 = 0;
        while (cls >= L.first[k0 + 1]) ++k0;
        const int g = L.g[k0], pos = cls - L.first[k0];
        const double H = L.H[k0];
        const int fx = g < 0 ? 0 : pos & ((1 << g) - 1), fy = g < 0 ? 0 : pos >> g;
        const double w = g < 0 ? 0.0 : 1.0 / (double)(1 << g);
        const double cx = near_first(fx, g) + c % NEAR_BOX + 0.5 - (g < 0 ? 0.0 : (fx + 0.5) * w);
        const double cy = near_first(fy, g) + c / NEAR_BOX + 0.5 - (g < 0 ? 0.0 : (fy + 0.5) * w);
        double v[9];
        for (int k = 0; k < 9; ++k) v[k] = 0.0;
        if (fabs(cx) < SG_NEAR_R && fabs(cy) < SG_NEAR_R) {
            if constexpr (Q == Q_POT) {
                unit_cell_potentials(cx, cy, v);
                v[0] *= -G * H;
                v[1] *= -G * H * H;
                v[2] *= -G * H * H;
            } else if constexpr (Q == Q_OFF) {
                unit_cell_offplane(cx, cy, z / H, v);
                for (int k = 0; k < 9; ++k) v[k] *= k % 3 == 0 ? G : G * H;
            } else {
                // unit_x_family: K^{x,0}, K^{x,x}, K^{x,y} at (cx, cy); the y family by exchange
                double x0, xx, xy, y0, yy, yx;
                if (unit_x_family(cx, cy, x0, xx, xy) && unit_x_family(cy, cx, y0, yy, yx)) {
                    v[0] = G * x0;
                    v[1] = G * H * xx;
                    v[2] = G * H * xy;
                    v[3] = G * y0;
                    v[4] = G * H * yx;
                    v[5] = G * H * yy;
                }
            }
        }
        for (int k = 0; k < q_planes<Q>(); ++k) {
            const float hi = (float)v[k];
            out[((int64_t)cls * q_planes<Q>() + k) * NEAR_CELLS + c] = make_float2(hi, (float)(v[k] - (double)hi));
        }
    }
}

// The near box of a target in patch p, clipped to the patch: cells [i0, i1] x [j0, j1].
__device__ __forceinline__ bool near_box(const sg_patch_dev &p, int x, int y, int &i0, int &i1, int &j0, int &j1)
{
    const int64_t L = p.step, RL = (int64_t)SG_NEAR_R * L;
    const int64_t ex = (int64_t)x - p.ox - L / 2, ey = (int64_t)y - p.oy - L / 2;
    i0 = max(0, floor_div(ex - RL, L) + 1);
    j0 = max(0, floor_div(ey - RL, L) + 1);
    i1 = min(p.nx - 1, -floor_div(-(ex + RL), L) - 1);
    j1 = min(p.ny - 1, -floor_div(-(ey + RL), L) - 1);
    return i0 <= i1 && j0 <= j1;
}

__device__ __forceinline__ int ilog2_pow2(int v) { return __ffs(v) - 1; }

// Table offset (in classes) of source cells `step` against target cells `ts`
// (lattice units), -1 if there is none: tab[log2 step][g + 1].
__device__ __forceinline__ int near_key(const int *__restrict__ tab, int step, int ts, int &g)
{
    g = max(-1, ilog2_pow2(step) - ilog2_pow2(ts));
    if (g > SG_NT_GMAX) return -1;
    return __ldg(&tab[ilog2_pow2(step) * SG_NT_KEYS + g + 1]);
}

constexpr int NEAR_WARPS = 8;

// Near field from the tables: one warp per target, lanes over the cells of its
// box; the lanes test 32 patches at a time. Bound by FP32 issue (11 operations
// per plane and cell) and the L2 reads of the tables (6.9 KB per position): 0.78 ms
// for the 865,000 boxes of six nested 256^2 levels (the FP64 corner form: 40 ms),
// 0.31 ms for the 199,000 off-plane boxes of three.
template <int Q>
__device__ __forceinline__ void near_field(const far_args &A, int cta)
{
    constexpr int NO = q_out<Q>(), NPL = q_planes<Q>();
    const sg_patch_dev *__restrict__ pd = A.pd;
    const float *__restrict__ sigma = A.sigma, *__restrict__ dx = A.dx, *__restrict__ dy = A.dy;
    const int *__restrict__ keys = A.keys;
    const int npatches = A.npatches;
    const int lane = threadIdx.x & 31;
    const int t = cta * NEAR_WARPS + (int)(threadIdx.x >> 5);
    if (t >= A.ntargets) return;
    const int4 tg = A.targets[t];
    const int ts = pd[tg.w].step;
    float hi[NO], lo[NO];
#pragma unroll
    for (int o = 0; o < NO; ++o) hi[o] = lo[o] = 0.f;
    for (int q0 = 0; q0 < npatches; q0 += 32) {
        bool hit = false;
        if (q0 + lane < npatches && q0 + lane != tg.w) {
            int i0, i1, j0, j1, g;
            hit = near_box(pd[q0 + lane], tg.x, tg.y, i0, i1, j0, j1) && near_key(keys, pd[q0 + lane].step, ts, g) >= 0;
        }
        for (unsigned m = __ballot_sync(0xffffffffu, hit); m; m &= m - 1) {
            const sg_patch_dev &p = pd[q0 + __ffs(m) - 1];
            int g;
            const int key = near_key(keys, p.step, ts, g);
            // the cell that holds the target, and its position in it
            const int x = tg.x - p.ox, y = tg.y - p.oy;
            const int sh = ilog2_pow2(p.step), I = x >> sh, J = y >> sh;
            const int fx = g < 0 ? 0 : (x & (p.step - 1)) / ts, fy = g < 0 ? 0 : (y & (p.step - 1)) / ts;
            const float2 *T = A.tab + ((int64_t)key + (g < 0 ? 0 : (fy << g) + fx)) * (NPL * NEAR_CELLS);
            const int ib = I + near_first(fx, g), jb = J + near_first(fy, g);
#pragma unroll
            for (int it = 0; it < (NEAR_CELLS + 31) / 32; ++it) {
                const int c = lane + 32 * it;
                const int i = ib + c % NEAR_BOX, j = jb + c / NEAR_BOX;
                if (c >= NEAR_CELLS || i < 0 || i >= p.nx || j < 0 || j >= p.ny) continue;
                const int64_t o = p.cell_off + (int64_t)j * p.nx + i;
                const float f[3] = {sigma[o], dx[o], dy[o]};
#pragma unroll
                for (int k = 0; k < NPL; ++k) mac2(hi[k / 3], lo[k / 3], f[k % 3], __ldg(&T[k * NEAR_CELLS + c]));
            }
        }
    }
#pragma unroll
    for (int o = 0; o < NO; ++o) {
        double v = (double)hi[o] + (double)lo[o];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (lane == 0) atomicAdd(&A.sums[(int64_t)t * NO + o], v);
    }
}

// The cross-patch sum in one launch: the CTAs of the middle and far field first, then
// those of the near field, which are short and fill the SMs while the last of the
// uneven far blocks run. Each target receives one addend from either, added to zero
// in either order (the same result). As two launches, one after the other: six nested 256^2 levels
// 3.23 ms, three off the plane 1.32, three in the plane 1.08; so 3.03, 1.10 and 0.92.
// (With targets for many waves the near field loses more by the far field's register
// count than the overlap gains: 5.7 M targets 30.3 ms as two launches, 32.4 as one.)
template <int Q>
__global__ void __launch_bounds__(NEAR_WARPS * 32, 3) k_near_far(far_args A)
{
    static_assert(NEAR_WARPS * 32 == 256, "one CTA size for both");
    sg_dep_trigger();
    sg_dep_wait();  // the composite sources, the charges, the cleared sums
    if ((int)blockIdx.x < A.ctas) far_field<Q>(A);
    else near_field<Q>(A, (int)blockIdx.x - A.ctas);
}

// Adds the sums, times scale (2^sum_exponent), to the targets' own-patch results.
template <int Q>
__global__ void __launch_bounds__(256) k_cross_add(const int4 *__restrict__ targets, int ntargets,
                                                   const double *__restrict__ sums, double scale, float *o0, float *o1,
                                                   float *o2)
{
    constexpr int NO = q_out<Q>();
    sg_dep_trigger();
    sg_dep_wait();
    const int t = blockIdx.x * 256 + threadIdx.x;
    if (t >= ntargets) return;
    const int at = targets[t].z;
    float *const out[3] = {o0, o1, o2};
#pragma unroll
    for (int o = 0; o < NO; ++o) {
        if (!out[o]) continue;  // sg_force on an off-plane plan takes Fx, Fy only
        out[o][at] = (float)((double)out[o][at] + scale * sums[(int64_t)t * NO + o]);
    }
}

// Near field without tables, added to near_out: one warp per target, the box of
// every patch that has no table for this pair of cell widths in the corner form
// in FP64. Every cell integral is a double difference over the cell's corners
// with weights A_c(t) = sum_i s_ic l_i(t), X_c, Y_c (l_i the reconstruction of
// cell i at the target; see direct.cu):
//   Fx = G sum_c [ -A g0 + X v g0y - Y r ],  Fy = G sum_c [ -A g0y + Y u g0 - X r ]
//   Phi = -G sum_c [ A F0 + X Fu + Y Fv ],  F0 = u g0 + v g0y, Fu = (v r + u^2 g0)/2, Fv = (u r + v^2 g0y)/2
// and off the plane, with R, G0, G0y, T = atan(u v / (|z| R)),
//   Fx = G sum_c [ -A G0 + X (v G0y - |z| T) - Y R ],  Fz = G sum_c [ -sgn(z) A T + z (X G0 + Y G0y) ].
// The warp stages the box's cell values with a zero border in shared memory and
// the logarithms of the corner columns and rows in lanes; lanes take corners.
constexpr int NEAR_SLOTS = (2 * SG_NEAR_R + 2) * (2 * SG_NEAR_R + 2);

template <int Q>
__global__ void __launch_bounds__(NEAR_WARPS * 32) k_near_corner(const int4 *__restrict__ targets, int ntargets,
                                                                 const sg_patch_dev *__restrict__ pd, int npatches,
                                                                 const float *__restrict__ sigma,
                                                                 const float *__restrict__ dx,
                                                                 const float *__restrict__ dy,
                                                                 const int *__restrict__ keys, double lambda, double G,
                                                                 double z, double *__restrict__ near_out)
{
    constexpr int NO = q_out<Q>();
    sg_dep_trigger();
    sg_dep_wait();
    __shared__ double cellv[NEAR_WARPS][3][NEAR_SLOTS];
    const int lane = threadIdx.x & 31;
    double *cl = cellv[threadIdx.x >> 5][0], *cx = cellv[threadIdx.x >> 5][1], *cy = cellv[threadIdx.x >> 5][2];
    const int t = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    if (t >= ntargets) return;
    const double az = fabs(z), z2 = z * z, sz = z > 0.0 ? 1.0 : -1.0;
    const int4 tg = targets[t];
    const int ts = pd[tg.w].step;
    double f[NO];
#pragma unroll
    for (int o = 0; o < NO; ++o) f[o] = 0.0;
    bool any = false;
    for (int q = 0; q < npatches; ++q) {
        if (q == tg.w) continue;
        const sg_patch_dev &p = pd[q];
        int i0, i1, j0, j1, g;
        if (near_key(keys, p.step, ts, g) >= 0 || !near_box(p, tg.x, tg.y, i0, i1, j0, j1)) continue;
        any = true;
        const int64_t L = p.step;
        const int nbx = i1 - i0 + 1, nby = j1 - j0 + 1, W = nbx + 2;
        __syncwarp();  // the previous box's values have been read
        for (int k = lane; k < W * (nby + 2); k += 32) {
            const int bi = k % W - 1, bj = k / W - 1;
            double l = 0.0, X = 0.0, Y = 0.0;
            if (bi >= 0 && bi < nbx && bj >= 0 && bj < nby) {
                const int i = i0 + bi, j = j0 + bj;
                const int64_t o = p.cell_off + (int64_t)j * p.nx + i;
                X = dx[o];
                Y = dy[o];
                // target minus cell centre, physical units
                const double ux = ((double)tg.x - ((double)p.ox + (i + 0.5) * (double)L)) * lambda;
                const double uy = ((double)tg.y - ((double)p.oy + (j + 0.5) * (double)L)) * lambda;
                l = fma(X, ux, fma(Y, uy, (double)sigma[o]));
            }
            cl[k] = l;
            cx[k] = X;
            cy[k] = Y;
        }
        // corner column ci (lane ci <= nbx) and row cj: u, v relative to the target; on u = 0 the
        // coincident-line form sgn(v) ln|v| is the general one with ln|u| replaced by ln 2
        const double LN2 = 0.69314718055994530942;
        const double uc = ((double)p.ox + (double)(i0 + lane) * L - tg.x) * lambda;
        const double vc = ((double)p.oy + (double)(j0 + lane) * L - tg.y) * lambda;
        double lnu = 0.0, lnv = 0.0;
        if (Q == Q_OFF) {
            if (lane <= nbx) lnu = 0.5 * log(fma(uc, uc, z2));
            if (lane <= nby) lnv = 0.5 * log(fma(vc, vc, z2));
        } else {
            if (lane <= nbx) lnu = uc == 0.0 ? LN2 : log(fabs(uc));
            if (lane <= nby) lnv = vc == 0.0 ? LN2 : log(fabs(vc));
        }
        __syncwarp();
        const int nci = nbx + 1, ncorner = nci * (nby + 1);
        for (int b0 = 0; b0 < ncorner; b0 += 32) {
            const int k = b0 + lane;
            const bool valid = k < ncorner;
            const int kk = valid ? k : 0;
            const int ci = kk % nci, cj = kk / nci;
            const double Lu = __shfl_sync(0xffffffffu, lnu, ci);
            const double Lv = __shfl_sync(0xffffffffu, lnv, cj);
            if (!valid) continue;
            // cells around corner (ci, cj) of the box: lower-left and upper-right count +1
            const int s00 = cj * W + ci, s10 = s00 + 1, s01 = s00 + W, s11 = s01 + 1;
            const double Aw = (cl[s00] - cl[s10]) - (cl[s01] - cl[s11]);
            const double X = (cx[s00] - cx[s10]) - (cx[s01] - cx[s11]);
            const double Y = (cy[s00] - cy[s10]) - (cy[s01] - cy[s11]);
            const double u = ((double)p.ox + (double)(i0 + ci) * L - tg.x) * lambda;
            const double v = ((double)p.oy + (double)(j0 + cj) * L - tg.y) * lambda;
            const double r = sqrt(fma(u, u, Q == Q_OFF ? fma(v, v, z2) : v * v));
            const double t0 = log(fabs(v) + r) - Lu, t1 = log(fabs(u) + r) - Lv;
            // the sign multiplies (ln|v| may be negative)
            double g0 = v > 0.0 ? t0 : (v < 0.0 ? -t0 : 0.0);
            double g0y = u > 0.0 ? t1 : (u < 0.0 ? -t1 : 0.0);
            if constexpr (Q == Q_POT) {
                if (u == 0.0 || v == 0.0) g0 = g0y = 0.0;  // multiplied by u, v
                const double ug = u * g0, vg = v * g0y;
                f[0] += fma(Aw, ug + vg, fma(X, 0.5 * fma(v, r, u * ug), Y * (0.5 * fma(u, r, v * vg))));
            } else if constexpr (Q == Q_OFF) {
                const double T = atan(u * v / (az * r));
                f[0] += fma(-Aw, g0, fma(X, fma(v, g0y, -az * T), -Y * r));
                f[1] += fma(-Aw, g0y, fma(Y, fma(u, g0, -az * T), -X * r));
                f[2] += fma(-sz * Aw, T, z * fma(X, g0, Y * g0y));
            } else {
                f[0] += fma(X * v, g0y, fma(-Aw, g0, -Y * r));
                f[1] += fma(Y * u, g0, fma(-Aw, g0y, -X * r));
            }
        }
    }
    if (!any) return;  // the same in every lane
#pragma unroll
    for (int o = 0; o < NO; ++o) {
        double v = f[o];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (lane == 0) near_out[(int64_t)t * NO + o] += (Q == Q_POT ? -G : G) * v;
    }
}

// The near tables and the targets' sums hold G times the integrals over 2^e, and
// k_cross_add multiplies by 2^e: G, or G H in the potential, and half of H's exponent
// are taken out, so that the tables' planes of sigma (as 1 / sqrt(H)) and of the slopes
// (as sqrt(H)) are of FP32's middle range whatever the units. Powers of two: no bit of
// an ordinary result changes. (Without it the potential's tables overflowed from
// G H^2 = 3e38 on, where the FP32 spectra of the patches' own convolutions, over Px Py,
// still fit. In k_cross_add and not in near_field: one FP64 multiplication more per
// component and warp there cost 6 % of a solve of 2048^2 cells in four patches.)
template <int Q>
int sum_exponent(const sg_plan *plan)
{
    const int h = ilogb(plan->lattice_unit), g = plan->geom.G != 0.0 ? ilogb(plan->geom.G) : 0;
    return g + (Q == Q_POT ? h : 0) + h / 2;
}

// ---------------------------------------------------------------- solve --

template <int Q>
sg_status solve(sg_plan *plan, const sg_workspace *ws, const float *sigma, const float *dx, const float *dy,
                float *o0, float *o1, float *o2, cudaStream_t st)
{
    sg_far &F = *plan->far;
    float *charges = (float *)ws->tile_w;
    sg_timing_begin(ws, SG_STAGE_WEIGHTS, st);
    SG_CUDA_TRY(sg_launch_dep(k_p2m, dim3((F.first[1] + 3) / 4), dim3(256), 0, st, F.desc, F.first[1], plan->patch_dev,
                              sigma, dx, dy, plan->lattice_unit, F.mat, charges, ws->partial,
                              (int64_t)plan->ntargets * q_out<Q>()));
    for (int k = 1; k < F.nlev; ++k) {
        const int n = F.first[k + 1] - F.first[k];
        SG_CUDA_TRY(sg_launch_dep(k_m2m, dim3((n + 3) / 4), dim3(256), 0, st, F.desc, F.first[k], n, F.patch, F.slot,
                                  F.mat, charges));
    }
    sg_timing_end(ws, SG_STAGE_WEIGHTS, st);
    sg_timing_begin(ws, SG_STAGE_DIRECT, st);
    const int grid_n = (plan->ntargets + NEAR_WARPS - 1) / NEAR_WARPS;
    const sg_near_tab &nt = Q == Q_POT ? F.ptab : F.tab;
    const double Gs = ldexp(plan->geom.G, -sum_exponent<Q>(plan));
    far_args A;
    memset(&A, 0, sizeof(A));
    A.blocks = plan->blocks;
    A.nblocks = plan->nblocks;
    A.targets = plan->targets;
    A.pd = plan->patch_dev;
    A.cp = F.patch;
    A.slot = F.slot;
    A.charges = charges;
    A.npatches = plan->npatches;
    A.sigma = sigma;
    A.dx = dx;
    A.dy = dy;
    A.lambda = plan->lattice_unit;
    A.G = Gs;
    A.zl = plan->geom.z / plan->lattice_unit;
    A.ctas = plan->far_grid;
    A.ntargets = plan->ntargets;
    A.keys = F.keys;
    A.tab = (const float2 *)nt.data;
    A.sums = ws->partial;
    SG_CUDA_TRY(sg_launch_dep(k_near_far<Q>, dim3(plan->far_grid + grid_n), dim3(256), 0, st, A));
    if (F.untabled)
        SG_CUDA_TRY(sg_launch_dep(k_near_corner<Q>, dim3(grid_n), dim3(NEAR_WARPS * 32), 0, st, plan->targets,
                                  plan->ntargets, plan->patch_dev, plan->npatches, sigma, dx, dy, F.keys,
                                  plan->lattice_unit, Gs, plan->geom.z, ws->partial));
    SG_CUDA_TRY(sg_launch_dep(k_cross_add<Q>, dim3((plan->ntargets + 255) / 256), dim3(256), 0, st, plan->targets,
                              plan->ntargets, A.sums, ldexp(1.0, sum_exponent<Q>(plan)), o0, o1, o2));
    SG_CUDA_TRY(cudaGetLastError());
    sg_timing_end(ws, SG_STAGE_DIRECT, st);
    return SG_OK;
}

template <int Q>
size_t table_bytes(const sg_far &F)
{
    return (size_t)std::max(1, F.nclass) * q_planes<Q>() * NEAR_CELLS * sizeof(float2);
}

// Give back tables whose build failed (nt.data set means built).
template <int Q>
void drop_tables(sg_plan *plan, sg_near_tab &nt)
{
    if (!nt.data) return;
    cudaFree(nt.data);
    nt.data = nullptr;
    plan->device_bytes -= (int64_t)table_bytes<Q>(*plan->far);
}

// Build the near tables of quantity Q (asynchronous on the legacy default stream).
template <int Q>
sg_status build_tables(sg_plan *plan, sg_near_tab &nt)
{
    sg_far &F = *plan->far;
    const size_t bytes = table_bytes<Q>(F);
    cudaError_t e = cudaMalloc(&nt.data, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        nt.data = nullptr;
        sg_set_last_cuda_error(e, "cudaMalloc");
        return e == cudaErrorMemoryAllocation ? SG_ENOMEM : SG_ECUDA;
    }
    plan->device_bytes += (int64_t)bytes;
    // the keys in the order of their classes
    near_list L;
    memset(&L, 0, sizeof(L));
    std::vector<std::pair<int, int>> order;  // first class, key
    for (int k = 0; k < SG_NT_STEPS * SG_NT_KEYS; ++k)
        if (F.keys_host[k] >= 0) order.push_back({F.keys_host[k], k});
    std::sort(order.begin(), order.end());
    for (const auto &o : order) {
        L.first[L.n] = o.first;
        L.g[L.n] = o.second % SG_NT_KEYS - 1;
        L.H[L.n] = (double)(1LL << (o.second / SG_NT_KEYS)) * plan->lattice_unit;
        ++L.n;
    }
    L.first[L.n] = F.nclass;
    if (F.nclass == 0) return SG_OK;
    const int grid = (int)std::min<int64_t>(((int64_t)F.nclass * NEAR_CELLS + 127) / 128, 1 << 16);
    k_near_table<Q><<<grid, 128>>>((float2 *)nt.data, L, ldexp(plan->geom.G, -sum_exponent<Q>(plan)), plan->geom.z);
    e = cudaGetLastError();
    if (e != cudaSuccess) {
        drop_tables<Q>(plan, nt);
        sg_set_last_cuda_error(e, "k_near_table");
        return SG_ECUDA;
    }
    return SG_OK;
}

// L_n(x) on the Chebyshev points, FP64
double lagrange(int n, double x)
{
    double v = 1.0;
    for (int r = 0; r < NP; ++r)
        if (r != n) v *= (x - cos((2 * r + 1) * M_PI / 16)) / (cos((2 * n + 1) * M_PI / 16) - cos((2 * r + 1) * M_PI / 16));
    return v;
}

// Keys of the near tables: the first class (position) of every source cell width
// 2^s (lattice units) and width ratio 2^g up to 2^gmax, -1 for none; returns the
// number of classes. A ratio has a table where its 4^g positions are at most the
// targets of the narrower level: a position's table takes about 3.4 corner
// evaluations to build.
int near_keys(int nlev, const int64_t *level_targets, int gmax, int *keys, bool &untabled)
{
    for (int k = 0; k < SG_NT_STEPS * SG_NT_KEYS; ++k) keys[k] = -1;
    int n = 0;
    untabled = false;
    for (int ls = 0; ls < nlev; ++ls)
        for (int lt = 0; lt < nlev; ++lt) {
            if (level_targets[lt] == 0) continue;
            const int g = std::max(-1, lt - ls);
            if (g > gmax || (g > 0 && (1LL << (2 * g)) > level_targets[lt])) {
                untabled = true;
                continue;
            }
            int &key = keys[(nlev - ls) * SG_NT_KEYS + g + 1];
            if (key >= 0) continue;
            key = n;
            n += g < 0 ? 1 : 1 << (2 * g);
        }
    return n;
}

}  // namespace

int64_t sg_near_table_bytes(int nlevels, const int64_t *level_targets, double z, int gmax)
{
    int keys[SG_NT_STEPS * SG_NT_KEYS];
    bool untabled;
    return (int64_t)near_keys(nlevels, level_targets, gmax, keys, untabled) *
           (z != 0.0 ? q_planes<Q_OFF>() : q_planes<Q_FORCE>()) * NEAR_CELLS * (int64_t)sizeof(float2);
}

int64_t sg_far_bytes(int64_t nclusters, int64_t ntargets, double z)
{
    return nclusters * (NQ * 4 + 24) + ntargets * (z != 0.0 ? 24 : 16);
}

void sg_far_free(sg_plan *plan)
{
    if (!plan->far) return;
    cudaFree(plan->far->patch);
    cudaFree(plan->far->slot);
    cudaFree(plan->far->desc);
    cudaFree(plan->far->mat);
    cudaFree(plan->far->keys);
    cudaFree(plan->far->tab.data);
    cudaFree(plan->far->ptab.data);
    delete plan->far;
    plan->far = nullptr;
}

sg_status sg_far_setup(sg_plan *plan, const int *const *codes, int nlevels, const int64_t *level_targets, int gmax)
{
    sg_far *F = new (std::nothrow) sg_far();
    if (!F) return SG_ENOMEM;
    memset(F, 0, sizeof(*F));
    plan->far = F;
    // cluster grids of every patch; slots of the clusters that hold an existing cell
    std::vector<sg_cl_patch> cp(plan->npatches);
    std::vector<int> slot;
    std::vector<int4> desc;
    int nlev = 1;
    for (int p = 0; p < plan->npatches; ++p) {
        sg_cl_patch &c = cp[p];
        memset(&c, 0, sizeof(c));
        const sg_patch_dev &d = plan->pp[p].d;
        int nx = (d.nx + CL - 1) / CL, ny = (d.ny + CL - 1) / CL;
        for (;;) {
            c.nx[c.nlev] = nx;
            c.ny[c.nlev] = ny;
            c.off[c.nlev] = (int)slot.size();
            slot.resize(slot.size() + (size_t)nx * ny, -1);
            ++c.nlev;
            if (nx == 1 && ny == 1) break;
            nx = (nx + 1) / 2;
            ny = (ny + 1) / 2;
        }
        nlev = std::max(nlev, c.nlev);
    }
    for (int k = 0; k < nlev; ++k) {
        F->first[k] = (int)desc.size();
        for (int p = 0; p < plan->npatches; ++p) {
            const sg_cl_patch &c = cp[p];
            const sg_patch_dev &d = plan->pp[p].d;
            if (k >= c.nlev) continue;
            for (int cy = 0; cy < c.ny[k]; ++cy)
                for (int cx = 0; cx < c.nx[k]; ++cx) {
                    bool any = false;
                    if (k == 0) {
                        for (int j = cy * CL; j < std::min(d.ny, (cy + 1) * CL) && !any; ++j)
                            for (int i = cx * CL; i < std::min(d.nx, (cx + 1) * CL) && !any; ++i)
                                any = codes[p][(size_t)j * d.nx + i] != SG_CELL_ABSENT;
                    } else {
                        for (int q = 0; q < 4 && !any; ++q) {
                            const int x = 2 * cx + (q & 1), y = 2 * cy + (q >> 1);
                            any = x < c.nx[k - 1] && y < c.ny[k - 1] && slot[c.off[k - 1] + y * c.nx[k - 1] + x] >= 0;
                        }
                    }
                    if (!any) continue;
                    slot[c.off[k] + cy * c.nx[k] + cx] = (int)desc.size();
                    desc.push_back(make_int4(p, cx, cy, k));
                }
        }
    }
    for (int k = nlev; k <= SG_CL_LEVELS; ++k) F->first[k] = (int)desc.size();
    // (the levels of a patch without an existing cell hold no cluster; a launch over none is an error)
    while (nlev > 1 && F->first[nlev] == F->first[nlev - 1]) --nlev;
    F->nlev = nlev;
    F->ncl = (int)desc.size();
    // interpolation matrices: A_n[i], B_n[i] (8-point Gauss-Legendre, exact for these degrees), C_h[n'][n]
    static const double gx[4] = {0.1834346424956498, 0.5255324099163290, 0.7966664774136267, 0.9602898564975363};
    static const double gw[4] = {0.3626837833783620, 0.3137066458778873, 0.2223810344533745, 0.1012285362903763};
    std::vector<float> mat(2 * NP * CL + 2 * NQ);
    for (int n = 0; n < NP; ++n)
        for (int i = 0; i < CL; ++i) {
            const double c = -1.0 + (i + 0.5) * (2.0 / CL), hw = 1.0 / CL;  // cell centre, half width
            double a = 0.0, b = 0.0;
            for (int u = 0; u < 8; ++u) {
                const double s = (u & 1 ? 1.0 : -1.0) * gx[u >> 1] * hw, w = gw[u >> 1] * hw;
                a += w * lagrange(n, c + s);
                b += w * s * lagrange(n, c + s);
            }
            mat[n * CL + i] = (float)a;
            mat[NP * CL + n * CL + i] = (float)b;
        }
    for (int h = 0; h < 2; ++h)
        for (int u = 0; u < NP; ++u)
            for (int n = 0; n < NP; ++n)
                mat[2 * NP * CL + h * NQ + u * NP + n] = (float)lagrange(n, 0.5 * (cos((2 * u + 1) * M_PI / 16) + (h ? 1.0 : -1.0)));
    F->nclass = near_keys(nlevels, level_targets, gmax, F->keys_host, F->untabled);
    SG_TRY(sg_plan_upload(plan, (void **)&F->patch, cp.data(), cp.size() * sizeof(sg_cl_patch)));
    SG_TRY(sg_plan_upload(plan, (void **)&F->slot, slot.data(), slot.size() * sizeof(int)));
    SG_TRY(sg_plan_upload(plan, (void **)&F->desc, desc.data(), desc.size() * sizeof(int4)));
    SG_TRY(sg_plan_upload(plan, (void **)&F->mat, mat.data(), mat.size() * sizeof(float)));
    SG_TRY(sg_plan_upload(plan, (void **)&F->keys, F->keys_host, sizeof(F->keys_host)));
    plan->ws_tile_bytes = (int64_t)F->ncl * NQ * (int64_t)sizeof(float);
    plan->ws_partial_bytes = (int64_t)plan->ntargets * (plan->geom.z != 0.0 ? 3 : 2) * (int64_t)sizeof(double);
    plan->far_grid = plan->nblocks;
    if (plan->geom.z != 0.0) return build_tables<Q_OFF>(plan, F->tab);
    return build_tables<Q_FORCE>(plan, F->tab);
}

sg_status sg_far_potential_tables(sg_plan *plan)
{
    if (!plan->far || plan->far->ptab.data) return SG_OK;
    sg_status s = build_tables<Q_POT>(plan, plan->far->ptab);
    cudaError_t e = cudaDeviceSynchronize();
    if (s == SG_OK && e != cudaSuccess) {
        drop_tables<Q_POT>(plan, plan->far->ptab);
        sg_set_last_cuda_error(e, "near tables of the potential");
        s = SG_ECUDA;
    }
    return s;
}

sg_status sg_far_solve(sg_plan *plan, const sg_workspace *ws, const float *sigma, const float *dx, const float *dy,
                       float *fx, float *fy, float *fz, cudaStream_t st)
{
    if (plan->geom.z != 0.0) return solve<Q_OFF>(plan, ws, sigma, dx, dy, fx, fy, fz, st);
    return solve<Q_FORCE>(plan, ws, sigma, dx, dy, fx, fy, nullptr, st);
}

sg_status sg_far_potential(sg_plan *plan, const sg_workspace *ws, const float *sigma, const float *dx, const float *dy,
                           float *phi, cudaStream_t st)
{
    return solve<Q_POT>(plan, ws, sigma, dx, dy, phi, nullptr, nullptr, st);
}
