// Cross-patch direct sum of an AMR hierarchy (Section 2, Eq. eqnXforce2 with
// the order-1 reconstruction of Eq. eqnGamma). The sources are the composite
// fields S_p of every patch (see amr.cu); each leaf target receives the sum
// over the cells of every patch other than its own, whose contribution comes
// from the FFT convolution of its own patch.
//
// FP64 plans: corner form. Every cell integral is a double difference over the
// cell's four corners, dd_i f = sum_c s_ic f(c - t) with s = +1 at the
// lower-left and upper-right corners and -1 at the other two. Writing the
// reconstruction of source i evaluated at the target, l_i(t) = sigma0_i +
// deltax_i (x_t - xc_i) + deltay_i (y_t - yc_i), the closed forms of Section 2 give
//   Fx(t) = G sum_c [ -A_c(t) g0(c - t) + X_c v g0y(c - t) - Y_c r(c - t) ]
//   Fy(t) = G sum_c [ -A_c(t) g0y(c - t) + Y_c u g0(c - t) - X_c r(c - t) ]
// with A_c(t) = sum_i s_ic l_i(t), X_c = sum_i s_ic deltax_i, Y_c = sum_i s_ic deltay_i,
//   g0(u, v) = asinh(v/|u|) = ln(v + r) - ln|u|,   g0y(u, v) = asinh(u/|v|),
// since the terms that depend on u alone (ln|u|) or v alone cancel in each
// cell's double difference. On u = 0 the coincident-line form of Section 2,
// sgn(v) ln|v|, is the same as g0 with ln|u| replaced by ln 2 (likewise for
// g0y on v = 0). A_c(t) = B_c + (x_t - x_T) X_c + (y_t - y_T) Y_c with B_c
// built relative to the tile origin (x_T, y_T). Pairs are summed in tiles of
// 16 x 16 corners staged in shared memory, per tile and across tiles in FP64.
//
// FP32 plans: cross32.cu. The corner form is unsuited to FP32: a corner's term is
// O(sigma) times an O(1) logarithm while a distant cell's integral is O(sigma H^2 /
// rho^2), so rounding of every corner term, not the integrals, would set the error
// (it grows like the square root of the number of corners).
//
// The mid-plane potential (sg_potential on hierarchies of this path) is the
// same sum with the kernel 1/r: its corner form and kernels follow the force's
// (see the potential section below).
#include "common.cuh"

#include <math.h>

namespace {

// ================================================================= FP64 ====

// One thread per (tile, corner): signed sums of the (up to) four cells of the
// patch around the corner, from the composite source fields.
template <typename T>
__global__ void k_corner_weights(const sg_tile_desc *__restrict__ tiles, int ntiles, const sg_patch_dev *__restrict__ pd,
                                 const T *__restrict__ sigma, const T *__restrict__ dx,
                                 const T *__restrict__ dy, double lambda, double *__restrict__ wout)
{
    const int64_t total = (int64_t)ntiles * SG_TILE_N;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int t = (int)(e / SG_TILE_N), k = (int)(e % SG_TILE_N);
        const sg_tile_desc td = tiles[t];
        const sg_patch_dev p = pd[td.patch];
        const int ci = td.ci0 + k % SG_TILE_X, cj = td.cj0 + k / SG_TILE_X;
        double B = 0.0, X = 0.0, Y = 0.0;
        if (ci <= p.nx && cj <= p.ny) {
            for (int q = 0; q < 4; ++q) {
                const int i = ci - 1 + (q & 1), j = cj - 1 + (q >> 1);
                if (i < 0 || i >= p.nx || j < 0 || j >= p.ny) continue;
                const double s = (q == 0 || q == 3) ? 1.0 : -1.0;
                const int64_t o = p.cell_off + (int64_t)j * p.nx + i;
                const double s0 = (double)sigma[o];
                const double sx = dx ? (double)dx[o] : 0.0;
                const double sy = dy ? (double)dy[o] : 0.0;
                // cell centre (lattice) = patch origin + (2i + 1) step / 2
                const double cx = p.ox + (2 * i + 1) * (p.step / 2);
                const double cy = p.oy + (2 * j + 1) * (p.step / 2);
                B += s * (s0 + sx * (td.ox - cx) * lambda + sy * (td.oy - cy) * lambda);
                X += s * sx;
                Y += s * sy;
            }
        }
        wout[e * 4 + 0] = B;
        wout[e * 4 + 1] = X * lambda;
        wout[e * 4 + 2] = Y * lambda;
        wout[e * 4 + 3] = 0.0;
    }
}

struct acc4 {
    double xl, xr, yl, yr;
};

// FP64 pair loop over one corner tile (natural logarithms).
__device__ __forceinline__ void tile_pairs_f64(const sg_dvec4 *__restrict__ w, double du0, double dv0, double st,
                                               double dxT, double dyT, acc4 &acc)
{
    double Lu[SG_TILE_X];
#pragma unroll
    for (int c = 0; c < SG_TILE_X; ++c) {
        const double u = fma((double)c, st, du0);
        Lu[c] = u == 0.0 ? 0.69314718055994530942 : log(fabs(u));
    }
    double sxl = 0, sxr = 0, syl = 0, syr = 0;
#pragma unroll 1
    for (int r = 0; r < SG_TILE_Y; ++r) {
        const double v = fma((double)r, st, dv0);
        const double av = fabs(v), v2 = v * v;
        const double Lv = v == 0.0 ? 0.69314718055994530942 : log(av);
#pragma unroll 4
        for (int c = 0; c < SG_TILE_X; ++c) {
            const sg_dvec4 wc = w[r * SG_TILE_X + c];
            const double u = fma((double)c, st, du0);
            const double rr = sqrt(fma(u, u, v2));
            const double la = log(av + rr);
            const double lb = log(fabs(u) + rr);
            const double g0 = v == 0.0 ? 0.0 : copysign(la - Lu[c], v);
            const double g0y = u == 0.0 ? 0.0 : copysign(lb - Lv, u);
            const double A = fma(dxT, wc.y, fma(dyT, wc.z, wc.x));
            sxl = fma(-A, g0, sxl);
            sxl = fma(wc.y, v * g0y, sxl);
            sxr = fma(-wc.z, rr, sxr);
            syl = fma(-A, g0y, syl);
            syl = fma(wc.z, u * g0, syl);
            syr = fma(-wc.y, rr, syr);
        }
    }
    acc.xl += sxl;
    acc.xr += sxr;
    acc.yl += syl;
    acc.yr += syr;
}

// grid (nblocks, nsplit); block SG_DIRECT_THREADS; one leaf target per thread.
__global__ void __launch_bounds__(SG_DIRECT_THREADS) k_cross_direct(
    const sg_target_block *__restrict__ blocks, const int4 *__restrict__ targets, const sg_tile_desc *__restrict__ tiles,
    int ntiles, const double *__restrict__ wts, int nsplit, double G, double *__restrict__ fx, double *__restrict__ fy,
    double *__restrict__ partial, int ntargets)
{
    __shared__ sg_dvec4 sw[SG_TILE_N];
    const sg_target_block blk = blocks[blockIdx.x];
    const int split = blockIdx.y;
    const int t0 = (int)((int64_t)ntiles * split / nsplit);
    const int t1 = (int)((int64_t)ntiles * (split + 1) / nsplit);
    const bool active = threadIdx.x < blk.count;
    int4 tg = make_int4(0, 0, -1, -1);
    if (active) tg = targets[blk.first + threadIdx.x];
    acc4 acc = {0.0, 0.0, 0.0, 0.0};
    const sg_dvec4 *wv = reinterpret_cast<const sg_dvec4 *>(wts);
    for (int t = t0; t < t1; ++t) {
        const sg_tile_desc td = tiles[t];
        if (td.patch == blk.patch) continue;  // same-patch pairs come from the FFT
        __syncthreads();
        for (int k = threadIdx.x; k < SG_TILE_N; k += SG_DIRECT_THREADS) sw[k] = wv[(int64_t)t * SG_TILE_N + k];
        __syncthreads();
        tile_pairs_f64(sw, (double)(td.ox - tg.x), (double)(td.oy - tg.y), (double)td.step, (double)(tg.x - td.ox),
                       (double)(tg.y - td.oy), acc);
    }
    if (!active) return;
    const double Fx = G * (acc.xl + acc.xr);
    const double Fy = G * (acc.yl + acc.yr);
    const int ti = blk.first + threadIdx.x;
    if (nsplit == 1) {
        fx[tg.z] += Fx;
        fy[tg.z] += Fy;
    } else {
        partial[((int64_t)split * ntargets + ti) * 2 + 0] = Fx;
        partial[((int64_t)split * ntargets + ti) * 2 + 1] = Fy;
    }
}

// Fixed-order sum of the per-split partials into the outputs.
__global__ void k_cross_reduce(const int4 *__restrict__ targets, int ntargets, int nsplit,
                               const double *__restrict__ partial, double *__restrict__ fx, double *__restrict__ fy)
{
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < ntargets; t += gridDim.x * blockDim.x) {
        double sx = 0.0, sy = 0.0;
        for (int s = 0; s < nsplit; ++s) {
            sx += partial[((int64_t)s * ntargets + t) * 2 + 0];
            sy += partial[((int64_t)s * ntargets + t) * 2 + 1];
        }
        const int o = targets[t].z;
        fx[o] += sx;
        fy[o] += sy;
    }
}

sg_status cross_solve_f64(sg_plan *plan, const sg_workspace *ws, const double *sigma, const double *dx,
                          const double *dy, double *fx, double *fy, cudaStream_t st)
{
    double *w = (double *)ws->tile_w;
    const int64_t nw = (int64_t)plan->ntiles * SG_TILE_N;
    int grid_w = (int)((nw + 255) / 256);
    if (grid_w > 65535) grid_w = 65535;
    sg_timing_begin(ws, SG_STAGE_WEIGHTS, st);
    k_corner_weights<double><<<grid_w, 256, 0, st>>>(plan->tiles, plan->ntiles, plan->patch_dev, sigma, dx, dy,
                                             plan->lattice_unit, w);
    SG_CUDA_TRY(cudaGetLastError());
    sg_timing_end(ws, SG_STAGE_WEIGHTS, st);
    sg_timing_begin(ws, SG_STAGE_DIRECT, st);
    dim3 grid(plan->nblocks, plan->nsplit);
    k_cross_direct<<<grid, SG_DIRECT_THREADS, 0, st>>>(plan->blocks, plan->targets, plan->tiles, plan->ntiles, w,
                                                       plan->nsplit, plan->geom.G, fx, fy, ws->partial,
                                                       plan->ntargets);
    SG_CUDA_TRY(cudaGetLastError());
    if (plan->nsplit > 1) {
        k_cross_reduce<<<(plan->ntargets + 255) / 256, 256, 0, st>>>(plan->targets, plan->ntargets, plan->nsplit,
                                                                      ws->partial, fx, fy);
        SG_CUDA_TRY(cudaGetLastError());
    }
    sg_timing_end(ws, SG_STAGE_DIRECT, st);
    return SG_OK;
}

// ============================================================ potential ====
//
// The same cross-patch sum for the mid-plane potential Phi = -G sum_i of the
// cell integrals of (sigma0_i + deltax_i (xbar - xc_i) + deltay_i (ybar - yc_i)) / r.
// With l_i(t) as above, xbar - xc_i = u + (x_t - xc_i), so the cell integral is
// l_i(t) P0 + deltax_i U + deltay_i V with P0, U, V the integrals of 1/r, u/r,
// v/r, and Section 2's antiderivatives give the corner form
//   Phi(t) = -G sum_c [ A_c(t) F0(c - t) + X_c Fu(c - t) + Y_c Fv(c - t) ],
//   F0 = u g0 + v g0y,  Fu = (v r + u^2 g0) / 2,  Fv = (u r + v^2 g0y) / 2
// (u ln(v + r) + v ln(u + r) and (v r + u^2 ln(v + r)) / 2 with the terms of one
// variable alone dropped, which cancel in each cell's double difference; every
// term vanishes where its factor u or v does, so the potential needs no
// coincident-line form).

// The corner functions of the potential at (u, v) = corner - target, r = |(u, v)|,
// from the logarithms ln(|v| + r) - ln|u| and ln(|u| + r) - ln|v| (t0, t1);
// accumulates A F0 + X Fu + Y Fv.
__device__ __forceinline__ double corner_pot(double u, double v, double r, double t0, double t1, double A, double X,
                                             double Y)
{
    const double g0 = (v == 0.0 || u == 0.0) ? 0.0 : (v > 0.0 ? t0 : -t0);   // multiplied by u, u^2
    const double g0y = (u == 0.0 || v == 0.0) ? 0.0 : (u > 0.0 ? t1 : -t1);  // multiplied by v, v^2
    const double ug = u * g0, vg = v * g0y;
    const double F0 = ug + vg;
    const double Fu = 0.5 * fma(v, r, u * ug);
    const double Fv = 0.5 * fma(u, r, v * vg);
    return fma(A, F0, fma(X, Fu, Y * Fv));
}

// FP64 corner form of the potential (k_cross_direct's layout; one output).
__global__ void __launch_bounds__(SG_DIRECT_THREADS) k_cross_direct_pot(
    const sg_target_block *__restrict__ blocks, const int4 *__restrict__ targets, const sg_tile_desc *__restrict__ tiles,
    int ntiles, const double *__restrict__ wts, int nsplit, double G, double lambda, double *__restrict__ phi,
    double *__restrict__ partial, int ntargets)
{
    __shared__ sg_dvec4 sw[SG_TILE_N];
    const sg_target_block blk = blocks[blockIdx.x];
    const int split = blockIdx.y;
    const int t0 = (int)((int64_t)ntiles * split / nsplit);
    const int t1 = (int)((int64_t)ntiles * (split + 1) / nsplit);
    const bool active = threadIdx.x < blk.count;
    int4 tg = make_int4(0, 0, -1, -1);
    if (active) tg = targets[blk.first + threadIdx.x];
    double acc = 0.0;
    const sg_dvec4 *wv = reinterpret_cast<const sg_dvec4 *>(wts);
    for (int t = t0; t < t1; ++t) {
        const sg_tile_desc td = tiles[t];
        if (td.patch == blk.patch) continue;  // same-patch pairs come from the FFT
        __syncthreads();
        for (int k = threadIdx.x; k < SG_TILE_N; k += SG_DIRECT_THREADS) sw[k] = wv[(int64_t)t * SG_TILE_N + k];
        __syncthreads();
        const double du0 = (double)(td.ox - tg.x), dv0 = (double)(td.oy - tg.y), st = (double)td.step;
        const double dxT = (double)(tg.x - td.ox), dyT = (double)(tg.y - td.oy);
        double Lu[SG_TILE_X];
#pragma unroll
        for (int c = 0; c < SG_TILE_X; ++c) {
            const double u = fma((double)c, st, du0);
            Lu[c] = u == 0.0 ? 0.0 : log(fabs(u));
        }
        double sum = 0.0;
#pragma unroll 1
        for (int r = 0; r < SG_TILE_Y; ++r) {
            const double v = fma((double)r, st, dv0);
            const double av = fabs(v), v2 = v * v;
            const double Lv = v == 0.0 ? 0.0 : log(av);
#pragma unroll 4
            for (int c = 0; c < SG_TILE_X; ++c) {
                const sg_dvec4 wc = sw[r * SG_TILE_X + c];
                const double u = fma((double)c, st, du0);
                const double rr = sqrt(fma(u, u, v2));
                const double A = fma(dxT, wc.y, fma(dyT, wc.z, wc.x));
                sum += corner_pot(u, v, rr, log(av + rr) - Lu[c], log(fabs(u) + rr) - Lv, A, wc.y, wc.z);
            }
        }
        acc += sum;
    }
    if (!active) return;
    // corner offsets are in lattice units: F0 is a length and Fu, Fv are lengths
    // squared, against weights X, Y that carry one lattice unit already, so one
    // factor lambda makes every term physical
    const double P = -G * lambda * acc;
    const int ti = blk.first + threadIdx.x;
    if (nsplit == 1) phi[tg.z] += P;
    else partial[(int64_t)split * ntargets + ti] = P;
}

__global__ void k_cross_reduce_pot(const int4 *__restrict__ targets, int ntargets, int nsplit,
                                   const double *__restrict__ partial, double *__restrict__ phi)
{
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < ntargets; t += gridDim.x * blockDim.x) {
        double sum = 0.0;
        for (int s = 0; s < nsplit; ++s) sum += partial[(int64_t)s * ntargets + t];
        phi[targets[t].z] += sum;
    }
}

sg_status cross_potential_f64(sg_plan *plan, const sg_workspace *ws, const double *sigma, const double *dx,
                              const double *dy, double *phi, cudaStream_t st)
{
    double *w = (double *)ws->tile_w;
    const int64_t nw = (int64_t)plan->ntiles * SG_TILE_N;
    int grid_w = (int)((nw + 255) / 256);
    if (grid_w > 65535) grid_w = 65535;
    sg_timing_begin(ws, SG_STAGE_WEIGHTS, st);
    k_corner_weights<double><<<grid_w, 256, 0, st>>>(plan->tiles, plan->ntiles, plan->patch_dev, sigma, dx, dy,
                                             plan->lattice_unit, w);
    SG_CUDA_TRY(cudaGetLastError());
    sg_timing_end(ws, SG_STAGE_WEIGHTS, st);
    sg_timing_begin(ws, SG_STAGE_DIRECT, st);
    dim3 grid(plan->nblocks, plan->nsplit);
    k_cross_direct_pot<<<grid, SG_DIRECT_THREADS, 0, st>>>(plan->blocks, plan->targets, plan->tiles, plan->ntiles, w,
                                                           plan->nsplit, plan->geom.G, plan->lattice_unit, phi,
                                                           ws->partial, plan->ntargets);
    SG_CUDA_TRY(cudaGetLastError());
    if (plan->nsplit > 1) {
        k_cross_reduce_pot<<<(plan->ntargets + 255) / 256, 256, 0, st>>>(plan->targets, plan->ntargets,
                                                                          plan->nsplit, ws->partial, phi);
        SG_CUDA_TRY(cudaGetLastError());
    }
    sg_timing_end(ws, SG_STAGE_DIRECT, st);
    return SG_OK;
}

// ============================================================ off plane ====
//
// Targets at height z != 0 above the plane of the sources (Section 2's kernels
// with R = sqrt(u^2 + v^2 + z^2)): every pair in the corner form with the
// off-plane antiderivatives.
// With the corner weights A_c(t), X_c, Y_c as in the plane,
//   Fx(t) = G sum_c [ -A_c G0 + X_c (v G0y - |z| T) - Y_c R ]
//   Fy(t) = G sum_c [ -A_c G0y + Y_c (u G0 - |z| T) - X_c R ]
//   Fz(t) = G sum_c [ -sgn(z) A_c T + z (X_c G0 + Y_c G0y) ]
// G0 = asinh(v / rho_u), rho_u = sqrt(u^2 + z^2), G0y = asinh(u / rho_v),
// T = atan(u v / (|z| R)): the x-family kernels K^{x,0} = -dd G0,
// K^{x,x} = -m K^{x,0} + dd[v G0y] - |z| dd T, K^{x,y} = -n K^{x,0} - dd R, and
// K^{z,0} = -sgn(z) dd T, K^{z,x} = -m K^{z,0} - z K^{x,0} (y-family by
// symmetry), the -m, -n terms folded into A_c(t). R >= |z| > 0: no coincident
// lines. asinh(v / rho) = sgn(v) (ln(|v| + R) - ln rho), rho per corner column
// (row) of the tile.

// grid (nblocks, nsplit); one leaf target per thread; partial[(split, target)][3].
__global__ void __launch_bounds__(SG_DIRECT_THREADS) k_cross_direct_z(
    const sg_target_block *__restrict__ blocks, const int4 *__restrict__ targets, const sg_tile_desc *__restrict__ tiles,
    int ntiles, const double *__restrict__ wts, int nsplit, double G, double zl, double *__restrict__ partial,
    int ntargets)
{
    __shared__ sg_dvec4 sw[SG_TILE_N];
    const sg_target_block blk = blocks[blockIdx.x];
    const int split = blockIdx.y;
    const int t0 = (int)((int64_t)ntiles * split / nsplit);
    const int t1 = (int)((int64_t)ntiles * (split + 1) / nsplit);
    const bool active = threadIdx.x < blk.count;
    int4 tg = make_int4(0, 0, -1, -1);
    if (active) tg = targets[blk.first + threadIdx.x];
    const double az = fabs(zl), z2 = zl * zl, sz = zl > 0.0 ? 1.0 : -1.0;
    double fx = 0.0, fy = 0.0, fz = 0.0;
    const sg_dvec4 *wv = reinterpret_cast<const sg_dvec4 *>(wts);
    for (int t = t0; t < t1; ++t) {
        const sg_tile_desc td = tiles[t];
        if (td.patch == blk.patch) continue;  // same-patch pairs come from the FFT
        __syncthreads();
        for (int k = threadIdx.x; k < SG_TILE_N; k += SG_DIRECT_THREADS) sw[k] = wv[(int64_t)t * SG_TILE_N + k];
        __syncthreads();
        const double du0 = (double)(td.ox - tg.x), dv0 = (double)(td.oy - tg.y), st = (double)td.step;
        const double dxT = (double)(tg.x - td.ox), dyT = (double)(tg.y - td.oy);
        double Lu[SG_TILE_X];
#pragma unroll
        for (int c = 0; c < SG_TILE_X; ++c) {
            const double u = fma((double)c, st, du0);
            Lu[c] = 0.5 * log(fma(u, u, z2));  // ln rho_u
        }
        double sx = 0.0, sy = 0.0, sz3 = 0.0;
#pragma unroll 1
        for (int r = 0; r < SG_TILE_Y; ++r) {
            const double v = fma((double)r, st, dv0);
            const double av = fabs(v), v2z = fma(v, v, z2);
            const double Lv = 0.5 * log(v2z);  // ln rho_v
#pragma unroll 2
            for (int c = 0; c < SG_TILE_X; ++c) {
                const sg_dvec4 wc = sw[r * SG_TILE_X + c];
                const double u = fma((double)c, st, du0);
                const double R = sqrt(fma(u, u, v2z));
                const double ta = log(av + R) - Lu[c];
                const double tb = log(fabs(u) + R) - Lv;
                const double g0 = v > 0.0 ? ta : (v < 0.0 ? -ta : 0.0);
                const double g0y = u > 0.0 ? tb : (u < 0.0 ? -tb : 0.0);
                const double T = atan(u * v / (az * R));
                const double A = fma(dxT, wc.y, fma(dyT, wc.z, wc.x));
                sx += fma(-A, g0, fma(wc.y, fma(v, g0y, -az * T), -wc.z * R));
                sy += fma(-A, g0y, fma(wc.z, fma(u, g0, -az * T), -wc.y * R));
                sz3 += fma(-sz * A, T, zl * fma(wc.y, g0, wc.z * g0y));
            }
        }
        fx += sx;
        fy += sy;
        fz += sz3;
    }
    if (!active) return;
    double *o = partial + ((int64_t)split * ntargets + blk.first + threadIdx.x) * 3;
    o[0] = G * fx;
    o[1] = G * fy;
    o[2] = G * fz;
}

// Fixed-order sum of the splits, added into the outputs.
template <typename T>
__global__ void k_cross_reduce_z(const int4 *__restrict__ targets, int ntargets, int nsplit,
                                 const double *__restrict__ partial, T *__restrict__ fx, T *__restrict__ fy,
                                 T *__restrict__ fz)
{
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < ntargets; t += gridDim.x * blockDim.x) {
        double a = 0.0, b = 0.0, c = 0.0;
        for (int s = 0; s < nsplit; ++s) {
            const double *q = partial + ((int64_t)s * ntargets + t) * 3;
            a += q[0];
            b += q[1];
            c += q[2];
        }
        const int o = targets[t].z;
        fx[o] = (T)((double)fx[o] + a);
        fy[o] = (T)((double)fy[o] + b);
        if (fz) fz[o] = (T)((double)fz[o] + c);  // sg_force on such a plan returns Fx, Fy only
    }
}

template <typename T>
sg_status cross_solve_z(sg_plan *plan, const sg_workspace *ws, const T *sigma, const T *dx, const T *dy, T *fx,
                        T *fy, T *fz, cudaStream_t st)
{
    double *w = (double *)ws->tile_w;
    const int64_t nw = (int64_t)plan->ntiles * SG_TILE_N;
    int grid_w = (int)((nw + 255) / 256);
    if (grid_w > 65535) grid_w = 65535;
    sg_timing_begin(ws, SG_STAGE_WEIGHTS, st);
    k_corner_weights<T><<<grid_w, 256, 0, st>>>(plan->tiles, plan->ntiles, plan->patch_dev, sigma, dx, dy,
                                                plan->lattice_unit, w);
    SG_CUDA_TRY(cudaGetLastError());
    sg_timing_end(ws, SG_STAGE_WEIGHTS, st);
    sg_timing_begin(ws, SG_STAGE_DIRECT, st);
    dim3 grid(plan->nblocks, plan->nsplit);
    k_cross_direct_z<<<grid, SG_DIRECT_THREADS, 0, st>>>(plan->blocks, plan->targets, plan->tiles, plan->ntiles, w,
                                                         plan->nsplit, plan->geom.G, plan->geom.z / plan->lattice_unit,
                                                         ws->partial, plan->ntargets);
    SG_CUDA_TRY(cudaGetLastError());
    k_cross_reduce_z<T><<<(plan->ntargets + 255) / 256, 256, 0, st>>>(plan->targets, plan->ntargets, plan->nsplit,
                                                                       ws->partial, fx, fy, fz);
    SG_CUDA_TRY(cudaGetLastError());
    sg_timing_end(ws, SG_STAGE_DIRECT, st);
    return SG_OK;
}

}  // namespace

sg_status sg_cross_solve(sg_plan *plan, const sg_workspace *ws, const void *sigma, const void *dx, const void *dy,
                         void *fx, void *fy, void *fz, cudaStream_t st)
{
    if (plan->ntiles == 0 || plan->ntargets == 0) return SG_OK;
    if (plan->prec == SG_FP32)
        return sg_far_solve(plan, ws, (const float *)sigma, (const float *)dx, (const float *)dy, (float *)fx,
                            (float *)fy, (float *)fz, st);
    if (plan->geom.z != 0.0)
        return cross_solve_z<double>(plan, ws, (const double *)sigma, (const double *)dx, (const double *)dy,
                                     (double *)fx, (double *)fy, (double *)fz, st);
    return cross_solve_f64(plan, ws, (const double *)sigma, (const double *)dx, (const double *)dy, (double *)fx,
                           (double *)fy, st);
}

sg_status sg_cross_potential(sg_plan *plan, const sg_workspace *ws, const void *sigma, const void *dx, const void *dy,
                             void *phi, cudaStream_t st)
{
    if (plan->ntiles == 0 || plan->ntargets == 0) return SG_OK;
    if (plan->prec == SG_FP64)
        return cross_potential_f64(plan, ws, (const double *)sigma, (const double *)dx, (const double *)dy,
                                   (double *)phi, st);
    return sg_far_potential(plan, ws, (const float *)sigma, (const float *)dx, (const float *)dy, (float *)phi, st);
}
