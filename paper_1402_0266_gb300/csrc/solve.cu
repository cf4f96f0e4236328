// solve.cu -- the deterministic single-domain solves (Sec. 4).
//
// The paper solves an implicit finite-difference discretisation of Eq. (3)
// on each subdomain, with the interface values as Dirichlet data, and gives no
// stencil. Since -(1/w) grad w . grad xi + lap xi = w div((1/w) grad xi), the
// implicit Euler step multiplied by 1/w reads, at an unknown node,
//
//   xi_ij / (w_ij Dt) + sum_nb c_nb (xi_ij - xi_nb) = xi^{n-1}_ij / (w_ij Dt),
//   c_nb = 1 / (wbar h^2),  wbar = (w_ij + w_nb) / 2,
//
// a symmetric positive definite M-matrix, solved per subdomain by Chebyshev
// iterations and conjugate gradients, both with the diagonal as preconditioner.
//
// Precision: the solution and its residual are double precision; the
// sweeps run on the residual equation A d = r in single precision (iterative
// refinement): each sweep reduces ||r|| by inner_tol or more,
// then x += d and r = b - A x are formed again in double precision, until
// ||r|| <= rtol ||b||. On GB300 double-precision arithmetic runs at a small
// fraction of the single-precision rate; only the residuals use it.
//
// Execution: one thread-block cluster per system; each block owns a band of
// the subdomain's rows. Dot products are reduced inside each block, then
// across the cluster through distributed shared memory, in a fixed order, so
// every block takes the same branch. All loops are bounded by max_iter and
// max_outer; non-convergence sets a status bit.
#include <cooperative_groups.h>

#include <algorithm>
#include <cstdlib>

#include "cluster.cuh"
#include "common.cuh"

namespace cg = cooperative_groups;

namespace sdd {

namespace {


__global__ void k_solve_setup(const float* __restrict__ w, const double* __restrict__ pxi,
                              const double* __restrict__ peta, int nx, int ny, double rDt, double* __restrict__ cx,
                              double* __restrict__ cy, double* __restrict__ dg, double* __restrict__ rhs0,
                              float* __restrict__ cxf, float* __restrict__ cyf, float* __restrict__ dgf,
                              float* __restrict__ dinvf, int* status)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= nx || j >= ny) return;
    const long long n = (long long)j * nx + i;
    const double ihx2 = (double)(nx - 1) * (double)(nx - 1);
    const double ihy2 = (double)(ny - 1) * (double)(ny - 1);
    if (bad_w(w[n])) atomicOr(status, STATUS_BAD_W);
    const double wc = (double)w[n];
    // (five divisions a node by the SM's two double-precision lanes took 40 us at 513^2)
    const double e = (i + 1 < nx) ? ihx2 * reciprocal(0.5 * (wc + (double)w[n + 1])) : 0.0;
    const double no = (j + 1 < ny) ? ihy2 * reciprocal(0.5 * (wc + (double)w[n + nx])) : 0.0;
    cx[n] = e;
    cy[n] = no;
    cxf[n] = (float)e;
    cyf[n] = (float)no;
    double d = rDt * reciprocal(wc);
    rhs0[n] = pxi[n] * d;
    rhs0[(long long)nx * ny + n] = peta[n] * d;
    if (i > 0 && i + 1 < nx && j > 0 && j + 1 < ny) {
        const double wwest = (double)w[n - 1], wsouth = (double)w[n - nx];
        d += e + no + ihx2 * reciprocal(0.5 * (wc + wwest)) + ihy2 * reciprocal(0.5 * (wc + wsouth));
    }
    dg[n] = d;
    dgf[n] = (float)d;
    dinvf[n] = (float)reciprocal(d);
}

// Dirichlet data of the new fields: the face data on the outer boundary, the
// interface estimates on the interface lines, and the previous values
// (initial guess) elsewhere.
__global__ void k_dirichlet(const double* __restrict__ faces, const double* __restrict__ pxi,
                            const double* __restrict__ peta, int nx, int ny, double* __restrict__ xo,
                            double* __restrict__ eo)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= nx || j >= ny) return;
    const long long n = (long long)j * nx + i;
    const long long per_field = 2LL * ny + 2LL * nx;
    double a = pxi[n], b = peta[n];
    // faces: left (x = 0, by j), right, bottom (y = 0, by i), top; first match wins
    if (i == 0) { a = faces[j]; b = faces[per_field + j]; }
    else if (i == nx - 1) { a = faces[ny + j]; b = faces[per_field + ny + j]; }
    else if (j == 0) { a = faces[2LL * ny + i]; b = faces[per_field + 2LL * ny + i]; }
    else if (j == ny - 1) { a = faces[2LL * ny + nx + i]; b = faces[per_field + 2LL * ny + nx + i]; }
    xo[n] = a;
    eo[n] = b;
}

__global__ void k_scatter_iface(const double* __restrict__ vx, const double* __restrict__ ve,
                                const int32_t* __restrict__ idx, int n, double* __restrict__ xo,
                                double* __restrict__ eo, uint32_t* step)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (step && k == 0) *step += 1u;   // the mesh step counter, when this closes the step
    if (k >= n) return;
    xo[idx[k]] = vx[k];
    eo[idx[k]] = ve[k];
}

__global__ void __launch_bounds__(SOLVE_THREADS) k_pcg_cluster(const SolveArgs a)
{
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks();
    const int rank = (int)cl.block_rank();
    const SolveSys S = a.sys[blockIdx.x / C];
    const int nx = a.nx;
    const int mx = S.i1 - S.i0, my = S.j1 - S.j0;
    const int row0 = S.j0 + (my * rank) / C, row1 = S.j0 + (my * (rank + 1)) / C;
    const int m = (row1 - row0) * mx;  // unknowns of this block
    double* __restrict__ x = a.x[S.field];
    float* __restrict__ r = a.r[S.field];
    float* __restrict__ p = a.p[S.field];
    float* __restrict__ q = a.q[S.field];
    float* __restrict__ d = a.d[S.field];
    const double* __restrict__ rhs = a.rhs0 + (long long)S.field * nx * a.ny;

    __shared__ ClusterSlots<double> red64[2];
    __shared__ ClusterSlots<float> red32[2];
    int seq = 0;  // one counter for both slot types: consecutive calls never share a slot set

    auto node = [&](int u) -> long long { return (long long)(row0 + u / mx) * nx + (S.i0 + u % mx); };

    // ||b||^2 with b = rhs + the Dirichlet neighbours' terms
    double bb = 0.0, unused = 0.0;
    for (int u = threadIdx.x; u < m; u += SOLVE_THREADS) {
        const long long n = node(u);
        const int i = S.i0 + u % mx, j = row0 + u / mx;
        double b = rhs[n];
        if (i == S.i0) b += a.cx[n - 1] * x[n - 1];
        if (i == S.i1 - 1) b += a.cx[n] * x[n + 1];
        if (j == S.j0) b += a.cy[n - nx] * x[n - nx];
        if (j == S.j1 - 1) b += a.cy[n] * x[n + nx];
        bb += b * b;
    }
    cluster_sum2(cl, red64, seq, bb, unused);
    const double stop2 = a.rtol * a.rtol * bb;

    int total = 0;
    bool converged = false;
    for (int outer = 0; outer < a.max_outer; ++outer) {
        // double-precision residual r = b - A x (x complete on every block: cluster-synchronised)
        double rr64 = 0.0, unused64 = 0.0;
        for (int u = threadIdx.x; u < m; u += SOLVE_THREADS) {
            const long long n = node(u);
            const double ax = a.dg[n] * x[n] - a.cx[n - 1] * x[n - 1] - a.cx[n] * x[n + 1] -
                              a.cy[n - nx] * x[n - nx] - a.cy[n] * x[n + nx];
            const double res = rhs[n] - ax;
            rr64 += res * res;
            const float rf = (float)res;
            r[n] = rf;
            d[n] = 0.0f;
            p[n] = rf * a.dinvf[n];
        }
        cluster_sum2(cl, red64, seq, rr64, unused64);
        if (rr64 <= stop2) {
            converged = true;
            break;
        }
        if (total >= a.max_iter) break;
        // single-precision PCG on A d = r, from d = 0 with p = z = r / diag
        float rz = 0.0f, rr = 0.0f;
        for (int u = threadIdx.x; u < m; u += SOLVE_THREADS) {
            const long long n = node(u);
            rz += r[n] * p[n];
            rr += r[n] * r[n];
        }
        cluster_sum2(cl, red32, seq, rz, rr);  // its barrier also publishes p to the neighbouring blocks
        if (!(rr > 0.0f)) continue;
        const float stop_in = a.inner_tol * a.inner_tol * rr;
        while (total < a.max_iter) {
            ++total;
            float pq = 0.0f, unused32 = 0.0f;
            for (int u = threadIdx.x; u < m; u += SOLVE_THREADS) {
                const long long n = node(u);
                // p is zero on every node that is not an unknown
                const float v = a.dgf[n] * p[n] - a.cxf[n - 1] * p[n - 1] - a.cxf[n] * p[n + 1] -
                                a.cyf[n - nx] * p[n - nx] - a.cyf[n] * p[n + nx];
                q[n] = v;
                pq += p[n] * v;
            }
            cluster_sum2(cl, red32, seq, pq, unused32);
            const float alpha = rz / pq;
            float rz_new = 0.0f, rr_new = 0.0f;
            for (int u = threadIdx.x; u < m; u += SOLVE_THREADS) {
                const long long n = node(u);
                d[n] += alpha * p[n];
                const float rn = r[n] - alpha * q[n];
                r[n] = rn;
                rz_new += rn * rn * a.dinvf[n];
                rr_new += rn * rn;
            }
            cluster_sum2(cl, red32, seq, rz_new, rr_new);
            if (rr_new <= stop_in) break;
            const float beta = rz_new / rz;
            rz = rz_new;
            for (int u = threadIdx.x; u < m; u += SOLVE_THREADS) {
                const long long n = node(u);
                p[n] = r[n] * a.dinvf[n] + beta * p[n];
            }
            cl.sync();  // p complete before the next product
        }
        // x += d in double precision; the next residual reads the neighbours' x
        for (int u = threadIdx.x; u < m; u += SOLVE_THREADS) {
            const long long n = node(u);
            x[n] += (double)d[n];
        }
        cl.sync();
    }
    if (threadIdx.x == 0 && rank == 0) {
        a.iters[blockIdx.x / C] = converged ? total : a.max_iter + 1;
        if (!converged) atomicOr(a.status, STATUS_NOCONV);
    }
    cl.sync();  // no block leaves while others may still read its shared memory
}

// log2 of a positive normal double, off the double-precision lanes (the library's logarithm and a division
// were 2 us of latency a sweep).
__device__ __forceinline__ float log2_of(double v)
{
    const int hi = __double2hiint(v);
    return (float)((hi >> 20) - 1023) + log2f(__int_as_float(0x3F800000 | ((hi & 0xFFFFF) << 3)));
}

// Chebyshev iterations for subdomains whose bands fit the blocks of a cluster, both fields together, and
// conjugate gradients (cg_solve) in the same launch for what they leave. Solves with their set-up, each waited for, ring
// density, Dt = 1e-3, in the kernel that ran conjugate gradients alone before and now: 4 x 19^2 unknowns 186 -> 72 us,
// 4 x 63^2 439 -> 120, 4 x 119^2 835 -> 252, 16 x 65^2 1307 -> 294, 9 x 119^2 2085 -> 446. The method:
// A d = r with the diagonal as preconditioner over the interval [lo, 1 + rho] of the eigenvalues of
// D^-1 A, in single precision, inside the double-precision refinement of the other kernels.
// rho is Gershgorin's bound, the largest row sum of D^-1 (D - A) (below 1: the mass term), so the upper
// end holds; lo adds to 1 - rho most of what the Dirichlet frame contributes with uniform coefficients.
// Where that is too much, the modes below lo fall more slowly than the rest, never grow, and cg_solve,
// which closes every solve, takes them over.
//
// Why not conjugate gradients alone: an iteration of theirs is a product, two barriers and a reduction of
// six sums, a latency chain of about 2.3 us whatever the cluster size; here it is one barrier (one block:
// a block barrier) and a product whose operands are in registers and shared memory, with no scalar to wait
// for: 0.39 us with one unknown a thread, 0.87 with four. (Which unknowns neighbour another block is found once: by a
// division per unknown and iteration, where the compiler left it in the loop, 9 x 100^2 took 808 us instead of 545.) The
// iteration count is 0.9 to 1.3 times theirs where the mass term counts (4 x 119^2 unknowns: up to Dt = 1e-2) and
// twice theirs without it, faster still (Dt = 1: 0.96 against 2.07 ms).
//
// What they lose: blocks of very different density (a 50 : 1 checkerboard at Dt >= 3e-2) have modes far below lo, and
// sweep after sweep falls short. A sweep that brings the residual down by less than a third of its factor
// (in the logarithm) is the last: with six of them 16 x 65^2 unknowns took 3.10 ms at Dt = 0.3, 2.40 in the kernel that ran
// conjugate gradients alone before, now 1.91; over Dt = 1e-4 to 1e3, 9^2 to 119^2 unknowns and five densities no
// solve takes longer than in that kernel (0.93 times at most).
//
// Layout: each thread keeps UPT unknowns (scaled coefficients and, per field, scaled residual z, step d,
// correction e) in registers; the steps d live in shared memory as pairs (both fields), a zero frame around
// the band and halo rows that the neighbouring blocks store into before the barrier. Planes alternate with the
// iteration's parity: a plane is rewritten only after the next iteration's barrier, which every reader has passed.
//
// planes: [parity] (rows_max + 2) x (mx + 2). True if the systems are solved; total: the iterations, at most a
// quarter of max_iter.
template <int UPT, bool ONE>
__device__ __forceinline__ bool cheb_solve(const SolveArgs& a, int rows_max, float2* planes, int& total)
{
    __shared__ ClusterSlots<double> red64[2];
    __shared__ float warp_max[SOLVE_WARPS], block_max;
    cg::cluster_group cl = cg::this_cluster();
    const int C = ONE ? 1 : (int)cl.num_blocks();
    const int rank = ONE ? 0 : (int)cl.block_rank();
    const int T = (int)blockDim.x;
    const SolveSys S = a.sys[blockIdx.x / C];
    const int nx = a.nx;
    const int mx = S.i1 - S.i0, my = S.j1 - S.j0;
    const int row0 = S.j0 + (my * rank) / C, rows = S.j0 + (my * (rank + 1)) / C - row0;
    const int m = rows * mx, W = mx + 2, plane = (rows_max + 2) * W;
    const int rows_below = rank > 0 ? ((my * rank) / C) - ((my * (rank - 1)) / C) : 0;
    double* __restrict__ x0 = a.x[0];
    double* __restrict__ x1 = a.x[1];
    const double* __restrict__ rhs0 = a.rhs0;
    const double* __restrict__ rhs1 = a.rhs0 + (long long)nx * a.ny;
    int seq = 0;
    auto sync = [&]() {
        if (ONE) __syncthreads();
        else cl.sync();
    };

    for (int k = threadIdx.x; k < 2 * plane; k += T) planes[k] = make_float2(0.f, 0.f);
    float2* nb_lo = (C > 1 && rank > 0) ? cl.map_shared_rank(planes, rank - 1) : nullptr;     // block below
    float2* nb_hi = (C > 1 && rank < C - 1) ? cl.map_shared_rank(planes, rank + 1) : nullptr; // block above

    int n_[UPT], sidx[UPT];   // grid index (-1: no unknown), place in a plane
    float cw[UPT], ce[UPT], cs[UPT], cn[UPT];   // couplings to unknowns over the diagonal (0 to Dirichlet nodes)
    float z[2][UPT], d[2][UPT], e[2][UPT];
    unsigned edge = 0;   // bit 2 k: unknown k is in the band's lowest row, another block below; 2 k + 1: highest, above
    float rho = 0.f;
    double bb[2] = {0.0, 0.0};
#pragma unroll
    for (int k = 0; k < UPT; ++k) {
        const int u = threadIdx.x + k * T;
        n_[k] = -1;
        sidx[k] = 0;
        cw[k] = ce[k] = cs[k] = cn[k] = 0.f;
#pragma unroll
        for (int f = 0; f < 2; ++f) z[f][k] = d[f][k] = e[f][k] = 0.f;
        if (u >= m) continue;
        const int lr = u / mx, lc = u - lr * mx;
        const int i = S.i0 + lc, j = row0 + lr, n = j * nx + i;
        n_[k] = n;
        sidx[k] = (lr + 1) * W + lc + 1;
        if (lr == 0 && nb_lo) edge |= 1u << 2 * k;
        if (lr == rows - 1 && nb_hi) edge |= 2u << 2 * k;
        const float di = a.dinvf[n];
        double b0 = rhs0[n], b1 = rhs1[n];
        if (i > S.i0) cw[k] = a.cxf[n - 1] * di;
        else b0 += a.cx[n - 1] * x0[n - 1], b1 += a.cx[n - 1] * x1[n - 1];
        if (i < S.i1 - 1) ce[k] = a.cxf[n] * di;
        else b0 += a.cx[n] * x0[n + 1], b1 += a.cx[n] * x1[n + 1];
        if (j > S.j0) cs[k] = a.cyf[n - nx] * di;
        else b0 += a.cy[n - nx] * x0[n - nx], b1 += a.cy[n - nx] * x1[n - nx];
        if (j < S.j1 - 1) cn[k] = a.cyf[n] * di;
        else b0 += a.cy[n] * x0[n + nx], b1 += a.cy[n] * x1[n + nx];
        rho = fmaxf(rho, cw[k] + ce[k] + cs[k] + cn[k]);
        bb[0] += b0 * b0;
        bb[1] += b1 * b1;
    }
    // the largest row sum over the cluster
    rho = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(rho)));   // nonnegative: ordered as integers
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = rho;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < T / 32; ++q) rho = fmaxf(rho, warp_max[q]);
        block_max = rho;
    }
    cluster_sum2(cl, red64, seq, bb[0], bb[1]);   // its barrier publishes block_max
    for (int q = 0; q < C; ++q) rho = fmaxf(rho, ONE ? block_max : *cl.map_shared_rank(&block_max, q));
    rho = fminf(fmaxf(rho, 1e-3f), 0.9999999f);
    const double stop2[2] = {a.rtol * a.rtol * bb[0], a.rtol * a.rtol * bb[1]};

    // the interval, and the factor per iteration
    const float ix = (float)(nx - 1), iy = (float)(a.ny - 1), px = ix * ix, py = iy * iy;
    const float frame = (px * (1.f - cospif(1.f / (float)(mx + 1))) + py * (1.f - cospif(1.f / (float)(my + 1)))) / (px + py);
    const float hi = 1.f + rho, lo = fminf((1.f - rho) + 0.7f * rho * frame, 0.5f * hi);
    const float theta = 0.5f * (hi + lo), delta = 0.5f * (hi - lo), sigma = theta / delta;
    const float per_iter = logf(sigma + sqrtf((sigma - 1.f) * (sigma + 1.f)));

    int b = 0;
    total = 0;
    bool converged = false;
    float goal = 1e30f;   // what a sweep has to leave at most for another (the logarithm of the reduction to come)
    for (int sweep = 0; sweep < 6; ++sweep) {
        // the residual, double precision
        double rr[2] = {0.0, 0.0};
#pragma unroll
        for (int k = 0; k < UPT; ++k) {
            const int n = n_[k];
            if (n < 0) continue;
            const float di = a.dinvf[n];
            const double g = a.dg[n], w = a.cx[n - 1], o = a.cx[n], s = a.cy[n - nx], t = a.cy[n];
#pragma unroll
            for (int f = 0; f < 2; ++f) {
                const double* x = f ? x1 : x0;
                const double r = (f ? rhs1[n] : rhs0[n]) -
                                 (g * x[n] - w * x[n - 1] - o * x[n + 1] - s * x[n - nx] - t * x[n + nx]);
                rr[f] += r * r;
                z[f][k] = (float)r * di;
                e[f][k] = 0.f;
            }
        }
        cluster_sum2(cl, red64, seq, rr[0], rr[1]);
        // iterations for what is left of the reduction, at most 1e-5 per sweep
        float left = 0.f;
        bool active[2], number = true;
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            active[f] = !(rr[f] <= stop2[f]);   // so that what is not a number never counts as solved
            number = number && (!active[f] || rr[f] > stop2[f]);
            if (active[f]) left = fmaxf(left, stop2[f] > 0.0 ? 0.34657359f * (log2_of(rr[f]) - log2_of(stop2[f])) : 100.f);
            else
#pragma unroll
                for (int k = 0; k < UPT; ++k) z[f][k] = 0.f;
        }
        converged = !active[0] && !active[1];
        // Left to conjugate gradients: what is not a number (they report it), what the sweep before brought too
        // little of, and what does not fit a quarter of max_iter, which bounds both methods together. (With half of
        // it, checkerboards of 10^4 : 1 at Dt = 1e3 that conjugate gradients solve in 885 iterations were not solved
        // within 970: of those a sweep that fell short had used 182.)
        const float sweeps = ceilf(left * (1.f / 11.5f));
        const bool leave = converged || !number || left > goal ||
                           left + 2.f * sweeps > per_iter * (0.25f * (float)a.max_iter - (float)total - sweeps);
        if (leave) break;
        goal = left - 0.35f * fminf(left, 11.5f);
        const int its = (int)ceilf((fminf(left, 11.5f) + 2.f) / per_iter);
        total += its;
        float r_old = 1.f / sigma, ca = 0.f, cb = 1.f / theta;
        const float two_delta = 2.f / delta;
        for (int it = 0; it < its; ++it, b ^= 1) {
            float2* mine = planes + b * plane;
#pragma unroll
            for (int k = 0; k < UPT; ++k) {
                if (n_[k] < 0) continue;
#pragma unroll
                for (int f = 0; f < 2; ++f) {
                    d[f][k] = ca * d[f][k] + cb * z[f][k];
                    e[f][k] += d[f][k];
                }
                const float2 v = make_float2(d[0][k], d[1][k]);
                mine[sidx[k]] = v;
                if (!ONE) {
                    if (edge & 1u << 2 * k) nb_lo[b * plane + sidx[k] + rows_below * W] = v;
                    if (edge & 2u << 2 * k) nb_hi[b * plane + sidx[k] - rows * W] = v;
                }
            }
            const float r_new = __frcp_rn(2.f * sigma - r_old);
            ca = r_new * r_old;
            cb = r_new * two_delta;
            r_old = r_new;
            sync();
#pragma unroll
            for (int k = 0; k < UPT; ++k) {
                const float2* v = mine + sidx[k];
                if (n_[k] < 0) continue;
                const float2 vw = v[-1], ve = v[1], vs = v[-W], vn = v[W];
                z[0][k] += cw[k] * vw.x + ce[k] * ve.x + cs[k] * vs.x + cn[k] * vn.x - d[0][k];
                z[1][k] += cw[k] * vw.y + ce[k] * ve.y + cs[k] * vs.y + cn[k] * vn.y - d[1][k];
            }
        }
#pragma unroll
        for (int k = 0; k < UPT; ++k)
            if (n_[k] >= 0) {
                x0[n_[k]] += (double)e[0][k];
                x1[n_[k]] += (double)e[1][k];
            }
        sync();   // the next residual reads the neighbours' x
    }
    return converged;   // the sum before has a barrier: no block writes into another's planes any more
}

// Register-resident conjugate gradients for subdomains whose band fits in the block, for
// the systems that cheb_solve left short of rtol (strong contrasts: the modes below its interval) or alone (max_iter):
// one cluster solves both fields of a subdomain (same matrix, two right-hand
// sides), so the cluster barriers are shared by the two solves. Each thread
// keeps UPT unknowns (coefficients and, per field, the CG vectors) in
// registers; the preconditioned residuals u live in shared memory with a
// halo row above and below. The inner iteration is the Chronopoulos--Gear
// form of preconditioned CG (Chronopoulos & Gear, "s-step iterative methods
// for symmetric linear systems", 1989): one fused reduction per iteration
// ((r,u), (w,u), (r,r) of both fields) after the product w = A u. Blocks push
// the edge rows of u and their reduction partials straight into the
// neighbours' shared memory before a cluster barrier, so an iteration is two
// barriers and no read crosses blocks. Halo rows and partial slots are
// double-buffered by the iteration's parity; a buffer is rewritten only two
// barriers after it was read. A field that has converged stops changing
// while the other one finishes.
//
// m_s: u, [parity][field] planes of (rows_max + 2) x (mx + 2), zero frame. before: iterations already made (they count towards max_iter).
template <int UPT, bool ONE>
__device__ __forceinline__ void cg_solve(const SolveArgs& a, int rows_max, float* m_s, int before)
{
    __shared__ float slots[2][16][8];   // [parity][block]: (gamma, delta, rr) of field 0, then field 1
    __shared__ float warp_part[2][SOLVE_WARPS][8];
    cg::cluster_group cl = cg::this_cluster();
    const int C = ONE ? 1 : (int)cl.num_blocks();
    const int rank = ONE ? 0 : (int)cl.block_rank();
    const int T = (int)blockDim.x;      // a multiple of 32, at most SOLVE_THREADS
    auto sync = [&]() {
        if (ONE) __syncthreads();
        else cl.sync();
    };
    const SolveSys S = a.sys[blockIdx.x / C];
    const int nx = a.nx;
    const int mx = S.i1 - S.i0, my = S.j1 - S.j0;
    const int row0 = S.j0 + (my * rank) / C, row1 = S.j0 + (my * (rank + 1)) / C;
    const int rows = row1 - row0;
    const int m = rows * mx;
    const int W = mx + 2;
    const int plane = (rows_max + 2) * W;
    const int rows_below = rank > 0 ? ((my * rank) / C) - ((my * (rank - 1)) / C) : 0;
    double* __restrict__ x0 = a.x[0];
    double* __restrict__ x1 = a.x[1];
    const double* __restrict__ rhs0 = a.rhs0;
    const double* __restrict__ rhs1 = a.rhs0 + (long long)nx * a.ny;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

    __shared__ ClusterSlots<double> red64[2];
    int seq = 0;

    for (int k = threadIdx.x; k < 4 * plane; k += T) m_s[k] = 0.0f;
    float* nb_lo = (C > 1 && rank > 0) ? cl.map_shared_rank(m_s, rank - 1) : nullptr;     // block below
    float* nb_hi = (C > 1 && rank < C - 1) ? cl.map_shared_rank(m_s, rank + 1) : nullptr; // block above

    int n_[UPT];      // grid index of the unknown
    int sidx[UPT];    // its place in a plane of m_s
    int lc_[UPT];     // its column in the band
    int edge[UPT];    // 1: first row of the band, 2: last row
    bool own[UPT];
    float cw[UPT], ce[UPT], cs[UPT], cn[UPT], dgv[UPT], dinv[UPT];
    float r[2][UPT], u[2][UPT], w[2][UPT], s[2][UPT], p[2][UPT], d[2][UPT];
#pragma unroll
    for (int k = 0; k < UPT; ++k) {
        const int uu0 = threadIdx.x + k * T;
        own[k] = uu0 < m;
        const int uu = own[k] ? uu0 : 0;
        const int lr = uu / mx;
        lc_[k] = uu % mx;
        n_[k] = (row0 + lr) * nx + (S.i0 + lc_[k]);
        sidx[k] = (lr + 1) * W + (lc_[k] + 1);
        edge[k] = (lr == 0 ? 1 : 0) | (lr == rows - 1 ? 2 : 0);
        if (own[k]) {
            const int n = n_[k];
            cw[k] = a.cxf[n - 1];
            ce[k] = a.cxf[n];
            cs[k] = a.cyf[n - nx];
            cn[k] = a.cyf[n];
            dgv[k] = a.dgf[n];
            dinv[k] = a.dinvf[n];
        } else {
            cw[k] = ce[k] = cs[k] = cn[k] = dgv[k] = dinv[k] = 0.0f;
        }
#pragma unroll
        for (int f = 0; f < 2; ++f) r[f][k] = u[f][k] = w[f][k] = s[f][k] = p[f][k] = d[f][k] = 0.0f;
    }

    // write both fields' u into buffer b and push their edge rows to the neighbours' halos
    auto publish = [&](int b) {
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            float* mine = m_s + (2 * b + f) * plane;
            const int off = (2 * b + f) * plane;
#pragma unroll
            for (int k = 0; k < UPT; ++k) {
                if (!own[k]) continue;
                mine[sidx[k]] = u[f][k];
                if ((edge[k] & 1) && nb_lo) nb_lo[off + (rows_below + 1) * W + lc_[k] + 1] = u[f][k];
                if ((edge[k] & 2) && nb_hi) nb_hi[off + lc_[k] + 1] = u[f][k];
            }
        }
    };
    auto apply_A = [&](int b, int f, int k) -> float {
        const float* v = m_s + (2 * b + f) * plane;
        const int c0 = sidx[k];
        return dgv[k] * v[c0] - cw[k] * v[c0 - 1] - ce[k] * v[c0 + 1] - cs[k] * v[c0 - W] - cn[k] * v[c0 + W];
    };
    // Six sums over the cluster, in two halves around a barrier. A warp's six values go through a
    // butterfly that halves the values with each of its first three steps (7 exchanges, then 2 more):
    // lane q & 7 ends with value q's warp sum. (Six full butterflies are 30 exchanges: with them and
    // their like after the barrier, the SM's one exchange a cycle took most of an iteration, 2.3 us.)
    auto push6 = [&](int b, const float (&v)[6]) {
        const bool h4 = lane & 4, h2 = lane & 2, h1 = lane & 1;
        const float in[8] = {v[0], v[1], v[2], v[3], v[4], v[5], 0.f, 0.f};
        float q4[4], q2[2], t;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            q4[k] = (h4 ? in[k + 4] : in[k]) + __shfl_xor_sync(0xffffffffu, h4 ? in[k] : in[k + 4], 4);
#pragma unroll
        for (int k = 0; k < 2; ++k)
            q2[k] = (h2 ? q4[k + 2] : q4[k]) + __shfl_xor_sync(0xffffffffu, h2 ? q4[k] : q4[k + 2], 2);
        t = (h1 ? q2[1] : q2[0]) + __shfl_xor_sync(0xffffffffu, h1 ? q2[0] : q2[1], 1);
        t += __shfl_xor_sync(0xffffffffu, t, 8);
        t += __shfl_xor_sync(0xffffffffu, t, 16);
        if (lane < 8) warp_part[b][warp][lane] = t;
        if (ONE) return;
        __syncthreads();
        if (warp == 0) {
            // value lane & 7 of the block, stored into every block's slot
            t = 0.f;
            for (int q = lane >> 3; q < (T >> 5); q += 4) t += warp_part[b][q][lane & 7];
            t += __shfl_xor_sync(0xffffffffu, t, 8);
            t += __shfl_xor_sync(0xffffffffu, t, 16);
            for (int q = lane >> 3; q < C; q += 4) cl.map_shared_rank(&slots[b][rank][0], q)[lane & 7] = t;
        }
    };
    // after the barrier, in every warp: the partials of the blocks (of the warps, for one block), in a fixed order
    auto read6 = [&](int b, float (&v)[6]) {
        float t = 0.f;
        for (int q = lane >> 3; q < (ONE ? T >> 5 : C); q += 4) t += ONE ? warp_part[b][q][lane & 7] : slots[b][q][lane & 7];
        t += __shfl_xor_sync(0xffffffffu, t, 8);
        t += __shfl_xor_sync(0xffffffffu, t, 16);
#pragma unroll
        for (int q = 0; q < 6; ++q) v[q] = __shfl_sync(0xffffffffu, t, q);
    };

    // ||b||^2 of both fields
    double bb[2] = {0.0, 0.0};
#pragma unroll
    for (int k = 0; k < UPT; ++k) {
        if (!own[k]) continue;
        const int n = n_[k];
        const int i = S.i0 + lc_[k], j = n / nx;
        double b0 = rhs0[n], b1 = rhs1[n];
        if (i == S.i0) { b0 += a.cx[n - 1] * x0[n - 1]; b1 += a.cx[n - 1] * x1[n - 1]; }
        if (i == S.i1 - 1) { b0 += a.cx[n] * x0[n + 1]; b1 += a.cx[n] * x1[n + 1]; }
        if (j == S.j0) { b0 += a.cy[n - nx] * x0[n - nx]; b1 += a.cy[n - nx] * x1[n - nx]; }
        if (j == S.j1 - 1) { b0 += a.cy[n] * x0[n + nx]; b1 += a.cy[n] * x1[n + nx]; }
        bb[0] += b0 * b0;
        bb[1] += b1 * b1;
    }
    cluster_sum2(cl, red64, seq, bb[0], bb[1]);
    const double stop2[2] = {a.rtol * a.rtol * bb[0], a.rtol * a.rtol * bb[1]};

    int total = before, it = 0;
    bool converged = false;
    for (int outer = 0; outer < a.max_outer; ++outer) {
        double rr64[2] = {0.0, 0.0};
#pragma unroll
        for (int k = 0; k < UPT; ++k) {
            if (!own[k]) continue;
            const int n = n_[k];
#pragma unroll
            for (int f = 0; f < 2; ++f) {
                const double* xf = f ? x1 : x0;
                const double ax = a.dg[n] * xf[n] - a.cx[n - 1] * xf[n - 1] - a.cx[n] * xf[n + 1] -
                                  a.cy[n - nx] * xf[n - nx] - a.cy[n] * xf[n + nx];
                const double res = (f ? rhs1[n] : rhs0[n]) - ax;
                rr64[f] += res * res;
                r[f][k] = (float)res;
                d[f][k] = 0.0f;
                u[f][k] = r[f][k] * dinv[k];
                s[f][k] = p[f][k] = 0.0f;
            }
        }
        cluster_sum2(cl, red64, seq, rr64[0], rr64[1]);
        bool active[2] = {!(rr64[0] <= stop2[0]), !(rr64[1] <= stop2[1])};
        if (!active[0] && !active[1]) {
            converged = true;
            break;
        }
        if (total >= a.max_iter) break;
        // a converged field has d = 0 and a zero residual in this sweep
#pragma unroll
        for (int f = 0; f < 2; ++f)
            if (!active[f]) {
#pragma unroll
                for (int k = 0; k < UPT; ++k) r[f][k] = u[f][k] = 0.0f;
            }
        // Chronopoulos--Gear iterations on A d = r from d = 0, u = M^-1 r, both fields in step
        float alpha[2] = {0.f, 0.f}, beta[2] = {0.f, 0.f}, gam_old[2] = {1.f, 1.f}, rr0[2] = {0.f, 0.f};
        bool first = true;
        for (;;) {
            if (!first) {
#pragma unroll
                for (int f = 0; f < 2; ++f) {
                    if (!active[f]) continue;
#pragma unroll
                    for (int k = 0; k < UPT; ++k) {
                        p[f][k] = u[f][k] + beta[f] * p[f][k];
                        s[f][k] = w[f][k] + beta[f] * s[f][k];
                        d[f][k] += alpha[f] * p[f][k];
                        r[f][k] -= alpha[f] * s[f][k];
                        u[f][k] = r[f][k] * dinv[k];
                    }
                }
            }
            const int b = it & 1;
            ++it;
            publish(b);
            sync();
            float v[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int f = 0; f < 2; ++f) {
#pragma unroll
                for (int k = 0; k < UPT; ++k) {
                    w[f][k] = own[k] ? apply_A(b, f, k) : 0.f;
                    v[3 * f + 0] += r[f][k] * u[f][k];
                    v[3 * f + 1] += w[f][k] * u[f][k];
                    v[3 * f + 2] += r[f][k] * r[f][k];
                }
            }
            push6(b, v);
            sync();
            read6(b, v);
#pragma unroll
            for (int f = 0; f < 2; ++f) {
                if (!active[f]) continue;
                const float gam = v[3 * f + 0], del = v[3 * f + 1], rr = v[3 * f + 2];
                if (first) {
                    rr0[f] = rr;
                    if (!(rr0[f] > 0.f) || !(del > 0.f)) {
                        active[f] = false;
                        continue;
                    }
                    alpha[f] = gam / del;
                    beta[f] = 0.f;
                } else {
                    if (rr <= a.inner_tol * a.inner_tol * rr0[f]) {
                        active[f] = false;
                        continue;
                    }
                    beta[f] = gam / gam_old[f];
                    alpha[f] = gam / (del - beta[f] * gam / alpha[f]);
                }
                gam_old[f] = gam;
            }
            first = false;
            if (!active[0] && !active[1]) break;
            if (total >= a.max_iter) break;
            ++total;
        }
        // x += d in double precision; the next residual reads the neighbours' x
#pragma unroll
        for (int k = 0; k < UPT; ++k)
            if (own[k]) {
                x0[n_[k]] += (double)d[0][k];
                x1[n_[k]] += (double)d[1][k];
            }
        sync();
    }
    if (threadIdx.x == 0 && rank == 0) {
        a.iters[blockIdx.x / C] = converged ? total : a.max_iter + 1;
        if (!converged) atomicOr(a.status, STATUS_NOCONV);
    }
    if (!ONE) cl.sync();  // no block leaves while others may still write into its shared memory
}

template <int UPT, bool ONE>
__global__ void __launch_bounds__(SOLVE_THREADS) k_solve(const SolveArgs a, int rows_max)
{
    extern __shared__ __align__(16) unsigned char solve_smem[];
    int total;
    const bool solved = cheb_solve<UPT, ONE>(a, rows_max, reinterpret_cast<float2*>(solve_smem), total);
    if (!solved) {
        cg_solve<UPT, ONE>(a, rows_max, reinterpret_cast<float*>(solve_smem), total);
        return;
    }
    cg::cluster_group cl = cg::this_cluster();
    const int C = ONE ? 1 : (int)cl.num_blocks();
    if (threadIdx.x == 0 && (ONE || cl.block_rank() == 0)) a.iters[blockIdx.x / C] = total;
    if (!ONE) cl.sync();   // no block leaves while others may still read its shared memory
}

__global__ void k_bump_step(uint32_t* step)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) *step += 1u;
}

}  // namespace

cudaError_t launch_solve_setup(const float* w, const double* prev_xi, const double* prev_eta, int nx, int ny,
                               double Dt, double* cx, double* cy, double* dg, double* rhs0, float* cxf, float* cyf,
                               float* dgf, float* dinvf, int* status, cudaStream_t s)
{
    const dim3 block(32, 8);
    const dim3 grid((nx + 31) / 32, (ny + 7) / 8);
    k_solve_setup<<<grid, block, 0, s>>>(w, prev_xi, prev_eta, nx, ny, 1.0 / Dt, cx, cy, dg, rhs0, cxf, cyf, dgf, dinvf,
                                       status);
    return cudaGetLastError();
}

cudaError_t launch_dirichlet(const double* faces64, const double* prev_xi, const double* prev_eta,
                             const double* iface_xi, const double* iface_eta, const int32_t* iface_idx,
                             int n_iface, int nx, int ny, double* xi_out, double* eta_out, cudaStream_t s)
{
    const dim3 block(32, 8);
    const dim3 grid((nx + 31) / 32, (ny + 7) / 8);
    k_dirichlet<<<grid, block, 0, s>>>(faces64, prev_xi, prev_eta, nx, ny, xi_out, eta_out);
    if (n_iface > 0)
        k_scatter_iface<<<(n_iface + 255) / 256, 256, 0, s>>>(iface_xi, iface_eta, iface_idx, n_iface, xi_out,
                                                             eta_out, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_dirichlet_faces(const double* faces64, const double* prev_xi, const double* prev_eta, int nx,
                                   int ny, double* xi_out, double* eta_out, cudaStream_t s)
{
    const dim3 block(32, 8);
    const dim3 grid((nx + 31) / 32, (ny + 7) / 8);
    k_dirichlet<<<grid, block, 0, s>>>(faces64, prev_xi, prev_eta, nx, ny, xi_out, eta_out);
    return cudaGetLastError();
}

cudaError_t launch_scatter_iface(const double* iface_xi, const double* iface_eta, const int32_t* iface_idx,
                                 int n_iface, double* xi_out, double* eta_out, uint32_t* step, cudaStream_t s)
{
    const int n = n_iface > 0 ? n_iface : 1;
    k_scatter_iface<<<(n + 255) / 256, 256, 0, s>>>(iface_xi, iface_eta, iface_idx, n_iface, xi_out, eta_out, step);
    return cudaGetLastError();
}

// Clusters of 2^k blocks that run at once on the current device, a block per SM (nine clusters of 16 do not, although 144 SMs
// would hold them: clusters stay inside the GPU's groups of SMs).
static int clusters_at_once(int k)
{
    const auto fn = k_solve<4, false>;
    cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1u << k);
    cfg.blockDim = dim3(SOLVE_THREADS);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1u << k;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) n = 0;
    cudaGetLastError();
    return n;
}

// Blocks per system (a power of two up to 16, no more than the smallest system's rows) for systems of at
// most max_mx columns and max_my rows: the least time by what the Chebyshev iterations measured, rounds of clusters that run
// at once x (0.4 us + 0.25 us per unknown of a thread) an iteration (0.3 + 0.16 since, the same proportion). One block (no cluster barrier) pays for
// up to 256 unknowns; above, its SM's few double-precision units make the residuals longer than the barrier.
// Bands that need more than 4 unknowns per thread leave the register-resident kernels and are the last choice.
// Asked for once per context, of the context's device.
int solve_cluster_size(int nsys, int min_rows, int max_mx, int max_my)
{
    if (max_mx * max_my <= 256) return 1;
    int best = 1;
    double least = 1e30;
    for (int k = 0; k < 5 && (1 << k) <= min_rows; ++k) {
        const int n = clusters_at_once(k), band = (max_my + (1 << k) - 1) / (1 << k) * max_mx;
        if (n < 1) continue;
        const double upt = std::max(0.25, (double)band / SOLVE_THREADS);
        const double t = (double)((nsys + n - 1) / n) * (0.4 + 0.25 * upt) * (solve_reg_upt(band) ? 1.0 : 100.0);
        if (t < least) {
            least = t;
            best = 1 << k;
        }
    }
    return best;
}

static cudaLaunchConfig_t cluster_config(const SolveArgs& a, size_t smem, cudaStream_t s, cudaLaunchAttribute* at)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.nsys * a.cluster));
    cfg.blockDim = dim3(SOLVE_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)a.cluster;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

template <int UPT>
static cudaError_t launch_reg(const SolveArgs& a, int rows_max, int max_mx, cudaStream_t s)
{
    const size_t smem = 4 * (size_t)(rows_max + 2) * (size_t)(max_mx + 2) * sizeof(float);
    const auto fn = a.cluster == 1 ? k_solve<UPT, true> : k_solve<UPT, false>;
    if (a.cluster > 8) cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (smem > 48 * 1024) {
        // the largest that any context asks for: another thread's launch keeps its limit
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSolveMaxSmem);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg = cluster_config(a, smem, s, at);
    // no more warps than the largest band needs (their sums cost exchanges)
    const int band = rows_max * max_mx;
    cfg.blockDim = dim3((unsigned)std::min(SOLVE_THREADS, ((band + UPT - 1) / UPT + 31) / 32 * 32));
    return cudaLaunchKernelEx(&cfg, fn, a, rows_max);
}

// Unknowns per thread of the register-resident kernel for these systems
// (0: too large, use the general kernel).
int solve_reg_upt(int max_band_unknowns)
{
    const int need = (max_band_unknowns + SOLVE_THREADS - 1) / SOLVE_THREADS;
    if (need <= 1) return 1;
    if (need <= 2) return 2;
    if (need <= 4) return 4;
    return 0;
}

cudaError_t launch_pcg(const SolveArgs& a, int upt, int rows_max, int max_mx, cudaStream_t s)
{
    if (a.nsys <= 0) return cudaSuccess;
    switch (upt) {
    case 1: return launch_reg<1>(a, rows_max, max_mx, s);
    case 2: return launch_reg<2>(a, rows_max, max_mx, s);
    case 4: return launch_reg<4>(a, rows_max, max_mx, s);
    default: {
        if (a.cluster > 8) cudaFuncSetAttribute(k_pcg_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        cudaLaunchAttribute at[1];
        cudaLaunchConfig_t cfg = cluster_config(a, 0, s, at);
        return cudaLaunchKernelEx(&cfg, k_pcg_cluster, a);
    }
    }
}

cudaError_t launch_bump_step(uint32_t* step, cudaStream_t s)
{
    k_bump_step<<<1, 32, 0, s>>>(step);
    return cudaGetLastError();
}

}  // namespace sdd
