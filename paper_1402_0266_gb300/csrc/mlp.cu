// mlp.cu -- the learned control variate's network on the device.
//
// The estimator of Eq. (7b) is a plain Monte Carlo mean (Sec. 4). A control
// variate subtracts from every path the sum of G(s_j, X_j) . sqrt(2) dW_j over
// the sub-steps it takes; any G keeps the mean, a G close to the solution's
// gradient removes most of the variance. Here G is the spatial gradient of a
// network g(x, y, t, w, |grad w| / w): two tanh layers of 64 units, one
// network per field, fitted by least squares to the method's own single-path
// scores. This file holds its kernels:
//
//   k_node_r / k_node_features  the node fields the network reads: w, r =
//                               |grad w| / w and their gradients, by the
//                               finite differences of the drift (FP64);
//   k_cv_scatter                training rows from single-path estimates;
//   k_moments / k_norm          feature standardisation (two-pass, FP64);
//   k_mlp_grad                  forward and backward pass over tiles of 64
//                               rows in shared memory, FP32 SIMT; per-block
//                               partial gradients, reduced in a fixed order;
//   k_mlp_reduce / k_mlp_adam   the batch gradient; Adam (Kingma & Ba 2015);
//   k_cv_tabulate               the table G at every node and time slice by
//                               forward-mode differentiation; the 64 x 64 layer
//                               on the tensor cores (tcgen05.mma, BF16 in, FP32
//                               accumulate in tensor memory), everything else FP32.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace sdd {
namespace {

constexpr int H = kMlpHidden;
constexpr int D = kMlpInputs;
constexpr int OW1 = 0, OB1 = H * D, OW2 = OB1 + H, OB2 = OW2 + H * H, OW3 = OB2 + H, OB3 = OW3 + H;
static_assert(OB3 + 1 == kMlpParams, "parameter layout");

constexpr int TILE = 64;     // rows of a tile of the training kernel
constexpr int LD = 68;       // row stride of the activation tiles (16-byte rows, conflict-free float4 reads)
constexpr int ZS = 8;        // row stride of the inputs (five, the fifth in the second float4)
constexpr int GRAD_THREADS = 256;

// ---------------------------------------------------------------- node fields

__device__ __forceinline__ double fd_x(const double* f, int nx, int i, int j, double rx)
{
    const double* row = f + (long long)j * nx;
    if (i == 0) return (-3.0 * row[0] + 4.0 * row[1] - row[2]) * rx;
    if (i == nx - 1) return (3.0 * row[nx - 1] - 4.0 * row[nx - 2] + row[nx - 3]) * rx;
    return (row[i + 1] - row[i - 1]) * rx;
}

__device__ __forceinline__ double fd_y(const double* f, int nx, int ny, int i, int j, double ry)
{
    const double* col = f + i;
    if (j == 0) return (-3.0 * col[0] + 4.0 * col[(long long)nx] - col[2LL * nx]) * ry;
    if (j == ny - 1)
        return (3.0 * col[(long long)(ny - 1) * nx] - 4.0 * col[(long long)(ny - 2) * nx] +
                col[(long long)(ny - 3) * nx]) * ry;
    return (col[(long long)(j + 1) * nx] - col[(long long)(j - 1) * nx]) * ry;
}

__global__ void k_node_w64(const float* __restrict__ w, long long n, double* __restrict__ w64)
{
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x)
        w64[k] = (double)w[k];
}

// grad w and r = |grad w| / w at every node (FP64).
__global__ void k_node_r(const double* __restrict__ w64, int nx, int ny, double* __restrict__ r64,
                         double2* __restrict__ gw)
{
    const long long n = (long long)nx * ny;
    const double rx = 0.5 * (nx - 1), ry = 0.5 * (ny - 1);
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(k % nx), j = (int)(k / nx);
        const double wx = fd_x(w64, nx, i, j, rx), wy = fd_y(w64, nx, ny, i, j, ry);
        gw[k] = make_double2(wx, wy);
        r64[k] = sqrt(wx * wx + wy * wy) / w64[k];
    }
}

// nfa = (w, r, dw/dx, dw/dy), nfb = (dr/dx, dr/dy) in FP32.
__global__ void k_node_features(const double* __restrict__ w64, const double* __restrict__ r64,
                                const double2* __restrict__ gw, int nx, int ny, float4* __restrict__ nfa,
                                float2* __restrict__ nfb)
{
    const long long n = (long long)nx * ny;
    const double rx = 0.5 * (nx - 1), ry = 0.5 * (ny - 1);
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(k % nx), j = (int)(k / nx);
        nfa[k] = make_float4((float)w64[k], (float)r64[k], (float)gw[k].x, (float)gw[k].y);
        nfb[k] = make_float2((float)fd_x(r64, nx, i, j, rx), (float)fd_y(r64, nx, ny, i, j, ry));
    }
}

struct alignas(16) Double4 {
    double x, y, z, w;
};

// The control variate's model from the fields at t_{n-1} themselves: one
// slice, (d xi/dx, d xi/dy, d eta/dx, d eta/dy) at every node by the same
// finite differences. Over a short mesh step the solution's gradient stays
// close to the previous field's.
__global__ void __launch_bounds__(256) k_field_grad(const double* __restrict__ xi, const double* __restrict__ eta, int nx,
                                                    int ny, double* __restrict__ table)
{
    const double rx = 0.5 * (nx - 1), ry = 0.5 * (ny - 1);
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= nx) return;
    for (int j = blockIdx.y; j < ny; j += gridDim.y) {
        Double4 o;
        o.x = fd_x(xi, nx, i, j, rx);
        o.y = fd_y(xi, nx, ny, i, j, ry);
        o.z = fd_x(eta, nx, i, j, rx);
        o.w = fd_y(eta, nx, ny, i, j, ry);
        reinterpret_cast<Double4*>(table)[(long long)j * nx + i] = o;
    }
}

// Weights C(order, m) 2^-order of the binomial filter, in single precision
// (exact up to order 24; rounded beyond), and the order.
struct BinomWeights {
    float w[kCvMaxOrder + 1];
    int order;
};

// Pass along x: tmp[j (nx - 1) + i] = sum_m w_m table[j][clamp(i - r + m)], all four components,
// for the cells i < nx - 1 along x and the node rows j < ny. A block stages its 256 cells' nodes of a row in single
// precision: converted once per node, not once per tap (the SM converts two doubles a cycle: at order 33
// on 1025^2 the pass took 232 us, now 23.5).
constexpr int SMOOTH_CELLS = 256;

__global__ void __launch_bounds__(SMOOTH_CELLS) k_cv_smooth_x(const double* __restrict__ table, int nx, int ny,
                                                              const BinomWeights W, float4* __restrict__ tmp)
{
    __shared__ float4 node[SMOOTH_CELLS + kCvMaxOrder];
    const int r = (W.order - 1) / 2, i0 = blockIdx.x * SMOOTH_CELLS, i = i0 + threadIdx.x;
    for (int j = blockIdx.y; j < ny; j += gridDim.y) {
        const double2* row = reinterpret_cast<const double2*>(table + 4LL * j * nx);
        for (int k = threadIdx.x; k < SMOOTH_CELLS + W.order; k += SMOOTH_CELLS) {
            const int q = min(max(i0 - r + k, 0), nx - 1);
            const double2 u = row[2LL * q], v = row[2LL * q + 1];
            node[k] = make_float4((float)u.x, (float)u.y, (float)v.x, (float)v.y);
        }
        __syncthreads();
        if (i < nx - 1) {
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int m = 0; m <= W.order; ++m) {
                const float4 v = node[threadIdx.x + m];
                const float wm = W.w[m];
                acc.x = fmaf(wm, v.x, acc.x);
                acc.y = fmaf(wm, v.y, acc.y);
                acc.z = fmaf(wm, v.z, acc.z);
                acc.w = fmaf(wm, v.w, acc.w);
            }
            tmp[(long long)j * (nx - 1) + i] = acc;
        }
        __syncthreads();
    }
}

// Pass along y: cells[j (nx - 1) + i] = sum_m w_m tmp[clamp(j - r + m)][i], j < ny - 1.
__global__ void __launch_bounds__(256) k_cv_smooth_y(const float4* __restrict__ tmp, int nx, int ny, const BinomWeights W,
                                                     float4* __restrict__ cells)
{
    const int r = (W.order - 1) / 2, i = blockIdx.x * 256 + threadIdx.x;
    if (i >= nx - 1) return;
    for (int j = blockIdx.y; j < ny - 1; j += gridDim.y) {
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int m = 0; m <= W.order; ++m) {
            const int q = min(max(j - r + m, 0), ny - 1);
            const float4 v = tmp[(long long)q * (nx - 1) + i];
            const float wm = W.w[m];
            acc.x = fmaf(wm, v.x, acc.x);
            acc.y = fmaf(wm, v.y, acc.y);
            acc.z = fmaf(wm, v.z, acc.z);
            acc.w = fmaf(wm, v.w, acc.w);
        }
        cells[(long long)j * (nx - 1) + i] = acc;
    }
}

// ---------------------------------------------------------------- training rows

__device__ __forceinline__ float bilin(const float4* __restrict__ nfa, int nx, int ny, double x, double y, int comp)
{
    double u = x * (nx - 1), v = y * (ny - 1);
    u = fmin(fmax(u, 0.0), nx - 1.0);
    v = fmin(fmax(v, 0.0), ny - 1.0);
    const int i = min((int)floor(u), nx - 2), j = min((int)floor(v), ny - 2);
    const double s = u - i, t = v - j;
    const long long k = (long long)j * nx + i;
    auto get = [&](long long q) { const float4 a = nfa[q]; return (double)(comp == 0 ? a.x : a.y); };
    return (float)((1 - s) * (1 - t) * get(k) + s * (1 - t) * get(k + 1) + (1 - s) * t * get(k + nx) +
                   s * t * get(k + nx + 1));
}

// Horizon k (1-based) of K, M samples: sample m goes to row m K + k - 1.
__global__ void k_cv_scatter(const double* __restrict__ xs, const double* __restrict__ ys,
                             const double* __restrict__ yxi, const double* __restrict__ yeta,
                             const float4* __restrict__ nfa, int nx, int ny, int k, int K, int M,
                             float* __restrict__ feats, float* __restrict__ targets)
{
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < M; m += gridDim.x * blockDim.x) {
        const long long row = (long long)m * K + (k - 1);
        float* f = feats + row * D;
        f[0] = (float)xs[m];
        f[1] = (float)ys[m];
        f[2] = (float)((double)k / (double)K);
        f[3] = bilin(nfa, nx, ny, xs[m], ys[m], 0);
        f[4] = bilin(nfa, nx, ny, xs[m], ys[m], 1);
        targets[2 * row + 0] = (float)yxi[m];
        targets[2 * row + 1] = (float)yeta[m];
    }
}

// ---------------------------------------------------------------- standardisation

constexpr int MOM_BLOCKS = 256;

// pass 0: per-block sums of f; pass 1: per-block sums of (f - mu)^2.
__global__ void k_moments(const float* __restrict__ feats, long long n, const double* __restrict__ mu, int pass,
                          double* __restrict__ part)
{
    __shared__ double red[D][256 / 32];
    double acc[D];
#pragma unroll
    for (int c = 0; c < D; ++c) acc[c] = 0.0;
    for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < n; r += (long long)gridDim.x * blockDim.x) {
#pragma unroll
        for (int c = 0; c < D; ++c) {
            const double v = (double)feats[r * D + c];
            const double d = pass ? v - mu[c] : v;
            acc[c] += pass ? d * d : d;
        }
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < D; ++c) {
        double v = acc[c];
        for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) red[c][wid] = v;
    }
    __syncthreads();
    if (threadIdx.x < D) {
        double v = 0.0;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) v += red[threadIdx.x][q];
        part[blockIdx.x * D + threadIdx.x] = v;
    }
}

// mu (pass 0) or s (pass 1) from the block sums, in block order.
__global__ void k_norm(const double* __restrict__ part, int nblk, long long n, double* __restrict__ mu, int pass,
                       float* __restrict__ norm)
{
    const int c = threadIdx.x;
    if (c >= D) return;
    double v = 0.0;
    for (int b = 0; b < nblk; ++b) v += part[b * D + c];
    v /= (double)n;
    if (pass == 0) {
        mu[c] = v;
        norm[c] = (float)v;
    } else {
        const double sd = sqrt(v);
        const double m = fabs(mu[c]);
        norm[D + c] = sd > 1e-6 * fmax(1.0, m) ? (float)(1.0 / sd) : 0.0f;
    }
}

// ---------------------------------------------------------------- training

struct GradSmem {
    float th[kMlpStride];      // the network's parameters; W2 in pairs of units: [j / 2][k] (W2[j][k], W2[j + 1][k])
    float2 w2t[H / 2 * H];     // W2 in pairs of inputs: [k / 2][j] (W2[j][k], W2[j][k + 1])
    float h1[TILE * LD];       // tanh(a1), later dL/da1
    float h2[TILE * LD];       // tanh(a2), later dL/da2
    float z[TILE * ZS];
    float y[TILE];
    float d[TILE];
    float quarter[4][H];       // sums over a quarter of the tile's rows
    float quarter2[4][H];
    float red[GRAD_THREADS / 32];
};

// A sum over tiles: value and rounding error (Knuth's two-sum), so that a block's tiles lose nothing that
// one tile's sum does not.
struct TileSum {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float v)
    {
        const float t = s + v;
        const float b = t - s;
        c += (s - (t - b)) + (v - b);
        s = t;
    }
    // the error of a sum that is infinite is not a number
    __device__ __forceinline__ float value() const { return isfinite(c) ? s + c : s; }
};

// acc[r][c] += sum_q a[row(r)][q] b[q][col(c)] over q < 64, even and odd q apart, columns 2 tx, 2 tx + 1 and 32 more
// (a warp's reads of b then touch every bank once): a row-major with stride LD,
// read four q at a time (a warp reads two rows of a and 64 columns of b), b in pairs of q, [q / 2][column].
template <int RPT>
__device__ __forceinline__ void tile_product(float2 (&acc)[RPT][4], const float* a, const float2* b, int tx, int ty)
{
#pragma unroll 4
    for (int q = 0; q < H; q += 4) {
        float4 bv[2][2];
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int c = 0; c < 2; ++c) bv[e][c] = *reinterpret_cast<const float4*>(&b[(q / 2 + e) * H + 2 * tx + 32 * c]);
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            const float4 av = *reinterpret_cast<const float4*>(&a[(ty + 16 * r) * LD + q]);
            const float2 ae[2] = {make_float2(av.x, av.y), make_float2(av.z, av.w)};
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                acc[r][0] = __ffma2_rn(ae[e], make_float2(bv[e][0].x, bv[e][0].y), acc[r][0]);
                acc[r][1] = __ffma2_rn(ae[e], make_float2(bv[e][0].z, bv[e][0].w), acc[r][1]);
                acc[r][2] = __ffma2_rn(ae[e], make_float2(bv[e][1].x, bv[e][1].y), acc[r][2]);
                acc[r][3] = __ffma2_rn(ae[e], make_float2(bv[e][1].z, bv[e][1].w), acc[r][3]);
            }
        }
    }
}

// Forward and backward over the block's tiles of one network (blockIdx.y): its share of the
// gradient of the batch loss (1 / batch) sum (g - y)^2, written to part[(f nblk + block) stride + p];
// part[.. + kMlpParams] = its sum of squared errors.
//
// Three 64 x 64 products and 128 tanhf per row: 4-by-4 register tiles, operands read four deep, W2's gradient kept in
// registers over the tiles. A tile's partial gradient is 18 KB, so blocks take several tiles and write one, and
// a tile's inputs are read while the one before is at work. Bound by the shared-memory loads (a 16-byte
// load of a warp takes four cycles, 81 % busy): the multiply-adds are in pairs, which halves their issue
// slots. 65,536 rows: 111 us (127 with single multiply-adds; 147 for a block and a partial per tile, whose sum took
// 163 us more, now 9). Blocks of 128 threads with 8-by-4 tiles load a third less, but hold 12 warps an SM: 121 us.
__global__ void __launch_bounds__(GRAD_THREADS, 2) k_mlp_grad(const float* __restrict__ theta,
                                                              const float* __restrict__ norm,
                                                              const float* __restrict__ feats,
                                                              const float* __restrict__ targets, long long row0,
                                                              long long rows, float inv_batch,
                                                              float* __restrict__ part)
{
    constexpr int ROWS = TILE, RPT = ROWS / 16, QROWS = ROWS / 4;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    GradSmem& S = *reinterpret_cast<GradSmem*>(smem_raw);
    const int f = blockIdx.y, t = threadIdx.x;
    const int lane = t & 31, wid = t >> 5, tx = t & 15, ty = t >> 4;
    const int j = t & 63, quarter = t >> 6;
    const float* th = theta + (long long)f * kMlpStride;
    for (int p = t; p < kMlpParams; p += GRAD_THREADS)
        if (p < OW2 || p >= OW2 + H * H) S.th[p] = th[p];
    float2* const w2 = reinterpret_cast<float2*>(&S.th[OW2]);
    for (int p = t; p < H * H / 2; p += GRAD_THREADS) {
        const int q = p / H, c = p % H;
        S.w2t[p] = make_float2(th[OW2 + c * H + 2 * q], th[OW2 + c * H + 2 * q + 1]);
        w2[p] = make_float2(th[OW2 + 2 * q * H + c], th[OW2 + (2 * q + 1) * H + c]);
    }

    TileSum gw2[4][4], small[2], loss;   // small: thread t's outputs of W1, b1 (t, t + 256)
    TileSum gw3, gb2, gb3;
    const int ntiles = (int)((rows + ROWS - 1) / ROWS);
    // a tile's inputs, read while the tile before is at work
    constexpr int NIN = (ROWS * D + GRAD_THREADS - 1) / GRAD_THREADS;
    float in[NIN], target = 0.f;
    auto load_inputs = [&](int tile) {
        const long long r0 = row0 + (long long)tile * ROWS;
        const int have = tile < ntiles ? (int)min((long long)ROWS, row0 + rows - r0) : 0;
#pragma unroll
        for (int q = 0; q < NIN; ++q) {
            const int p = t + q * GRAD_THREADS;
            in[q] = p < have * D ? feats[r0 * D + p] : 0.f;
        }
        target = t < have ? targets[2 * (r0 + t) + f] : 0.f;
    };
    load_inputs(blockIdx.x);
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int have = (int)min((long long)ROWS, rows - (long long)tile * ROWS);
        __syncthreads();   // the tile before is done (and the parameters are in place)
#pragma unroll
        for (int q = 0; q < NIN; ++q) {
            const int p = t + q * GRAD_THREADS, c = p % D;
            if (p < ROWS * D) S.z[p / D * ZS + c] = p < have * D ? (in[q] - norm[c]) * norm[D + c] : 0.f;
        }
        if (t < ROWS) S.y[t] = target;
        __syncthreads();
        load_inputs(tile + (int)gridDim.x);

        // layer 1: thread owns unit j and rows quarter + 4 m
        {
            float wj[D];
#pragma unroll
            for (int c = 0; c < D; ++c) wj[c] = S.th[OW1 + j * D + c];
            const float bj = S.th[OB1 + j];
#pragma unroll 4
            for (int i = quarter; i < ROWS; i += 4) {
                const float4 z = *reinterpret_cast<const float4*>(&S.z[i * ZS]);
                float a = fmaf(wj[0], z.x, bj);
                a = fmaf(wj[1], z.y, a);
                a = fmaf(wj[2], z.z, a);
                a = fmaf(wj[3], z.w, a);
                a = fmaf(wj[4], S.z[i * ZS + 4], a);
                S.h1[i * LD + j] = tanhf(a);
            }
        }
        __syncthreads();

        // layer 2: a2[i][j] = b2[j] + sum_k h1[i][k] W2[j][k], rows ty + 16 r, units 4 tx..
        {
            float2 acc[RPT][4];
#pragma unroll
            for (int r = 0; r < RPT; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[r][c] = make_float2(S.th[OB2 + 2 * tx + (c & 1) + 16 * (c & 2)], 0.f);
            tile_product<RPT>(acc, S.h1, S.w2t, tx, ty);
#pragma unroll
            for (int r = 0; r < RPT; ++r)
#pragma unroll
                for (int c = 0; c < 4; c += 2)
                    *reinterpret_cast<float2*>(&S.h2[(ty + 16 * r) * LD + 2 * tx + 16 * c]) =
                        make_float2(tanhf(acc[r][c].x + acc[r][c].y), tanhf(acc[r][c + 1].x + acc[r][c + 1].y));
        }
        __syncthreads();

        // output and dL/dg: 256 / ROWS neighbouring threads per row, each with its share of the units
        {
            constexpr int SPLIT = GRAD_THREADS / ROWS, UNITS = H / SPLIT;
            const int i = t / SPLIT, part0 = (t % SPLIT) * UNITS;
            float v = 0.f;
#pragma unroll
            for (int u = 0; u < UNITS; u += 4) {
                const float4 h = *reinterpret_cast<const float4*>(&S.h2[i * LD + part0 + u]);
                const float4 w = *reinterpret_cast<const float4*>(&S.th[OW3 + part0 + u]);
                v += (w.x * h.x + w.y * h.y) + (w.z * h.z + w.w * h.w);
            }
#pragma unroll
            for (int o = SPLIT / 2; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            const float e = i < have ? v + S.th[OB3] - S.y[i] : 0.f;
            float sq = t % SPLIT == 0 ? e * e : 0.f;
            if (t % SPLIT == 0) S.d[i] = 2.f * e * inv_batch;
            for (int o = 16; o; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
            if (lane == 0) S.red[wid] = sq;
        }
        __syncthreads();
        // dL/dw3[j] = sum_i d_i h2[i][j] by quarters of the rows, dL/db3 = sum_i d_i, the loss;
        // then dL/da2 = d_i w3_j (1 - h2^2) in place, rows by the same threads, dL/db2 its sum
        {
            const float w3 = S.th[OW3 + j];
            float a = 0.f, b = 0.f;
#pragma unroll 8
            for (int i = quarter * QROWS; i < (quarter + 1) * QROWS; ++i) {
                const float h = S.h2[i * LD + j], d = S.d[i];
                a = fmaf(d, h, a);
                const float g = d * w3 * (1.f - h * h);
                b += g;
                S.h2[i * LD + j] = g;
            }
            S.quarter[quarter][j] = a;
            S.quarter2[quarter][j] = b;
        }
        __syncthreads();
        if (t < H) {
            gw3.add((S.quarter[0][t] + S.quarter[1][t]) + (S.quarter[2][t] + S.quarter[3][t]));
        } else if (t >= 128 && t < 128 + H) {
            const int o = t - 128;
            gb2.add((S.quarter2[0][o] + S.quarter2[1][o]) + (S.quarter2[2][o] + S.quarter2[3][o]));
        } else if (wid == 2) {
            float a = 0.f;
            for (int i = lane; i < ROWS; i += 32) a += S.d[i];
            for (int o = 16; o; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            gb3.add(a);
        } else if (t == 96) {
            float a = 0.f;
            for (int q = 0; q < GRAD_THREADS / 32; ++q) a += S.red[q];
            loss.add(a);
        }
        // dL/dW2[j][k] = sum_i g2[i][j] h1[i][k] (units 4 ty.., inputs 4 tx..)
        {
            float2 acc[4][2] = {};
#pragma unroll 4
            for (int i = 0; i < ROWS; ++i) {
                const float4 g = *reinterpret_cast<const float4*>(&S.h2[i * LD + 4 * ty]);
                const float4 h = *reinterpret_cast<const float4*>(&S.h1[i * LD + 4 * tx]);
                const float2 gv[4] = {make_float2(g.x, g.x), make_float2(g.y, g.y), make_float2(g.z, g.z),
                                      make_float2(g.w, g.w)};
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    acc[r][0] = __ffma2_rn(gv[r], make_float2(h.x, h.y), acc[r][0]);
                    acc[r][1] = __ffma2_rn(gv[r], make_float2(h.z, h.w), acc[r][1]);
                }
            }
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    gw2[r][2 * c].add(acc[r][c].x);
                    gw2[r][2 * c + 1].add(acc[r][c].y);
                }
        }
        __syncthreads();   // h1 is overwritten next
        // dL/da1[i][k] = (sum_j g2[i][j] W2[j][k]) (1 - h1[i][k]^2), rows ty + 16 r, inputs 4 tx..;
        // each thread overwrites only its own h1 entries, which no other thread reads in this phase
        {
            float2 acc[RPT][4] = {};
            tile_product<RPT>(acc, S.h2, w2, tx, ty);
#pragma unroll
            for (int r = 0; r < RPT; ++r)
#pragma unroll
                for (int c = 0; c < 4; c += 2) {
                    float2* const h = reinterpret_cast<float2*>(&S.h1[(ty + 16 * r) * LD + 2 * tx + 16 * c]);
                    const float2 v = *h;
                    *h = make_float2((acc[r][c].x + acc[r][c].y) * (1.f - v.x * v.x),
                                     (acc[r][c + 1].x + acc[r][c + 1].y) * (1.f - v.y * v.y));
                }
        }
        __syncthreads();
        // dL/dW1[j][c] = sum_i g1[i][j] z[i][c], dL/db1[j] = sum_i g1[i][j], by quarters of the rows
        {
            float a[D + 1] = {};
#pragma unroll 4
            for (int i = quarter * QROWS; i < (quarter + 1) * QROWS; ++i) {
                const float g = S.h1[i * LD + j];
                const float4 z = *reinterpret_cast<const float4*>(&S.z[i * ZS]);
                a[0] = fmaf(g, z.x, a[0]);
                a[1] = fmaf(g, z.y, a[1]);
                a[2] = fmaf(g, z.z, a[2]);
                a[3] = fmaf(g, z.w, a[3]);
                a[4] = fmaf(g, S.z[i * ZS + 4], a[4]);
                a[D] += g;
            }
            // dL/da2 is no longer needed: its place takes the quarters' sums
#pragma unroll
            for (int c = 0; c <= D; ++c) S.h2[(quarter * (D + 1) + c) * H + j] = a[c];
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int o = t + q * GRAD_THREADS;
            constexpr int Q = H * (D + 1);
            if (o < Q) small[q].add((S.h2[o] + S.h2[Q + o]) + (S.h2[2 * Q + o] + S.h2[3 * Q + o]));
        }
    }

    float* out = part + ((long long)f * gridDim.x + blockIdx.x) * kMlpStride;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int o = t + q * GRAD_THREADS;
        if (o < H * D) out[OW1 + (o & 63) * D + (o >> 6)] = small[q].value();
        else if (o < H * (D + 1)) out[OB1 + (o & 63)] = small[q].value();
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        *reinterpret_cast<float4*>(&out[OW2 + (4 * ty + r) * H + 4 * tx]) =
            make_float4(gw2[r][0].value(), gw2[r][1].value(), gw2[r][2].value(), gw2[r][3].value());
    }
    if (t < H) out[OW3 + t] = gw3.value();
    else if (t == 64) out[OB3] = gb3.value();
    else if (t == 96) out[kMlpParams] = loss.value();
    else if (t >= 128 && t < 128 + H) out[OB2 + t - 128] = gb2.value();
}

// Sum over the blocks' partials of parameter p (kMlpParams: the loss) in double precision: SUM_SPLIT threads
// (threadIdx.y) each take every SUM_SPLIT-th block, thread y = 0 gets the total. (One thread per parameter
// and 1,024 partials took 163 us, a chain of loads and additions on 36 SMs.)
constexpr int SUM_SPLIT = 16;

__device__ __forceinline__ double part_sum(const float* __restrict__ part, int nblk, int f, int p)
{
    __shared__ double red[SUM_SPLIT][32];
    double a = 0.0;
    if (p <= kMlpParams)
        for (int b = threadIdx.y; b < nblk; b += SUM_SPLIT) a += (double)part[((long long)f * nblk + b) * kMlpStride + p];
    red[threadIdx.y][threadIdx.x] = a;
    __syncthreads();
    if (threadIdx.y == 0)
        for (int q = 1; q < SUM_SPLIT; ++q) a += red[q][threadIdx.x];
    return a;
}

// The batch gradient and mean loss from the blocks' partials.
__global__ void __launch_bounds__(32 * SUM_SPLIT) k_mlp_reduce(const float* __restrict__ part, int nblk, float inv_rows,
                                                               float* __restrict__ grad, float* __restrict__ loss)
{
    const int f = blockIdx.y;
    const int p = blockIdx.x * 32 + threadIdx.x;
    const double a = part_sum(part, nblk, f, p);
    if (threadIdx.y != 0 || p > kMlpParams) return;
    if (p < kMlpParams) {
        grad[(long long)f * kMlpStride + p] = (float)a;
    } else if (loss) {
        loss[f] = (float)(a * inv_rows);
    }
}

struct AdamArgs {
    float lr;        // step size of this update
    float c1, c2;    // 1 / (1 - beta1^t), 1 / (1 - beta2^t)
    float beta1, beta2, eps;
    float inv_rows;
    int nblk;
    long long step;  // index into the loss record
};

// Adam (Kingma & Ba 2015, Algorithm 1) on the batch gradient, reduced from
// the blocks' partials.
__global__ void __launch_bounds__(32 * SUM_SPLIT) k_mlp_adam(float* __restrict__ theta, float* __restrict__ m, float* __restrict__ v,
                           const float* __restrict__ part, AdamArgs a, float* __restrict__ losses, long long steps)
{
    const int f = blockIdx.y;
    const int p = blockIdx.x * 32 + threadIdx.x;
    const double s = part_sum(part, a.nblk, f, p);
    if (threadIdx.y != 0 || p > kMlpParams) return;
    if (p == kMlpParams) {
        if (losses) losses[(long long)f * steps + a.step] = (float)(s * a.inv_rows);
        return;
    }
    const long long q = (long long)f * kMlpStride + p;
    const float g = (float)s;
    const float mm = a.beta1 * m[q] + (1.f - a.beta1) * g;
    const float vv = a.beta2 * v[q] + (1.f - a.beta2) * g * g;
    m[q] = mm;
    v[q] = vv;
    theta[q] -= a.lr * (mm * a.c1) / (sqrtf(vv * a.c2) + a.eps);
}

// ---------------------------------------------------------------- tabulation

__device__ __forceinline__ float tanh_approx(float x)
{
    float y;
    asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

struct TabArgs {
    const float* theta;     // [2][kMlpStride]
    const float* norm;      // mu[5], s[5]
    const float4* nfa;      // (w, r, dw/dx, dw/dy) per node
    const float2* nfb;      // (dr/dx, dr/dy) per node
    int nx, ny, slices;
    double* table;          // (slices, ny, nx, 4)
    int* status;            // STATUS_TIMEOUT if a bounded wait runs out
    float tfrac[kMaxCvSlices];
};

// ---- the 64 x 64 layer on the fifth-generation tensor cores
//
// A CTA of 256 threads takes tiles of 128 points (point p = slice * nodes +
// node). Layer 1: a thread takes 16 units of points t % 64 and t % 64 + 64, paired in its multiply-adds so that a
// weight is read once for both, and writes its part of three BF16 rows into shared memory: h1 = tanh(a1),
// u1 = (1 - h1^2) W1 dz/dx, v1 = (1 - h1^2) W1
// dz/dy. One thread issues the three products h1 W2^T, u1 W2^T, v1 W2^T as
// tcgen05.mma (M = 128, N = 64, K = 16, BF16 in, FP32 accumulate) into three
// 64-column accumulators in tensor memory, committed to an mbarrier; then
// warp w reads lanes 32 (w % 4) .. 32 (w % 4) + 31 (point t % 128), half of the columns, back with
// tcgen05.ld and forms its half of
// d/dx = sum_j w3_j (1 - tanh(a2_j)^2) (W2 u1)_j, d/dy likewise; the halves
// meet in shared memory. The operands are double-buffered: layer 1 of the next tile runs while the tensor cores
// work on this one. Bound by the instructions around the products (tensor pipe below 5 %): 2.1e5 points of two networks
// 59 us with a barrier between the stages and a weight read per point and unit, now 54.
//
// Operands are K-major without swizzle: 8 x 8 BF16 core matrices of 128
// contiguous bytes (a row's 8 consecutive k at 16-byte pitch); core matrices
// adjacent in k are 128 B apart (leading byte offset), 8-row groups 1024 B
// (stride byte offset). Byte offset of (row r, k): (r / 8) 1024 + (k / 8) 128
// + (r % 8) 16 + (k % 8) 2.

constexpr int TC_ROWS = 128;                         // points per tile = MMA M
constexpr int TC_THREADS = 2 * TC_ROWS;              // two threads per point
constexpr int TC_OPERAND_BYTES = TC_ROWS * H * 2;    // one 128 x 64 BF16 operand
constexpr int TC_W2_BYTES = H * H * 2;
constexpr int TC_TMEM_COLS = 256;                    // three 64-column FP32 accumulators, rounded to a power of two
// Dynamic shared memory requested per CTA: above a third of the SM's 228 KB,
// so that at most two CTAs (2 x 256 tensor-memory columns of 512) share an SM
// and tcgen05.alloc never waits.
constexpr int TC_SMEM_REQUEST = 112 * 1024;
constexpr long long TC_WAIT_LIMIT = 1LL << 26;       // polls of the MMA mbarrier before giving up

struct TcSmem {
    alignas(1024) unsigned char a[2][3][TC_OPERAND_BYTES];   // by parity of the tile
    alignas(1024) unsigned char b[TC_W2_BYTES];
    alignas(16) float w1[H][8];   // a unit's weights and bias of layer 1: w0 .. w4, b
    alignas(16) float b2[H], w3[H];
    float2 half_g[2][TC_ROWS];   // the second half's (d/dx, d/dy) partial sums, by parity of the tile
    alignas(8) unsigned long long mbar;
    uint32_t tmem;
    int abort;
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t core_off(int r, int k) { return (r >> 3) * 1024 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2; }

// Shared-memory matrix descriptor: start, leading and stride byte offsets (all
// >> 4), the fixed 0b001 at bits 46-48, no swizzle (bits 61-63 zero).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | (1ULL << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), BF16 A
// and B (bits 7-9, 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 at bits
// 17-22, M >> 4 at bits 24-28.
constexpr uint32_t tc_idesc(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        :: "r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}

// 16 consecutive accumulator columns of the thread's lane from each of three accumulators; the wait is in the
// same statement, so no use of the registers can be scheduled before it.
__device__ __forceinline__ void tc_ld16x3(uint32_t ta, uint32_t tb, uint32_t tc, float (&a)[16], float (&b)[16], float (&c)[16])
{
    uint32_t r[48];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%48];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, "
        "%29, %30, %31}, [%49];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, "
        "%45, %46, %47}, [%50];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=&r"(r[0]), "=&r"(r[1]), "=&r"(r[2]), "=&r"(r[3]), "=&r"(r[4]), "=&r"(r[5]), "=&r"(r[6]), "=&r"(r[7]),
          "=&r"(r[8]), "=&r"(r[9]), "=&r"(r[10]), "=&r"(r[11]), "=&r"(r[12]), "=&r"(r[13]), "=&r"(r[14]), "=&r"(r[15]),
          "=&r"(r[16]), "=&r"(r[17]), "=&r"(r[18]), "=&r"(r[19]), "=&r"(r[20]), "=&r"(r[21]), "=&r"(r[22]), "=&r"(r[23]),
          "=&r"(r[24]), "=&r"(r[25]), "=&r"(r[26]), "=&r"(r[27]), "=&r"(r[28]), "=&r"(r[29]), "=&r"(r[30]), "=&r"(r[31]),
          "=&r"(r[32]), "=&r"(r[33]), "=&r"(r[34]), "=&r"(r[35]), "=&r"(r[36]), "=&r"(r[37]), "=&r"(r[38]), "=&r"(r[39]),
          "=&r"(r[40]), "=&r"(r[41]), "=&r"(r[42]), "=&r"(r[43]), "=&r"(r[44]), "=&r"(r[45]), "=&r"(r[46]), "=&r"(r[47])
        : "r"(ta), "r"(tb), "r"(tc));
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        a[k] = __uint_as_float(r[k]);
        b[k] = __uint_as_float(r[16 + k]);
        c[k] = __uint_as_float(r[32 + k]);
    }
}

__global__ void __launch_bounds__(TC_THREADS) k_cv_tabulate(const TabArgs a)
{
    extern __shared__ unsigned char smem_raw[];
    TcSmem& S = *reinterpret_cast<TcSmem*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int f = blockIdx.y;
    const int t = threadIdx.x, warp = t >> 5;
    const int row = t % TC_ROWS, half = t / TC_ROWS;   // the point and the half of the units
    const float* th = a.theta + (long long)f * kMlpStride;

    // weights: layer 1 and the biases in FP32, W2 (B operand, rows n, k-major) in BF16
    for (int p = t; p < H * D; p += TC_THREADS) S.w1[p / D][p % D] = th[OW1 + p];
    for (int p = t; p < H; p += TC_THREADS) {
        S.w1[p][D] = th[OB1 + p];
        S.b2[p] = th[OB2 + p];
        S.w3[p] = th[OW3 + p];
    }
    for (int p = t; p < H * H / 8; p += TC_THREADS) {
        const int n = p / (H / 8), k0 = (p % (H / 8)) * 8;
        const float* wr = th + OW2 + n * H + k0;
        const uint4 v = make_uint4(pack_bf16(wr[0], wr[1]), pack_bf16(wr[2], wr[3]), pack_bf16(wr[4], wr[5]),
                                   pack_bf16(wr[6], wr[7]));
        *reinterpret_cast<uint4*>(S.b + core_off(n, k0)) = v;
    }
    if (t == 0) {
        S.abort = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&S.mbar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&S.tmem)), "n"(TC_TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = S.tmem;

    float mu[D], sc[D];
#pragma unroll
    for (int c = 0; c < D; ++c) {
        mu[c] = a.norm[c];
        sc[c] = a.norm[D + c];
    }
    const long long nn = (long long)a.nx * a.ny;
    const long long points = nn * a.slices;
    const long long tiles = (points + TC_ROWS - 1) / TC_ROWS;
    constexpr uint32_t idesc = tc_idesc(TC_ROWS, H);
    uint32_t phase = 0;
    // layer 1 of tile tl: 16 units of two of its points per thread (clamped in the ragged last tile; not written)
    auto layer1 = [&](long long tl, int par) {
        const int first = t % (TC_ROWS / 2), share = t / (TC_ROWS / 2);
        float2 z[D], dx3, dx4, dy3, dy4;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const long long pt = tl * TC_ROWS + first + q * (TC_ROWS / 2);
            const long long pc = pt < points ? pt : points - 1;
            int sl, i, j;
            long long node;
            if (points <= 0x7fffffffLL) {
                const uint32_t n = (uint32_t)nn, p32 = (uint32_t)pc, k = p32 / n, m = p32 - k * n;
                sl = (int)k;
                j = (int)(m / (uint32_t)a.nx);
                i = (int)(m - (uint32_t)j * (uint32_t)a.nx);
                node = m;
            } else {
                sl = (int)(pc / nn);
                node = pc - (long long)sl * nn;
                i = (int)(node % a.nx);
                j = (int)(node / a.nx);
            }
            const float4 fa = a.nfa[node];
            const float2 fb = a.nfb[node];
            auto put = [&](float2& v, float x) { (q ? v.y : v.x) = x; };
            put(z[0], ((float)i / (float)(a.nx - 1) - mu[0]) * sc[0]);
            put(z[1], ((float)j / (float)(a.ny - 1) - mu[1]) * sc[1]);
            put(z[2], (a.tfrac[sl] - mu[2]) * sc[2]);
            put(z[3], (fa.x - mu[3]) * sc[3]);
            put(z[4], (fa.y - mu[4]) * sc[4]);
            put(dx3, fa.z * sc[3]);
            put(dx4, fb.x * sc[4]);
            put(dy3, fa.w * sc[3]);
            put(dy4, fb.y * sc[4]);
        }
        const float2 dx0 = make_float2(sc[0], sc[0]), dy1 = make_float2(sc[1], sc[1]), one = make_float2(1.f, 1.f);
#pragma unroll 1
        for (int k0 = share * (H / 4); k0 < (share + 1) * (H / 4); k0 += 8) {
            uint32_t ph[2][4], pu[2][4], pv[2][4];   // by point
#pragma unroll
            for (int e = 0; e < 8; e += 2) {
                float2 hv[2], uv[2], vv[2];   // by unit
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const float4 wa = *reinterpret_cast<const float4*>(&S.w1[k0 + e + q][0]);
                    const float2 wb = *reinterpret_cast<const float2*>(&S.w1[k0 + e + q][4]);
                    const float2 w0 = make_float2(wa.x, wa.x), w1 = make_float2(wa.y, wa.y),
                                 w2 = make_float2(wa.z, wa.z), w3 = make_float2(wa.w, wa.w),
                                 w4 = make_float2(wb.x, wb.x);
                    float2 a1 = __ffma2_rn(w0, z[0], make_float2(wb.y, wb.y));
                    a1 = __ffma2_rn(w1, z[1], a1);
                    a1 = __ffma2_rn(w2, z[2], a1);
                    a1 = __ffma2_rn(w3, z[3], a1);
                    a1 = __ffma2_rn(w4, z[4], a1);
                    const float2 t1 = make_float2(tanh_approx(a1.x), tanh_approx(a1.y));
                    const float2 k1 = __ffma2_rn(make_float2(-t1.x, -t1.y), t1, one);
                    // the inputs' derivatives along x are zero in 1 and 2, along y in 0 and 2
                    const float2 ux = __ffma2_rn(w4, dx4, __ffma2_rn(w3, dx3, __fmul2_rn(w0, dx0)));
                    const float2 uy = __ffma2_rn(w4, dy4, __ffma2_rn(w3, dy3, __fmul2_rn(w1, dy1)));
                    hv[q] = t1;
                    uv[q] = __fmul2_rn(k1, ux);
                    vv[q] = __fmul2_rn(k1, uy);
                }
                ph[0][e / 2] = pack_bf16(hv[0].x, hv[1].x);
                pu[0][e / 2] = pack_bf16(uv[0].x, uv[1].x);
                pv[0][e / 2] = pack_bf16(vv[0].x, vv[1].x);
                ph[1][e / 2] = pack_bf16(hv[0].y, hv[1].y);
                pu[1][e / 2] = pack_bf16(uv[0].y, uv[1].y);
                pv[1][e / 2] = pack_bf16(vv[0].y, vv[1].y);
            }
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const uint32_t o = core_off(first + q * (TC_ROWS / 2), k0);
                *reinterpret_cast<uint4*>(S.a[par][0] + o) = make_uint4(ph[q][0], ph[q][1], ph[q][2], ph[q][3]);
                *reinterpret_cast<uint4*>(S.a[par][1] + o) = make_uint4(pu[q][0], pu[q][1], pu[q][2], pu[q][3]);
                *reinterpret_cast<uint4*>(S.a[par][2] + o) = make_uint4(pv[q][0], pv[q][1], pv[q][2], pv[q][3]);
            }
        }
        // the operands, written through the generic proxy, become visible to the tensor cores
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    };
    auto issue = [&](int par) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t bbase = smem_u32(S.b);
#pragma unroll
        for (int g = 0; g < 3; ++g) {
            const uint32_t abase = smem_u32(S.a[par][g]);
#pragma unroll
            for (int kk = 0; kk < H / 16; ++kk)
                tc_mma(tmem + (uint32_t)(H * g), smem_desc(abase + 256 * kk, 128, 1024),
                       smem_desc(bbase + 256 * kk, 128, 1024), idesc, kk > 0 ? 1u : 0u);
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                     :: "r"(smem_u32(&S.mbar)) : "memory");
    };
    // layer 1 of the next tile while the tensor cores work on this one; one barrier a tile: it says that the
    // accumulators have been read and that the next operands are in place (those of the tile before last are
    // free then: their products were waited for)
    if (blockIdx.x < tiles) {
        layer1(blockIdx.x, 0);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (t == 0) issue(0);
    }
    int par = 0;
    for (long long tl = blockIdx.x; tl < tiles; tl += gridDim.x, par ^= 1) {
        const bool more = tl + gridDim.x < tiles;
        if (more) layer1(tl + gridDim.x, par ^ 1);
        // wait for the products (bounded)
        {
            uint32_t done = 0;
            for (long long it = 0; it < TC_WAIT_LIMIT && !done; ++it)
                asm volatile(
                    "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                    "selp.u32 %0, 1, 0, p;\n\t}"
                    : "=r"(done) : "r"(smem_u32(&S.mbar)), "r"(phase) : "memory");
            if (!done) S.abort = 1;
        }
        phase ^= 1u;
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // epilogue: this thread's row from the three accumulators, 16 columns at a time
        float2 g = make_float2(0.f, 0.f);   // (d/dx, d/dy)
        const uint32_t lane_base = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
#pragma unroll 1
        for (int c0 = half * (H / 2); c0 < (half + 1) * (H / 2); c0 += 16) {
            float vh[16], vu[16], vv[16];
            tc_ld16x3(lane_base + (uint32_t)c0, lane_base + (uint32_t)(H + c0), lane_base + (uint32_t)(2 * H + c0), vh, vu, vv);
#pragma unroll
            for (int k = 0; k < 16; k += 2) {
                const float2 b = *reinterpret_cast<const float2*>(&S.b2[c0 + k]), w = *reinterpret_cast<const float2*>(&S.w3[c0 + k]);
                const float2 a2 = __fadd2_rn(make_float2(vh[k], vh[k + 1]), b);
                const float2 h2 = make_float2(tanh_approx(a2.x), tanh_approx(a2.y));
                const float2 wq = __fmul2_rn(w, __ffma2_rn(make_float2(-h2.x, -h2.y), h2, make_float2(1.f, 1.f)));
                g = __ffma2_rn(make_float2(wq.x, wq.x), make_float2(vu[k], vv[k]), g);
                g = __ffma2_rn(make_float2(wq.y, wq.y), make_float2(vu[k + 1], vv[k + 1]), g);
            }
        }
        if (half == 1) S.half_g[par][row] = g;
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (S.abort) {
            if (t == 0) atomicOr(a.status, STATUS_TIMEOUT);
            break;
        }
        if (more && t == 0) issue(par ^ 1);
        const long long pt = tl * TC_ROWS + row;
        if (half == 0 && pt < points) {
            const float2 o2 = S.half_g[par][row];
            double* o = a.table + pt * 4 + 2 * f;
            o[0] = (double)(g.x + o2.x);
            o[1] = (double)(g.y + o2.y);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "n"(TC_TMEM_COLS));
    }
}

int grid_for(long long n, int block)
{
    const long long b = (n + block - 1) / block;
    return (int)std::min<long long>(std::max<long long>(b, 1), 4096);
}

}  // namespace

// ---------------------------------------------------------------- launchers

cudaError_t launch_node_features(const float* w, int nx, int ny, double* w64, double* r64, double2* gw, float4* nfa,
                                 float2* nfb, cudaStream_t s)
{
    const long long n = (long long)nx * ny;
    k_node_w64<<<grid_for(n, 256), 256, 0, s>>>(w, n, w64);
    k_node_r<<<grid_for(n, 256), 256, 0, s>>>(w64, nx, ny, r64, gw);
    k_node_features<<<grid_for(n, 256), 256, 0, s>>>(w64, r64, gw, nx, ny, nfa, nfb);
    return cudaGetLastError();
}

cudaError_t launch_field_grad(const double* xi, const double* eta, int nx, int ny, double* table, cudaStream_t s)
{
    k_field_grad<<<dim3((unsigned)(nx + 255) / 256, (unsigned)std::min(ny, 65535)), 256, 0, s>>>(xi, eta, nx, ny, table);
    return cudaGetLastError();
}

cudaError_t launch_cv_smooth(const double* table, int nx, int ny, int order, float4* tmp, float4* cells,
                             cudaStream_t s)
{
    if (order < 1 || order > kCvMaxOrder || (order & 1) == 0) return cudaErrorInvalidValue;
    BinomWeights W{};
    W.order = order;
    double c = 1.0;   // C(order, m)
    for (int m = 0; m <= order; ++m) {
        W.w[m] = (float)std::ldexp(c, -order);
        c = c * (double)(order - m) / (double)(m + 1);
    }
    const dim3 grid((unsigned)(nx - 1 + 255) / 256, (unsigned)std::min(ny, 65535));
    k_cv_smooth_x<<<grid, SMOOTH_CELLS, 0, s>>>(table, nx, ny, W, tmp);
    k_cv_smooth_y<<<grid, 256, 0, s>>>(tmp, nx, ny, W, cells);
    return cudaGetLastError();
}

cudaError_t launch_cv_scatter(const double* xs, const double* ys, const double* yxi, const double* yeta,
                              const float4* nfa, int nx, int ny, int k, int K, int M, float* feats, float* targets,
                              cudaStream_t s)
{
    k_cv_scatter<<<grid_for(M, 256), 256, 0, s>>>(xs, ys, yxi, yeta, nfa, nx, ny, k, K, M, feats, targets);
    return cudaGetLastError();
}

size_t mlp_norm_scratch_doubles() { return (size_t)MOM_BLOCKS * D + D; }

cudaError_t launch_mlp_norm(const float* feats, long long n, double* scratch, float* norm, cudaStream_t s)
{
    double* part = scratch;
    double* mu = scratch + MOM_BLOCKS * D;
    const int nb = (int)std::min<long long>(MOM_BLOCKS, std::max<long long>(1, (n + 255) / 256));
    k_moments<<<nb, 256, 0, s>>>(feats, n, mu, 0, part);
    k_norm<<<1, 32, 0, s>>>(part, nb, n, mu, 0, norm);
    k_moments<<<nb, 256, 0, s>>>(feats, n, mu, 1, part);
    k_norm<<<1, 32, 0, s>>>(part, nb, n, mu, 1, norm);
    return cudaGetLastError();
}

int mlp_tile_rows() { return TILE; }

// Two blocks per SM, one for each network (three, at 80 registers, took as long).
int mlp_grad_blocks(long long rows, int sm_count)
{
    return (int)std::min<long long>(sm_count, (rows + TILE - 1) / TILE);
}

cudaError_t launch_mlp_grad(const float* theta, const float* norm, const float* feats, const float* targets,
                            long long row0, long long rows, float inv_batch, float* part, int sm_count,
                            cudaStream_t s)
{
    const size_t smem = sizeof(GradSmem);
    cudaError_t e = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)mlp_grad_blocks(rows, sm_count), 2);
    k_mlp_grad<<<grid, GRAD_THREADS, smem, s>>>(theta, norm, feats, targets, row0, rows, inv_batch, part);
    return cudaGetLastError();
}

cudaError_t launch_mlp_reduce(const float* part, int nblk, float inv_rows, float* grad, float* loss, cudaStream_t s)
{
    const dim3 grid((kMlpParams + 1 + 31) / 32, 2);
    k_mlp_reduce<<<grid, dim3(32, SUM_SPLIT), 0, s>>>(part, nblk, inv_rows, grad, loss);
    return cudaGetLastError();
}

cudaError_t launch_mlp_adam(float* theta, float* m, float* v, const float* part, int nblk, double lr, long long t,
                            float inv_rows, float* losses, long long steps, long long step, cudaStream_t s)
{
    AdamArgs a;
    const double b1 = 0.9, b2 = 0.999;
    a.lr = (float)lr;
    a.c1 = (float)(1.0 / (1.0 - std::pow(b1, (double)t)));
    a.c2 = (float)(1.0 / (1.0 - std::pow(b2, (double)t)));
    a.beta1 = (float)b1;
    a.beta2 = (float)b2;
    a.eps = 1e-8f;
    a.inv_rows = inv_rows;
    a.nblk = nblk;
    a.step = step;
    const dim3 grid((kMlpParams + 1 + 31) / 32, 2);
    k_mlp_adam<<<grid, dim3(32, SUM_SPLIT), 0, s>>>(theta, m, v, part, a, losses, steps);
    return cudaGetLastError();
}

cudaError_t launch_cv_tabulate(const float* theta, const float* norm, const float4* nfa, const float2* nfb, int nx,
                               int ny, int slices, const float* tfrac, double* table, int* status, int sm_count,
                               cudaStream_t s)
{
    static_assert(sizeof(TcSmem) + 1024 <= TC_SMEM_REQUEST, "tabulation shared memory");
    TabArgs a{};
    a.theta = theta;
    a.norm = norm;
    a.nfa = nfa;
    a.nfb = nfb;
    a.nx = nx;
    a.ny = ny;
    a.slices = slices;
    a.table = table;
    a.status = status;
    for (int q = 0; q < slices && q < kMaxCvSlices; ++q) a.tfrac[q] = tfrac[q];
    const long long tiles = ((long long)nx * ny * slices + TC_ROWS - 1) / TC_ROWS;
    if (tiles <= 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k_cv_tabulate, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM_REQUEST);
    if (e != cudaSuccess) return e;
    // two CTAs per SM and network at most (tensor-memory columns), both networks side by side
    const int grid = (int)std::min<long long>(tiles, (long long)sm_count);
    k_cv_tabulate<<<dim3(grid, 2), TC_THREADS, TC_SMEM_REQUEST, s>>>(a);
    return cudaGetLastError();
}

}  // namespace sdd
