// fields.cu -- per-mesh-step field preparation (the path kernel's tables).
//
//  * drift b = -grad w / w at the grid nodes by finite differences (Eq. 6;
//    Sec. 4 "derivatives ... approximated using finite differences"):
//    second-order central differences inside, second-order one-sided
//    differences (-3 w0 + 4 w1 - w2) / 2h on the edges, in double precision;
//  * per cell, the bilinear interpolant of b and of (xi, eta) written as
//    a0 + a1 s + a2 t + a3 s t over the cell's local coordinates (s, t), with
//    a0 = f00, a1 = f10 - f00, a2 = f01 - f00, a3 = f11 - f10 - f01 + f00,
//    formed in double and stored in single precision, the two components
//    interleaved (Sec. 4: bilinear interpolation between grid points);
//  * the boundary data of Sec. 3: xi = 0 / 1 on x = 0 / 1, eta = 0 / 1 on
//    y = 0 / 1, and on the other faces the 1D Winslow solution
//    int_0^s w / int_0^1 w (cumulative trapezoid, double precision).
#include <cuda_fp16.h>

#include <algorithm>

#include "common.cuh"

namespace sdd {

namespace {

__device__ __forceinline__ double2 node_drift(const float* __restrict__ w, int nx, int ny, int i, int j,
                                              double rx, double ry)
{
    // rx = 1 / (2 hx) = (nx - 1) / 2, ry likewise
    const float* row = w + (long long)j * nx;
    double wx, wy;
    if (i == 0)
        wx = (-3.0 * (double)row[0] + 4.0 * (double)row[1] - (double)row[2]) * rx;
    else if (i == nx - 1)
        wx = (3.0 * (double)row[nx - 1] - 4.0 * (double)row[nx - 2] + (double)row[nx - 3]) * rx;
    else
        wx = ((double)row[i + 1] - (double)row[i - 1]) * rx;
    const float* col = w + i;
    if (j == 0)
        wy = (-3.0 * (double)col[0] + 4.0 * (double)col[(long long)nx] - (double)col[2LL * nx]) * ry;
    else if (j == ny - 1)
        wy = (3.0 * (double)col[(long long)(ny - 1) * nx] - 4.0 * (double)col[(long long)(ny - 2) * nx] +
              (double)col[(long long)(ny - 3) * nx]) * ry;
    else
        wy = ((double)col[(long long)(j + 1) * nx] - (double)col[(long long)(j - 1) * nx]) * ry;
    const double r = -reciprocal((double)row[i]);
    return make_double2(wx * r, wy * r);
}

// Bilinear coefficients of two fields u, v on one cell, interleaved so that one
// paired single-precision FMA evaluates both: (a0u, a0v, a1u, a1v) and
// (a2u, a2v, a3u, a3v).
__device__ __forceinline__ void bilinear_coefs2(double u00, double u10, double u01, double u11, double v00,
                                                double v10, double v01, double v11, float4& lo, float4& hi)
{
    lo = make_float4((float)u00, (float)v00, (float)(u10 - u00), (float)(v10 - v00));
    hi = make_float4((float)(u01 - u00), (float)(v01 - v00), (float)((u11 - u10) - (u01 - u00)),
                     (float)((v11 - v10) - (v01 - v00)));
}

// Face data of one line of w: the cumulative trapezoid over its total, by one block: each thread sums a
// contiguous run of intervals, the run totals are scanned over the block, then each thread writes its run.
// (By one warp per line a 2049^2 grid's faces took 280 us, 64 dependent loads a thread.)
constexpr int FACE_THREADS = 256;
constexpr int FACE_BLOCKS = 5;   // blocks a grid's faces take

template <int T>
__device__ void block_cumtrapz(const float* __restrict__ v, long long stride, int n, double* __restrict__ out,
                               float* __restrict__ out32)
{
    __shared__ double part[T / 32];
    const int t = threadIdx.y * blockDim.x + threadIdx.x, lane = t & 31, warp = t >> 5;
    const int run = (n - 1 + T - 1) / T;
    const int k0 = min(1 + t * run, n), k1 = min(k0 + run, n);
    double mine = 0.0;
    for (int k = k0; k < k1; ++k) mine += 0.5 * ((double)v[(k - 1) * stride] + (double)v[k * stride]);
    double incl = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const double o = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += o;
    }
    if (lane == 31) part[warp] = incl;
    __syncthreads();
    double acc = incl - mine, total = 0.0;
    for (int q = 0; q < T / 32; ++q) {
        if (q < warp) acc += part[q];
        total += part[q];
    }
    if (t == 0) {
        out[0] = 0.0;
        if (out32) out32[0] = 0.f;
    }
    for (int k = k0; k < k1; ++k) {
        acc += 0.5 * ((double)v[(k - 1) * stride] + (double)v[k * stride]);
        const double f = acc / total;
        out[k] = f;
        if (out32) out32[k] = (float)f;
    }
}

// Part b of a grid's faces by a block of T threads. 0, 1: xi on y = 0, 1; 2, 3: eta on x = 0, 1; 4: xi on x = 0, 1
// and eta on y = 0, 1 (0 and 1).
template <int T>
__device__ void face_block(int b, const float* __restrict__ w, int nx, int ny, double* __restrict__ faces,
                           float* __restrict__ faces32)
{
    const long long per_field = 2LL * ny + 2LL * nx;
    // line q of a field: left, right (ny), bottom, top (nx)
    auto line = [&](int field, int q) { return field * per_field + (q < 2 ? q * (long long)ny : 2LL * ny + (q - 2) * (long long)nx); };
    if (b < 4) {
        const long long at = b < 2 ? line(0, 2 + b) : line(1, b - 2);
        const float* v = b == 0 ? w : b == 1 ? w + (long long)(ny - 1) * nx : b == 2 ? w : w + (nx - 1);
        block_cumtrapz<T>(v, b < 2 ? 1 : nx, b < 2 ? nx : ny, faces + at, faces32 ? faces32 + at : nullptr);
        return;
    }
    for (int q = 0; q < 4; ++q) {
        const long long at = q < 2 ? line(0, q) : line(1, q);
        const int n = q < 2 ? ny : nx;
        const double f = q & 1 ? 1.0 : 0.0;
        for (int k = threadIdx.y * blockDim.x + threadIdx.x; k < n; k += T) {
            faces[at + k] = f;
            if (faces32) faces32[at + k] = (float)f;
        }
    }
}

__global__ void __launch_bounds__(FACE_THREADS) k_winslow_faces(const float* __restrict__ w, int nx, int ny,
                                                                double* __restrict__ faces,
                                                                float* __restrict__ faces32)
{
    face_block<FACE_THREADS>(blockIdx.x, w, nx, ny, faces, faces32);
}

// The tables of one to N grids in one launch. Per grid five blocks for its faces where they are wanted, then
// one block per 32 x TY cells: the drift at the tile's 33 x (TY + 1) nodes once (in
// shared memory, double precision), then each cell's records. TY is 8, or 2 where blocks of 8 rows
// would not give every SM four of them: the kernel is bound by the double-precision lanes of the SMs in use.
// A small grid's faces and cells take 5 and 7 us by themselves, latency for the most part: with a launch for
// each, 16 grids of 65^2 to 513^2 spent 250 of the 1650 us of a batch's estimate on them; with one launch it took
// 1444 (1371 with the path kernel's gathers left out where there is no drift).
constexpr int PREP_TX = 32;
constexpr int PREP_MANY = 16;

template <int N>
struct PrepArgs {
    PrepItem it[N];
    int32_t block0[N];   // first block of each
    int32_t n;
};

// The zero maps of several grids, cleared before their cells mark them.
__global__ void k_clear_zmaps(const __grid_constant__ PrepArgs<PREP_MANY> a)
{
    uint8_t* z = a.it[blockIdx.x].zmap;
    if (!z || !a.it[blockIdx.x].bcoef) return;
    for (int k = threadIdx.x; k < kZmapBytes / 4; k += blockDim.x) reinterpret_cast<uint32_t*>(z)[k] = 0u;
}

template <int PREP_TY, int N>
__global__ void __launch_bounds__(PREP_TX * PREP_TY) k_prep_cells(const __grid_constant__ PrepArgs<N> a)
{
    __shared__ double2 bn[PREP_TY + 1][PREP_TX + 1];
    int g = 0;
    while (N > 1 && g + 1 < a.n && (int)blockIdx.x >= a.block0[g + 1]) ++g;
    const PrepItem& I = a.it[g];
    const float* __restrict__ w = I.w;
    const double* __restrict__ xi = I.xi;
    const double* __restrict__ eta = I.eta;
    float4* __restrict__ bcoef = I.bcoef;
    float4* __restrict__ fcoef = I.fcoef;
    uint8_t* __restrict__ zmap = I.zmap;
    int* status = I.status;
    const int nx = I.nx, ny = I.ny;
    int b = (int)blockIdx.x - a.block0[g];
    if (I.faces64) {
        if (b < FACE_BLOCKS) {
            face_block<PREP_TX * PREP_TY>(b, w, nx, ny, I.faces64, I.faces32);
            return;
        }
        b -= FACE_BLOCKS;
    }
    const int tiles = (nx - 1 + PREP_TX - 1) / PREP_TX;
    const int ix0 = b % tiles * PREP_TX, iy0 = b / tiles * PREP_TY;
    const int ix = ix0 + threadIdx.x, iy = iy0 + threadIdx.y;
    const bool cell_in = ix < nx - 1 && iy < ny - 1;
    if (bcoef) {
        bool nonzero = false;
        const double rx = 0.5 * (double)(nx - 1), ry = 0.5 * (double)(ny - 1);
        const int tid = threadIdx.y * PREP_TX + threadIdx.x;
        for (int k = tid; k < (PREP_TX + 1) * (PREP_TY + 1); k += PREP_TX * PREP_TY) {
            const int ti = k % (PREP_TX + 1), tj = k / (PREP_TX + 1);
            const int i = ix0 + ti, j = iy0 + tj;
            if (i < nx && j < ny) bn[tj][ti] = node_drift(w, nx, ny, i, j, rx, ry);
        }
        __syncthreads();
        if (cell_in) {
            // every node is checked by the cell that has it as lower-left corner,
            // the last row and column by the cells next to them
            bool bad = bad_w(w[(long long)iy * nx + ix]);
            if (ix == nx - 2) bad |= bad_w(w[(long long)iy * nx + ix + 1]);
            if (iy == ny - 2) bad |= bad_w(w[(long long)(iy + 1) * nx + ix]);
            if (ix == nx - 2 && iy == ny - 2) bad |= bad_w(w[(long long)(iy + 1) * nx + ix + 1]);
            if (bad) atomicOr(status, STATUS_BAD_W);
            const int tx = threadIdx.x, ty = threadIdx.y;
            const double2 b00 = bn[ty][tx], b10 = bn[ty][tx + 1], b01 = bn[ty + 1][tx], b11 = bn[ty + 1][tx + 1];
            const long long cell = (long long)iy * (nx - 1) + ix;
            float4 lo, hi;
            bilinear_coefs2(b00.x, b10.x, b01.x, b11.x, b00.y, b10.y, b01.y, b11.y, lo, hi);
            bcoef[2 * cell + 0] = lo;
            bcoef[2 * cell + 1] = hi;
            nonzero = lo.x != 0.f || lo.y != 0.f || lo.z != 0.f || lo.w != 0.f || hi.x != 0.f || hi.y != 0.f ||
                      hi.z != 0.f || hi.w != 0.f;
        }
        if (zmap) {
            // mark the tiles that the cell reaches, once per run of cells of a warp's row in the same tiles
            const float fx = (float)kZmapTiles / (float)(nx - 1), fy = (float)kZmapTiles / (float)(ny - 1);
            const int x0 = max(0, (int)floorf(((float)ix - 0.01f) * fx));
            const int x1 = min(kZmapTiles - 1, (int)floorf(((float)ix + 1.01f) * fx));
            const int run = nonzero ? x0 * kZmapTiles + x1 : -1;
            const int before = __shfl_up_sync(0xffffffffu, run, 1);
            if (nonzero && (threadIdx.x == 0 || run != before)) {
                const int y0 = max(0, (int)floorf(((float)iy - 0.01f) * fy));
                const int y1 = min(kZmapTiles - 1, (int)floorf(((float)iy + 1.01f) * fy));
                for (int ty = y0; ty <= y1; ++ty)
                    for (int tx = x0; tx <= x1; ++tx) zmap[ty * kZmapTiles + tx] = 1;
            }
        }
    }
    if (fcoef && cell_in) {
        const long long cell = (long long)iy * (nx - 1) + ix;
        const long long n00 = (long long)iy * nx + ix;
        const long long n01 = n00 + nx;
        bilinear_coefs2(xi[n00], xi[n00 + 1], xi[n01], xi[n01 + 1], eta[n00], eta[n00 + 1], eta[n01], eta[n01 + 1],
                        fcoef[2 * cell + 0], fcoef[2 * cell + 1]);
    }
}

// Control-variate table: node values (slice, j, i, 4) of the two models'
// gradients -> one 32-byte record per slice and cell holding the cell's four
// corner values in half precision (round to nearest even): the xi model's
// (d/dx, d/dy) at corners 00, 10, 01, 11, then the eta model's. The model the
// estimator uses is the bilinear interpolation of these rounded node values
// (continuous across cells: neighbouring cells hold the same rounded values).
__global__ void k_cv_cells(const double* __restrict__ g, int slices, int nx, int ny, uint4* __restrict__ cv)
{
    const int ix = blockIdx.x * blockDim.x + threadIdx.x;
    const int iy = blockIdx.y * blockDim.y + threadIdx.y;
    const int q = blockIdx.z;
    if (ix >= nx - 1 || iy >= ny - 1 || q >= slices) return;
    const double* T = g + (long long)q * nx * ny * 4;
    const long long n00 = (long long)iy * nx + ix;
    const long long corner[4] = {n00, n00 + 1, n00 + nx, n00 + nx + 1};
    const long long cell = (long long)q * (nx - 1) * (ny - 1) + (long long)iy * (nx - 1) + ix;
    uint32_t w[8];
    for (int f = 0; f < 2; ++f)
        for (int k = 0; k < 4; ++k) {
            const double* v = T + 4 * corner[k] + 2 * f;
            const __half hx = __double2half(v[0]), hy = __double2half(v[1]);
            w[4 * f + k] = (uint32_t)__half_as_ushort(hx) | ((uint32_t)__half_as_ushort(hy) << 16);
        }
    cv[2 * cell + 0] = make_uint4(w[0], w[1], w[2], w[3]);
    cv[2 * cell + 1] = make_uint4(w[4], w[5], w[6], w[7]);
}

__global__ void k_faces32(const double* __restrict__ f64, float* __restrict__ f32, int n)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) f32[k] = (float)f64[k];
}

}  // namespace

template <int TY, int N>
static cudaError_t launch_prep_n(const PrepItem* items, int n, cudaStream_t s)
{
    PrepArgs<N> a;
    a.n = n;
    long long blocks = 0;
    for (int k = 0; k < n; ++k) {
        a.it[k] = items[k];
        a.block0[k] = (int32_t)blocks;
        blocks += (items[k].faces64 ? FACE_BLOCKS : 0);
        if (items[k].bcoef || items[k].fcoef)
            blocks += (long long)((items[k].nx - 1 + PREP_TX - 1) / PREP_TX) * ((items[k].ny - 1 + TY - 1) / TY);
    }
    if constexpr (N == 1) {
        if (items[0].bcoef && items[0].zmap) {
            const cudaError_t e = cudaMemsetAsync(items[0].zmap, 0, kZmapBytes, s);
            if (e != cudaSuccess) return e;
        }
    } else {
        k_clear_zmaps<<<n, 256, 0, s>>>(a);
    }
    if (blocks > 0) k_prep_cells<TY, N><<<(unsigned)blocks, dim3(PREP_TX, TY), 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_prep(const PrepItem* items, int n, int sm_count, cudaStream_t s)
{
    for (int k0 = 0; k0 < n; k0 += PREP_MANY) {
        const int m = std::min(n - k0, PREP_MANY);
        long long blocks8 = 0;
        for (int k = k0; k < k0 + m; ++k)
            blocks8 += (long long)((items[k].nx - 1 + PREP_TX - 1) / PREP_TX) * ((items[k].ny - 1 + 7) / 8);
        const bool tall = blocks8 >= 4LL * sm_count;
        const PrepItem* q = items + k0;
        const cudaError_t e = m == 1 ? (tall ? launch_prep_n<8, 1>(q, m, s) : launch_prep_n<2, 1>(q, m, s))
                                     : (tall ? launch_prep_n<8, PREP_MANY>(q, m, s) : launch_prep_n<2, PREP_MANY>(q, m, s));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_cv_cells(const double* grad, int slices, int nx, int ny, uint4* cvcoef, cudaStream_t s)
{
    const dim3 block(32, 8);
    const dim3 grid((nx - 1 + 31) / 32, (ny - 1 + 7) / 8, slices);
    k_cv_cells<<<grid, block, 0, s>>>(grad, slices, nx, ny, cvcoef);
    return cudaGetLastError();
}

cudaError_t launch_winslow_faces(const float* w, int nx, int ny, double* faces64, float* faces32, cudaStream_t s)
{
    k_winslow_faces<<<FACE_BLOCKS, FACE_THREADS, 0, s>>>(w, nx, ny, faces64, faces32);
    return cudaGetLastError();
}

cudaError_t launch_faces32(const double* faces64, float* faces32, int n, cudaStream_t s)
{
    k_faces32<<<(n + 255) / 256, 256, 0, s>>>(faces64, faces32, n);
    return cudaGetLastError();
}

}  // namespace sdd
