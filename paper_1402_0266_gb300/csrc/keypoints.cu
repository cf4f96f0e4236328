// keypoints.cu -- key-point placement and interface fill (Sec. 4, Sec. 5).
//
// Sec. 4 evaluates the stochastic solution only near the maxima and minima of
// rho_x, rho_xx along the horizontal interfaces and of rho_y, rho_yy along the
// vertical ones (rho = 1 / w as in Sec. 5); Sec. 5 fills the other interface
// points by piecewise cubic Hermite interpolation. Along a line with positions
// t = 0 .. n - 1 (t = 0 and n - 1 on the boundary):
//
//   D1(t) = rho(t + 1) - rho(t - 1),  D2(t) = (rho(t + 1) - rho(t)) - (rho(t) - rho(t - 1))
//
// for t = 1 .. n - 2 in double precision (undivided: the grid spacing does not
// move an extremum). A position t in 2 .. n - 3 is a key point when D1 or D2
// has a local extremum there (p(t) > p(t - 1) and p(t) >= p(t + 1), or the
// mirror) of size |p(t)| >= max |p| / 100 (smaller ones are rounding noise
// where rho is flat); crossings of a vertical and a horizontal line are
// always key points, and so, with a spacing g > 0, is every position t with
// t mod g = 0 (the mesh also moves where rho is flat along a line). The fill is the monotone PCHIP interpolant (Fritsch &
// Carlson's scheme with Fritsch & Butland's derivative formula) through the
// line's two boundary values and its key points' estimates.
#include <algorithm>

#include "common.cuh"

namespace sdd {
namespace {

constexpr int KP_THREADS = 1024;

__device__ __forceinline__ long long line_node(const KeyLine& L, int nx, int t)
{
    // vertical line: column fixed, row t; horizontal line: row fixed, column t
    return L.orient == 0 ? (long long)t * nx + L.fixed : (long long)L.fixed * nx + t;
}

// The larger of two nonnegative doubles: ordered as integers, so the comparison stays
// off the SM's two double-precision lanes.
__device__ __forceinline__ double larger(double a, double b)
{
    return __longlong_as_double(max(__double_as_longlong(a), __double_as_longlong(b)));
}

// |d|, 0 where d is not a number: beside a density that is none the other differences keep their maximum.
__device__ __forceinline__ double magnitude(double d)
{
    const double m = fabs(d);
    return __double_as_longlong(m) > 0x7ff0000000000000LL ? 0.0 : m;
}

// One block per line: the profiles in shared memory, their largest sizes, then
// the extremum test at every position the line owns. Two 41-position lines: 27 us with every
// thread of 1,024 comparing 32 warps' maxima in double precision, 7 us now.
__global__ void __launch_bounds__(KP_THREADS) k_keypoints(const float* __restrict__ w, int nx,
                                                           const KeyLine* __restrict__ lines,
                                                           const int32_t* __restrict__ pos_idx,
                                                           const uint8_t* __restrict__ pos_cross,
                                                           int spacing, uint8_t* __restrict__ mask)
{
    extern __shared__ double prof[];   // D1 at [0, n), D2 at [n, 2n): entry t for t = 1 .. n - 2
    __shared__ double red[2][KP_THREADS / 32];
    const KeyLine L = lines[blockIdx.x];
    const int n = L.n;
    double m1 = 0.0, m2 = 0.0;
    for (int t = 1 + threadIdx.x; t <= n - 2; t += blockDim.x) {
        const double rm = 1.0 / (double)w[line_node(L, nx, t - 1)];
        const double r0 = 1.0 / (double)w[line_node(L, nx, t)];
        const double rp = 1.0 / (double)w[line_node(L, nx, t + 1)];
        const double d1 = rp - rm;
        const double d2 = (rp - r0) - (r0 - rm);
        prof[t] = d1;
        prof[n + t] = d2;
        m1 = larger(m1, magnitude(d1));
        m2 = larger(m2, magnitude(d2));
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 16; o; o >>= 1) {
        m1 = larger(m1, __shfl_xor_sync(0xffffffffu, m1, o));
        m2 = larger(m2, __shfl_xor_sync(0xffffffffu, m2, o));
    }
    if (lane == 0) {
        red[0][wid] = m1;
        red[1][wid] = m2;
    }
    __syncthreads();
    double big[2] = {0.0, 0.0};
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) {
        big[0] = larger(big[0], red[0][q]);
        big[1] = larger(big[1], red[1][q]);
    }
    for (int t = 1 + threadIdx.x; t <= n - 2; t += blockDim.x) {
        const int k = L.start + t - 1;
        if (pos_cross[k]) {
            if (L.orient == 0) mask[pos_idx[k]] = 1;   // a crossing belongs to its vertical line
            continue;
        }
        uint8_t key = (spacing > 0 && t % spacing == 0) ? 1 : 0;
        if (t >= 2 && t <= n - 3) {
            for (int q = 0; q < 2; ++q) {
                const double* p = prof + q * n;
                const double pm = p[t - 1], p0 = p[t], pp = p[t + 1];
                if (big[q] == 0.0 || fabs(p0) * 100.0 < big[q]) continue;
                if ((p0 > pm && p0 >= pp) || (p0 < pm && p0 <= pp)) key = 1;
            }
        }
        mask[pos_idx[k]] = key;
    }
}

// Derivative of the PCHIP interpolant at anchor k of m (positions ax, values ay): the slope of the only
// interval, Fritsch and Butland's weighted harmonic mean inside, shape-preserving three-point ends.
template <typename IT, typename DT>
__device__ __forceinline__ double pchip_derivative(const IT* ax, const DT* ay, int m, int k)
{
    if (m == 2) return (ay[1] - ay[0]) / (double)(ax[1] - ax[0]);
    if (k > 0 && k < m - 1) {
        const double h0 = (double)(ax[k] - ax[k - 1]), h1 = (double)(ax[k + 1] - ax[k]);
        const double s0 = (ay[k] - ay[k - 1]) * reciprocal(h0), s1 = (ay[k + 1] - ay[k]) * reciprocal(h1);
        if (s0 == 0.0 || s1 == 0.0 || (s0 > 0.0) != (s1 > 0.0)) return 0.0;
        const double w1 = 2.0 * h1 + h0, w2 = h1 + 2.0 * h0;
        // (w1 + w2) / (w1 / s0 + w2 / s1) by one division, with no product of the slopes that could underflow
        return (w1 + w2) * s0 * (s1 / (w1 * s1 + w2 * s0));
    }
    // end derivative from the first (last) two intervals
    const int a = k == 0 ? 0 : m - 1, b = k == 0 ? 1 : m - 2, c = k == 0 ? 2 : m - 3;
    const double h0 = fabs((double)(ax[b] - ax[a])), h1 = fabs((double)(ax[c] - ax[b]));
    const double s0 = (ay[b] - ay[a]) / (double)(ax[b] - ax[a]), s1 = (ay[c] - ay[b]) / (double)(ax[c] - ax[b]);
    const double d = ((2.0 * h0 + h1) * s0 - h0 * s1) / (h0 + h1);
    const auto sgn = [](double v) { return (v > 0.0) - (v < 0.0); };
    if (sgn(d) != sgn(s0)) return 0.0;
    if (sgn(s0) != sgn(s1) && fabs(d) > fabs(3.0 * s0)) return 3.0 * s0;
    return d;
}

// The interpolant at position t of the interval from anchor k to k + 1.
template <typename IT, typename DT>
__device__ __forceinline__ double pchip_value(const IT* ax, const DT* ay, const DT* ad, int k, int t)
{
    const double rh = reciprocal((double)(ax[k + 1] - ax[k]));
    const double s = (ay[k + 1] - ay[k]) * rh;
    const double e = ad[k] + ad[k + 1] - 2.0 * s;
    const double c3 = e * rh * rh;
    const double c2 = (s - ad[k] - e) * rh;
    const double u = (double)t - (double)ax[k];
    return ((c3 * u + c2) * u + ad[k]) * u + ay[k];
}

// The boundary values of field f at the two ends of line L.
__device__ __forceinline__ void line_ends(const KeyLine& L, const double* faces, int f, int nx, int ny, double& y0,
                                          double& y1)
{
    // face data: per field left[ny] right[ny] bottom[nx] top[nx]
    const double* F = faces + (long long)f * (2LL * ny + 2LL * nx);
    y0 = L.orient == 0 ? F[2 * ny + L.fixed] : F[L.fixed];
    y1 = L.orient == 0 ? F[2 * ny + nx + L.fixed] : F[ny + L.fixed];
}

constexpr int PCHIP_THREADS = 512;

// Lines of up to this many bytes' positions are filled in shared memory.
size_t pchip_smem_bytes(int n) { return (size_t)n * (6 * sizeof(double) + 3 * sizeof(int32_t) + 1); }

// One block per line: the key positions' places among the anchors by a count of the key flags before
// them (a ballot per 32 positions), then the derivatives, then the positions the line owns that are not key,
// each in parallel over the anchors or positions and both fields. (With one thread per field and line
// the fill of four 41-position lines took 80 us, a chain of double-precision divisions; now 10 us, a third of the divisions.)
__global__ void __launch_bounds__(PCHIP_THREADS) k_pchip_smem(const KeyLine* __restrict__ lines,
                                                              const int32_t* __restrict__ pos_idx,
                                                              const uint8_t* __restrict__ pos_cross,
                                                              const uint8_t* __restrict__ mask,
                                                              const double* __restrict__ faces, int nx, int ny,
                                                              double* __restrict__ mean_xi,
                                                              double* __restrict__ mean_eta, int max_n)
{
    extern __shared__ double sp[];
    const KeyLine L = lines[blockIdx.x];
    const int n = L.n, words = (n + 31) / 32;
    double* ay = sp;                                    // [2][max_n] anchor values
    double* ad = sp + 2LL * max_n;                      // [2][max_n] derivatives there
    int32_t* ax = reinterpret_cast<int32_t*>(sp + 4LL * max_n);   // [max_n] anchor positions
    uint32_t* keys = reinterpret_cast<uint32_t*>(ax + max_n);     // [words] key flags, bit t & 31 of word t / 32
    int32_t* before = reinterpret_cast<int32_t*>(keys + words);   // [words + 1] key positions before each word
    const int lane = threadIdx.x & 31;
    for (int t0 = (int)(threadIdx.x - lane); t0 < words * 32; t0 += blockDim.x) {
        const int t = t0 + lane;
        const bool key = t >= 1 && t <= n - 2 && mask[pos_idx[L.start + t - 1]] != 0;
        const uint32_t bits = __ballot_sync(0xffffffffu, key);
        if (lane == 0) keys[t0 >> 5] = bits;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        int sum = 0;
        for (int w0 = 0; w0 < words; w0 += 32) {
            const int mine = w0 + lane < words ? __popc(keys[w0 + lane]) : 0;
            int incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            if (w0 + lane < words) before[w0 + lane] = sum + incl - mine;
            sum += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) before[words] = sum;
    }
    __syncthreads();
    const int m = before[words] + 2;   // anchors: the key positions and the two ends
    // the last anchor at or before position t
    auto anchor = [&](int t) { return before[t >> 5] + __popc(keys[t >> 5] & (0xffffffffu >> (31 - (t & 31)))); };
    for (int t = 1 + threadIdx.x; t <= n - 2; t += blockDim.x)
        if ((keys[t >> 5] >> (t & 31)) & 1u) {
            const int a = anchor(t), i = pos_idx[L.start + t - 1];
            ax[a] = t;
            ay[a] = mean_xi[i];
            ay[max_n + a] = mean_eta[i];
        }
    if (threadIdx.x < 2) {
        const int f = threadIdx.x;
        double y0, y1;
        line_ends(L, faces, f, nx, ny, y0, y1);
        ay[(long long)f * max_n] = y0;
        ay[(long long)f * max_n + m - 1] = y1;
        ax[f == 0 ? 0 : m - 1] = f == 0 ? 0 : n - 1;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < 2 * m; k += blockDim.x) {
        const long long f = k >= m ? max_n : 0;
        ad[f + k - (k >= m ? m : 0)] = pchip_derivative(ax, ay + f, m, k >= m ? k - m : k);
    }
    __syncthreads();
    for (int t = 1 + threadIdx.x; t <= n - 2; t += blockDim.x) {
        const int p = L.start + t - 1;
        if (((keys[t >> 5] >> (t & 31)) & 1u) || (L.orient == 1 && pos_cross[p])) continue;
        const int a = anchor(t), i = pos_idx[p];
        mean_xi[i] = pchip_value(ax, ay, ad, a, t);
        mean_eta[i] = pchip_value(ax, ay + max_n, ad + max_n, a, t);
    }
}

// Lines too long for shared memory: one block per line, thread f < 2
// interpolates field f with its anchors in global scratch.
__global__ void k_pchip(const KeyLine* __restrict__ lines, const int32_t* __restrict__ pos_idx,
                        const uint8_t* __restrict__ pos_cross, const uint8_t* __restrict__ mask,
                        const double* __restrict__ faces, int nx, int ny, double* __restrict__ mean_xi,
                        double* __restrict__ mean_eta, double* __restrict__ scratch)
{
    const int f = threadIdx.x;
    if (f >= 2) return;
    const KeyLine L = lines[blockIdx.x];
    const int n = L.n;
    double* mean = f == 0 ? mean_xi : mean_eta;
    double y0, y1;
    line_ends(L, faces, f, nx, ny, y0, y1);
    // anchors: (x, y) and their derivatives, in this line's scratch region (three arrays of n per field;
    // the lines before this one hold L.start + 2 blockIdx.x positions in all)
    double* ax = scratch + 6LL * (L.start + 2LL * blockIdx.x) + 3LL * f * n;
    double* ay = ax + n;
    double* ad = ay + n;
    auto key = [&](int t) { return mask[pos_idx[L.start + t - 1]] != 0; };
    int m = 0;
    ax[m] = 0;
    ay[m++] = y0;
    for (int t = 1; t <= n - 2; ++t)
        if (key(t)) {
            ax[m] = t;
            ay[m++] = mean[pos_idx[L.start + t - 1]];
        }
    ax[m] = n - 1;
    ay[m++] = y1;
    for (int k = 0; k < m; ++k) ad[k] = pchip_derivative(ax, ay, m, k);
    int seg = 0;
    for (int t = 1; t <= n - 2; ++t) {
        if (key(t) || (L.orient == 1 && pos_cross[L.start + t - 1])) continue;
        while (seg < m - 2 && ax[seg + 1] < (double)t) ++seg;
        mean[pos_idx[L.start + t - 1]] = pchip_value(ax, ay, ad, seg, t);
    }
}

}  // namespace

cudaError_t launch_keypoints(const float* w, int nx, const KeyLine* lines, int nlines, int max_n,
                             const int32_t* pos_idx, const uint8_t* pos_cross, int spacing, uint8_t* mask,
                             cudaStream_t s)
{
    if (nlines <= 0) return cudaSuccess;
    const size_t smem = 2 * (size_t)max_n * sizeof(double);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_keypoints, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const int threads = std::min(KP_THREADS, (max_n + 31) / 32 * 32);
    k_keypoints<<<nlines, threads, smem, s>>>(w, nx, lines, pos_idx, pos_cross, spacing, mask);
    return cudaGetLastError();
}

size_t pchip_scratch_doubles(long long total_positions, int nlines)
{
    return (size_t)(6 * (total_positions + 2LL * nlines) + 16);
}

cudaError_t launch_pchip(const KeyLine* lines, int nlines, int max_n, const int32_t* pos_idx,
                         const uint8_t* pos_cross, const uint8_t* mask, const double* faces, int nx, int ny,
                         double* mean_xi, double* mean_eta, double* scratch, cudaStream_t s)
{
    if (nlines <= 0) return cudaSuccess;
    const size_t smem = pchip_smem_bytes(max_n);
    if (smem <= 200 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_pchip_smem, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_pchip_smem<<<nlines, std::min(PCHIP_THREADS, (max_n + 31) / 32 * 32), smem, s>>>(lines, pos_idx, pos_cross, mask, faces, nx, ny, mean_xi,
                                                         mean_eta, max_n);
    } else {
        k_pchip<<<nlines, 32, 0, s>>>(lines, pos_idx, pos_cross, mask, faces, nx, ny, mean_xi, mean_eta, scratch);
    }
    return cudaGetLastError();
}

}  // namespace sdd
