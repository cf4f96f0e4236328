// mg.cu -- multigrid-preconditioned conjugate gradients for large subdomains.
//
// The subdomain systems of Sec. 4 (the implicit step of Eq. (3) in the
// symmetric form xi / (w Dt) + sum_nb c_nb (xi - xi_nb) = rhs, an SPD
// M-matrix) become ill-conditioned as the grid is refined: the Jacobi preconditioner needs
// O(sqrt(Dt) / h) iterations, about 1,800 at 2049^2 with Dt = 1e-3. A
// geometric multigrid V-cycle as preconditioner brings that to a few tens.
//
// Levels: every system is a box of mx x my unknowns with a Dirichlet frame;
// while both sizes are odd and at least 3, the next level keeps every second
// node (M = (m - 1) / 2; coarse node I sits on fine node 2I). Coarse
// operators are rediscretised from the fine coefficients: the mass term
// 1 / (w Dt) is sampled, a coarse face's coefficient is the series
// combination of the two fine faces it spans, (1/2) c1 c2 / (c1 + c2), which
// keeps the scaling c / H^2 = c / (4 h^2) of a uniform medium. Smoother:
// red-black Gauss-Seidel, two sweeps before (red, black) and after (black,
// red) the coarse correction; restriction full weighting, prolongation
// bilinear (restriction = transpose / 4), so the V-cycle is symmetric. Levels
// of at most 4096 unknowns run inside one block per system; a larger level is
// one launch down and one up.
//
// Precision, as in the Jacobi kernels: the residual b - A x and the
// update x += d are double precision; the inner conjugate gradients on A d = r
// and the V-cycle are single precision (iterative refinement). Every dot
// product is reduced per block, then in block order. The solve runs inside a
// CUDA graph whose while-nodes stop once every field has converged; systems
// (and fields) that have converged before stop changing.
#include <algorithm>
#include <type_traits>

#include "common.cuh"

namespace sdd {
namespace {

constexpr int MG_THREADS = 256;
constexpr int TAIL_THREADS = 1024;
constexpr int TAIL_MAX_SMEM = 214200;   // of k_mg_tail, over every shape that mg_levels admits

// padded index -> (i, j) of level l
struct Lv {
    int W, H, mx, my;
    long long off;   // this system's first element
};

__device__ __forceinline__ Lv level(const MgArgs& a, int l, int s)
{
    Lv v;
    v.mx = a.mx[l];
    v.my = a.my[l];
    v.W = v.mx + 2;
    v.H = v.my + 2;
    v.off = a.off[l] + (long long)s * v.W * v.H;
    return v;
}

__device__ __forceinline__ bool any_active(const MgArgs& a, int s)
{
    return a.act_i[2 * s] | a.act_i[2 * s + 1];
}

// ---------------------------------------------------------------- setup

// Level 0 from the grid: D and the face coefficients (single precision
// copies), the mass term, and every level-0 vector zeroed (the frame stays
// zero for the whole solve).
__global__ void k_mg_coef0(const MgArgs a)
{
    const int s = blockIdx.y;
    const SolveSys S = a.sys[s];
    const Lv v = level(a, 0, s);
    const int P = v.W * v.H;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < P; idx += gridDim.x * blockDim.x) {
        const int ip = idx % v.W, jp = idx / v.W;
        const long long g = (long long)(S.j0 - 1 + jp) * a.nx + (S.i0 - 1 + ip);
        const bool in = ip >= 1 && ip <= v.mx && jp >= 1 && jp <= v.my;
        const long long e = v.off + idx;
        a.D[e] = in ? a.dgf[g] : 0.f;
        a.MS[e] = in ? (float)(1.0 / ((double)a.w[g] * a.Dt)) : 0.f;
        a.CX[e] = (ip <= v.mx && jp >= 1 && jp <= v.my) ? a.cxf[g] : 0.f;
        a.CY[e] = (jp <= v.my && ip >= 1 && ip <= v.mx) ? a.cyf[g] : 0.f;
        for (int f = 0; f < 2; ++f) {
            a.U[f][e] = 0.f;
            a.F[f][e] = 0.f;
            a.Z[f][e] = 0.f;
            a.Pv[f][idx + (long long)s * P] = 0.f;
            a.Qv[f][idx + (long long)s * P] = 0.f;
            a.Cv[f][idx + (long long)s * P] = 0.f;
        }
    }
}

__device__ __forceinline__ float series(float c1, float c2)
{
    return (c1 > 0.f && c2 > 0.f) ? 0.5f * c1 * c2 / (c1 + c2) : 0.f;
}

// Level l + 1 from level l (see the header: sampled mass, series faces).
__global__ void k_mg_coarsen(const MgArgs a, int l)
{
    const int s = blockIdx.y;
    const Lv h = level(a, l, s), c = level(a, l + 1, s);
    const int P = c.W * c.H;
    const float* CXh = a.CX + h.off;
    const float* CYh = a.CY + h.off;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < P; idx += gridDim.x * blockDim.x) {
        const int I = idx % c.W, J = idx / c.W;
        const int fi = 2 * I, fj = 2 * J;   // fine padded coordinates of the coarse node
        auto cxH = [&](int Ic, int Jc) { return series(CXh[2 * Jc * h.W + 2 * Ic], CXh[2 * Jc * h.W + 2 * Ic + 1]); };
        auto cyH = [&](int Ic, int Jc) {
            return series(CYh[2 * Jc * h.W + 2 * Ic], CYh[(2 * Jc + 1) * h.W + 2 * Ic]);
        };
        const bool in = I >= 1 && I <= c.mx && J >= 1 && J <= c.my;
        const long long e = c.off + idx;
        a.CX[e] = (I <= c.mx && J >= 1 && J <= c.my) ? cxH(I, J) : 0.f;
        a.CY[e] = (J <= c.my && I >= 1 && I <= c.mx) ? cyH(I, J) : 0.f;
        if (in) {
            const float ms = a.MS[h.off + (long long)fj * h.W + fi];
            a.MS[e] = ms;
            a.D[e] = ms + cxH(I - 1, J) + cxH(I, J) + cyH(I, J - 1) + cyH(I, J);
        } else {
            a.MS[e] = 0.f;
            a.D[e] = 0.f;
        }
        a.U[0][e] = a.U[1][e] = 0.f;
        a.F[0][e] = a.F[1][e] = 0.f;
        a.Z[0][e] = a.Z[1][e] = 0.f;
    }
}

// Per-block sums of two values per field -> part[s][block][4].
__device__ __forceinline__ void block_sum4(float v0, float v1, float v2, float v3, float* out)
{
    __shared__ float red[4][MG_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float v[4] = {v0, v1, v2, v3};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        for (int o = 16; o; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
        if (lane == 0) red[k][warp] = v[k];
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        float t = 0.f;
        for (int q = 0; q < MG_THREADS / 32; ++q) t += red[threadIdx.x][q];
        out[threadIdx.x] = t;
    }
}

__device__ __forceinline__ void block_sum4d(double v0, double v1, double v2, double v3, double* out)
{
    __shared__ double red[4][MG_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double v[4] = {v0, v1, v2, v3};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        for (int o = 16; o; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
        if (lane == 0) red[k][warp] = v[k];
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        double t = 0.0;
        for (int q = 0; q < MG_THREADS / 32; ++q) t += red[threadIdx.x][q];
        out[threadIdx.x] = t;
    }
}

// ---------------------------------------------------------------- V-cycle pieces
//
// Levels above `tail` run as two launches a level, one on the way down and one on the way up, each tile of
// 32 x 32 nodes by one block with the level's data in shared memory: a half-sweep needs its neighbours' values of
// the half-sweep before, so a block computes the four half-sweeps of a smoothing on regions that shrink by one
// node a side each, ending with its own tile (about twice the arithmetic, a fifth of the launches and of the
// memory traffic of a launch per half-sweep: the two levels above the tail of four 255^2 subdomains took 21 launches
// of about 10 us each for a V-cycle, now four of 15 us; they wait on barriers and shared memory).

constexpr int TILE = 32;
constexpr int PRE_R = TILE + 12, POST_R = TILE + 8;   // sides of the regions held

struct TileRegion {
    int x0, y0;   // padded coordinates of the region's first node
};

// One node of a Gauss-Seidel half-sweep in a region of side R: u = (f + sum of neighbours) / diagonal, both fields.
template <int R>
__device__ __forceinline__ void region_smooth(float2* u, const float2* f, const float* id, const float* cx,
                                              const float* cy, int e)
{
    const float2 w = u[e - 1], o = u[e + 1], s = u[e - R], n = u[e + R], b = f[e];
    const float cw = cx[e - 1], ce = cx[e], cs = cy[e - R], cn = cy[e], d = id[e];
    u[e] = make_float2((b.x + cw * w.x + ce * o.x + cs * s.x + cn * n.x) * d,
                       (b.y + cw * w.y + ce * o.y + cs * s.y + cn * n.y) * d);
}

// Half-sweep of a color on the region's nodes at least `in` from its sides. A node of color c has
// (padded column + padded row) & 1 == c. Nodes outside the box have id = 0 and keep u = 0.
template <int R>
__device__ __forceinline__ void region_sweep(float2* u, const float2* f, const float* id, const float* cx,
                                             const float* cy, TileRegion g, int in, int color)
{
    const int side = R - 2 * in, half = (side + 1) / 2;
    for (int k = threadIdx.x; k < side * half; k += MG_THREADS) {
        const int r = k / half, j = in + r;
        const int first = (g.x0 + g.y0 + in + j + color) & 1;   // 1: the row's first node has the other color
        const int i = in + 2 * (k - r * half) + first;
        if (i < R - in) region_smooth<R>(u, f, id, cx, cy, j * R + i);
    }
    __syncthreads();
}

// The level's data of the region: right-hand side, inverse diagonal (0 outside the box) and couplings.
template <int R>
__device__ __forceinline__ void region_load(const MgArgs& a, const Lv& v, TileRegion g, float2* f, float* id, float* cx,
                                            float* cy, float* dg)
{
    for (int k = threadIdx.x; k < R * R; k += MG_THREADS) {
        const int jp = g.y0 + k / R, ip = g.x0 + k % R;
        const bool held = ip >= 0 && ip < v.W && jp >= 0 && jp < v.H;
        const long long e = v.off + (long long)jp * v.W + ip;
        const float d = held ? a.D[e] : 0.f;
        id[k] = d > 0.f ? 1.f / d : 0.f;
        if (dg) dg[k] = d;
        cx[k] = held ? a.CX[e] : 0.f;
        cy[k] = held ? a.CY[e] : 0.f;
        f[k] = held ? make_float2(a.F[0][e], a.F[1][e]) : make_float2(0.f, 0.f);
    }
}

struct PreSmem {
    float2 u[PRE_R * PRE_R], f[PRE_R * PRE_R];
    float id[PRE_R * PRE_R], cx[PRE_R * PRE_R], cy[PRE_R * PRE_R], dg[PRE_R * PRE_R];
};

// Down: from U_l = 0, nu = 2 sweeps (red, black), then F_{l+1} = full weighting of F_l - A_l U_l and U_{l+1} = 0.
// The coarse nodes of a tile need the residual one node past it, and that the iterate one node further.
__global__ void __launch_bounds__(MG_THREADS) k_mg_down(const MgArgs a, int l, int tiles_x)
{
    extern __shared__ __align__(16) unsigned char mg_smem[];
    PreSmem& S = *reinterpret_cast<PreSmem*>(mg_smem);
    const int s = blockIdx.y;
    if (!any_active(a, s)) return;
    const Lv v = level(a, l, s), c = level(a, l + 1, s);
    const int bx = blockIdx.x % tiles_x, by = blockIdx.x / tiles_x;
    constexpr int R = PRE_R;
    const TileRegion g{TILE * bx - 4, TILE * by - 4};   // own nodes: TILE b + 1 .. TILE b + TILE
    for (int k = threadIdx.x; k < R * R; k += MG_THREADS) S.u[k] = make_float2(0.f, 0.f);
    region_load<R>(a, v, g, S.f, S.id, S.cx, S.cy, S.dg);
    __syncthreads();
    for (int h = 0; h < 4; ++h) region_sweep<R>(S.u, S.f, S.id, S.cx, S.cy, g, 1 + h, h & 1);
    // own nodes
    for (int k = threadIdx.x; k < TILE * TILE; k += MG_THREADS) {
        const int i = 5 + k % TILE, j = 5 + k / TILE, ip = g.x0 + i, jp = g.y0 + j;
        if (ip > v.mx || jp > v.my) continue;
        const float2 u = S.u[j * R + i];
        const long long e = v.off + (long long)jp * v.W + ip;
        a.U[0][e] = u.x;
        a.U[1][e] = u.y;
    }
    // residuals in the place of the right-hand side, from own nodes to one past them
    for (int k = threadIdx.x; k < (TILE + 2) * (TILE + 2); k += MG_THREADS) {
        const int e = (5 + k / (TILE + 2)) * R + 5 + k % (TILE + 2);
        const float2 u = S.u[e], w = S.u[e - 1], o = S.u[e + 1], t = S.u[e - R], n = S.u[e + R], b = S.f[e];
        const float d = S.dg[e], cw = S.cx[e - 1], ce = S.cx[e], cs = S.cy[e - R], cn = S.cy[e];
        const bool in = S.id[e] > 0.f;
        S.f[e] = in ? make_float2(b.x - (d * u.x - cw * w.x - ce * o.x - cs * t.x - cn * n.x),
                                  b.y - (d * u.y - cw * w.y - ce * o.y - cs * t.y - cn * n.y))
                    : make_float2(0.f, 0.f);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < TILE * TILE / 4; k += MG_THREADS) {
        const int I = TILE / 2 * bx + 1 + k % (TILE / 2), J = TILE / 2 * by + 1 + k / (TILE / 2);
        if (I > c.mx || J > c.my) continue;
        const float2* r = S.f + (2 * J - g.y0) * R + (2 * I - g.x0);
        auto sum2 = [](float2 p, float2 q) { return make_float2(p.x + q.x, p.y + q.y); };
        const float2 cross = sum2(sum2(r[-1], r[1]), sum2(r[-R], r[R]));
        const float2 diag = sum2(sum2(r[-R - 1], r[-R + 1]), sum2(r[R - 1], r[R + 1]));
        const long long e = c.off + (long long)J * c.W + I;
        a.F[0][e] = (4.f * r[0].x + 2.f * cross.x + diag.x) * (1.f / 16.f);
        a.F[1][e] = (4.f * r[0].y + 2.f * cross.y + diag.y) * (1.f / 16.f);
        a.U[0][e] = a.U[1][e] = 0.f;
    }
}

struct PostSmem {
    float2 u[POST_R * POST_R], f[POST_R * POST_R];
    float id[POST_R * POST_R], cx[POST_R * POST_R], cy[POST_R * POST_R];
};

// Up: Z_l = U_l + bilinear interpolation of the coarse iterate, then two sweeps (black, red). The result goes to
// arrays of its own: a block reads its neighbours' nodes of U_l. At level 0 the block also sums its part of (r, z).
__global__ void __launch_bounds__(MG_THREADS) k_mg_up(const MgArgs a, int l, int tiles_x)
{
    extern __shared__ __align__(16) unsigned char mg_smem[];
    PostSmem& S = *reinterpret_cast<PostSmem*>(mg_smem);
    const int s = blockIdx.y;
    const bool on = any_active(a, s);
    if (!on && l > 0) return;
    const Lv v = level(a, l, s), c = level(a, l + 1, s);
    const int bx = blockIdx.x % tiles_x, by = blockIdx.x / tiles_x;
    constexpr int R = POST_R;
    const TileRegion g{TILE * bx - 3, TILE * by - 3};   // own nodes at 4 .. 4 + TILE - 1
    float rz[2] = {0.f, 0.f};
    if (on) {
        // the coarse iterate: the level below `tail` leaves it in U, the others in Z
        const float* uc0 = (l + 1 == a.tail ? a.U[0] : a.Z[0]) + c.off;
        const float* uc1 = (l + 1 == a.tail ? a.U[1] : a.Z[1]) + c.off;
        region_load<R>(a, v, g, S.f, S.id, S.cx, S.cy, nullptr);
        for (int k = threadIdx.x; k < R * R; k += MG_THREADS) {
            const int jp = g.y0 + k / R, ip = g.x0 + k % R;
            float2 u = make_float2(0.f, 0.f);
            if (ip >= 1 && ip <= v.mx && jp >= 1 && jp <= v.my) {
                const long long e = v.off + (long long)jp * v.W + ip;
                const int c00 = (jp >> 1) * c.W + (ip >> 1), c10 = (jp >> 1) * c.W + ((ip + 1) >> 1);
                const int c01 = ((jp + 1) >> 1) * c.W + (ip >> 1), c11 = ((jp + 1) >> 1) * c.W + ((ip + 1) >> 1);
                u.x = a.U[0][e] + 0.25f * (uc0[c00] + uc0[c10] + uc0[c01] + uc0[c11]);
                u.y = a.U[1][e] + 0.25f * (uc1[c00] + uc1[c10] + uc1[c01] + uc1[c11]);
            }
            S.u[k] = u;
        }
        __syncthreads();
        for (int h = 0; h < 4; ++h) region_sweep<R>(S.u, S.f, S.id, S.cx, S.cy, g, 1 + h, (h + 1) & 1);
        for (int k = threadIdx.x; k < TILE * TILE; k += MG_THREADS) {
            const int i = 4 + k % TILE, j = 4 + k / TILE, ip = g.x0 + i, jp = g.y0 + j;
            if (ip > v.mx || jp > v.my) continue;
            const float2 u = S.u[j * R + i], f = S.f[j * R + i];
            const long long e = v.off + (long long)jp * v.W + ip;
            a.Z[0][e] = u.x;
            a.Z[1][e] = u.y;
            rz[0] += f.x * u.x;
            rz[1] += f.y * u.y;
        }
    }
    if (l == 0) block_sum4(rz[0], rz[1], 0.f, 0.f, a.part + ((long long)s * a.T0 + blockIdx.x) * 4);
}


// The levels from `tail` down in shared memory, one block per system: a row of a level per warp and step, so
// that no index is divided. The 50 phases of the levels from 63^2 down are a chain of block barriers, the
// bound here: 29 us (51 from a cold cache, where the levels in global memory took 61). A level of at most 4096
// unknowns and all below it fill at most 214,200 bytes (31 x 543) over every shape that mg_levels admits.
struct TailSmem {
    float2* u[kMgMaxLevels];
    float2* f[kMgMaxLevels];
    float* id[kMgMaxLevels];
    float* cx[kMgMaxLevels];
    float* cy[kMgMaxLevels];
};

size_t tail_smem_bytes(const MgArgs& a)
{
    size_t nodes = 0;
    for (int l = a.tail; l < a.levels; ++l) nodes += (size_t)(a.mx[l] + 2) * (a.my[l] + 2);
    return nodes * (2 * sizeof(float2) + 3 * sizeof(float)) + (size_t)(a.mx[a.tail] + 2) * (a.my[a.tail] + 2) * sizeof(float2);
}

__global__ void __launch_bounds__(TAIL_THREADS) k_mg_tail(const MgArgs a)
{
    extern __shared__ __align__(16) unsigned char mg_smem[];
    __shared__ TailSmem T;
    const int s = blockIdx.x;
    if (!any_active(a, s)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int WARPS = TAIL_THREADS / 32;
    const int lt = a.tail, L = a.levels;
    auto size = [&](int l) { return (a.mx[l] + 2) * (a.my[l] + 2); };
    if (threadIdx.x == 0) {
        float2* p = reinterpret_cast<float2*>(mg_smem) + size(lt);   // first the residuals
        for (int l = lt; l < L; ++l) {
            T.u[l] = p;
            T.f[l] = p + size(l);
            p += 2 * size(l);
        }
        float* q = reinterpret_cast<float*>(p);
        for (int l = lt; l < L; ++l) {
            T.id[l] = q;
            T.cx[l] = q + size(l);
            T.cy[l] = q + 2 * size(l);
            q += 3 * size(l);
        }
    }
    float2* const res = reinterpret_cast<float2*>(mg_smem);
    __syncthreads();
    for (int l = lt; l < L; ++l) {
        const Lv v = level(a, l, s);
        const int n = v.W * v.H;
        // five nodes a thread in flight (a 65^2 box in one round)
        constexpr int BATCH = 5;
        for (int k0 = threadIdx.x; k0 < n; k0 += BATCH * TAIL_THREADS) {
            float d[BATCH], cx[BATCH], cy[BATCH];
            float2 f[BATCH];
#pragma unroll
            for (int q = 0; q < BATCH; ++q) {
                const int k = k0 + q * TAIL_THREADS;
                d[q] = 0.f;
                f[q] = make_float2(0.f, 0.f);
                if (k >= n) continue;
                const long long e = v.off + k;
                d[q] = a.D[e];
                cx[q] = a.CX[e];
                cy[q] = a.CY[e];
                if (l == lt) f[q] = make_float2(a.F[0][e], a.F[1][e]);
            }
#pragma unroll
            for (int q = 0; q < BATCH; ++q) {
                const int k = k0 + q * TAIL_THREADS;
                if (k >= n) continue;
                T.id[l][k] = d[q] > 0.f ? 1.f / d[q] : 0.f;
                T.cx[l][k] = cx[q];
                T.cy[l][k] = cy[q];
                T.u[l][k] = make_float2(0.f, 0.f);
                T.f[l][k] = f[q];
            }
        }
    }
    __syncthreads();
    // the first level's coefficients in registers where a thread has two nodes of each colour at most
    const int W0 = a.mx[lt] + 2;
    const bool held = a.mx[lt] <= 64 && a.my[lt] <= 2 * WARPS;
    float hw[2][2], he[2][2], hs[2][2], hn[2][2], hd[2][2];   // [colour][row]
    float2 hf[2][2];
    auto held_at = [&](int color, int r, int& e) {
        const int j = 1 + warp + r * WARPS, i = 1 + 2 * lane + ((j + 1 + color) & 1);
        e = j * W0 + i;
        return j <= a.my[lt] && i <= a.mx[lt];
    };
#pragma unroll
    for (int color = 0; color < 2; ++color)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            int e;
            hw[color][r] = he[color][r] = hs[color][r] = hn[color][r] = hd[color][r] = 0.f;
            hf[color][r] = make_float2(0.f, 0.f);
            if (!held || !held_at(color, r, e)) continue;
            hw[color][r] = T.cx[lt][e - 1];
            he[color][r] = T.cx[lt][e];
            hs[color][r] = T.cy[lt][e - W0];
            hn[color][r] = T.cy[lt][e];
            hd[color][r] = T.id[lt][e];
            hf[color][r] = T.f[lt][e];
        }
    auto held_sweep = [&](auto colour) {
        constexpr int color = decltype(colour)::value;
        float2* const u = T.u[lt];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            int e;
            if (!held_at(color, r, e)) continue;
            const float2 w = u[e - 1], o = u[e + 1], t = u[e - W0], n = u[e + W0], b = hf[color][r];
            const float cw = hw[color][r], ce = he[color][r], cs = hs[color][r], cn = hn[color][r], d = hd[color][r];
            u[e] = make_float2((b.x + cw * w.x + ce * o.x + cs * t.x + cn * n.x) * d,
                               (b.y + cw * w.y + ce * o.y + cs * t.y + cn * n.y) * d);
        }
        __syncthreads();
    };
    auto sweep = [&](int l, int color) {
        if (held && l == lt) {
            if (color == 0) held_sweep(std::integral_constant<int, 0>());
            else held_sweep(std::integral_constant<int, 1>());
            return;
        }
        const int mx = a.mx[l], my = a.my[l], W = mx + 2;
        float2* const u = T.u[l];
        for (int j = 1 + warp; j <= my; j += WARPS)
            for (int i = 1 + 2 * lane + ((j + 1 + color) & 1); i <= mx; i += 64) {
                const int e = j * W + i;
                const float2 w = u[e - 1], o = u[e + 1], t = u[e - W], n = u[e + W], b = T.f[l][e];
                const float cw = T.cx[l][e - 1], ce = T.cx[l][e], cs = T.cy[l][e - W], cn = T.cy[l][e], d = T.id[l][e];
                u[e] = make_float2((b.x + cw * w.x + ce * o.x + cs * t.x + cn * n.x) * d,
                                   (b.y + cw * w.y + ce * o.y + cs * t.y + cn * n.y) * d);
            }
        __syncthreads();
    };
    for (int l = lt; l < L - 1; ++l) {
        for (int k = 0; k < a.nu; ++k) {
            sweep(l, 0);
            sweep(l, 1);
        }
        const int mx = a.mx[l], my = a.my[l], W = mx + 2, mc = a.mx[l + 1], Wc = mc + 2;
        for (int j = warp; j < my + 2; j += WARPS)
            for (int i = lane; i < W; i += 32) {
                const int e = j * W + i;
                float2 r = make_float2(0.f, 0.f);
                if (i >= 1 && i <= mx && j >= 1 && j <= my) {
                    const float2* u = T.u[l] + e;
                    const float2 b = T.f[l][e];
                    const float cw = T.cx[l][e - 1], ce = T.cx[l][e], cs = T.cy[l][e - W], cn = T.cy[l][e], d = 1.f / T.id[l][e];
                    r.x = b.x - (d * u[0].x - cw * u[-1].x - ce * u[1].x - cs * u[-W].x - cn * u[W].x);
                    r.y = b.y - (d * u[0].y - cw * u[-1].y - ce * u[1].y - cs * u[-W].y - cn * u[W].y);
                }
                res[e] = r;
            }
        __syncthreads();
        for (int J = 1 + warp; J <= a.my[l + 1]; J += WARPS)
            for (int I = 1 + lane; I <= mc; I += 32) {
                const float2* r = res + 2 * J * W + 2 * I;
                auto sum2 = [](float2 p, float2 q) { return make_float2(p.x + q.x, p.y + q.y); };
                const float2 cross = sum2(sum2(r[-1], r[1]), sum2(r[-W], r[W]));
                const float2 diag = sum2(sum2(r[-W - 1], r[-W + 1]), sum2(r[W - 1], r[W + 1]));
                T.f[l + 1][J * Wc + I] = make_float2((4.f * r[0].x + 2.f * cross.x + diag.x) * (1.f / 16.f),
                                                     (4.f * r[0].y + 2.f * cross.y + diag.y) * (1.f / 16.f));
            }
        __syncthreads();
    }
    // coarsest level: one unknown is solved exactly (by any sweep), a larger box by many sweeps
    const int last = a.mx[L - 1] == 1 && a.my[L - 1] == 1 ? 1 : a.coarse_sweeps;
    for (int k = 0; k < last; ++k) {
        sweep(L - 1, 0);
        sweep(L - 1, 1);
    }
    if (last > 1)
        for (int k = 0; k < last; ++k) {
            sweep(L - 1, 1);
            sweep(L - 1, 0);
        }
    for (int l = L - 2; l >= lt; --l) {
        const int mx = a.mx[l], my = a.my[l], W = mx + 2, Wc = a.mx[l + 1] + 2;
        const float2* const uc = T.u[l + 1];
        for (int j = 1 + warp; j <= my; j += WARPS)
            for (int i = 1 + lane; i <= mx; i += 32) {
                const int r0 = (j >> 1) * Wc, r1 = ((j + 1) >> 1) * Wc, c0 = i >> 1, c1 = (i + 1) >> 1;
                const float2 p = uc[r0 + c0], q = uc[r0 + c1], r = uc[r1 + c0], t = uc[r1 + c1];
                float2& u = T.u[l][j * W + i];
                u = make_float2(u.x + 0.25f * (p.x + q.x + r.x + t.x), u.y + 0.25f * (p.y + q.y + r.y + t.y));
            }
        __syncthreads();
        for (int k = 0; k < a.nu; ++k) {
            sweep(l, 1);
            sweep(l, 0);
        }
    }
    const Lv v = level(a, lt, s);
    for (int k = threadIdx.x; k < v.W * v.H; k += TAIL_THREADS) {
        const float2 u = T.u[lt][k];
        a.U[0][v.off + k] = u.x;
        a.U[1][v.off + k] = u.y;
    }
}

// ---------------------------------------------------------------- Krylov pieces (level-0 vectors)

// Values 0 and 1 of a system's `count` block partials summed by one warp, the same order in every caller.
__device__ __forceinline__ float2 warp_part_sums(const float* part, int s, int count)
{
    float x = 0.f, y = 0.f;
    for (int b = threadIdx.x & 31; b < count; b += 32) {
        const float2 v = *reinterpret_cast<const float2*>(part + ((long long)s * count + b) * 4);
        x += v.x;
        y += v.y;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
    }
    return make_float2(x, y);
}

// The same for every thread of a block (one thread after another took 5 us for 64 partials).
__device__ __forceinline__ float2 block_part_sums(const float* part, int s, int count)
{
    __shared__ float2 total;
    if (threadIdx.x < 32) {
        const float2 t = warp_part_sums(part, s, count);
        if (threadIdx.x == 0) total = t;
    }
    __syncthreads();
    return total;
}

// Double-precision residual of the current fields on every unknown; writes it
// (single precision) as the V-cycle's level-0 right-hand side, zeroes the
// correction; per-block sums of ||r||^2 and
// ||b||^2 (b = rhs + the Dirichlet neighbours' terms).
__global__ void __launch_bounds__(MG_THREADS) k_mg_res64(const MgArgs a)
{
    const int s = blockIdx.y;
    const SolveSys S = a.sys[s];
    const Lv v = level(a, 0, s);
    const int n = v.mx * v.my;
    const int nx = a.nx;
    double rr[2] = {0.0, 0.0}, bb[2] = {0.0, 0.0};
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int ip = 1 + k % v.mx, jp = 1 + k / v.mx;
        const int i = S.i0 - 1 + ip, j = S.j0 - 1 + jp;
        const long long g = (long long)j * nx + i;
        const long long e = (long long)jp * v.W + ip;
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            const double* x = a.x[f];
            const double* rhs = a.rhs0 + (long long)f * nx * a.ny;
            const double ax = a.dg[g] * x[g] - a.cx[g - 1] * x[g - 1] - a.cx[g] * x[g + 1] - a.cy[g - nx] * x[g - nx] -
                              a.cy[g] * x[g + nx];
            const double r = rhs[g] - ax;
            double b = rhs[g];
            if (i == S.i0) b += a.cx[g - 1] * x[g - 1];
            if (i == S.i1 - 1) b += a.cx[g] * x[g + 1];
            if (j == S.j0) b += a.cy[g - nx] * x[g - nx];
            if (j == S.j1 - 1) b += a.cy[g] * x[g + nx];
            rr[f] += r * r;
            bb[f] += b * b;
            a.F[f][v.off + e] = (float)r;
            a.Cv[f][(long long)s * v.W * v.H + e] = 0.f;
        }
    }
    block_sum4d(rr[0], rr[1], bb[0], bb[1], a.part64 + ((long long)s * a.B0 + blockIdx.x) * 4);
}

// Per system and field: outer convergence. first: stop2 = rtol^2 ||b||^2 and
// every field starts active. final: the status and iteration counts. The two
// fields of a system are lanes 0 and 1 of its warp.
__global__ void k_mg_outer(const MgArgs a, int first, int final)
{
    // one warp per system: lane q sums value q & 3 (||r||^2, then ||b||^2, of both fields) over every eighth block
    const int lane = threadIdx.x & 31, s = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (s >= a.nsys) return;   // uniform over the warp
    double rr = 0.0;
    for (int b = lane >> 2; b < a.B0; b += 8) rr += a.part64[((long long)s * a.B0 + b) * 4 + (lane & 3)];
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) rr += __shfl_xor_sync(0xffffffffu, rr, o);
    const double bb = __shfl_down_sync(0xffffffffu, rr, 2);
    const bool valid = lane < 2;
    const int f = lane, t = 2 * s + f;
    if (valid && first) {
        a.stop2[t] = a.rtol * a.rtol * bb;
        a.act_o[t] = 1;
        a.iters[t] = 0;
    }
    const bool conv = valid ? rr <= a.stop2[t] : true;
    if (final) {
        const unsigned other = __shfl_xor_sync(0xffffffffu, conv ? 1u : 0u, 1);
        const int it_other = __shfl_xor_sync(0xffffffffu, valid ? a.iters[t] : 0, 1);
        if (!valid) return;
        if (!conv) atomicOr(a.status, STATUS_NOCONV);
        if (f == 0) a.sys_iters[s] = (conv && other) ? max(a.iters[t], it_other) : a.max_iter + 1;
        return;
    }
    if (!valid) return;
    if (conv) a.act_o[t] = 0;
    a.act_i[t] = a.act_o[t];
    a.rr0[t] = (float)rr;
}

// Level-0 vectors of a system: z (the V-cycle's U), r (its F), p, q, d.
struct V0 {
    long long off, base;
    int W, H, mx, my;
};

__device__ __forceinline__ V0 v0(const MgArgs& a, int s)
{
    V0 v;
    v.mx = a.mx[0];
    v.my = a.my[0];
    v.W = v.mx + 2;
    v.H = v.my + 2;
    v.base = (long long)s * v.W * v.H;
    v.off = a.off[0] + v.base;
    return v;
}

// p = z + beta p with beta = rz_new / rz_old (first: p = z); rz slots by parity.
__global__ void __launch_bounds__(MG_THREADS) k_mg_pupdate(const MgArgs a, int first, int parity)
{
    const int s = blockIdx.y;
    if (!any_active(a, s)) return;
    if (parity < 0) parity = a.loop[1] & 1;   // inside a graph loop: the inner iteration counter
    const V0 v = v0(a, s);
    const int n = v.mx * v.my;
    float beta[2];
    const float2 rz2 = block_part_sums(a.part, s, a.T0);
#pragma unroll
    for (int f = 0; f < 2; ++f) {
        const float rz_new = f ? rz2.y : rz2.x;
        const float rz_old = a.rz[(2 * s + f) * 2 + (parity ^ 1)];
        beta[f] = (!first && a.act_i[2 * s + f] && rz_old > 0.f) ? rz_new / rz_old : 0.f;
        if (blockIdx.x == 0 && threadIdx.x == 0) a.rz[(2 * s + f) * 2 + parity] = rz_new;
    }
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const long long e = (long long)(1 + k / v.mx) * v.W + 1 + k % v.mx;
#pragma unroll
        for (int f = 0; f < 2; ++f) a.Pv[f][v.base + e] = a.Z[f][v.off + e] + beta[f] * a.Pv[f][v.base + e];
    }
}

// q = A p (level 0, single precision), (p, q) partials
__global__ void __launch_bounds__(MG_THREADS) k_mg_spmv(const MgArgs a)
{
    const int s = blockIdx.y;
    const V0 v = v0(a, s);
    const int n = v.mx * v.my;
    float t[2] = {0.f, 0.f};
    if (any_active(a, s))
        for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
            const long long e = (long long)(1 + k / v.mx) * v.W + 1 + k % v.mx;
            const long long c = v.off + e;
            const float d = a.D[c], cw = a.CX[c - 1], ce = a.CX[c], cs = a.CY[c - v.W], cn = a.CY[c];
#pragma unroll
            for (int f = 0; f < 2; ++f) {
                const float* p = a.Pv[f] + v.base;
                const float q = d * p[e] - cw * p[e - 1] - ce * p[e + 1] - cs * p[e - v.W] - cn * p[e + v.W];
                a.Qv[f][v.base + e] = q;
                t[f] += p[e] * q;
            }
        }
    block_sum4(t[0], t[1], 0.f, 0.f, a.part + ((long long)s * a.B0 + blockIdx.x) * 4);
}

// d += alpha p, r -= alpha q; (r, r) partials, to an array of their own: other blocks still read (p, q)'s.
__global__ void __launch_bounds__(MG_THREADS) k_mg_update(const MgArgs a, int parity)
{
    const int s = blockIdx.y;
    if (parity < 0) parity = a.loop[1] & 1;
    const V0 v = v0(a, s);
    const int n = v.mx * v.my;
    float t[2] = {0.f, 0.f};
    if (any_active(a, s)) {
        float alpha[2];
        const float2 pq2 = block_part_sums(a.part, s, a.B0);
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            const float pq = f ? pq2.y : pq2.x;
            const float rz = a.rz[(2 * s + f) * 2 + parity];
            alpha[f] = (a.act_i[2 * s + f] && pq > 0.f) ? rz / pq : 0.f;
        }
        for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
            const long long e = (long long)(1 + k / v.mx) * v.W + 1 + k % v.mx;
#pragma unroll
            for (int f = 0; f < 2; ++f) {
                a.Cv[f][v.base + e] += alpha[f] * a.Pv[f][v.base + e];
                const float r = a.F[f][v.off + e] - alpha[f] * a.Qv[f][v.base + e];
                a.F[f][v.off + e] = r;
                t[f] += r * r;
            }
        }
    }
    block_sum4(t[0], t[1], 0.f, 0.f, a.part_rr + ((long long)s * a.B0 + blockIdx.x) * 4);
}

// Loop control inside a graph: counter `which` (0 refinement sweeps, 1 inner iterations) counts this pass, and the
// while-node's condition becomes "some field still active (act_o for 0, act_i for 1) and fewer than cap
// passes". One block. For the inner iterations it first ends those of a field once ||r||^2 <= inner_tol^2
// ||r_0||^2 (or on a breakdown), from k_mg_update's partials.
__global__ void __launch_bounds__(MG_THREADS) k_mg_cond(const MgArgs a, cudaGraphConditionalHandle h, int which, int cap,
                                                        int body_kernels)
{
    int any = 0;
    if (which == 0) {
        for (int t = threadIdx.x; t < 2 * a.nsys; t += blockDim.x) any |= a.act_o[t];
    } else {
        const int lane = threadIdx.x & 31;
        for (int s = threadIdx.x >> 5; s < a.nsys; s += MG_THREADS / 32) {
            const float2 rr = warp_part_sums(a.part_rr, s, a.B0);
            const int t = 2 * s + lane;
            if (lane < 2 && a.act_i[t]) {
                a.iters[t] += 1;
                if ((lane ? rr.y : rr.x) > a.inner_tol * a.inner_tol * a.rr0[t]) any = 1;
                else a.act_i[t] = 0;
            }
        }
    }
    any = __syncthreads_or(any);
    if (threadIdx.x != 0) return;
    if (a.launches) *a.launches += body_kernels;   // the pass of the loop body that ends here
    const int c = a.loop[which] + 1;
    a.loop[which] = c;
    cudaGraphSetConditional(h, (any && c < cap) ? 1u : 0u);
}

// Start a loop: counter `which` to zero and the loop's condition to "some field active".
__global__ void k_mg_loop_reset(const MgArgs a, cudaGraphConditionalHandle h, int which)
{
    const int32_t* act = which == 0 ? a.act_o : a.act_i;
    int any = 0;
    for (int t = threadIdx.x; t < 2 * a.nsys; t += blockDim.x) any |= act[t];
    any = __syncthreads_or(any);
    if (threadIdx.x != 0) return;
    if (which == 0 && a.launches) *a.launches = 0;
    a.loop[which] = 0;
    cudaGraphSetConditional(h, any ? 1u : 0u);
}

// x += d (double precision) on every unknown of the fields still iterating
__global__ void __launch_bounds__(MG_THREADS) k_mg_xupdate(const MgArgs a)
{
    const int s = blockIdx.y;
    const SolveSys S = a.sys[s];
    const V0 v = v0(a, s);
    const int n = v.mx * v.my;
    const bool on[2] = {a.act_o[2 * s] != 0, a.act_o[2 * s + 1] != 0};
    if (!on[0] && !on[1]) return;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int ip = 1 + k % v.mx, jp = 1 + k / v.mx;
        const long long g = (long long)(S.j0 - 1 + jp) * a.nx + (S.i0 - 1 + ip);
        const long long e = (long long)jp * v.W + ip;
#pragma unroll
        for (int f = 0; f < 2; ++f)
            if (on[f]) a.x[f][g] += (double)a.Cv[f][v.base + e];
    }
}

int blocks_for(long long n)
{
    const long long b = (n + MG_THREADS * 4 - 1) / (MG_THREADS * 4);
    return (int)std::max<long long>(1, std::min<long long>(b, 64));
}

}  // namespace

// ---------------------------------------------------------------- host side

static int tiles(int m) { return (m + TILE - 1) / TILE; }

bool mg_levels(int mx, int my, MgArgs& a)
{
    if (mx < 1 || my < 1) return false;
    int L = 1;
    a.mx[0] = mx;
    a.my[0] = my;
    while (L < kMgMaxLevels && (a.mx[L - 1] & 1) && (a.my[L - 1] & 1) && a.mx[L - 1] >= 3 && a.my[L - 1] >= 3) {
        a.mx[L] = (a.mx[L - 1] - 1) / 2;
        a.my[L] = (a.my[L - 1] - 1) / 2;
        ++L;
    }
    a.levels = L;
    // the coarsest level is solved by sweeps; only worthwhile when it is small
    if ((long long)a.mx[L - 1] * a.my[L - 1] > 64) return false;
    a.tail = 1;   // level 0 always by the tile kernels
    while (a.tail < L - 1 && (long long)a.mx[a.tail] * a.my[a.tail] > 4096) ++a.tail;
    return L >= 2;
}

long long mg_layout(MgArgs& a, int nsys)
{
    long long off = 0;
    for (int l = 0; l < a.levels; ++l) {
        a.off[l] = off;
        off += (long long)nsys * (a.mx[l] + 2) * (a.my[l] + 2);
    }
    a.nsys = nsys;
    a.B0 = blocks_for((long long)a.mx[0] * a.my[0]);
    a.T0 = tiles(a.mx[0]) * tiles(a.my[0]);
    return off;
}

cudaError_t launch_mg_setup(const MgArgs& a, cudaStream_t s)
{
    const long long P0 = (long long)(a.mx[0] + 2) * (a.my[0] + 2);
    k_mg_coef0<<<dim3(blocks_for(P0), a.nsys), MG_THREADS, 0, s>>>(a);
    for (int l = 0; l + 1 < a.levels; ++l) {
        const long long P = (long long)(a.mx[l + 1] + 2) * (a.my[l + 1] + 2);
        k_mg_coarsen<<<dim3(blocks_for(P), a.nsys), MG_THREADS, 0, s>>>(a, l);
    }
    return cudaGetLastError();
}

// kernels one V-cycle launches
static int vcycle_kernels(const MgArgs& a) { return 2 * a.tail + 1; }

static cudaError_t vcycle(const MgArgs& a, cudaStream_t s)
{
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k_mg_down, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PreSmem))) != cudaSuccess)
        return e;
    if ((e = cudaFuncSetAttribute(k_mg_up, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PostSmem))) != cudaSuccess)
        return e;
    auto grid = [&](int l) { return dim3((unsigned)(tiles(a.mx[l]) * tiles(a.my[l])), (unsigned)a.nsys); };
    for (int l = 0; l < a.tail; ++l) k_mg_down<<<grid(l), MG_THREADS, sizeof(PreSmem), s>>>(a, l, tiles(a.mx[l]));
    // the limit is that of every shape, so that another thread's launch keeps it
    const size_t smem = tail_smem_bytes(a);
    if ((e = cudaFuncSetAttribute(k_mg_tail, cudaFuncAttributeMaxDynamicSharedMemorySize, TAIL_MAX_SMEM)) != cudaSuccess)
        return e;
    k_mg_tail<<<a.nsys, TAIL_THREADS, smem, s>>>(a);
    for (int l = a.tail - 1; l >= 0; --l)
        k_mg_up<<<grid(l), MG_THREADS, sizeof(PostSmem), s>>>(a, l, tiles(a.mx[l]));
    return cudaGetLastError();
}

// A condition handle of the graph that stream s is capturing into. The
// handle's default (1) applies only when the whole graph is launched, so a
// loop entered more than once per launch has its handle set by a kernel first.
static cudaError_t make_handle(cudaStream_t s, cudaGraphConditionalHandle* h)
{
    cudaStreamCaptureStatus st;
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamGetCaptureInfo(s, &st, nullptr, &g, nullptr, nullptr, nullptr);
    if (e != cudaSuccess) return e;
    if (st != cudaStreamCaptureStatusActive) return cudaErrorStreamCaptureImplicit;
    return cudaGraphConditionalHandleCreate(h, g, 1, cudaGraphCondAssignDefault);
}

// Add a while-node on handle h after the capture's current dependencies on
// stream s and start capturing its body on stream b.
static cudaError_t begin_while(cudaStream_t s, cudaStream_t b, cudaGraphConditionalHandle h, cudaGraphNode_t* node)
{
    cudaStreamCaptureStatus st;
    cudaGraph_t g = nullptr;
    const cudaGraphNode_t* deps = nullptr;
    size_t nd = 0;
    cudaError_t e = cudaStreamGetCaptureInfo(s, &st, nullptr, &g, &deps, nullptr, &nd);
    if (e != cudaSuccess) return e;
    if (st != cudaStreamCaptureStatusActive) return cudaErrorStreamCaptureImplicit;
    cudaGraphNodeParams p{};
    p.type = cudaGraphNodeTypeConditional;
    p.conditional.handle = h;
    p.conditional.type = cudaGraphCondTypeWhile;
    p.conditional.size = 1;
    if ((e = cudaGraphAddNode(node, g, deps, nullptr, nd, &p)) != cudaSuccess) return e;
    return cudaStreamBeginCaptureToGraph(b, p.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                         cudaStreamCaptureModeRelaxed);
}

// Close the body captured on b; s continues after the while-node.
static cudaError_t end_while(cudaStream_t s, cudaStream_t b, cudaGraphNode_t node)
{
    cudaGraph_t body = nullptr;
    cudaError_t e = cudaStreamEndCapture(b, &body);
    if (e != cudaSuccess) return e;
    return cudaStreamUpdateCaptureDependencies(s, &node, nullptr, 1, cudaStreamSetCaptureDependencies);
}

static cudaError_t mg_graph_body(const MgArgs& a, cudaStream_t s, cudaStream_t s2, cudaStream_t s3)
{
    const dim3 g0(a.B0, a.nsys);
    const int sc = (a.nsys + 3) / 4;   // k_mg_outer: a warp per system
    cudaError_t e;
    cudaGraphConditionalHandle ho, hi;
    cudaGraphNode_t no, ni;
    k_mg_res64<<<g0, MG_THREADS, 0, s>>>(a);
    k_mg_outer<<<sc, 128, 0, s>>>(a, 1, 0);
    if ((e = make_handle(s, &ho)) != cudaSuccess) return e;
    k_mg_loop_reset<<<1, MG_THREADS, 0, s>>>(a, ho, 0);
    if ((e = begin_while(s, s2, ho, &no)) != cudaSuccess) return e;
    // one refinement sweep: the inner PCG on A d = r, then x += d and the new residual
    if ((e = vcycle(a, s2)) != cudaSuccess) return e;
    if ((e = make_handle(s2, &hi)) != cudaSuccess) return e;
    k_mg_loop_reset<<<1, MG_THREADS, 0, s2>>>(a, hi, 1);
    k_mg_pupdate<<<g0, MG_THREADS, 0, s2>>>(a, 1, -1);
    if ((e = begin_while(s2, s3, hi, &ni)) != cudaSuccess) return e;
    k_mg_spmv<<<g0, MG_THREADS, 0, s3>>>(a);
    k_mg_update<<<g0, MG_THREADS, 0, s3>>>(a, -1);
    k_mg_cond<<<1, MG_THREADS, 0, s3>>>(a, hi, 1, a.inner, 4 + vcycle_kernels(a));
    if ((e = vcycle(a, s3)) != cudaSuccess) return e;
    k_mg_pupdate<<<g0, MG_THREADS, 0, s3>>>(a, 0, -1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = end_while(s2, s3, ni)) != cudaSuccess) return e;
    k_mg_xupdate<<<g0, MG_THREADS, 0, s2>>>(a);
    k_mg_res64<<<g0, MG_THREADS, 0, s2>>>(a);
    k_mg_outer<<<sc, 128, 0, s2>>>(a, 0, 0);
    k_mg_cond<<<1, MG_THREADS, 0, s2>>>(a, ho, 0, a.outer, 6 + vcycle_kernels(a));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = end_while(s, s2, no)) != cudaSuccess) return e;
    k_mg_outer<<<sc, 128, 0, s>>>(a, 0, 1);
    return cudaGetLastError();
}

// The solve, for a stream that is being captured: the refinement sweeps
// and the inner iterations are while-nodes whose condition kernels stop them
// once every field has converged (at most outer x inner passes), so a graph
// replay runs only the iterations the systems need.
cudaError_t launch_mg_solve_graph(const MgArgs& a, cudaStream_t s, cudaStream_t s2, cudaStream_t s3)
{
    const cudaError_t e = mg_graph_body(a, s, s2, s3);
    if (e != cudaSuccess) {
        // leave no body capture open: the caller ends (and discards) the main capture
        for (cudaStream_t b : {s3, s2}) {
            cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
            if (cudaStreamIsCapturing(b, &st) == cudaSuccess && st != cudaStreamCaptureStatusNone) {
                cudaGraph_t g = nullptr;
                cudaStreamEndCapture(b, &g);
                if (g) cudaGraphDestroy(g);
            }
        }
    }
    return e;
}

}  // namespace sdd
