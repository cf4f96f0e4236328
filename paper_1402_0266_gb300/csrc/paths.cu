// paths.cu -- the interface Monte Carlo path kernel and the per-node reduction.
//
// Each path solves dX = -(1/w) grad w dt + sqrt(2) dW (Eq. 7a with the
// Winslow coefficients of Eq. 6) from its node by Euler--Maruyama over the K
// sub-steps of one mesh step (Sec. 4), with dW = sqrt(dt) N(0,1), the drift
// interpolated bilinearly between the grid nodes, and a boundary test after
// every sub-step. A path that leaves scores the boundary data f, g at its exit
// point; a path that stays scores xi, eta of the start of the mesh step at its
// end point (Eq. 7b). The node's estimate is the mean over its paths (Sec. 4).
//
// Execution: a persistent grid; each warp repeatedly takes a task (one node,
// a contiguous range of its paths) from a counter, on its own. Each lane runs one path at
// a time; idle lanes take the task's next unstarted paths when some path of the
// warp reaches the end of the step or enough lanes are idle. In the paper's
// (plain) exit mode one Philox block supplies the normals of two consecutive
// sub-steps, so a warp advances its paths by sub-step pairs. Scores are summed per lane with
// compensation (single precision, shifted by the node's start coordinates),
// then per warp in double precision; the per-node reduction over tasks runs in
// a fixed order, so results do not depend on scheduling.
//
// Deferred scoring: when the fields of the step's start are still being
// computed beside the path kernel (pipelined mesh steps), a surviving path
// leaves its end point (and control-variate sums) in a record array instead,
// and so does a path that leaves by the plain test (the sub-step that crossed
// the boundary: scoring it here would hold its warp on the face-table loads);
// k_score_surv scores the records once the fields are final, then runs the
// per-node reduction.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "cluster.cuh"
#include "common.cuh"

namespace sdd {

namespace {

constexpr unsigned FULL = 0xffffffffu;

// Positions and both components of every bilinear field travel as float2 so
// that GB300's paired single-precision instructions (FFMA2, FADD2, FMUL2)
// handle x and y together.
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

struct Cell {
    float2 st;        // local coordinates (s, t) in [0, 1)
    uint32_t idx;     // row-major cell index (plus kCellBits in the kernels of one instance of at most kOneMaxCells cells)
};

// Cell of pos, strictly inside the unit square, and local coordinates. g = pos (n - 1) stays below n - 1: the
// largest single-precision pos below 1 is 1 - 2^-24, and (n - 1)(1 - 2^-24) lies more than half an ulp below
// n - 1 (or is the float below it, for a power of two). floor() through a directed add of 2^23:
// for 0 <= g < 2^23, (g + 2^23) rounded down is 2^23 + floor(g) exactly, and
// its bits are 0x4B000000 + floor(g). ONE (at most kOneMaxCells cells): the cell index by one exact
// multiply-add in single precision, 2^23 + j (nx - 1) + i, left in its float bits; the table
// pointers take the offset of those bits (rec2). Otherwise cell_bias removes the offset from the
// row-major cell index in 32-bit wrap-around arithmetic.
constexpr uint32_t kCellBits = 0x4B000000u;

template <bool ONE>
__device__ __forceinline__ Cell locate(const InstDev& I, float2 pos)
{
    const float2 g = __fmul2_rn(pos, f2(I.sx, I.sy));
    const float2 t = __fadd2_rd(g, f2(8388608.0f, 8388608.0f));
    const float2 fl = __fadd2_rn(t, f2(-8388608.0f, -8388608.0f));    // floor(g), exact
    Cell c;
    c.st = __ffma2_rn(fl, f2(-1.0f, -1.0f), g);                        // g - floor(g), exact
    c.idx = ONE ? __float_as_uint(__fmaf_rn(fl.y, I.sx, t.x))
                : __float_as_uint(t.y) * (uint32_t)(I.nx - 1) + __float_as_uint(t.x) - I.cell_bias;
    return c;
}

// The record of cell idx in a table of records.
template <bool ONE, typename T>
__device__ __forceinline__ const T* record(const T* base, uint32_t idx, int per_cell)
{
    const long long bytes = (long long)sizeof(T) * per_cell;
    return reinterpret_cast<const T*>(reinterpret_cast<const char*>(base) - (ONE ? bytes * (long long)kCellBits : 0) +
                                      bytes * (long long)idx);
}

template <bool ONE>
__device__ __forceinline__ const float4* rec2(const float4* base, uint32_t idx)
{
    return record<ONE>(base, idx, 2);
}

// A cell's two records in one 256-bit read-only load (records are 32-byte
// aligned): one L1 request per gather instead of two for the same sector.
__device__ __forceinline__ void load_cell(const float4* p, float4& lo, float4& hi)
{
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(lo.x), "=f"(lo.y), "=f"(lo.z), "=f"(lo.w), "=f"(hi.x), "=f"(hi.y), "=f"(hi.z), "=f"(hi.w)
        : "l"(p));
}

// Both components of a bilinear field from the cell's records
// lo = (a0u, a0v, a1u, a1v), hi = (a2u, a2v, a3u, a3v): (a0 + a1 s) + t (a2 + a3 s).
__device__ __forceinline__ float2 eval2(const float4& lo, const float4& hi, float2 st)
{
    const float2 ss = f2(st.x, st.x), tt = f2(st.y, st.y);
    const float2 r = __ffma2_rn(f2(lo.z, lo.w), ss, f2(lo.x, lo.y));
    const float2 q = __ffma2_rn(f2(hi.z, hi.w), ss, f2(hi.x, hi.y));
    return __ffma2_rn(q, tt, r);
}

// One Euler--Maruyama sub-step from pos with increment z = sqrt(2 dt) N(0,1)^2:
// pos + b(pos) dt + z, b bilinear from the cell's drift records.
__device__ __forceinline__ float2 em(const float4& lo, const float4& hi, float2 st, float2 pos, float2 dt2, float2 z)
{
    return __fadd2_rn(__ffma2_rn(eval2(lo, hi, st), dt2, pos), z);
}

// Strictly inside the unit square: x^2 < x and y^2 < y. Rounding keeps the order
// (x^2 and x are at least an ulp of x apart, or x^2 underflows below x). False for a NaN.
__device__ __forceinline__ bool inside2(float2 p)
{
    const float2 q = __fmul2_rn(p, p);
    return q.x < p.x && q.y < p.y;
}

// Face `face` at tangential coordinate s: the offset of its table (field 0;
// field 1 follows 2 ny + 2 nx entries later), the interval k and the fraction f.
__device__ __forceinline__ void face_interval(const InstDev& I, int face, float s, long long& off, int& k, float& f)
{
    const int n = (face < 2) ? I.ny : I.nx;
    off = 0;
    if (face >= 1) off += I.ny;
    if (face >= 2) off += I.ny;
    if (face >= 3) off += I.nx;
    const float g = s * (float)(n - 1);
    k = (int)floorf(g);
    k = max(0, min(k, n - 2));
    f = g - (float)k;
}

// Linear interpolation of face `face` of `field` at tangential coordinate s.
__device__ __forceinline__ float face_value(const InstDev& I, int field, int face, float s)
{
    long long off;
    int k;
    float f;
    face_interval(I, face, s, off, k, f);
    const float* v = I.faces32 + off + (long long)field * (2LL * I.ny + 2LL * I.nx);
    return fmaf(f, v[k + 1] - v[k], v[k]);
}

// The boundary crossing of the sub-step X_j = (x, y) -> X_{j+1} = (xn, yn):
// the segment is cut at the smallest crossing fraction over the violated
// faces, ties to the face listed first (left, right, bottom, top); t is the
// tangential coordinate of the crossing on that face.
__device__ __forceinline__ void exit_crossing(float x, float y, float xn, float yn, int& face, float& t)
{
    float best = 2.0f;
    int f = -1;
    if (xn <= 0.0f) { const float s = x / (x - xn); if (s < best) { best = s; f = 0; } }
    if (xn >= 1.0f) { const float s = (1.0f - x) / (xn - x); if (s < best) { best = s; f = 1; } }
    if (yn <= 0.0f) { const float s = y / (y - yn); if (s < best) { best = s; f = 2; } }
    if (yn >= 1.0f) { const float s = (1.0f - y) / (yn - y); if (s < best) { best = s; f = 3; } }
    if (f < 0) { f = 0; best = 0.0f; }  // only for a non-finite position
    float tt = (f < 2) ? fmaf(best, yn - y, y) : fmaf(best, xn - x, x);
    t = fminf(fmaxf(tt, 0.0f), 1.0f);
    face = f;
}

// Brownian-bridge test between two inside points: the half plane behind face
// k is touched with probability exp(-d0 d1 / dt) (sigma^2 = 2); the faces
// combine as 1 - prod (1 - p_k). On exit: the face of largest p_k, at the
// projection t of the sub-step midpoint. inv: 1 / dt.
__device__ __forceinline__ bool bridge_test(float x, float y, float xn, float yn, float inv, float u, int& face, float& t)
{
    const float d0[4] = {x, 1.0f - x, y, 1.0f - y};
    const float d1[4] = {xn, 1.0f - xn, yn, 1.0f - yn};
    float stay = 1.0f, pmax = -1.0f;
    int f = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float p = __expf(-d0[k] * d1[k] * inv);
        stay *= (1.0f - p);
        if (p > pmax) { pmax = p; f = k; }
    }
    if (!(u < 1.0f - stay)) return false;
    t = (f < 2) ? 0.5f * (y + yn) : 0.5f * (x + xn);
    t = fminf(fmaxf(t, 0.0f), 1.0f);
    face = f;
    return true;
}

// Distance of a point inside the square to the nearest face.
__device__ __forceinline__ float face_distance(float2 p)
{
    return fminf(fminf(p.x, 1.0f - p.x), fminf(p.y, 1.0f - p.y));
}

// The boundary data at tangential coordinate t of a face, and the point.
__device__ __forceinline__ void face_point(const InstDev& I, int face, float t, float& yxi, float& yeta, float& xe,
                                           float& ye)
{
    yxi = face_value(I, 0, face, t);
    yeta = face_value(I, 1, face, t);
    xe = (face == 0) ? 0.0f : (face == 1) ? 1.0f : t;
    ye = (face == 2) ? 0.0f : (face == 3) ? 1.0f : t;
}

// Exit through the boundary between X_j and X_{j+1}: the boundary data at the crossing.
__device__ __forceinline__ void plain_exit(const InstDev& I, float x, float y, float xn, float yn, int& face,
                                        float& yxi, float& yeta, float& xe, float& ye)
{
    float t;
    exit_crossing(x, y, xn, yn, face, t);
    face_point(I, face, t, yxi, yeta, xe, ye);
}

// 32 bytes through the non-coherent path as eight words.
__device__ __forceinline__ void load_words(const uint4* p, uint4& lo, uint4& hi)
{
    asm("ld.global.nc.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(lo.x), "=r"(lo.y), "=r"(lo.z), "=r"(lo.w), "=r"(hi.x), "=r"(hi.y), "=r"(hi.z), "=r"(hi.w)
        : "l"(p));
}

__device__ __forceinline__ float2 half2_to_float2(uint32_t u)
{
    __half2 h;
    memcpy(&h, &u, sizeof h);
    return __half22float2(h);
}

// Bilinear interpolation of four corner values (00, 10, 01, 11) at (s, t):
// ((1 - s) f00 + s f10) (1 - t) + ((1 - s) f01 + s f11) t, both components.
__device__ __forceinline__ float2 corners2(const uint4& r, float2 ss, float2 oms, float2 tt, float2 omt)
{
    const float2 r0 = __ffma2_rn(ss, half2_to_float2(r.y), __fmul2_rn(oms, half2_to_float2(r.x)));
    const float2 r1 = __ffma2_rn(ss, half2_to_float2(r.w), __fmul2_rn(oms, half2_to_float2(r.z)));
    return __ffma2_rn(tt, r1, __fmul2_rn(omt, r0));
}

// Control variate: the model gradients of xi and eta at the cell's point
// (slice q), gxi = (d/dx, d/dy) of the xi model, geta of the eta model.
template <bool ONE>
__device__ __forceinline__ void cv_eval(const InstDev& I, const Cell& c, int q, float2& gxi, float2& geta)
{
    const uint4* r = record<ONE>(I.cvcoef + 2 * ((size_t)q * (size_t)(I.nx - 1) * (size_t)(I.ny - 1)), c.idx, 2);
    uint4 gx, ge;
    load_words(r, gx, ge);
    const float2 ss = f2(c.st.x, c.st.x), tt = f2(c.st.y, c.st.y);
    const float2 oms = f2(1.f - c.st.x, 1.f - c.st.x), omt = f2(1.f - c.st.y, 1.f - c.st.y);
    gxi = corners2(gx, ss, oms, tt, omt);
    geta = corners2(ge, ss, oms, tt, omt);
}

// Control variate of one value per cell: (d/dx, d/dy) of xi, then of eta, on
// the cell holding the point, in one 128-bit read-only load.
template <bool ONE>
__device__ __forceinline__ void cv_cell(const InstDev& I, const Cell& c, float2& gxi, float2& geta)
{
    const float4 g = __ldg(record<ONE>(I.cvcell, c.idx, 1));
    gxi = f2(g.x, g.y);
    geta = f2(g.z, g.w);
}

// The gradients times the sub-step's increment z = sqrt(2 dt) N(0,1)^2, added to
// the running sums (acc_xi, acc_eta hold the x and y parts separately).
__device__ __forceinline__ void cv_acc(float2 gxi, float2 geta, float2 z, float2& acc_xi, float2& acc_eta)
{
    acc_xi = __ffma2_rn(gxi, z, acc_xi);
    acc_eta = __ffma2_rn(geta, z, acc_eta);
}

// Compensated sums of a lane's scores and their squares.
struct Acc {
    float s, cs, q, cq;
    __device__ __forceinline__ void add(float v)
    {
        float y1 = v - cs;
        float t1 = s + y1;
        cs = (t1 - s) - y1;
        s = t1;
        const float v2 = v * v;
        float y2 = v2 - cq;
        float t2 = q + y2;
        cq = (t2 - q) - y2;
        q = t2;
    }
    __device__ __forceinline__ double sum() const { return (double)s - (double)cs; }
    __device__ __forceinline__ double sumsq() const { return (double)q - (double)cq; }
};

// Sums of four values over the warp, value lane & 3 in each lane: the first two
// steps halve the values held, so a lane makes 6 double-precision additions where
// four butterflies make 20. A warp's addition takes 16 cycles of its SM's two
// double-precision lanes: with 32-path tasks the sums were a sixth of an estimate.
__device__ __forceinline__ double warp_sum4(double v0, double v1, double v2, double v3)
{
    const bool h2 = threadIdx.x & 2, h1 = threadIdx.x & 1;
    const double a = (h2 ? v2 : v0) + __shfl_xor_sync(FULL, h2 ? v0 : v2, 2);
    const double b = (h2 ? v3 : v1) + __shfl_xor_sync(FULL, h2 ? v1 : v3, 2);
    double t = (h1 ? b : a) + __shfl_xor_sync(FULL, h1 ? a : b, 1);
#pragma unroll
    for (int off = 4; off < 32; off <<= 1) t += __shfl_xor_sync(FULL, t, off);
    return t;
}

// Sum of nonnegative 64-bit integers below 2^58 over the warp.
__device__ __forceinline__ long long warp_sum_ll(long long v)
{
    const unsigned lo = __reduce_add_sync(FULL, (unsigned)(v & 0xffff));
    const unsigned mid = __reduce_add_sync(FULL, (unsigned)((v >> 16) & 0xffff));
    const unsigned hi = __reduce_add_sync(FULL, (unsigned)(v >> 32));
    return (long long)lo + ((long long)mid << 16) + ((long long)hi << 32);
}

// A lane's counts over a task (each nonnegative, below 2^31).
__device__ __forceinline__ long long warp_sum_int(int v)
{
    return (long long)__reduce_add_sync(FULL, (unsigned)v & 0xffffu) +
           ((long long)__reduce_add_sync(FULL, (unsigned)v >> 16) << 16);
}

// The sums of a task: lanes 0 to 3 hold the sums of Partial's order.
__device__ __forceinline__ void put_partial(Partial* p, double sum, long long exits, long long steps)
{
    const int lane = threadIdx.x & 31;
    if (lane < 4) reinterpret_cast<double*>(p)[lane] = sum;
    if (lane == 0) {
        p->exits = exits;
        p->steps = steps;
    }
}

// Deferred scoring: a path's record in the survivor buffer, one float2 (two
// with CV, the second holding the control-variate sums): a survivor leaves its
// end point (x, y), x > 0; a path that left by the plain test the crossing of
// its last sub-step with the boundary, (-1 - face, t) with t the tangential
// coordinate on that face (the face data are interpolated there later); a path
// scored in the kernel (bridge exits) REC_SKIP. No point inside the square has
// a negative x, so the sign tells the kinds apart.
constexpr float REC_SKIP = -8.0f;

template <bool CV>
__device__ __forceinline__ void put_record(void* surv, long long i, float2 r, float cxi, float ceta)
{
    float2* q = static_cast<float2*>(surv) + (CV ? 2 * i : i);
    q[0] = r;
    if (CV) q[1] = f2(cxi, ceta);
}

// The record of a plain exit through the sub-step (x, y) -> (xn, yn).
__device__ __forceinline__ float2 exit_record(float x, float y, float xn, float yn)
{
    int face;
    float t;
    exit_crossing(x, y, xn, yn, face, t);
    return f2(-1.0f - (float)face, t);
}

// Idle lanes that call for a refill. A lane whose path left the domain waits until this many have, or until some
// path of the warp reaches the end of the step; then all that ended are scored and replaced together (the crossing,
// the boundary data and the sums take more instructions than a pass). 601 nodes of a 194 x 131 grid, 45 sub-steps:
// 297 us with each exit scored in its pass, now 277; 4 lanes or 18 instead of 8 are up to 1 % slower.
constexpr int REFILL_MIN = 8;

// The draws of one path: Philox block d of path p, its first two rounds reduced
// to what changes with d. With counter (p, node, d, step), round 1 multiplies p
// and d, round 2 multiplies a word of d and the node and one of p and the step:
// of the two rounds' four products only the two of d are formed per draw.
struct PathWords {
    uint32_t u, v, w;
};

__device__ __forceinline__ PathWords path_words(uint32_t path, uint32_t step, const PhiloxKeys& K)
{
    const unsigned long long p0 = (unsigned long long)0xD2511F53u * path;
    const uint32_t z1 = (uint32_t)(p0 >> 32) ^ step ^ K.rk[1];
    const unsigned long long p1 = (unsigned long long)0xCD9E8D57u * z1;
    return PathWords{(uint32_t)(p1 >> 32) ^ K.rk[2], (uint32_t)p1, (uint32_t)p0 ^ K.rk[3]};
}

// Rounds 1 and 2 of block d: nodek is the node word xor round 1's first key.
__device__ __forceinline__ uint4 draw_begin(const PathWords& q, uint32_t nodek, uint32_t d)
{
    const unsigned long long p1 = (unsigned long long)0xCD9E8D57u * d;
    const unsigned long long p0 = (unsigned long long)0xD2511F53u * ((uint32_t)(p1 >> 32) ^ nodek);
    return make_uint4(q.u ^ (uint32_t)p1, q.v, (uint32_t)(p0 >> 32) ^ q.w, (uint32_t)p0);
}

// Tile of the zero map that holds p (shared-memory offset): floor(T p) per axis,
// T = kZmapTiles, by one fused multiply-add rounded down at 2, whose unit is
// 2^-22: the float bits are 0x40000000 + tile, and with the pitch T = 4 q - 1 the
// two offsets cancel (0x40000000 * 4 q = 0 mod 2^32). Positions outside the
// square land on any byte of the map: their lanes' results are not used.
__device__ __forceinline__ uint32_t zmap_offset(float2 p)
{
    static_assert(kZmapTiles % 4 == 3, "the pitch cancels the offset of the float bits");
    constexpr float scale = kZmapTiles * (1.0f / 4194304.0f);
    const float2 t = __ffma2_rd(p, f2(scale, scale), f2(2.0f, 2.0f));
    return min(__float_as_uint(t.y) * (uint32_t)kZmapTiles + __float_as_uint(t.x), (uint32_t)kZmapBytes - 1u);
}

// MODE 0: the paper's test, sub-step pairs; MODE 1: with the bridge test;
// MODE 2: as MODE 0 when K is even (every pair has both sub-steps).
// CVM: 0 no control variate; otherwise subtract sum_j G(s_j, X_j) . sqrt(2) dW_j
// from both scores, G from node values interpolated bilinearly in time slices
// (1, cv_eval) or one value per cell (2, cv_cell).
// VAR_MULTI: each task's instance from the instance table (batches); VAR_ONE: a
// single instance whose tables are kernel parameters, with its zero map if it has one; VAR_BIG: the same for
// grids of more than kOneMaxCells cells, with an integer cell index. Its blocks stay at paths_min_blocks an SM (32 warps, 24
// with a control variate): where L2 does not hold the records, more warps spread the gathers over more of them. 4,774
// nodes x 8,000 paths x 100 sub-steps at 4097^2: drift everywhere 17.3 ms (19.6 with 40 warps, 17.3 in the batch
// kernel), with cell gradients 39.2 (45.7 with 32 warps, 39.1); the ring 11.7 (10.9 with 40, 17.0 in the batch kernel, which has
// no map) and 22.3 with cell gradients (38.2).
// DEFER: survivors and plain exits leave records for k_score_surv.
constexpr int VAR_MULTI = 0, VAR_ONE = 1, VAR_BIG = 2;
int variant(const PathArgs& a)
{
    return !a.single ? VAR_MULTI : (long long)(a.one.nx - 1) * (a.one.ny - 1) > kOneMaxCells ? VAR_BIG : VAR_ONE;
}
constexpr int kOneMaxBlock = 256;
constexpr int paths_max_block(int cvm, int var) { return cvm ? kCvMaxBlock : var != VAR_MULTI ? kOneMaxBlock : 512; }
constexpr int paths_min_blocks(int mode, int cvm, int var)
{
    return cvm ? (var == VAR_ONE ? 4 : 3) : var == VAR_MULTI ? 2 : var == VAR_BIG || mode == 1 ? 4 : 5;
}

// A lane's sums over a task, in shared memory: they change once per path, and the
// registers they would hold through every sub-step are worth more there.
// Word k of thread i at [k][i]: no bank conflicts.
template <int BLOCK, bool SCORES>
struct LaneSums {
    int exits[BLOCK], steps[BLOCK];
    float acc[SCORES ? 8 : 1][SCORES ? BLOCK : 1];

    __device__ __forceinline__ void clear()
    {
        exits[threadIdx.x] = steps[threadIdx.x] = 0;
        if (SCORES)
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[k][threadIdx.x] = 0.f;
    }
    __device__ __forceinline__ Acc get(int f) const
    {
        return Acc{acc[4 * f][threadIdx.x], acc[4 * f + 1][threadIdx.x], acc[4 * f + 2][threadIdx.x],
                   acc[4 * f + 3][threadIdx.x]};
    }
    __device__ __forceinline__ void add(int f, float v)
    {
        Acc x = get(f);
        x.add(v);
        acc[4 * f][threadIdx.x] = x.s;
        acc[4 * f + 1][threadIdx.x] = x.cs;
        acc[4 * f + 2][threadIdx.x] = x.q;
        acc[4 * f + 3][threadIdx.x] = x.cq;
    }
};

// How a lane's path left, until the warp scores it: the sub-step's two ends (a bridge exit: the second holds
// the tangential coordinate), sub-steps taken and face, the control-variate sums.
template <int BLOCK, bool CV>
struct LaneExits {
    float2 p0[BLOCK], p1[BLOCK];
    int info[BLOCK];
    float cv[CV ? 2 : 1][CV ? BLOCK : 1];

    __device__ __forceinline__ void put(float2 a, float2 b, int i, float cxi, float ceta)
    {
        p0[threadIdx.x] = a;
        p1[threadIdx.x] = b;
        info[threadIdx.x] = i;
        if (CV) {
            cv[0][threadIdx.x] = cxi;
            cv[CV ? 1 : 0][threadIdx.x] = ceta;
        }
    }
    __device__ __forceinline__ void get(float2& a, float2& b, int& i, float& cxi, float& ceta) const
    {
        a = p0[threadIdx.x];
        b = p1[threadIdx.x];
        i = info[threadIdx.x];
        if (CV) {
            cxi = cv[0][threadIdx.x];
            ceta = cv[CV ? 1 : 0][threadIdx.x];
        }
    }
};

// Node data read again where a path starts or ends rather than held in registers
// (volatile: the compiler would otherwise keep the first read).
__device__ __forceinline__ float2 node_start(const NodeDev* nd)
{
    float2 v;
    asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(&nd->xf));
    return v;
}

__device__ __forceinline__ long long node_records(const NodeDev* nd)
{
    long long v;
    asm volatile("ld.global.nc.s64 %0, [%1];" : "=l"(v) : "l"(&nd->rec0));
    return v;
}

__device__ __forceinline__ unsigned lanes_below()
{
    unsigned m;
    asm volatile("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// The tasks of one warp. MAP: the drift is read through the zero map zsm: a lane in
// an unmarked tile has zero drift (it reads nothing; with the bridge test or time slices the all-zero
// record), and a warp without a lane in a marked tile only adds the increment.
//
// What bounds it (GB300, two sub-steps of a warp's 32 paths = one pass): a gather of 32 records that
// miss L1 takes 34 cycles of the SM whatever its width (32 bytes per cycle from L2), so a pass with
// drift everywhere costs 64 or more (2.7e11 path-steps/s at 2049^2, L1 data pipe 80 % busy); a pass
// without drift is 119 instructions, 45 cycles, bound by issue slots and the FMA pipe's wide
// multiplies (4.5e11). Hence the branch around the gather, the draws' shared first rounds, the sums
// in shared memory and 48 registers (40 warps per SM; 32 and 48 warps are within 2 %), a draw made
// where it is used rather than a pass ahead (fewer registers and moves; the other warps cover the
// gathers), and bookkeeping only when a path ends. On a 2049^2 ring (28,609 nodes x 2e4 paths x 100
// sub-steps): 144 ms per launch and 75 instructions per path-step, against 179 ms and 92 for the kernel that tested
// every path in every pass and redirected gathers without skipping them.
template <int MODE, bool RECORD, int CVM, int VAR, bool DEFER, bool MAP>
__device__ __forceinline__ void walk_tasks(const PathArgs& a, const uint8_t* zsm,
                                           LaneSums<paths_max_block(CVM, VAR), !DEFER || MODE == 1>& sums,
                                           LaneExits<paths_max_block(CVM, VAR), CVM != 0>& left)
{
    constexpr int LEFT = 7;   // a path that left by the plain test; otherwise the face of a bridge exit
    constexpr bool CV = CVM != 0;
    constexpr bool CVT = CVM == 1;   // node values in time slices
    constexpr bool ONE = VAR == VAR_ONE;
    constexpr bool PAIRS = MODE != 1;
    constexpr bool ACC = !DEFER || MODE == 1;   // some scores are summed here
    const uint32_t step = a.step_ptr ? *a.step_ptr : a.step_index;
    const int K = a.K;
    const int P = PAIRS ? (K + 1) >> 1 : K;   // passes of a path: sub-step pairs, or sub-steps
    const float2 dt2 = f2(a.dt, a.dt);
    // records that lanes without a cell read: the all-zero one, the first cell's
    constexpr bool READ_ZERO = MODE == 1 || CVT;
    [[maybe_unused]] const uint32_t zcell = (ONE ? kCellBits : 0u) + a.zcell;
    const uint32_t cell0 = ONE ? kCellBits : 0u;

    // Each warp takes the next task as soon as its last one is done (no wait
    // for the block's other warps); tasks go node by node, so warps started
    // together share the node's neighbourhood in L1.
    for (;;) {
        int tq = 0;
        if (lanes_below() == 0) tq = atomicAdd(a.queue, 1);
        const int t = __shfl_sync(FULL, tq, 0);
        if (t >= a.ntasks) return;

        const Task task = a.tasks[t];
        if (a.node_mask && !a.node_mask[task.node]) continue;   // not a key point this step
        const NodeDev* const nd = a.nodes + task.node;
        // a single instance's tables come from the kernel parameters (no registers held for them)
        InstDev Iloc;
        if (VAR == VAR_MULTI) Iloc = a.inst[nd->inst];
        const InstDev& I = VAR != VAR_MULTI ? a.one : Iloc;
        const uint32_t nodek = nd->ctr ^ a.keys.rk[0];
        const uint32_t end = (uint32_t)task.path0 + (uint32_t)task.npaths;
        uint32_t next = (uint32_t)task.path0, path = 0;
        bool alive = false, ended = false;   // ended: a path that left, to be scored
        PathWords pw{};
        float2 pos = f2(0.5f, 0.5f);
        int m = 0;        // the path's pass: its draw
        float dm = 0.f;   // bridge test: the position's distance to the boundary
        float2 cvx = f2(0.f, 0.f), cve = f2(0.f, 0.f);  // control-variate sums of the path
        int cvq = 0, cvn = CVT ? a.cv_bound[1] : 0;      // slice of the current sub-step, start of the next
        sums.clear();

        float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;   // the cell record read last
        // One sub-step from p with increment z, for lanes with ok (the others' results are not used,
        // and their p may lie anywhere): p + b(p) dt + z.
        auto advance = [&](float2 p, float2 z, bool ok, bool count, int j) -> float2 {
            bool g = ok;
            if (MAP) g = zsm[zmap_offset(p)] != 0 && ok;
            float2 q = __fadd2_rn(p, z);
            if (CV || !MAP || __any_sync(FULL, g)) {
                Cell c = locate<ONE>(I, p);
                if (CV) c.idx = ok ? c.idx : cell0;
                // lanes without drift or path do not read: beside lanes that miss L1 their hit on the zero record costs
                // the warp three cycles, and unread it saves one each (257^2 steps 8053 -> 7853 us, a batch of 16
                // grids 1441 -> 1360, 1025^2 with field cells 2864 -> 2717). Bound by instructions, the bridge test and
                // the time slices read the zero record instead of clearing eight registers (732 against 744 us, 133 against 136).
                if (MAP && READ_ZERO) {
                    load_cell(rec2<ONE>(I.bcoef, g ? c.idx : zcell), lo, hi);
                } else {
                    if (MAP && !g) lo = hi = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (g) load_cell(rec2<ONE>(I.bcoef, c.idx), lo, hi);
                }
                if (CV) {
                    // the model at X_j; the sub-step counts only when the path takes it
                    const float2 zt = count ? z : f2(0.f, 0.f);
                    float2 gx, ge;
                    if (CVT) {
                        if (count && j >= cvn) cvn = a.cv_bound[++cvq + 1];
                        cv_eval<ONE>(I, c, cvq, gx, ge);
                    } else {
                        cv_cell<ONE>(I, c, gx, ge);
                    }
                    cv_acc(gx, ge, zt, cvx, cve);
                }
                q = em(lo, hi, c.st, p, dt2, z);
            }
            return q;
        };

        int k = 0;   // passes until a path of the warp ends with the step
        for (;;) {
            if (k == 0) {
                // the lanes without a path take the task's next ones, in lane order
                const unsigned idle = __ballot_sync(FULL, !alive);
                if (next < end) {
                    const uint32_t cand = next + __popc(idle & lanes_below());
                    next += __popc(idle);
                    if (!alive && cand < end) {
                        alive = true;
                        path = cand;
                        pw = path_words(path, step, a.keys);
                        pos = node_start(nd);
                        if (!PAIRS) dm = face_distance(pos);
                        m = 0;
                        if (CV) cvx = cve = f2(0.f, 0.f);
                        if (CVT) {
                            cvq = 0;
                            cvn = a.cv_bound[1];
                        }
                    }
                } else if (idle == FULL) {
                    break;
                }
                k = __reduce_min_sync(FULL, alive ? P - m : 0x7fffffff);
            }
            // one pass: the sub-step pair (bridge mode: the sub-step) of draw m
            uint4 r = draw_begin(pw, nodek, (uint32_t)m);
            philox_rounds_rk<2, 10>(r, a.keys);
            float2 zA, zB = f2(0.f, 0.f);
            if (PAIRS) box_muller2(r, a.bm_scale, zA, zB);
            else box_muller(r.x, r.y, a.bm_scale, zA.x, zA.y);
            const float2 pa = advance(pos, zA, alive, alive, PAIRS ? 2 * m : m);
            const bool inA = inside2(pa);
            float2 pn = pa;   // where the pass ends
            bool out;
            int face = LEFT;
            float tb = 0.f;
            if (PAIRS) {
                // an odd K: the last pair has no sub-step B
                const bool haveB = MODE == 2 || 2 * m + 1 < K;
                const float2 pb = advance(pa, zB, alive && inA, alive && inA && haveB, 2 * m + 1);
                if (haveB) pn = pb;
                out = alive && !(inA && (!haveB || inside2(pb)));
            } else {
                out = alive && !inA;
                const float dm1 = face_distance(pa);
                if (alive && inA && dm * dm1 < a.bridge_cut &&
                    bridge_test(pos.x, pos.y, pa.x, pa.y, a.inv_dt, uniform_pos(r.z), face, tb))
                    out = true;
                dm = dm1;
            }
            --k;
            if (__any_sync(FULL, out)) {
                // the paths that left wait for the next refill: now if enough lanes are idle, or all
                if (out) {
                    const float2 p0 = PAIRS && inA ? pa : pos, p1 = PAIRS && inA ? pn : pa;
                    const int taken = !PAIRS ? m + 1 : inA ? 2 * m + 2 : 2 * m + 1;
                    left.put(p0, !PAIRS && face != LEFT ? f2(tb, 0.f) : p1, taken | face << 28, cvx.x + cvx.y, cve.x + cve.y);
                    alive = false;
                    ended = true;
                }
                const int idle = 32 - __popc(__ballot_sync(FULL, alive));
                if (idle == 32 || (idle >= REFILL_MIN && next < end)) k = 0;
            }
            if (k == 0 && (ended || (alive && m == P - 1))) {
                const long long ri = DEFER || RECORD ? node_records(nd) + (long long)path : 0;
                int taken = K, code = -1;
                bool later = DEFER;   // scored by k_score_surv once the fields are final
                float yxi = 0.f, yeta = 0.f, xe = 0.f, ye = 0.f, cxi = 0.f, ceta = 0.f;
                if (CV) {
                    cxi = cvx.x + cvx.y;
                    ceta = cve.x + cve.y;
                }
                if (ended) {
                    ++sums.exits[threadIdx.x];
                    float2 p0, p1;
                    int info;
                    left.get(p0, p1, info, cxi, ceta);
                    taken = info & 0x0fffffff;
                    face = info >> 28;
                    if (MODE == 1 && face != LEFT) {
                        // a bridge exit is scored here; its record holds the skip mark
                        face_point(I, face, p1.x, yxi, yeta, xe, ye);
                        code = face + 4;
                        later = false;
                        if (DEFER) put_record<CV>(a.surv, ri, f2(REC_SKIP, 0.f), cxi, ceta);
                    } else if (DEFER) {
                        put_record<CV>(a.surv, ri, exit_record(p0.x, p0.y, p1.x, p1.y), cxi, ceta);
                    } else {
                        plain_exit(I, p0.x, p0.y, p1.x, p1.y, code, yxi, yeta, xe, ye);
                    }
                } else if (DEFER) {
                    put_record<CV>(a.surv, ri, pn, cxi, ceta);
                } else {
                    // survived the mesh step: xi, eta of its start at the end point
                    const Cell c = locate<ONE>(I, pn);
                    float4 f0, f1;
                    load_cell(rec2<ONE>(I.fcoef, c.idx), f0, f1);
                    const float2 v = eval2(f0, f1, c.st);
                    yxi = v.x;
                    yeta = v.y;
                    xe = pn.x;
                    ye = pn.y;
                }
                sums.steps[threadIdx.x] += taken;
                if (ACC && !later) {
                    if (CV) {
                        yxi -= cxi;
                        yeta -= ceta;
                    }
                    const float2 c = node_start(nd);
                    sums.add(0, yxi - c.x);
                    sums.add(1, yeta - c.y);
                }
                if (RECORD) {
                    if (a.rec.steps) a.rec.steps[ri] = taken;
                    if (a.rec.code) a.rec.code[ri] = code;
                    if (a.rec.score_xi) a.rec.score_xi[ri] = yxi;
                    if (a.rec.score_eta) a.rec.score_eta[ri] = yeta;
                    if (a.rec.x_end) a.rec.x_end[ri] = xe;
                    if (a.rec.y_end) a.rec.y_end[ri] = ye;
                }
                alive = ended = false;
            }
            pos = pn;
            ++m;
        }

        double tot = 0.0;
        if (ACC) {
            const Acc ax = sums.get(0), ae = sums.get(1);
            tot = warp_sum4(ax.sum(), ax.sumsq(), ae.sum(), ae.sumsq());
        }
        put_partial(a.partials + t, tot, warp_sum_int(sums.exits[threadIdx.x]), warp_sum_int(sums.steps[threadIdx.x]));
    }
}

template <int MODE, bool RECORD, int CVM, int VAR, bool DEFER>
__global__ void __launch_bounds__(paths_max_block(CVM, VAR), paths_min_blocks(MODE, CVM, VAR))
    k_paths(const PathArgs a)
{
    __shared__ LaneSums<paths_max_block(CVM, VAR), !DEFER || MODE == 1> sums;
    __shared__ LaneExits<paths_max_block(CVM, VAR), CVM != 0> left;
    if (VAR != VAR_MULTI && a.zmap) {
        // stage the zero map, and leave it unused where nearly every tile is marked
        extern __shared__ __align__(16) uint8_t zsm[];
        __shared__ int marked;
        if (threadIdx.x == 0) marked = 0;
        __syncthreads();
        int mine = 0;
        for (int k = threadIdx.x; k < kZmapBytes / 16; k += blockDim.x) {
            const uint4 v = reinterpret_cast<const uint4*>(a.zmap)[k];
            reinterpret_cast<uint4*>(zsm)[k] = v;
            mine += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);   // marks are ones
        }
        atomicAdd(&marked, mine);
        __syncthreads();
        if (marked < kZmapTiles * kZmapTiles * 7 / 8) {
            walk_tasks<MODE, RECORD, CVM, VAR, DEFER, true>(a, zsm, sums, left);
            return;
        }
    }
    walk_tasks<MODE, RECORD, CVM, VAR, DEFER, false>(a, nullptr, sums, left);
}

// Exponential time-stepping (exit_mode 2), the alternative integrator Sec. 4
// names: sub-step j of a path has length tau_j = -dt ln u with u = (2^23 - m)
// 2^-23 from word 3 of the block (path, node, j, step), cut at the end of the
// mesh step (and after 4K + 16 sub-steps); normals from words 0, 1 scaled by
// sqrt(2 tau_j); the plain test, then the Brownian-bridge test over tau_j with
// the uniform of word 2.
//
// The paths of a warp end at different sub-steps, one or two of them in nearly every pass: a lane whose
// path is done waits, so that the scores, the sums and the new paths (as many instructions as a
// pass) are made for EXP_REFILL lanes at a time. Bound by issue slots. 253 nodes x 8000 paths at K = 20:
// 406 us with a path's end handled in its pass and ten rounds a draw, now 372.
constexpr int EXP_REFILL = 6;

template <bool RECORD>
__global__ void __launch_bounds__(512, 2) k_paths_exp(const PathArgs a)
{
    __shared__ LaneSums<512, true> sums;
    const uint32_t step = a.step_ptr ? *a.step_ptr : a.step_index;
    const int cap = 4 * a.K + 16;
    const float T = a.horizon;
    const float ln2dt = a.dt * 0.69314718055994530942f;
    constexpr int SURVIVED = -1, LEFT = -2;   // otherwise 4 + the face of a bridge exit
    for (;;) {
        int tq = 0;
        if (lanes_below() == 0) tq = atomicAdd(a.queue, 1);
        const int t = __shfl_sync(FULL, tq, 0);
        if (t >= a.ntasks) return;
        const Task task = a.tasks[t];
        if (a.node_mask && !a.node_mask[task.node]) continue;
        const NodeDev* const nd = a.nodes + task.node;
        const InstDev I = a.inst[nd->inst];
        const uint32_t nodek = nd->ctr ^ a.keys.rk[0];
        const uint32_t end = (uint32_t)task.path0 + (uint32_t)task.npaths;
        uint32_t next = (uint32_t)task.path0, path = 0;
        bool alive = false, ended = false;
        PathWords pw{};
        float2 pos = f2(0.5f, 0.5f), pe = f2(0.f, 0.f);   // pe: the point past an exit, or (t, -) of a bridge exit
        int j = 0, code = SURVIVED;
        float tm = 0.f, dm = 0.f;   // time, distance to the boundary
        sums.clear();
        bool refill = true;
        for (;;) {
            if (refill) {
                if (ended) {
                    ended = false;
                    const long long ri = a.surv || RECORD ? node_records(nd) + (long long)path : 0;
                    float yxi = 0.f, yeta = 0.f, xe = 0.f, ye = 0.f;
                    bool later = a.surv != nullptr;   // scored by k_score_surv once the fields are final
                    if (code != SURVIVED) ++sums.exits[threadIdx.x];
                    if (code >= 4) {
                        face_point(I, code - 4, pe.x, yxi, yeta, xe, ye);
                        if (a.surv) put_record<false>(a.surv, ri, f2(REC_SKIP, 0.f), 0.f, 0.f);
                        later = false;
                    } else if (a.surv) {
                        put_record<false>(a.surv, ri, code == LEFT ? exit_record(pos.x, pos.y, pe.x, pe.y) : pos, 0.f, 0.f);
                    } else if (code == LEFT) {
                        plain_exit(I, pos.x, pos.y, pe.x, pe.y, code, yxi, yeta, xe, ye);
                    } else {
                        const Cell cf = locate<false>(I, pos);
                        float4 f0, f1;
                        load_cell(rec2<false>(I.fcoef, cf.idx), f0, f1);
                        const float2 v = eval2(f0, f1, cf.st);
                        yxi = v.x;
                        yeta = v.y;
                        xe = pos.x;
                        ye = pos.y;
                    }
                    sums.steps[threadIdx.x] += j;
                    if (!later) {
                        const float2 c = node_start(nd);
                        sums.add(0, yxi - c.x);
                        sums.add(1, yeta - c.y);
                    }
                    if (RECORD) {
                        if (a.rec.steps) a.rec.steps[ri] = j;
                        if (a.rec.code) a.rec.code[ri] = code;
                        if (a.rec.score_xi) a.rec.score_xi[ri] = yxi;
                        if (a.rec.score_eta) a.rec.score_eta[ri] = yeta;
                        if (a.rec.x_end) a.rec.x_end[ri] = xe;
                        if (a.rec.y_end) a.rec.y_end[ri] = ye;
                    }
                }
                // the lanes without a path take the task's next ones, in lane order
                const unsigned idle = __ballot_sync(FULL, !alive);
                if (next < end) {
                    const uint32_t cand = next + __popc(idle & lanes_below());
                    next += __popc(idle);
                    if (!alive && cand < end) {
                        alive = true;
                        path = cand;
                        pw = path_words(path, step, a.keys);
                        pos = node_start(nd);
                        dm = face_distance(pos);
                        j = 0;
                        tm = 0.f;
                    }
                } else if (idle == FULL) {
                    break;
                }
            }
            if (alive) {
                uint4 r = draw_begin(pw, nodek, (uint32_t)j);
                philox_rounds_rk<2, 10>(r, a.keys);
                const float u3 = 2.0f - __uint_as_float(0x3F800000u | (r.w & 0x7FFFFFu));
                float tau = -ln2dt * __log2f(u3);
                bool last = false;
                if (tm + tau >= T || j + 1 >= cap) {
                    tau = T - tm;
                    last = true;
                }
                float2 z;
                box_muller(r.x, r.y, -2.77258872223978123767f * tau, z.x, z.y);   // -4 ln 2 tau: sqrt(2 tau) N(0,1)
                const Cell c = locate<false>(I, pos);
                float4 g0, g1;
                load_cell(rec2<false>(I.bcoef, c.idx), g0, g1);
                const float2 pn = em(g0, g1, c.st, pos, f2(tau, tau), z);
                ++j;
                if (!inside2(pn)) {
                    code = LEFT;
                    ended = true;
                    pe = pn;
                } else {
                    const float dm1 = face_distance(pn);
                    if (dm * dm1 < 18.0f * tau &&
                        bridge_test(pos.x, pos.y, pn.x, pn.y, 1.0f / tau, uniform_pos(r.z), code, pe.x)) {
                        code += 4;
                        ended = true;
                    } else {
                        pos = pn;
                        dm = dm1;
                        tm += tau;
                        code = SURVIVED;
                        ended = last;
                    }
                }
                alive = !ended;
            }
            const int idle = 32 - __popc(__ballot_sync(FULL, alive));
            refill = idle == 32 || (idle >= EXP_REFILL && next < end);
        }
        const Acc ax = sums.get(0), ae = sums.get(1);
        const double tot = warp_sum4(ax.sum(), ax.sumsq(), ae.sum(), ae.sumsq());
        put_partial(a.partials + t, tot, warp_sum_int(sums.exits[threadIdx.x]), warp_sum_int(sums.steps[threadIdx.x]));
    }
}

__device__ __forceinline__ double face_value64(const InstDev& I, int field, int face, double s)
{
    const int n = (face < 2) ? I.ny : I.nx;
    long long off = (long long)field * (2LL * I.ny + 2LL * I.nx);
    if (face >= 1) off += I.ny;
    if (face >= 2) off += I.ny;
    if (face >= 3) off += I.nx;
    const double* v = I.faces64 + off;
    const double g = s * (double)(n - 1);
    int k = (int)floor(g);
    k = max(0, min(k, n - 2));
    const double f = g - (double)k;
    return (1.0 - f) * v[k] + f * v[k + 1];
}

// A node that no path was walked for (left to the interface fill, or on the boundary): its outputs by one warp.
__device__ bool pathless_node(const FinalArgs& a, int node, const NodeDev& nd, int lane)
{
    const bool filled = a.node_mask && !a.node_mask[node];
    if (!filled && nd.ntasks != 0) return false;
    const OutDev o = a.out_table ? a.out_table[nd.inst] : a.out0;
    const int k = nd.local;
    double vx = 0.0, ve = 0.0;
    if (!filled) {
        // a node on the boundary: its Dirichlet value, every path exits at time 0
        const InstDev I = a.inst[nd.inst];
        int face;
        double tg;
        if (nd.x <= 0.0) { face = 0; tg = nd.y; }
        else if (nd.x >= 1.0) { face = 1; tg = nd.y; }
        else if (nd.y <= 0.0) { face = 2; tg = nd.x; }
        else { face = 3; tg = nd.x; }
        vx = face_value64(I, 0, face, tg);
        ve = face_value64(I, 1, face, tg);
        for (int p = lane; p < nd.n_paths; p += 32) {
            const long long ri = nd.rec0 + p;
            if (a.rec.steps) a.rec.steps[ri] = 0;
            if (a.rec.code) a.rec.code[ri] = face;
            if (a.rec.score_xi) a.rec.score_xi[ri] = (float)vx;
            if (a.rec.score_eta) a.rec.score_eta[ri] = (float)ve;
            if (a.rec.x_end) a.rec.x_end[ri] = nd.xf;
            if (a.rec.y_end) a.rec.y_end[ri] = nd.yf;
        }
    }
    if (lane == 0) {
        if (o.mean_xi) o.mean_xi[k] = vx;
        if (o.mean_eta) o.mean_eta[k] = ve;
        if (o.se_xi) o.se_xi[k] = 0.0;
        if (o.se_eta) o.se_eta[k] = 0.0;
        if (o.n_exit) o.n_exit[k] = filled ? 0 : nd.n_paths;
        if (o.path_steps) o.path_steps[k] = 0;
    }
    return true;
}

// Thread t of T: compensated sums of the node's task partials t, t + T, ...
__device__ __forceinline__ void task_sums(const FinalArgs& a, const NodeDev& nd, int t, int T, double (&v)[4],
                                          long long& ex, long long& st)
{
    double c[4] = {0, 0, 0, 0};
    ex = st = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = 0.0;
    for (int k = t; k < nd.ntasks; k += T) {
        const Partial p = a.partials[nd.task0 + k];
        const double in[4] = {p.s_xi, p.q_xi, p.s_eta, p.q_eta};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (k == t) {
                v[q] = in[q];
                continue;
            }
            const double y = in[q] - c[q];
            const double tt = v[q] + y;
            c[q] = (tt - v[q]) - y;
            v[q] = tt;
        }
        ex += p.exits;
        st += p.steps;
    }
    if (T < nd.ntasks)
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] -= c[q];
}

// The node's mean and standard error s / sqrt(N), s^2 = (Q - S^2 / N) / (N - 1) of the shifted scores,
// by one warp with sum lane & 3 in each lane: lane 0 for xi, lane 2 for eta.
__device__ __forceinline__ void node_outputs(const FinalArgs& a, const NodeDev& nd, int lane, double tot, long long ex,
                                             long long st)
{
    const OutDev o = a.out_table ? a.out_table[nd.inst] : a.out0;
    const int k = nd.local;
    const double sq = __shfl_down_sync(FULL, tot, 1);   // lane 0: Q of xi, lane 2: Q of eta
    if (lane == 0 || lane == 2) {
        const double N = (double)nd.n_paths;
        const double m = tot / N;
        const double var = nd.n_paths > 1 ? fmax(0.0, (sq - tot * m) * reciprocal(N - 1.0)) : 0.0;
        double* const mean = lane ? o.mean_eta : o.mean_xi;
        double* const se = lane ? o.se_eta : o.se_xi;
        if (mean) mean[k] = (double)(lane ? nd.yf : nd.xf) + m;
        if (se) se[k] = sqrt(var * reciprocal(N));
    }
    if (lane == 0) {
        if (o.n_exit) o.n_exit[k] = ex;
        if (o.path_steps) o.path_steps[k] = st;
    }
}

// What a warp or a block contributes to a node.
struct NodeSums {
    double v[4];
    long long ex, st;
};

__device__ __forceinline__ void put_sums(NodeSums* p, int lane, double v, long long ex, long long st)
{
    if (lane < 4) p->v[lane] = v;
    if (lane == 0) {
        p->ex = ex;
        p->st = st;
    }
}

// Sums of n contributions by one warp, in a fixed order: sum lane & 3 in each lane, the counts in all.
__device__ __forceinline__ double join_sums(const NodeSums* p, int n, int lane, long long& ex, long long& st)
{
    double v = 0.0;
    ex = st = 0;
    for (int g = lane >> 2; g < n; g += 8) v += p[g].v[lane & 3];
    for (int off = 4; off < 32 && off < 4 * n; off <<= 1) v += __shfl_xor_sync(FULL, v, off);
    for (int g = 0; g < n; ++g) {
        ex += p[g].ex;
        st += p[g].st;
    }
    return v;
}

constexpr int FINAL_WARPS = 8;

// One node by `warps` warps (a block; one: a warp of a two-warp block). A node's task partials are a
// chain of loads and of double-precision additions on lanes that hold two of them an SM cycle: one warp a node took
// 16 us for 253 nodes of 8,000 paths, four take 9.
__global__ void __launch_bounds__(FINAL_WARPS * 32) k_finalize(const FinalArgs a, int warps)
{
    __shared__ NodeSums part[FINAL_WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int node = warps == 1 ? blockIdx.x * (int)(blockDim.x >> 5) + warp : blockIdx.x;
    if (node >= a.nnodes) return;
    const NodeDev nd = a.nodes[node];
    if (nd.ntasks == 0 || (a.node_mask && !a.node_mask[node])) {
        if (warps == 1 || warp == 0) pathless_node(a, node, nd, lane);
        return;   // uniform over the node's warps
    }
    double v[4];
    long long ex, st;
    task_sums(a, nd, warps == 1 ? lane : (int)threadIdx.x, 32 * warps, v, ex, st);
    double tot = warp_sum4(v[0], v[1], v[2], v[3]);
    ex = warp_sum_ll(ex);
    st = warp_sum_ll(st);
    if (warps > 1) {
        put_sums(part + warp, lane, tot, ex, st);
        __syncthreads();
        if (warp != 0) return;
        tot = join_sums(part, warps, lane, ex, st);
    }
    node_outputs(a, nd, lane, tot, ex, st);
}

// Scores of the paths that survived a mesh step, once the fields of the step's
// start are final (the estimate of the next mesh step runs beside the
// subdomain solve that produces them), then the node's reduction. A cluster of C blocks of T threads per node: the
// node's paths end in one neighbourhood, so a block's gathers share L1; thread k of the cluster's C T takes paths
// k, k + C T, ... SCORE_BATCH at a time (records, then gathers, in flight
// together) and sums xi and eta at the end points minus the paths'
// control-variate sums; task partials are dealt to the cluster's threads as well. Each block leaves its sums
// with block 0, whose first warp writes the outputs. The next batch's records are read while the
// current batch's gathers are in flight. T = 256 threads at 64 registers puts four blocks on an SM (many nodes: one
// wave for up to four per SM); with no more nodes than SMs, four blocks per node make one wave of them. (One block
// of 1024 threads per node left half the SMs idle on a 41 x 41 grid's 77 nodes, and the task partials went
// through one warp: 26.6 us, now 16.9.)
constexpr int SCORE_BATCH = 2;
constexpr int SCORE_THREADS = 256;
constexpr int SCORE_MAX_CLUSTER = 4;

template <bool CV>
__global__ void __launch_bounds__(SCORE_THREADS, 4) k_score_surv(const ScoreArgs a)
{
    __shared__ double task_v[4][SCORE_THREADS];
    __shared__ long long task_n[2][SCORE_THREADS];
    __shared__ NodeSums part[SCORE_THREADS / 32], blocks[SCORE_MAX_CLUSTER];
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int node = blockIdx.x / C;
    const NodeDev& nd = a.nodes[node];
    if (nd.ntasks == 0 || (a.fin.node_mask && !a.fin.node_mask[node])) {
        // a boundary node or one left to the interface fill: no paths to score
        if (warp == 0 && rank == 0) pathless_node(a.fin, node, nd, lane);
        return;   // uniform over the cluster
    }
    // a block's shared memory may be written by the others of its cluster once it has started: every block arrives
    // here, and waits for all before the first remote store (the scoring lies between, so the wait is short)
    if (C > 1) cl.barrier_arrive();
    const InstDev I = a.inst[nd.inst];
    const float x0 = nd.xf, y0 = nd.yf;
    const int first = rank * SCORE_THREADS + threadIdx.x, threads = C * SCORE_THREADS, end = nd.n_paths;
    Acc ax{0.f, 0.f, 0.f, 0.f}, ae{0.f, 0.f, 0.f, 0.f};
    // the records of the batch that starts at path p0 (past the end: the skip mark)
    auto load_batch = [&](int p0, float2 (&r)[SCORE_BATCH], float2 (&cvs)[SCORE_BATCH]) {
#pragma unroll
        for (int u = 0; u < SCORE_BATCH; ++u) {
            const int p = p0 + u * threads;
            r[u] = f2(REC_SKIP, 0.f);
            cvs[u] = f2(0.f, 0.f);
            if (p < end) {
                const long long si = nd.rec0 + p;
                const float2* q = static_cast<const float2*>(a.surv) + (CV ? 2 * si : si);
                r[u] = q[0];
                if (CV) cvs[u] = q[1];
            }
        }
    };
    float2 r[SCORE_BATCH];
    float2 cvs[SCORE_BATCH];
    load_batch(first, r, cvs);
    {
        // this thread's share of the task partials, kept in shared memory over the scoring
        double v[4];
        long long ex, st;
        task_sums(a.fin, nd, first, threads, v, ex, st);
#pragma unroll
        for (int q = 0; q < 4; ++q) task_v[q][threadIdx.x] = v[q];
        task_n[0][threadIdx.x] = ex;
        task_n[1][threadIdx.x] = st;
    }
    for (int p0 = first; p0 < end; p0 += SCORE_BATCH * threads) {
        // one round of loads for the batch: a survivor gathers the field record at its
        // end point, a plain exit the face data on both sides of its crossing
        // (f0 = xi[k], xi[k + 1], eta[k], eta[k + 1]; st.x the fraction)
        float4 f0[SCORE_BATCH], f1[SCORE_BATCH];
        float2 st[SCORE_BATCH];
#pragma unroll
        for (int u = 0; u < SCORE_BATCH; ++u) {
            if (r[u].x >= 0.f) {
                const Cell c = locate<false>(I, r[u]);
                load_cell(rec2<false>(I.fcoef, c.idx), f0[u], f1[u]);
                st[u] = c.st;
            } else if (r[u].x != REC_SKIP) {
                int k;
                float f;
                long long off;
                const int face = (int)(-1.0f - r[u].x);
                face_interval(I, face, r[u].y, off, k, f);
                const float* v0 = I.faces32 + off + k;
                const float* v1 = v0 + (2LL * I.ny + 2LL * I.nx);
                f0[u] = make_float4(v0[0], v0[1], v1[0], v1[1]);
                st[u] = f2(f, 0.f);
            }
        }
        // the next batch's records while this batch's gathers are in flight
        float2 rn[SCORE_BATCH];
        float2 cn[SCORE_BATCH];
        load_batch(p0 + SCORE_BATCH * threads, rn, cn);
#pragma unroll
        for (int u = 0; u < SCORE_BATCH; ++u) {
            if (r[u].x == REC_SKIP) continue;   // scored in the path kernel, or past the end
            float yxi, yeta;
            if (r[u].x >= 0.f) {
                const float2 v = eval2(f0[u], f1[u], st[u]);
                yxi = v.x;
                yeta = v.y;
            } else {
                // left the domain in the sub-step (x0, y0) -> (x1, y1): the boundary data there,
                // as face_value interpolates it
                yxi = fmaf(st[u].x, f0[u].y - f0[u].x, f0[u].x);
                yeta = fmaf(st[u].x, f0[u].w - f0[u].z, f0[u].z);
            }
            ax.add(yxi - cvs[u].x - x0);
            ae.add(yeta - cvs[u].y - y0);
        }
#pragma unroll
        for (int u = 0; u < SCORE_BATCH; ++u) {
            r[u] = rn[u];
            cvs[u] = cn[u];
        }
    }
    double tot = warp_sum4(ax.sum() + task_v[0][threadIdx.x], ax.sumsq() + task_v[1][threadIdx.x],
                           ae.sum() + task_v[2][threadIdx.x], ae.sumsq() + task_v[3][threadIdx.x]);
    long long ex = warp_sum_ll(task_n[0][threadIdx.x]), st = warp_sum_ll(task_n[1][threadIdx.x]);
    put_sums(part + warp, lane, tot, ex, st);
    __syncthreads();
    if (warp == 0) tot = join_sums(part, SCORE_THREADS / 32, lane, ex, st);
    if (C > 1) {
        cl.barrier_wait();
        if (warp == 0) put_sums(cl.map_shared_rank(blocks, 0) + rank, lane, tot, ex, st);
        cl.sync();
        if (rank == 0 && warp == 0) tot = join_sums(blocks, C, lane, ex, st);
    }
    if (rank == 0 && warp == 0) node_outputs(a.fin, nd, lane, tot, ex, st);
}

__global__ void k_rng_draw(uint64_t seed, const uint32_t* __restrict__ ctrs, long long count,
                           uint32_t* __restrict__ words, float* __restrict__ normals)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= count) return;
    const uint4 c = make_uint4(ctrs[4 * i], ctrs[4 * i + 1], ctrs[4 * i + 2], ctrs[4 * i + 3]);
    const uint4 r = philox4x32_10(c, (uint32_t)seed, (uint32_t)(seed >> 32));
    words[4 * i + 0] = r.x;
    words[4 * i + 1] = r.y;
    words[4 * i + 2] = r.z;
    words[4 * i + 3] = r.w;
    if (normals) {
        const float scale = -1.38629436111989061883f;  // -2 ln 2: unit variance
        float z0, z1, z2, z3;
        box_muller(r.x, r.y, scale, z0, z1);
        box_muller(r.z, r.w, scale, z2, z3);
        normals[4 * i + 0] = z0;
        normals[4 * i + 1] = z1;
        normals[4 * i + 2] = z2;
        normals[4 * i + 3] = z3;
    }
}

template <int MODE, int CVM, int VAR>
const void* pick_out(bool record, bool defer)
{
    if (defer) return (const void*)k_paths<MODE, false, CVM, VAR, true>;
    return record ? (const void*)k_paths<MODE, true, CVM, VAR, false> : (const void*)k_paths<MODE, false, CVM, VAR, false>;
}

template <int CVM, int VAR>
const void* pick_mode(int mode, bool record, bool defer)
{
    if (mode == 0) return pick_out<0, CVM, VAR>(record, defer);
    if (mode == 2) return pick_out<2, CVM, VAR>(record, defer);
    return pick_out<1, CVM, VAR>(record, defer);
}

template <int VAR>
const void* pick_var(int mode, bool record, int cvm, bool defer)
{
    if (cvm == 2) return pick_mode<2, VAR>(mode, record, defer);
    return cvm ? pick_mode<1, VAR>(mode, record, defer) : pick_mode<0, VAR>(mode, record, defer);
}

// cvm: 0 no control variate, 1 node values in time slices, 2 one value per cell
const void* pick(int mode, bool record, int cvm, int var, bool defer)
{
    if (mode == 3) return record ? (const void*)k_paths_exp<true> : (const void*)k_paths_exp<false>;
    if (var == VAR_ONE) return pick_var<VAR_ONE>(mode, record, cvm, defer);
    if (var == VAR_BIG) return pick_var<VAR_BIG>(mode, record, cvm, defer);
    return pick_var<VAR_MULTI>(mode, record, cvm, defer);
}

int kernel_mode(int exit_mode, int K)
{
    if (exit_mode == 2) return 3;   // exponential time-stepping
    return exit_mode == 1 ? 1 : ((K & 1) == 0 ? 2 : 0);
}

}  // namespace

int path_kernel_max_block(int exit_mode, int cvm, bool single)
{
    return exit_mode == 2 ? 512 : paths_max_block(cvm, single ? VAR_ONE : VAR_MULTI);
}

int path_kernel_blocks_per_sm(int exit_mode, bool record, int block, int cvm, const PathArgs* a)
{
    int n = 0;
    // the even-K kernel has the same footprint class; size the grid for the larger of the two
    const int mode = exit_mode == 2 ? 3 : exit_mode == 1 ? 1 : 0;
    const size_t smem = a && a->zmap && mode != 3 ? kZmapBytes : 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &n, pick(mode, record, cvm, a ? variant(*a) : VAR_MULTI, a && a->surv), block, smem) != cudaSuccess)
        return 1;
    if (a && variant(*a) == VAR_BIG) n = std::min(n, paths_min_blocks(mode, cvm, VAR_BIG));
    return n > 0 ? n : 1;
}

cudaError_t launch_paths(const PathArgs& a, int exit_mode, bool record, int grid, int block, cudaStream_t s, int cvm)
{
    const int mode = kernel_mode(exit_mode, a.K);
    const size_t smem = a.zmap && mode != 3 ? kZmapBytes : 0;
    void* args[] = {(void*)&a};
    return cudaLaunchKernel(pick(mode, record, cvm, variant(a), a.surv != nullptr), dim3((unsigned)grid),
                            dim3((unsigned)block), args, smem, s);
}

cudaError_t launch_score_surv(const ScoreArgs& a, bool cv, cudaStream_t s)
{
    if (a.nnodes <= 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int C = a.nnodes <= sms ? SCORE_MAX_CLUSTER : 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.nnodes * C));
    cfg.blockDim = dim3(SCORE_THREADS);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cv ? cudaLaunchKernelEx(&cfg, k_score_surv<true>, a) : cudaLaunchKernelEx(&cfg, k_score_surv<false>, a);
}

cudaError_t launch_finalize(const FinalArgs& a, long long ntasks, cudaStream_t s)
{
    if (a.nnodes <= 0) return cudaSuccess;
    // two of a node's task partials per thread on average
    int warps = 1;
    while (warps < FINAL_WARPS && 64LL * warps * a.nnodes < ntasks) warps *= 2;
    // blocks of a few warps: their double-precision sums spread over the SMs
    const int per_block = warps == 1 ? 2 : 1;
    k_finalize<<<(unsigned)((a.nnodes + per_block - 1) / per_block), 32 * std::max(2, warps), 0, s>>>(a, warps);
    return cudaGetLastError();
}

cudaError_t launch_rng_draw(uint64_t seed, const uint32_t* ctrs, long long count, uint32_t* words, float* normals,
                            cudaStream_t s)
{
    if (count <= 0) return cudaSuccess;
    const int block = 256;
    k_rng_draw<<<(unsigned)((count + block - 1) / block), block, 0, s>>>(seed, ctrs, count, words, normals);
    return cudaGetLastError();
}

}  // namespace sdd
