// Hybrid coarse-to-fine update of Sec. 3.3 (Algorithm 1) and the exact grid
// k-nearest-neighbour search it rests on.
//
// Grid: the cube anchored at the per-axis minimum `lo` of a point set, side
// = the largest per-axis extent, split into n^3 cells of side h = side / n.
// Cell of p: floor((p - lo) / h) per axis in fp32 round-to-nearest, clamped
// to [0, n-1] for members of the set; id = (iz n + iy) n + ix.
//
// Voxel reduction: (id, index) pairs are radix-sorted (stable, so a voxel's
// points stay in input order); each run of equal ids becomes one point
// whose parameters are the run's means, one warp per voxel with lanes over
// the parameters, compensated fp32 sums in ascending input index.
//
// kNN: d2 = (dx dx + dy dy) + dz dz in fp32 round-to-nearest, ties by lower
// index.  The reference points lie in cell order as {x, y, z, index} (a
// counting sort: the order inside a cell is arbitrary, and the result does
// not depend on it), with a dense cell-start table, so the points of a run of
// consecutive cells are a contiguous slice.  A search visits cubic shells of
// cells around the query's cell; shell r is (2r+1)^2 rows along x (a whole row
// where |dy| or |dz| is r, else the row's two end cells).  Once shell r is
// done every unvisited point lies beyond a face of the visited cube of
// cells, so the search stops when the K-th best d2 is below the squared
// distance to the nearest such face (less a relative slack for the
// roundings of d2 and an absolute one for the cell coordinates), or when
// every cell has been seen.  Three kernels, each taking the queries the one
// before leaves open:
//   - one thread per query (knn_thread_kernel): the query's list in registers,
//     a few shells, rows beyond the K-th best skipped; queries in cell order
//     where there is one, so that a warp's lanes walk the same rows;
//   - one warp per query (knn_kernel) on a grid 8 times coarser, built only
//     when a query is left open: lane j holds the j-th best so far, one row per
//     lane; runs of up to 32 points are walked by their lanes side by side,
//     longer ones by the whole warp;
//   - an exhaustive scan, one block per query (neighbours across a wide
//     empty region).
// Sets too small for the first kernel, lists above its 16 entries and grids
// too large for a cell table (binary search over the sorted ids) start with a
// warp per query.
//
// Outlier removal: per point, the population standard deviation of its K
// neighbour distances, fp32 sums in neighbour order; survivors are
// compacted in order.  Generation: one warp per survivor averages its K
// nearest survivors' parameters (compensated fp32 sums in neighbour order); the same
// kernel, from attribute 3 on, moves parameters between frames.
#include <cfloat>

#include "pbr_internal.cuh"

namespace pbr {

constexpr int BBOX_PARTS = 608; // partial boxes of the first reduction pass

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int BBOX_THREADS = 256;

// Cell coordinate of p along one axis.  Members of the set are clamped into
// [0, n-1]; queries into [-n, 2n-1], which only moves a far query's cell
// towards the grid and so keeps every point of a cell at Chebyshev cell
// distance d > 0 more than (d - 1) h away from the query.
__device__ __forceinline__ int cell_coord(float p, float lo, float h, int n, bool member)
{
    if (h == 0.0f) return 0;
    float t = __fdiv_rn(__fsub_rn(p, lo), h);
    t = fminf(fmaxf(t, -1.0e9f), 1.0e9f); // keeps the conversion in range
    const int c = (int)floorf(t);
    return member ? min(max(c, 0), n - 1) : min(max(c, -n), 2 * n - 1);
}

__device__ __forceinline__ float sq_dist(float ax, float ay, float az, float bx, float by,
                                         float bz)
{
    const float dx = __fsub_rn(bx, ax), dy = __fsub_rn(by, ay), dz = __fsub_rn(bz, az);
    return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

// ------------------------------------------------------------------ grid
__global__ void __launch_bounds__(BBOX_THREADS)
bbox_partial_kernel(const float *__restrict__ pos, int64_t n, float *__restrict__ part)
{
    float mn[3] = {FLT_MAX, FLT_MAX, FLT_MAX}, mx[3] = {-FLT_MAX, -FLT_MAX, -FLT_MAX};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float v = pos[3 * i + a];
            mn[a] = fminf(mn[a], v);
            mx[a] = fmaxf(mx[a], v);
        }
    }
    __shared__ float s_v[6][BBOX_THREADS / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        for (int o = 16; o > 0; o >>= 1) {
            mn[a] = fminf(mn[a], __shfl_xor_sync(FULL, mn[a], o));
            mx[a] = fmaxf(mx[a], __shfl_xor_sync(FULL, mx[a], o));
        }
        if (lane == 0) {
            s_v[a][w] = mn[a];
            s_v[3 + a][w] = mx[a];
        }
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        const int a = threadIdx.x;
        float r = s_v[a][0];
        for (int j = 1; j < BBOX_THREADS / 32; ++j)
            r = a < 3 ? fminf(r, s_v[a][j]) : fmaxf(r, s_v[a][j]);
        part[6 * blockIdx.x + a] = r;
    }
}

// One block: the box of the partial boxes (minima and maxima, so the order
// does not matter) and the grid over it.  A single thread walking the 608
// partial boxes took 43 us, more than any other kernel of a small search.
__global__ void __launch_bounds__(BBOX_THREADS)
grid_params_kernel(const float *__restrict__ part, int n_parts, int n_cells, GridParams *gp,
                   int n_coarse, GridParams *coarse)
{
    __shared__ float s_v[6][BBOX_THREADS / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int a = 0; a < 6; ++a) {
        float v = a < 3 ? FLT_MAX : -FLT_MAX;
        for (int b = threadIdx.x; b < n_parts; b += BBOX_THREADS)
            v = a < 3 ? fminf(v, part[6 * b + a]) : fmaxf(v, part[6 * b + a]);
        for (int o = 16; o > 0; o >>= 1) {
            const float t = __shfl_xor_sync(FULL, v, o);
            v = a < 3 ? fminf(v, t) : fmaxf(v, t);
        }
        if (lane == 0) s_v[a][w] = v;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    float lo[3], hi[3];
    for (int a = 0; a < 3; ++a) {
        lo[a] = s_v[a][0];
        hi[a] = s_v[3 + a][0];
        for (int j = 1; j < BBOX_THREADS / 32; ++j) {
            lo[a] = fminf(lo[a], s_v[a][j]);
            hi[a] = fmaxf(hi[a], s_v[3 + a][j]);
        }
    }
    float side = 0.0f, amax = 0.0f;
    for (int a = 0; a < 3; ++a) {
        side = fmaxf(side, __fsub_rn(hi[a], lo[a]));
        amax = fmaxf(amax, fmaxf(fabsf(lo[a]), fabsf(hi[a])));
    }
    for (int level = 0; level < 2; ++level) {
        GridParams *p = level ? coarse : gp;
        const int n = level ? n_coarse : n_cells;
        if (!p) continue;
        for (int a = 0; a < 3; ++a) p->lo[a] = lo[a];
        p->n = n;
        p->h = __fdiv_rn(side, (float)n);
        // a coordinate's cell can be off across a boundary by the rounding of
        // (p - lo) / h: a few ulps of the coordinates' magnitude
        p->slack = 4.0e-6f * (side + amax);
    }
}

__device__ __forceinline__ uint32_t cell_id(const GridParams &g, float x, float y, float z)
{
    const int ix = cell_coord(x, g.lo[0], g.h, g.n, true);
    const int iy = cell_coord(y, g.lo[1], g.h, g.n, true);
    const int iz = cell_coord(z, g.lo[2], g.h, g.n, true);
    return ((uint32_t)iz * (uint32_t)g.n + (uint32_t)iy) * (uint32_t)g.n + (uint32_t)ix;
}

__global__ void cell_ids_kernel(const float *__restrict__ pos, int64_t n,
                                const GridParams *__restrict__ gp, uint32_t *__restrict__ keys,
                                uint32_t *__restrict__ vals)
{
    const GridParams g = *gp;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        keys[i] = cell_id(g, pos[3 * i], pos[3 * i + 1], pos[3 * i + 2]);
        vals[i] = (uint32_t)i;
    }
}

// Points in cell order by counting: points per cell into table[cell + 1],
// the exclusive scan of those turns table[cell + 1] into the first slot of
// `cell`, and the scatter's atomics move it past its last point, which is
// the first slot of cell + 1: table[c] ends as the start of cell c.
// gate: when set, the kernels do nothing while *gate is 0.
__global__ void cell_hist_kernel(const float *__restrict__ pos, int64_t n,
                                 const GridParams *__restrict__ gp, uint32_t *__restrict__ ids,
                                 uint32_t *__restrict__ table, const uint32_t *gate)
{
    if (gate && *gate == 0) return;
    const GridParams g = *gp;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t c = cell_id(g, pos[3 * i], pos[3 * i + 1], pos[3 * i + 2]);
        ids[i] = c;
        atomicAdd(table + 1 + c, 1u);
    }
}

__global__ void cell_scatter_kernel(const float *__restrict__ pos, int64_t n,
                                    const uint32_t *__restrict__ ids, uint32_t *__restrict__ table,
                                    float4 *__restrict__ pts, const uint32_t *gate)
{
    if (gate && *gate == 0) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        pts[atomicAdd(table + 1 + ids[i], 1u)] =
            make_float4(pos[3 * i], pos[3 * i + 1], pos[3 * i + 2], __uint_as_float((uint32_t)i));
}

// Exclusive scan of p[0..n) in place by one block, for tables small enough
// (GATED_CELLS) that three launches would cost more.
__global__ void __launch_bounds__(1024) gated_scan_kernel(uint32_t *p, int n, const uint32_t *gate)
{
    if (gate && *gate == 0) return;
    __shared__ uint32_t s_w[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t run = 0;
    for (int base = 0; base < n; base += 4096) {
        const int i = base + 4 * (int)threadIdx.x;
        uint32_t v[4], sum = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = i + k < n ? p[i + k] : 0u;
            sum += v[k];
        }
        uint32_t inc = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(FULL, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) s_w[w] = inc;
        __syncthreads();
        if (w == 0) {
            uint32_t x = s_w[lane];
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(FULL, x, o);
                if (lane >= o) x += t;
            }
            s_w[lane] = x;
        }
        __syncthreads();
        uint32_t at = run + inc - sum + (w > 0 ? s_w[w - 1] : 0u);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (i + k < n) p[i + k] = at;
            at += v[k];
        }
        run += s_w[31];
        __syncthreads();
    }
}

// Points in the order of a sorted (id, index) list (grids without a table).
__global__ void gather_points_kernel(const float *__restrict__ pos, const uint32_t *__restrict__ idx,
                                     int64_t n, float4 *__restrict__ pts)
{
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n;
         j += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t i = idx[j];
        pts[j] = make_float4(pos[3 * (size_t)i], pos[3 * (size_t)i + 1], pos[3 * (size_t)i + 2],
                             __uint_as_float(i));
    }
}

// -------------------------------------------------------- voxel runs
__global__ void run_flags_kernel(const uint32_t *__restrict__ keys, int64_t n,
                                 uint32_t *__restrict__ flags)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        flags[i] = (i == 0 || keys[i] != keys[i - 1]) ? 1u : 0u;
}

// After the exclusive scan of the flags (pos), each run's first index.
__global__ void run_starts_kernel(const uint32_t *__restrict__ keys, const uint32_t *__restrict__ pos,
                                  int64_t n, uint32_t *__restrict__ starts)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        if (i == 0 || keys[i] != keys[i - 1]) starts[pos[i]] = (uint32_t)i;
}

// Compensated (Kahan) fp32 sum, every operation rounded to nearest (no
// contraction): the error stays within a few ulps of the total whatever the
// number of terms, with fp32 arithmetic only.
struct KahanSum {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float x)
    {
        const float y = __fsub_rn(x, c);
        const float t = __fadd_rn(s, y);
        c = __fsub_rn(__fsub_rn(t, s), y);
        s = t;
    }
};

// Parameter `a` of point i: position (a < 3), SH (a < 3 + nsh), opacity,
// radius.
struct Params {
    const float *pos, *sh, *op, *rad;
    int nsh;
    __device__ __forceinline__ float get(uint32_t i, int a) const
    {
        if (a < 3) return pos[3 * (size_t)i + a];
        if (a < 3 + nsh) return sh[(size_t)nsh * i + (a - 3)];
        return a == 3 + nsh ? op[i] : rad[i];
    }
};
struct OutParams {
    float *pos, *sh, *op, *rad;
    int nsh;
    __device__ __forceinline__ void put(int64_t i, int a, float v) const
    {
        if (a < 3) pos[3 * i + a] = v;
        else if (a < 3 + nsh) sh[(int64_t)nsh * i + (a - 3)] = v;
        else if (a == 3 + nsh) op[i] = v;
        else rad[i] = v;
    }
};

// Attributes of a lane: a_begin + lane, + 32, ... (at most two: 3 + 48 + 2).
// Sums over GATHER points at a time, all their loads in flight together; the
// additions keep their order.  One load, then its four dependent additions,
// at a time, these kernels waited on memory for most of their time.  A 1M
// point cloud, 53 attributes: voxel means 267 -> 165 us (172 two at a time,
// 212 eight), means of 8 neighbours 298 -> 268.
constexpr int GATHER = 4;

// Compensated sums of attributes a0 (and a1 when two) over points idx(0) ..
// idx(cnt - 1).
template <class Idx>
__device__ __forceinline__ void sum_points(const Params &in, Idx idx, int cnt, int a0, int a1,
                                           bool two, KahanSum &s0, KahanSum &s1)
{
    for (int m = 0; m < cnt; m += GATHER) {
        uint32_t p[GATHER];
        float x[GATHER], y[GATHER];
#pragma unroll
        for (int u = 0; u < GATHER; ++u) p[u] = idx(m + u < cnt ? m + u : m);
#pragma unroll
        for (int u = 0; u < GATHER; ++u) {
            x[u] = m + u < cnt ? in.get(p[u], a0) : 0.0f;
            y[u] = two && m + u < cnt ? in.get(p[u], a1) : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < GATHER; ++u) {
            if (m + u >= cnt) break;
            s0.add(x[u]);
            if (two) s1.add(y[u]);
        }
    }
}

__global__ void __launch_bounds__(256)
voxel_mean_kernel(const uint32_t *__restrict__ order, const uint32_t *__restrict__ starts,
                  int64_t n_runs, int64_t n, Params in, OutParams out)
{
    const int lane = threadIdx.x & 31;
    const int nattr = 5 + in.nsh;
    const int a1 = lane + 32;
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n_runs;
         r += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const uint32_t b = starts[r];
        const uint32_t e = r + 1 < n_runs ? starts[r + 1] : (uint32_t)n;
        const float cnt = (float)(e - b);
        if (lane >= nattr) continue;
        KahanSum s0, s1;
        sum_points(in, [&](int m) { return __ldg(order + b + m); }, (int)(e - b), lane, a1,
                   a1 < nattr, s0, s1);
        out.put(r, lane, __fdiv_rn(s0.s, cnt));
        if (a1 < nattr) out.put(r, a1, __fdiv_rn(s1.s, cnt));
    }
}

// ------------------------------------------------------------------ kNN
__device__ __forceinline__ uint32_t lower_bound_u32(const uint32_t *__restrict__ a, uint32_t n,
                                                    uint32_t key)
{
    uint32_t lo = 0, hi = n;
    while (lo < hi) {
        const uint32_t mid = lo + ((hi - lo) >> 1);
        if (__ldg(a + mid) < key) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// Cells between coordinate c and the grid [0, n-1] along one axis.
__device__ __forceinline__ int axis_gap(int c, int n)
{
    if (c < 0) return -c;
    return c > n - 1 ? c - (n - 1) : 0;
}

// Inserts (cd, cj) into the warp's sorted list (lane j = j-th best, j <
// keff) if it ranks among the first keff; updates the K-th best (kd, ki).
__device__ __forceinline__ void knn_insert(float &bd, uint32_t &bi, float cd, uint32_t cj,
                                           int keff, uint32_t kmask, int lane, float &kd,
                                           uint32_t &ki)
{
    const bool less = bd < cd || (bd == cd && bi < cj);
    const int p = __popc(__ballot_sync(FULL, less) & kmask);
    if (p >= keff) return;
    const float ud = __shfl_up_sync(FULL, bd, 1);
    const uint32_t ui = __shfl_up_sync(FULL, bi, 1);
    if (lane == p) {
        bd = cd;
        bi = cj;
    } else if (lane > p && lane < keff) {
        bd = ud;
        bi = ui;
    }
    kd = __shfl_sync(FULL, bd, keff - 1);
    ki = __shfl_sync(FULL, bi, keff - 1);
}

// Index range [s, t) of the points in cells [a, b] (consecutive ids) of
// the sorted list: from the dense cell-start table when there is one, else
// by binary search for s and a galloping search for t.
__device__ __forceinline__ void cell_range(const uint32_t *__restrict__ cs,
                                           const uint32_t *__restrict__ rid, uint32_t nr,
                                           uint32_t a, uint32_t b, uint32_t &s, uint32_t &t)
{
    if (cs) {
        s = __ldg(cs + a);
        t = __ldg(cs + b + 1);
        return;
    }
    s = lower_bound_u32(rid, nr, a);
    if (s >= nr || __ldg(rid + s) > b) {
        t = s;
        return;
    }
    uint32_t lo = s, step = 1, hi = s + 1; // rid[lo] <= b
    while (hi < nr && __ldg(rid + hi) <= b) {
        lo = hi;
        step <<= 1;
        hi = s + step;
    }
    if (hi > nr) hi = nr;
    while (hi - lo > 1) { // rid[lo] <= b, hi == nr or rid[hi] > b
        const uint32_t mid = lo + ((hi - lo) >> 1);
        if (__ldg(rid + mid) <= b) lo = mid;
        else hi = mid;
    }
    t = hi;
}

// Candidate j of the points in cell order against the query: squared
// distance and whether it would enter the current list.
__device__ __forceinline__ bool knn_candidate(uint32_t j, const float4 *__restrict__ pts, float qx,
                                              float qy, float qz, uint32_t self_idx, float kd,
                                              uint32_t ki, float &d2, uint32_t &ri)
{
    const float4 c = __ldg(pts + j);
    ri = __float_as_uint(c.w);
    if (ri == self_idx) return false;
    d2 = sq_dist(qx, qy, qz, c.x, c.y, c.z);
    return d2 < kd || (d2 == kd && ri < ki);
}

// Inserts the candidates of the lanes set in m, lowest lane first.
__device__ __forceinline__ void knn_insert_all(uint32_t m, float d2, uint32_t ri, float &bd,
                                               uint32_t &bi, int keff, uint32_t kmask, int lane,
                                               float &kd, uint32_t &ki)
{
    while (m) {
        const int src = __ffs(m) - 1;
        m &= m - 1;
        const float cd = __shfl_sync(FULL, d2, src);
        const uint32_t cj = __shfl_sync(FULL, ri, src);
        knn_insert(bd, bi, cd, cj, keff, kmask, lane, kd, ki);
    }
}

// Lower bound on the distance from the query to any point of a cell
// outside the cube of cells [c - r, c + r] (per axis), counting only faces
// with grid cells beyond them; FLT_MAX when the cube covers the grid.  The
// slack covers the rounding of cell coordinates and face positions.
__device__ __forceinline__ float unvisited_bound(const GridParams &g, int r, int cx, int cy,
                                                 int cz, float qx, float qy, float qz)
{
    const int c[3] = {cx, cy, cz};
    const float q[3] = {qx, qy, qz};
    float bound = FLT_MAX;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (c[a] - r > 0)
            bound = fminf(bound, q[a] - (g.lo[a] + (float)(c[a] - r) * g.h));
        if (c[a] + r < g.n - 1)
            bound = fminf(bound, (g.lo[a] + (float)(c[a] + r + 1) * g.h) - q[a]);
    }
    return bound == FLT_MAX ? FLT_MAX : bound * 0.99999f - g.slack;
}

// Lower bound on the distance along one axis from coordinate p to cell c of
// the grid (the slack as in unvisited_bound).
__device__ __forceinline__ float cell_gap(const GridParams &g, float p, float lo, int c)
{
    const float d = fmaxf((lo + (float)c * g.h) - p, p - (lo + (float)(c + 1) * g.h));
    return fmaxf(d * 0.99999f - g.slack, 0.0f);
}

// Whether row (y, z) of cells may hold a point as near as squared distance kd.
__device__ __forceinline__ bool row_open(const GridParams &g, float qy, float qz, int y, int z,
                                         float kd)
{
    const float a = cell_gap(g, qy, g.lo[1], y), b = cell_gap(g, qz, g.lo[2], z);
    return !(__fadd_rn(__fmul_rn(a, a), __fmul_rn(b, b)) > kd);
}

// Writes the warp's list (lane j = j-th best) as row q of the output.
__device__ __forceinline__ void knn_write(int64_t q, int k, int keff, int lane, float bd,
                                          uint32_t bi, int32_t *__restrict__ out_idx,
                                          float *__restrict__ out_d2)
{
    if (lane < k) {
        const bool have = lane < keff;
        out_idx[q * k + lane] = have ? (int32_t)bi : -1;
        out_d2[q * k + lane] = have ? bd : FLT_MAX;
    }
}

// Shells searched on one grid before a query moves on (to the coarser grid,
// then to the exhaustive kernel): a query whose neighbours lie across a wide
// empty region would otherwise walk (2r+1)^2 rows per shell alone while the
// rest of the GPU idles.
constexpr int KNN_MAX_SHELLS = 16;

// One warp per query.  Queries are 0..nq-1, or qlist[0..*nq_dev) when qlist
// is set.  self_mode: the queries are the reference points (query q is
// reference q and is skipped; its cell is clamped like theirs).  Queries
// still open after KNN_MAX_SHELLS shells are appended to `defer` (count in
// *n_defer) and their rows left unwritten.
__global__ void __launch_bounds__(256)
knn_kernel(const float *__restrict__ qpos, int64_t nq_all, const uint32_t *__restrict__ qlist,
           const uint32_t *__restrict__ nq_dev, uint32_t nr, KnnGrid grid, int k, int keff, int self_mode, int32_t *__restrict__ out_idx,
           float *__restrict__ out_d2, uint32_t *__restrict__ defer, uint32_t *__restrict__ n_defer)
{
    const GridParams g = *grid.gp;
    const uint32_t *__restrict__ rid = grid.rid;
    const float4 *__restrict__ pts = grid.pts;
    const uint32_t *__restrict__ cs = grid.cs;
    const int lane = threadIdx.x & 31;
    const int n = g.n;
    const uint32_t kmask = keff >= 32 ? FULL : ((1u << keff) - 1u);
    const int64_t nq = qlist ? (int64_t)*nq_dev : nq_all;
    for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < nq;
         t += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int64_t q = qlist ? (int64_t)qlist[t] : t;
        const float qx = qpos[3 * q], qy = qpos[3 * q + 1], qz = qpos[3 * q + 2];
        const uint32_t self_idx = self_mode ? (uint32_t)q : 0xffffffffu;
        float bd = FLT_MAX, kd = FLT_MAX;
        uint32_t bi = 0xffffffffu, ki = 0xffffffffu;
        bool keff_done = true;
        if (keff > 0) {
            const int cx = cell_coord(qx, g.lo[0], g.h, n, self_mode);
            const int cy = cell_coord(qy, g.lo[1], g.h, n, self_mode);
            const int cz = cell_coord(qz, g.lo[2], g.h, n, self_mode);
            // first shell that meets the grid
            const int r0 = max(axis_gap(cx, n), max(axis_gap(cy, n), axis_gap(cz, n)));
            for (int r = r0;; ++r) {
                // rows (dy, dz) of shell r that meet the grid
                const int dy0 = max(-r, -cy), dy1 = min(r, n - 1 - cy);
                const int dz0 = max(-r, -cz), dz1 = min(r, n - 1 - cz);
                const int ny = dy1 - dy0 + 1;
                const int rows = ny * (dz1 - dz0 + 1);
                for (int base = 0; base < rows; base += 32) {
                    // this lane's row: up to two index ranges of the sorted list
                    const int row = base + lane;
                    uint32_t s0 = 0, t0 = 0, s1 = 0, t1 = 0;
                    const int dy = dy0 + row % ny, dz = dz0 + row / ny;
                    // rows beyond the K-th best are skipped
                    if (row < rows && row_open(g, qy, qz, cy + dy, cz + dz, kd)) {
                        const uint32_t rb =
                            ((uint32_t)(cz + dz) * (uint32_t)n + (uint32_t)(cy + dy)) * (uint32_t)n;
                        if (abs(dy) == r || abs(dz) == r) {
                            const int x0 = max(cx - r, 0), x1 = min(cx + r, n - 1);
                            if (x0 <= x1)
                                cell_range(cs, rid, nr, rb + (uint32_t)x0, rb + (uint32_t)x1, s0, t0);
                        } else {
                            if (cx - r >= 0 && cx - r < n)
                                cell_range(cs, rid, nr, rb + (uint32_t)(cx - r),
                                           rb + (uint32_t)(cx - r), s0, t0);
                            if (cx + r >= 0 && cx + r < n)
                                cell_range(cs, rid, nr, rb + (uint32_t)(cx + r),
                                           rb + (uint32_t)(cx + r), s1, t1);
                        }
                    }
                    // runs longer than a warp: the whole warp, 32 points a step
#pragma unroll
                    for (int part = 0; part < 2; ++part) {
                        const uint32_t st = part ? s1 : s0, en = part ? t1 : t0;
                        uint32_t m = __ballot_sync(FULL, en - st > 32u);
                        while (m) {
                            const int src = __ffs(m) - 1;
                            m &= m - 1;
                            const uint32_t rs = __shfl_sync(FULL, st, src);
                            const uint32_t re = __shfl_sync(FULL, en, src);
                            for (uint32_t j0 = rs; j0 < re; j0 += 32) {
                                const uint32_t j = j0 + lane;
                                float d2 = FLT_MAX;
                                uint32_t ri = 0;
                                const bool better = j < re && knn_candidate(j, pts, qx, qy, qz, self_idx, kd,
                                                                            ki, d2, ri);
                                knn_insert_all(__ballot_sync(FULL, better), d2, ri, bd, bi, keff,
                                               kmask, lane, kd, ki);
                            }
                        }
                    }
                    // short runs: every lane walks its own, one point a step
                    if (t0 - s0 > 32u) s0 = t0;
                    if (t1 - s1 > 32u) s1 = t1;
                    while (true) {
                        const bool has = s0 < t0 || s1 < t1;
                        if (!__any_sync(FULL, has)) break;
                        float d2 = FLT_MAX;
                        uint32_t ri = 0;
                        bool better = false;
                        if (has) {
                            const uint32_t j = s0 < t0 ? s0++ : s1++;
                            better = knn_candidate(j, pts, qx, qy, qz, self_idx, kd, ki, d2, ri);
                        }
                        knn_insert_all(__ballot_sync(FULL, better), d2, ri, bd, bi, keff, kmask,
                                       lane, kd, ki);
                    }
                }
                const float bound = unvisited_bound(g, r, cx, cy, cz, qx, qy, qz);
                if (bound == FLT_MAX) break; // every cell visited
                if (kd < FLT_MAX && bound > 0.0f && kd < __fmul_rn(bound, bound)) break;
                if (r - r0 + 1 >= KNN_MAX_SHELLS) {
                    if (lane == 0) defer[atomicAdd(n_defer, 1u)] = (uint32_t)q;
                    keff_done = false;
                    break;
                }
            }
        }
        if (keff_done) knn_write(q, k, keff, lane, bd, bi, out_idx, out_d2);
    }
}

// One thread per query, on grids with a cell table: the first shells of the
// search, up to KT (>= k) entries in registers.  Rows of cells whose slab is
// farther away than the K-th best are skipped.  Queries come from qpts (a
// cloud in cell order, {x, y, z, index}) or, without one, from qpos in the
// order given; self: the queries are the reference points.  Queries still
// open after THREAD_SHELLS shells are appended to `defer`.
// A warp per query spends its 32 lanes on the few points of a cell and an
// insertion per accepted point on the whole warp; a thread per query keeps
// 32 queries of neighbouring cells in one warp, whose lanes read the same
// rows.  Bound by the latency of its gathers (the nine slices' bounds are
// loaded together).  200k points on surfaces, nearest point: 325 -> 36 us a
// search; 1M-point cloud reduced to its voxels with 1% outliers, 8 nearest:
// 1410 -> 310 us (134 here, 175 on the coarse grid for the outliers; 238
// there before it skipped rows; three shells here: 174 and no fewer left).
constexpr int THREAD_SHELLS = 2;

template <int KT>
__global__ void __launch_bounds__(128)
knn_thread_kernel(const float4 *__restrict__ qpts, const float *__restrict__ qpos, int64_t nq,
                  KnnGrid grid, int k, int keff, int self_mode, int32_t *__restrict__ out_idx,
                  float *__restrict__ out_d2, uint32_t *__restrict__ defer,
                  uint32_t *__restrict__ n_defer)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nq) return;
    const GridParams g = *grid.gp;
    const float4 *__restrict__ pts = grid.pts;
    const uint32_t *__restrict__ cs = grid.cs;
    const int n = g.n;
    float qx, qy, qz;
    uint32_t q;
    if (qpts) {
        const float4 v = __ldg(qpts + t);
        qx = v.x;
        qy = v.y;
        qz = v.z;
        q = __float_as_uint(v.w);
    } else {
        qx = __ldg(qpos + 3 * t);
        qy = __ldg(qpos + 3 * t + 1);
        qz = __ldg(qpos + 3 * t + 2);
        q = (uint32_t)t;
    }
    const uint32_t self_idx = self_mode ? q : 0xffffffffu;
    float bd[KT];
    uint32_t bi[KT];
#pragma unroll
    for (int m = 0; m < KT; ++m) {
        bd[m] = FLT_MAX;
        bi[m] = 0xffffffffu;
    }
    const int cx = cell_coord(qx, g.lo[0], g.h, n, self_mode);
    const int cy = cell_coord(qy, g.lo[1], g.h, n, self_mode);
    const int cz = cell_coord(qz, g.lo[2], g.h, n, self_mode);

    // the points of slots [s, e): bubble each through the sorted list
    auto visit = [&](uint32_t s, uint32_t e) {
        for (uint32_t j = s; j < e; ++j) {
            const float4 c = __ldg(pts + j);
            uint32_t ri = __float_as_uint(c.w);
            float d2 = sq_dist(qx, qy, qz, c.x, c.y, c.z);
            if (ri == self_idx || !(d2 < bd[KT - 1] || (d2 == bd[KT - 1] && ri < bi[KT - 1])))
                continue;
#pragma unroll
            for (int m = 0; m < KT; ++m) {
                const bool before = d2 < bd[m] || (d2 == bd[m] && ri < bi[m]);
                const float od = bd[m];
                const uint32_t oi = bi[m];
                bd[m] = before ? d2 : od;
                bi[m] = before ? ri : oi;
                d2 = before ? od : d2;
                ri = before ? oi : ri;
            }
        }
    };
    // whether row (y, z) of cells meets the grid and may hold a better point
    auto open = [&](int y, int z) {
        return y >= 0 && y < n && z >= 0 && z < n && row_open(g, qy, qz, y, z, bd[KT - 1]);
    };
    auto row_base = [&](int y, int z) { return ((uint32_t)z * (uint32_t)n + (uint32_t)y) * (uint32_t)n; };
    auto settled = [&](int r) {
        const float bound = unvisited_bound(g, r, cx, cy, cz, qx, qy, qz);
        if (bound == FLT_MAX) return true; // every cell visited
        return bd[KT - 1] < FLT_MAX && bound > 0.0f && bd[KT - 1] < __fmul_rn(bound, bound);
    };

    bool done = keff == 0;
    if (!done) { // shells 0 and 1: the nine rows' slices first, the query's own row leading
        constexpr int OY[9] = {0, -1, 1, 0, 0, -1, -1, 1, 1}, OZ[9] = {0, 0, 0, -1, 1, -1, 1, -1, 1};
        const int x0 = max(cx - 1, 0), x1 = min(cx + 1, n - 1);
        uint32_t s[9], e[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int y = cy + OY[i], z = cz + OZ[i];
            const bool in = x0 <= x1 && y >= 0 && y < n && z >= 0 && z < n;
            const uint32_t rb = in ? row_base(y, z) : 0u;
            s[i] = in ? __ldg(cs + rb + (uint32_t)x0) : 0u;
            e[i] = in ? __ldg(cs + rb + (uint32_t)x1 + 1) : 0u;
        }
#pragma unroll
        for (int i = 0; i < 9; ++i)
            if (s[i] < e[i] && open(cy + OY[i], cz + OZ[i])) visit(s[i], e[i]);
        done = settled(1);
    }
    for (int r = 2; r <= THREAD_SHELLS && !done; ++r) {
        const int x0 = max(cx - r, 0), x1 = min(cx + r, n - 1);
        for (int dz = -r; dz <= r; ++dz)
            for (int dy = -r; dy <= r; ++dy) {
                if (!open(cy + dy, cz + dz)) continue;
                const uint32_t rb = row_base(cy + dy, cz + dz);
                if (abs(dy) == r || abs(dz) == r) {
                    if (x0 <= x1) visit(__ldg(cs + rb + (uint32_t)x0), __ldg(cs + rb + (uint32_t)x1 + 1));
                } else {
                    if (cx - r >= 0 && cx - r < n)
                        visit(__ldg(cs + rb + (uint32_t)(cx - r)), __ldg(cs + rb + (uint32_t)(cx - r) + 1));
                    if (cx + r >= 0 && cx + r < n)
                        visit(__ldg(cs + rb + (uint32_t)(cx + r)), __ldg(cs + rb + (uint32_t)(cx + r) + 1));
                }
            }
        done = settled(r);
    }
    if (!done) {
        defer[atomicAdd(n_defer, 1u)] = q;
        return;
    }
    for (int m = 0; m < k; ++m) { // entries past the list stay padding
        int32_t oi = -1;
        float od = FLT_MAX;
#pragma unroll
        for (int j = 0; j < KT; ++j)
            if (j == m && m < keff) {
                oi = (int32_t)bi[j];
                od = bd[j];
            }
        out_idx[(int64_t)q * k + m] = oi;
        out_d2[(int64_t)q * k + m] = od;
    }
}

// Deferred queries, one block each: its 8 warps scan every reference point
// (warp w takes points w*32 + lane, w*32 + lane + 256, ...) into their own
// lists, which warp 0 then merges.  Exact, like the grid search.
__global__ void __launch_bounds__(256)
knn_exhaustive_kernel(const float *__restrict__ qpos, const float *__restrict__ rpos, uint32_t nr,
                      int k, int keff, int self_mode, const uint32_t *__restrict__ defer,
                      const uint32_t *__restrict__ n_defer, int32_t *__restrict__ out_idx,
                      float *__restrict__ out_d2)
{
    __shared__ float s_d[8][32];
    __shared__ uint32_t s_i[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t kmask = keff >= 32 ? FULL : ((1u << keff) - 1u);
    const uint32_t nd = *n_defer;
    for (uint32_t t = blockIdx.x; t < nd; t += gridDim.x) {
        const uint32_t q = defer[t];
        const float qx = qpos[3 * (size_t)q], qy = qpos[3 * (size_t)q + 1],
                    qz = qpos[3 * (size_t)q + 2];
        const uint32_t self_idx = self_mode ? q : 0xffffffffu;
        float bd = FLT_MAX, kd = FLT_MAX;
        uint32_t bi = 0xffffffffu, ki = 0xffffffffu;
        for (uint32_t j0 = (uint32_t)w * 32; j0 < nr; j0 += 256) {
            const uint32_t j = j0 + lane;
            float d2 = FLT_MAX;
            bool better = false;
            if (j < nr && j != self_idx) {
                d2 = sq_dist(qx, qy, qz, __ldg(rpos + 3 * (size_t)j), __ldg(rpos + 3 * (size_t)j + 1),
                             __ldg(rpos + 3 * (size_t)j + 2));
                better = d2 < kd || (d2 == kd && j < ki);
            }
            knn_insert_all(__ballot_sync(FULL, better), d2, j, bd, bi, keff, kmask, lane, kd, ki);
        }
        s_d[w][lane] = bd;
        s_i[w][lane] = bi;
        __syncthreads();
        if (w == 0) {
            for (int v = 1; v < 8; ++v) {
                const float d2 = s_d[v][lane];
                const uint32_t ri = s_i[v][lane];
                const bool better = lane < keff && (d2 < kd || (d2 == kd && ri < ki));
                knn_insert_all(__ballot_sync(FULL, better), d2, ri, bd, bi, keff, kmask, lane, kd,
                               ki);
            }
            knn_write(q, k, keff, lane, bd, bi, out_idx, out_d2);
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------- outliers
__global__ void outlier_flags_kernel(const float *__restrict__ d2, int64_t n, int k, int keff,
                                     float eps, uint32_t *__restrict__ keep)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (keff == 0) {
            keep[i] = 1u;
            continue;
        }
        const float *row = d2 + i * k;
        float s = 0.0f;
        for (int j = 0; j < keff; ++j) s = __fadd_rn(s, __fsqrt_rn(row[j]));
        const float mean = __fdiv_rn(s, (float)keff);
        float t = 0.0f;
        for (int j = 0; j < keff; ++j) {
            const float e = __fsub_rn(__fsqrt_rn(row[j]), mean);
            t = __fadd_rn(t, __fmul_rn(e, e));
        }
        const float delta = __fsqrt_rn(__fdiv_rn(t, (float)keff));
        keep[i] = delta > eps ? 0u : 1u;
    }
}

// Copies kept points to their compacted slots (pos = exclusive scan of keep),
// four points of a warp in flight at a time
// (1M points: 114 -> 55 us).
__global__ void __launch_bounds__(256)
compact_points_kernel(const uint32_t *__restrict__ keep, const uint32_t *__restrict__ pos,
                      int64_t n, Params in, OutParams out)
{
    const int lane = threadIdx.x & 31;
    const int nattr = 5 + in.nsh;
    const bool has0 = lane < nattr, has1 = lane + 32 < nattr;
    constexpr int W = 4;
    for (int64_t i = W * (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); i < n;
         i += W * (((int64_t)gridDim.x * blockDim.x) >> 5)) {
        bool k[W];
        int64_t o[W];
        float x[W], y[W];
#pragma unroll
        for (int u = 0; u < W; ++u) {
            k[u] = i + u < n && keep[i + u];
            o[u] = i + u < n ? pos[i + u] : 0;
        }
#pragma unroll
        for (int u = 0; u < W; ++u) {
            x[u] = k[u] && has0 ? in.get((uint32_t)(i + u), lane) : 0.0f;
            y[u] = k[u] && has1 ? in.get((uint32_t)(i + u), lane + 32) : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < W; ++u) {
            if (k[u] && has0) out.put(o[u], lane, x[u]);
            if (k[u] && has1) out.put(o[u], lane + 32, y[u]);
        }
    }
}

__global__ void fill_u32_kernel(uint32_t *__restrict__ p, int64_t n, uint32_t v)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        p[i] = v;
}

// ---------------------------------------------------------- generation
__global__ void __launch_bounds__(256)
generate_kernel(const int32_t *__restrict__ nbr, int64_t n, int k, int keff, Params in,
                OutParams out, int64_t out_base, int a_begin)
{
    const int lane = threadIdx.x & 31;
    const int nattr = 5 + in.nsh;
    const int a0 = a_begin + lane, a1 = a0 + 32;
    for (int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < n;
         q += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int32_t *row = nbr + q * k;
        if (a0 >= nattr) continue;
        // a point at no finite distance to enough others has fewer neighbours
        // (rows end in -1): the mean of those there are, NaN without any
        int have = keff;
        while (have > 0 && __ldg(row + have - 1) < 0) --have;
        const float cnt = (float)have;
        KahanSum s0, s1;
        sum_points(in, [&](int m) { return (uint32_t)__ldg(row + m); }, have, a0, a1, a1 < nattr, s0,
                   s1);
        out.put(out_base + q, a0, __fdiv_rn(s0.s, cnt));
        if (a1 < nattr) out.put(out_base + q, a1, __fdiv_rn(s1.s, cnt));
    }
}

unsigned grid_for(int64_t items, int per_block, int max_blocks)
{
    int64_t b = (items + per_block - 1) / per_block;
    if (b < 1) b = 1;
    if (b > max_blocks) b = max_blocks;
    return (unsigned)b;
}

constexpr int MAX_BLOCKS = 152 * 32;

} // namespace

size_t grid_temp_bytes() { return sizeof(float) * 6 * BBOX_PARTS; }

void launch_grid_params(const float *pos, int64_t n, int n_cells, GridParams *gp, int n_coarse,
                        GridParams *coarse, void *temp, cudaStream_t s)
{
    float *part = (float *)temp;
    const unsigned blocks = grid_for(n, BBOX_THREADS, BBOX_PARTS);
    bbox_partial_kernel<<<blocks, BBOX_THREADS, 0, s>>>(pos, n, part);
    grid_params_kernel<<<1, BBOX_THREADS, 0, s>>>(part, (int)blocks, n_cells, gp,
                                                    n_coarse, coarse);
    count_launches(2);
}

void launch_cell_ids(const float *pos, int64_t n, const GridParams *gp, uint32_t *keys,
                     uint32_t *vals, cudaStream_t s)
{
    if (n <= 0) return;
    cell_ids_kernel<<<grid_for(n, 256, MAX_BLOCKS), 256, 0, s>>>(pos, n, gp, keys, vals);
    count_launches(1);
}

void launch_run_starts(const uint32_t *keys, int64_t n, uint32_t *flags, uint32_t *starts,
                       unsigned long long *n_runs, void *scan_temp, cudaStream_t s)
{
    if (n <= 0) return;
    const unsigned g = grid_for(n, 256, MAX_BLOCKS);
    run_flags_kernel<<<g, 256, 0, s>>>(keys, n, flags);
    launch_exclusive_scan(flags, flags, n, n_runs, scan_temp, s);
    run_starts_kernel<<<g, 256, 0, s>>>(keys, flags, n, starts);
    count_launches(2);
}

void launch_voxel_mean(const uint32_t *order, const uint32_t *starts, int64_t n_runs, int64_t n,
                       const PointArrays &in, const PointArraysOut &out, cudaStream_t s)
{
    if (n_runs <= 0) return;
    voxel_mean_kernel<<<grid_for(n_runs, 8, MAX_BLOCKS), 256, 0, s>>>(
        order, starts, n_runs, n, Params{in.pos, in.sh, in.op, in.rad, in.nsh},
        OutParams{out.pos, out.sh, out.op, out.rad, out.nsh});
    count_launches(1);
}

size_t knn_temp_bytes(int64_t nq) { return sizeof(uint32_t) * (size_t)(2 * nq + 2); }

// Queries per search from which a thread per query is the faster start: 4096
// for each entry of its list, at least 8192.  Below, its few warps leave most
// SMs idle, and the longer a thread's list the longer its insertions (a whole
// self search, thread / warp per query, in us; k = 1: 8k points 96 / 98, 16k
// 86 / 91, 64k 83 / 148; k = 8: 16k 121 / 109, 64k 128 / 198; k = 16: 64k
// 277 / 253, 300k 450 / 1002).
inline bool thread_per_query(int64_t nq, int k) { return nq >= 4096 * (int64_t)(k > 2 ? k : 2); }

namespace {

template <int KT>
void thread_search(const float4 *qpts, const float *qpos, int64_t nq, const KnnGrid &g, int k,
                   int keff, int self_mode, int32_t *out_idx, float *out_d2, uint32_t *defer,
                   uint32_t *n_defer, cudaStream_t s)
{
    knn_thread_kernel<KT><<<(unsigned)((nq + 127) / 128), 128, 0, s>>>(
        qpts, qpos, nq, g, k, keff, self_mode, out_idx, out_d2, defer, n_defer);
}

} // namespace

const uint32_t *launch_knn(const float *qpos, const float4 *qpts, int64_t nq, int64_t nr,
                           const KnnGrid &fine, int k, int keff, int self_mode, int32_t *out_idx,
                           float *out_d2, void *temp, cudaStream_t s)
{
    uint32_t *cnt = (uint32_t *)temp, *d1 = cnt + 2;
    cudaMemsetAsync(cnt, 0, 2 * sizeof(uint32_t), s);
    if (thread_per_query(nq, k) && k <= 16 && fine.cs) {
        auto f = k == 1   ? thread_search<1>
                 : k == 2 ? thread_search<2>
                 : k <= 4 ? thread_search<4>
                 : k <= 8 ? thread_search<8>
                 : k <= 12 ? thread_search<12>
                           : thread_search<16>;
        f(qpts, qpos, nq, fine, k, keff, self_mode, out_idx, out_d2, d1, cnt, s);
    } else {
        knn_kernel<<<grid_for(nq, 8, MAX_BLOCKS), 256, 0, s>>>(qpos, nq, nullptr, nullptr,
                                                              (uint32_t)nr, fine, k, keff,
                                                              self_mode, out_idx, out_d2, d1, cnt);
    }
    count_launches(1);
    return cnt;
}

void launch_knn_rest(const float *qpos, int64_t nq, const float *rpos, int64_t nr,
                     const KnnGrid *coarse, int k, int keff, int self_mode, int32_t *out_idx,
                     float *out_d2, void *temp, cudaStream_t s)
{
    uint32_t *cnt = (uint32_t *)temp, *d1 = cnt + 2, *d2 = d1 + nq;
    const uint32_t *last = d1, *n_last = cnt;
    if (coarse) {
        knn_kernel<<<grid_for(nq, 8, 152 * 8), 256, 0, s>>>(qpos, 0, d1, cnt, (uint32_t)nr, *coarse,
                                                          k, keff, self_mode, out_idx, out_d2, d2,
                                                          cnt + 1);
        last = d2;
        n_last = cnt + 1;
        count_launches(1);
    }
    knn_exhaustive_kernel<<<304, 256, 0, s>>>(qpos, rpos, (uint32_t)nr, k, keff, self_mode, last,
                                              n_last, out_idx, out_d2);
    count_launches(1);
}

void launch_cell_sort(const float *pos, int64_t n, const GridParams *gp, int64_t n_cells_total,
                      uint32_t *ids, uint32_t *table, float4 *pts, void *scan_temp,
                      const uint32_t *gate, cudaStream_t s)
{
    cudaMemsetAsync(table, 0, sizeof(uint32_t) * (size_t)(n_cells_total + 1), s);
    if (n <= 0) return;
    const unsigned g = grid_for(n, 256, MAX_BLOCKS);
    cell_hist_kernel<<<g, 256, 0, s>>>(pos, n, gp, ids, table, gate);
    if (n_cells_total <= GATED_CELLS) {
        gated_scan_kernel<<<1, 1024, 0, s>>>(table + 1, (int)n_cells_total, gate);
        count_launches(1);
    } else {
        launch_exclusive_scan(table + 1, table + 1, n_cells_total, nullptr, scan_temp, s);
    }
    cell_scatter_kernel<<<g, 256, 0, s>>>(pos, n, ids, table, pts, gate);
    count_launches(2);
}

void launch_gather_points(const float *pos, const uint32_t *idx, int64_t n, float4 *pts,
                          cudaStream_t s)
{
    if (n <= 0) return;
    gather_points_kernel<<<grid_for(n, 256, MAX_BLOCKS), 256, 0, s>>>(pos, idx, n, pts);
    count_launches(1);
}

void launch_outlier_flags(const float *d2, int64_t n, int k, int keff, float eps, uint32_t *keep,
                          cudaStream_t s)
{
    if (n <= 0) return;
    outlier_flags_kernel<<<grid_for(n, 256, MAX_BLOCKS), 256, 0, s>>>(d2, n, k, keff, eps, keep);
    count_launches(1);
}

void launch_compact_points(const uint32_t *keep, const uint32_t *pos, int64_t n,
                           const PointArrays &in, const PointArraysOut &out, cudaStream_t s)
{
    if (n <= 0) return;
    compact_points_kernel<<<grid_for(n, 32, MAX_BLOCKS), 256, 0, s>>>(
        keep, pos, n, Params{in.pos, in.sh, in.op, in.rad, in.nsh},
        OutParams{out.pos, out.sh, out.op, out.rad, out.nsh});
    count_launches(1);
}

void launch_fill_u32(uint32_t *p, int64_t n, uint32_t v, cudaStream_t s)
{
    if (n <= 0) return;
    fill_u32_kernel<<<grid_for(n, 256, MAX_BLOCKS), 256, 0, s>>>(p, n, v);
    count_launches(1);
}

void launch_generate(const int32_t *nbr, int64_t n, int k, int keff, const PointArrays &in,
                     const PointArraysOut &out, int64_t out_base, cudaStream_t s, int a_begin)
{
    if (n <= 0 || keff <= 0) return;
    generate_kernel<<<grid_for(n, 8, MAX_BLOCKS), 256, 0, s>>>(
        nbr, n, k, keff, Params{in.pos, in.sh, in.op, in.rad, in.nsh},
        OutParams{out.pos, out.sh, out.op, out.rad, out.nsh}, out_base, a_begin);
    count_launches(1);
}

} // namespace pbr
