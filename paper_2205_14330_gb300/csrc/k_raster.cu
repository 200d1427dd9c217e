// Per-tile compositing of Sec. 3.2 and its adjoint.
//
// Per pixel centre u and listed point (records {px, py, rc^2, q'} {o, rgb}):
//   d2 = (ux - px)^2 + (uy - py)^2            (fp32, round-to-nearest; the persistent
//                                             schedule fuses the second square)
//   if d2 <= rc^2:                             (the cutoff of Sec. 3.2)
//     alpha = min(alpha_max, o * 2^(q' d2))    (Eq. 5, q' = -log2(e)/(2 s^2))
//     C += T alpha c ;  T *= (1 - alpha)       (Eqs. 6-7, front to back)
// stopping after the point that takes T below t_eps or reaches the count
// cap.  Outputs C + T bg, T and the list position just after the last
// composited point.
//
// The adjoint walks each pixel's list back to front from that position.  T
// before a point is recovered as T_after/(1-alpha); S accumulates the colour
// behind the point, so
//   dL/dc     = alpha T g
//   dL/dalpha = T (c.g) - S / (1 - alpha)
// and, below the alpha_max clamp, with dG = dL/dalpha G,
//   dL/do = dG,  dL/dp = o dG q (u - p),  dL/dq = -o dG d2 / 2   (q = 1/s^2).
// The kernels sum {dG (u - p), dG d2}, without the per-point factors o, q and
// -1/2, which the point stage applies once per point-view: the terms are
// {dG dx, dG dy, dG d2, do, dr, dg, db}.
// The 7 per-point terms of a warp go to the per-(view, point) buffer with
// 16-byte atomics: straight from each contributing lane when few lanes
// contribute, else summed first with a transposed shuffle reduction (two
// atomics per warp and point) in the warp-streamed schedules.
//
// The pair keys carry the mask of the tile's 8 x 8 pixel blocks that hold a
// pixel including the point, so a warp takes from its tile's list only the
// entries of its own block, and it skips those whose cutoff disc misses its
// still active pixels.  Three schedules:
//   - warp-streamed (batch depth 0, default): a block covers one TW x TH
//     screen tile, each warp an 8 x 8 block of it (a lane owns two pixels of
//     a column, four rows apart) or, where few long lists decide the time,
//     half of one (one pixel a lane; the rule is raster_lanes').  Every warp
//     walks its entries by itself, 32 per step, culls them with one ballot,
//     steps through the hits in lockstep and stops as soon as its own pixels
//     have saturated.  No block barriers.
//   - persistent (batch depth 0, persistent): the same walk in one launch;
//     warps take (tile, unit) items longest list first from an atomic
//     counter.
//   - block-staged (batch depth > 0): the block stages `depth` records in
//     shared memory and each warp culls the batch into its own list; block
//     barriers between batches, per-block shared-memory gradient sums.
// What bounds the walks: 92 M (8 x 8 block, hit) steps on the 1M-point,
// 64-view batch, of whose 64 pixels 44 are still active and 17 include the
// point.  The forward is bound by instruction issue (about 45 a step; one
// pixel's weight, three colour sums and T are 6 of them), the backward by
// issue (85 a step, 71% of the slots) and the L1 data path (82%) together: a
// shared-memory read of 16 bytes a lane takes four cycles of that path even
// when every lane reads the same address, and so do the atomics' operands.
// So hits are staged compacted, the loops over them carry no bit scans and
// are unrolled with the loads first, a point's own scalars stay scalar
// operands (a packed operation would need them duplicated), the blend is
// predicated per pixel instead of masked, and a chunk whose amplitudes are
// all below the clamp skips the clamp.  Measured against lockstep loops over
// hit masks (8 x 4 one-pixel warps in the streamed schedule), 1M points, 64
// views, 16 x 32 tiles, persistent: forward 5.31 -> 4.09 ms, backward 9.34 ->
// 8.84 ms; 500k points, 4 views of 800 x 800, 16 x 16 tiles, streamed: forward
// 257 -> 188 us, backward 423 -> 363 us, in store mode 333 -> 304 us and 569 ->
// 528 us; one 1920 x 1080 view of 1M points: forward 216 -> 151 us.
// Store mode (STORE): the forward also keeps T before each of a pixel's
// first store_depth composited points, and the backward reads it there
// instead of dividing, each value one composited point ahead of its use.
#include "pbr_internal.cuh"

namespace pbr {

namespace {

__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ uint32_t lanemask_lt_r()
{
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

__device__ __forceinline__ int find_view_by_tile(const Batch &b, uint32_t tile)
{
    int lo = 0, hi = b.n_views - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (b.views[mid].tile_base <= tile) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// The calling thread's pixel and its warp's 8 x 4 rectangle of pixel
// centres [xl, xh] x [yl, yh] inside tile `tile`.
struct PixelGeom {
    const DevView *V;
    int x, y;
    bool inside;
    float ux, uy, xl, xh, yl, yh;
};

// Pixel (sx0 + (lane & 7), sy0 + (lane >> 3)) of view V and the 8 x 4
// rectangle of pixel centres with corner (sx0, sy0).
__device__ __forceinline__ PixelGeom pixel_geom_at(const DevView *V, int sx0, int sy0, int lane)
{
    PixelGeom g;
    g.V = V;
    g.x = sx0 + (lane & 7);
    g.y = sy0 + (lane >> 3);
    g.inside = g.x < g.V->W && g.y < g.V->H;
    g.ux = (float)g.x + 0.5f;
    g.uy = (float)g.y + 0.5f;
    g.xl = (float)sx0 + 0.5f;
    g.xh = (float)sx0 + 7.5f;
    g.yl = (float)sy0 + 0.5f;
    g.yh = (float)sy0 + 3.5f;
    return g;
}

// Sub-block `w` of tile `tile` (sub-blocks numbered row-major, TW/8 per row).
template <int TW, int TH>
__device__ __forceinline__ PixelGeom pixel_geom(const Batch &b, uint32_t tile, int w, int lane)
{
    const DevView *V = &b.views[find_view_by_tile(b, tile)];
    const uint32_t local = tile - V->tile_base;
    const int tx = (int)(local % (uint32_t)V->tiles_x), ty = (int)(local / (uint32_t)V->tiles_x);
    return pixel_geom_at(V, tx * TW + (w % (TW / 8)) * 8, ty * TH + (w / (TW / 8)) * 4, lane);
}

// Culling test of one record against a rectangle of pixel centres: the
// per-pixel cutoff test (the same fp32 operations, see pair_d2) applied to the
// rectangle's pixel centre nearest the splat centre, floor(p) + 0.5 clamped
// into the rectangle per axis.  Rounding is monotone, of products and sums as
// of a fused multiply-add, so that centre has the smallest fp32 squared
// distance of all the rectangle's centres: the test keeps exactly the points
// some pixel of the rectangle includes.  Which points a pixel composites
// therefore does not hang on the rectangle, and the forward and the backward
// may cull with different ones.
template <bool FUSED>
__device__ __forceinline__ bool disc_meets_rect(const float4 a, const PixelGeom &g)
{
    const float cx = fminf(fmaxf(floorf(a.x) + 0.5f, g.xl), g.xh);
    const float cy = fminf(fmaxf(floorf(a.y) + 0.5f, g.yl), g.yh);
    const float ex = __fsub_rn(cx, a.x), ey = __fsub_rn(cy, a.y);
    const float ex2 = __fmul_rn(ex, ex);
    return (FUSED ? __fmaf_rn(ey, ey, ex2) : __fadd_rn(ex2, __fmul_rn(ey, ey))) <= a.z;
}

// The rectangle of the centres of the still active pixels of a warp that
// owns P pixels per lane, one column, rows 4 apart (g[q] below g[q-1]).
// Warp-wide reductions: all 32 lanes must call it together, outside any
// lane-dependent branch or short-circuit.
template <int P>
__device__ __forceinline__ PixelGeom active_rect_rows(const PixelGeom (&g)[P], const bool (&act)[P])
{
    PixelGeom r = g[0];
    bool any = false;
    uint32_t ylo = 0xffffffffu, yhi = 0u;
#pragma unroll
    for (int q = P - 1; q >= 0; --q) {
        any = any || act[q];
        if (act[q]) ylo = (uint32_t)g[q].y;
    }
#pragma unroll
    for (int q = 0; q < P; ++q)
        if (act[q]) yhi = (uint32_t)g[q].y;
    const uint32_t x = (uint32_t)g[0].x;
    const uint32_t x0 = __reduce_min_sync(0xffffffffu, any ? x : 0xffffffffu);
    const uint32_t x1 = __reduce_max_sync(0xffffffffu, any ? x : 0u);
    const uint32_t y0 = __reduce_min_sync(0xffffffffu, ylo);
    const uint32_t y1 = __reduce_max_sync(0xffffffffu, yhi);
    r.xl = (float)x0 + 0.5f;
    r.xh = (float)x1 + 0.5f;
    r.yl = (float)y0 + 0.5f;
    r.yh = (float)y1 + 0.5f;
    return r;
}

// Sum of 8 per-lane values over the warp; lane l returns the total of value
// (l >> 2) & 7.  Three halving exchanges then two butterfly steps.
__device__ __forceinline__ float warp_sum8_transposed(const float v[8], int lane)
{
    float a[4];
    bool hi = lane & 16;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float send = hi ? v[k] : v[k + 4];
        const float keep = hi ? v[k + 4] : v[k];
        a[k] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
    float c2[2];
    hi = lane & 8;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float send = hi ? a[k] : a[k + 2];
        const float keep = hi ? a[k + 2] : a[k];
        c2[k] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
    hi = lane & 4;
    float r;
    {
        const float send = hi ? c2[0] : c2[1];
        const float keep = hi ? c2[1] : c2[0];
        r = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
    r += __shfl_xor_sync(0xffffffffu, r, 2);
    r += __shfl_xor_sync(0xffffffffu, r, 1);
    return r;
}

// Adds the warp's 7 per-point terms to g2d[pv][0..6] with two 16-byte
// atomics: after the transposed reduction lane 4k holds term k; lanes 0 and
// 16 gather four terms each.
__device__ __forceinline__ void warp_add_terms(const float v[8], int lane, float *g2d, uint32_t pv)
{
    const float t = warp_sum8_transposed(v, lane);
    const float t1 = __shfl_down_sync(0xffffffffu, t, 4);
    const float t2 = __shfl_down_sync(0xffffffffu, t, 8);
    const float t3 = __shfl_down_sync(0xffffffffu, t, 12);
    if ((lane & 15) == 0) {
        float4 *dst = reinterpret_cast<float4 *>(g2d + 8 * (size_t)pv) + (lane >> 4);
        atomicAdd(dst, make_float4(t, t1, t2, lane ? 0.f : t3));
    }
}

// ------------------------------------------------------ block-mask queues
// The pair keys carry the mask of the 8 x 8 pixel blocks of the tile that
// hold a pixel including the point (pair key = tile << B | mask), so a warp
// working on one block takes from its tile's list only the entries with its
// block's bit: the queue below holds their list positions (relative to the
// tile's first entry) and point-view ids, in compositing order, and the
// compositing loops consume it 32 entries at a time.  bit == 0 (tiles of
// one block) takes every entry.
// The queue is a ring of QCAP entries read from `head`; a fill scans
// FILL_GROUPS groups of 32 list entries per step, their loads in flight
// together (a warp's block takes a fraction of its tile's entries, so a
// refill scans several groups).
constexpr int QCAP = 128;
constexpr int FILL_GROUPS = 3; // 32 + 3 x 32 entries fit the ring
struct WarpQueue {
    uint32_t pos[QCAP]; // list positions, relative to the tile's first entry
    uint32_t pv[QCAP];  // point-view ids
};

// Front to back: scans the list from position p (absolute, < e), appending
// the entries with `bit`, until the queue holds 32 or the list ends.
// Warp-uniform.
__device__ __forceinline__ void queue_fill_front(const uint32_t *__restrict__ keys,
                                                 const uint32_t *__restrict__ pv_list, uint32_t s,
                                                 uint32_t e, uint32_t bit, uint32_t &p, int &qn,
                                                 uint32_t qh, WarpQueue &q, int lane)
{
    const uint32_t lt = lanemask_lt_r();
    while (qn < 32 && p < e) {
        uint32_t k[FILL_GROUPS];
#pragma unroll
        for (int g = 0; g < FILL_GROUPS; ++g) {
            const uint32_t i = p + 32 * g + lane;
            k[g] = bit && i < e ? __ldg(keys + i) : 0u;
        }
#pragma unroll
        for (int g = 0; g < FILL_GROUPS; ++g) {
            const uint32_t i = p + 32 * g + lane;
            const bool take = i < e && (bit == 0 || (k[g] & bit) != 0);
            const uint32_t m = __ballot_sync(0xffffffffu, take);
            if (take) {
                const uint32_t slot = (qh + (uint32_t)qn + __popc(m & lt)) & (QCAP - 1);
                q.pos[slot] = i - s;
                q.pv[slot] = __ldg(pv_list + i);
            }
            qn += __popc(m);
        }
        p = e - p > 32u * FILL_GROUPS ? p + 32u * FILL_GROUPS : e;
    }
    __syncwarp();
}

// Back to front: scans the relative positions [0, c + 32) downwards from
// the aligned chunk c (c < 0: nothing left), entries below `lim` only,
// appending the entries with `bit` in descending position order.
__device__ __forceinline__ void queue_fill_back(const uint32_t *__restrict__ keys,
                                                const uint32_t *__restrict__ pv_list, uint32_t s,
                                                uint32_t lim, uint32_t bit, int64_t &c, int &qn,
                                                uint32_t qh, WarpQueue &q, int lane)
{
    const uint32_t gt = ~(lanemask_lt_r() | (1u << lane));
    while (qn < 32 && c >= 0) {
        uint32_t k[FILL_GROUPS];
#pragma unroll
        for (int g = 0; g < FILL_GROUPS; ++g) {
            const int64_t cg = c - 32 * g;
            const uint32_t i = (uint32_t)cg + lane;
            k[g] = bit && cg >= 0 && i < lim ? __ldg(keys + s + i) : 0u;
        }
#pragma unroll
        for (int g = 0; g < FILL_GROUPS; ++g) {
            const int64_t cg = c - 32 * g;
            const uint32_t i = (uint32_t)cg + lane;
            const bool take = cg >= 0 && i < lim && (bit == 0 || (k[g] & bit) != 0);
            const uint32_t m = __ballot_sync(0xffffffffu, take);
            if (take) {
                const uint32_t slot = (qh + (uint32_t)qn + __popc(m & gt)) & (QCAP - 1);
                q.pos[slot] = i;
                q.pv[slot] = __ldg(pv_list + s + i);
            }
            qn += __popc(m);
        }
        c -= 32 * FILL_GROUPS;
    }
    __syncwarp();
}

// Takes the next min(qn, 32) queued entries: lane l < the count receives
// entry l (its relative position and point-view).  Returns the count.
__device__ __forceinline__ int queue_take(WarpQueue &q, int &qn, uint32_t &qh, int lane,
                                          uint32_t &pos, uint32_t &pv)
{
    const int take = qn < 32 ? qn : 32;
    if (lane < take) {
        const uint32_t slot = (qh + (uint32_t)lane) & (QCAP - 1);
        pos = q.pos[slot];
        pv = q.pv[slot];
    }
    qh += (uint32_t)take;
    qn -= take;
    __syncwarp();
    return take;
}

// Keeps the compiler from fusing the product that produced v into a later
// add (a product feeding an add can be merged into one fused multiply-add
// even across __fmul_rn, which changes the rounding of a distance and with
// it the exact cutoff decision).
__device__ __forceinline__ float unfused1(float v)
{
    asm("" : "+f"(v));
    return v;
}

// One composited point, front to back.  Returns true when the pixel stops.
// Every rounding is explicit: alpha = min(alpha_max, o 2^(q' d2)), weight
// alpha T, C += weight c (fused), T -= weight.
__device__ __forceinline__ bool pixel_blend(float d2, const float4 a, const float4 c,
                                            const DevOpts &o, float &T, float &C0, float &C1,
                                            float &C2, uint32_t &cnt)
{
    const float alpha = fminf(o.alpha_max, __fmul_rn(c.x, ex2_approx(__fmul_rn(d2, a.w))));
    const float wgt = __fmul_rn(alpha, T);
    C0 = fmaf(wgt, c.y, C0);
    C1 = fmaf(wgt, c.z, C1);
    C2 = fmaf(wgt, c.w, C2);
    T = __fsub_rn(T, wgt);
    ++cnt;
    return T < o.t_eps || cnt == (uint32_t)o.max_per_pixel;
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Per-pixel adjoint of one composited point (see the file comment).  On
// return v[0..6] = {dG dx, dG dy, dG d2, do, dr, dg, db}; T and S are
// updated.
__device__ __forceinline__ void pixel_adjoint(float d2, float dx, float dy, const float4 a,
                                              const float4 c, float amax, float g0, float g1,
                                              float g2, float &T, float &S, float v[8])
{
    const float G = ex2_approx(d2 * a.w);
    const float raw = c.x * G;
    const float alpha = fminf(amax, raw);
    const float rom = __frcp_rn(1.0f - alpha);
    const float Tb = T * rom;
    const float wgt = alpha * Tb;
    const float cg = c.y * g0 + c.z * g1 + c.w * g2;
    v[4] = wgt * g0;
    v[5] = wgt * g1;
    v[6] = wgt * g2;
    const float dalpha = Tb * cg - S * rom;
    S = fmaf(wgt, cg, S);
    T = Tb;
    if (raw < amax) {
        const float dG = dalpha * G;
        v[0] = dG * dx;
        v[1] = dG * dy;
        v[2] = dG * d2;
        v[3] = dG;
    }
}

__device__ __forceinline__ float pixel_d2(float ux, float uy, float px, float py, float &dx,
                                          float &dy)
{
    dx = __fsub_rn(ux, px);
    dy = __fsub_rn(uy, py);
    return __fadd_rn(unfused1(__fmul_rn(dx, dx)), unfused1(__fmul_rn(dy, dy)));
}

// Index of the pixel in the packed per-pixel arrays (valid when inside).
__device__ __forceinline__ int64_t pixel_index(const PixelGeom &g)
{
    return g.V->pix_base + (int64_t)g.y * g.V->W + g.x;
}

// Store mode: T before the cnt-th composited point of pixel pix.
__device__ __forceinline__ void store_T(const StoreBuf &sto, int64_t pix, uint32_t cnt, float T)
{
    if (cnt < (uint32_t)sto.depth) sto.T[pix * sto.depth + cnt] = T;
}

// Store mode, backward: one pixel's list read back to front, each value
// fetched one composited point ahead of its use.
struct StoreRow {
    const float *p;
    uint32_t k, depth; // composited points not yet visited
    float nxt;         // T before point k - 1 (when k - 1 < depth)
};

__device__ __forceinline__ StoreRow store_row(const StoreBuf &sto, int64_t pix, bool inside)
{
    StoreRow r;
    r.p = sto.T + pix * sto.depth;
    r.depth = (uint32_t)sto.depth;
    r.k = inside ? sto.n[pix] : 0u;
    r.nxt = r.k > 0 && r.k <= r.depth ? r.p[r.k - 1] : 0.0f;
    return r;
}

// Visits the pixel's next composited point if `take`: whether its T was
// stored, and T.
__device__ __forceinline__ bool row_next(StoreRow &r, bool take, float &T)
{
    const bool has = take && r.k <= r.depth;
    T = r.nxt;
    r.k -= take;
    if (take && r.k - 1u < r.depth) r.nxt = r.p[r.k - 1u];
    return has;
}

__device__ __forceinline__ void write_pixel(const PixelGeom &g, const DevOpts &o, float T,
                                            float C0, float C1, float C2, uint32_t last,
                                            float *out_rgb, float *T_final, uint32_t *n_contrib)
{
    if (!g.inside) return;
    const int64_t local = (int64_t)g.y * g.V->W + g.x;
    const int64_t pix = g.V->pix_base + local;
    float *dst = g.V->out ? g.V->out + 3 * local : out_rgb + 3 * pix;
    dst[0] = C0 + T * o.bg[0];
    dst[1] = C1 + T * o.bg[1];
    dst[2] = C2 + T * o.bg[2];
    T_final[pix] = T;
    n_contrib[pix] = last;
}

__device__ __forceinline__ void add_stats(unsigned long long *stats, uint32_t a, uint32_t b,
                                          int lane)
{
    if (!stats) return;
    const uint32_t wa = __reduce_add_sync(0xffffffffu, a);
    const uint32_t wb = __reduce_add_sync(0xffffffffu, b);
    if (lane == 0) {
        atomicAdd(stats, (unsigned long long)wa);
        atomicAdd(stats + 1, (unsigned long long)wb);
    }
}

// ------------------------------------------------- packed two-pixel math
// A lane of the 8 x 8-pixel warps owns two pixels of one column, rows 4
// apart (A above B); their per-point arithmetic runs in packed fp32x2
// operations (.x pixel A, .y pixel B), one instruction for both pixels.
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// Squared fp32 distances from the lane's two pixel centres (ux, uy.x) and
// (ux, uy.y) to the splat centre: dx = ux - px (shared), dy = uy - py, d2 =
// dx dx + dy dy.  FUSED 0 (streamed): each operation rounded to nearest, as
// in pixel_d2.  FUSED 1 (persistent): dy dy + dx dx rounded once.  Each
// schedule keeps its own rounding, forward and backward alike: whether a
// pixel on the edge of a disc includes the point can turn on the last bit.
template <bool FUSED>
__device__ __forceinline__ float2 pair_d2(float ux, float2 uy, float px, float py, float &dx,
                                          float2 &dy)
{
    dx = __fsub_rn(ux, px);
    dy = make_float2(__fsub_rn(uy.x, py), __fsub_rn(uy.y, py));
    const float dx2 = __fmul_rn(dx, dx);
    if (FUSED) return make_float2(__fmaf_rn(dy.x, dy.x, dx2), __fmaf_rn(dy.y, dy.y, dx2));
    const float2 dy2 = mul2(dy, dy); // the sums are scalar: no packed add to fuse it into
    return make_float2(__fadd_rn(dx2, dy2.x), __fadd_rn(dx2, dy2.y));
}

// One warp's shared memory of the forward.
struct FwdWarp {
    float4 a[32], c[32]; // the chunk's hits: record halves
    uint32_t pos[32];    // and their list positions
    WarpQueue q;
};

// Forward of one 8 x 8 block by one warp: lane l owns the pixels A = (l & 7, l
// >> 3) and B = (l & 7, 4 + (l >> 3)).  The warp takes the tile list's
// entries with its block's bit (`bit`) 32 at a time from its queue, culls
// them against the rectangle of its active pixels and stages the hits in list
// order; then it steps through them, every lane testing and blending the
// point at both of its pixels; the blend of a pixel the point does not
// include (or that has stopped) is predicated off.  Each pixel's blend
// sequence and roundings are the one-pixel walk's.
// A pixel is active until its T is below t_eps (-1 outside the image; t_eps at
// most 1, see scheduled_opts).  Whether a pixel's two conditions are joined by &
// or && only moves the schedule of instructions: & and && take 3.88 and 3.99 ms in
// the persistent forward of the 1M-point, 64-view step, 616 and 606 us streamed,
// counting, on 16 views of 257 x 1023 to 1279 x 719.
// COUNT: the points composited per pixel are counted (pair counts, store
// mode, the count cap).
// FUSED: the rounding of the squared distance (pair_d2).
// NP: pixels a lane owns; with 1 the warp's pixels are the 8 x 4 sub-block
// with first pixel (sx0, sy0), and what concerns pixel B compiles away.
template <int NP, bool COUNT, bool STORE, bool FUSED>
__device__ __forceinline__ void fwd_pair_item(const DevView *V, int sx0, int sy0, uint32_t s,
                                              uint32_t e, uint32_t bit, const DevOpts &o, int lane,
                                              const uint32_t *__restrict__ keys,
                                              const uint32_t *__restrict__ pv_list,
                                              const float4 *__restrict__ rec,
                                              float *__restrict__ out_rgb,
                                              float *__restrict__ T_final,
                                              uint32_t *__restrict__ n_contrib,
                                              uint32_t &examined_acc, uint32_t &composited_acc,
                                              FwdWarp &m, const StoreBuf &sto)
{
    PixelGeom g[NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) g[q] = pixel_geom_at(V, sx0, sy0 + 4 * q, lane);
    const PixelGeom &gA = g[0], &gB = g[NP - 1];
    const int64_t pixA = STORE && gA.inside ? pixel_index(gA) : 0;
    const int64_t pixB = STORE && gB.inside ? pixel_index(gB) : 0;
    float2 T = make_float2(gA.inside ? 1.0f : -1.0f, NP == 2 && gB.inside ? 1.0f : -1.0f);
    float2 C0 = f2(0.0f), C1 = f2(0.0f), C2 = f2(0.0f);
    uint32_t cntA = 0, cntB = 0, lastA = 0, lastB = 0, examined = 0;
    const float ux = gA.ux;
    const float2 uy = make_float2(gA.uy, gB.uy);
    const float eps = o.t_eps, amax = o.alpha_max;
    // pixels that reached the count cap
    const uint32_t cmax = COUNT && o.max_per_pixel ? (uint32_t)o.max_per_pixel : 0xffffffffu;
    const uint32_t lt = lanemask_lt_r();
    uint32_t p = s;
    int qn = 0;
    uint32_t qh = 0;
    while (true) {
        bool act[NP];
        act[NP - 1] = !(T.y < eps) && cntB < cmax;
        act[0] = !(T.x < eps) && cntA < cmax;
        if (!__any_sync(0xffffffffu, act[0] || act[NP - 1])) break;
        queue_fill_front(keys, pv_list, s, e, bit, p, qn, qh, m.q, lane);
        if (qn == 0) break;
        uint32_t rel = 0, pv = 0;
        const int take = queue_take(m.q, qn, qh, lane, rel, pv);
        const bool valid = lane < take;
        float4 a = make_float4(0.f, 0.f, -1.f, 0.f), c = make_float4(0.f, 0.f, 0.f, 0.f);
        if (valid) {
            a = __ldg(rec + 2 * (size_t)pv);
            c = __ldg(rec + 2 * (size_t)pv + 1);
        }
        // every lane takes part in the reductions, whatever its entry
        const PixelGeom ar = active_rect_rows<NP>(g, act);
        const bool hit = valid && disc_meets_rect<FUSED>(a, ar);
        const uint32_t hm = __ballot_sync(0xffffffffu, hit);
        const int nh = __popc(hm);
        // the slots behind the hits are filled with points no pixel includes
        const int slot = hit ? __popc(hm & lt) : nh + __popc(~hm & lt);
        m.a[slot] = hit ? a : make_float4(0.f, 0.f, -1.f, 0.f);
        m.c[slot] = hit ? c : make_float4(0.f, 0.f, 0.f, 0.f);
        m.pos[slot] = rel;
        __syncwarp();
        if (COUNT) examined += (uint32_t)nh * ((uint32_t)act[0] + (uint32_t)(NP == 2 && act[NP - 1]));
        // the chunk's last composited hit of each pixel
        int jA = -1, jB = -1;
        constexpr int FWD_UNROLL = STORE ? 2 : 4;
        for (int j0 = 0; j0 < nh; j0 += FWD_UNROLL) {
#pragma unroll
            for (int u = 0; u < FWD_UNROLL; ++u) {
                const float4 aj = m.a[j0 + u], cj = m.c[j0 + u];
                float dx;
                float2 dy;
                const float2 d2 = pair_d2<FUSED>(ux, uy, aj.x, aj.y, dx, dy);
                bool inA = FUSED ? !(T.x < eps) & (d2.x <= aj.z) : d2.x <= aj.z && !(T.x < eps);
                bool inB = NP == 2 && (FUSED ? !(T.y < eps) & (d2.y <= aj.z)
                                             : d2.y <= aj.z && !(T.y < eps));
                if (COUNT) {
                    inA = inA && cntA < cmax;
                    inB = inB && cntB < cmax;
                }
                const float rawA = __fmul_rn(cj.x, ex2_approx(__fmul_rn(d2.x, aj.w)));
                const float rawB = NP == 2 ? __fmul_rn(cj.x, ex2_approx(__fmul_rn(d2.y, aj.w))) : 0.0f;
                if (STORE) {
                    if (inA) store_T(sto, pixA, cntA, T.x);
                    if (inB) store_T(sto, pixB, cntB, T.y);
                }
                const float2 wgt = mul2(make_float2(fminf(amax, rawA), fminf(amax, rawB)), T);
                if (inA) {
                    C0.x = fmaf(wgt.x, cj.y, C0.x);
                    C1.x = fmaf(wgt.x, cj.z, C1.x);
                    C2.x = fmaf(wgt.x, cj.w, C2.x);
                    T.x = __fsub_rn(T.x, wgt.x);
                    jA = j0 + u;
                    if (COUNT) ++cntA;
                }
                if (inB) {
                    C0.y = fmaf(wgt.y, cj.y, C0.y);
                    C1.y = fmaf(wgt.y, cj.z, C1.y);
                    C2.y = fmaf(wgt.y, cj.w, C2.y);
                    T.y = __fsub_rn(T.y, wgt.y);
                    jB = j0 + u;
                    if (COUNT) ++cntB;
                }
            }
        }
        if (jA >= 0) lastA = m.pos[jA] + 1;
        if (jB >= 0) lastB = m.pos[jB] + 1;
        __syncwarp(); // chunk consumed before the buffers are refilled
    }
    if (COUNT) {
        examined_acc += examined;
        composited_acc += cntA + cntB;
    }
    if (STORE) {
        if (gA.inside) sto.n[pixA] = cntA;
        if (NP == 2 && gB.inside) sto.n[pixB] = cntB;
    }
    write_pixel(gA, o, T.x, C0.x, C1.x, C2.x, lastA, out_rgb, T_final, n_contrib);
    if (NP == 2) write_pixel(gB, o, T.y, C0.y, C1.y, C2.y, lastB, out_rgb, T_final, n_contrib);
}

// ------------------------------------------------------------- backward
// Up to this many lanes with a contributing pixel add their terms (the sums
// over both their pixels) with their own vector atomics; more go through the
// transposed warp reduction, which costs some 35 instructions whatever the
// count, where the atomics cost L1 and L2 throughput per lane.  On the
// 1M-point, 64-view batch an earlier form of the loop took 10.13 ms at 24,
// 10.14 at 20, 10.61 at 28, 11.39 with the reduction for every point.
// Summing a batch of 8 or 16 hits at once instead (recursion terms to shared
// memory, then one lane per hit and column group) needed two atomics a hit
// and no reduction, but its shared-memory traffic made the L1 path the bound:
// 8.84-9.3 ms against 8.87.
constexpr int BWD_DIRECT_MAX = 24;
// One-pixel lanes: an earlier form of the loop took 13.0 ms at 12 and 16, 13.4
// at 20, 14.5 at 2 and 22.1 with atomics only on the same batch.
constexpr int BWD_DIRECT_MAX_ONE = 16;

// One warp's shared memory of the backward.
struct BwdWarp {
    float4 a[32], c[32]; // the chunk's hits: record halves
    uint2 ip[32];        // their list positions and point-views
    WarpQueue q;
};

// Adjoint state of one pixel: T after its last composited point, the colour
// behind (S, starting from the background term), dL/dC and the list length.
struct BwdPixel {
    float T, S, g0, g1, g2;
    uint32_t L;
};

__device__ __forceinline__ BwdPixel bwd_pixel(const PixelGeom &g, const DevOpts &o,
                                              const float *__restrict__ T_final,
                                              const uint32_t *__restrict__ n_contrib,
                                              const float *__restrict__ grad_rgb)
{
    BwdPixel p{1.0f, 0.f, 0.f, 0.f, 0.f, 0u};
    if (g.inside) {
        const int64_t pix = g.V->pix_base + (int64_t)g.y * g.V->W + g.x;
        p.T = T_final[pix];
        p.L = n_contrib[pix];
        p.g0 = grad_rgb[3 * pix];
        p.g1 = grad_rgb[3 * pix + 1];
        p.g2 = grad_rgb[3 * pix + 2];
    }
    p.S = p.T * (o.bg[0] * p.g0 + o.bg[1] * p.g1 + o.bg[2] * p.g2);
    return p;
}

// Adjoint state of a lane's two pixels (see BwdPixel), packed.
struct BwdPair {
    float2 T, S, g0, g1, g2;
    uint32_t LA, LB;
};

// What a point contributes to the recursions of a lane's two pixels before T
// and S enter: alpha, G and 1 / (1 - alpha) (0, 0 and 1 where the point was
// not composited; G 0 also where alpha is clamped, which has no geometry
// terms), and c.g.
struct PairAlpha {
    float2 alpha, G, rom, cg;
};

// tA, tB: whether the point was composited at the lane's pixels; d2: its
// squared distances.  CLAMP 0: the point's amplitude is below the clamp, so
// alpha is too.  Operands that are the point's own stay scalar (a packed
// operation would need them duplicated).
template <int NP, bool CLAMP>
__device__ __forceinline__ PairAlpha pair_alpha(bool tA, bool tB, float2 d2, const float4 a,
                                                const float4 c, float amax, const BwdPair &p)
{
    PairAlpha r;
    r.G.x = ex2_approx(__fmul_rn(d2.x, a.w));
    r.G.y = NP == 2 ? ex2_approx(__fmul_rn(d2.y, a.w)) : 0.0f;
    if (CLAMP) {
        const float rawA = c.x * r.G.x, rawB = c.x * r.G.y;
        r.alpha = make_float2(tA ? fminf(amax, rawA) : 0.0f, tB ? fminf(amax, rawB) : 0.0f);
        r.G = make_float2(tA && rawA < amax ? r.G.x : 0.0f, tB && rawB < amax ? r.G.y : 0.0f);
    } else {
        r.G = make_float2(tA ? r.G.x : 0.0f, tB ? r.G.y : 0.0f);
        r.alpha = make_float2(c.x * r.G.x, c.x * r.G.y);
    }
    const float2 om = fma2(r.alpha, f2(-1.0f), f2(1.0f));
    r.rom = make_float2(rcp_approx(om.x), NP == 2 ? rcp_approx(om.y) : 1.0f);
    r.cg = make_float2(fmaf(c.w, p.g2.x, fmaf(c.z, p.g1.x, c.y * p.g0.x)),
                       NP == 2 ? fmaf(c.w, p.g2.y, fmaf(c.z, p.g1.y, c.y * p.g0.y)) : 0.0f);
    return r;
}

// The recursions at one point and its terms summed over the lane's two
// pixels: v = {t0, t1, t2, do, dr, dg, db, 0}; updates T and S.  hasA /
// hasB: tb holds the stored transmittance before the point (store mode)
// instead of the one recovered by division.
template <int NP>
__device__ __forceinline__ void pair_recur(const PairAlpha &r, float2 d2, float dx, float2 dy,
                                           BwdPair &p, bool hasA, bool hasB, float2 tb, float v[8])
{
    float2 Tb = mul2(p.T, r.rom);
    if (hasA) Tb.x = tb.x;
    if (hasB) Tb.y = tb.y;
    const float2 w = mul2(r.alpha, Tb);
    const float2 sr = mul2(p.S, r.rom);
    const float2 dalpha = fma2(Tb, r.cg, make_float2(-sr.x, -sr.y));
    p.S = fma2(w, r.cg, p.S);
    p.T = Tb;
    const float2 dG = mul2(dalpha, r.G);
    const float2 t1 = mul2(dG, dy), t2 = mul2(dG, d2);
    const float2 t4 = mul2(w, p.g0), t5 = mul2(w, p.g1), t6 = mul2(w, p.g2);
    auto sum = [](float2 t) { return NP == 2 ? t.x + t.y : t.x; };
    v[3] = sum(dG);
    v[0] = v[3] * dx;
    v[1] = sum(t1);
    v[2] = sum(t2);
    v[4] = sum(t4);
    v[5] = sum(t5);
    v[6] = sum(t6);
    v[7] = 0.0f;
}

// Adds one point's terms to its slot of the gradient buffer; cm: the lanes
// with a contributing pixel.
template <int NP>
__device__ __forceinline__ void bwd_add(uint32_t cm, bool any, const float v[8], int lane,
                                        float *__restrict__ g2d, uint32_t pv)
{
    if (__popc(cm) > (NP == 2 ? BWD_DIRECT_MAX : BWD_DIRECT_MAX_ONE)) {
        warp_add_terms(v, lane, g2d, pv);
    } else if (any) { // few lanes: each adds its own terms
        float4 *dst = reinterpret_cast<float4 *>(g2d) + 2 * (size_t)pv;
        atomicAdd(dst, make_float4(v[0], v[1], v[2], v[3]));
        atomicAdd(dst + 1, make_float4(v[4], v[5], v[6], 0.f));
    }
}

// Back-propagates one chunk of nh staged hits through the lane's pixels.
template <int NP, bool CLAMP, bool STATS, bool STORE, bool FUSED>
__device__ __forceinline__ void bwd_chunk(const BwdWarp &m, int nh, float ux, float2 uy,
                                          float amax, int lane, BwdPair &p,
                                          float *__restrict__ g2d, uint32_t &examined,
                                          uint32_t &used, StoreRow &rowA, StoreRow &rowB)
{
    // two hits in flight: 363 against 368 us on the 4-view step; store mode's
    // list pointers leave no registers for it (526 against 585 us)
    constexpr int BWD_UNROLL = STORE ? 1 : 2;
    for (int j0 = 0; j0 < nh; j0 += BWD_UNROLL) {
        // BWD_UNROLL hits at a time: their loads and weights first, which do
        // not depend on one another, then the recursions
        PairAlpha pr[BWD_UNROLL];
        bool hasA[BWD_UNROLL], hasB[BWD_UNROLL], any[BWD_UNROLL];
        float2 tb[BWD_UNROLL], d2[BWD_UNROLL], dy[BWD_UNROLL];
        float dx[BWD_UNROLL];
        uint32_t pv[BWD_UNROLL];
#pragma unroll
        for (int u = 0; u < BWD_UNROLL; ++u) {
            const float4 aj = m.a[j0 + u], cj = m.c[j0 + u];
            const uint2 ip = m.ip[j0 + u];
            pv[u] = ip.y;
            d2[u] = pair_d2<FUSED>(ux, uy, aj.x, aj.y, dx[u], dy[u]);
            const bool bA = ip.x < p.LA, bB = NP == 2 && ip.x < p.LB;
            const bool tA = bA && d2[u].x <= aj.z, tB = bB && d2[u].y <= aj.z;
            if (STATS) {
                examined += (uint32_t)bA + (uint32_t)bB;
                used += (uint32_t)tA + (uint32_t)tB;
            }
            any[u] = tA || tB;
            hasA[u] = hasB[u] = false;
            tb[u] = f2(0.0f);
            if (STORE) {
                hasA[u] = row_next(rowA, tA, tb[u].x);
                if (NP == 2) hasB[u] = row_next(rowB, tB, tb[u].y);
            }
            pr[u] = pair_alpha<NP, CLAMP>(tA, tB, d2[u], aj, cj, amax, p);
        }
#pragma unroll
        for (int u = 0; u < BWD_UNROLL; ++u) {
            const uint32_t cm = __ballot_sync(0xffffffffu, any[u]);
            if (!cm) continue;
            float v[8];
            pair_recur<NP>(pr[u], d2[u], dx[u], dy[u], p, hasA[u], hasB[u], tb[u], v);
            bwd_add<NP>(cm, any[u], v, lane, g2d, pv[u]);
        }
    }
}

// Backward of one 8 x 8 block with first pixel (sx0, sy0) of view V by one
// warp: lane l owns the pixels A = (l & 7, l >> 3) and B = (l & 7, 4 + (l >>
// 3)).  The warp takes the tile list's entries with its block's bit (`bit`)
// from its queue, back to front, 32 at a time, and keeps those whose disc
// meets the rectangle of the pixels whose composited list reaches them; the
// records of the next 32 are in flight while these are processed.  Per hit
// the lane forms the adjoint at both pixels (packed fp32x2) and adds the two
// term vectors, so the per-point warp work serves 64 pixels.  s: the start
// of the tile's list.  NP: see fwd_pair_item.
template <int NP, bool STATS, bool STORE, bool FUSED>
__device__ __forceinline__ void bwd_pair_item(const DevView *V, int sx0, int sy0, uint32_t s,
                                              uint32_t bit, const DevOpts &o, int lane,
                                              const uint32_t *__restrict__ keys,
                                              const uint32_t *__restrict__ pv_list,
                                              const float4 *__restrict__ rec,
                                              const float *__restrict__ T_final,
                                              const uint32_t *__restrict__ n_contrib,
                                              const float *__restrict__ grad_rgb,
                                              float *__restrict__ g2d, uint32_t &examined,
                                              uint32_t &used, BwdWarp &m, const StoreBuf &sto)
{
    PixelGeom g[NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) g[q] = pixel_geom_at(V, sx0, sy0 + 4 * q, lane);
    const BwdPixel pa = bwd_pixel(g[0], o, T_final, n_contrib, grad_rgb);
    BwdPixel pb{1.0f, 0.f, 0.f, 0.f, 0.f, 0u};
    if (NP == 2) pb = bwd_pixel(g[NP - 1], o, T_final, n_contrib, grad_rgb);
    BwdPair p;
    p.T = make_float2(pa.T, pb.T);
    p.S = make_float2(pa.S, pb.S);
    p.g0 = make_float2(pa.g0, pb.g0);
    p.g1 = make_float2(pa.g1, pb.g1);
    p.g2 = make_float2(pa.g2, pb.g2);
    p.LA = pa.L;
    p.LB = pb.L;
    const uint32_t wmax = __reduce_max_sync(0xffffffffu, max(p.LA, p.LB));
    if (wmax == 0) return;
    // store mode: composited points not yet visited, per pixel
    StoreRow rowA, rowB;
    if (STORE) {
        rowA = store_row(sto, g[0].inside ? pixel_index(g[0]) : 0, g[0].inside);
        if (NP == 2)
            rowB = store_row(sto, g[NP - 1].inside ? pixel_index(g[NP - 1]) : 0, g[NP - 1].inside);
    }
    const uint32_t lt = lanemask_lt_r();
    const float ux = g[0].ux;
    const float2 uy = make_float2(g[0].uy, g[NP - 1].uy);
    int64_t c = (int64_t)((wmax - 1) & ~31u);
    int qn = 0;
    uint32_t qh = 0;
    uint32_t rel = 0, pv = 0;
    float4 ra = make_float4(0.f, 0.f, -1.f, 0.f), rc = ra;
    int take = 0;
    auto fetch = [&]() {
        queue_fill_back(keys, pv_list, s, wmax, bit, c, qn, qh, m.q, lane);
        take = qn > 0 ? queue_take(m.q, qn, qh, lane, rel, pv) : 0;
        if (lane < take) {
            ra = __ldg(rec + 2 * (size_t)pv);
            rc = __ldg(rec + 2 * (size_t)pv + 1);
        }
    };
    fetch();
    while (take > 0) {
        // pixels whose composited list reaches the chunk's nearest entry;
        // every lane takes part in the reductions, whatever its entry
        const uint32_t lowest = __shfl_sync(0xffffffffu, rel, take - 1);
        bool act[NP];
        act[NP - 1] = p.LB > lowest;
        act[0] = p.LA > lowest;
        const PixelGeom ar = active_rect_rows<NP>(g, act);
        const bool hit = lane < take && disc_meets_rect<FUSED>(ra, ar);
        const uint32_t hm = __ballot_sync(0xffffffffu, hit);
        // amplitudes that may reach the clamp (a NaN counts as one)
        const bool clamp = __any_sync(0xffffffffu, hit && !(rc.x < o.alpha_max));
        const int nh = __popc(hm);
        const int slot = hit ? __popc(hm & lt) : nh + __popc(~hm & lt);
        // the slots behind the hits are filled with points no pixel includes
        m.a[slot] = hit ? ra : make_float4(0.f, 0.f, -1.f, 0.f);
        m.c[slot] = rc;
        m.ip[slot] = make_uint2(rel, pv);
        __syncwarp();
        fetch();
        if (clamp)
            bwd_chunk<NP, true, STATS, STORE, FUSED>(m, nh, ux, uy, o.alpha_max, lane, p, g2d,
                                                 examined, used, rowA, rowB);
        else
            bwd_chunk<NP, false, STATS, STORE, FUSED>(m, nh, ux, uy, o.alpha_max, lane, p, g2d,
                                                  examined, used, rowA, rowB);
        __syncwarp(); // chunk consumed before the buffers are refilled
    }
}

// First pixel of unit `w` of a tile, and its block's bit in the pair keys'
// masks (0 when a tile is a single block).  NP 2: the units are the tile's 8 x
// 8 blocks, numbered like the masks' bits; NP 1: their upper and lower halves.
template <int TW, int TH, int NP>
__device__ __forceinline__ uint32_t unit_of(int tx, int ty, int w, int &sx0, int &sy0)
{
    const int blk = NP == 2 ? w : w >> 1;
    sx0 = tx * TW + (blk % (TW / 8)) * 8;
    sy0 = ty * TH + (blk / (TW / 8)) * 8 + (NP == 2 ? 0 : 4 * (w & 1));
    return block_bits(TW, TH) ? 1u << blk : 0u;
}

template <int TW, int TH, int NP>
__host__ __device__ constexpr int units()
{
    return TW * TH / (32 * NP);
}

// Warp-streamed: one block per tile, warp w takes the tile's unit w.
template <int TW, int TH, int NP, bool COUNT, bool STORE>
__global__ void __launch_bounds__(units<TW, TH, NP>() * 32)
raster_fwd_stream_kernel(Batch b, DevOpts o, const uint2 *__restrict__ ranges,
                         const uint32_t *__restrict__ keys, const uint32_t *__restrict__ pv_list,
                         const float4 *__restrict__ rec, float *__restrict__ out_rgb,
                         float *__restrict__ T_final, uint32_t *__restrict__ n_contrib,
                         unsigned long long *__restrict__ stats, StoreBuf sto)
{
    __shared__ FwdWarp s_fwd[units<TW, TH, NP>()];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const DevView *V = &b.views[find_view_by_tile(b, blockIdx.x)];
    const uint32_t local = blockIdx.x - V->tile_base;
    const int tx = (int)(local % (uint32_t)V->tiles_x), ty = (int)(local / (uint32_t)V->tiles_x);
    int sx0, sy0;
    const uint32_t bit = unit_of<TW, TH, NP>(tx, ty, w, sx0, sy0);
    const uint2 rg = ranges[blockIdx.x];
    uint32_t ex = 0, co = 0;
    fwd_pair_item<NP, COUNT, STORE, false>(V, sx0, sy0, rg.x, rg.y > rg.x ? rg.y : rg.x, bit, o,
                                           lane, keys, pv_list, rec, out_rgb, T_final, n_contrib,
                                           ex, co, s_fwd[w], sto);
    if (COUNT) add_stats(stats, ex, co, lane);
}

template <int TW, int TH, int NP, bool STATS, bool STORE>
__global__ void __launch_bounds__(units<TW, TH, NP>() * 32)
raster_bwd_stream_kernel(Batch b, DevOpts o, const uint2 *__restrict__ ranges,
                         const uint32_t *__restrict__ keys, const uint32_t *__restrict__ pv_list,
                         const float4 *__restrict__ rec, const float *__restrict__ T_final,
                         const uint32_t *__restrict__ n_contrib, const float *__restrict__ grad_rgb,
                         float *__restrict__ g2d, unsigned long long *__restrict__ stats,
                         StoreBuf sto)
{
    __shared__ BwdWarp s_bwd[units<TW, TH, NP>()];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const DevView *V = &b.views[find_view_by_tile(b, blockIdx.x)];
    const uint32_t local = blockIdx.x - V->tile_base;
    const int tx = (int)(local % (uint32_t)V->tiles_x), ty = (int)(local / (uint32_t)V->tiles_x);
    int sx0, sy0;
    const uint32_t bit = unit_of<TW, TH, NP>(tx, ty, w, sx0, sy0);
    uint32_t ex = 0, us = 0;
    bwd_pair_item<NP, STATS, STORE, false>(V, sx0, sy0, ranges[blockIdx.x].x, bit, o, lane, keys,
                                           pv_list, rec, T_final, n_contrib, grad_rgb, g2d, ex, us,
                                           s_bwd[w], sto);
    if (STATS) add_stats(stats ? stats + 2 : nullptr, ex, us, lane);
}

// ------------------------------------------------------------ persistent
// Persistent warps: each warp takes (tile, sub-block) items from an atomic
// counter over `order` (tiles sorted longest list first), so long tiles
// start early and no warp idles while work remains.
constexpr int PERSIST_THREADS = 256;
constexpr int BWD_PERSIST_BLOCKS = 4;
constexpr int FWD_PERSIST_BLOCKS = 5; // forward blocks per SM (see the kernel)

__device__ __forceinline__ uint32_t next_item(uint32_t *work, int lane)
{
    uint32_t it = 0;
    if (lane == 0) it = atomicAdd(work, 1u);
    return __shfl_sync(0xffffffffu, it, 0);
}

// Tile descriptor of the persistent order: {view, tx | ty << 16, list start,
// list end}, so that a warp starting an item needs one load, not a search
// of the view table, a division and the ranges.
__device__ __forceinline__ uint4 tile_desc(const Batch &b, const uint2 *ranges, uint32_t tile)
{
    const int v = find_view_by_tile(b, tile);
    const DevView &V = b.views[v];
    const uint32_t local = tile - V.tile_base;
    const uint32_t tx = local % (uint32_t)V.tiles_x, ty = local / (uint32_t)V.tiles_x;
    const uint2 r = ranges[tile];
    return make_uint4((uint32_t)v, tx | (ty << 16), r.x, r.y > r.x ? r.y : r.x);
}

// COUNT / STATS: count composited points and, with stats non-null, the
// examined / composited pairs; without, the loops carry no counting.  The
// forward's warps run five blocks per SM (48 registers): 4.05 ms on the
// 1M-point, 64-view step against 4.10 at four and 4.27 at six (unrolled by
// two).  The backward runs best at four (64 registers): 8.87 ms, 9.07 at
// three, 8.96 at five.
template <int TW, int TH, int NP, bool COUNT, bool STORE>
__global__ void __launch_bounds__(PERSIST_THREADS, FWD_PERSIST_BLOCKS)
raster_fwd_persist_kernel(Batch b, DevOpts o, const uint2 *__restrict__ ranges,
                          const uint32_t *__restrict__ keys, const uint32_t *__restrict__ pv_list,
                          const float4 *__restrict__ rec, float *__restrict__ out_rgb,
                          float *__restrict__ T_final, uint32_t *__restrict__ n_contrib,
                          unsigned long long *__restrict__ stats, const uint4 *__restrict__ order,
                          uint32_t *work, StoreBuf sto)
{
    constexpr uint32_t SUBS = units<TW, TH, NP>();
    constexpr int NW = PERSIST_THREADS / 32;
    __shared__ FwdWarp s_fwd[NW];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t n_items = b.n_tiles * SUBS;
    uint32_t ex = 0, co = 0;
    for (uint32_t it = next_item(work, lane); it < n_items; it = next_item(work, lane)) {
        const uint4 d = order[it / SUBS];
        const int sub = (int)(it % SUBS);
        int sx0, sy0;
        const uint32_t bit =
            unit_of<TW, TH, NP>((int)(d.y & 0xffffu), (int)(d.y >> 16), sub, sx0, sy0);
        fwd_pair_item<NP, COUNT, STORE, true>(&b.views[d.x], sx0, sy0, d.z, d.w, bit, o, lane,
                                              keys, pv_list, rec, out_rgb, T_final, n_contrib, ex,
                                              co, s_fwd[w], sto);
        __syncwarp(); // the item's shared memory is read before the next one writes it
    }
    if (COUNT) add_stats(stats, ex, co, lane);
}

template <int TW, int TH, int NP, bool STATS, bool STORE>
__global__ void __launch_bounds__(PERSIST_THREADS, BWD_PERSIST_BLOCKS)
raster_bwd_persist_kernel(Batch b, DevOpts o, const uint2 *__restrict__ ranges,
                          const uint32_t *__restrict__ keys, const uint32_t *__restrict__ pv_list,
                          const float4 *__restrict__ rec, const float *__restrict__ T_final,
                          const uint32_t *__restrict__ n_contrib,
                          const float *__restrict__ grad_rgb, float *__restrict__ g2d,
                          unsigned long long *__restrict__ stats, const uint4 *__restrict__ order,
                          uint32_t *work, StoreBuf sto)
{
    constexpr uint32_t SUBS = units<TW, TH, NP>();
    __shared__ BwdWarp s_bwd[PERSIST_THREADS / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t n_items = b.n_tiles * SUBS;
    uint32_t ex = 0, us = 0;
    for (uint32_t it = next_item(work, lane); it < n_items; it = next_item(work, lane)) {
        const uint4 d = order[it / SUBS];
        const int sub = (int)(it % SUBS);
        int sx0, sy0;
        const uint32_t bit =
            unit_of<TW, TH, NP>((int)(d.y & 0xffffu), (int)(d.y >> 16), sub, sx0, sy0);
        bwd_pair_item<NP, STATS, STORE, true>(&b.views[d.x], sx0, sy0, d.z, bit, o, lane, keys,
                                              pv_list, rec, T_final, n_contrib, grad_rgb, g2d, ex,
                                              us, s_bwd[w], sto);
        __syncwarp(); // the item's shared memory is read before the next one writes it
    }
    if (STATS) add_stats(stats ? stats + 2 : nullptr, ex, us, lane);
}

// Tile order, longest list first: bucket = floor(log2(length)), buckets in
// descending order (order inside a bucket is arbitrary; it only affects
// scheduling).  work[0] = forward item counter, work[1] = backward item
// counter, work[2..34) = bucket counts / offsets.
__global__ void tile_bucket_count_kernel(const uint2 *__restrict__ ranges, uint32_t n_tiles,
                                         uint32_t *work)
{
    __shared__ uint32_t s_c[32];
    if (threadIdx.x < 32) s_c[threadIdx.x] = 0;
    __syncthreads();
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n_tiles) {
        const uint2 r = ranges[t];
        const uint32_t len = r.y > r.x ? r.y - r.x : 0u;
        atomicAdd(&s_c[31 - (len ? __clz(len) : 31)], 1u);
    }
    __syncthreads();
    if (threadIdx.x < 32 && s_c[threadIdx.x]) atomicAdd(work + 2 + threadIdx.x, s_c[threadIdx.x]);
}

__global__ void tile_bucket_scan_kernel(uint32_t *work)
{
    if (threadIdx.x == 0) {
        work[0] = 0;
        work[1] = 0;
        uint32_t run = 0;
        for (int bkt = 31; bkt >= 0; --bkt) { // longest first
            const uint32_t c = work[2 + bkt];
            work[2 + bkt] = run;
            run += c;
        }
    }
}

// Stable inside a block: the block's tiles of one bucket keep their id
// order and take one contiguous range of the bucket (one atomic per block
// and bucket), so neighbouring tiles of similar length run close together
// in time and share their records through L2.
__global__ void __launch_bounds__(256)
tile_bucket_scatter_kernel(Batch b, const uint2 *__restrict__ ranges, uint32_t n_tiles,
                           uint32_t *work, uint4 *__restrict__ order)
{
    __shared__ uint32_t s_w[8][33]; // per warp and bucket: count, then offset
    __shared__ uint32_t s_base[32];
    const int w = threadIdx.x >> 5;
    for (int j = threadIdx.x; j < 8 * 33; j += 256) (&s_w[0][0])[j] = 0;
    __syncthreads();
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t bkt = 32; // none
    if (t < n_tiles) {
        const uint2 r = ranges[t];
        const uint32_t len = r.y > r.x ? r.y - r.x : 0u;
        bkt = 31 - (len ? __clz(len) : 31);
    }
    const uint32_t peers = __match_any_sync(0xffffffffu, bkt);
    const uint32_t rank = __popc(peers & lanemask_lt_r());
    if (bkt < 32 && rank == 0) s_w[w][bkt] = __popc(peers);
    __syncthreads();
    if (threadIdx.x < 32) {
        const int b = threadIdx.x;
        uint32_t run = 0;
        for (int v = 0; v < 8; ++v) {
            const uint32_t c = s_w[v][b];
            s_w[v][b] = run;
            run += c;
        }
        s_base[b] = run ? atomicAdd(work + 2 + b, run) : 0u;
    }
    __syncthreads();
    if (bkt < 32) order[s_base[bkt] + s_w[w][bkt] + rank] = tile_desc(b, ranges, t);
}

// ========================================================= block-staged
// Builds, in shared memory, the ascending list of batch entries whose cutoff
// disc reaches the warp's rectangle.  Returns the count.
__device__ __forceinline__ int warp_cull(const float4 *s_a, int nb, const PixelGeom &g,
                                         uint16_t *list, int lane)
{
    int cnt = 0;
    const uint32_t lt = lanemask_lt_r();
    for (int k0 = 0; k0 < nb; k0 += 32) {
        const int k = k0 + lane;
        const bool hit = k < nb && disc_meets_rect<false>(s_a[k], g);
        const uint32_t m = __ballot_sync(0xffffffffu, hit);
        if (hit) list[cnt + __popc(m & lt)] = (uint16_t)k;
        cnt += __popc(m);
    }
    __syncwarp();
    return cnt;
}

template <int TW, int TH>
__global__ void __launch_bounds__(TW * TH)
raster_fwd_staged_kernel(Batch b, DevOpts o, int depth, const uint2 *__restrict__ ranges,
                         const uint32_t *__restrict__ pv_list, const float4 *__restrict__ rec,
                         float *__restrict__ out_rgb, float *__restrict__ T_final,
                         uint32_t *__restrict__ n_contrib, unsigned long long *__restrict__ stats)
{
    constexpr int NT = TW * TH;
    extern __shared__ float4 s_rec[]; // [depth] a-part, [depth] b-part, per-warp lists
    float4 *s_a = s_rec, *s_b = s_rec + depth;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint16_t *s_list = (uint16_t *)(s_rec + 2 * depth) + w * depth;
    const uint32_t tile = blockIdx.x;
    const PixelGeom g = pixel_geom<TW, TH>(b, tile, w, lane);
    const uint2 rg = ranges[tile];
    const uint32_t s = rg.x, e = rg.y > rg.x ? rg.y : rg.x;

    float T = 1.0f, C0 = 0.f, C1 = 0.f, C2 = 0.f;
    uint32_t cnt = 0, last = 0, examined = 0;
    bool done = !g.inside;
    for (uint32_t base = s; base < e; base += depth) {
        if (__syncthreads_count(!done) == 0) break;
        const int nb = (int)min((uint32_t)depth, e - base);
        for (int k = threadIdx.x; k < nb; k += NT) {
            const uint32_t pv = pv_list[base + k];
            s_a[k] = rec[2 * (size_t)pv];
            s_b[k] = rec[2 * (size_t)pv + 1];
        }
        __syncthreads();
        if (!__any_sync(0xffffffffu, !done)) continue;
        const int nl = warp_cull(s_a, nb, g, s_list, lane);
        if (done) continue;
        int j = 0;
        for (; j < nl; ++j) {
            const int k = s_list[j];
            const float4 a = s_a[k];
            float dx, dy;
            const float d2 = pixel_d2(g.ux, g.uy, a.x, a.y, dx, dy);
            if (d2 <= a.z) {
                last = base + k - s + 1;
                if (pixel_blend(d2, a, s_b[k], o, T, C0, C1, C2, cnt)) {
                    done = true;
                    ++j;
                    break;
                }
            }
        }
        examined += j;
    }
    add_stats(stats, examined, cnt, lane);
    write_pixel(g, o, T, C0, C1, C2, last, out_rgb, T_final, n_contrib);
}

template <int TW, int TH>
__global__ void __launch_bounds__(TW * TH)
raster_bwd_staged_kernel(Batch b, DevOpts o, int depth, const uint2 *__restrict__ ranges,
                         const uint32_t *__restrict__ pv_list, const float4 *__restrict__ rec,
                         const float *__restrict__ T_final, const uint32_t *__restrict__ n_contrib,
                         const float *__restrict__ grad_rgb, float *__restrict__ g2d,
                         unsigned long long *__restrict__ stats)
{
    constexpr int NT = TW * TH;
    extern __shared__ float4 s_rec[];
    float4 *s_a = s_rec, *s_b = s_rec + depth;
    float *s_acc = (float *)(s_rec + 2 * depth); // [depth][8] block sums of the terms
    uint32_t *s_pv = (uint32_t *)(s_acc + 8 * depth);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint16_t *s_list = (uint16_t *)(s_pv + depth) + w * depth;
    __shared__ uint32_t s_max[NT / 32];
    const uint32_t tile = blockIdx.x;
    const PixelGeom g = pixel_geom<TW, TH>(b, tile, w, lane);
    const uint32_t s = ranges[tile].x;

    float T = 1.0f, g0 = 0.f, g1 = 0.f, g2 = 0.f;
    uint32_t L = 0;
    if (g.inside) {
        const int64_t pix = g.V->pix_base + (int64_t)g.y * g.V->W + g.x;
        T = T_final[pix];
        L = n_contrib[pix];
        g0 = grad_rgb[3 * pix];
        g1 = grad_rgb[3 * pix + 1];
        g2 = grad_rgb[3 * pix + 2];
    }
    float S = T * (o.bg[0] * g0 + o.bg[1] * g1 + o.bg[2] * g2);
    const uint32_t wmax = __reduce_max_sync(0xffffffffu, L);
    if (lane == 0) s_max[w] = wmax;
    __syncthreads();
    uint32_t maxL = 0;
#pragma unroll
    for (int j = 0; j < NT / 32; ++j) maxL = max(maxL, s_max[j]);

    uint32_t examined = 0, used = 0;
    for (int64_t bend = maxL; bend > 0; bend -= depth) {
        const uint32_t bstart = (uint32_t)(bend > depth ? bend - depth : 0);
        const int nb = (int)(bend - bstart);
        __syncthreads(); // previous batch fully consumed
        for (int k = threadIdx.x; k < nb; k += NT) {
            const uint32_t pv = pv_list[s + bstart + k];
            s_pv[k] = pv;
            s_a[k] = rec[2 * (size_t)pv];
            s_b[k] = rec[2 * (size_t)pv + 1];
            reinterpret_cast<float4 *>(s_acc)[2 * k] = make_float4(0.f, 0.f, 0.f, 0.f);
            reinterpret_cast<float4 *>(s_acc)[2 * k + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        __syncthreads();
        // warps whose pixels all stop before this batch skip it
        const int nwb = bstart < wmax ? (int)min((uint32_t)nb, wmax - bstart) : 0;
        const int nl = nwb > 0 ? warp_cull(s_a, nwb, g, s_list, lane) : 0;
        for (int j = nl - 1; j >= 0; --j) {
            const int k = s_list[j];
            float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            bool contrib = false;
            if (bstart + k < L) {
                ++examined;
                const float4 a = s_a[k];
                float dx, dy;
                const float d2 = pixel_d2(g.ux, g.uy, a.x, a.y, dx, dy);
                if (d2 <= a.z) {
                    contrib = true;
                    ++used;
                    pixel_adjoint(d2, dx, dy, a, s_b[k], o.alpha_max, g0, g1, g2, T, S, v);
                }
            }
            if (__any_sync(0xffffffffu, contrib)) {
                const float tot = warp_sum8_transposed(v, lane);
                const int which = (lane >> 2) & 7;
                if ((lane & 3) == 0 && which < 7) atomicAdd(s_acc + 8 * k + which, tot);
            }
        }
        __syncthreads();
        // one global atomic per (block, point, term)
        for (int t = threadIdx.x; t < nb * 7; t += NT) {
            const int k = t / 7, cc = t - 7 * k;
            const float val = s_acc[8 * k + cc];
            if (val != 0.f) atomicAdd(g2d + 8 * (size_t)s_pv[k] + cc, val);
        }
    }
    add_stats(stats ? stats + 2 : nullptr, examined, used, lane);
}

// ------------------------------------------------------------ dispatch
int persist_grid(const void *kernel)
{
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, PERSIST_THREADS, 0);
    return sms * (per_sm > 0 ? per_sm : 1);
}

template <int TW, int TH, int NP, bool COUNT, bool STORE>
void fwd_launch(const Batch &b, const DevOpts &o, const uint2 *ranges, const uint32_t *keys,
                const uint32_t *pv_list, const float4 *rec, float *out_rgb, float *T_final,
                uint32_t *n_contrib, unsigned long long *stats, const uint4 *order, uint32_t *work,
                cudaStream_t s, const StoreBuf &sto)
{
    if (order) {
        static const int grid =
            persist_grid((const void *)raster_fwd_persist_kernel<TW, TH, NP, COUNT, STORE>);
        raster_fwd_persist_kernel<TW, TH, NP, COUNT, STORE><<<grid, PERSIST_THREADS, 0, s>>>(
            b, o, ranges, keys, pv_list, rec, out_rgb, T_final, n_contrib, stats, order, work,
            sto);
    } else {
        raster_fwd_stream_kernel<TW, TH, NP, COUNT, STORE><<<b.n_tiles, units<TW, TH, NP>() * 32, 0, s>>>(
            b, o, ranges, keys, pv_list, rec, out_rgb, T_final, n_contrib, stats, sto);
    }
}

template <int TW, int TH, int NP, bool STATS, bool STORE>
void bwd_launch(const Batch &b, const DevOpts &o, const uint2 *ranges, const uint32_t *keys,
                const uint32_t *pv_list, const float4 *rec, const float *T_final,
                const uint32_t *n_contrib, const float *grad_rgb, float4 *g2d,
                unsigned long long *stats, const uint4 *order, uint32_t *work, cudaStream_t s,
                const StoreBuf &sto)
{
    if (order) {
        static const int grid =
            persist_grid((const void *)raster_bwd_persist_kernel<TW, TH, NP, STATS, STORE>);
        raster_bwd_persist_kernel<TW, TH, NP, STATS, STORE><<<grid, PERSIST_THREADS, 0, s>>>(
            b, o, ranges, keys, pv_list, rec, T_final, n_contrib, grad_rgb, (float *)g2d, stats,
            order, work + 1, sto);
    } else {
        raster_bwd_stream_kernel<TW, TH, NP, STATS, STORE><<<b.n_tiles, units<TW, TH, NP>() * 32, 0, s>>>(
            b, o, ranges, keys, pv_list, rec, T_final, n_contrib, grad_rgb, (float *)g2d, stats,
            sto);
    }
}

// The kernels are instantiated with and without pair counting (STATS, COUNT)
// and store mode (STORE, which counts too), so that the variants the graphs
// run carry neither; the count cap needs the forward's counting variant.
template <int TW, int TH>
void fwd_dispatch(const Batch &b, const DevOpts &o, int depth, const uint2 *ranges,
                  const uint32_t *keys, const uint32_t *pv_list, const float4 *rec,
                  float *out_rgb, float *T_final,
                  uint32_t *n_contrib, unsigned long long *stats, const uint4 *order,
                  uint32_t *work, cudaStream_t s, const StoreBuf &sto, bool two)
{
    const bool store = sto.T != nullptr;
    if (depth == 0) {
        const bool count = stats || o.max_per_pixel;
        auto f = two ? (store ? fwd_launch<TW, TH, 2, true, true>
                        : count ? fwd_launch<TW, TH, 2, true, false>
                                : fwd_launch<TW, TH, 2, false, false>)
                     : (store ? fwd_launch<TW, TH, 1, true, true>
                        : count ? fwd_launch<TW, TH, 1, true, false>
                                : fwd_launch<TW, TH, 1, false, false>);
        f(b, o, ranges, keys, pv_list, rec, out_rgb, T_final, n_contrib, stats, order, work, s,
          sto);
    } else {
        const size_t smem =
            (size_t)depth * (2 * sizeof(float4) + (TW * TH / 32) * sizeof(uint16_t));
        static const bool attr = cudaFuncSetAttribute(raster_fwd_staged_kernel<TW, TH>,
                                                      cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                      160 * 1024) == cudaSuccess;
        (void)attr;
        raster_fwd_staged_kernel<TW, TH><<<b.n_tiles, TW * TH, smem, s>>>(
            b, o, depth, ranges, pv_list, rec, out_rgb, T_final, n_contrib, stats);
    }
    count_launches(1);
}

template <int TW, int TH>
void bwd_dispatch(const Batch &b, const DevOpts &o, int depth, const uint2 *ranges,
                  const uint32_t *keys, const uint32_t *pv_list, const float4 *rec,
                  const float *T_final,
                  const uint32_t *n_contrib, const float *grad_rgb, float4 *g2d,
                  unsigned long long *stats, const uint4 *order, uint32_t *work,
                  cudaStream_t s, const StoreBuf &sto, bool two)
{
    const bool store = sto.T != nullptr;
    if (depth == 0) {
        auto f = two ? (store ? bwd_launch<TW, TH, 2, true, true>
                        : stats ? bwd_launch<TW, TH, 2, true, false>
                                : bwd_launch<TW, TH, 2, false, false>)
                     : (store ? bwd_launch<TW, TH, 1, true, true>
                        : stats ? bwd_launch<TW, TH, 1, true, false>
                                : bwd_launch<TW, TH, 1, false, false>);
        f(b, o, ranges, keys, pv_list, rec, T_final, n_contrib, grad_rgb, g2d, stats, order, work,
          s, sto);
    } else {
        const size_t smem = (size_t)depth * (4 * sizeof(float4) + sizeof(uint32_t) +
                                             (TW * TH / 32) * sizeof(uint16_t));
        static const bool attr = cudaFuncSetAttribute(raster_bwd_staged_kernel<TW, TH>,
                                                      cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                      160 * 1024) == cudaSuccess;
        (void)attr;
        raster_bwd_staged_kernel<TW, TH><<<b.n_tiles, TW * TH, smem, s>>>(
            b, o, depth, ranges, pv_list, rec, T_final, n_contrib, grad_rgb, (float *)g2d, stats);
    }
    count_launches(1);
}

} // namespace

void launch_tile_order(const Batch &b, const uint2 *ranges, uint32_t n_tiles, uint4 *order,
                       uint32_t *work, cudaStream_t s)
{
    cudaMemsetAsync(work, 0, 34 * sizeof(uint32_t), s);
    if (n_tiles == 0) return;
    const unsigned nb = (n_tiles + 255) / 256;
    tile_bucket_count_kernel<<<nb, 256, 0, s>>>(ranges, n_tiles, work);
    tile_bucket_scan_kernel<<<1, 32, 0, s>>>(work);
    tile_bucket_scatter_kernel<<<nb, 256, 0, s>>>(b, ranges, n_tiles, work, order);
    count_launches(3);
}

void reset_work_counters(uint32_t *work, cudaStream_t s)
{
    cudaMemsetAsync(work, 0, 2 * sizeof(uint32_t), s);
}

void launch_raster_fwd(const Batch &b, const DevOpts &o, int depth, const uint2 *ranges,
                       const uint32_t *keys, const uint32_t *pv_list, const float4 *rec,
                       float *out_rgb, float *T_final, uint32_t *n_contrib,
                       unsigned long long *stats, cudaStream_t s, bool two, const uint4 *order,
                       uint32_t *work, const StoreBuf &sto)
{
    if (b.n_tiles == 0) return;
    if (o.tile_w == 8 && o.tile_h == 8)
        fwd_dispatch<8, 8>(b, o, depth, ranges, keys, pv_list, rec, out_rgb, T_final, n_contrib,
                           stats, order, work, s, sto, two);
    else if (o.tile_w == 16 && o.tile_h == 32)
        fwd_dispatch<16, 32>(b, o, depth, ranges, keys, pv_list, rec, out_rgb, T_final,
                             n_contrib, stats, order, work, s, sto, two);
    else
        fwd_dispatch<16, 16>(b, o, depth, ranges, keys, pv_list, rec, out_rgb, T_final,
                             n_contrib, stats, order, work, s, sto, two);
}

void launch_raster_bwd(const Batch &b, const DevOpts &o, int depth, const uint2 *ranges,
                       const uint32_t *keys, const uint32_t *pv_list, const float4 *rec,
                       const float *T_final, const uint32_t *n_contrib, const float *grad_rgb,
                       float4 *g2d, unsigned long long *stats, cudaStream_t s, bool two,
                       const uint4 *order, uint32_t *work, const StoreBuf &sto)
{
    if (b.n_tiles == 0) return;
    if (o.tile_w == 8 && o.tile_h == 8)
        bwd_dispatch<8, 8>(b, o, depth, ranges, keys, pv_list, rec, T_final, n_contrib, grad_rgb,
                           g2d, stats, order, work, s, sto, two);
    else if (o.tile_w == 16 && o.tile_h == 32)
        bwd_dispatch<16, 32>(b, o, depth, ranges, keys, pv_list, rec, T_final, n_contrib,
                             grad_rgb, g2d, stats, order, work, s, sto, two);
    else
        bwd_dispatch<16, 16>(b, o, depth, ranges, keys, pv_list, rec, T_final, n_contrib,
                             grad_rgb, g2d, stats, order, work, s, sto, two);
}

} // namespace pbr
