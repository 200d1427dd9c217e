// C entry points of the visual-hull initialisation and the consistency
// check (Sec. 3.1 and the appendix).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "api_internal.h"

using namespace pbr;

namespace {

constexpr uint64_t SH_STREAM = 0x5DEECE66Dull; // SH draws: stream seed ^ this

// Views of the check on the device, `zeros` words of 0 behind them; validates
// cameras and z_near.
int upload_views(TempBufs &tb, const pbr_camera *cams, int32_t n_cams, float z_near,
                 HullView **d_views, cudaStream_t s, int zeros = 0)
{
    if (!cams || n_cams < 1 || !(z_near >= 0.0f) || !std::isfinite(z_near))
        return set_error(PBR_ERR_INVALID_ARG, "consistency check: bad cameras or z_near");
    const size_t bytes = sizeof(HullView) * n_cams + sizeof(uint32_t) * zeros;
    std::vector<HullView> v((bytes + sizeof(HullView) - 1) / sizeof(HullView));
    std::memset(v.data(), 0, sizeof(HullView) * v.size());
    int64_t base = 0;
    for (int i = 0; i < n_cams; ++i) {
        const pbr_camera &c = cams[i];
        if (c.width <= 0 || c.height <= 0)
            return set_error(PBR_ERR_INVALID_ARG, "camera %d: size", i);
        HullView &h = v[i];
        h.fx = c.fx;
        h.fy = c.fy;
        h.cx = c.cx;
        h.cy = c.cy;
        for (int k = 0; k < 9; ++k) h.R[k] = c.R[k];
        for (int k = 0; k < 3; ++k) h.t[k] = c.t[k];
        h.W = c.width;
        h.H = c.height;
        h.pix_base = base;
        base += (int64_t)c.width * c.height;
    }
    PBR_TRY(tb.alloc(d_views, bytes));
    upload_small(*d_views, v.data(), bytes, s);
    return PBR_OK;
}

int read_u64(const unsigned long long *dev, unsigned long long *out, cudaStream_t s)
{
    PBR_CUDA(cudaMemcpyAsync(out, dev, sizeof(*out), cudaMemcpyDeviceToHost, s));
    PBR_CUDA(cudaStreamSynchronize(s));
    return PBR_OK;
}

} // namespace

extern "C" int pbr_consistency_check(pbr_ctx *ctx, const float *pos, int64_t n,
                                     const pbr_camera *cams, int32_t n_cams,
                                     const uint8_t *masks, float z_near, uint8_t *keep,
                                     pbr_stream_t stream)
{
    if (!ctx || n < 0 || (n > 0 && (!pos || !masks || !keep)))
        return set_error(PBR_ERR_INVALID_ARG, "pbr_consistency_check: bad arguments");
    if (n == 0) return PBR_OK;
    cudaStream_t s = (cudaStream_t)stream;
    PBR_CUDA(cudaSetDevice(ctx->device));
    TempBufs tb(s);
    HullView *views;
    PBR_TRY(upload_views(tb, cams, n_cams, z_near, &views, s));
    launch_consistency(pos, n, views, n_cams, masks, z_near, keep, nullptr, s);
    PBR_CUDA(cudaGetLastError());
    return PBR_OK;
}

extern "C" int pbr_consistency_filter(pbr_ctx *ctx, const pbr_points *in, const pbr_camera *cams,
                                      int32_t n_cams, const uint8_t *masks, float z_near,
                                      float *out_pos, float *out_sh, float *out_opacity,
                                      float *out_radius, int64_t *n_out, pbr_stream_t stream)
{
    if (!ctx || !in || !n_out || in->n < 0 || in->n > 0x7fffffffLL || in->sh_degree < 0 ||
        in->sh_degree > 3)
        return set_error(PBR_ERR_INVALID_ARG, "pbr_consistency_filter: bad arguments");
    *n_out = 0;
    const int64_t n = in->n;
    if (n == 0) return PBR_OK;
    if (!in->pos || !in->sh || !in->opacity || !in->radius || !masks || !out_pos || !out_sh ||
        !out_opacity || !out_radius)
        return set_error(PBR_ERR_INVALID_ARG, "pbr_consistency_filter: null array");
    cudaStream_t s = (cudaStream_t)stream;
    PBR_CUDA(cudaSetDevice(ctx->device));
    const int nsh = 3 * (in->sh_degree + 1) * (in->sh_degree + 1);
    TempBufs tb(s);
    HullView *views;
    PBR_TRY(upload_views(tb, cams, n_cams, z_near, &views, s));
    uint32_t *keep, *newpos;
    void *stmp;
    unsigned long long *tot;
    PBR_TRY(tb.alloc(&keep, sizeof(uint32_t) * n));
    PBR_TRY(tb.alloc(&newpos, sizeof(uint32_t) * n));
    PBR_TRY(tb.alloc(&stmp, scan_temp_bytes(n)));
    PBR_TRY(tb.alloc(&tot, sizeof(unsigned long long)));
    launch_consistency(in->pos, n, views, n_cams, masks, z_near, nullptr, keep, s);
    launch_exclusive_scan(keep, newpos, n, tot, stmp, s);
    launch_compact_points(keep, newpos, n,
                          PointArrays{in->pos, in->sh, in->opacity, in->radius, nsh},
                          PointArraysOut{out_pos, out_sh, out_opacity, out_radius, nsh}, s);
    unsigned long long m = 0;
    PBR_TRY(read_u64(tot, &m, s));
    *n_out = (int64_t)m;
    PBR_CUDA(cudaGetLastError());
    return PBR_OK;
}

extern "C" int pbr_visual_hull_init(pbr_ctx *ctx, const float lo[3], const float hi[3],
                                    const pbr_camera *cams, int32_t n_cams, const uint8_t *masks,
                                    float z_near, uint64_t seed, int64_t n_target,
                                    int64_t max_candidates, int32_t sh_degree, float *out_pos,
                                    float *out_sh, int64_t *n_out, int64_t *n_drawn,
                                    pbr_stream_t stream)
{
    if (!ctx || !lo || !hi || !masks || !n_out || !n_drawn || n_target < 0 ||
        n_target > 0x7fffffffLL || max_candidates < 0 || sh_degree < 0 || sh_degree > 3 ||
        (n_target > 0 && !out_pos))
        return set_error(PBR_ERR_INVALID_ARG, "pbr_visual_hull_init: bad arguments");
    float ext[3];
    for (int a = 0; a < 3; ++a) {
        if (!std::isfinite(lo[a]) || !std::isfinite(hi[a]) || !(hi[a] >= lo[a]))
            return set_error(PBR_ERR_INVALID_ARG, "pbr_visual_hull_init: bad box");
        ext[a] = hi[a] - lo[a];
    }
    *n_out = 0;
    *n_drawn = 0;
    if (max_candidates == 0) max_candidates = 1ll << 40;
    cudaStream_t s = (cudaStream_t)stream;
    PBR_CUDA(cudaSetDevice(ctx->device));
    TempBufs tb(s);
    HullView *views;
    PBR_TRY(upload_views(tb, cams, n_cams, z_near, &views, s, HULL_CHUNKS));
    // Batches of candidates in counter order; the first n_target accepted.
    // A batch costs a host synchronisation, candidates beyond the last one
    // taken cost their draws, but for those the kernel sees to be beyond it: the
    // first batch allows for one candidate in 32 accepted, the next ones for the
    // share seen so far and a little more.
    constexpr int64_t BATCH = HULL_BATCH, LEAST = 1ll << 16;
    auto sized = [&](double want) {
        const int64_t c = want < (double)BATCH ? (int64_t)want : BATCH;
        return std::max(LEAST, (c + 4 * HULL_BLOCK - 1) / (4 * HULL_BLOCK) * (4 * HULL_BLOCK));
    };
    int64_t size = sized(32.0 * (double)n_target);
    unsigned long long *result; // and counts, bits: one allocation
    PBR_TRY(tb.alloc(&result, 2 * sizeof(unsigned long long) +
                                  sizeof(uint32_t) * (BATCH / HULL_BLOCK) + BATCH / 8));
    uint32_t *counts = (uint32_t *)(result + 2), *bits = counts + BATCH / HULL_BLOCK,
             *found = (uint32_t *)(views + n_cams);
    int64_t done = 0, drawn = 0;
    while (done < n_target && drawn < max_candidates) {
        const int64_t cnt = std::min<int64_t>(size, max_candidates - drawn);
        const uint32_t need = (uint32_t)(n_target - done);
        launch_hull_batch(seed, (uint64_t)drawn, cnt, lo, ext, views, n_cams, masks, z_near, bits,
                          counts, found, need, out_pos, done, result, s);
        unsigned long long got[2] = {0, 0};
        PBR_CUDA(cudaMemcpyAsync(got, result, sizeof got, cudaMemcpyDeviceToHost, s));
        PBR_CUDA(cudaStreamSynchronize(s));
        if ((int64_t)got[0] >= (int64_t)need) {
            drawn += (int64_t)got[1] + 1;
            done = n_target;
        } else {
            drawn += cnt;
            done += (int64_t)got[0];
            size = done > 0 ? sized(1.05 * (double)(n_target - done) * (double)drawn / (double)done)
                            : BATCH;
        }
    }
    // SH of the kept points: standard normals
    if (out_sh && done > 0) {
        const int64_t coef = 3ll * (sh_degree + 1) * (sh_degree + 1);
        launch_sh_normals(seed ^ SH_STREAM, done * coef, out_sh, s);
    }
    *n_out = done;
    *n_drawn = drawn;
    PBR_CUDA(cudaGetLastError());
    PBR_CUDA(cudaStreamSynchronize(s));
    return PBR_OK;
}
