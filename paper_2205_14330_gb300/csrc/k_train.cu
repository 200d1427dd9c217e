// Training objective and optimiser step of Sec. 3.3.
//
// loss_tv: per view image, L = sum (I_hat - I)^2 (or |I_hat - I|) +
// lambda * TV(I_hat), TV = l1 norm of forward differences along x and y
// per channel (anisotropic, no wrap-around), and dL/dI_hat with
// d|d|/dd = sign(d), sign(0) = 0; each forward difference is counted once, by
// its left / upper pixel.  One thread takes TV_ROWS pixels of a column of one
// channel: neighbouring threads read neighbouring floats, a value is loaded
// once for its column and twice (from L1) for its row's differences, all of a
// thread's loads are in flight together, and a pixel's place is found by one
// division per run.  One thread per pixel, with a 64-bit division each, its
// loads 12 bytes apart and a block per 256 pixels adding to the loss, took
// 60.6 us on four views of 800 x 800; this 34.5 (39.7 with two rows a thread,
// 35.8 with eight).
//
// optimizer: p <- p - lr g (SGD) or the bias-corrected Adam update, with the
// learning rate and the step number read from device memory so a captured
// training step can change them between replays (per-epoch decay).  Bound by
// memory (28 bytes an element): four elements a thread where the arrays allow
// 16-byte accesses, one otherwise: 15M elements
// (420 MB) 98 -> 74 us, 600k elements 8.2 -> 4.3.
#include <algorithm>

#include "pbr_internal.cuh"

namespace pbr {

namespace {

__device__ __forceinline__ float sgnf(float d) { return d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f); }

constexpr int TV_ROWS = 4;

__global__ void __launch_bounds__(256)
loss_tv_kernel(const DevView *__restrict__ views, int kind, float lam,
               const float *__restrict__ pred, const float *__restrict__ target,
               float *__restrict__ grad, double *loss)
{
    const DevView &V = views[blockIdx.y];
    const int H = V.H;
    const int64_t row = 3 * (int64_t)V.W; // floats
    const int64_t runs = row * (((int64_t)H + TV_ROWS - 1) / TV_ROWS);
    // compensated fp32 per thread, fp64 across threads: no per-element fp64
    float acc = 0.0f, comp = 0.0f;
    auto add = [&](float x) {
        const float y = __fsub_rn(x, comp);
        const float t = __fadd_rn(acc, y);
        comp = __fsub_rn(__fsub_rn(t, acc), y);
        acc = t;
    };
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < runs;
         r += (int64_t)gridDim.x * blockDim.x) {
        const int64_t run = runs <= 0xffffffffll ? (int64_t)((uint32_t)r / (uint32_t)row) : r / row;
        const int64_t x = r - run * row; // column, in floats
        const int y0 = (int)run * TV_ROWS;
        const int rows = min(TV_ROWS, H - y0);
        const int64_t q = 3 * V.pix_base + (int64_t)y0 * row + x;
        const bool tv_on = lam != 0.0f, left = tv_on && x >= 3, right = tv_on && x + 3 < row;
        float c[TV_ROWS + 2], t[TV_ROWS], l[TV_ROWS], rt[TV_ROWS];
#pragma unroll
        for (int i = 0; i < TV_ROWS + 2; ++i) {
            const bool in = i >= 1 && i <= rows;
            const bool edge = tv_on && (i == 0 ? y0 > 0 : i == rows + 1 && y0 + rows < H);
            c[i] = in || edge ? __ldg(pred + q + (i - 1) * row) : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < TV_ROWS; ++i) {
            t[i] = i < rows ? __ldg(target + q + i * row) : 0.0f;
            l[i] = i < rows && left ? __ldg(pred + q + i * row - 3) : 0.0f;
            rt[i] = i < rows && right ? __ldg(pred + q + i * row + 3) : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < TV_ROWS; ++i) {
            if (i >= rows) break;
            const float a = c[i + 1];
            const float d = a - t[i];
            float gv;
            if (kind == 0) {
                add(d * d);
                gv = 2.0f * d;
            } else {
                add(fabsf(d));
                gv = sgnf(d);
            }
            if (tv_on) {
                float tv = 0.0f;
                if (right) {
                    const float dx = rt[i] - a;
                    add(lam * fabsf(dx));
                    tv -= sgnf(dx);
                }
                if (left) tv += sgnf(a - l[i]);
                if (y0 + i + 1 < H) {
                    const float dy = c[i + 2] - a;
                    add(lam * fabsf(dy));
                    tv -= sgnf(dy);
                }
                if (y0 + i > 0) tv += sgnf(a - c[i]);
                gv += lam * tv;
            }
            grad[q + i * row] = gv;
        }
    }
    double tot = (double)acc - (double)comp;
    for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    __shared__ double s_w[32];
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = tot;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += s_w[w];
        if (t != 0.0) atomicAdd(loss, t);
    }
}

struct Rates {
    float lr, bc1, bc2;
};

__device__ __forceinline__ void update(const OptParams &prm, const Rates &r, float gi, float &p,
                                       float &m, float &v)
{
    const float mi = prm.beta1 * m + (1.0f - prm.beta1) * gi;
    const float vi = prm.beta2 * v + (1.0f - prm.beta2) * gi * gi;
    m = mi;
    v = vi;
    p -= r.lr * (mi / r.bc1) / (sqrtf(vi / r.bc2) + prm.eps);
}

// T: float, or float4 where all arrays are 16-byte aligned (n counts Ts).
template <typename T>
__global__ void __launch_bounds__(256)
optimizer_kernel(OptParams prm, const OptState *__restrict__ dev, int group, T *__restrict__ p,
                 const T *__restrict__ g, T *__restrict__ m, T *__restrict__ v, int64_t n)
{
    Rates r;
    r.lr = prm.lr;
    int t = prm.step;
    if (dev) {
        r.lr = dev->lr[group];
        t = dev->step;
    }
    if (r.lr == 0.0f) return;
    r.bc1 = 1.0f - powf(prm.beta1, (float)t);
    r.bc2 = 1.0f - powf(prm.beta2, (float)t);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const T gi = g[i];
        T pi = p[i];
        if constexpr (sizeof(T) == sizeof(float)) {
            if (prm.kind == 0) {
                pi -= r.lr * gi;
            } else {
                T mi = m[i], vi = v[i];
                update(prm, r, gi, pi, mi, vi);
                m[i] = mi;
                v[i] = vi;
            }
        } else {
            if (prm.kind == 0) {
                pi.x -= r.lr * gi.x;
                pi.y -= r.lr * gi.y;
                pi.z -= r.lr * gi.z;
                pi.w -= r.lr * gi.w;
            } else {
                T mi = m[i], vi = v[i];
                update(prm, r, gi.x, pi.x, mi.x, vi.x);
                update(prm, r, gi.y, pi.y, mi.y, vi.y);
                update(prm, r, gi.z, pi.z, mi.z, vi.z);
                update(prm, r, gi.w, pi.w, mi.w, vi.w);
                m[i] = mi;
                v[i] = vi;
            }
        }
        p[i] = pi;
    }
}

template <typename T>
void run_optimizer(const OptParams &prm, const OptState *dev, int group, float *p, const float *g,
                   float *m, float *v, int64_t n, cudaStream_t s)
{
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, 152 * 16);
    optimizer_kernel<T><<<(unsigned)blocks, 256, 0, s>>>(prm, dev, group, (T *)p, (const T *)g,
                                                         (T *)m, (T *)v, n);
    count_launches(1);
}

__global__ void step_counter_kernel(OptState *dev) { dev->step += 1; }

} // namespace

void launch_loss_tv(const DevView *views, int n_views, int64_t max_pix, int kind, float lam,
                    const float *pred, const float *target, float *grad, double *loss,
                    cudaStream_t s)
{
    if (n_views <= 0 || max_pix <= 0) return;
    // a pass or a few over the GPU: every block ends in an fp64 atomic on one
    // address.  Views differ in size, so the blocks are not divided among all.
    const int64_t runs = (3 * max_pix + TV_ROWS - 1) / TV_ROWS;
    const int64_t bx = std::min<int64_t>((runs + 255) / 256, 152 * 8 / std::min(n_views, 4));
    loss_tv_kernel<<<dim3((unsigned)bx, (unsigned)n_views), 256, 0, s>>>(views, kind, lam, pred,
                                                                          target, grad, loss);
    count_launches(1);
}

void launch_optimizer(const OptParams &prm, const OptState *dev, int group, float *p,
                      const float *g, float *m, float *v, int64_t n, cudaStream_t s)
{
    if (n <= 0) return;
    const uintptr_t at = (uintptr_t)p | (uintptr_t)g | (uintptr_t)m | (uintptr_t)v;
    const int64_t quads = at % 16 == 0 ? n / 4 : 0, rest = n - 4 * quads;
    if (quads) run_optimizer<float4>(prm, dev, group, p, g, m, v, quads, s);
    if (rest) {
        const int64_t o = 4 * quads;
        run_optimizer<float>(prm, dev, group, p + o, g + o, m ? m + o : m, v ? v + o : v, rest, s);
    }
}

void launch_step_counter(OptState *dev, cudaStream_t s)
{
    step_counter_kernel<<<1, 1, 0, s>>>(dev);
    count_launches(1);
}

} // namespace pbr
