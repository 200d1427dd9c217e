// Visual-hull initialisation and consistency check (Sec. 3.1 and the
// appendix): a point is consistent when its projection (Eq. 1) lands on a
// foreground pixel of every view's mask; the initial cloud is the first
// n_target consistent points of a counter-based uniform stream over the
// scene box, with SH coefficients drawn from N(0, 1).
//
// Projection in fp32 round-to-nearest with the renderer's operation order:
// X = ((R0 px + R1 py) + R2 pz) + t per row, u = fx (X.x / X.z) + cx; pixel
// (floor u, floor v); behind z_near or outside the image = background.
// Random numbers: SplitMix64 (Steele, Lea and Flood, OOPSLA 2014), output i
// of stream s = finaliser of s + (i + 1) * 0x9E3779B97F4A7C15; uniforms are
// the top 24 bits times 2^-24.
#include "pbr_internal.cuh"

namespace pbr {

namespace {

__device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t i)
{
    uint64_t z = seed + (i + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ float uniform24(uint64_t z)
{
    return (float)(uint32_t)(z >> 40) * 5.9604644775390625e-8f; // 2^-24, exact
}

// Whether the point lands on a foreground pixel of every view in [v0, v1).
__device__ __forceinline__ bool consistent(float px, float py, float pz,
                                           const HullView *__restrict__ views, int v0, int v1,
                                           const uint8_t *__restrict__ masks, float z_near)
{
    for (int v = v0; v < v1; ++v) {
        const HullView &V = views[v];
        float X[3];
#pragma unroll
        for (int r = 0; r < 3; ++r)
            X[r] = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(V.R[3 * r], px),
                                                  __fmul_rn(V.R[3 * r + 1], py)),
                                       __fmul_rn(V.R[3 * r + 2], pz)),
                             V.t[r]);
        if (!(X[2] > z_near)) return false;
        const float u = __fadd_rn(__fmul_rn(V.fx, __fdiv_rn(X[0], X[2])), V.cx);
        const float w = __fadd_rn(__fmul_rn(V.fy, __fdiv_rn(X[1], X[2])), V.cy);
        if (!(u >= 0.0f && w >= 0.0f && u < (float)V.W && w < (float)V.H)) return false;
        const int64_t x = (int64_t)floorf(u), y = (int64_t)floorf(w);
        if (__ldg(masks + V.pix_base + y * V.W + x) == 0) return false;
    }
    return true;
}

__global__ void __launch_bounds__(256)
cc_flags_kernel(const float *__restrict__ pos, int64_t n, const HullView *__restrict__ views,
                int nv, const uint8_t *__restrict__ masks, float z_near,
                uint8_t *__restrict__ flags8, uint32_t *__restrict__ flags32)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const bool ok = consistent(pos[3 * i], pos[3 * i + 1], pos[3 * i + 2], views, 0, nv, masks,
                                   z_near);
        if (flags8) flags8[i] = ok ? 1 : 0;
        if (flags32) flags32[i] = ok ? 1u : 0u;
    }
}

// Position of candidate j of stream `seed` in the box.
struct HullBox {
    uint64_t seed;
    float lo[3], ex[3];
};

__device__ __forceinline__ void candidate(const HullBox &b, uint64_t j, float p[3])
{
#pragma unroll
    for (int a = 0; a < 3; ++a)
        p[a] = __fadd_rn(__fmul_rn(b.ex[a], uniform24(splitmix64(b.seed, 3 * j + a))), b.lo[a]);
}

// Acceptance of HB candidates per block, as a bit each (candidate i
// of the batch in bit i & 31 of word i / 32) and a count per block.
// A warp of candidates runs until its last one fails, so testing every view
// at once keeps a warp for all views while a few lanes live (196 us for 4 M
// candidates and 16 views).  The views are taken in groups of 1, 1, 2, 4, ...
// instead, the survivors of each group packed into a shared queue, so that
// the next group runs with full warps; a survivor's position is drawn again
// (kept in shared memory it cost occupancy: 95 -> 127 us for 6.4 M
// candidates).  Bound by issue (three draws a candidate, two exact divisions
// a test) and by the latency of the mask reads.
// The batch allows for few accepted; where the masks take more, the blocks that
// start after `need` have been found among lower candidates test none: found[c]
// adds up what the blocks of chunk c accepted, and a block looks at the chunks
// below its own.  The blocks that start at once stay: 2,048 candidates a block keep
// them few (4,096: 307 us a call as 2,048 on 8.6 M candidates of which one in 54 is
// accepted), 1,024 in batches below HULL_FEW, which last as long as one block.
// 500k points, every candidate accepted, 16 views, a first batch of 16 M: 1647 ->
// 489 us.
constexpr int HULL_THREADS = 256;

template <int HB>
__global__ void __launch_bounds__(HULL_THREADS)
hull_accept_kernel(HullBox box, uint64_t first, int64_t count, const HullView *__restrict__ views,
                   int nv, const uint8_t *__restrict__ masks, float z_near,
                   uint32_t need, uint32_t *__restrict__ bits, uint32_t *__restrict__ counts,
                   uint32_t *found)
{
    __shared__ uint16_t s_q[2][HB];
    __shared__ uint32_t s_bits[HB / 32];
    __shared__ uint32_t s_n[2];
    __shared__ bool s_enough;
    const int64_t base = (int64_t)blockIdx.x * HB;
    const int lane = threadIdx.x & 31;
    for (int j = threadIdx.x; j < HB / 32; j += HULL_THREADS) s_bits[j] = 0;
    if (threadIdx.x < 2) s_n[threadIdx.x] = 0;
    const uint32_t chunk = blockIdx.x / HULL_CHUNK;
    if (threadIdx.x < 32) {
        const uint32_t below = __reduce_add_sync(
            0xffffffffu, (uint32_t)lane < chunk ? __ldcg(found + lane) : 0u);
        if (lane == 0) s_enough = below >= need;
    }
    __syncthreads();
    if (s_enough) { // its candidates' ranks are all beyond `need`
        if (threadIdx.x == 0) counts[blockIdx.x] = 0;
        return;
    }
    int n = (int)(count - base < HB ? count - base : HB);
    int cur = 0;
    bool all = true; // the first group tests every candidate, without a queue
    for (int v0 = 0; v0 < nv && n > 0;) {
        const int v1 = v0 < 2 ? v0 + 1 : (2 * v0 < nv ? 2 * v0 : nv);
        for (int q0 = 0; q0 < n; q0 += HULL_THREADS) {
            const int q = q0 + (int)threadIdx.x;
            bool ok = false;
            uint32_t i = 0;
            if (q < n) {
                i = all ? (uint32_t)q : s_q[cur][q];
                float p[3];
                candidate(box, first + (uint64_t)base + i, p);
                ok = consistent(p[0], p[1], p[2], views, v0, v1, masks, z_near);
            }
            const uint32_t m = __ballot_sync(0xffffffffu, ok);
            uint32_t at = 0;
            if (lane == 0 && m) at = atomicAdd(&s_n[cur ^ 1], (uint32_t)__popc(m));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (ok) s_q[cur ^ 1][at + __popc(m & ((1u << lane) - 1u))] = (uint16_t)i;
        }
        __syncthreads();
        cur ^= 1;
        n = (int)s_n[cur];
        if (threadIdx.x == 0) s_n[cur ^ 1] = 0;
        __syncthreads();
        all = false;
        v0 = v1;
    }
    for (int q = threadIdx.x; q < n; q += HULL_THREADS) {
        const uint32_t i = all ? (uint32_t)q : s_q[cur][q];
        atomicOr(&s_bits[i >> 5], 1u << (i & 31));
    }
    __syncthreads();
    for (int j = threadIdx.x; j < HB / 32; j += HULL_THREADS)
        bits[(int64_t)blockIdx.x * (HB / 32) + j] = s_bits[j];
    if (threadIdx.x == 0) {
        counts[blockIdx.x] = (uint32_t)n;
        if (n) atomicAdd(found + chunk, (uint32_t)n);
    }
}

// One block: exclusive scan of the nb block counts in place, out[0] = total; found
// is 0 again.
__global__ void __launch_bounds__(1024)
hull_scan_kernel(uint32_t *counts, int nb, uint32_t *found, unsigned long long *out)
{
    __shared__ uint32_t s_w[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t run = 0;
    for (int base = 0; base < nb; base += 1024) {
        const int i = base + (int)threadIdx.x;
        const uint32_t v = i < nb ? counts[i] : 0u;
        uint32_t inc = v;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) s_w[w] = inc;
        __syncthreads();
        if (w == 0) {
            uint32_t x = s_w[lane];
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += t;
            }
            s_w[lane] = x;
        }
        __syncthreads();
        if (i < nb) counts[i] = run + inc - v + (w > 0 ? s_w[w - 1] : 0u);
        run += s_w[31];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = run;
    if (threadIdx.x < HULL_CHUNKS) found[threadIdx.x] = 0;
}

// Accepted candidates of rank < need go to out[done + rank]; the candidate
// of rank need - 1 reports its index.  One thread per word of bits.
template <int HB>
__global__ void __launch_bounds__(HB / 32)
hull_take_kernel(HullBox box, uint64_t first, const uint32_t *__restrict__ bits,
                 const uint32_t *__restrict__ offsets, uint32_t need, float *__restrict__ out,
                 int64_t done, unsigned long long *last)
{
    constexpr int WORDS = HB / 32;
    __shared__ uint32_t s_w[WORDS / 32];
    if (offsets[blockIdx.x] >= need) return; // whole block (untested ones among them)
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t word = (int64_t)blockIdx.x * WORDS + threadIdx.x;
    uint32_t m = bits[word];
    const uint32_t c = (uint32_t)__popc(m);
    uint32_t inc = c;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) s_w[w] = inc;
    __syncthreads();
    uint32_t k = offsets[blockIdx.x] + inc - c;
    for (int j = 0; j < w; ++j) k += s_w[j];
    for (; m && k < need; m &= m - 1, ++k) {
        const uint64_t i = 32ull * (uint64_t)word + (uint64_t)(__ffs(m) - 1);
        float p[3];
        candidate(box, first + i, p);
        float *dst = out + 3 * (done + k);
        dst[0] = p[0];
        dst[1] = p[1];
        dst[2] = p[2];
        if (k == need - 1) *last = i;
    }
}

// Standard normals for the flattened [points, coefficients] array, Box-Muller
// on stream seed: coefficients 2p and 2p + 1 are the cosine and the sine of
// pair p, from outputs 2p and 2p + 1; one thread per pair.  fp32 (logf,
// sincospif): no decision depends on these values, and fp64 transcendentals
// run at a small fraction of the fp32 rate on this GPU.  u1 and u2 are exact
// in fp32 (24-bit integers times 2^-24).
__global__ void sh_normals_kernel(uint64_t seed, int64_t count, float *__restrict__ out)
{
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; 2 * p < count;
         p += (int64_t)gridDim.x * blockDim.x) {
        const float u1 =
            ((float)(uint32_t)(splitmix64(seed, 2 * (uint64_t)p) >> 40) + 1.0f) * 0x1p-24f;
        const float u2 = (float)(uint32_t)(splitmix64(seed, 2 * (uint64_t)p + 1) >> 40) * 0x1p-24f;
        const float r = sqrtf(-2.0f * logf(u1));
        float sn, cs;
        sincospif(2.0f * u2, &sn, &cs);
        out[2 * p] = r * cs;
        if (2 * p + 1 < count) out[2 * p + 1] = r * sn;
    }
}

unsigned grid_of(int64_t n)
{
    int64_t b = (n + 255) / 256;
    if (b < 1) b = 1;
    if (b > 152 * 32) b = 152 * 32;
    return (unsigned)b;
}

} // namespace

void launch_consistency(const float *pos, int64_t n, const HullView *views, int nv,
                        const uint8_t *masks, float z_near, uint8_t *flags8, uint32_t *flags32,
                        cudaStream_t s)
{
    if (n <= 0) return;
    cc_flags_kernel<<<grid_of(n), 256, 0, s>>>(pos, n, views, nv, masks, z_near, flags8, flags32);
    count_launches(1);
}

namespace {

constexpr int64_t HULL_FEW = 1ll << 21;
static_assert(HULL_BATCH / (2 * HULL_BLOCK) <= HULL_CHUNK * HULL_CHUNKS &&
                  HULL_FEW / HULL_BLOCK <= HULL_CHUNK * HULL_CHUNKS && HULL_CHUNKS <= 32,
              "a lane per chunk");

template <int HB>
void run_batch(const HullBox &box, uint64_t first, int64_t count, const HullView *views, int nv,
               const uint8_t *masks, float z_near, uint32_t *bits, uint32_t *counts,
               uint32_t *found, uint32_t need, float *out, int64_t done,
               unsigned long long *result, cudaStream_t s)
{
    const unsigned nb = (unsigned)((count + HB - 1) / HB);
    hull_accept_kernel<HB><<<nb, HULL_THREADS, 0, s>>>(box, first, count, views, nv, masks, z_near,
                                                       need, bits, counts, found);
    hull_scan_kernel<<<1, 1024, 0, s>>>(counts, (int)nb, found, result);
    hull_take_kernel<HB><<<nb, HB / 32, 0, s>>>(box, first, bits, counts, need, out, done,
                                                result + 1);
    count_launches(3);
}

} // namespace

void launch_hull_batch(uint64_t seed, uint64_t first, int64_t count, const float lo[3],
                       const float ext[3], const HullView *views, int nv, const uint8_t *masks,
                       float z_near, uint32_t *bits, uint32_t *counts, uint32_t *found,
                       uint32_t need, float *out, int64_t done, unsigned long long *result,
                       cudaStream_t s)
{
    if (count <= 0 || need == 0) return;
    HullBox box;
    box.seed = seed;
    for (int a = 0; a < 3; ++a) {
        box.lo[a] = lo[a];
        box.ex[a] = ext[a];
    }
    if (count < HULL_FEW)
        run_batch<HULL_BLOCK>(box, first, count, views, nv, masks, z_near, bits, counts, found, need,
                              out, done, result, s);
    else
        run_batch<2 * HULL_BLOCK>(box, first, count, views, nv, masks, z_near, bits, counts, found,
                                  need, out, done, result, s);
}

void launch_sh_normals(uint64_t seed, int64_t count, float *out, cudaStream_t s)
{
    if (count <= 0) return;
    sh_normals_kernel<<<grid_of((count + 1) / 2), 256, 0, s>>>(seed, count, out);
    count_launches(1);
}

} // namespace pbr
