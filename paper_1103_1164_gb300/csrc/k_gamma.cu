// Gamma-index comparison of two dose distributions (the 3 %-3 mm 3-D gamma
// of the paper's accuracy evaluation, Section 3 and Tables 2-3):
//   gamma(r) = min(R / dta, min over whole-voxel offsets o, |o| <= R, r + o in
//              the grid, of sqrt(|o|^2 / dta^2 + (D_eval(r + o) - D_ref(r))^2 / dD^2)),
// dD = pct / 100 * max D_ref, and its statistics (gamma_max, the mean gamma
// and the pass rate gamma < 1 inside the reference's 50 % isodose line).
//
// One thread per reference voxel walks the offsets in order of increasing
// length and stops at the first whose distance term alone is not below the
// best value so far (no later offset can do better); consecutive threads hold
// consecutive x, so each offset's evaluated doses are read coalesced.  The
// reductions (max dose, statistics) run in a fixed order, so results do not
// depend on scheduling.
//
// Two launches, one upload and one read-back per call: the last block of each
// kernel to finish folds the blocks' partials, and the statistics are taken as
// gamma is computed.  With five kernels, a wait for the maximum between them and
// five device blocks allocated and freed per call, a comparison on 128 x 128 x 96
// voxels took 297 us, of which 45 us were kernels; now 88 to 111, of which 36 are (on
// a host whose launches take longer, 351 and 149).
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <string>
#include <vector>

#include "dc_internal.cuh"

namespace dc {
namespace {

constexpr int kGammaThreads = 256;
constexpr int kMaxBlocks = 304;     // partials of the maximum (two blocks per multiprocessor)
constexpr int kPartBlocks = 2432;   // partials of the statistics
constexpr int kMaxReach = 64;       // search radius in voxels along each axis

// Per block: max gamma, sum of gamma, voxel count and pass count inside the
// 50 % isodose of the reference.
struct GammaPart {
    double sum50;
    long long n50, pass50;
    float gmax;
    float dmax;   // the result's: max D_ref
};

// Device scratch of one call.  `done` counts finished blocks and is zero between
// kernels (the last block resets it).
constexpr int kSlotOffsets = 4096;  // search spheres of a radius up to 9.9 voxels
struct GammaScratch {
    GammaPart part[kPartBlocks];
    GammaPart out;
    float maxpart[kMaxBlocks];
    float dmax;
    unsigned int done;
    int4 off[kSlotOffsets];
};

// Scratch of the calls in flight: a call takes a free slot and returns it when its
// work has ended (the call waits for it); with none free, or for a larger search
// sphere, it allocates.  One set per device, as all device variables.
constexpr int kSlots = 4;
__device__ GammaScratch g_scratch[kSlots];
std::atomic<unsigned> g_busy{0};

struct GammaArgs {
    const float* ref;
    const float* ev;
    float* gamma;
    int nx, ny, nz;
    const int4* off;     // (i, j, k, bits of |o|^2 / dta^2), |o| ascending
    int n_off;
    float frac;          // pct / 100
    float cap2;          // (R / dta)^2
    GammaScratch* sc;
};

// Sums and maximum over the block in a fixed order: shuffles inside the warps, then
// the warps in order.  The result is thread 0's.
__device__ __forceinline__ GammaPart block_fold(GammaPart x, GammaPart* sh)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        x.sum50 += __shfl_xor_sync(0xffffffffu, x.sum50, o);
        x.n50 += __shfl_xor_sync(0xffffffffu, x.n50, o);
        x.pass50 += __shfl_xor_sync(0xffffffffu, x.pass50, o);
        x.gmax = fmaxf(x.gmax, __shfl_xor_sync(0xffffffffu, x.gmax, o));
    }
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < kGammaThreads / 32; ++w) {
            x.sum50 += sh[w].sum50;
            x.n50 += sh[w].n50;
            x.pass50 += sh[w].pass50;
            x.gmax = fmaxf(x.gmax, sh[w].gmax);
        }
    __syncthreads();
    return x;
}

__device__ __forceinline__ float block_max(float x, float* sh)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < kGammaThreads / 32; ++w) x = fmaxf(x, sh[w]);
    __syncthreads();
    return x;
}

// Whether this block is the kernel's last to get here, its writes and the other
// blocks' before it visible to it.
__device__ __forceinline__ bool last_block(unsigned int* done)
{
    __shared__ unsigned int s_turn;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_turn = atomicAdd(done, 1u);
    __syncthreads();
    const bool last = s_turn == gridDim.x - 1;
    if (last) {
        if (threadIdx.x == 0) *done = 0;
        __threadfence();
    }
    return last;
}

// max D_ref (values >= 0): contiguous chunks per block, then the blocks' maxima.
__global__ void __launch_bounds__(kGammaThreads) k_gamma_max(const float* __restrict__ d, int64_t n, GammaScratch* sc)
{
    __shared__ float sh[kGammaThreads / 32];
    const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
    const int64_t lo = blockIdx.x * chunk, hi = min(n, lo + chunk);
    float m = 0.f;
    for (int64_t v = lo + threadIdx.x; v < hi; v += 4 * kGammaThreads) {
        float x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = v + q * kGammaThreads < hi ? __ldg(d + v + q * kGammaThreads) : 0.f;
#pragma unroll
        for (int q = 0; q < 4; ++q) m = fmaxf(m, x[q]);
    }
    m = block_max(m, sh);
    if (threadIdx.x == 0) sc->maxpart[blockIdx.x] = m;
    if (!last_block(&sc->done)) return;
    m = 0.f;
    for (int q = threadIdx.x; q < gridDim.x; q += kGammaThreads) m = fmaxf(m, __ldcg(sc->maxpart + q));
    m = block_max(m, sh);
    if (threadIdx.x == 0) sc->dmax = m;
}

// Gamma and its statistics; nothing is computed without a positive maximum.
__global__ void __launch_bounds__(kGammaThreads) k_gamma(const GammaArgs a)
{
    __shared__ GammaPart sh[kGammaThreads / 32];
    const float dmax = a.sc->dmax;
    if (!(dmax > 0.f)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) a.sc->out = GammaPart{0.0, 0, 0, 0.f, dmax};
        return;
    }
    const int64_t V = (int64_t)a.nx * a.ny * a.nz;
    const float dD = a.frac * dmax, half = 0.5f * dmax;
    const float inv = 1.0f / (dD * dD);
    GammaPart mine{0.0, 0, 0, 0.f, dmax};
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < V; v += (int64_t)gridDim.x * blockDim.x) {
        int x, y, z;
        if (V <= 0xffffffffll) {   // 32-bit division
            const uint32_t u = (uint32_t)v, q = u / (uint32_t)a.nx;
            x = (int)(u - q * (uint32_t)a.nx);
            y = (int)(q % (uint32_t)a.ny);
            z = (int)(q / (uint32_t)a.ny);
        } else {
            x = (int)(v % a.nx);
            y = (int)((v / a.nx) % a.ny);
            z = (int)(v / ((int64_t)a.nx * a.ny));
        }
        const float dr = __ldg(a.ref + v);
        float best = a.cap2;
        for (int q = 0; q < a.n_off; ++q) {
            const int4 o = __ldg(a.off + q);
            const float d2 = __int_as_float(o.w);
            if (d2 >= best) break;
            const int xx = x + o.x, yy = y + o.y, zz = z + o.z;
            if ((unsigned)xx >= (unsigned)a.nx || (unsigned)yy >= (unsigned)a.ny || (unsigned)zz >= (unsigned)a.nz)
                continue;
            const float diff = __ldg(a.ev + ((int64_t)zz * a.ny + yy) * a.nx + xx) - dr;
            best = fminf(best, fmaf(diff * diff, inv, d2));
        }
        const float gv = sqrtf(best);
        a.gamma[v] = gv;
        mine.gmax = fmaxf(mine.gmax, gv);
        if (dr >= half) {
            mine.sum50 += (double)gv;
            ++mine.n50;
            mine.pass50 += gv < 1.0f ? 1 : 0;
        }
    }
    mine = block_fold(mine, sh);
    if (threadIdx.x == 0) a.sc->part[blockIdx.x] = mine;
    if (!last_block(&a.sc->done)) return;
    mine = GammaPart{0.0, 0, 0, 0.f, dmax};
    for (int q = threadIdx.x; q < gridDim.x; q += kGammaThreads) {
        const volatile GammaPart& t = a.sc->part[q];
        mine.gmax = fmaxf(mine.gmax, t.gmax);
        mine.sum50 += t.sum50;
        mine.n50 += t.n50;
        mine.pass50 += t.pass50;
    }
    mine = block_fold(mine, sh);
    if (threadIdx.x == 0) a.sc->out = mine;
}

int float_bits(float f)
{
    int i;
    memcpy(&i, &f, sizeof(i));
    return i;
}

// Device memory of one call: its scratch, and copies of host arrays.  Waits for the
// call's work and gives everything back on every return path.
struct GammaBuffers {
    cudaStream_t stream;
    int slot = -1;
    std::vector<void*> ptrs;
    explicit GammaBuffers(cudaStream_t s) : stream(s) {}
    ~GammaBuffers()
    {
        if (slot >= 0) {
            cudaStreamSynchronize(stream);
            g_busy.fetch_and(~(1u << slot));
        }
        for (void* p : ptrs) cudaFree(p);
        cudaGetLastError();   // what failed has been reported: not for a later call's launch check
    }
    template <typename T>
    cudaError_t get(T** p, size_t n)
    {
        void* q = nullptr;
        const cudaError_t e = dc::dev_malloc(&q, n * sizeof(T) > 0 ? n * sizeof(T) : 16);
        if (e == cudaSuccess) ptrs.push_back(q);
        *p = reinterpret_cast<T*>(q);
        return e;
    }
    cudaError_t scratch(GammaScratch** sc)
    {
        for (int k = 0; k < kSlots && slot < 0; ++k)
            if (!(g_busy.fetch_or(1u << k) & (1u << k))) slot = k;
        cudaError_t e;
        if (slot >= 0) {
            void* p = nullptr;
            e = cudaGetSymbolAddress(&p, g_scratch);
            *sc = reinterpret_cast<GammaScratch*>(p) + slot;
        } else {
            e = get(sc, 1);
            if (e == cudaSuccess) e = cudaMemsetAsync(&(*sc)->done, 0, sizeof(unsigned int), stream);
        }
        return e;
    }
};

}  // namespace
}  // namespace dc

using namespace dc;

extern "C" dc_status dc_gamma_index(const float* ref, const float* eval, const dc_grid* grid, float dose_pct,
                                    float dta_cm, float search_cm, float* gamma, dc_gamma_stats* stats,
                                    void* cuda_stream, uint32_t flags)
{
    DC_NVTX("dc_gamma_index");
    if (!ref || !eval || !grid) {
        set_error("dc_gamma_index: NULL argument");
        return DC_EINVAL;
    }
    const dc_grid g = *grid;
    if (g.nx < 1 || g.ny < 1 || g.nz < 1 || !(g.dx > 0 && g.dy > 0 && g.dz > 0)) {
        set_error("dc_gamma_index: empty grid or non-positive voxel size");
        return DC_EINVAL;
    }
    if (!(dose_pct > 0 && dta_cm > 0 && search_cm >= dta_cm)) {
        set_error("dc_gamma_index: need dose_pct > 0, dta_cm > 0 and search_cm >= dta_cm");
        return DC_EINVAL;
    }
    const int ri = (int)floor(search_cm / g.dx + 1e-9), rj = (int)floor(search_cm / g.dy + 1e-9),
              rk = (int)floor(search_cm / g.dz + 1e-9);
    if (ri > kMaxReach || rj > kMaxReach || rk > kMaxReach) {
        set_error("dc_gamma_index: the search radius spans more than 64 voxels along an axis");
        return DC_EINVAL;
    }
    const int64_t V = (int64_t)g.nx * g.ny * g.nz;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);

    GammaBuffers buf(s);
    const bool dev = (flags & DC_DEVICE_PTRS) != 0;
    const float* d_ref = ref;
    const float* d_ev = eval;
    float* d_g = dev ? gamma : nullptr;
    GammaScratch* sc = nullptr;
    DC_CUDA(buf.scratch(&sc));
    if (!dev) {
        float *r = nullptr, *e = nullptr;
        DC_CUDA(buf.get(&r, V));
        DC_CUDA(buf.get(&e, V));
        DC_CUDA(cudaMemcpyAsync(r, ref, V * sizeof(float), cudaMemcpyHostToDevice, s));
        DC_CUDA(cudaMemcpyAsync(e, eval, V * sizeof(float), cudaMemcpyHostToDevice, s));
        d_ref = r;
        d_ev = e;
    }
    if (!d_g) DC_CUDA(buf.get(&d_g, V));
    const int64_t want = (V + kGammaThreads - 1) / kGammaThreads;
    k_gamma_max<<<(int)std::min<int64_t>(want, kMaxBlocks), kGammaThreads, 0, s>>>(d_ref, V, sc);

    // offsets within the search sphere, by increasing length (ties in a fixed order)
    struct Off {
        double d2;
        int i, j, k;
    };
    std::vector<Off> offs;
    const double R2 = (double)search_cm * search_cm * (1 + 1e-12);
    for (int k = -rk; k <= rk; ++k)
        for (int j = -rj; j <= rj; ++j)
            for (int i = -ri; i <= ri; ++i) {
                const double d2 = (i * (double)g.dx) * (i * (double)g.dx) + (j * (double)g.dy) * (j * (double)g.dy) +
                                  (k * (double)g.dz) * (k * (double)g.dz);
                if (d2 <= R2) offs.push_back(Off{d2, i, j, k});
            }
    std::stable_sort(offs.begin(), offs.end(), [](const Off& a, const Off& b) { return a.d2 < b.d2; });
    std::vector<int4> h_off(offs.size());
    const double inv_dta2 = 1.0 / ((double)dta_cm * dta_cm);
    for (size_t q = 0; q < offs.size(); ++q) {
        const float d2 = (float)(offs[q].d2 * inv_dta2);
        h_off[q] = make_int4(offs[q].i, offs[q].j, offs[q].k, float_bits(d2));
    }
    int4* d_off = sc->off;
    if (h_off.size() > (size_t)kSlotOffsets) DC_CUDA(buf.get(&d_off, h_off.size()));
    DC_CUDA(cudaMemcpyAsync(d_off, h_off.data(), h_off.size() * sizeof(int4), cudaMemcpyHostToDevice, s));

    GammaArgs a;
    a.ref = d_ref;
    a.ev = d_ev;
    a.gamma = d_g;
    a.nx = g.nx;
    a.ny = g.ny;
    a.nz = g.nz;
    a.off = d_off;
    a.n_off = (int)h_off.size();
    a.frac = dose_pct / 100.f;
    a.cap2 = (float)(((double)search_cm / dta_cm) * ((double)search_cm / dta_cm));
    a.sc = sc;
    k_gamma<<<(int)std::min<int64_t>(want, kPartBlocks), kGammaThreads, 0, s>>>(a);
    count_launches(2);
    DC_CUDA(cudaGetLastError());
    GammaPart h{};
    DC_CUDA(cudaMemcpyAsync(&h, &sc->out, sizeof(h), cudaMemcpyDeviceToHost, s));
    DC_CUDA(cudaStreamSynchronize(s));
    if (!(h.dmax > 0.f)) {
        set_error("dc_gamma_index: the reference dose is zero everywhere");
        return DC_EINVAL;
    }
    if (gamma && !dev) {
        DC_CUDA(cudaMemcpyAsync(gamma, d_g, V * sizeof(float), cudaMemcpyDeviceToHost, s));
        DC_CUDA(cudaStreamSynchronize(s));
    }
    if (stats) {
        stats->gamma_max = h.gmax;
        stats->n50 = h.n50;
        stats->gamma_avg50 = h.n50 > 0 ? h.sum50 / (double)h.n50 : 0.0;
        stats->pass50_pct = h.n50 > 0 ? 100.0 * (double)h.pass50 / (double)h.n50 : 0.0;
        stats->dose_max = h.dmax;
    }
    return DC_OK;
}
