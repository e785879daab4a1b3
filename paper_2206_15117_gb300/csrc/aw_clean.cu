// Cleaning: Cotton-Schwab major cycles around a Hogbom minor cycle.
//
// arXiv:2206.15117 Sec. 2.1: the imager cleans with the Cotton-Schwab
// algorithm (number of clean cycles, loop gain, cycle factor, threshold);
// Sec. 4 names Hogbom cleaning as its iterative, hard-to-parallelise part.
// The readings the paper leaves open are stated with the declarations in
// aw.h.  Major-cycle transforms reuse the gridding, image and degridding
// paths; the minor cycle keeps the maximum of every tile so that an iteration
// rescans only the tiles its subtraction touched.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>

#include "aw_internal.h"

namespace {

inline cudaStream_t S_(void *s) { return reinterpret_cast<cudaStream_t>(s); }

int use_device(int dev) {
    int cur = -1;
    AW_CUDA_TRY(cudaGetDevice(&cur));
    if (cur != dev) AW_CUDA_TRY(cudaSetDevice(dev));
    return AW_OK;
}

int nblk(int64_t n, int t) {
    int64_t b = (n + t - 1) / t;
    if (b < 1) b = 1;
    if (b > 152 * 32) b = 152 * 32;
    return (int)b;
}

// ctx->d_scratch words used here
constexpr int SCR_R0 = 4;        // main-lobe radius
constexpr int SCR_SIDE = 5;      // sidelobe level (float bits, >= 0)
constexpr int SCR_PEAK = 6;      // window peak |I| (float bits, >= 0)
constexpr int SCR_NITER = 7;     // Hogbom iterations
constexpr int SCR_BAR_COUNT = 8; // grid barrier: arrivals
constexpr int SCR_BAR_ERR = 10;  // grid barrier: set when a wait gave up
// spin limit of one barrier wait: polls of 0.37 to 0.39 us (2^24 of them 6.2 s, 3 x 2^23 9.7 s), about 9 s
constexpr long long BAR_SPIN_LIMIT = 24000000ll;

// ---------------------------------------------------------------- sidelobe
// r0 = first x > 0 with psf[c][c + x] <= 0 (N/2 if none), one warp.
__global__ void psf_r0_kernel(const float *psf, int N, unsigned int *scr) {
    const int c = N / 2, lane = threadIdx.x;
    int r0 = N / 2;
    for (int base = 1; base < N - c; base += 32) {
        const int x = base + lane;
        const bool hit = x < N - c && psf[(int64_t)c * N + c + x] <= 0.f;
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        if (m) { r0 = base + __ffs(m) - 1; break; }
    }
    if (lane == 0) scr[SCR_R0] = (unsigned)r0;
}

__global__ void psf_side_kernel(const float *psf, int N, unsigned int *scr) {
    const int c = N / 2;
    const int64_t r0 = scr[SCR_R0];
    float m = 0.f;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (int64_t)N * N;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t dy = i / N - c, dx = i % N - c;
        const int64_t q = N / 4;
        if (dx * dx + dy * dy > r0 * r0 && dx < q && -dx < q && dy < q && -dy < q) m = fmaxf(m, fabsf(psf[i]));
    }
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&scr[SCR_SIDE], __float_as_uint(m));
}

// ---------------------------------------------------------------- window peak
__global__ void window_peak_kernel(const float *img, int N, int x0, int y0, int x1, int y1, unsigned int *scr) {
    const int w = x1 - x0;
    const int64_t cnt = (int64_t)w * (y1 - y0);
    float m = 0.f;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < cnt; e += (int64_t)gridDim.x * blockDim.x)
        m = fmaxf(m, fabsf(img[(int64_t)(y0 + e / w) * N + x0 + e % w]));
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&scr[SCR_PEAK], __float_as_uint(m));
}

// ---------------------------------------------------------------- Hogbom
// |I| and the pixel index packed so that the unsigned maximum is the largest
// |I| with the lowest index; 0 means "no pixel".
__device__ __forceinline__ unsigned long long hb_pack(float v, uint32_t idx) {
    return ((unsigned long long)__float_as_uint(fabsf(v)) << 32) | (unsigned long long)(0xFFFFFFFFu - idx);
}

struct HbGeom {
    int N, T, TX;
    int x0, y0, x1, y1;
};

// What a tile shows the others: its largest |I| over the window (packed with the
// pixel) and the residual of every plane there.
struct __align__(16) HbRec {
    unsigned long long best;
    unsigned long long pad;
    float v[4];
};

constexpr int HB_GROUP = 256;                  // threads that work on one tile
constexpr int HB_GROUPS = 4;                   // tiles a block works on at once
constexpr int HB_THREADS = HB_GROUP * HB_GROUPS;
constexpr int HB_TILES_AXIS = 64;              // tiles an axis, at most

__device__ __forceinline__ unsigned long long max_u64(unsigned long long a, unsigned long long b) { return a > b ? a : b; }
__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
    for (int o = 16; o; o >>= 1) v = max_u64(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// One tile by a group of HB_GROUP threads: with SUB, comp[s] x psf is subtracted
// inside the patch [xa, xb) x [ya, yb) about (py, px) (FP32, one rounding per
// multiply and per subtraction); then the tile's record is written.  Every pixel
// of the tile is read by one thread only, through L2 (another block may have
// written it an iteration ago).  `bar`: the group's barrier; red: 8 words.
template <bool SUB>
__device__ __forceinline__ void hb_tile(float *R, const float *psf, int npol, const HbGeom &g, int t, int py, int px,
                                        int ya, int yb, int xa, int xb, const float (&comp)[4], HbRec *out, int bar,
                                        unsigned long long *red) {
    const int64_t NN = (int64_t)g.N * g.N;
    const int c = g.N / 2, gt = threadIdx.x % HB_GROUP, lane = gt & 31, warp = gt >> 5;
    const int tx0 = (t % g.TX) * g.T, ty0 = (t / g.TX) * g.T;
    const int tx1 = min(tx0 + g.T, g.N), ty1 = min(ty0 + g.T, g.N);
    unsigned long long best = 0ull;
    float bv[4] = {0.f, 0.f, 0.f, 0.f};
    for (int y = ty0 + warp; y < ty1; y += HB_GROUP / 32)
        for (int x = tx0 + lane; x < tx1; x += 32) {
            const bool sub = SUB && y >= ya && y < yb && x >= xa && x < xb;
            const bool win = y >= g.y0 && y < g.y1 && x >= g.x0 && x < g.x1;
            if (!sub && !win) continue;
            const uint32_t idx = (uint32_t)y * (uint32_t)g.N + (uint32_t)x;
            float v[4];
#pragma unroll
            for (int s = 0; s < 4; ++s) v[s] = s < npol ? __ldcg(R + s * NN + idx) : 0.f;
            if (sub) {
                const float p = __ldg(psf + (int64_t)(c + y - py) * g.N + (c + x - px));
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    if (s < npol) {
                        v[s] = __fsub_rn(v[s], __fmul_rn(comp[s], p));
                        __stcg(R + s * NN + idx, v[s]);
                    }
            }
            const unsigned long long k = hb_pack(v[0], idx);
            if (win && k > best) {
                best = k;
#pragma unroll
                for (int s = 0; s < 4; ++s) bv[s] = v[s];
            }
        }
    const unsigned long long wb = warp_max_u64(best);
    if (lane == 0) red[warp] = wb;
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(HB_GROUP) : "memory");
    unsigned long long gb = 0ull;
#pragma unroll
    for (int w = 0; w < HB_GROUP / 32; ++w) gb = max_u64(gb, red[w]);
    if (gb == 0ull ? gt == 0 : best == gb) {   // (a pixel index is in one thread only)
        uint4 *o = reinterpret_cast<uint4 *>(out);
        __stcg(o, make_uint4((uint32_t)gb, (uint32_t)(gb >> 32), 0u, 0u));
        __stcg(o + 1, make_uint4(__float_as_uint(bv[0]), __float_as_uint(bv[1]), __float_as_uint(bv[2]),
                                 __float_as_uint(bv[3])));
    }
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(HB_GROUP) : "memory");   // red is free again
}

// The first records, one group a block.
__global__ void __launch_bounds__(HB_GROUP) hb_tiles_kernel(float *R, int npol, HbGeom g, HbRec *rec) {
    __shared__ unsigned long long red[HB_GROUP / 32];
    const float none[4] = {0.f, 0.f, 0.f, 0.f};
    hb_tile<false>(R, nullptr, npol, g, blockIdx.x, 0, 0, 0, 0, 0, 0, none, rec + blockIdx.x, 1, red);
}

// Barrier over all blocks of a cooperative launch (co-residency guaranteed by
// the launch): the arrival count only grows, and the call that a block makes as
// its n-th waits for n x nblocks arrivals.  The wait is bounded: one that runs out
// sets the error word and returns false, so that no block can wait for ever; the
// caller then leaves its loop.
__device__ bool grid_barrier(unsigned int *scr, unsigned int nblocks, unsigned int n, int *s_ok) {
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned int target = n * nblocks;   // (compared as a difference: the count may wrap)
        __threadfence();
        int ok = 1;
        if ((int)(atomicAdd(scr + SCR_BAR_COUNT, 1u) + 1u - target) < 0) {
            long long spins = 0;
            while ((int)(*(volatile unsigned int *)(scr + SCR_BAR_COUNT) - target) < 0) {
                if (++spins > BAR_SPIN_LIMIT || *(volatile unsigned int *)(scr + SCR_BAR_ERR)) {
                    atomicExch(scr + SCR_BAR_ERR, 1u);
                    ok = 0;
                    break;
                }
                __nanosleep(20);
            }
        }
        __threadfence();
        *s_ok = ok;
    }
    __syncthreads();
    return *s_ok != 0;
}

// Self-test of the barrier's bounded wait: one block that expects a second
// arrival which never comes (the arrival count is never reached).
__global__ void barrier_timeout_kernel(unsigned int *scr) {
    __shared__ int s_ok;
    grid_barrier(scr, 2u, 1u, &s_ok);
}

struct __align__(16) HbSmem {
    unsigned long long best[HB_TILES_AXIS * HB_TILES_AXIS];   // every tile's maximum
    float4 v[HB_TILES_AXIS * HB_TILES_AXIS];                  // and the residual there
    unsigned long long row[HB_TILES_AXIS];                    // maxima of the tile rows
    unsigned long long red[HB_GROUPS][HB_GROUP / 32];
    int ok;
};

// The minor cycle as one cooperative grid with one barrier an iteration.  Every
// block holds all tiles' maxima and the residuals there in shared memory, so all
// find the same peak and component (gain x residual, all planes) without another
// block's help.  The tiles the patch touches are dealt to groups of 256 threads;
// a group subtracts its part of component x psf and finds the tile's new maximum
// in the same pass over the tile, and publishes it.  After the barrier every
// block reads the touched tiles' records.  Records alternate between two buffers,
// so that a block ahead by an iteration does not write what another still reads.
// Latency bounds it: L2 round trips for the records, the tile and the barrier.
// 2048^2 x 4, patch 513^2: 23.2 us an iteration with three barriers (peak read,
// patch subtracted, tiles rescanned), 6.8 us now.
__global__ void __launch_bounds__(HB_THREADS) hogbom_kernel(float *R, const float *psf, float *model, int npol,
                                                            HbGeom g, float gain, float thr, int max_iter, int h,
                                                            HbRec *rec, unsigned int *scr) {
    extern __shared__ __align__(16) char hb_smem[];
    HbSmem &sm = *reinterpret_cast<HbSmem *>(hb_smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, group = tid / HB_GROUP;
    const int ntiles = g.TX * g.TX;
    const int64_t NN = (int64_t)g.N * g.N;
    // tiles whose records the next decision reads: all of them at first
    int tx0 = 0, ty0 = 0, ntx = g.TX, nty = g.TX;
    for (int n = 0;; ++n) {
        // ---- refresh the touched tiles, then their rows
        const HbRec *in = rec + (int64_t)((n + 1) & 1) * ntiles;
        for (int k = tid; k < ntx * nty; k += HB_THREADS) {
            const int t = (ty0 + k / ntx) * g.TX + tx0 + k % ntx;
            const uint4 a = __ldcg(reinterpret_cast<const uint4 *>(in + t));
            const uint4 b = __ldcg(reinterpret_cast<const uint4 *>(in + t) + 1);
            sm.best[t] = (unsigned long long)a.y << 32 | a.x;
            sm.v[t] = make_float4(__uint_as_float(b.x), __uint_as_float(b.y), __uint_as_float(b.z), __uint_as_float(b.w));
        }
        __syncthreads();
        for (int y = ty0 + warp; y < ty0 + nty; y += HB_THREADS / 32) {
            unsigned long long v = lane < g.TX ? sm.best[y * g.TX + lane] : 0ull;
            if (lane + 32 < g.TX) v = max_u64(v, sm.best[y * g.TX + lane + 32]);
            v = warp_max_u64(v);
            if (lane == 0) sm.row[y] = v;
        }
        __syncthreads();
        // ---- the peak and the component, the same in every thread of every block
        unsigned long long v = lane < g.TX ? sm.row[lane] : 0ull;
        if (lane + 32 < g.TX) v = max_u64(v, sm.row[lane + 32]);
        const unsigned long long best = warp_max_u64(v);
        bool stop = best == 0ull || n >= max_iter;
        const uint32_t idx = 0xFFFFFFFFu - (uint32_t)(best & 0xFFFFFFFFull);
        int py = 0, px = 0;
        float comp[4] = {0.f, 0.f, 0.f, 0.f};
        if (!stop) {
            py = (int)(idx / (uint32_t)g.N);
            px = (int)(idx % (uint32_t)g.N);
            const float4 at = sm.v[(py / g.T) * g.TX + px / g.T];
            stop = fabsf(at.x) < thr;
            comp[0] = __fmul_rn(gain, at.x);
            comp[1] = __fmul_rn(gain, at.y);
            comp[2] = __fmul_rn(gain, at.z);
            comp[3] = __fmul_rn(gain, at.w);
        }
        if (stop) {
            if (blockIdx.x == 0 && tid == 0) scr[SCR_NITER] = (unsigned)n;
            break;
        }
        if (blockIdx.x == 0 && tid < npol) {
            const int64_t o = tid * NN + idx;
            model[o] = __fadd_rn(model[o], tid == 0 ? comp[0] : tid == 1 ? comp[1] : tid == 2 ? comp[2] : comp[3]);
        }
        // ---- subtract and rescan the touched tiles
        const int ya = max(0, py - h), yb = min(g.N, py + h + 1);
        const int xa = max(0, px - h), xb = min(g.N, px + h + 1);
        tx0 = xa / g.T;
        ty0 = ya / g.T;
        ntx = (xb - 1) / g.T - tx0 + 1;
        nty = (yb - 1) / g.T - ty0 + 1;
        HbRec *out = rec + (int64_t)(n & 1) * ntiles;
        for (int k = group * gridDim.x + blockIdx.x; k < ntx * nty; k += gridDim.x * HB_GROUPS) {
            const int t = (ty0 + k / ntx) * g.TX + tx0 + k % ntx;
            hb_tile<true>(R, psf, npol, g, t, py, px, ya, yb, xa, xb, comp, out + t, 1 + group, sm.red[group]);
        }
        if (!grid_barrier(scr, gridDim.x, (unsigned)(n + 1), &sm.ok)) break;   // the records are current
    }
}

// ---------------------------------------------------------------- clean helpers
__global__ void unit_vis_kernel(float2 *v, int64_t nvis, int npol) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nvis * npol;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(i % npol);
        v[i] = make_float2((c == 0 || c == 3) ? 1.f : 0.f, 0.f);
    }
}

__global__ void psf_norm_kernel(const float *plane0, int N, float *psf) {
    const float p0 = plane0[(int64_t)(N / 2) * N + N / 2];
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (int64_t)N * N;
         i += (int64_t)gridDim.x * blockDim.x)
        psf[i] = plane0[i] / p0;
}

int check_window(const int32_t *win, int N) {
    if (!win) return aw_set_error(AW_EINVAL, "window is NULL");
    if (win[0] < 0 || win[1] < 0 || win[2] > N || win[3] > N || win[0] >= win[2] || win[1] >= win[3])
        return aw_set_error(AW_EINVAL, "window (%d, %d, %d, %d) not a non-empty box inside the %d^2 image",
                            win[0], win[1], win[2], win[3], N);
    return AW_OK;
}

HbGeom geom_of(int N, const int32_t *win) {
    HbGeom g;
    g.N = N;
    g.T = std::max(32, (N + HB_TILES_AXIS - 1) / HB_TILES_AXIS);
    g.TX = (N + g.T - 1) / g.T;
    g.x0 = win[0];
    g.y0 = win[1];
    g.x1 = win[2];
    g.y1 = win[3];
    return g;
}

// Run barrier_timeout_kernel: AW_ETIMEOUT once the wait has given up.
int barrier_selftest_impl(aw_ctx *ctx, cudaStream_t s) {
    AW_CUDA_TRY(cudaMemsetAsync(ctx->d_scratch + SCR_BAR_COUNT, 0, 3 * sizeof(unsigned int), s));
    barrier_timeout_kernel<<<1, 32, 0, s>>>(ctx->d_scratch);
    AW_CHECK_LAUNCH();
    unsigned int w = 0;
    AW_CUDA_TRY(cudaMemcpyAsync(&w, ctx->d_scratch + SCR_BAR_ERR, sizeof(w), cudaMemcpyDeviceToHost, s));
    AW_CUDA_TRY(cudaStreamSynchronize(s));
    AW_CUDA_TRY(cudaMemsetAsync(ctx->d_scratch + SCR_BAR_COUNT, 0, 3 * sizeof(unsigned int), s));
    AW_CUDA_TRY(cudaStreamSynchronize(s));
    return w ? aw_set_error(AW_ETIMEOUT, "grid barrier wait gave up") : AW_OK;
}

int hogbom_impl(aw_ctx *ctx, float *R, const float *psf, int npol, int N, float gain, float thr, int max_iter,
                int h, const int32_t *win, float *model, int32_t *n_iter, cudaStream_t s) {
    HbGeom g = geom_of(N, win);
    const int ntiles = g.TX * g.TX;
    HbRec *rec = nullptr;
    AW_CUDA_TRY(cudaMallocAsync(&rec, 2 * sizeof(HbRec) * ntiles, s));
    hb_tiles_kernel<<<ntiles, HB_GROUP, 0, s>>>(R, npol, g, rec + ntiles);   // iteration 0 reads the second buffer
    cudaError_t e = cudaGetLastError();
    int per_sm = 0;
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(hogbom_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(HbSmem));
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, hogbom_kernel, HB_THREADS, sizeof(HbSmem));
    if (e == cudaSuccess && per_sm < 1) e = cudaErrorCooperativeLaunchTooLarge;
    if (e == cudaSuccess) e = cudaMemsetAsync(ctx->d_scratch + SCR_BAR_COUNT, 0, 3 * sizeof(unsigned int), s);
    if (e == cudaSuccess) {
        // a group of threads for every tile a patch can touch, two groups' tiles a block at
        // most, one block per SM: the barrier's cost grows with the blocks
        const int across = std::min(2 * h / g.T + 2, g.TX);
        const int blocks = std::min(ctx->sm_count, std::max(1, (across * across + 1) / 2));
        void *args[] = {&R, (void *)&psf, &model, &npol, &g, &gain, &thr, &max_iter, &h, &rec, &ctx->d_scratch};
        e = cudaLaunchCooperativeKernel((const void *)hogbom_kernel, dim3(blocks), dim3(HB_THREADS), args,
                                        sizeof(HbSmem), s);
    }
    cudaFreeAsync(rec, s);
    if (e != cudaSuccess) return aw_set_error(AW_ECUDA, "hogbom: %s", cudaGetErrorString(e));
    unsigned int w[4] = {0, 0, 0, 0};  // iterations, barrier count, -, error
    AW_CUDA_TRY(cudaMemcpyAsync(w, ctx->d_scratch + SCR_NITER, sizeof(w), cudaMemcpyDeviceToHost, s));
    AW_CUDA_TRY(cudaStreamSynchronize(s));
    if (w[3]) return aw_set_error(AW_ETIMEOUT, "hogbom: a grid barrier wait gave up; results are invalid");
    *n_iter = (int32_t)w[0];
    return AW_OK;
}

int sidelobe_impl(aw_ctx *ctx, const float *psf, int N, float *out, cudaStream_t s) {
    AW_CUDA_TRY(cudaMemsetAsync(ctx->d_scratch + SCR_SIDE, 0, sizeof(unsigned int), s));
    psf_r0_kernel<<<1, 32, 0, s>>>(psf, N, ctx->d_scratch);
    AW_CHECK_LAUNCH();
    psf_side_kernel<<<nblk((int64_t)N * N, 256), 256, 0, s>>>(psf, N, ctx->d_scratch);
    AW_CHECK_LAUNCH();
    unsigned int bits = 0;
    AW_CUDA_TRY(cudaMemcpyAsync(&bits, ctx->d_scratch + SCR_SIDE, sizeof(bits), cudaMemcpyDeviceToHost, s));
    AW_CUDA_TRY(cudaStreamSynchronize(s));
    std::memcpy(out, &bits, sizeof(float));
    return AW_OK;
}

int window_peak_impl(aw_ctx *ctx, const float *img, int N, const int32_t *win, float *out, cudaStream_t s) {
    AW_CUDA_TRY(cudaMemsetAsync(ctx->d_scratch + SCR_PEAK, 0, sizeof(unsigned int), s));
    const int64_t cnt = (int64_t)(win[2] - win[0]) * (win[3] - win[1]);
    window_peak_kernel<<<nblk(cnt, 256), 256, 0, s>>>(img, N, win[0], win[1], win[2], win[3], ctx->d_scratch);
    AW_CHECK_LAUNCH();
    unsigned int bits = 0;
    AW_CUDA_TRY(cudaMemcpyAsync(&bits, ctx->d_scratch + SCR_PEAK, sizeof(bits), cudaMemcpyDeviceToHost, s));
    AW_CUDA_TRY(cudaStreamSynchronize(s));
    std::memcpy(out, &bits, sizeof(float));
    return AW_OK;
}

struct DevMem {
    void *p = nullptr;
    ~DevMem() { if (p) aw_dev_free(p); }
};

int check_plan_kset(const aw_plan *p, const aw_kernel_set *k) {
    if (!p || !k) return aw_set_error(AW_EINVAL, "plan/kset is NULL");
    if (p->N != k->spec.N || p->OS != k->spec.OS || p->npol != k->spec.npol || p->nbins != k->nbins || p->ntype != k->ntype ||
        p->bin_support != k->bin_support)
        return aw_set_error(AW_EINVAL, "kernel set geometry does not match the plan");
    return AW_OK;
}

#define CL_GUARD_BEGIN \
    AW_TRACE();         \
    try {
#define CL_GUARD_END                                                   \
    }                                                                  \
    catch (const std::bad_alloc &) {                                   \
        return aw_set_error(AW_ENOMEM, "host allocation failed");      \
    }                                                                  \
    catch (...) {                                                      \
        return aw_set_error(AW_EINVAL, "unexpected C++ exception");    \
    }

}  // namespace

int aw_barrier_selftest(aw_ctx *ctx, cudaStream_t s) { return barrier_selftest_impl(ctx, s); }

extern "C" {

int aw_image_to_grid(aw_ctx *ctx, const aw_kernel_set *k, const float *image, void *grid, void *stream) {
    CL_GUARD_BEGIN
    if (!ctx || !k || !image || !grid) return aw_set_error(AW_EINVAL, "NULL argument");
    int rc = use_device(ctx->device);
    if (rc) return rc;
    return aw_image_to_grid_impl(ctx, k->spec.N, k->spec.npol, k->spec.W, image, grid, S_(stream));
    CL_GUARD_END
}

int aw_degrid_subtract(aw_ctx *ctx, const aw_plan *p, const aw_kernel_set *k, const void *grid, const void *vis,
                       void *vis_out, void *stream) {
    CL_GUARD_BEGIN
    if (!ctx) return aw_set_error(AW_EINVAL, "ctx is NULL");
    int rc = check_plan_kset(p, k);
    if (rc) return rc;
    if (!grid || ((!vis || !vis_out) && p->nvis)) return aw_set_error(AW_EINVAL, "grid/vis/vis_out is NULL");
    rc = use_device(ctx->device);
    if (rc) return rc;
    return aw_launch_degrid(p, k, grid, vis_out, S_(stream), vis);
    CL_GUARD_END
}

int aw_psf_sidelobe(aw_ctx *ctx, const float *psf, int32_t N, float *sidelobe, void *stream) {
    CL_GUARD_BEGIN
    if (!ctx || !psf || !sidelobe) return aw_set_error(AW_EINVAL, "NULL argument");
    if (N < 2) return aw_set_error(AW_EINVAL, "N=%d", N);
    int rc = use_device(ctx->device);
    if (rc) return rc;
    return sidelobe_impl(ctx, psf, N, sidelobe, S_(stream));
    CL_GUARD_END
}

int aw_hogbom(aw_ctx *ctx, float *residual, const float *psf, int32_t npol, int32_t N, float gain,
              float threshold, int32_t max_iter, int32_t patch_half, const int32_t *window, float *model,
              int32_t *n_iter, void *stream) {
    CL_GUARD_BEGIN
    if (!ctx || !residual || !psf || !model || !n_iter) return aw_set_error(AW_EINVAL, "NULL argument");
    if (npol != 1 && npol != 4) return aw_set_error(AW_EINVAL, "npol %d", npol);
    if (N < 4 || (int64_t)N * N > 0xFFFFFFFFll) return aw_set_error(AW_EINVAL, "N=%d", N);
    if (!(gain > 0.f && gain <= 1.f)) return aw_set_error(AW_EINVAL, "gain %g outside (0, 1]", (double)gain);
    if (max_iter < 0) return aw_set_error(AW_EINVAL, "max_iter %d", max_iter);
    if (patch_half < 0 || patch_half >= N / 2) return aw_set_error(AW_EINVAL, "patch_half %d", patch_half);
    int rc = check_window(window, N);
    if (rc) return rc;
    rc = use_device(ctx->device);
    if (rc) return rc;
    return hogbom_impl(ctx, residual, psf, npol, N, gain, threshold, max_iter, patch_half, window, model, n_iter,
                       S_(stream));
    CL_GUARD_END
}

int aw_grid_batched(aw_ctx *ctx, aw_plan *p, const aw_kernel_set *k, const void *vis, const float *weight,
                    void *grid, aw_stats *stats, void *stream);

int aw_clean(aw_ctx *ctx, aw_plan *p, const aw_kernel_set *kg, const aw_kernel_set *kd, const void *vis,
             const float *weight, const aw_clean_cfg *cfg, float *model, float *residual, float *psf,
             aw_clean_report *report, void *stream) {
    CL_GUARD_BEGIN
    if (!ctx || !cfg || !model || !residual || !psf || !report) return aw_set_error(AW_EINVAL, "NULL argument");
    int rc = check_plan_kset(p, kg);
    if (rc) return rc;
    rc = check_plan_kset(p, kd);
    if (rc) return rc;
    if (kg->spec.role != AW_ROLE_GRID) return aw_set_error(AW_EINVAL, "kgrid is not a GRID kernel set");
    if (kd->spec.role == AW_ROLE_GRID) return aw_set_error(AW_EINVAL, "kdegrid is a GRID kernel set");
    if (!vis && p->nvis) return aw_set_error(AW_EINVAL, "vis is NULL");
    const int N = p->N, npol = p->npol;
    if (cfg->n_major < 1 || cfg->max_minor < 0 || !(cfg->gain > 0.f && cfg->gain <= 1.f) ||
        !(cfg->cycle_factor >= 0.f) || cfg->patch_half < 0 || cfg->patch_half >= N / 2)
        return aw_set_error(AW_EINVAL, "clean configuration out of range");
    int32_t win[4] = {cfg->window[0], cfg->window[1], cfg->window[2], cfg->window[3]};
    if (!win[0] && !win[1] && !win[2] && !win[3]) {
        win[0] = win[1] = N / 4;
        win[2] = win[3] = 3 * N / 4;
    }
    rc = check_window(win, N);
    if (rc) return rc;
    rc = use_device(ctx->device);
    if (rc) return rc;
    cudaStream_t s = S_(stream);
    const int64_t plane = (int64_t)N * N;
    const size_t vbytes = sizeof(float2) * (size_t)npol * (size_t)std::max<int64_t>(p->nvis, 1);
    DevMem rv, gr;
    AW_CUDA_TRY(aw_dev_malloc(&rv.p, vbytes));
    AW_CUDA_TRY(aw_dev_malloc(&gr.p, sizeof(float2) * (size_t)npol * plane));
    float2 *res_vis = reinterpret_cast<float2 *>(rv.p);
    aw_clean_report rep{};
    aw_stats st{};
    // point-spread function: unit Stokes I visibilities, same weights and kernels
    unit_vis_kernel<<<nblk(p->nvis * npol, 256), 256, 0, s>>>(res_vis, p->nvis, npol);
    AW_CHECK_LAUNCH();
    AW_CUDA_TRY(cudaMemsetAsync(gr.p, 0, sizeof(float2) * (size_t)npol * plane, s));
    rc = aw_grid_batched(ctx, p, kg, res_vis, weight, gr.p, &st, stream);
    if (rc) return rc;
    if (!(st.weight_sum > 0)) return aw_set_error(AW_EINVAL, "no visibility was gridded (weight sum %g)", st.weight_sum);
    rep.weight_sum = st.weight_sum;
    rc = aw_fft_to_image_impl(ctx, N, npol, kg->spec.W, gr.p, st.weight_sum, residual, s);
    if (rc) return rc;
    psf_norm_kernel<<<nblk(plane, 256), 256, 0, s>>>(residual, N, psf);
    AW_CHECK_LAUNCH();
    rc = sidelobe_impl(ctx, psf, N, &rep.sidelobe, s);
    if (rc) return rc;
    // major cycles
    AW_CUDA_TRY(cudaMemsetAsync(model, 0, sizeof(float) * (size_t)npol * plane, s));
    AW_CUDA_TRY(cudaMemcpyAsync(res_vis, vis, vbytes, cudaMemcpyDeviceToDevice, s));
    bool stopped = false;
    for (int k = 0; k < cfg->n_major; ++k) {
        AW_CUDA_TRY(cudaMemsetAsync(gr.p, 0, sizeof(float2) * (size_t)npol * plane, s));
        rc = aw_grid_batched(ctx, p, kg, res_vis, weight, gr.p, &st, stream);
        if (rc) return rc;
        rc = aw_fft_to_image_impl(ctx, N, npol, kg->spec.W, gr.p, st.weight_sum, residual, s);
        if (rc) return rc;
        float peak = 0.f;
        rc = window_peak_impl(ctx, residual, N, win, &peak, s);
        if (rc) return rc;
        if (k == 0) rep.peak_first = peak;
        rep.peak_last = peak;
        if (peak < cfg->threshold) { stopped = true; break; }
        const float thr = std::max(cfg->threshold, (cfg->cycle_factor * rep.sidelobe) * peak);
        int32_t n = 0;
        rc = hogbom_impl(ctx, residual, psf, npol, N, cfg->gain, thr, cfg->max_minor, cfg->patch_half, win, model,
                         &n, s);
        if (rc) return rc;
        rep.n_minor += n;
        rep.n_major += 1;
        rc = aw_image_to_grid_impl(ctx, N, npol, kd->spec.W, model, gr.p, s);
        if (rc) return rc;
        rc = aw_launch_degrid(p, kd, gr.p, res_vis, s, vis);
        if (rc) return rc;
    }
    if (!stopped) {
        // the residual image of the last prediction
        AW_CUDA_TRY(cudaMemsetAsync(gr.p, 0, sizeof(float2) * (size_t)npol * plane, s));
        rc = aw_grid_batched(ctx, p, kg, res_vis, weight, gr.p, &st, stream);
        if (rc) return rc;
        rc = aw_fft_to_image_impl(ctx, N, npol, kg->spec.W, gr.p, st.weight_sum, residual, s);
        if (rc) return rc;
        rc = window_peak_impl(ctx, residual, N, win, &rep.peak_last, s);
        if (rc) return rc;
    }
    AW_CUDA_TRY(cudaStreamSynchronize(s));
    *report = rep;
    return AW_OK;
    CL_GUARD_END
}

}  // extern "C"
