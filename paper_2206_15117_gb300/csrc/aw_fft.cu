// The two-dimensional transforms between image and uv grid for N = 256 ... 4096,
// two passes over memory with the image step in the first or last of them.
//
// A line of N values is transformed by N / 16 threads with 16 values each in
// registers: radix 16 at every step (the last one 2 ... 16), exchanged through
// shared memory in between (padded by one value in 16: no bank conflicts).  Before
// and after the transform thread t has the values t + m N / 16, so loads and
// stores are coalesced and need no exchange.  Twiddle factors are tables
// rounded from double.  A row CTA takes whole rows, a column CTA COLS
// neighbouring columns (32 or 64 bytes a row).
//
// What bounds it, 4096^2 x 4 grid to image: rows 170 us, HBM (6.0 TB/s); columns 455 us, the
// L1 tags of 12,288 pieces of 16 or 32 bytes a tile and, one CTA filling the SM's
// registers, the load phase that the copy ahead does not cover (2 columns a CTA:
// 875 us in all).  Against cuFFT's three passes and a pass for the image step, to
// image / to grid: 512^2 15 / 15 us against 19 / 19, 1024^2 x 4 37 / 36 against 44 / 44,
// 2048^2 x 4 148 / 131 against 170 / 168, 4096^2 x 4 623 / 560 against 653 / 641; relative
// error at 4096^2 1.8e-7 against 3.6e-7.  Smaller and larger N stay with cuFFT: below
// 256 two launches are the whole time, and 8192 values of four columns do not fit in shared
// memory.
#include <algorithm>
#include <cmath>

#include "aw_internal.h"

namespace {

constexpr int PTS = 16;    // values a thread
// columns a CTA: eight where they fit in the registers of one and enough CTAs are left
template <int N> constexpr int COLS = N == 1024 || N == 2048 ? 8 : 4;

__device__ __forceinline__ int padded(int i) { return i + (i >> 4); }
template <int N> constexpr int LINE_WORDS = N + N / 16;

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
// a * exp(+-i pi / 2)
template <bool INV>
__device__ __forceinline__ float2 crot(float2 a) { return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x); }
// a * exp(+-i pi k / 8)
template <bool INV>
__device__ __forceinline__ float2 croot16(float2 a, int k) {
    constexpr float c1 = 0.92387953251128676f, s1 = 0.38268343236508977f, h = 0.70710678118654752f;
    const float c[10] = {1.f, c1, h, s1, 0.f, -s1, -h, -c1, -1.f, -c1};
    const float s[10] = {0.f, s1, h, c1, 1.f, c1, h, s1, 0.f, -s1};
    return cmul(a, make_float2(c[k], INV ? s[k] : -s[k]));
}

template <bool INV>
__device__ __forceinline__ void dft4(float2 &a, float2 &b, float2 &c, float2 &d) {
    const float2 s0 = cadd(a, c), s1 = csub(a, c), s2 = cadd(b, d), s3 = crot<INV>(csub(b, d));
    a = cadd(s0, s2);
    b = cadd(s1, s3);
    c = csub(s0, s2);
    d = csub(s1, s3);
}

// Transform of R values; output k is left at place<R>(k).
template <int R>
__device__ __forceinline__ constexpr int place(int k) {
    return R == 16 ? 4 * (k & 3) + (k >> 2) : R == 8 ? 2 * (k & 3) + (k >> 2) : k;
}
template <int R, bool INV>
__device__ __forceinline__ void dft(float2 (&a)[R]) {
    if constexpr (R == 2) {
        const float2 b = a[1];
        a[1] = csub(a[0], b);
        a[0] = cadd(a[0], b);
    } else if constexpr (R == 4) {
        dft4<INV>(a[0], a[1], a[2], a[3]);
    } else {
        constexpr int M = R / 4;
#pragma unroll
        for (int n = 0; n < M; ++n) dft4<INV>(a[n], a[M + n], a[2 * M + n], a[3 * M + n]);
#pragma unroll
        for (int k = 1; k < 4; ++k)
#pragma unroll
            for (int n = 1; n < M; ++n) a[M * k + n] = croot16<INV>(a[M * k + n], n * k * (16 / R));
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if constexpr (M == 4) {
                dft4<INV>(a[4 * k], a[4 * k + 1], a[4 * k + 2], a[4 * k + 3]);
            } else {
                const float2 b = a[2 * k + 1];
                a[2 * k + 1] = csub(a[2 * k], b);
                a[2 * k] = cadd(a[2 * k], b);
            }
        }
    }
}

// One step of radix R on transforms of NS values: v[m] is value t + m T of the
// line; on return v[q + r (16 / R)] is output r of butterfly t + q T.
template <int R, int NS, int T, bool INV>
__device__ __forceinline__ void step(float2 (&v)[PTS], int t, const float2 *tw) {
    constexpr int Q = PTS / R;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        float2 a[R];
        const int k = (t + q * T) % NS;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            a[r] = v[q + r * Q];
            if (NS > 1 && r) {
                float2 w = tw[(r - 1) * NS + k];
                if (!INV) w.y = -w.y;
                a[r] = cmul(a[r], w);
            }
        }
        dft<R, INV>(a);
#pragma unroll
        for (int r = 0; r < R; ++r) v[q + r * Q] = a[place<R>(r)];
    }
}

// After a step of radix 16 on NS values: the outputs to their places in the line,
// and the thread's values of the next step back.  STRIDE: lines interleaved.
template <int NS, int T, int STRIDE, bool SYNC>
__device__ __forceinline__ void exchange(float2 (&v)[PTS], int t, float2 *line) {
    const int base = (t / NS) * NS * 16 + t % NS;
    if (SYNC) __syncthreads();         // what others still read there
#pragma unroll
    for (int r = 0; r < PTS; ++r) line[padded(base + r * NS) * STRIDE] = v[r];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < PTS; ++m) v[m] = line[padded(t + m * T) * STRIDE];
}

// `last` runs before the last step, when the thread has its values in registers.
template <int N, int STRIDE, bool INV, bool SYNC, class F>
__device__ __forceinline__ void line_fft(float2 (&v)[PTS], int t, float2 *line, const float2 *tw, F last) {
    constexpr int T = N / PTS;
    step<16, 1, T, INV>(v, t, nullptr);
    exchange<1, T, STRIDE, SYNC>(v, t, line);
    if constexpr (N == 256) {
        last();
        step<16, 16, T, INV>(v, t, tw);
    } else {
        step<16, 16, T, INV>(v, t, tw);
        exchange<16, T, STRIDE, true>(v, t, line);
        last();
        step<N / 256, 256, T, INV>(v, t, tw + 15 * 16);
    }
}

template <int N> constexpr int ROW_LINES = N >= 2048 ? 1 : 2048 / N;   // rows a CTA: 128 threads, 256 at 4096

// Rows in place (INV), or rows of the image prepared as the grid (forward):
// (-1)^(qx+qy) I(q) / (c[qx] c[qy]), zero on row/col 0, N/2 further on.
template <int N, bool INV>
__global__ void __launch_bounds__(ROW_LINES<N> * N / PTS) fft_rows_kernel(float2 *g, const float *img,
                                                                         const float *corr, const float2 *tw) {
    extern __shared__ float2 sm[];
    constexpr int T = N / PTS;
    const int t = threadIdx.x % T, l = threadIdx.x / T;
    const int64_t row = (int64_t)blockIdx.x * ROW_LINES<N> + l;      // plane * N + row: a multiple of ROW_LINES rows
    float2 *z = g + row * N;
    float2 v[PTS];
    if constexpr (INV) {
#pragma unroll
        for (int m = 0; m < PTS; ++m) v[m] = __ldcs(z + t + m * T);
    } else {
        const int y = ((int)(row & (N - 1)) + N / 2) & (N - 1);
        const float *i = img + (row - (row & (N - 1)) + y) * N;
        float in[PTS];
#pragma unroll
        for (int m = 0; m < PTS; ++m) in[m] = __ldcs(i + ((t + m * T + N / 2) & (N - 1)));
        const float cy = corr[y];
#pragma unroll
        for (int m = 0; m < PTS; ++m) {
            const int x = (t + m * T + N / 2) & (N - 1);
            float p = 0.f;
            if (x != 0 && y != 0) {
                p = in[m] / (corr[x] * cy);
                if ((x + y) & 1) p = -p;
            }
            v[m] = make_float2(p, 0.f);
        }
    }
    line_fft<N, 1, INV, false>(v, t, sm + l * LINE_WORDS<N>, tw, [] {});
#pragma unroll
    for (int m = 0; m < PTS; ++m) z[t + m * T] = v[m];
}

template <int N> constexpr bool AHEAD = N == 4096;

// Columns in place; the inverse also leaves the image: (-1)^(qx+qy) Re / (c[qx]
// c[qy]) / weight_sum, zero on row/col 0.  A CTA takes tiles of COLS columns in
// turn (`per` a plane) and copies the next one to shared memory during the last
// step and the stores of this one.
template <int N, bool INV>
__global__ void __launch_bounds__(COLS<N> *N / PTS, 1024 / (COLS<N> * N / PTS)) fft_cols_kernel(float2 *g, float *img, const float *corr,
                                                                     float inv_wsum, int ntile, const float2 *tw) {
    extern __shared__ float2 sm[];
    constexpr int T = N / PTS, C = COLS<N>, per = N / C;
    const int c = threadIdx.x % C, t = threadIdx.x / C;
    float2 *line = sm + c;
    auto src = [&](int tile) { return g + (int64_t)(tile / per) * N * N + (tile % per) * C + c; };
    // .L2::128B: the neighbouring CTAs' sectors of the line come to L2 with it
    auto fetch = [&](int tile) {
        const float2 *z = src(tile);
#pragma unroll
        for (int m = 0; m < PTS; ++m) {
            const unsigned dst = (unsigned)__cvta_generic_to_shared(line + padded(t + m * T) * C);
            asm volatile("cp.async.ca.shared.global.L2::128B [%0], [%1], 8;"
                         :: "r"(dst), "l"(z + (int64_t)(t + m * T) * N) : "memory");
        }
    };
    if (AHEAD<N> && blockIdx.x < ntile) fetch(blockIdx.x);
    for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
        float2 v[PTS];
        if constexpr (AHEAD<N>) {
            asm volatile("cp.async.wait_all;" ::: "memory");      // a thread reads what it copied itself
#pragma unroll
            for (int m = 0; m < PTS; ++m) v[m] = line[padded(t + m * T) * C];
        } else {
            const float2 *z = src(tile);
#pragma unroll
            for (int m = 0; m < PTS; ++m)
                asm volatile("ld.global.L1::no_allocate.L2::128B.v2.f32 {%0, %1}, [%2];"
                             : "=f"(v[m].x), "=f"(v[m].y) : "l"(z + (int64_t)(t + m * T) * N) : "memory");
        }
        line_fft<N, C, INV, AHEAD<N>>(v, t, line, tw, [&] {
            if constexpr (AHEAD<N>) {
                __syncthreads();                                   // everyone has its values of the last exchange
                if (tile + (int)gridDim.x < ntile) fetch(tile + gridDim.x);
            }
        });
        const int zx = (tile % per) * C + c;
        const int64_t plane = (int64_t)(tile / per) * N * N;
        float2 *z = g + plane + zx;
#pragma unroll
        for (int m = 0; m < PTS; ++m) z[(int64_t)(t + m * T) * N] = v[m];
        if constexpr (INV) {
            const int x = (zx + N / 2) & (N - 1);
            const float cx = corr[x];
            float *o = img + plane + x;
#pragma unroll
            for (int m = 0; m < PTS; ++m) {
                const int y = (t + m * T + N / 2) & (N - 1);
                float p = 0.f;
                if (x != 0 && y != 0) p = (((x + y) & 1) ? -v[m].x : v[m].x) / (cx * corr[y]) * inv_wsum;
                o[(int64_t)y * N] = p;
            }
        }
    }
}

template <int N, bool INV>
int launch(aw_ctx *ctx, float2 *g, float *img_out, const float *img_in, const float *corr, float inv_wsum, int npol,
           const float2 *tw, cudaStream_t s) {
    constexpr int L = ROW_LINES<N>;
    const size_t rs = sizeof(float2) * LINE_WORDS<N> * L, cs = sizeof(float2) * LINE_WORDS<N> * COLS<N>;
    AW_CUDA_TRY(cudaFuncSetAttribute(fft_rows_kernel<N, INV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rs));
    AW_CUDA_TRY(cudaFuncSetAttribute(fft_cols_kernel<N, INV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cs));
    fft_rows_kernel<N, INV><<<(unsigned)(npol * N / L), L * N / PTS, rs, s>>>(g, img_in, corr, tw);
    AW_CHECK_LAUNCH();
    const int ntile = npol * (N / COLS<N>);
    const int nb = AHEAD<N> ? std::min(ntile, std::max(ctx->sm_count, 1)) : ntile;
    fft_cols_kernel<N, INV><<<nb, COLS<N> * N / PTS, cs, s>>>(g, img_out, corr, inv_wsum, ntile, tw);
    AW_CHECK_LAUNCH();
    return AW_OK;
}

template <bool INV>
int launch_n(aw_ctx *ctx, int N, float2 *g, float *img_out, const float *img_in, const float *corr, float inv_wsum, int npol,
             const float2 *tw, cudaStream_t s) {
    switch (N) {
        case 256: return launch<256, INV>(ctx, g, img_out, img_in, corr, inv_wsum, npol, tw, s);
        case 512: return launch<512, INV>(ctx, g, img_out, img_in, corr, inv_wsum, npol, tw, s);
        case 1024: return launch<1024, INV>(ctx, g, img_out, img_in, corr, inv_wsum, npol, tw, s);
        case 2048: return launch<2048, INV>(ctx, g, img_out, img_in, corr, inv_wsum, npol, tw, s);
        case 4096: return launch<4096, INV>(ctx, g, img_out, img_in, corr, inv_wsum, npol, tw, s);
    }
    return aw_set_error(AW_EINVAL, "transform size %d", N);
}

// Twiddle factors exp(2 pi i r k / (NS R)), r = 1 ... R-1, k < NS, of the steps
// after the first.
int twiddles(aw_ctx *ctx, int N, float2 **out) {
    auto it = ctx->twiddle.find(N);
    if (it != ctx->twiddle.end()) { *out = it->second; return AW_OK; }
    std::vector<float2> w;
    for (int NS = 16; NS < N; NS *= 16) {
        const int R = N / NS < 16 ? N / NS : 16;
        for (int r = 1; r < R; ++r)
            for (int k = 0; k < NS; ++k) {
                const double a = 2.0 * M_PI * r * k / ((double)NS * R);
                w.push_back(make_float2((float)cos(a), (float)sin(a)));
            }
    }
    float2 *d = nullptr;
    AW_CUDA_TRY(aw_dev_malloc(&d, sizeof(float2) * w.size()));
    cudaError_t e = cudaMemcpy(d, w.data(), sizeof(float2) * w.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
    if (e != cudaSuccess) {
        aw_dev_free(d);
        return aw_set_error(AW_ECUDA, "twiddle table: %s", cudaGetErrorString(e));
    }
    ctx->twiddle[N] = d;
    *out = d;
    return AW_OK;
}

}  // namespace

bool aw_fft_has(int N) { return N >= 256 && N <= 4096; }

int aw_fft_grid_to_image(aw_ctx *ctx, int N, int npol, float2 *g, const float *corr, float inv_wsum, float *image,
                         cudaStream_t s) {
    float2 *tw = nullptr;
    const int rc = twiddles(ctx, N, &tw);
    if (rc) return rc;
    return launch_n<true>(ctx, N, g, image, nullptr, corr, inv_wsum, npol, tw, s);
}

int aw_fft_image_to_grid(aw_ctx *ctx, int N, int npol, const float *image, const float *corr, float2 *g,
                         cudaStream_t s) {
    float2 *tw = nullptr;
    const int rc = twiddles(ctx, N, &tw);
    if (rc) return rc;
    return launch_n<false>(ctx, N, g, nullptr, image, corr, 0.f, npol, tw, s);
}
