// uv grid -> dirty image (Sec. 2.2: FFTs on the GPU) and the mosaic
// weighting gamma(l, m) of Eq. 1 (Sec. 2.2).
#include <cmath>

#include "aw_internal.h"

namespace {

// The centring phases (-1)^(x + y) of both sides of a transform: those of one
// side are a shift of the other side by N/2 on each axis (N a multiple of 4), so
// they are applied as signs on the image side and as a shifted position, also on
// the image side, and the grid needs no pass of its own.  The kernels here are for
// the N that have no transform of the library's own.  A CTA works on one
// row of one plane (blockIdx.y, blockIdx.z), a thread on V pixels of it; V = 4
// for arrays aligned to 16 bytes.

// image = (-1)^(qx+qy) Re(Z) / (c[qx] c[qy]) / weight_sum, zero on row/col 0; Z is
// the transform of the plain grid, read N/2 further on
template <int V>
__global__ void gridcorr_kernel(const float2 *Z, const float *corr, int N, float inv_wsum, float *img) {
    const int y = blockIdx.y, x = V * (blockIdx.x * blockDim.x + threadIdx.x);
    if (x >= N) return;
    const int64_t plane = (int64_t)blockIdx.z * N * N;
    const float2 *z = Z + plane + (int64_t)((y + N / 2) & (N - 1)) * N + ((x + N / 2) & (N - 1));
    float re[V], v[V];
    if constexpr (V == 4) {
        const float4 a = reinterpret_cast<const float4 *>(z)[0], b = reinterpret_cast<const float4 *>(z)[1];
        re[0] = a.x; re[1] = a.z; re[2] = b.x; re[3] = b.z;
    } else {
        re[0] = z[0].x;
    }
    const float cy = corr[y];
#pragma unroll
    for (int j = 0; j < V; ++j) {
        v[j] = 0.f;
        if (x + j != 0 && y != 0) v[j] = (((x + j + y) & 1) ? -re[j] : re[j]) / (corr[x + j] * cy) * inv_wsum;
    }
    float *o = img + plane + (int64_t)y * N + x;
    if constexpr (V == 4) *reinterpret_cast<float4 *>(o) = make_float4(v[0], v[1], v[2], v[3]);
    else o[0] = v[0];
}

// grid = (-1)^(qx+qy) I(q) / (c[qx] c[qy]) as complex, zero on row/col 0, written
// N/2 further on: a plain forward FFT then gives the model's uv grid
template <int V>
__global__ void image_prep_kernel(const float *img, const float *corr, int N, float2 *g) {
    const int y = blockIdx.y, x = V * (blockIdx.x * blockDim.x + threadIdx.x);
    if (x >= N) return;
    const int64_t plane = (int64_t)blockIdx.z * N * N;
    const float *i = img + plane + (int64_t)y * N + x;
    float in[V], v[V];
    if constexpr (V == 4) {
        const float4 a = *reinterpret_cast<const float4 *>(i);
        in[0] = a.x; in[1] = a.y; in[2] = a.z; in[3] = a.w;
    } else {
        in[0] = i[0];
    }
    const float cy = corr[y];
#pragma unroll
    for (int j = 0; j < V; ++j) {
        v[j] = 0.f;
        if (x + j != 0 && y != 0) {
            v[j] = in[j] / (corr[x + j] * cy);
            if ((x + j + y) & 1) v[j] = -v[j];
        }
    }
    float2 *o = g + plane + (int64_t)((y + N / 2) & (N - 1)) * N + ((x + N / 2) & (N - 1));
    if constexpr (V == 4) {
        reinterpret_cast<float4 *>(o)[0] = make_float4(v[0], 0.f, v[1], 0.f);
        reinterpret_cast<float4 *>(o)[1] = make_float4(v[2], 0.f, v[3], 0.f);
    } else {
        o[0] = make_float2(v[0], 0.f);
    }
}

// gamma at sum B^2 = s, max sqrt(sum B^2) = mx
__device__ __forceinline__ float gamma_of(float s, float mx, float eps) {
    const float pbp = (mx > 0.f) ? sqrtf(s) / mx : 0.f;   // [sqrt(sum B^2) / max]_pbp
    const float wc = (s > 0.f) ? 1.0f / s : 0.f;           // [1 / sum B^2]_wc
    return (pbp < eps || s == 0.f) ? 0.f : pbp * wc;
}

__global__ void gamma_max_kernel(const float *B, int nfield, int64_t npix, unsigned int *maxbits) {
    float m = 0.f;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < npix;
         i += (int64_t)gridDim.x * blockDim.x) {
        float s = 0.f;
        for (int f = 0; f < nfield; ++f) {
            const float b = B[(int64_t)f * npix + i];
            s = fmaf(b, b, s);
        }
        m = fmaxf(m, sqrtf(s));
    }
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(maxbits, __float_as_uint(m));
}

__global__ void gamma_apply_kernel(const float *B, int nfield, int64_t npix, const unsigned int *maxbits,
                                   float eps, float *gamma) {
    const float mx = __uint_as_float(*maxbits);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < npix;
         i += (int64_t)gridDim.x * blockDim.x) {
        float s = 0.f;
        for (int f = 0; f < nfield; ++f) {
            const float b = B[(int64_t)f * npix + i];
            s = fmaf(b, b, s);
        }
        gamma[i] = gamma_of(s, mx, eps);
    }
}

// The same two passes on four pixels a thread (arrays 16-byte aligned, npix a
// multiple of 4): the first leaves sum B^2 in gamma, so that the beams are read
// once.
__global__ void __launch_bounds__(256) gamma_sum4_kernel(const float4 *B, int nfield, int64_t nq,
                                                         unsigned int *maxbits, float4 *sum) {
    float m = 0.f;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nq; i += (int64_t)gridDim.x * blockDim.x) {
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int f = 0; f < nfield; ++f) {
            const float4 b = __ldcs(B + (int64_t)f * nq + i);
            s.x = fmaf(b.x, b.x, s.x);
            s.y = fmaf(b.y, b.y, s.y);
            s.z = fmaf(b.z, b.z, s.z);
            s.w = fmaf(b.w, b.w, s.w);
        }
        sum[i] = s;
        m = fmaxf(m, fmaxf(fmaxf(sqrtf(s.x), sqrtf(s.y)), fmaxf(sqrtf(s.z), sqrtf(s.w))));
    }
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(maxbits, __float_as_uint(m));
}

__global__ void __launch_bounds__(256) gamma_final4_kernel(int64_t nq, const unsigned int *maxbits, float eps,
                                                           float4 *gamma) {
    const float mx = __uint_as_float(*maxbits);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nq; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 s = gamma[i];
        gamma[i] = make_float4(gamma_of(s.x, mx, eps), gamma_of(s.y, mx, eps), gamma_of(s.z, mx, eps),
                               gamma_of(s.w, mx, eps));
    }
}

int nblocks(int64_t n, int t) {
    int64_t b = (n + t - 1) / t;
    if (b < 1) b = 1;
    if (b > 152 * 32) b = 152 * 32;
    return (int)b;
}

bool aligned16(const void *a, const void *b) { return ((uintptr_t)a | (uintptr_t)b) % 16 == 0; }

// Launch shape of the row kernels above with V pixels a thread.
void row_shape(int N, int npol, int V, dim3 &grid, dim3 &block) {
    const int n = (N + V - 1) / V;
    block = dim3((unsigned)(n < 256 ? n : 256));
    grid = dim3((unsigned)((n + block.x - 1) / block.x), (unsigned)N, (unsigned)npol);
}

}  // namespace

int aw_ctx_gridcorr(aw_ctx *ctx, int N, double W, float **out) {
    auto key = std::make_pair(N, W);
    auto it = ctx->gridcorr.find(key);
    if (it != ctx->gridcorr.end()) { *out = it->second; return AW_OK; }
    const aw_pswf p = aw_pswf_make(M_PI * W / 2.0);
    std::vector<float> c(N);
    for (int q = 0; q < N; ++q) c[q] = (q == 0) ? 0.f : (float)p.eval((q - N / 2) * 2.0 / N);
    float *d = nullptr;
    AW_CUDA_TRY(aw_dev_malloc(&d, sizeof(float) * N));
    AW_CUDA_TRY(cudaMemcpy(d, c.data(), sizeof(float) * N, cudaMemcpyHostToDevice));
    ctx->gridcorr[key] = d;
    *out = d;
    return AW_OK;
}

int aw_fft_to_image_impl(aw_ctx *ctx, int N, int npol, double W, void *grid, double weight_sum,
                         float *image, cudaStream_t s) {
    if (N % 4) return aw_set_error(AW_EINVAL, "N must be a multiple of 4");
    if (!(weight_sum > 0)) return aw_set_error(AW_EINVAL, "weight_sum must be positive");
    float *corr = nullptr;
    int rc = aw_ctx_gridcorr(ctx, N, W, &corr);
    if (rc) return rc;
    float2 *g = reinterpret_cast<float2 *>(grid);
    const float inv = (float)(1.0 / weight_sum);
    if (aw_fft_has(N)) return aw_fft_grid_to_image(ctx, N, npol, g, corr, inv, image, s);
    cufftHandle plan;
    rc = aw_ctx_fft_plan(ctx, 2, N, npol, CUFFT_C2C, &plan);
    if (rc) return rc;
    AW_CUFFT_TRY(cufftSetStream(plan, s));
    AW_CUFFT_TRY(cufftExecC2C(plan, reinterpret_cast<cufftComplex *>(g), reinterpret_cast<cufftComplex *>(g),
                              CUFFT_INVERSE));
    dim3 nb, nt;
    if (aligned16(g, image)) {
        row_shape(N, npol, 4, nb, nt);
        gridcorr_kernel<4><<<nb, nt, 0, s>>>(g, corr, N, inv, image);
    } else {
        row_shape(N, npol, 1, nb, nt);
        gridcorr_kernel<1><<<nb, nt, 0, s>>>(g, corr, N, inv, image);
    }
    AW_CHECK_LAUNCH();
    return AW_OK;
}

// G(g) = sum_q I(q) / c(q) exp(-2 pi i (g - N/2)(q - N/2) / N): with N a multiple
// of 4 the centring phases reduce to (-1)^(q) and a shift of the image by N/2
// before a plain forward FFT.
int aw_image_to_grid_impl(aw_ctx *ctx, int N, int npol, double W, const float *image, void *grid,
                          cudaStream_t s) {
    if (N % 4) return aw_set_error(AW_EINVAL, "N must be a multiple of 4");
    float *corr = nullptr;
    int rc = aw_ctx_gridcorr(ctx, N, W, &corr);
    if (rc) return rc;
    float2 *g = reinterpret_cast<float2 *>(grid);
    if (aw_fft_has(N)) return aw_fft_image_to_grid(ctx, N, npol, image, corr, g, s);
    cufftHandle plan;
    rc = aw_ctx_fft_plan(ctx, 2, N, npol, CUFFT_C2C, &plan);
    if (rc) return rc;
    AW_CUFFT_TRY(cufftSetStream(plan, s));
    dim3 nb, nt;
    if (aligned16(g, image)) {
        row_shape(N, npol, 4, nb, nt);
        image_prep_kernel<4><<<nb, nt, 0, s>>>(image, corr, N, g);
    } else {
        row_shape(N, npol, 1, nb, nt);
        image_prep_kernel<1><<<nb, nt, 0, s>>>(image, corr, N, g);
    }
    AW_CHECK_LAUNCH();
    AW_CUFFT_TRY(cufftExecC2C(plan, reinterpret_cast<cufftComplex *>(g), reinterpret_cast<cufftComplex *>(g),
                              CUFFT_FORWARD));
    return AW_OK;
}

int aw_mosaic_gamma_impl(aw_ctx *ctx, const float *beams, int nfield, int N, float eps, float *gamma,
                         cudaStream_t s) {
    const int64_t npix = (int64_t)N * N;
    AW_CUDA_TRY(cudaMemsetAsync(ctx->d_scratch, 0, sizeof(unsigned int), s));
    if (npix % 4 == 0 && aligned16(beams, gamma) &&
        (gamma + npix <= beams || gamma >= beams + (int64_t)nfield * npix)) {
        const int64_t nq = npix / 4;
        gamma_sum4_kernel<<<nblocks(nq, 256), 256, 0, s>>>(reinterpret_cast<const float4 *>(beams), nfield, nq,
                                                          ctx->d_scratch, reinterpret_cast<float4 *>(gamma));
        AW_CHECK_LAUNCH();
        gamma_final4_kernel<<<nblocks(nq, 256), 256, 0, s>>>(nq, ctx->d_scratch, eps, reinterpret_cast<float4 *>(gamma));
        AW_CHECK_LAUNCH();
        return AW_OK;
    }
    gamma_max_kernel<<<nblocks(npix, 256), 256, 0, s>>>(beams, nfield, npix, ctx->d_scratch);
    AW_CHECK_LAUNCH();
    gamma_apply_kernel<<<nblocks(npix, 256), 256, 0, s>>>(beams, nfield, npix, ctx->d_scratch, eps, gamma);
    AW_CHECK_LAUNCH();
    return AW_OK;
}
