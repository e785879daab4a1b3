// Internal declarations shared by the libaw translation units.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <cufft.h>
#include <nvtx3/nvToolsExt.h>
#include <stdint.h>

#include <cstdarg>
#include <map>
#include <string>
#include <tuple>
#include <vector>

#include "aw.h"

#define AW_C_LIGHT 299792458.0

// ---------------------------------------------------------------- errors
int aw_set_error(int code, const char *fmt, ...);

#define AW_CUDA_TRY(call)                                                             \
    do {                                                                              \
        cudaError_t e_ = (call);                                                      \
        if (e_ != cudaSuccess)                                                        \
            return aw_set_error(e_ == cudaErrorMemoryAllocation ? AW_ENOMEM : AW_ECUDA, \
                                "%s: %s (%s:%d)", #call, cudaGetErrorString(e_),       \
                                __FILE__, __LINE__);                                  \
    } while (0)

#define AW_CUFFT_TRY(call)                                                            \
    do {                                                                              \
        cufftResult r_ = (call);                                                      \
        if (r_ != CUFFT_SUCCESS)                                                      \
            return aw_set_error(r_ == CUFFT_ALLOC_FAILED ? AW_ENOMEM : AW_ECUDA,        \
                                "%s: cufft error %d (%s:%d)", #call, (int)r_,          \
                                __FILE__, __LINE__);                                  \
    } while (0)

#define AW_CHECK_LAUNCH() AW_CUDA_TRY(cudaGetLastError())

// ---------------------------------------------------------------- tracing
// An NVTX range named after the ABI function for the duration of the call
// (visible to profilers that attach; free otherwise).
struct AwTrace {
    explicit AwTrace(const char *name) { nvtxRangePushA(name); }
    ~AwTrace() { nvtxRangePop(); }
    AwTrace(const AwTrace &) = delete;
    AwTrace &operator=(const AwTrace &) = delete;
};
#define AW_TRACE() AwTrace aw_trace_(__func__)

// ---------------------------------------------------------------- device memory
// Every device buffer of the library goes through these: they count the live
// buffers and let aw_debug_fail_alloc make a chosen allocation fail.
cudaError_t aw_dev_malloc_raw(void **p, size_t bytes);
void aw_dev_free(void *p);
template <class T>
inline cudaError_t aw_dev_malloc(T **p, size_t bytes) {
    return aw_dev_malloc_raw(reinterpret_cast<void **>(p), bytes);
}

// ---------------------------------------------------------------- handles
struct aw_ctx {
    int device = 0;
    int sm_count = 0;
    // cuFFT plans keyed by (rank tag, size, batch, type)
    std::map<std::tuple<int, int, int, int>, cufftHandle> fft_plans;
    // grid-correction vectors keyed by (N, W)
    std::map<std::pair<int, double>, float *> gridcorr;
    // twiddle factors of the library's own transforms, by N
    std::map<int, float2 *> twiddle;
    // small device scratch: [0] reduction word for mosaic_gamma
    unsigned int *d_scratch = nullptr;
    // last aw_autotune result (used by aw_plan_create when given no tune)
    bool has_tune = false;
    aw_tune tune_cache{};
};

struct aw_kernel_set {
    int device = 0;
    aw_kernel_spec spec{};          // copied; pointer members re-pointed to the vectors
    std::vector<int32_t> supports;  // per w plane
    std::vector<double> pa, fbin_freqs;
    std::vector<double> type_leak;  // [ntype][4] per-type leakage (ntype >= 2)
    int ntype = 1;                  // antenna types; baseline classes = ntype^2 if >= 2
    int nclass = 1;
    int nbins = 0;
    int P = 1;                      // npol * npol
    int max_support = 0;
    std::vector<int32_t> bin_support;
    std::vector<int64_t> bin_offset;  // element offset of each bin (complex elements)
    int64_t total_elems = 0;
    int elem_bytes = 8;
    // complex values per 16-byte chunk of the table layout (see aw_tab_index)
    int ce = 1;
    void *d_table = nullptr;
    int32_t *d_bin_support = nullptr;
    int64_t *d_bin_offset = nullptr;
    int n_rejected = 0;
    // tables hold K * scale (a power of two; != 1 only for FP16 storage, to keep
    // the kernel values inside the FP16 normal range)
    float scale = 1.0f;
};

// One sorted visibility: 16 bytes.
struct __align__(16) aw_rec {
    uint32_t orig;   // caller index
    uint16_t x0, y0; // first footprint cell
    uint16_t bin;
    uint8_t fx, fy;  // fine offsets
    uint8_t flip;
    uint8_t pad0;
    uint16_t pad1;
};
static_assert(sizeof(aw_rec) == 16, "aw_rec must be 16 bytes");

struct aw_plan {
    int device = 0;
    int64_t nvis = 0, nvalid = 0, n_outside = 0, n_flagged = 0, nitems = 0;
    int N = 0, OS = 0, npol = 1, nbins = 0, nw = 1, npa = 1, nfb = 1;
    int ntype = 1;                  // baseline classes are ntype^2 when ntype >= 2
    aw_tune tune{};
    double mean_taps = 0;
    aw_rec *d_rec = nullptr;        // [nvis] sorted (valid first) by (bin, tile, position)
    int4 *d_items = nullptr;        // [nitems] {start, count, bin, 0}
    // degridding order: the valid visibilities by (bin, super-tile, oversampled
    // offset, position), cut into items of at most AW_DG_CHUNK visibilities
    aw_rec *d_rec_dg = nullptr;     // [nvalid]
    int4 *d_items_dg = nullptr;     // [nitems_dg] {start, count, bin, 0}
    int64_t nitems_dg = 0;
    int dg_tile = 1024;
    int32_t *d_plane_support = nullptr;  // [nw] support per w plane
    double *d_fl = nullptr;              // [nchan] frequency / c
    std::vector<int32_t> bin_support;
    // grid-time statistics (device): [0] weight sum (double), [1] non-finite count
    double *d_wsum = nullptr;
    unsigned long long *d_nonfinite = nullptr;
    unsigned int *d_counter = nullptr;  // persistent work-queue head
    // AW_GRID_HYBRID: the gridding items of the low w planes (TILES) and the
    // degridding items of the others (OFFSETS), and the second stream the
    // OFFSETS part runs on (fork and join through the two events)
    int4 *d_items_ht = nullptr;
    int64_t nitems_ht = 0;
    int4 *d_items_ho = nullptr;
    int64_t nitems_ho = 0;
    cudaStream_t aux = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    // AW_GRID_REGION: the valid visibilities of the bins on the region kernels,
    // by (bin, region tile, oversampled offset, position), cut into tasks
    // {start, count, bin, aw_rg_pack(tile, footprint block)}.  The other bins'
    // degridding items (d_items_ho) take the OFFSETS schedule on the second
    // stream.
    aw_rec *d_rec_rg = nullptr;
    int64_t nreg = 0;
    int4 *d_items_rg = nullptr;
    int64_t nitems_rg = 0;
    // Stokes I: the region degridding tasks over the same records (all blocks of
    // a footprint in one task)
    int4 *d_items_rgd = nullptr;
    int64_t nitems_rgd = 0;
    unsigned int *d_rcounter = nullptr;   // work-queue head of the region gridding (behind d_counter)
    // coordinate inputs kept for aw_plan_coords
    aw_vis_desc vis{};
    double uscale = 0, half = 0, winv = 0;
    // graphs of aw_grid_batched for the last two argument sets (double-buffered
    // callers alternate between two), least recently used replaced first
    struct GraphSlot {
        cudaGraphExec_t exec = nullptr;
        const void *vis = nullptr, *weight = nullptr, *grid = nullptr, *kset = nullptr;
        cudaStream_t stream = nullptr;
        uint64_t used = 0;
    };
    GraphSlot gslots[2];
    uint64_t gclock = 0;
    void drop_graphs() {
        for (auto &g : gslots) {
            if (g.exec) cudaGraphExecDestroy(g.exec);
            g = GraphSlot{};
        }
    }
};

// ---------------------------------------------------------------- regions
// REGION schedule: a CTA accumulates one plane of a grid region of AW_RG_R x
// AW_RG_R cells in shared memory.  A footprint of S x S taps is cut along each
// axis into blocks of 24 or 16 taps (one of 8 for S <= 8; the last block may
// reach past the footprint, its absent taps have kernel value 0), and a task
// is one block of the footprints that start in one T x T grid tile, T + block
// - 1 <= AW_RG_R.
constexpr int AW_RG_R = 56;
constexpr int AW_RG_MAXV = 1024;      // visibilities per gridding task
constexpr int AW_RG_MAXV_DG = 256;   // visibilities per degridding task

// blocks along an axis: n24 of 24 taps, then n16 of 16 (S <= 8: one of 8)
__host__ __device__ inline int aw_rg_n24(int S) {
    const int k = (S + 7) / 8;
    return k <= 1 ? 0 : (k - (k % 3 == 0 ? 0 : k % 3 == 2 ? 2 : 4)) / 3;
}
__host__ __device__ inline int aw_rg_nblk(int S) {
    const int k = (S + 7) / 8;
    return k <= 1 ? 1 : aw_rg_n24(S) + (k % 3 == 0 ? 0 : k % 3 == 2 ? 1 : 2);
}
__host__ __device__ inline int aw_rg_blk_width(int S, int i) { return S <= 8 ? 8 : i < aw_rg_n24(S) ? 24 : 16; }
__host__ __device__ inline int aw_rg_blk_first(int S, int i) {
    const int a = aw_rg_n24(S);
    return i <= a ? 24 * i : 24 * a + 16 * (i - a);
}
__host__ __device__ inline int aw_rg_tile(int S) {
    return AW_RG_R + 1 - (S <= 8 ? 8 : aw_rg_n24(S) ? 24 : 16);
}
// Supports on the region kernels: padding the footprint to a multiple of 8 taps
// a side costs at most 1.8 times the taps (about what OFFSETS costs more).
// Stokes I: up to 48 cells (wider ones hold few visibilities a tile).  A set with
// no support above AW_RG_MIN_SUPPORT stays on OFFSETS: blocks of 8 x 8 taps alone
// give the region kernel too little to do between its barriers (300k full-pol
// visibilities of 8 x 8 taps: 149 us against 189; 126k of 7 x 7 in Stokes I: 29
// against 35), beside wider ones they are better off there than on OFFSETS' one CTA
// per SM (3M with supports 8-64: 5.0 ms against 6.3).
constexpr int AW_RG_MIN_SUPPORT = 8;
inline bool aw_rg_eligible(int S, int npol) {
    const int p = (S + 7) / 8 * 8;
    return S >= 2 && S <= (npol == 1 ? 48 : 128) && 10 * p * p <= 18 * S * S;
}
// task word: tile column and row (9 bits each: at most 16384 / 33), block column and row (3 bits each)
__host__ __device__ inline int aw_rg_pack(int tx, int ty, int bx, int by) {
    return tx | ty << 9 | bx << 18 | by << 21;
}
// Whether 32-bit words hold the task positions and the queue head, which counts a
// task once a plane and, at the end, once more for every CTA: a set of more tasks
// (above a thousand million segments of one visibility or so) takes OFFSETS.
inline bool aw_rg_fits(unsigned long long ntasks, int npol) {
    return ntasks <= (0xffffffffull - (1ull << 20)) / (unsigned)npol;
}

// Visibilities per degridding work item: 8 warps x 4 visibilities.
constexpr int AW_DG_VB = 4;
constexpr int AW_DG_CHUNK = 8 * AW_DG_VB;

// ---------------------------------------------------------------- table layout
// Inside one (bin, fy, fx) block of L = S*S taps, the P Mueller values of a tap
// are split into 16-byte chunks of `ce` complex values (ce = 2 for FP32, 4 for
// 16-bit storage, or P if P is smaller) and stored chunk-major, tap-minor:
// index(tap, m) = ((m / ce) * L + tap) * ce + m % ce.  Threads that handle
// consecutive taps then read consecutive 16-byte words (coalesced loads).
__host__ __device__ inline int64_t aw_tab_index(int ce, int64_t L, int64_t tap, int m) {
    return ((int64_t)(m / ce) * L + tap) * ce + (m % ce);
}

// ---------------------------------------------------------------- helpers
int aw_ctx_fft_plan(aw_ctx *ctx, int rank_tag, int n, int batch, cufftType type, cufftHandle *out);
int aw_ctx_gridcorr(aw_ctx *ctx, int N, double W, float **out);

// PSWF taper psi(x), psi(0) = 1, from the Legendre eigen-expansion (host).
struct aw_pswf {
    std::vector<double> beta;  // coefficients of Pbar_{2k}
    double norm = 1.0;         // 1 / psi_unnormalised(0)
    double eval(double x) const;
};
aw_pswf aw_pswf_make(double c, int nterms = 48);

// Exclusive scan of uint32 (n up to 2^31) with caller scratch from aw_scan_scratch_bytes.
size_t aw_scan_scratch_bytes(int64_t n);
int aw_exclusive_scan_u32(const uint32_t *in, uint32_t *out, int64_t n, void *scratch,
                          cudaStream_t s);

// Grid / degrid launchers (aw_grid.cu).
struct aw_grid_launch {
    const aw_plan *plan;
    const aw_kernel_set *kset;
    const void *vis;
    const float *weight;
    void *grid;
    bool persistent;
    int ctas;
    cudaStream_t stream;
    // one schedule over a subset of its items (the parts of AW_GRID_HYBRID);
    // mode < 0: the plan's own schedule over all its items
    int mode = -1;
    const int4 *items = nullptr;
    int64_t nitems = 0;
};
int aw_launch_grid(const aw_grid_launch &L);
// REGION schedule (aw_grid_region.cu): the gridding tasks of a plan on stream s.
int aw_launch_grid_region(const aw_plan *p, const aw_kernel_set *k, const void *vis, const float *weight, void *grid,
                          cudaStream_t s);
int aw_region_bounds_status(unsigned int *v, int reset);
// Region degridding (aw_degrid_region.cu) of the plan's region tasks, and zero
// (or sub_from) for the visibilities that are not gridded.
int aw_launch_degrid_region(const aw_plan *p, const aw_kernel_set *k, const void *grid, void *vis_out,
                            cudaStream_t s, const void *sub_from);
int aw_degrid_region_bounds_status(unsigned int *v, int reset);
// cum[q] = share of the plan's visibility-taps (sum of S^2) in w planes < q, q = 0..nw
int aw_plan_plane_taps(const aw_plan *plan, std::vector<double> &cum, cudaStream_t s);
int aw_launch_degrid(const aw_plan *plan, const aw_kernel_set *kset, const void *grid,
                     void *vis_out, cudaStream_t stream, const void *sub_from = nullptr);
// The library's own two-pass transforms (aw_fft.cu), for the N that it has.
bool aw_fft_has(int N);
int aw_fft_grid_to_image(aw_ctx *ctx, int N, int npol, float2 *g, const float *corr, float inv_wsum, float *image,
                         cudaStream_t s);
int aw_fft_image_to_grid(aw_ctx *ctx, int N, int npol, const float *image, const float *corr, float2 *g,
                         cudaStream_t s);
int aw_fft_to_image_impl(aw_ctx *ctx, int N, int npol, double W, void *grid, double weight_sum,
                         float *image, cudaStream_t s);
int aw_image_to_grid_impl(aw_ctx *ctx, int N, int npol, double W, const float *image, void *grid,
                          cudaStream_t s);

// Storage conversion (aw_synth.cu).
int aw_export_table(const void *src, float2 *dst, int64_t nblocks, int L, int P, int ce, int storage,
                    float inv_scale, cudaStream_t s);
int aw_convert_table_scaled(const float2 *src, void *dst, int64_t nblocks, int L, int P, int ce, int storage,
                            float scale, cudaStream_t s);
int aw_table_absmax(const float2 *src, int64_t n, float *out_host, cudaStream_t s);
