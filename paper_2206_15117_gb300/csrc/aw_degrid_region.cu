// Stokes-I degridding of REGION plans: a grid region in shared memory, kernel
// taps in registers.
//
// arXiv:2206.15117 Sec. 3.2: a predicted visibility is the model grid under its
// footprint weighted with the kernel of its bin and oversampled offset, V =
// sum_j K(jy, jx; fy, fx) G[y0 + jy][x0 + jx].
//
// A task is the visibilities of one bin whose footprints start in one grid tile
// (the order and tiles of the region gridding), at most RD_MAXV.  For each block
// of the footprint (24 or 16 taps a side) the CTA copies the tile's region into
// shared memory; a warp then takes runs of equal offset, holds the block's taps
// in registers (lane (r, c) of 4 x 8 the taps (r + 4 i, c + 8 j)) and forms four
// visibilities at a time, whose eight partial sums are reduced over the lanes
// together.  A warp alone adds to a visibility, so no atomics are needed.
//
// What bounds it: the shared-memory pipe (8 bytes a visibility-tap) and, at the
// small supports, the reductions.  20.16M visibilities at 2048^2, supports 8-64:
// 2.9 ms (that pipe 74 % busy) against 5.8 ms reading the grid through L1, one
// gather per tap (load latency).  On a GPU where 128 threads and 6 CTAs an SM take
// 2.76 ms: 4 CTAs 3.60, 64 threads and 8 CTAs 3.72, 256 threads and 4 CTAs 3.06 ms.
#include <algorithm>

#include "aw_internal.h"

#ifdef AW_BOUNDS_CHECK
__device__ unsigned int g_bounds_status_rd;
#endif

namespace {

#ifdef AW_BOUNDS_CHECK
__device__ __forceinline__ bool rd_bounds_ok(bool ok, unsigned int code) {
    if (!ok) atomicCAS(&g_bounds_status_rd, 0u, code);
    return ok;
}
#define RD_BOK(cond, code) rd_bounds_ok((cond), (code))
#else
#define RD_BOK(cond, code) true
#endif

enum : unsigned int { BC_P_REC = 19, BC_P_CELL, BC_P_TAB, BC_P_SMEM };

constexpr int RR = AW_RG_R;           // region side = row stride in cells
constexpr int RD_MAXV = AW_RG_MAXV_DG;
constexpr int RD_THREADS = 128;
constexpr int RD_CTAS = 6;

struct RegionDegridArgs {
    const aw_rec *rec_all;      // grid order: [nvalid, nvis) are the visibilities not gridded
    const aw_rec *rec;          // region order
    const int4 *items;          // {start, count, bin, aw_rg_pack(tile, -)}
    int64_t nitems;
    const void *ktab;
    const int64_t *bin_offset;
    const int32_t *bin_support;
    const float2 *grid;
    float2 *vis_out;
    const float2 *sub_from;     // SUB: vis_out = sub_from - prediction (may alias vis_out)
    int N, OS;
    float inv_scale;
    int64_t nvis, nvalid, nreg, tab_elems;
};

struct __align__(16) DegridSmem {
    float2 reg[RR * RR];
    float2 out[RD_MAXV];
    int cell[RD_MAXV + 4];      // (read ahead in fours)
    uint16_t off[RD_MAXV];
    uint16_t run[RD_MAXV + 1];  // starts of the runs of equal offset
    int nrun;
    int wsum[RD_THREADS / 32];
};

template <int ST>
__device__ __forceinline__ float2 tap_value(const void *tab, int64_t idx) {
    if constexpr (ST == AW_STORAGE_FP32) {
        return __ldg(reinterpret_cast<const float2 *>(tab) + idx);
    } else {
        const uint32_t w = __ldg(reinterpret_cast<const uint32_t *>(tab) + idx);
        if constexpr (ST == AW_STORAGE_BF16) return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w));
        else return __half22float2(*reinterpret_cast<const __half2 *>(&w));
    }
}

// The runs of a task on one footprint block of 8 CB columns and 4 RB rows.
// PAD: the block may reach past the footprint; cells of absent taps are not used.
template <int ST, int CB, int RB, bool PAD>
__device__ __forceinline__ void run_block(DegridSmem &sm, const RegionDegridArgs &a, int64_t tab0, int S, int fy,
                                          int fx) {
    constexpr int NT = CB * RB;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r = lane >> 3, c = lane & 7;
    // a long run is shared by all warps, four visibilities at a time; the short
    // ones go to the warps in turn
    for (int run = 0; run < sm.nrun; ++run) {
        const int j0 = sm.run[run], j1 = sm.run[run + 1];
        const bool shared_run = j1 - j0 > 4 * (RD_THREADS / 32);
        if (!shared_run && run % (RD_THREADS / 32) != warp) continue;
        const int64_t kb = tab0 + (int64_t)sm.off[j0] * S * S;
        const bool kok = RD_BOK(kb >= 0 && kb + (int64_t)S * S <= a.tab_elems, BC_P_TAB);
        float2 k[NT];
        unsigned on = 0;
#pragma unroll
        for (int i = 0; i < RB; ++i)
#pragma unroll
            for (int j = 0; j < CB; ++j) {
                const int ty = fy + r + 4 * i, tx = fx + c + 8 * j;
                const bool ok = (!PAD || (ty < S && tx < S)) && kok;
                if (ok) on |= 1u << (i * CB + j);
                k[i * CB + j] = ok ? tap_value<ST>(a.ktab, kb + ty * S + tx) : make_float2(0.f, 0.f);
            }
        const float2 *base = sm.reg + r * RR + c;
        const int jb = shared_run ? j0 + 4 * warp : j0, js = shared_run ? 4 * (RD_THREADS / 32) : 4;
#pragma unroll 1
        for (int j = jb; j < j1; j += js) {
            float x[8];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                // (past the run's end: another visibility's cell, its sum dropped)
                const float2 *p = base + sm.cell[j + q];
                float re = 0.f, im = 0.f;
                if (RD_BOK(p >= sm.reg && p + (RB - 1) * 4 * RR + (CB - 1) * 8 < sm.reg + RR * RR, BC_P_SMEM)) {
#pragma unroll
                    for (int t = 0; t < NT; ++t) {
                        float2 g = p[(t / CB) * 4 * RR + (t % CB) * 8];
                        if (PAD && !(on >> t & 1u)) g = make_float2(0.f, 0.f);
                        re = fmaf(k[t].x, g.x, re);
                        re = fmaf(-k[t].y, g.y, re);
                        im = fmaf(k[t].x, g.y, im);
                        im = fmaf(k[t].y, g.x, im);
                    }
                }
                x[2 * q] = re;
                x[2 * q + 1] = im;
            }
            // reduce-scatter over lane bits 4, 3, 2 (value index bits 2, 1, 0), then bits 1, 0
#pragma unroll
            for (int h = 4; h >= 1; h >>= 1) {
                const bool up = lane & (4 * h);
#pragma unroll
                for (int i = 0; i < h; ++i) {
                    const float send = up ? x[i] : x[i + h];
                    const float keep = up ? x[i + h] : x[i];
                    x[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * h);
                }
            }
            x[0] += __shfl_xor_sync(0xffffffffu, x[0], 2);
            x[0] += __shfl_xor_sync(0xffffffffu, x[0], 1);
            const int v = j + (lane >> 3);   // value index lane >> 2: visibility, then re / im
            if ((lane & 3) == 0 && v < j1) {
                float *o = reinterpret_cast<float *>(&sm.out[v]) + ((lane >> 2) & 1);
                *o += x[0];
            }
        }
    }
}

template <int ST, bool SUB>
__global__ void __launch_bounds__(RD_THREADS, RD_CTAS) degrid_region_kernel(RegionDegridArgs a) {
    extern __shared__ __align__(16) char rd_smem[];
    DegridSmem &sm = *reinterpret_cast<DegridSmem *>(rd_smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if ((int64_t)blockIdx.x < a.nitems) {
        // last items first: the wide supports of the high w planes are the long tasks
        const int4 it = a.items[a.nitems - 1 - blockIdx.x];
        const int start = it.x, count = min(it.y, RD_MAXV), S = a.bin_support[it.z];
        const int T = aw_rg_tile(S), nb = aw_rg_nblk(S);
        const int tx0 = (it.w & 511) * T, ty0 = ((it.w >> 9) & 511) * T;
        const int64_t tab0 = a.bin_offset[it.z];
        // ---- the task's cells, offsets and runs
        for (int i = tid; i < RD_MAXV + 4; i += RD_THREADS) {
            int cell = 0;
            if (i < count) {
                aw_rec r{};
                if (RD_BOK((int64_t)start + i < a.nreg, BC_P_REC)) r = a.rec[(int64_t)start + i];
                const int ly = (int)r.y0 - ty0, lx = (int)r.x0 - tx0;
                const bool inr = RD_BOK(ly >= 0 && lx >= 0 && ly < T && lx < T, BC_P_CELL);
                cell = inr ? ly * RR + lx : 0;
                sm.off[i] = (uint16_t)((int)r.fy * a.OS + (int)r.fx);
                sm.out[i] = make_float2(0.f, 0.f);
            }
            sm.cell[i] = cell;
        }
        __syncthreads();
        int before = 0;
        for (int c0 = 0; c0 < count; c0 += RD_THREADS) {
            const int i = c0 + tid;
            const bool head = i < count && (i == 0 || sm.off[i] != sm.off[i - 1]);
            const unsigned m = __ballot_sync(0xffffffffu, head);
            if (lane == 0) sm.wsum[warp] = __popc(m);
            __syncthreads();
            int at = before;
            for (int w = 0; w < RD_THREADS / 32; ++w) {
                if (w < warp) at += sm.wsum[w];
                before += sm.wsum[w];
            }
            if (head) sm.run[at + __popc(m & ((1u << lane) - 1u))] = (uint16_t)i;
            __syncthreads();
        }
        if (tid == 0) {
            sm.run[before] = (uint16_t)count;
            sm.nrun = before;
        }
        // ---- footprint blocks
        for (int b = 0; b < nb * nb; ++b) {
            const int by = b / nb, bx = b - by * nb;
            const int bw = aw_rg_blk_width(S, bx), bh = aw_rg_blk_width(S, by);
            const int fx = aw_rg_blk_first(S, bx), fy = aw_rg_blk_first(S, by);
            const int rows = T + bh - 1, cols = T + bw - 1;
            __syncthreads();   // the runs are listed / the previous block's readers are done
            for (int y = warp; y < rows; y += RD_THREADS / 32) {
                const int gy = ty0 + fy + y;
                const float2 *src = a.grid + (int64_t)gy * a.N + tx0 + fx;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int x = lane + 32 * h;
                    if (x < cols)
                        sm.reg[y * RR + x] = gy < a.N && tx0 + fx + x < a.N ? __ldg(src + x) : make_float2(0.f, 0.f);
                }
            }
            __syncthreads();
#define RD_BLOCK(CB, RB)                                                       \
    (S % 8 ? run_block<ST, CB, RB, true>(sm, a, tab0, S, fy, fx)              \
           : run_block<ST, CB, RB, false>(sm, a, tab0, S, fy, fx))
            if (bw == 8) RD_BLOCK(1, 2);
            else if (bw == 16 && bh == 16) RD_BLOCK(2, 4);
            else if (bw == 24 && bh == 24) RD_BLOCK(3, 6);
            else if (bw == 24) RD_BLOCK(3, 4);
            else RD_BLOCK(2, 6);
#undef RD_BLOCK
        }
        __syncthreads();
        for (int i = tid; i < count; i += RD_THREADS) {
            if (!RD_BOK((int64_t)start + i < a.nreg, BC_P_REC)) continue;
            const aw_rec r = a.rec[(int64_t)start + i];
            if (!RD_BOK(r.orig < a.nvis, BC_P_REC)) continue;
            float2 o = make_float2(sm.out[i].x * a.inv_scale, sm.out[i].y * a.inv_scale);
            if (r.flip) o.y = -o.y;
            if constexpr (SUB) {
                const float2 w = a.sub_from[r.orig];
                o = make_float2(w.x - o.x, w.y - o.y);
            }
            a.vis_out[r.orig] = o;
        }
    }
    // visibilities that were not gridded (outside or flagged) predict zero
    for (int64_t i = a.nvalid + (int64_t)blockIdx.x * RD_THREADS + tid; i < a.nvis;
         i += (int64_t)gridDim.x * RD_THREADS) {
        const int64_t o = a.rec_all[i].orig;
        a.vis_out[o] = SUB ? a.sub_from[o] : make_float2(0.f, 0.f);
    }
}

template <int ST, bool SUB>
int launch_t(const RegionDegridArgs &a, cudaStream_t s) {
    auto kern = degrid_region_kernel<ST, SUB>;
    AW_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DegridSmem)));
    kern<<<(unsigned)a.nitems, RD_THREADS, sizeof(DegridSmem), s>>>(a);
    AW_CHECK_LAUNCH();
    return AW_OK;
}

template <int ST>
int launch_st(const RegionDegridArgs &a, cudaStream_t s) {
    return a.sub_from ? launch_t<ST, true>(a, s) : launch_t<ST, false>(a, s);
}

}  // namespace

int aw_launch_degrid_region(const aw_plan *p, const aw_kernel_set *k, const void *grid, void *vis_out,
                            cudaStream_t s, const void *sub_from) {
    RegionDegridArgs a;
    a.rec_all = p->d_rec;
    a.rec = p->d_rec_rg;
    a.items = p->d_items_rgd;
    a.nitems = p->nitems_rgd;
    a.ktab = k->d_table;
    a.bin_offset = k->d_bin_offset;
    a.bin_support = k->d_bin_support;
    a.grid = reinterpret_cast<const float2 *>(grid);
    a.vis_out = reinterpret_cast<float2 *>(vis_out);
    a.sub_from = reinterpret_cast<const float2 *>(sub_from);
    a.N = p->N;
    a.OS = p->OS;
    a.inv_scale = 1.0f / k->scale;
    a.nvis = p->nvis;
    a.nvalid = p->nvalid;
    a.nreg = p->nreg;
    a.tab_elems = k->total_elems;
    const int st = k->spec.storage;
    if (st == AW_STORAGE_FP32) return launch_st<AW_STORAGE_FP32>(a, s);
    if (st == AW_STORAGE_BF16) return launch_st<AW_STORAGE_BF16>(a, s);
    return launch_st<AW_STORAGE_FP16>(a, s);
}

int aw_degrid_region_bounds_status(unsigned int *v, int reset) {
#ifdef AW_BOUNDS_CHECK
    AW_CUDA_TRY(cudaMemcpyFromSymbol(v, g_bounds_status_rd, sizeof(*v)));
    if (reset) {
        const unsigned int z = 0;
        AW_CUDA_TRY(cudaMemcpyToSymbol(g_bounds_status_rd, &z, sizeof(z)));
    }
#else
    (void)reset;
    *v = 0;
#endif
    return AW_OK;
}
