// Gridding, REGION schedule: a CTA of two warps accumulates one plane of a grid
// region in shared memory.
//
// arXiv:2206.15117 Sec. 3.2: every visibility is convolved onto the uv grid
// with the oversampled kernel of its bin, G_s[y0 + jy][x0 + jx] +=
// sum_c K_{s,c}(jy, jx; fy, fx) w_c V_c (Sec. 2.1: w-projection planes; Sec. 3.2:
// the Mueller-cell kernels of the A term).
//
// A task is (visibilities of one bin whose footprints start in one T x T grid
// tile, at most AW_RG_MAXV; one block of the footprint; one grid plane s).  The
// visibilities come sorted by oversampled offset.  For each run of equal offset
// a thread holds its taps of the kernel block (row s of the Mueller matrix, NPOL
// complex values a tap) in registers, lane (r, c) of 4 x 8 having the taps
// (r + 4 i, c + 8 j) of the warp's half of the block, and adds K V of every
// visibility of the run to the region with a plain shared-memory
// read-modify-write per tap.  A barrier of the two warps after each visibility
// orders those of neighbouring footprints.  The addresses of a thread's taps
// differ by constants, so a visibility costs one address; the half-warps of a
// 64-bit access touch two rows of 8 cells, which with 56 cells a row fall on
// different banks.  At the end the region is added to the grid (one vector
// atomic per non-zero cell).  Any support works: blocks are 24 or 16 taps a
// side, and a smaller block leaves a larger tile, hence longer runs.
//
// What bounds it: the shared-memory pipe (128 B a clock), 16 bytes per
// visibility-tap and plane plus the kernel loads of every run; at full
// polarisation the FP32 pipe has the same limit of 0.5 clocks per
// visibility-tap.  Measured on 12M full-pol visibilities at 4096^2 (supports
// 16-72): 26.7 ms (the pipe 79 % busy) against 37.0 ms for the former form, four
// planes a CTA with the warps kept apart by footprint-row residues and OFFSETS
// beside it; 20.16M Stokes-I visibilities at 2048^2: 3.9 against 7.4 ms.  On a GPU
// where it takes 24.9 ms, one warp a region took 29.6 (two warps a scheduler do
// not hide their own latencies) and loading the next run's kernel values into a
// second register set 36-45 ms.
#include <algorithm>

#include "aw_internal.h"

// Checked builds (-DAW_BOUNDS_CHECK): a bad index records a code here (the
// first one wins) and the access is skipped; aw_debug_bounds_status reports it.
#ifdef AW_BOUNDS_CHECK
__device__ unsigned int g_bounds_status_rg;
#endif

namespace {

#ifdef AW_BOUNDS_CHECK
__device__ __forceinline__ bool rg_bounds_ok(bool ok, unsigned int code) {
    if (!ok) atomicCAS(&g_bounds_status_rg, 0u, code);
    return ok;
}
#define RG_BOK(cond, code) rg_bounds_ok((cond), (code))
#else
#define RG_BOK(cond, code) true
#endif

enum : unsigned int { BC_R_REC = 14, BC_R_CELL, BC_R_TAB, BC_R_GRID, BC_R_SMEM };

constexpr int RR = AW_RG_R;          // region side = row stride in cells
constexpr int RG_CTAS_SM = 8;        // 8 x (25 KB region + 3 KB staging) fill the shared memory

struct RegionArgs {
    const aw_rec *rec;          // region order
    const int4 *items;          // {start, count, bin, aw_rg_pack(tile, block)}
    int64_t nitems;
    unsigned int *counter;      // work-queue head (zeroed before the launch)
    const void *ktab;
    const int64_t *bin_offset;
    const int32_t *bin_support;
    const float2 *vis;
    const float *weight;
    float2 *grid;
    int N, OS;
    double *wsum;
    unsigned long long *nonfinite;
    float inv_scale;
    int64_t nvis, nvalid, tab_elems;
};

template <int ST>
__device__ __forceinline__ float2 widen(uint32_t w) {
    if constexpr (ST == AW_STORAGE_BF16) return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w));
    else return __half22float2(*reinterpret_cast<const __half2 *>(&w));
}

// Row s (NPOL values) of the Mueller kernel of tap t in the block of L taps
// that starts at complex element idx (chunk layout of aw_tab_index).
template <int ST, int NPOL>
__device__ __forceinline__ void load_row(const void *tab, int64_t idx, int L, int t, int s, float2 (&k)[NPOL]) {
    if constexpr (ST == AW_STORAGE_FP32) {
        const float2 *p = reinterpret_cast<const float2 *>(tab) + idx;
        if constexpr (NPOL == 4) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float4 v = __ldg(reinterpret_cast<const float4 *>(p) + (2 * s + h) * L + t);
                k[2 * h] = make_float2(v.x, v.y);
                k[2 * h + 1] = make_float2(v.z, v.w);
            }
        } else {
            k[0] = __ldg(p + t);
        }
    } else {
        const uint32_t *p = reinterpret_cast<const uint32_t *>(tab) + idx;
        if constexpr (NPOL == 4) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(p) + s * L + t);
            k[0] = widen<ST>(v.x);
            k[1] = widen<ST>(v.y);
            k[2] = widen<ST>(v.z);
            k[3] = widen<ST>(v.w);
        } else {
            k[0] = widen<ST>(__ldg(p + t));
        }
    }
}

__device__ __forceinline__ void cmac(float2 &a, float2 k, float2 v) {
    a.x = fmaf(k.x, v.x, a.x);
    a.x = fmaf(-k.y, v.y, a.x);
    a.y = fmaf(k.x, v.y, a.y);
    a.y = fmaf(k.y, v.x, a.y);
}

typedef unsigned long long u64;
__device__ __forceinline__ u64 pk(float x, float y) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 unpk(u64 a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
    u64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
constexpr int RG_THREADS = 64;
constexpr int RG_ROUND = RG_THREADS;   // visibilities staged at a time, one a thread

// Shared memory of a CTA: the region and one round of staged visibilities.
template <int NPOL>
struct __align__(16) RegionSmem {
    float2 reg[RR * RR];
    float2 v[RG_ROUND][NPOL];  // flipped, weighted, scaled
    int cell[RG_ROUND];        // footprint cell in the region
    int off[RG_ROUND];         // oversampled offset
    unsigned heads[2];         // bit j: visibility j starts a run of equal offset
    unsigned int next;
};

// One task's constants.
struct Task {
    int start, count, S, L, T, s, fx, fy, tx0, ty0;
    int64_t tab0;
    bool stats;
};

// g + K V for the thread's taps.  Full polarisation in packed pairs (fma.rn.f32x2
// runs at the FFMA rate with half the issue slots: 25.8 against 28.4 ms on that
// GPU): q1 = g + sum (kx, ky) vr, q2 = sum (kx, ky) vi, and g + K V =
// (q1.x - q2.y, q1.y + q2.x).
template <int NPOL, int CB, int RB, bool PAD>
__device__ __forceinline__ void add_vis(float2 *p, const float2 (&v)[NPOL], const float2 (&k)[CB * RB][NPOL],
                                        unsigned on) {
    constexpr int NT = CB * RB;
    float2 g[NT];
#pragma unroll
    for (int t = 0; t < NT; ++t) g[t] = p[(t / CB) * 4 * RR + (t % CB) * 8];
    if constexpr (NPOL == 4) {
        u64 vr[NPOL], vi[NPOL];
#pragma unroll
        for (int m = 0; m < NPOL; ++m) { vr[m] = pk(v[m].x, v[m].x); vi[m] = pk(v[m].y, v[m].y); }
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            u64 q1 = pk(g[t].x, g[t].y), q2 = 0;
#pragma unroll
            for (int m = 0; m < NPOL; ++m) {
                const u64 kk = pk(k[t][m].x, k[t][m].y);
                q1 = fma2(kk, vr[m], q1);
                q2 = m ? fma2(kk, vi[m], q2) : mul2(kk, vi[m]);
            }
            const float2 a1 = unpk(q1), a2 = unpk(q2);
            g[t] = make_float2(a1.x - a2.y, a1.y + a2.x);
            if (!PAD || (on >> t & 1u)) p[(t / CB) * 4 * RR + (t % CB) * 8] = g[t];
        }
    } else {
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            cmac(g[t], k[t][0], v[0]);
            if (!PAD || (on >> t & 1u)) p[(t / CB) * 4 * RR + (t % CB) * 8] = g[t];
        }
    }
}

// All visibilities of one task on a block of 8 CB columns and 8 RB rows, warp w
// taking the rows [4 RB w, 4 RB (w + 1)).  PAD: the block may reach past the
// footprint; absent taps have value 0 and write nothing.  Not inlined: each shape
// gets its own register allocation, within 128.
template <int ST, int NPOL, int CB, int RB, bool PAD>
__device__ __noinline__ void run_task(const RegionArgs a, const Task t, double *wsum_out,
                                      unsigned long long *nbad_out) {
    extern __shared__ __align__(16) char rg_smem[];
    RegionSmem<NPOL> &sm = *reinterpret_cast<RegionSmem<NPOL> *>(rg_smem);
    constexpr int NT = CB * RB;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int c0 = 0; c0 < t.count; c0 += RG_ROUND) {
        const int n = min(RG_ROUND, t.count - c0);
        __syncthreads();   // the region is zeroed / the previous round is done
        // ---- stage the round (flipped, weighted, NaN-checked)
        int key = -1;
        if (tid < n) {
            const int64_t ri = (int64_t)t.start + c0 + tid;
            aw_rec r{};
            if (RG_BOK(ri < a.nvalid, BC_R_REC)) r = a.rec[ri];
            const int64_t orig = RG_BOK(r.orig < a.nvis, BC_R_REC) ? (int64_t)r.orig : 0;
            float2 v[NPOL];
            float w[NPOL];
            bool bad = false;
#pragma unroll
            for (int m = 0; m < NPOL; ++m) {
                v[m] = a.vis[orig * NPOL + m];
                w[m] = a.weight ? a.weight[orig * NPOL + m] : 1.0f;
                bad |= !isfinite(v[m].x) || !isfinite(v[m].y) || !isfinite(w[m]);
            }
            if (r.flip) {
#pragma unroll
                for (int m = 0; m < NPOL; ++m) v[m].y = -v[m].y;
                if constexpr (NPOL == 4) {
                    const float2 x = v[1]; v[1] = v[2]; v[2] = x;
                    const float xw = w[1]; w[1] = w[2]; w[2] = xw;
                }
            }
            if (bad) {
#pragma unroll
                for (int m = 0; m < NPOL; ++m) { v[m] = make_float2(0.f, 0.f); w[m] = 0.f; }
            }
            if (t.stats) {
                double wm = 0.0;
#pragma unroll
                for (int m = 0; m < NPOL; ++m) wm += (double)w[m];
                *wsum_out += wm / NPOL;
                *nbad_out += bad;
            }
#pragma unroll
            for (int m = 0; m < NPOL; ++m) {
                const float ws = w[m] * a.inv_scale;
                sm.v[tid][m] = make_float2(ws * v[m].x, ws * v[m].y);
            }
            const int ly = (int)r.y0 - t.ty0, lx = (int)r.x0 - t.tx0;
            const bool inr = RG_BOK(ly >= 0 && lx >= 0 && ly < t.T && lx < t.T, BC_R_CELL);
            sm.cell[tid] = inr ? ly * RR + lx : 0;
            key = (int)r.fy * a.OS + (int)r.fx;
            sm.off[tid] = key;
        }
        __syncthreads();
        // ---- runs of equal offset
        const unsigned hd = __ballot_sync(0xffffffffu, tid < n && (tid == 0 || key != sm.off[tid - 1]));
        if (lane == 0) sm.heads[warp] = hd;
        __syncthreads();
        u64 heads = (u64)sm.heads[1] << 32 | sm.heads[0];
        while (heads) {
            const int j0 = __ffsll((long long)heads) - 1;
            heads &= heads - 1;
            const int j1 = heads ? __ffsll((long long)heads) - 1 : n;
            const int64_t kb = t.tab0 + (int64_t)sm.off[j0] * t.L * (NPOL * NPOL);
            const bool kok = RG_BOK(kb >= 0 && kb + (int64_t)t.L * NPOL * NPOL <= a.tab_elems, BC_R_TAB);
            const int r = warp * 4 * RB + (lane >> 3), c = lane & 7;   // block row, column of tap 0
            float2 k[NT][NPOL];
            unsigned on = 0;
#pragma unroll
            for (int i = 0; i < RB; ++i)
#pragma unroll
                for (int j = 0; j < CB; ++j) {
                    const int ty = t.fy + r + 4 * i, tx = t.fx + c + 8 * j;
                    if ((!PAD || (ty < t.S && tx < t.S)) && kok) {
                        on |= 1u << (i * CB + j);
                        load_row<ST, NPOL>(a.ktab, kb, t.L, ty * t.S + tx, t.s, k[i * CB + j]);
                    } else {
#pragma unroll
                        for (int m = 0; m < NPOL; ++m) k[i * CB + j][m] = make_float2(0.f, 0.f);
                    }
                }
            float2 *base = sm.reg + r * RR + c;
#pragma unroll 1
            for (int j = j0; j < j1; ++j) {
                float2 v[NPOL];
                if constexpr (NPOL == 4) {
                    const float4 v01 = *reinterpret_cast<const float4 *>(&sm.v[j][0]);
                    const float4 v23 = *reinterpret_cast<const float4 *>(&sm.v[j][2]);
                    v[0] = make_float2(v01.x, v01.y); v[1] = make_float2(v01.z, v01.w);
                    v[2] = make_float2(v23.x, v23.y); v[3] = make_float2(v23.z, v23.w);
                } else {
                    v[0] = sm.v[j][0];
                }
                float2 *p = base + sm.cell[j];
                if (RG_BOK(p >= sm.reg && p + (RB - 1) * 4 * RR + (CB - 1) * 8 < sm.reg + RR * RR, BC_R_SMEM))
                    add_vis<NPOL, CB, RB, PAD>(p, v, k, on);
                // the next visibility's cells may be this one's cells of other threads
                __syncthreads();
            }
        }
    }
    __syncthreads();
}

template <int ST, int NPOL>
__global__ void __launch_bounds__(RG_THREADS, RG_CTAS_SM) grid_region_kernel(RegionArgs a) {
    extern __shared__ __align__(16) char rg_smem[];
    RegionSmem<NPOL> &sm = *reinterpret_cast<RegionSmem<NPOL> *>(rg_smem);
    const int tid = threadIdx.x;
    double wloc = 0.0;
    unsigned long long nbad = 0;
    for (;;) {
        if (tid == 0) sm.next = atomicAdd(a.counter, 1u);
        __syncthreads();
        const unsigned int q = sm.next;
        if ((int64_t)q >= a.nitems * NPOL) break;
        // last items first: the wide supports of the high w planes are the long tasks
        const int4 it = a.items[a.nitems - 1 - q / NPOL];
        Task t;
        t.s = (int)(q % NPOL);
        t.start = it.x;
        t.count = it.y;
        t.S = a.bin_support[it.z];
        t.L = t.S * t.S;
        t.T = aw_rg_tile(t.S);
        t.tab0 = a.bin_offset[it.z];
        const int bx = (it.w >> 18) & 7, by = it.w >> 21;
        const int bw = aw_rg_blk_width(t.S, bx), bh = aw_rg_blk_width(t.S, by);
        t.fx = aw_rg_blk_first(t.S, bx);
        t.fy = aw_rg_blk_first(t.S, by);
        t.tx0 = (it.w & 511) * t.T;          // the tile's first cell
        t.ty0 = ((it.w >> 9) & 511) * t.T;
        t.stats = t.s == 0 && bx == 0 && by == 0;
        const int rows = t.T + bh - 1;
        float4 *z = reinterpret_cast<float4 *>(sm.reg);
        for (int i = tid; i < rows * RR / 2; i += RG_THREADS) z[i] = make_float4(0.f, 0.f, 0.f, 0.f);
#define RG_TASK(CB, RB)                                                  \
    (t.S % 8 ? run_task<ST, NPOL, CB, RB, true>(a, t, &wloc, &nbad)     \
             : run_task<ST, NPOL, CB, RB, false>(a, t, &wloc, &nbad))
        if (bw == 8) RG_TASK(1, 1);
        else if (bw == 16 && bh == 16) RG_TASK(2, 2);
        else if (bw == 24 && bh == 24) RG_TASK(3, 3);
        else if (bw == 24) RG_TASK(3, 2);
        else RG_TASK(2, 3);
#undef RG_TASK
        // ---- add the region to the grid (cells that received nothing are skipped)
        float2 *dst = a.grid + ((int64_t)t.s * a.N + t.ty0 + t.fy) * a.N + t.tx0 + t.fx;
        const int cols = t.T + bw - 1;
        for (int y = tid >> 5; y < rows; y += 2)
            for (int x = tid & 31; x < cols; x += 32) {
                const float2 v = sm.reg[y * RR + x];
                if ((v.x != 0.f || v.y != 0.f) &&
                    RG_BOK(t.ty0 + t.fy + y < a.N && t.tx0 + t.fx + x < a.N, BC_R_GRID))
                    atomicAdd(dst + (int64_t)y * a.N + x, v);
            }
        __syncthreads();
    }
    // statistics: one atomic per warp
    for (int o = 16; o; o >>= 1) {
        wloc += __shfl_xor_sync(0xffffffffu, wloc, o);
        nbad += __shfl_xor_sync(0xffffffffu, nbad, o);
    }
    if ((tid & 31) == 0) {
        if (wloc != 0.0) atomicAdd(a.wsum, wloc);
        if (nbad) atomicAdd(a.nonfinite, nbad);
    }
}

template <int ST, int NPOL>
int launch_region_t(const RegionArgs &a, int sm_count, cudaStream_t s) {
    auto kern = grid_region_kernel<ST, NPOL>;
    const size_t smem = sizeof(RegionSmem<NPOL>);
    AW_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int64_t blocks = std::min<int64_t>(a.nitems * NPOL, (int64_t)sm_count * RG_CTAS_SM);
    kern<<<(unsigned)blocks, RG_THREADS, smem, s>>>(a);
    AW_CHECK_LAUNCH();
    return AW_OK;
}

}  // namespace

int aw_launch_grid_region(const aw_plan *p, const aw_kernel_set *k, const void *vis, const float *weight, void *grid,
                          cudaStream_t s) {
    if (p->nitems_rg == 0) return AW_OK;
    RegionArgs a;
    a.rec = p->d_rec_rg;
    a.items = p->d_items_rg;
    a.nitems = p->nitems_rg;
    a.counter = p->d_rcounter;
    a.ktab = k->d_table;
    a.bin_offset = k->d_bin_offset;
    a.bin_support = k->d_bin_support;
    a.vis = reinterpret_cast<const float2 *>(vis);
    a.weight = weight;
    a.grid = reinterpret_cast<float2 *>(grid);
    a.N = p->N;
    a.OS = p->OS;
    a.wsum = p->d_wsum;
    a.nonfinite = p->d_nonfinite;
    a.inv_scale = 1.0f / k->scale;
    a.nvis = p->nvis;
    a.nvalid = p->nreg;
    a.tab_elems = k->total_elems;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    AW_CUDA_TRY(cudaMemsetAsync(p->d_rcounter, 0, sizeof(unsigned int), s));
    const int st = k->spec.storage;
    if (p->npol == 4) {
        if (st == AW_STORAGE_FP32) return launch_region_t<AW_STORAGE_FP32, 4>(a, sms, s);
        if (st == AW_STORAGE_BF16) return launch_region_t<AW_STORAGE_BF16, 4>(a, sms, s);
        return launch_region_t<AW_STORAGE_FP16, 4>(a, sms, s);
    }
    if (st == AW_STORAGE_FP32) return launch_region_t<AW_STORAGE_FP32, 1>(a, sms, s);
    if (st == AW_STORAGE_BF16) return launch_region_t<AW_STORAGE_BF16, 1>(a, sms, s);
    return launch_region_t<AW_STORAGE_FP16, 1>(a, sms, s);
}

int aw_region_bounds_status(unsigned int *v, int reset) {
#ifdef AW_BOUNDS_CHECK
    AW_CUDA_TRY(cudaMemcpyFromSymbol(v, g_bounds_status_rg, sizeof(*v)));
    if (reset) {
        const unsigned int z = 0;
        AW_CUDA_TRY(cudaMemcpyToSymbol(g_bounds_status_rg, &z, sizeof(z)));
    }
#else
    (void)reset;
    *v = 0;
#endif
    return AW_OK;
}
