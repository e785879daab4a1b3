// Plan creation: per-visibility FP64 coordinates (uvw in wavelengths, Eq. 2)
// and the device key sort that orders visibilities by (bin, grid tile,
// position in tile) and cuts them into work items.
#include <algorithm>
#include <cmath>
#include <vector>

#include "aw_internal.h"

namespace {

struct CoordArgs {
    int64_t nvis;
    const double *uvw;
    const uint32_t *row;
    const uint16_t *chan;
    const double *freq;
    const double *fl;          // channels [0, nchan): frequency / c, one correctly rounded division
    const uint8_t *pa_bin;
    const uint8_t *fbin;
    const uint8_t *flags;
    const uint8_t *row_types;  // [nrow][2] or NULL
    int N, OS, nw, npa, nfb, ntype;
    double uscale, half, winv;
    const int32_t *support;  // per w plane
    int tile, tbits, ntx, nty;
    int64_t nrow;
    int32_t nchan;
};

struct CoordOut {
    int x0, y0, fx, fy, bin, flip, valid, S;
};

// floor(a / d), in 32 bits where a fits (nearly every visibility)
__device__ __forceinline__ long long floor_div(long long a, int d) {
    if (a >= 0 && a <= 0x7fffffffll) return (long long)((uint32_t)a / (uint32_t)d);
    long long q = a / d;
    if (a < 0 && q * d != a) q -= 1;
    return q;
}

__global__ void channel_kernel(const double *freq, int nchan, double *fl) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < nchan) fl[c] = __ddiv_rn(freq[c], AW_C_LIGHT);
}

// The FP64 coordinate step with a fixed operation order (no contraction).
// FP64 runs at 2 lanes a clock and SM here, so the step holds ten FP64 operations
// and three conversions; the division by c is done once a channel (a channel that
// the descriptor's nchan does not count takes the same division here), signs are
// tested and changed on the bits.
__device__ __forceinline__ CoordOut coord_of(const CoordArgs &a, int64_t k) {
    CoordOut o;
    const uint32_t r = a.row[k];
    const uint16_t c = a.chan[k];
    const double f = (int)c < a.nchan ? __ldg(a.fl + c) : __ddiv_rn(a.freq[c], AW_C_LIGHT);
    double u = __dmul_rn(a.uvw[3 * (int64_t)r + 0], f);
    double v = __dmul_rn(a.uvw[3 * (int64_t)r + 1], f);
    double w = __dmul_rn(a.uvw[3 * (int64_t)r + 2], f);
    // w < 0, and the sign change, on the bits (comparisons run in the FP64 pipe too)
    const unsigned long long wb = (unsigned long long)__double_as_longlong(w);
    o.flip = wb - 0x8000000000000001ull <= 0x7ff0000000000000ull - 1ull ? 1 : 0;   // -inf .. the smallest negative
    const unsigned long long sign = (unsigned long long)o.flip << 63;
    u = __longlong_as_double((long long)((unsigned long long)__double_as_longlong(u) ^ sign));
    v = __longlong_as_double((long long)((unsigned long long)__double_as_longlong(v) ^ sign));
    w = __longlong_as_double((long long)(wb ^ sign));
    const double xr = __dadd_rn(__dadd_rn(__dmul_rn(u, a.uscale), a.half), 0.5);
    const double yr = __dadd_rn(__dadd_rn(__dmul_rn(v, a.uscale), a.half), 0.5);
    // rounded down and clamped far out, where they are invalid anyway (the conversion
    // saturates and takes a NaN to the lowest value)
    const long long lim = 4000000000000000ll;
    const long long Xi = min(max(__double2ll_rd(xr), -lim), lim);
    const long long Yi = min(max(__double2ll_rd(yr), -lim), lim);
    int wp = 0;
    if (a.winv > 0.0) {
        // (a NaN counts as far out, as the minimum with a large plane number takes it)
        const double wt = __dmul_rn(w, a.winv);
        const bool nan = ((unsigned long long)__double_as_longlong(wt) & 0x7fffffffffffffffull) > 0x7ff0000000000000ull;
        wp = nan ? a.nw - 1 : min(max(__double2int_rd(wt), 0), a.nw - 1);
    }
    const int pa = a.pa_bin ? (int)a.pa_bin[r] : 0;
    const int fb = a.fbin ? (int)a.fbin[c] : 0;
    int cls = 0;
    if (a.ntype >= 2 && a.row_types) {
        // the flipped sample is the reversed baseline: its class swaps the types
        int ti = min((int)a.row_types[2 * (int64_t)r], a.ntype - 1);
        int tj = min((int)a.row_types[2 * (int64_t)r + 1], a.ntype - 1);
        if (o.flip) { const int t = ti; ti = tj; tj = t; }
        cls = ti * a.ntype + tj;
    }
    o.bin = ((cls * a.nw + wp) * a.npa + min(pa, a.npa - 1)) * a.nfb + min(fb, a.nfb - 1);
    const int S = a.support[wp];
    o.S = S;
    const long long rho = (long long)(S - 2) * a.OS / 2;
    const long long Ax = Xi - rho, Ay = Yi - rho;
    const long long ix = floor_div(Ax, a.OS), iy = floor_div(Ay, a.OS);
    o.fx = (int)(Ax - ix * a.OS);
    o.fy = (int)(Ay - iy * a.OS);
    int valid = 1;
    if (ix < 0 || ix + S > a.N) valid = 0;
    if (iy < 0 || iy + S > a.N) valid = 0;
    o.x0 = valid ? (int)ix : 0;
    o.y0 = valid ? (int)iy : 0;
    o.valid = valid;
    return o;
}

template <typename K>
__global__ void coords_kernel(CoordArgs a, K invalid_key, K *keys, aw_rec *recs, unsigned long long *counts /* outside, flagged, valid, taps */) {
    unsigned long long n_out = 0, n_flag = 0, n_val = 0, taps = 0;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < a.nvis;
         k += (int64_t)gridDim.x * blockDim.x) {
        const CoordOut o = coord_of(a, k);
        const bool flagged = a.flags && a.flags[k];
        const bool ok = o.valid && !flagged;
        if (!o.valid) n_out++;
        else if (flagged) n_flag++;
        K key = invalid_key;
        if (ok) {
            n_val++;
            taps += (unsigned long long)o.S * o.S;
            const int tx = o.x0 >> a.tbits, ty = o.y0 >> a.tbits;
            const int lx = o.x0 & (a.tile - 1), ly = o.y0 & (a.tile - 1);
            key = ((((K)o.bin * a.nty + ty) * a.ntx + tx) << (2 * a.tbits)) | ((K)ly << a.tbits) | (K)lx;
        }
        keys[k] = key;
        aw_rec rc;
        rc.orig = (uint32_t)k;
        rc.x0 = (uint16_t)o.x0;
        rc.y0 = (uint16_t)o.y0;
        rc.bin = (uint16_t)o.bin;
        rc.fx = (uint8_t)o.fx;
        rc.fy = (uint8_t)o.fy;
        rc.flip = (uint8_t)o.flip;
        rc.pad0 = ok ? 1 : 0;   // gridded
        rc.pad1 = 0;
        recs[k] = rc;
    }
    // warp-aggregated counters
    for (int off = 16; off; off >>= 1) {
        n_out += __shfl_xor_sync(0xffffffffu, n_out, off);
        n_flag += __shfl_xor_sync(0xffffffffu, n_flag, off);
        n_val += __shfl_xor_sync(0xffffffffu, n_val, off);
        taps += __shfl_xor_sync(0xffffffffu, taps, off);
    }
    if ((threadIdx.x & 31) == 0) {
        if (n_out) atomicAdd(&counts[0], n_out);
        if (n_flag) atomicAdd(&counts[1], n_flag);
        if (n_val) atomicAdd(&counts[2], n_val);
        if (taps) atomicAdd(&counts[3], taps);
    }
}

__global__ void coords_out_kernel(CoordArgs a, int32_t *x0, int32_t *y0, int32_t *fx, int32_t *fy,
                                  int32_t *bin, uint8_t *flip, uint8_t *valid) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < a.nvis;
         k += (int64_t)gridDim.x * blockDim.x) {
        const CoordOut o = coord_of(a, k);
        const bool ok = o.valid && !(a.flags && a.flags[k]);
        if (x0) x0[k] = o.x0;
        if (y0) y0[k] = o.y0;
        if (fx) fx[k] = o.fx;
        if (fy) fy[k] = o.fy;
        if (bin) bin[k] = o.bin;
        if (flip) flip[k] = (uint8_t)o.flip;
        if (valid) valid[k] = ok ? 1 : 0;
    }
}

// ------------------------------------------------------------ LSD radix sort
// One pass = per-tile digit histogram -> exclusive scan over [digit][tile] ->
// stable scatter, with digits of up to 9 bits and keys of 32 or 64 bits.  A tile
// is RS_TILE keys; each warp owns a contiguous run of RS_ITEMS * 32 of them and
// ranks equal digits with __match_any_sync against its own running counters, so
// the order of equal keys is preserved.  The tile is put in digit order in shared
// memory first, so that a digit's run leaves as consecutive words: written
// straight from the registers, every store touched 32 sectors, and a pass over
// 12M 64-bit keys took 146 us (116 now; 64 with 32-bit keys).
constexpr int RS_THREADS = 512;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_ITEMS = 16;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;
constexpr int RS_BITS = 9;
constexpr int RS_DIGITS = 1 << RS_BITS;
static_assert(RS_DIGITS == RS_THREADS, "one digit a thread");

template <typename K>
__global__ void __launch_bounds__(RS_THREADS) radix_hist_kernel(const K *keys, int64_t n, int shift, int nd,
                                                                uint32_t *counts, int ntiles) {
    __shared__ uint32_t h[RS_DIGITS];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * RS_TILE;
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i) {
        const int64_t k = base + (int64_t)i * RS_THREADS + threadIdx.x;
        if (k < n) atomicAdd(&h[(int)(keys[k] >> shift) & (nd - 1)], 1u);
    }
    __syncthreads();
    if ((int)threadIdx.x < nd) counts[(int64_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

template <typename K>
struct RadixSmem {
    union {
        K key[RS_TILE];
        uint32_t val[RS_TILE];            // (after the keys have left)
    };
    uint32_t out[RS_DIGITS];              // output position of the digit's first key, less its place in the tile
    uint16_t cnt[RS_WARPS][RS_DIGITS];    // running counts, then the digit's place before each warp
    uint32_t wsum[RS_WARPS];
};

template <typename K>
__global__ void __launch_bounds__(RS_THREADS, 2) radix_scatter_kernel(const K *keys, const uint32_t *vals, int64_t n,
                                                                   int shift, int nd, const uint32_t *offsets,
                                                                   int ntiles, K *keys_out, uint32_t *vals_out) {
    extern __shared__ __align__(16) char rs_smem[];
    RadixSmem<K> &sm = *reinterpret_cast<RadixSmem<K> *>(rs_smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int w = 0; w < RS_WARPS; ++w) sm.cnt[w][tid] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * RS_TILE;
    const int ntile = (int)min((int64_t)RS_TILE, n - base);
    const int w0 = warp * RS_ITEMS * 32 + lane;        // the thread's first key of the tile
    keys += base;
    K kk[RS_ITEMS];
    uint16_t rank[RS_ITEMS];
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r) kk[r] = (w0 + r * 32 < ntile) ? keys[w0 + r * 32] : 0;
    const unsigned lt = (1u << lane) - 1u;
    // 1) rank among the warp's keys of the same digit
    if (ntile == RS_TILE) {
#pragma unroll
        for (int r = 0; r < RS_ITEMS; ++r) {
            const int d = (int)(kk[r] >> shift) & (nd - 1);
            const unsigned peers = __match_any_sync(0xffffffffu, d);
            const uint32_t before = sm.cnt[warp][d], mine = __popc(peers & lt);
            rank[r] = (uint16_t)(before + mine);
            __syncwarp();
            if (mine == 0) sm.cnt[warp][d] = (uint16_t)(before + __popc(peers));
            __syncwarp();
        }
    } else {
        for (int r = 0; r < RS_ITEMS; ++r) {
            const bool in = w0 + r * 32 < ntile;
            const int d = in ? (int)(keys[w0 + r * 32] >> shift) & (nd - 1) : nd;   // (absent keys match one another)
            const unsigned peers = __match_any_sync(0xffffffffu, d);
            const uint32_t before = in ? sm.cnt[warp][d] : 0, mine = __popc(peers & lt);
#pragma unroll
            for (int q = 0; q < RS_ITEMS; ++q)
                if (q == r) rank[q] = (uint16_t)(before + mine);
            __syncwarp();
            if (in && mine == 0) sm.cnt[warp][d] = (uint16_t)(before + __popc(peers));
            __syncwarp();
        }
    }
    __syncthreads();
    // 2) a digit's place before each warp, its total, and the digits' places in the tile
    uint32_t total = 0;
#pragma unroll
    for (int w = 0; w < RS_WARPS; ++w) {
        const uint32_t c = sm.cnt[w][tid];
        sm.cnt[w][tid] = (uint16_t)total;
        total += c;
    }
    uint32_t incl = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) sm.wsum[warp] = incl;
    __syncthreads();
    uint32_t place = incl - total;
    for (int w = 0; w < warp; ++w) place += sm.wsum[w];
    if (tid < nd) sm.out[tid] = offsets[(int64_t)tid * ntiles + blockIdx.x] - place;
#pragma unroll
    for (int w = 0; w < RS_WARPS; ++w) sm.cnt[w][tid] += (uint16_t)place;
    __syncthreads();
    // 3) the keys in digit order, and out; then the values the same way (loaded while
    // the keys leave)
    uint16_t (&at)[RS_ITEMS] = rank;
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r)
        if (w0 + r * 32 < ntile) {
            const int d = (int)(kk[r] >> shift) & (nd - 1);
            at[r] = (uint16_t)(sm.cnt[warp][d] + rank[r]);
            sm.key[at[r]] = kk[r];
        }
    uint32_t vv[RS_ITEMS];
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r)
        vv[r] = w0 + r * 32 < ntile && vals ? __ldg(vals + base + w0 + r * 32) : (uint32_t)(base + w0 + r * 32);
    __syncthreads();
    uint32_t pos[RS_ITEMS];
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r) {
        const int i = r * RS_THREADS + tid;
        if (i < ntile) {
            const K key = sm.key[i];
            pos[r] = sm.out[(int)(key >> shift) & (nd - 1)] + (uint32_t)i;
            keys_out[pos[r]] = key;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r) {
        if (w0 + r * 32 < ntile) sm.val[at[r]] = vv[r];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r) {
        const int i = r * RS_THREADS + tid;
        if (i < ntile) vals_out[pos[r]] = sm.val[i];
    }
}

// ------------------------------------------------------------ items
// Starts of the segments of equal key >> shift, in two passes over the keys:
// heads per block of SEG_BLOCK keys, and, after a scan of those counts, the heads
// themselves.
constexpr int SEG_THREADS = 256;
constexpr int SEG_ITEMS = 8;
constexpr int SEG_BLOCK = SEG_THREADS * SEG_ITEMS;

template <typename K>
__device__ __forceinline__ bool seg_head(const K *keys, int64_t i, int64_t n, int shift) {
    return i < n && (i == 0 || (keys[i] >> shift) != (keys[i - 1] >> shift));
}

template <typename K>
__global__ void __launch_bounds__(SEG_THREADS) seg_count_kernel(const K *keys, int64_t n, int shift, uint32_t *nhead) {
    __shared__ uint32_t total;
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * SEG_BLOCK;
    uint32_t c = 0;
#pragma unroll
    for (int r = 0; r < SEG_ITEMS; ++r)
        c += __popc(__ballot_sync(0xffffffffu, seg_head(keys, base + r * SEG_THREADS + threadIdx.x, n, shift)));
    if ((threadIdx.x & 31) == 0) atomicAdd(&total, c);
    __syncthreads();
    if (threadIdx.x == 0) nhead[blockIdx.x] = total;
}

template <typename K>
__global__ void __launch_bounds__(SEG_THREADS) seg_start_kernel(const K *keys, int64_t n, int shift,
                                                                const uint32_t *first, uint32_t *starts) {
    __shared__ uint32_t wsum[SEG_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t at = first[blockIdx.x];
    for (int r = 0; r < SEG_ITEMS; ++r) {
        const int64_t i = (int64_t)blockIdx.x * SEG_BLOCK + r * SEG_THREADS + threadIdx.x;
        const bool head = seg_head(keys, i, n, shift);
        const unsigned m = __ballot_sync(0xffffffffu, head);
        if (lane == 0) wsum[warp] = __popc(m);
        __syncthreads();
        uint32_t before = 0, all = 0;
        for (int w = 0; w < SEG_THREADS / 32; ++w) {
            if (w < warp) before += wsum[w];
            all += wsum[w];
        }
        if (head) starts[at + before + __popc(m & ((1u << lane) - 1u))] = (uint32_t)i;
        at += all;
        __syncthreads();
    }
}

__global__ void seg_chunks_kernel(const uint32_t *starts, int64_t nseg, uint32_t nvalid, int chunk,
                                  uint32_t *nch) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < nseg;
         s += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t a = starts[s];
        const uint32_t b = (s + 1 < nseg) ? starts[s + 1] : nvalid;
        nch[s] = (b - a + chunk - 1) / chunk;
    }
}

__global__ void emit_items_kernel(const uint32_t *starts, const uint32_t *itembase, int64_t nseg,
                                  uint32_t nvalid, int chunk, const aw_rec *rec, int4 *items) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < nseg;
         s += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t a = starts[s];
        const uint32_t b = (s + 1 < nseg) ? starts[s + 1] : nvalid;
        const int bin = rec[a].bin;
        uint32_t pos = itembase[s];
        for (uint32_t st = a; st < b; st += chunk) {
            const uint32_t cnt = min((uint32_t)chunk, b - st);
            items[pos++] = make_int4((int)st, (int)cnt, bin, 0);
        }
    }
}

// REGION tasks of the segments (one bin and one region tile each): ceil(count /
// cap) pieces times blk^2 footprint blocks, geo[bin] = {tile side, cap, blk, -}.
// *total: their number, in 64 bits (the positions in the list have 32).
__global__ void rg_count_kernel(const uint32_t *starts, int64_t nseg, uint32_t nreg, const aw_rec *rec,
                                const int4 *geo, uint32_t *ntask, unsigned long long *total) {
    unsigned long long sum = 0;
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < nseg;
         s += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t a = starts[s], b = (s + 1 < nseg) ? starts[s + 1] : nreg;
        const int4 g = geo[rec[a].bin];
        const uint32_t n = (b - a + g.y - 1) / g.y * g.z * g.z;
        ntask[s] = n;
        sum += n;
    }
    for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if ((threadIdx.x & 31) == 0 && sum) atomicAdd(total, sum);
}

__global__ void rg_emit_kernel(const uint32_t *starts, const uint32_t *base, int64_t nseg, uint32_t nreg,
                               const aw_rec *rec, const int4 *geo, int4 *tasks) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < nseg;
         s += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t a = starts[s], b = (s + 1 < nseg) ? starts[s + 1] : nreg;
        const aw_rec r = rec[a];
        const int4 g = geo[r.bin];
        const int tx = r.x0 / g.x, ty = r.y0 / g.x;
        uint32_t pos = base[s];
        for (uint32_t st = a; st < b; st += g.y)
            for (int k = 0; k < g.z * g.z; ++k)
                tasks[pos++] = make_int4((int)st, (int)min((uint32_t)g.y, b - st), (int)r.bin,
                                         aw_rg_pack(tx, ty, k % g.z, k / g.z));
    }
}

// REGION key of the i-th visibility in degridding order: (bin, region tile row,
// region tile column); the order by oversampled offset inside a bin and
// super-tile is there already, and the sort is stable.  geo[bin].x = tile side
// (0: the bin takes no region); those bins get invalid_key (sorted last);
// eligible ones are counted in *nreg.
template <typename K>
__global__ void rg_key_kernel(const aw_rec *rec, int64_t nv, const int4 *geo, int nt, K invalid_key, K *keys,
                              unsigned long long *nreg) {
    unsigned long long cnt = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nv;
         i += (int64_t)gridDim.x * blockDim.x) {
        const aw_rec r = rec[i];
        const int T = geo[r.bin].x;
        K key = invalid_key;
        if (T > 0) {
            key = ((K)r.bin * nt + (int)r.y0 / T) * nt + (int)r.x0 / T;
            cnt++;
        }
        keys[i] = key;
    }
    for (int o = 16; o; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(nreg, cnt);
}

__global__ void gather_rec_kernel(const aw_rec *in, const uint32_t *perm, int64_t n, aw_rec *out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = in[perm[i]];
}

__global__ void rec_orig_kernel(const aw_rec *rec, int64_t n, uint32_t *perm) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        perm[i] = rec[i].orig;
}

// Degridding key of the i-th valid visibility (grid order): (bin, super-tile
// row, super-tile column, fy, fx); inside a group the grid order (tile, then
// position) stays.
template <typename K>
__global__ void dg_key_kernel(const aw_rec *rec, int64_t nv, int OS, int stbits, int nst, K *keys) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nv;
         i += (int64_t)gridDim.x * blockDim.x) {
        const aw_rec r = rec[i];
        keys[i] = (((K)r.bin * nst + (r.y0 >> stbits)) * nst + (r.x0 >> stbits)) * (OS * OS) + (int)r.fy * OS + r.fx;
    }
}

int grid_blocks(int64_t n, int threads) {
    int64_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > 152 * 64) b = 152 * 64;
    return (int)b;
}

struct DevBuf {
    void *p = nullptr;
    ~DevBuf() { if (p) aw_dev_free(p); }
};

int ilog2(int v) {
    int r = 0;
    while ((1 << r) < v) ++r;
    return r;
}

int fill_coord_args(const aw_vis_desc *vis, const aw_kernel_set *ks, int tile, CoordArgs &a,
                    aw_plan *plan) {
    const aw_kernel_spec &sp = ks->spec;
    a.nvis = vis->nvis;
    a.uvw = vis->uvw;
    a.row = vis->row_of_vis;
    a.chan = vis->chan_of_vis;
    a.freq = vis->freq;
    a.fl = plan->d_fl;
    a.pa_bin = vis->pa_bin;
    a.fbin = vis->fbin;
    a.flags = vis->flags;
    a.row_types = vis->row_types;
    a.N = sp.N;
    a.OS = sp.OS;
    a.nw = sp.nw;
    a.npa = sp.npa;
    a.nfb = sp.nfb;
    a.ntype = ks->ntype;
    a.uscale = (double)sp.N * sp.dl * (double)sp.OS;
    a.half = (double)(sp.N / 2) * (double)sp.OS;
    a.winv = (sp.nw > 1 && sp.w_max > 0.0) ? (double)sp.nw / sp.w_max : 0.0;
    a.support = plan->d_plane_support;  // first nw entries hold the per-plane supports
    a.tile = tile;
    a.tbits = ilog2(tile);
    a.ntx = (sp.N + tile - 1) / tile;
    a.nty = a.ntx;
    a.nrow = vis->nrow;
    a.nchan = vis->nchan;
    return AW_OK;
}

// The temporaries: one device allocation handed out in pieces.
struct Arena {
    DevBuf buf;
    size_t size = 0, used = 0;
    static size_t round(size_t b) { return (b + 255) / 256 * 256; }
    template <class T>
    T *take(size_t count) {
        T *p = reinterpret_cast<T *>(static_cast<char *>(buf.p) + used);
        used += round(count * sizeof(T));
        return p;
    }
};

// Sort buffers: two (key, value) arrays for n visibilities (64-bit keys), the
// tile counts and their scan, and per-segment words.
struct SortBufs {
    uint64_t *k0, *k1;
    uint32_t *v0, *v1;
    uint32_t *words[3];   // max(tile counts, n + 1) words each
    void *scratch;
};

int key_bits(uint64_t maxkey) {   // bits that hold 0 .. maxkey
    int b = 1;
    while (b < 64 && (maxkey >> b)) ++b;
    return b;
}

// LSD radix sort of n keys of `bits` bits, the values being 0 .. n-1 at the
// start; on return kin / vout point at the sorted arrays.
template <typename K>
int radix_sort(K *&kin, uint32_t *&vout, int64_t n, int bits, SortBufs &b, cudaStream_t s) {
    const int ntiles = (int)((n + RS_TILE - 1) / RS_TILE);
    const int passes = (bits + RS_BITS - 1) / RS_BITS, db = (bits + passes - 1) / passes, nd = 1 << db;
    AW_CUDA_TRY(cudaFuncSetAttribute(radix_scatter_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(RadixSmem<K>)));
    K *k0 = kin, *k1 = reinterpret_cast<K *>(kin == reinterpret_cast<K *>(b.k0) ? b.k1 : b.k0);
    const uint32_t *v0 = nullptr;
    uint32_t *v1 = b.v0;
    for (int pass = 0; pass < passes; ++pass) {
        const int shift = pass * db;
        radix_hist_kernel<K><<<ntiles, RS_THREADS, 0, s>>>(k0, n, shift, nd, b.words[0], ntiles);
        AW_CHECK_LAUNCH();
        int rc = aw_exclusive_scan_u32(b.words[0], b.words[1], (int64_t)nd * ntiles, b.scratch, s);
        if (rc) return rc;
        radix_scatter_kernel<K><<<ntiles, RS_THREADS, sizeof(RadixSmem<K>), s>>>(k0, v0, n, shift, nd, b.words[1], ntiles,
                                                                                k1, v1);
        AW_CHECK_LAUNCH();
        std::swap(k0, k1);
        v0 = v1;
        v1 = v1 == b.v0 ? b.v1 : b.v0;
    }
    kin = k0;
    vout = const_cast<uint32_t *>(v0);
    return AW_OK;
}

// Exclusive scan of the n per-segment counts `cnt` into `base`, and their total (host).
int scan_counts(const uint32_t *cnt, uint32_t *base, int64_t n, void *scratch, int64_t *total, cudaStream_t s) {
    int rc = aw_exclusive_scan_u32(cnt, base, n, scratch, s);
    if (rc) return rc;
    uint32_t lb = 0, ln = 0;
    AW_CUDA_TRY(cudaMemcpyAsync(&lb, base + n - 1, 4, cudaMemcpyDeviceToHost, s));
    AW_CUDA_TRY(cudaMemcpyAsync(&ln, cnt + n - 1, 4, cudaMemcpyDeviceToHost, s));
    AW_CUDA_TRY(cudaStreamSynchronize(s));
    *total = (int64_t)lb + ln;
    return AW_OK;
}

// Starts (b.words[2]) of the *nseg segments of equal key >> shift in nv sorted keys.
template <typename K>
int build_segments(const K *keys, int64_t nv, int shift, SortBufs &b, int64_t *nseg, cudaStream_t s) {
    const int64_t nblk = (nv + SEG_BLOCK - 1) / SEG_BLOCK;
    seg_count_kernel<K><<<(unsigned)nblk, SEG_THREADS, 0, s>>>(keys, nv, shift, b.words[0]);
    AW_CHECK_LAUNCH();
    const int rc = scan_counts(b.words[0], b.words[1], nblk, b.scratch, nseg, s);
    if (rc) return rc;
    seg_start_kernel<K><<<(unsigned)nblk, SEG_THREADS, 0, s>>>(keys, nv, shift, b.words[1], b.words[2]);
    AW_CHECK_LAUNCH();
    return AW_OK;
}

// Cut the sorted keys of the nv valid visibilities into segments of equal
// key >> shift and the segments into items of at most `chunk` visibilities;
// allocates *items.
template <typename K>
int build_items(const K *keys, int64_t nv, int shift, int chunk, const aw_rec *rec, SortBufs &b, int4 **items,
                int64_t *nitems, cudaStream_t s) {
    int64_t nseg = 0;
    int rc = build_segments<K>(keys, nv, shift, b, &nseg, s);
    if (rc) return rc;
    seg_chunks_kernel<<<grid_blocks(nseg, 256), 256, 0, s>>>(b.words[2], nseg, (uint32_t)nv, chunk, b.words[0]);
    AW_CHECK_LAUNCH();
    rc = scan_counts(b.words[0], b.words[1], nseg, b.scratch, nitems, s);
    if (rc) return rc;
    AW_CUDA_TRY(aw_dev_malloc(items, sizeof(int4) * std::max<int64_t>(*nitems, 1)));
    emit_items_kernel<<<grid_blocks(nseg, 256), 256, 0, s>>>(b.words[2], b.words[1], nseg, (uint32_t)nv, chunk, rec,
                                                            *items);
    AW_CHECK_LAUNCH();
    return AW_OK;
}

// The region tasks of the nseg segments (b.words[2]) of the nreg records `rec`
// under the per-bin geometry geo; allocates *tasks.  *ntasks = 0 and no list if
// they are more than aw_rg_fits allows or hold fewer than min_mean visibilities on
// average.
int build_region_tasks(int64_t nseg, int64_t nreg, int npol, int64_t min_mean, const aw_rec *rec, const int4 *geo,
                       unsigned long long *d_total, SortBufs &b, int4 **tasks, int64_t *ntasks, cudaStream_t s) {
    unsigned long long total = 0;
    *ntasks = 0;
    AW_CUDA_TRY(cudaMemsetAsync(d_total, 0, sizeof(total), s));
    rg_count_kernel<<<grid_blocks(nseg, 256), 256, 0, s>>>(b.words[2], nseg, (uint32_t)nreg, rec, geo, b.words[0], d_total);
    AW_CHECK_LAUNCH();
    const int rc = aw_exclusive_scan_u32(b.words[0], b.words[1], nseg, b.scratch, s);
    if (rc) return rc;
    AW_CUDA_TRY(cudaMemcpyAsync(&total, d_total, sizeof(total), cudaMemcpyDeviceToHost, s));
    AW_CUDA_TRY(cudaStreamSynchronize(s));
    if (!aw_rg_fits(total, npol) || nreg < min_mean * (int64_t)total) return AW_OK;
    AW_CUDA_TRY(aw_dev_malloc(tasks, sizeof(int4) * std::max<int64_t>((int64_t)total, 1)));
    rg_emit_kernel<<<grid_blocks(nseg, 256), 256, 0, s>>>(b.words[2], b.words[1], nseg, (uint32_t)nreg, rec, geo, *tasks);
    AW_CHECK_LAUNCH();
    *ntasks = (int64_t)total;
    return AW_OK;
}

}  // namespace

// AW_GRID_HYBRID: the gridding items of w planes [0, split_planes) for the
// TILES part and the degridding items of the other planes for the OFFSETS
// part (order kept), plus the second stream and the fork / join events.  The
// w plane of bin ((k nw + p) npa + a) nfb + f is p.  Once per plan, on the host.
static int build_hybrid_items(aw_plan *plan, cudaStream_t s) {
    const int split = plan->tune.split_planes, per_plane = plan->npa * plan->nfb;
    auto filter = [&](const int4 *d_src, int64_t n, bool low, int4 **d_out, int64_t *n_out) -> int {
        std::vector<int4> h((size_t)n), keep;
        if (n) AW_CUDA_TRY(cudaMemcpyAsync(h.data(), d_src, sizeof(int4) * n, cudaMemcpyDeviceToHost, s));
        AW_CUDA_TRY(cudaStreamSynchronize(s));
        keep.reserve((size_t)n);
        for (const int4 &it : h)
            if (((it.z / per_plane) % plan->nw < split) == low) keep.push_back(it);
        *n_out = (int64_t)keep.size();
        if (!keep.empty()) {
            AW_CUDA_TRY(aw_dev_malloc(d_out, sizeof(int4) * keep.size()));
            AW_CUDA_TRY(cudaMemcpyAsync(*d_out, keep.data(), sizeof(int4) * keep.size(), cudaMemcpyHostToDevice, s));
            AW_CUDA_TRY(cudaStreamSynchronize(s));
        }
        return AW_OK;
    };
    int rc = filter(plan->d_items, plan->nitems, true, &plan->d_items_ht, &plan->nitems_ht);
    if (rc) return rc;
    rc = filter(plan->d_items_dg, plan->nitems_dg, false, &plan->d_items_ho, &plan->nitems_ho);
    if (rc) return rc;
    AW_CUDA_TRY(cudaStreamCreateWithFlags(&plan->aux, cudaStreamNonBlocking));
    AW_CUDA_TRY(cudaEventCreateWithFlags(&plan->ev_fork, cudaEventDisableTiming));
    AW_CUDA_TRY(cudaEventCreateWithFlags(&plan->ev_join, cudaEventDisableTiming));
    return AW_OK;
}

constexpr int64_t RDG_MIN = 128;   // visibilities a region degridding task, on average
// Sparse full-pol sets take OFFSETS alone: below RG_SPARSE visibilities a bin and
// region tile, clearing and adding the four planes of a region costs more than
// atomics (25k visibilities of 128 bins on 4096^2, 4 a tile: 506 us against 173; 45 sets of
// 20k-2.9M: OFFSETS the faster one in all 26 below 28, equal about 60, up to 0.55 of
// its speed above 200).
constexpr int64_t RG_SPARSE = 24;
// The region order of the eligible bins and its tasks; the sort buffers are the
// plan builder's (>= nv).
template <typename K>
static int sort_region(aw_plan *plan, int64_t nv, const int4 *d_geo, int nb, int nt, uint64_t maxkey,
                       unsigned long long *d_nreg, SortBufs &b, cudaStream_t s) {
    K *keys = reinterpret_cast<K *>(b.k0);
    uint32_t *perm = nullptr;
    rg_key_kernel<K><<<grid_blocks(nv, 256), 256, 0, s>>>(plan->d_rec_dg, nv, d_geo, nt, (K)maxkey, keys, d_nreg);
    AW_CHECK_LAUNCH();
    int rc = radix_sort<K>(keys, perm, nv, key_bits(maxkey), b, s);
    if (rc) return rc;
    unsigned long long nreg = 0;
    AW_CUDA_TRY(cudaMemcpyAsync(&nreg, d_nreg, sizeof(nreg), cudaMemcpyDeviceToHost, s));
    AW_CUDA_TRY(cudaStreamSynchronize(s));
    plan->nreg = (int64_t)nreg;
    if (plan->nreg == 0) return AW_OK;
    int64_t nseg = 0;
    rc = build_segments<K>(keys, plan->nreg, 0, b, &nseg, s);
    if (rc == AW_OK && plan->npol == 4 && plan->nreg < RG_SPARSE * nseg) {
        plan->nreg = 0;
        return AW_OK;
    }
    if (rc == AW_OK) {
        AW_CUDA_TRY(aw_dev_malloc(&plan->d_rec_rg, sizeof(aw_rec) * plan->nreg));
        gather_rec_kernel<<<grid_blocks(plan->nreg, 256), 256, 0, s>>>(plan->d_rec_dg, perm, plan->nreg, plan->d_rec_rg);
        AW_CHECK_LAUNCH();
        rc = build_region_tasks(nseg, plan->nreg, plan->npol, 0, plan->d_rec_rg, d_geo, d_nreg, b, &plan->d_items_rg,
                                &plan->nitems_rg, s);
    }
    if (rc == AW_OK && plan->nitems_rg == 0) {   // too many tasks
        aw_dev_free(plan->d_rec_rg);
        plan->d_rec_rg = nullptr;
        plan->nreg = 0;
        return AW_OK;
    }
    // Region degridding pays a region's load (and its latency) per task: taken where the
    // tasks, as they are cut for this set, are half full on average (20.16M Stokes-I
    // visibilities, 237 a task: 2.9 against 5.8 ms; 1M, 80 a task: 472 against 357 us).
    // Their size is limited by the set's as well as by the tiles' density, so sets below
    // RDG_MIN x 12 tasks an SM (233,000 visibilities on 152 SMs) never take it.
    if (rc == AW_OK && plan->npol == 1 && plan->nreg >= RDG_MIN * nseg)
        rc = build_region_tasks(nseg, plan->nreg, 1, RDG_MIN, plan->d_rec_rg, d_geo + nb, d_nreg, b, &plan->d_items_rgd,
                                &plan->nitems_rgd, s);
    return rc;
}

// AW_GRID_REGION: the region order of the valid visibilities of the bins on
// the region kernel, its tasks, and the OFFSETS items of the other bins with
// the second stream.  The region kernel is the faster one at every support it
// takes (aw_rg_eligible), so every plane goes there, split_planes or not.
static int build_region(aw_plan *plan, const aw_kernel_set *ks, int64_t nv, SortBufs &b, cudaStream_t s) {
    const int nb = ks->nbins;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // gridding geometry of every bin, then the degridding one
    std::vector<int4> geo((size_t)nb * 2, make_int4(0, 0, 0, 0));
    bool all = true, any = false;
    for (int i = 0; i < nb; ++i) {
        const int S = ks->bin_support[(size_t)i];
        if (ks->max_support > AW_RG_MIN_SUPPORT && aw_rg_eligible(S, plan->npol)) {
            // visibilities a task: enough tasks to fill the SMs twice (8 gridding CTAs, 6
            // degridding CTAs each), as far as the limits allow (126k visibilities of 7 x 7 taps
            // on 512^2: 35 us, 106 with the largest tasks)
            const int64_t k = (int64_t)aw_rg_nblk(S) * aw_rg_nblk(S) * plan->npol;
            const int64_t cap = std::min<int64_t>(std::max<int64_t>(nv * k / (sms * 16) / 64 * 64, 64), AW_RG_MAXV);
            const int64_t capd = std::min<int64_t>(std::max<int64_t>(nv / (sms * 12) / 32 * 32, 32), AW_RG_MAXV_DG);
            geo[(size_t)i] = make_int4(aw_rg_tile(S), (int)cap, aw_rg_nblk(S), 0);
            geo[(size_t)nb + i] = make_int4(aw_rg_tile(S), (int)capd, 1, 0);
            any = true;
        } else {
            all = false;
        }
    }
    if (any) {
        DevBuf dgeo, dcnt;
        AW_CUDA_TRY(aw_dev_malloc(&dgeo.p, sizeof(int4) * geo.size()));
        AW_CUDA_TRY(cudaMemcpyAsync(dgeo.p, geo.data(), sizeof(int4) * geo.size(), cudaMemcpyHostToDevice, s));
        AW_CUDA_TRY(aw_dev_malloc(&dcnt.p, sizeof(unsigned long long)));
        AW_CUDA_TRY(cudaMemsetAsync(dcnt.p, 0, sizeof(unsigned long long), s));
        const int nt = (plan->N + aw_rg_tile(128) - 1) / aw_rg_tile(128);   // tiles an axis at the smallest tile side
        const uint64_t maxkey = (uint64_t)nb * nt * nt;                     // also the key of the bins that take no region
        const int4 *d_geo = (const int4 *)dgeo.p;
        unsigned long long *d_nreg = (unsigned long long *)dcnt.p;
        const int rc = key_bits(maxkey) <= 32 ? sort_region<uint32_t>(plan, nv, d_geo, nb, nt, maxkey, d_nreg, b, s)
                                              : sort_region<uint64_t>(plan, nv, d_geo, nb, nt, maxkey, d_nreg, b, s);
        if (rc) return rc;
        AW_CUDA_TRY(cudaStreamSynchronize(s));   // the geometry is freed here
    }
    if (plan->nreg == 0) {
        all = false;
        std::fill(geo.begin(), geo.end(), make_int4(0, 0, 0, 0));
    }
    // the other bins: their degridding items on the OFFSETS schedule
    if (!all) {
        std::vector<int4> hd((size_t)plan->nitems_dg), keep;
        if (plan->nitems_dg)
            AW_CUDA_TRY(cudaMemcpyAsync(hd.data(), plan->d_items_dg, sizeof(int4) * plan->nitems_dg, cudaMemcpyDeviceToHost, s));
        AW_CUDA_TRY(cudaStreamSynchronize(s));
        for (const int4 &it : hd)
            if (geo[(size_t)it.z].x == 0) keep.push_back(it);
        plan->nitems_ho = (int64_t)keep.size();
        if (!keep.empty()) {
            AW_CUDA_TRY(aw_dev_malloc(&plan->d_items_ho, sizeof(int4) * keep.size()));
            AW_CUDA_TRY(cudaMemcpyAsync(plan->d_items_ho, keep.data(), sizeof(int4) * keep.size(), cudaMemcpyHostToDevice, s));
            AW_CUDA_TRY(cudaStreamSynchronize(s));
        }
        AW_CUDA_TRY(cudaStreamCreateWithFlags(&plan->aux, cudaStreamNonBlocking));
        AW_CUDA_TRY(cudaEventCreateWithFlags(&plan->ev_fork, cudaEventDisableTiming));
        AW_CUDA_TRY(cudaEventCreateWithFlags(&plan->ev_join, cudaEventDisableTiming));
    }
    AW_CUDA_TRY(cudaStreamSynchronize(s));
    return AW_OK;
}

int aw_plan_plane_taps(const aw_plan *plan, std::vector<double> &cum, cudaStream_t s) {
    cum.assign((size_t)plan->nw + 1, 0.0);
    std::vector<int4> h((size_t)plan->nitems);
    if (plan->nitems) AW_CUDA_TRY(cudaMemcpyAsync(h.data(), plan->d_items, sizeof(int4) * plan->nitems,
                                                  cudaMemcpyDeviceToHost, s));
    AW_CUDA_TRY(cudaStreamSynchronize(s));
    const int per_plane = plan->npa * plan->nfb;
    for (const int4 &it : h) {
        const double S = plan->bin_support[(size_t)it.z];
        cum[(size_t)((it.z / per_plane) % plan->nw) + 1] += (double)it.y * S * S;
    }
    for (size_t q = 1; q < cum.size(); ++q) cum[q] += cum[q - 1];
    if (cum.back() > 0)
        for (double &c : cum) c /= cum.back();
    return AW_OK;
}

int aw_plan_build(aw_ctx *ctx, const aw_vis_desc *vis, const aw_kernel_set *ks, const aw_tune *tune,
                  aw_plan *plan, cudaStream_t s) {
    if (!vis || vis->nvis < 0 || (vis->nvis > 0 && (!vis->uvw || !vis->row_of_vis || !vis->chan_of_vis || !vis->freq)))
        return aw_set_error(AW_EINVAL, "vis descriptor incomplete");
    if (vis->nvis > 0x7fffffffLL) return aw_set_error(AW_EINVAL, "nvis %lld above 2^31-1", (long long)vis->nvis);
    const aw_kernel_spec &sp = ks->spec;
    aw_tune t = tune ? *tune : aw_tune{32, 256, 5, 0, AW_GRID_TILES};
    if (t.tile < 8 || t.tile > 256 || (t.tile & (t.tile - 1))) return aw_set_error(AW_EINVAL, "tile %d", t.tile);
    if (t.chunk < 32 || t.chunk > 2048) return aw_set_error(AW_EINVAL, "chunk %d", t.chunk);
    if (t.ctas_per_sm < 1 || t.ctas_per_sm > 8) t.ctas_per_sm = 2;
    if (t.dg_tile == 0) t.dg_tile = 1024;
    if (t.dg_tile < 32 || t.dg_tile > 4096 || (t.dg_tile & (t.dg_tile - 1)))
        return aw_set_error(AW_EINVAL, "dg_tile %d", t.dg_tile);
    if (t.grid_mode != AW_GRID_TILES && t.grid_mode != AW_GRID_OFFSETS && t.grid_mode != AW_GRID_HYBRID &&
        t.grid_mode != AW_GRID_REGION)
        return aw_set_error(AW_EINVAL, "grid_mode %d", t.grid_mode);
    if ((t.grid_mode == AW_GRID_HYBRID || t.grid_mode == AW_GRID_REGION) &&
        (t.split_planes < 0 || t.split_planes > sp.nw))
        return aw_set_error(AW_EINVAL, "split_planes %d outside 0..%d", t.split_planes, sp.nw);
    plan->tune = t;
    plan->dg_tile = t.dg_tile;
    plan->nvis = vis->nvis;
    plan->N = sp.N;
    plan->OS = sp.OS;
    plan->npol = sp.npol;
    plan->nbins = ks->nbins;
    plan->nw = sp.nw;
    plan->npa = sp.npa;
    plan->nfb = sp.nfb;
    plan->ntype = ks->ntype;
    plan->vis = *vis;
    // per-plane supports first (the coordinate step indexes by w plane), then per bin
    std::vector<int32_t> sup(ks->supports.begin(), ks->supports.end());
    plan->bin_support = ks->bin_support;
    const int64_t n = vis->nvis;
    const int nchan = std::min(std::max(vis->nchan, 0), 65536);   // (chan_of_vis has 16 bits)
    AW_CUDA_TRY(aw_dev_malloc(&plan->d_plane_support, sizeof(int32_t) * std::max<size_t>(sup.size(), 1)));
    AW_CUDA_TRY(aw_dev_malloc(&plan->d_fl, sizeof(double) * std::max(nchan, 1)));
    AW_CUDA_TRY(aw_dev_malloc(&plan->d_wsum, sizeof(double)));
    AW_CUDA_TRY(aw_dev_malloc(&plan->d_nonfinite, sizeof(unsigned long long)));
    AW_CUDA_TRY(aw_dev_malloc(&plan->d_counter, sizeof(unsigned int) * 5));
    plan->d_rcounter = plan->d_counter + 4;
    AW_CUDA_TRY(aw_dev_malloc(&plan->d_rec, sizeof(aw_rec) * std::max<int64_t>(n, 1)));
    AW_CUDA_TRY(cudaMemcpyAsync(plan->d_plane_support, sup.data(), sizeof(int32_t) * sup.size(),
                                cudaMemcpyHostToDevice, s));
    if (n == 0) {
        AW_CUDA_TRY(aw_dev_malloc(&plan->d_items, sizeof(int4)));
        AW_CUDA_TRY(cudaStreamSynchronize(s));
        return AW_OK;
    }
    if (nchan > 0) {
        channel_kernel<<<grid_blocks(nchan, 256), 256, 0, s>>>(vis->freq, nchan, plan->d_fl);
        AW_CHECK_LAUNCH();
    }
    CoordArgs a;
    fill_coord_args(vis, ks, t.tile, a, plan);
    plan->uscale = a.uscale;
    plan->half = a.half;
    plan->winv = a.winv;
    // keys: bins x tiles x (tile position), and one value for invalid ones
    const uint64_t maxkey = ((uint64_t)ks->nbins * a.nty * a.ntx) << (2 * a.tbits);
    const int kbits = key_bits(maxkey);

    // the temporaries, in one allocation
    const int64_t ntiles = (n + RS_TILE - 1) / RS_TILE;
    const size_t words = (size_t)std::max<int64_t>(ntiles * RS_DIGITS, n + 1);
    Arena ar;
    ar.size = 2 * Arena::round(sizeof(uint64_t) * n) + 2 * Arena::round(sizeof(uint32_t) * n) +
              Arena::round(sizeof(aw_rec) * n) + 3 * Arena::round(sizeof(uint32_t) * words) +
              Arena::round(aw_scan_scratch_bytes((int64_t)words)) + Arena::round(sizeof(unsigned long long) * 4);
    AW_CUDA_TRY(aw_dev_malloc(&ar.buf.p, ar.size));
    SortBufs b;
    b.k0 = ar.take<uint64_t>(n);
    b.k1 = ar.take<uint64_t>(n);
    b.v0 = ar.take<uint32_t>(n);
    b.v1 = ar.take<uint32_t>(n);
    aw_rec *rec = ar.take<aw_rec>(n);
    for (auto &w : b.words) w = ar.take<uint32_t>(words);
    b.scratch = ar.take<char>(aw_scan_scratch_bytes((int64_t)words));
    unsigned long long *d_cnt = ar.take<unsigned long long>(4);
    AW_CUDA_TRY(cudaMemsetAsync(d_cnt, 0, sizeof(unsigned long long) * 4, s));
    // the gridding order and its items: runs of equal (bin, tile), then chunks
    auto grid_order = [&](auto key) -> int {
        using K = decltype(key);
        K *keys = reinterpret_cast<K *>(b.k0);
        uint32_t *perm = nullptr;
        coords_kernel<K><<<grid_blocks(n, 256), 256, 0, s>>>(a, (K)maxkey, keys, rec, d_cnt);
        AW_CHECK_LAUNCH();
        int rc = radix_sort<K>(keys, perm, n, kbits, b, s);
        if (rc) return rc;
        gather_rec_kernel<<<grid_blocks(n, 256), 256, 0, s>>>(rec, perm, n, plan->d_rec);
        AW_CHECK_LAUNCH();
        unsigned long long hc[4];
        AW_CUDA_TRY(cudaMemcpyAsync(hc, d_cnt, sizeof(hc), cudaMemcpyDeviceToHost, s));
        AW_CUDA_TRY(cudaStreamSynchronize(s));
        plan->n_outside = (int64_t)hc[0];
        plan->n_flagged = (int64_t)hc[1];
        plan->nvalid = (int64_t)hc[2];
        plan->mean_taps = hc[2] ? (double)hc[3] / (double)hc[2] : 0.0;
        if (plan->nvalid == 0) {
            AW_CUDA_TRY(aw_dev_malloc(&plan->d_items, sizeof(int4)));
            plan->nitems = 0;
            return AW_OK;
        }
        return build_items<K>(keys, plan->nvalid, 2 * a.tbits, t.chunk, plan->d_rec, b, &plan->d_items,
                              &plan->nitems, s);
    };
    int rc = kbits <= 32 ? grid_order(uint32_t()) : grid_order(uint64_t());
    if (rc || plan->nvalid == 0) return rc;
    const int64_t nv = plan->nvalid;
    // CTAs an SM of the default schedule: five for Stokes I (5083 items 125 us against 179
    // with two, 353 items 27.3 / 27.3).  At full polarisation they meet on the cells of
    // the few tiles that are in work, so three (9815 items 2.69 ms against 3.06; five 2.69) and
    // two for small sets (490 items 70.7 us against 75.3 with three and 78.5 with five, 624
    // items 59.3 / 64.2 / 67.5, 1222 items equal, 1297 items 427 / 360 / 342).
    if (!tune && plan->npol == 4) plan->tune.ctas_per_sm = plan->nitems >= 8 * (int64_t)ctx->sm_count ? 3 : 2;

    // degridding order: (bin, super-tile, oversampled offset), the grid order inside
    const int stbits = ilog2(plan->dg_tile);
    const int nst = (sp.N + plan->dg_tile - 1) >> stbits;
    const uint64_t ngroups = (uint64_t)ks->nbins * nst * nst * sp.OS * sp.OS;
    auto degrid_order = [&](auto key) -> int {
        using K = decltype(key);
        K *keys = reinterpret_cast<K *>(b.k0);
        uint32_t *perm = nullptr;
        dg_key_kernel<K><<<grid_blocks(nv, 256), 256, 0, s>>>(plan->d_rec, nv, sp.OS, stbits, nst, keys);
        AW_CHECK_LAUNCH();
        int r = radix_sort<K>(keys, perm, nv, key_bits(ngroups), b, s);
        if (r) return r;
        AW_CUDA_TRY(aw_dev_malloc(&plan->d_rec_dg, sizeof(aw_rec) * nv));
        gather_rec_kernel<<<grid_blocks(nv, 256), 256, 0, s>>>(plan->d_rec, perm, nv, plan->d_rec_dg);
        AW_CHECK_LAUNCH();
        return build_items<K>(keys, nv, 0, AW_DG_CHUNK, plan->d_rec_dg, b, &plan->d_items_dg, &plan->nitems_dg, s);
    };
    rc = key_bits(ngroups) <= 32 ? degrid_order(uint32_t()) : degrid_order(uint64_t());
    if (rc) return rc;
    if (t.grid_mode == AW_GRID_HYBRID) {
        rc = build_hybrid_items(plan, s);
        if (rc) return rc;
    }
    if (t.grid_mode == AW_GRID_REGION) {
        rc = build_region(plan, ks, nv, b, s);
        if (rc) return rc;
    }
    AW_CUDA_TRY(cudaStreamSynchronize(s));
    return AW_OK;
}

int aw_plan_coords_impl(const aw_plan *plan, const aw_kernel_set *ks_unused, int32_t *x0, int32_t *y0,
                        int32_t *fx, int32_t *fy, int32_t *bin, uint8_t *flip, uint8_t *valid,
                        cudaStream_t s) {
    (void)ks_unused;
    if (plan->nvis == 0) return AW_OK;
    CoordArgs a;
    const aw_vis_desc *vis = &plan->vis;
    a.nvis = vis->nvis;
    a.uvw = vis->uvw;
    a.row = vis->row_of_vis;
    a.chan = vis->chan_of_vis;
    a.freq = vis->freq;
    a.fl = plan->d_fl;
    a.pa_bin = vis->pa_bin;
    a.fbin = vis->fbin;
    a.flags = vis->flags;
    a.row_types = vis->row_types;
    a.N = plan->N;
    a.OS = plan->OS;
    a.nw = plan->nw;
    a.npa = plan->npa;
    a.nfb = plan->nfb;
    a.ntype = plan->ntype;
    a.uscale = plan->uscale;
    a.half = plan->half;
    a.winv = plan->winv;
    a.support = plan->d_plane_support;
    a.nchan = vis->nchan;
    a.tile = plan->tune.tile;
    a.tbits = ilog2(plan->tune.tile);
    a.ntx = a.nty = (plan->N + plan->tune.tile - 1) / plan->tune.tile;
    coords_out_kernel<<<grid_blocks(plan->nvis, 256), 256, 0, s>>>(a, x0, y0, fx, fy, bin, flip, valid);
    AW_CHECK_LAUNCH();
    return AW_OK;
}

int aw_plan_order_impl(const aw_plan *plan, uint32_t *perm, cudaStream_t s) {
    if (plan->nvis == 0) return AW_OK;
    rec_orig_kernel<<<grid_blocks(plan->nvis, 256), 256, 0, s>>>(plan->d_rec, plan->nvis, perm);
    AW_CHECK_LAUNCH();
    return AW_OK;
}

// ------------------------------------------------------------ exclusive scan
// Three phases over blocks of SCAN_BLOCK elements: block sums, a scan of the
// block sums by one block, then the block-local scan plus its offset.
constexpr int SCAN_THREADS = 512;
constexpr int SCAN_ITEMS = 4;
constexpr int SCAN_BLOCK = SCAN_THREADS * SCAN_ITEMS;

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *total) {
    __shared__ uint32_t warp_sums[SCAN_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t ws = (lane < SCAN_THREADS / 32) ? warp_sums[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, ws, o);
            if (lane >= o) ws += y;
        }
        if (lane < SCAN_THREADS / 32) warp_sums[lane] = ws;
    }
    __syncthreads();
    const uint32_t before = (warp > 0 ? warp_sums[warp - 1] : 0) + x - v;
    if (total) *total = warp_sums[SCAN_THREADS / 32 - 1];
    __syncthreads();
    return before;
}

__global__ void scan_reduce_kernel(const uint32_t *in, int64_t n, uint32_t *bsum) {
    const int64_t base = (int64_t)blockIdx.x * SCAN_BLOCK + (int64_t)threadIdx.x * SCAN_ITEMS;
    uint32_t s = 0;
    for (int i = 0; i < SCAN_ITEMS; ++i)
        if (base + i < n) s += in[base + i];
    uint32_t total;
    block_exclusive_scan(s, &total);
    if (threadIdx.x == 0) bsum[blockIdx.x] = total;
}

__global__ void scan_sums_kernel(uint32_t *bsum, int64_t nb) {
    __shared__ uint32_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int64_t base = 0; base < nb; base += SCAN_THREADS) {
        const int64_t i = base + threadIdx.x;
        const uint32_t v = (i < nb) ? bsum[i] : 0;
        uint32_t total;
        const uint32_t ex = block_exclusive_scan(v, &total);
        if (i < nb) bsum[i] = carry + ex;
        __syncthreads();
        if (threadIdx.x == 0) carry += total;
        __syncthreads();
    }
}

__global__ void scan_apply_kernel(const uint32_t *in, int64_t n, const uint32_t *bsum, uint32_t *out) {
    const int64_t base = (int64_t)blockIdx.x * SCAN_BLOCK + (int64_t)threadIdx.x * SCAN_ITEMS;
    uint32_t v[SCAN_ITEMS];
    uint32_t s = 0;
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        v[i] = (base + i < n) ? in[base + i] : 0;
        s += v[i];
    }
    uint32_t run = block_exclusive_scan(s, nullptr) + bsum[blockIdx.x];
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        if (base + i < n) out[base + i] = run;
        run += v[i];
    }
}

size_t aw_scan_scratch_bytes(int64_t n) {
    const int64_t nb = (n + SCAN_BLOCK - 1) / SCAN_BLOCK;
    return sizeof(uint32_t) * (size_t)std::max<int64_t>(nb, 1);
}

int aw_exclusive_scan_u32(const uint32_t *in, uint32_t *out, int64_t n, void *scratch, cudaStream_t s) {
    if (n <= 0) return AW_OK;
    const int64_t nb = (n + SCAN_BLOCK - 1) / SCAN_BLOCK;
    if (nb > 0x7fffffffLL) return aw_set_error(AW_EINVAL, "scan too large");
    uint32_t *bsum = (uint32_t *)scratch;
    scan_reduce_kernel<<<(unsigned)nb, SCAN_THREADS, 0, s>>>(in, n, bsum);
    AW_CHECK_LAUNCH();
    scan_sums_kernel<<<1, SCAN_THREADS, 0, s>>>(bsum, nb);
    AW_CHECK_LAUNCH();
    scan_apply_kernel<<<(unsigned)nb, SCAN_THREADS, 0, s>>>(in, n, bsum, out);
    AW_CHECK_LAUNCH();
    return AW_OK;
}
