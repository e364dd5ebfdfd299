// Device spatial index: cell keys, a stable LSD radix sort of (key, index),
// the sorted point arrays and the first-slot table of every cell.
//
// Replaces the paper's node-local k-d tree (Algorithm 1, "search node-local
// k-d tree for neighbors"; Sec. 5.1, FP32 tree search) with a uniform grid of
// side >= rmax/s whose cells are ordered by (catalog, Morton(cy, cz), cx): an
// x-row of cells is one contiguous slot range, so a sphere of radius rmax is
// covered by a few dozen contiguous ranges.  Everything here is HBM-bound
// streaming (a few passes over 8-16 bytes per point).
#include "internal.h"

#include <cstdio>

namespace g3 {

namespace {

// Radix tiles: up to kSmallSort points 1,024 keys, one per thread, so that a small
// catalog spreads over the chip, ranks its keys in one round, and every CTA forms the
// digit offsets from all tiles' counts by itself (no scan launches); above, 4,096 keys,
// 16 per thread, and scan launches, as that sum grows with the square of the tiles.  The
// whole index in the small / large form: 37 / 70 us at 1,000 points, 40 / 94 at 20,000,
// 46 / 110 at 2^17, 64 / 113 at 2^18, 117 / 115 at 2^19, 256 / 143 at 2^20.
constexpr int64_t kSmallSort = 1 << 18;
constexpr int kSmallThreads = 1024, kSmallItems = 1;
constexpr int kLargeThreads = 256, kLargeItems = 16;
constexpr int kPrimTile = 1024;  // slots per counter of the primaries' compaction
constexpr int kScanBlock = 1024;

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Position i of the input in FP64 (0 where it is out of range: flagged in k_keys).
__device__ __forceinline__ bool load_pos(const IndexArgs& a, int64_t i, double (&x)[3]) {
    if (a.pos_f64) {
        const double* p = static_cast<const double*>(a.pos) + 3 * i;
        x[0] = p[0]; x[1] = p[1]; x[2] = p[2];
    } else {
        const float* p = static_cast<const float*>(a.pos) + 3 * i;
        x[0] = p[0]; x[1] = p[1]; x[2] = p[2];
    }
    bool ok = true;
    for (int d = 0; d < 3; ++d)
        if (!(x[d] >= 0.0 && x[d] < a.g.boxd)) {  // also catches NaN
            ok = false;
            x[d] = 0.0;
        }
    return ok;
}

// ---- keys and the first digit's histogram --------------------------------------

// hist: [tile][256] counts of the lowest digit; zero[0 .. nzero): cleared for the
// later passes' histograms and the primaries' counters.
template <int THREADS, int ITEMS>
__global__ void __launch_bounds__(THREADS) k_keys(IndexArgs a, const int64_t* cat_off, int ncat, unsigned* key,
                                                       int* status, int* hist, int* zero, int64_t nzero) {
    __shared__ int h[256];
    if (threadIdx.x < 256) h[threadIdx.x] = 0;
    for (int64_t k = blockIdx.x * (int64_t)THREADS + threadIdx.x; k < nzero; k += (int64_t)gridDim.x * THREADS)
        zero[k] = 0;
    __syncthreads();
    const int64_t base = blockIdx.x * (int64_t)(THREADS * ITEMS) + threadIdx.x;
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const int64_t i = base + it * THREADS;
        if (i >= a.n) continue;
        double x[3];
        const bool ok = load_pos(a, i, x);
        if (!ok || !isfinite(a.w[i])) atomicOr(status, kStatusRange);
        int c[3];
        for (int d = 0; d < 3; ++d) {
            const float xf = (float)x[d];
            const int n = d == 0 ? a.g.ncx : a.g.nc;
            const int cc = (int)(xf * (d == 0 ? a.g.inv_cellx : a.g.inv_cell));
            c[d] = cc < 0 ? 0 : (cc >= n ? n - 1 : cc);
        }
        long long cat = 0;
        if (cat_off) {
            int lo = 0, hi = ncat - 1;  // last catalog with cat_off[c] <= i
            while (lo < hi) {
                int mid = (lo + hi + 1) >> 1;
                if (cat_off[mid] <= i) lo = mid; else hi = mid - 1;
            }
            cat = lo;
        }
        const unsigned k = (unsigned)(cat * a.g.cells_per_cat + (long long)morton2(c[1], c[2]) * a.g.ncx + c[0]);
        key[i] = k;
        atomicAdd(&h[k & 255u], 1);
    }
    __syncthreads();
    if (threadIdx.x < 256) hist[blockIdx.x * 256 + threadIdx.x] = h[threadIdx.x];
}

// ---- exclusive scan (int32) --------------------------------------------

__device__ int block_scan_excl(int v, int* sh, int& total) {
    // blockDim.x == kScanBlock; warp shuffles then warp totals
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int s = (lane < (int)(blockDim.x >> 5)) ? sh[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        sh[lane] = s;  // inclusive over warps
    }
    __syncthreads();
    int pre = (wid > 0 ? sh[wid - 1] : 0) + x - v;
    total = sh[(blockDim.x >> 5) - 1];
    __syncthreads();
    return pre;
}

// The radix offsets: an exclusive scan of hist in (digit, tile) order, in place of
// [tile][digit].  Element e = digit * ntiles + tile.
__device__ __forceinline__ int64_t hist_at(int64_t e, int ntiles) { return (e % ntiles) * 256 + e / ntiles; }

__global__ void k_scan_reduce(const int* in, int ntiles, int64_t n, int* bsum) {
    __shared__ int sh[32];
    const int64_t i = blockIdx.x * (int64_t)kScanBlock + threadIdx.x;
    int tot;
    block_scan_excl(i < n ? in[hist_at(i, ntiles)] : 0, sh, tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

__global__ void k_scan_top(int* bsum, int nb) {
    __shared__ int sh[32];
    int carry = 0;
    for (int base = 0; base < nb; base += kScanBlock) {
        int i = base + threadIdx.x;
        int v = i < nb ? bsum[i] : 0;
        int tot;
        int pre = block_scan_excl(v, sh, tot);
        if (i < nb) bsum[i] = carry + pre;
        carry += tot;
    }
}

__global__ void k_scan_final(int* io, int ntiles, int64_t n, const int* bsum) {
    __shared__ int sh[32];
    const int64_t i = blockIdx.x * (int64_t)kScanBlock + threadIdx.x;
    int tot;
    const int v = i < n ? io[hist_at(i, ntiles)] : 0;
    const int pre = block_scan_excl(v, sh, tot);
    if (i < n) io[hist_at(i, ntiles)] = bsum[blockIdx.x] + pre;
}

// ---- radix sort -----------------------------------------------------------

struct ScatterArgs {
    const unsigned* key;
    const int* val;        // null in the first pass: value i
    int64_t n;
    int shift, ntiles;
    const int* hist;       // [tile][256]: counts (SCANNED = false) or offsets
    unsigned* key_out;
    int* val_out;          // not written by the last pass
    int* hist_next;        // next digit's histogram (not the last pass)
    // last pass: the sorted arrays
    float4* pts;
    double* pts64;
    int* orig;
    int* negw;
    int64_t n_primary;     // < n: count the primaries per kPrimTile slots
    int* prim_count;
};

// Stable scatter: warp w of a tile owns 32 ITEMS consecutive items and ranks them
// round by round (32 at a time) with per-warp digit counters; the warps' counters
// are then prefix-summed per digit in warp order.  With few tiles every CTA forms
// its own digit offsets from the tiles' counts (no scan launches); the pass counts
// the next digit while it scatters, and the last one writes the sorted points.
template <int THREADS, int ITEMS, bool SCANNED, bool LAST>
__global__ void __launch_bounds__(THREADS) k_radix_scatter(ScatterArgs s, IndexArgs a) {
    constexpr int kWarps = THREADS / 32;
    constexpr int kPerWarp = 32 * ITEMS;
    constexpr int kTile = THREADS * ITEMS;
    constexpr int kParts = THREADS / 256;  // threads per digit
    __shared__ int wcnt[kWarps][257];
    __shared__ int soff[256];
    __shared__ int wsum[8];
    __shared__ int2 part[kParts][256];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int d = threadIdx.x; d < kWarps * 257; d += THREADS) (&wcnt[0][0])[d] = 0;
    const int dig = threadIdx.x & 255, grp = threadIdx.x >> 8;
    if constexpr (SCANNED) {
        if (grp == 0) soff[dig] = s.hist[(int64_t)blockIdx.x * 256 + dig];
    } else {
        // items of lower digits, plus those of the digit in earlier tiles
        int before = 0, tot = 0;
#pragma unroll 8
        for (int t = grp; t < s.ntiles; t += kParts) {
            const int v = __ldg(s.hist + t * 256 + dig);
            before += t < (int)blockIdx.x ? v : 0;
            tot += v;
        }
        part[grp][dig] = make_int2(before, tot);
        __syncthreads();
        int x = 0;
        if (grp == 0) {
            for (int k = 1; k < kParts; ++k) {
                before += part[k][dig].x;
                tot += part[k][dig].y;
            }
            x = tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (lane == 31) wsum[wid] = x;
        }
        __syncthreads();
        if (grp == 0) {
            int pre = 0;
            for (int w = 0; w < wid; ++w) pre += wsum[w];
            soff[dig] = pre + x - tot + before;
        }
    }
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kTile + wid * kPerWarp;
    unsigned kk[ITEMS];
    int vv[ITEMS], loc[ITEMS];
    const unsigned lt = lanemask_lt();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int64_t i = base + r * 32 + lane;
        kk[r] = 0;
        vv[r] = 0;
        if (i < s.n) {
            kk[r] = s.key[i];
            vv[r] = s.val ? s.val[i] : (int)i;
        }
    }
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int dg = base + r * 32 + lane < s.n ? (kk[r] >> s.shift) & 255u : 256;  // 256: past the end
        const unsigned peers = __match_any_sync(0xffffffffu, dg);
        const int b = wcnt[wid][dg];
        loc[r] = b + __popc(peers & lt);
        __syncwarp();
        if ((peers & lt) == 0u) wcnt[wid][dg] = b + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    if (grp == 0) {
        int run = soff[dig];
        for (int w = 0; w < kWarps; ++w) {
            const int t = wcnt[w][dig];
            wcnt[w][dig] = run;
            run += t;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        if (base + r * 32 + lane >= s.n) continue;
        const int pos = wcnt[wid][(kk[r] >> s.shift) & 255u] + loc[r];
        s.key_out[pos] = kk[r];
        if constexpr (!LAST) {
            s.val_out[pos] = vv[r];
            atomicAdd(&s.hist_next[(int64_t)(pos / kTile) * 256 + ((kk[r] >> (s.shift + 8)) & 255u)], 1);
        } else {
            double x[3];
            load_pos(a, vv[r], x);
            float w = a.w[vv[r]];
            if (!isfinite(w)) w = 0.f;
            if (w < 0.f) *s.negw = 1;
            s.pts[pos] = make_float4((float)x[0], (float)x[1], (float)x[2], w);
            if (s.pts64) {
                s.pts64[3 * (int64_t)pos + 0] = x[0];
                s.pts64[3 * (int64_t)pos + 1] = x[1];
                s.pts64[3 * (int64_t)pos + 2] = x[2];
            }
            s.orig[pos] = vv[r];
            if (s.prim_count && vv[r] < s.n_primary) atomicAdd(&s.prim_count[pos / kPrimTile], 1);
        }
    }
}

// ---- cell starts, primary list ------------------------------------------------

__global__ void k_cell_start(const unsigned* key, int64_t n, long long ncells, int* cstart) {
    long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (c > ncells) return;
    int64_t lo = 0, hi = n;  // first slot with key >= c
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if ((long long)key[mid] < c) lo = mid + 1; else hi = mid;
    }
    cstart[c] = (int)lo;
}

// Sorted slots of the primaries (original index < n_primary), in slot order: block
// t compacts the kPrimTile slots of counter t behind the counts before it.
__global__ void __launch_bounds__(kPrimTile) k_prim_compact(const int* orig, int64_t n, int64_t n_primary,
                                                            const int* count, int* plist) {
    __shared__ int sh[32];
    __shared__ int off;
    int before = 0;
    for (int t = threadIdx.x; t < (int)blockIdx.x; t += kPrimTile) before += count[t];
    if (threadIdx.x == 0) off = 0;
    __syncthreads();
    for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
    if ((threadIdx.x & 31) == 0 && before) atomicAdd(&off, before);
    const int64_t p = blockIdx.x * (int64_t)kPrimTile + threadIdx.x;
    const int flag = p < n && orig[p] < n_primary;
    int tot;
    const int pre = block_scan_excl(flag, sh, tot);
    if (flag) plist[off + pre] = (int)p;
}

// Batch: the slot ranges of the catalogs end to end (nr ranges, out ascending).
__global__ void k_iota_ranges(const int* rstart, const int* rlen, const int* rout, int nr, int64_t n, int* plist) {
    const int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (o >= n) return;
    int lo = 0, hi = nr - 1;  // last range with out <= o (empty ranges share their start)
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (rout[mid] <= o) lo = mid; else hi = mid - 1;
    }
    const int k = (int)o - rout[lo];
    if (k < rlen[lo]) plist[o] = rstart[lo] + k;
}

inline int grid_of(int64_t n, int b) { return (int)((n + b - 1) / b); }

}  // namespace

namespace {
constexpr int kSmallTile = kSmallThreads * kSmallItems, kLargeTile = kLargeThreads * kLargeItems;

template <int THREADS, int ITEMS, bool SCANNED>
void scatter_pass(const ScatterArgs& s, const IndexArgs& a, bool last, cudaStream_t st) {
    if (last)
        k_radix_scatter<THREADS, ITEMS, SCANNED, true><<<s.ntiles, THREADS, 0, st>>>(s, a);
    else
        k_radix_scatter<THREADS, ITEMS, SCANNED, false><<<s.ntiles, THREADS, 0, st>>>(s, a);
}
}  // namespace

// Histograms of up to 4 passes, the primaries' counters, and the scan's block sums.
size_t index_scratch_ints(int64_t n) {
    const int64_t tiles = n <= kSmallSort ? grid_of(n, kSmallTile) : grid_of(n, kLargeTile);
    return (size_t)(4 * 256 * tiles + grid_of(n, kPrimTile) + grid_of(256 * tiles, kScanBlock) + 1);
}

int build_index(IndexBuffers& b, const IndexArgs& a, const int64_t* cat_off_dev, int ncat,
                long long ncells, int64_t n_primary, const PrimRanges* ranges,
                cudaStream_t st) {
    const int64_t n = a.n;
    if (n <= 0) return 0;
    const int T = 256;
    int launches = 1;
    const bool small = n <= kSmallSort;
    const int ntiles = small ? grid_of(n, kSmallTile) : grid_of(n, kLargeTile);
    const int nprim_tiles = grid_of(n, kPrimTile);
    const int64_t hist = (int64_t)256 * ntiles;
    int* prim_count = b.scratch + 4 * hist;
    int* bsum = prim_count + nprim_tiles;
    // LSD radix sort on the bits in use
    int bits = 1;
    while (bits < 32 && ((unsigned long long)1 << bits) <= (unsigned long long)ncells) ++bits;
    const int passes = (bits + 7) / 8;
    if (small)
        k_keys<kSmallThreads, kSmallItems><<<ntiles, kSmallThreads, 0, st>>>(
            a, cat_off_dev, ncat, b.key_a, b.status, b.scratch, b.scratch + hist, 3 * hist + nprim_tiles);
    else
        k_keys<kLargeThreads, kLargeItems><<<ntiles, kLargeThreads, 0, st>>>(
            a, cat_off_dev, ncat, b.key_a, b.status, b.scratch, b.scratch + hist, 3 * hist + nprim_tiles);
    const bool subset = !ranges && n_primary < n;
    ScatterArgs s{};
    s.key = b.key_a;
    s.n = n;
    s.ntiles = ntiles;
    s.key_out = b.key_b;
    s.val_out = b.val_a;
    s.pts = b.pts;
    s.pts64 = b.pts64;
    s.orig = b.orig;
    s.negw = b.status + kNegWeightSlot;
    s.n_primary = n_primary;
    s.prim_count = subset ? prim_count : nullptr;
    for (int p = 0; p < passes; ++p) {
        s.shift = 8 * p;
        int* h = b.scratch + p * hist;
        s.hist = h;
        s.hist_next = h + hist;
        const bool last = p + 1 == passes;
        if (small) {
            scatter_pass<kSmallThreads, kSmallItems, false>(s, a, last, st);
            launches += 1;
        } else {
            const int nb = grid_of(hist, kScanBlock);
            k_scan_reduce<<<nb, kScanBlock, 0, st>>>(h, ntiles, hist, bsum);
            k_scan_top<<<1, kScanBlock, 0, st>>>(bsum, nb);
            k_scan_final<<<nb, kScanBlock, 0, st>>>(h, ntiles, hist, bsum);
            scatter_pass<kLargeThreads, kLargeItems, true>(s, a, last, st);
            launches += 4;
        }
        // the other buffers for the next pass
        unsigned* kin = const_cast<unsigned*>(s.key);
        s.key = s.key_out;
        s.key_out = kin;
        int* vin = s.val ? const_cast<int*>(s.val) : b.val_b;
        s.val = s.val_out;
        s.val_out = vin;
    }
    b.key_sorted = const_cast<unsigned*>(s.key);
    k_cell_start<<<(int)((ncells + 1 + T - 1) / T), T, 0, st>>>(b.key_sorted, n, ncells, b.cstart);
    launches += 1;
    // primary list
    if (ranges) {
        k_iota_ranges<<<grid_of(n, T), T, 0, st>>>(ranges->start, ranges->len, ranges->out, ranges->n, n, b.plist);
        launches += 1;
    } else if (subset) {
        k_prim_compact<<<nprim_tiles, kPrimTile, 0, st>>>(b.orig, n, n_primary, prim_count, b.plist);
        launches += 1;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        fprintf(stderr, "g3pcf index: %s\n", cudaGetErrorString(e));
        return -1;
    }
    return launches;
}

}  // namespace g3
