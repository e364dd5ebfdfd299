// zeta contraction, plain-FP32 form, and the FP64 reduction to zeta.
//
// Paper: Sec. 3.1 -- about one primary the coefficient is a_lm(r1) a*_l'm(r2),
// "repeated for all primaries"; Sec. 3.2/3.3 -- per-thread partial multipoles
// are combined at the end and reduced across nodes.  Here the sum over
// primaries is a per-m Gram matrix over the A rows,
//      C_m = sum_i w_i v_i v_i^T,   v_i = [Re a_m(i) | Im a_m(i)]  (m >= 1),
// from which zeta_m = (C_XX + C_YY) + i (C_YX - C_XY) (and zeta_0 = C_XX).
// Only upper tiles of the symmetric C_m are formed.  Every (segment of
// primaries, tile) pair is one CTA writing its own partial (FP64), and the
// reduction adds the segments of a catalog in a fixed order, so reruns give
// bit-identical zeta.
#include "internal.h"

namespace g3 {

namespace {

// One warp per 32 x 32 tile and range of primaries, four warps (row ranges) per
// CTA; a lane holds 8 x 4 entries of the tile.  Bound by issue: per primary and
// warp 16 packed FMAs (two issue cycles each) and about 20 other instructions.
// 32-wide tiles leave 1.5 entries computed per entry of the triangle (64-wide
// ones 2.1 at B = lmax = 10).  Runs of kFlushRows primaries are summed in FP32 (2^-24 per
// addition, which sets the error), the runs in double-float (head + tail, 2^-48 per
// addition; the warps' sums and the partials' reduction in FP64): FP64 additions, at 1/58
// of the FP32 rate, would take a third of the kernel's time.  20,000 primaries, B = lmax = 10:
// 0.20 ms (10 row parts, 1,220 CTAs) against 1.29 ms for 64-wide tiles with 4 x 4 scalar
// FMAs per thread, whose 129 CTAs left most SMs one block of 8,192 rows.
constexpr int kT = 32;           // tile edge
constexpr int kKC = 8;           // rows per shared-memory stage
constexpr int kCWarps = 4;
constexpr int kThreads = kCWarps * 32;
constexpr int kFlushRows = 256;  // FP32 run length
static_assert(kFlushRows % kKC == 0, "a run is whole stages");

struct ContractSmem {
    float a[kKC][kT];            // weighted rows, left side
    float b[kKC][kT];
    float2 tot[32][32];          // [entry of a lane][lane]: sum of the finished runs
};

__device__ __forceinline__ float2 neg2(float2 x) { return make_float2(-x.x, -x.y); }
// (h, l) += v for two sums at once: error-free addition to the head, its rounding
// error into the tail
__device__ __forceinline__ void run_add(float2& h, float2& l, float2 v) {
    const float2 s = __fadd2_rn(h, v);
    const float2 bb = __fadd2_rn(s, neg2(h));
    const float2 e = __fadd2_rn(__fadd2_rn(h, neg2(__fadd2_rn(s, neg2(bb)))), __fadd2_rn(v, neg2(bb)));
    l = __fadd2_rn(l, e);
    h = s;
}

__global__ void __launch_bounds__(kThreads, 4) k_contract_fp32(const float* __restrict__ A, int RLP,
                                                               const float* __restrict__ wrow,
                                                               const Tile* tiles, const Segment* segs,
                                                               double* partials, int part_stride) {
    extern __shared__ __align__(16) unsigned char cs_raw[];
    ContractSmem* sm = reinterpret_cast<ContractSmem*>(cs_raw);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    ContractSmem& S = sm[wid];
    const Tile t = tiles[blockIdx.x];
    const Segment sg = segs[blockIdx.y];
    // lane: rows 8 ty .. + 7 and columns 4 tx .. + 3 of the tile
    const int tx = lane & 7, ty = lane >> 3;
    // this warp's runs of the segment
    const int nruns = (sg.row1 - sg.row0 + kFlushRows - 1) / kFlushRows;
    const int first = sg.row0 + wid * nruns / kCWarps * kFlushRows;
    const int last = min(sg.row1, sg.row0 + (wid + 1) * nruns / kCWarps * kFlushRows);
    const bool va = lane < t.rows, vb = lane < t.cols, diag = t.r0 == t.c0;
    const float* pa = A + (int64_t)first * RLP + t.col0 + t.r0 + (va ? lane : 0);
    const float* pb = A + (int64_t)first * RLP + t.col0 + t.c0 + (vb ? lane : 0);
#pragma unroll
    for (int e = 0; e < 32; ++e) S.tot[e][lane] = make_float2(0.f, 0.f);
    // acc[j][i]: rows 8 ty + 2 i, + 1 (the packed pair) of column 4 tx + j
    float2 acc[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[j][i] = make_float2(0.f, 0.f);
    float ra[kKC], rb[kKC], rw[kKC];
    auto fetch = [&](int r0) {
#pragma unroll
        for (int k = 0; k < kKC; ++k) {
            const bool in = r0 + k < last;
            rw[k] = in ? __ldg(wrow + r0 + k) : 0.f;
            ra[k] = in && va ? __ldg(pa) : 0.f;
            rb[k] = diag ? ra[k] : (in && vb ? __ldg(pb) : 0.f);
            pa += RLP;
            pb += RLP;
        }
    };
    if (first < last) fetch(first);
    for (int r0 = first; r0 < last; r0 += kKC) {
        __syncwarp();
#pragma unroll
        for (int k = 0; k < kKC; ++k) {
            S.a[k][lane] = ra[k] * rw[k];
            S.b[k][lane] = rb[k];
        }
        __syncwarp();
        if (r0 + kKC < last) fetch(r0 + kKC);
#pragma unroll
        for (int k = 0; k < kKC; ++k) {
            const float4 a0 = *reinterpret_cast<const float4*>(&S.a[k][8 * ty]);
            const float4 a1 = *reinterpret_cast<const float4*>(&S.a[k][8 * ty + 4]);
            const float4 b4 = *reinterpret_cast<const float4*>(&S.b[k][4 * tx]);
            const float2 av[4] = {make_float2(a0.x, a0.y), make_float2(a0.z, a0.w), make_float2(a1.x, a1.y),
                                  make_float2(a1.z, a1.w)};
            const float bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[j][i] = __ffma2_rn(av[i], make_float2(bv[j], bv[j]), acc[j][i]);
        }
        if ((r0 + kKC - sg.row0) % kFlushRows == 0 || r0 + kKC >= last) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float2* to = &S.tot[2 * (4 * j + i)][lane];
                    float2 x = to[0], y = to[32];  // (head, tail) of the pair's two entries
                    float2 h = make_float2(x.x, y.x), l = make_float2(x.y, y.y);
                    run_add(h, l, acc[j][i]);
                    to[0] = make_float2(h.x, l.x);
                    to[32] = make_float2(h.y, l.y);
                    acc[j][i] = make_float2(0.f, 0.f);
                }
        }
    }
    // the four warps' sums, in warp order: warp w takes the lanes' entries 8 w .. + 7
    __syncthreads();
    double* out = partials + (int64_t)blockIdx.y * part_stride + t.out_off;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int e = 8 * wid + q;  // = 2 (4 j + i) + part
        float h = 0.f, l = 0.f;
#pragma unroll
        for (int w = 0; w < kCWarps; ++w) {
            const float2 v = sm[w].tot[e][lane];
            const float s = __fadd_rn(h, v.x), bb = __fsub_rn(s, h);
            const float er = __fadd_rn(__fsub_rn(h, __fsub_rn(s, bb)), __fsub_rn(v.x, bb));
            l = __fadd_rn(l, __fadd_rn(v.y, er));
            h = s;
        }
        const int j = e >> 3, i = (e >> 1) & 3, part = e & 1;
        out[(8 * ty + 2 * i + part) * kT + 4 * tx + j] = (double)h + (double)l;
    }
}

struct BlockInfo {
    int tile_base[kMaxL + 1];
    int ntile[kMaxL + 1];
    int width[kMaxL + 1];
    int zoff[kMaxL + 1];  // complex offset of block m inside one catalog's zeta
};

__device__ __forceinline__ double c_lookup(const double* part, const Tile* tiles,
                                           const BlockInfo& bi, int m, int a, int b, int T,
                                           int colmajor) {
    if (a > b) {
        const int t = a;
        a = b;
        b = t;
    }
    const int ti = a / T, tj = b / T, nt = bi.ntile[m];
    const int idx = bi.tile_base[m] + ti * nt - ti * (ti - 1) / 2 + (tj - ti);
    const Tile& tl = tiles[idx];
    return colmajor ? part[tl.out_off + (b - tl.c0) * T + (a - tl.r0)]
                    : part[tl.out_off + (a - tl.r0) * T + (b - tl.c0)];
}

__global__ void k_reduce(const double* partials, int part_stride, const int* seg_first, int ncat,
                         const Tile* tiles, BlockInfo bi, int nbins, int lmax, int T, int cm,
                         int64_t zsize, double* zeta, const unsigned long long* counts, int64_t* counts_out) {
    const int cat = blockIdx.y;
    if (counts_out && blockIdx.x == 0 && threadIdx.x < nbins && cat < ncat)
        counts_out[cat * nbins + threadIdx.x] = (int64_t)counts[cat * nbins + threadIdx.x];
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= zsize || cat >= ncat) return;
    int m = 0;
    while (m < lmax && e >= bi.zoff[m + 1]) ++m;
    const int K = nbins * (lmax + 1 - m);
    const int64_t loc = e - bi.zoff[m];
    const int r = (int)(loc / K), c = (int)(loc % K);
    double re = 0.0, im = 0.0;
    for (int s = seg_first[cat]; s < seg_first[cat + 1]; ++s) {
        const double* p = partials + (int64_t)s * part_stride;
        if (m == 0) {
            re += c_lookup(p, tiles, bi, 0, r, c, T, cm);
        } else {
            re += c_lookup(p, tiles, bi, m, r, c, T, cm) + c_lookup(p, tiles, bi, m, K + r, K + c, T, cm);
            im += c_lookup(p, tiles, bi, m, K + r, c, T, cm) - c_lookup(p, tiles, bi, m, r, K + c, T, cm);
        }
    }
    double* z = zeta + 2 * ((int64_t)cat * zsize + e);
    z[0] = re;
    z[1] = im;
}

// Isotropic 3PCF from zeta: out[c][l][b1][b2] = Re zeta^0_ll(b1,b2)
// + 2 sum_{m=1}^{l} Re zeta^m_ll(b1,b2) (the m < 0 blocks folded in by
// zeta^{-m} = conj(zeta^m) for real weights).
__global__ void k_isotropic(const double* zeta, BlockInfo bi, int nbins, int lmax, int64_t zsize,
                            int ncat, double* out) {
    const int64_t per_cat = (int64_t)(lmax + 1) * nbins * nbins;
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= per_cat * ncat) return;
    const int cat = (int)(e / per_cat);
    const int64_t r = e - cat * per_cat;
    const int l = (int)(r / ((int64_t)nbins * nbins));
    const int b1 = (int)((r / nbins) % nbins), b2 = (int)(r % nbins);
    const double* z = zeta + 2 * (int64_t)cat * zsize;
    double acc = 0.0;
    for (int m = 0; m <= l; ++m) {
        const int K = nbins * (lmax + 1 - m);
        const int64_t idx = bi.zoff[m] + (int64_t)((l - m) * nbins + b1) * K + (l - m) * nbins + b2;
        acc += (m == 0 ? 1.0 : 2.0) * z[2 * idx];
    }
    out[e] = acc;
}

// out[e] = sum_c coef[c] zeta_c[e] over the 2 zsize doubles of a zeta block,
// catalogs in index order (fixed summation order: reruns are bit-identical).
__global__ void k_combine(const double* zeta, int64_t n2, int ncat, CombineCoef cf, double* out) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n2; e += (int64_t)gridDim.x * blockDim.x) {
        double acc = 0.0;
        for (int c = 0; c < ncat; ++c) acc = fma(cf.c[c], zeta[(int64_t)c * n2 + e], acc);
        out[e] = acc;
    }
}

}  // namespace

int launch_combine(const double* zeta, int64_t zsize, int ncat, const double* coef, double* out, cudaStream_t st) {
    if (ncat < 1 || ncat > kMaxCombine) return -1;
    CombineCoef cf{};
    for (int c = 0; c < ncat; ++c) cf.c[c] = coef[c];
    const int64_t n2 = 2 * zsize;
    int64_t blocks = (n2 + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) blocks = 1;
    k_combine<<<(unsigned)blocks, 256, 0, st>>>(zeta, n2, ncat, cf, out);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int contract_tile_dim_fp32() { return kT; }

// Rows per segment when the base segments (of `seg` rows) alone leave the chip
// idle: about three CTAs per slot (4 per SM), whole runs for every warp.
int64_t contract_fp32_split(int64_t seg, int64_t nbase, int ntiles, int nsm) {
    const int64_t step = (int64_t)kCWarps * kFlushRows;
    const int64_t have = nbase * ntiles, want = (int64_t)nsm * 4 * 3;
    if (have <= 0 || have >= want) return seg;
    const int64_t parts = (want + have - 1) / have;
    const int64_t rows = ((seg + parts - 1) / parts + step - 1) / step * step;
    return rows < seg ? rows : seg;
}

// Tiles of edge T over the upper triangle of every C_m (row-major in (ti, tj)).
int make_tiles(int nbins, int lmax, int T, Tile* out, int max_tiles) {
    return fill_tiles(nbins, lmax, T, out, max_tiles);
}

int launch_contract_fp32(const float* A, int RLP, const float* wrow, const Tile* tiles, int ntiles,
                         const Segment* segs, int nsegs, double* partials, int part_stride,
                         cudaStream_t st) {
    if (ntiles <= 0 || nsegs <= 0) return 0;
    const size_t smem = sizeof(ContractSmem) * kCWarps;
    if (cudaFuncSetAttribute(k_contract_fp32, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return -1;
    dim3 grid(ntiles, nsegs);
    k_contract_fp32<<<grid, kThreads, smem, st>>>(A, RLP, wrow, tiles, segs, partials, part_stride);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_reduce(const double* partials, int part_stride, const int* seg_first, int ncat,
                  int nbins, int lmax, const Tile* tiles, int T, double* zeta, cudaStream_t st,
                  int colmajor, const unsigned long long* counts, int64_t* counts_out) {
    BlockInfo bi;
    int base = 0;
    int64_t zo = 0;
    for (int m = 0; m <= lmax; ++m) {
        const int K = nbins * (lmax + 1 - m);
        const int W = (m == 0) ? K : 2 * K;
        const int nt = (W + T - 1) / T;
        bi.tile_base[m] = base;
        bi.ntile[m] = nt;
        bi.width[m] = W;
        bi.zoff[m] = (int)zo;
        base += nt * (nt + 1) / 2;
        zo += (int64_t)K * K;
    }
    const int64_t zsize = zo;
    dim3 grid((unsigned)((zsize + 255) / 256), ncat);
    k_reduce<<<grid, 256, 0, st>>>(partials, part_stride, seg_first, ncat, tiles, bi, nbins, lmax,
                                   T, colmajor, zsize, zeta, counts, counts_out);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_isotropic(const double* zeta, int nbins, int lmax, int ncat, double* out, cudaStream_t st) {
    BlockInfo bi{};
    int64_t zo = 0;
    for (int m = 0; m <= lmax; ++m) {
        const int64_t K = (int64_t)nbins * (lmax + 1 - m);
        bi.zoff[m] = (int)zo;
        zo += K * K;
    }
    const int64_t total = (int64_t)(lmax + 1) * nbins * nbins * ncat;
    if (total == 0) return 0;
    k_isotropic<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(zeta, bi, nbins, lmax, zo, ncat, out);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace g3
