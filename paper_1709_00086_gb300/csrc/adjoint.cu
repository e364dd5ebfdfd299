// Adjoint of zeta with respect to the weights and positions (not in the
// paper; the derivative of its Sec. 3.1 estimator with the pair set and
// radial bins held fixed).
//
// With G_m = dL/dzeta_m / 2 (the caller passes dL/d(Re zeta, Im zeta)),
// M_m = G_m + G_m^H and A_i the primary's multipoles,
//      V_i = M_m A_i                    (k_vgemm, per m block, FP32; k_vgemm_df
//                                        in double-float for the double-float
//                                        pair pass)
//      dL/dw_i (as a primary) = Re(A_i^H V_i)   (FP32: fused into k_vgemm;
//                                        double-float: in k_adj_df)
//      H_i = w_i V_i                    (applied by the adjoint pair pass)
// (per catalog c of a batched forward, M is built from that catalog's dL/dzeta_c)
// and the pair pass (k_adj over the pair lists, or the fused k_pair mode 1)
// adds, for every pair (i, j) in bin b,
// 2 Re(conj(H_i,b) . Y(rhat_ij)) to dL/dw_j and the gradient of the same
// quantity with respect to the separation to dL/dpos_j and -dL/dpos_i.
// In the real form of an A row ([Re | Im] halves for m >= 1) M acts as
// [[Re M, -Im M], [Im M, Re M]]; for m = 0 only Re M enters because a_l0
// and Y_l0 are real.
#include "internal.h"

namespace g3 {

namespace {

constexpr int kRows = 8;         // primaries per CTA in k_vgemm and k_vgemm_df
constexpr int kVThreads = 256;

struct MInfo {
    int K[kMaxL + 1];
    int W[kMaxL + 1];
    int col0[kMaxL + 1];   // first A column of block m
    int moff[kMaxL + 1];   // offset of block m in the M buffer (floats)
    long long zoff[kMaxL + 1];  // complex offset of block m in zeta
};

// an M entry of the double-float path: head + tail
__device__ __forceinline__ float2 m_entry(double v) {
    const float h = (float)v;
    return make_float2(h, (float)(v - (double)h));
}

__global__ void k_build_mreal(const double* dz, MInfo mi, int lmax, int64_t zsize, size_t mfloats,
                              float* Mr) {
    const int m = blockIdx.y, cat = blockIdx.z;
    if (m > lmax) return;
    const int K = mi.K[m], W = mi.W[m];
    const double* Z = dz + 2 * ((int64_t)cat * zsize + mi.zoff[m]);
    float* out = Mr + (size_t)cat * mfloats + mi.moff[m];
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < W * W; e += gridDim.x * blockDim.x) {
        const int rr = e / W, cc = e % W;
        const int r = rr % K, c = cc % K;
        // M = G + G^H, G = dz / 2
        const double re = 0.5 * (Z[2 * ((int64_t)r * K + c)] + Z[2 * ((int64_t)c * K + r)]);
        const double im = 0.5 * (Z[2 * ((int64_t)r * K + c) + 1] - Z[2 * ((int64_t)c * K + r) + 1]);
        double v;
        if (m == 0) {
            v = re;
        } else {
            const bool rlo = rr < K, clo = cc < K;
            v = (rlo == clo) ? re : (rlo ? -im : im);
        }
        out[e] = (float)v;
    }
}

// One CTA per block of up to kRows rows of one catalog: blk = {catalog, first
// row, rows}; the catalog picks its M.  Without a block table (blks null) block
// b covers rows row_lo + kRows b .. of catalog 0 below row_hi.  The row's
// primary-weight term is added to dw[row], or, for rows of a chunk of
// primaries (rorig non-null), to dw[rorig[rplist ? rplist[q0 + row] : q0 + row]].
// FP32 M, V and sums.
__global__ void __launch_bounds__(kVThreads) k_vgemm(const float* __restrict__ A, int RLP, int RL,
                                                     const int4* __restrict__ blks, int64_t row_lo,
                                                     int64_t row_hi, const float* __restrict__ Mall,
                                                     size_t mfloats, MInfo mi, int lmax, float* V,
                                                     double* dw, const int* rplist, const int* rorig,
                                                     int64_t q0) {
    extern __shared__ float sA[];  // kRows x RL
    __shared__ float red[kRows][kVThreads / 32];
    int4 blk;
    if (blks) {
        blk = blks[blockIdx.x];
    } else {
        const int64_t b0 = row_lo + (int64_t)blockIdx.x * kRows;
        blk = make_int4(0, (int)b0, (int)(row_hi - b0 < kRows ? row_hi - b0 : kRows), 0);
    }
    const float* __restrict__ Mr = Mall + (size_t)blk.x * mfloats;
    const int64_t r0 = blk.y;
    const int64_t rows = r0 + blk.z;
    for (int k = threadIdx.x; k < kRows * RL; k += kVThreads) {
        const int rr = k / RL, c = k % RL;
        sA[k] = (r0 + rr < rows) ? A[(r0 + rr) * RLP + c] : 0.f;
    }
    __syncthreads();
    float dwp[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) dwp[r] = 0.f;
    for (int col = threadIdx.x; col < RL; col += kVThreads) {
        int m = 0;
        while (m < lmax && col >= mi.col0[m + 1]) ++m;
        const int W = mi.W[m], c = col - mi.col0[m];
        const float* Mrow = Mr + mi.moff[m] + (int64_t)c * W;
        const float* As = sA + mi.col0[m];
        float acc[kRows];
#pragma unroll
        for (int r = 0; r < kRows; ++r) acc[r] = 0.f;
        for (int k = 0; k < W; ++k) {
            const float mv = __ldg(Mrow + k);
#pragma unroll
            for (int r = 0; r < kRows; ++r) acc[r] = fma(mv, As[r * RL + k], acc[r]);
        }
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            if (r0 + r < rows) V[(r0 + r) * RLP + col] = acc[r];
            dwp[r] = fma(sA[r * RL + col], acc[r], dwp[r]);
        }
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        float v = dwp[r];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) red[r][wid] = v;
    }
    __syncthreads();
    if (threadIdx.x < kRows && r0 + threadIdx.x < rows) {
        double s = 0.0;
        for (int k = 0; k < kVThreads / 32; ++k) s += (double)red[threadIdx.x][k];
        const int64_t row = r0 + threadIdx.x;
        int64_t idx = row;
        if (rorig) {
            const int64_t q = q0 + row;
            idx = rorig[rplist ? rplist[q] : q];
        }
        dw[idx] += s;  // the primary-weight term (dw starts at zero; pair terms add atomically)
    }
}

// M of one catalog for the double-float path, one CTA per order m and bin b1, one warp per
// row c of that bin: entries as head + tail, and for every bin b2 the largest row sum of |M|
// over the columns of b2 (norm[m][b1][b2]), which bounds the sums of k_vgemm_df.  The real
// form is symmetric, so that row c is also column c.  Lane = b2 + nbins x share: 32 / nbins
// lanes share a bin's columns.
constexpr int kBWarps = 16;
__global__ void __launch_bounds__(kBWarps * 32) k_build_m_df(const double* dz, MInfo mi, int nbins, int64_t zsize,
                                                            size_t mfloats, size_t nfloats, float2* Mr, float* norm) {
    __shared__ float s_max[kBWarps][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, cat = blockIdx.y;
    const int m = blockIdx.x / nbins, b1 = blockIdx.x - m * nbins;
    const int K = mi.K[m], W = mi.W[m], shares = 32 / nbins;
    const double* Z = dz + 2 * ((int64_t)cat * zsize + mi.zoff[m]);
    float most = 0.f;
    for (int rr = b1 + wid * nbins; rr < W; rr += kBWarps * nbins) {
        const int r = rr % K;
        float2* out = Mr + (size_t)cat * mfloats + mi.moff[m] + (int64_t)rr * W;
        float sum = 0.f;
        for (int cc = lane; lane < shares * nbins && cc < W; cc += shares * nbins) {
            const int c = cc % K;
            // M = G + G^H, G = dz / 2
            const double re = 0.5 * (Z[2 * ((int64_t)r * K + c)] + Z[2 * ((int64_t)c * K + r)]);
            const double im = 0.5 * (Z[2 * ((int64_t)r * K + c) + 1] - Z[2 * ((int64_t)c * K + r) + 1]);
            const bool rlo = rr < K, clo = cc < K;
            const float2 v = m_entry(m == 0 || rlo == clo ? re : (rlo ? -im : im));
            out[cc] = v;
            sum += fabsf(v.x);
        }
        float tot = sum;
        for (int sh = 1; sh < shares; ++sh) tot += __shfl_sync(0xffffffffu, sum, (lane + sh * nbins) & 31);
        most = fmaxf(most, tot);
    }
    s_max[wid][lane] = most;
    __syncthreads();
    if (wid == 0 && lane < nbins) {
        for (int w = 1; w < kBWarps; ++w) most = fmaxf(most, s_max[w][lane]);
        norm[cat * nfloats + blockIdx.x * nbins + lane] = most;
    }
}

__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
// V = M A in double-float (M head + tail, A exact), 8 rows of one catalog per CTA,
// one column per thread at a time, two rows per packed operation.  The head of
// every sum carries a bias of three times its bound, so that the difference to the next
// head is exact and one FMA returns the rounding error: 5 operations per multiply-add (10
// with an error-free addition).  The tail gathers half an ulp of the bias per term, about
// 2^-44 of the bound (rms, 140 terms), so the bound keeps apart what the gradient keeps
// apart: it is formed per row (neighbours of any size share a CTA), and per bin of the
// column as the sum over the bins b of M's largest row sum in b times the row's largest
// |A| there (bins that dL/dzeta leaves out count nothing).  Bound by issue; M (from L2) is read once per 8 rows,
// coalesced by its symmetry (16 rows per CTA: the same time).  20,000 rows at B =
// lmax = 10: 0.68 ms against 1.73 with error-free additions (0.65 with one bias per CTA
// and order); 80 registers and three CTAs per SM, as 64 and four take 0.82.
// The primary-weight term Re(A^H V) is the pair pass's (k_adj_df).
__global__ void __launch_bounds__(kVThreads, 3) k_vgemm_df(
    const float* __restrict__ A, int RLP, int RL, const int4* __restrict__ blks, int64_t row_lo, int64_t row_hi,
    const float2* __restrict__ Mall, const float* __restrict__ norm, size_t mfloats, MInfo mi, int nbins, int lmax,
    float2* V) {
    constexpr int R = kRows, RS = R + 4;  // rows, column stride in shared memory
    extern __shared__ __align__(16) float sA[];  // RL x RS
    const int nmb = (lmax + 1) * nbins;
    float* amax = sA + (size_t)RL * RS;  // [m][bin][row]: largest |A|
    float* bias = amax + nmb * R;        // [m][bin][row]
    int4 blk;
    if (blks) {
        blk = blks[blockIdx.x];
    } else {
        const int64_t b0 = row_lo + (int64_t)blockIdx.x * R;
        blk = make_int4(0, (int)b0, (int)(row_hi - b0 < R ? row_hi - b0 : R), 0);
    }
    const float2* __restrict__ Mr = Mall + (size_t)blk.x * mfloats;
    const float* __restrict__ nr = norm + (size_t)blk.x * (lmax + 1) * nbins * nbins;
    const int64_t r0 = blk.y;
    const int nrow = blk.z;
    for (int c = threadIdx.x; c < RL; c += kVThreads) {
#pragma unroll
        for (int rr = 0; rr < R; ++rr) sA[c * RS + rr] = rr < nrow ? __ldg(A + (r0 + rr) * RLP + c) : 0.f;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < nmb * R; k += kVThreads) {
        // (a block's columns: the bin varies fastest)
        const int rr = k % R, m = k / R / nbins, b = k / R - m * nbins, W = mi.W[m];
        float mx = 0.f;
        for (int c = b; c < W; c += nbins) mx = fmaxf(mx, fabsf(sA[(mi.col0[m] + c) * RS + rr]));
        amax[k] = mx;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < nmb * R; k += kVThreads) {
        const int rr = k % R, mb = k / R, m = mb / nbins;
        float s = 0.f;
        for (int b = 0; b < nbins; ++b) s = fmaf(__ldg(nr + mb * nbins + b), amax[(m * nbins + b) * R + rr], s);
        bias[k] = 3.f * s;
    }
    __syncthreads();
    for (int col = threadIdx.x; col < RL; col += kVThreads) {
        int m = 0;
        while (m < lmax && col >= mi.col0[m + 1]) ++m;
        const int W = mi.W[m], c = col - mi.col0[m];
        const float2* Mc = Mr + mi.moff[m] + c;
        const float4* As = reinterpret_cast<const float4*>(sA + mi.col0[m] * RS);
        const float4* bs = reinterpret_cast<const float4*>(bias + (m * nbins + c % nbins) * R);
        float2 H[R / 2], Lo[R / 2];
#pragma unroll
        for (int r = 0; r < R / 4; ++r) {
            const float4 b4 = bs[r];
            H[2 * r] = make_float2(b4.x, b4.y);
            H[2 * r + 1] = make_float2(b4.z, b4.w);
            Lo[2 * r] = Lo[2 * r + 1] = dup(0.f);
        }
#pragma unroll 8
        for (int k = 0; k < W; ++k) {
            const float2 mv = __ldg(Mc + (int64_t)k * W);
            const float2 Mh = dup(mv.x), Ml = dup(mv.y);
#pragma unroll
            for (int r = 0; r < R / 4; ++r) {
                const float4 a4 = As[k * (RS / 4) + r];
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const float2 x = half ? make_float2(a4.z, a4.w) : make_float2(a4.x, a4.y);
                    float2& h = H[2 * r + half];
                    float2& l = Lo[2 * r + half];
                    const float2 s = __ffma2_rn(Mh, x, h);
                    const float2 e = __ffma2_rn(Mh, x, __fadd2_rn(h, neg2(s)));
                    l = __ffma2_rn(Ml, x, __fadd2_rn(l, e));
                    h = s;
                }
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float hb = __fsub_rn(r & 1 ? H[r / 2].y : H[r / 2].x, reinterpret_cast<const float*>(bs)[r]);  // exact
            const float lb = r & 1 ? Lo[r / 2].y : Lo[r / 2].x;
            // renormalised
            const float h = __fadd_rn(hb, lb), bb = __fsub_rn(h, hb);
            const float l = __fadd_rn(__fsub_rn(hb, __fsub_rn(h, bb)), __fsub_rn(lb, bb));
            if (r < nrow) V[(r0 + r) * RLP + col] = make_float2(h, l);
        }
    }
}

MInfo make_info(int nbins, int lmax) {
    MInfo mi{};
    int col = 0, moff = 0;
    long long z = 0;
    for (int m = 0; m <= lmax; ++m) {
        const int K = nbins * (lmax + 1 - m);
        const int W = m == 0 ? K : 2 * K;
        mi.K[m] = K;
        mi.W[m] = W;
        mi.col0[m] = col;
        mi.moff[m] = moff;
        mi.zoff[m] = z;
        col += W;
        moff += W * W;
        z += (long long)K * K;
    }
    return mi;
}

}  // namespace

size_t adjoint_m_floats(int nbins, int lmax) {
    size_t s = 0;
    for (int m = 0; m <= lmax; ++m) {
        const size_t K = (size_t)nbins * (lmax + 1 - m);
        const size_t W = m == 0 ? K : 2 * K;
        s += W * W;
    }
    return s;
}

size_t adjoint_norm_floats(int nbins, int lmax) { return (size_t)(lmax + 1) * nbins * nbins; }

int adjoint_rows_per_block() { return kRows; }

int launch_adjoint_m(const double* dzeta, int nbins, int lmax, int ncat, int64_t zsize, float* Mr,
                     cudaStream_t st) {
    const MInfo mi = make_info(nbins, lmax);
    dim3 g1(64, lmax + 1, ncat);
    k_build_mreal<<<g1, 256, 0, st>>>(dzeta, mi, lmax, zsize, adjoint_m_floats(nbins, lmax), Mr);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_adjoint_m_df(const double* dzeta, int nbins, int lmax, int ncat, int64_t zsize, float2* Mr, float* norm,
                        cudaStream_t st) {
    const MInfo mi = make_info(nbins, lmax);
    dim3 grid((lmax + 1) * nbins, ncat);
    k_build_m_df<<<grid, kBWarps * 32, 0, st>>>(dzeta, mi, nbins, zsize, adjoint_m_floats(nbins, lmax),
                                                adjoint_norm_floats(nbins, lmax), Mr, norm);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_adjoint_prep(const double* dzeta, int nbins, int lmax, int ncat, int64_t zsize, const float* A,
                        int RLP, int RL, const int4* blks, int nblks, float* Mr, float* V, double* dw,
                        cudaStream_t st) {
    if (launch_adjoint_m(dzeta, nbins, lmax, ncat, zsize, Mr, st) != 0) return -1;
    if (nblks > 0) {
        const MInfo mi = make_info(nbins, lmax);
        const size_t smem = sizeof(float) * kRows * RL;
        if (cudaFuncSetAttribute(k_vgemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
            cudaSuccess)
            return -1;
        k_vgemm<<<(unsigned)nblks, kVThreads, smem, st>>>(A, RLP, RL, blks, 0, 0, Mr,
                                                                 adjoint_m_floats(nbins, lmax), mi, lmax, V, dw,
                                                                 nullptr, nullptr, 0);
    }
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_vgemm_rows(const float* A, int RLP, int RL, int64_t row_lo, int64_t row_hi, const float* Mr,
                      int nbins, int lmax, float* V, double* dw, const int* plist, const int* orig,
                      int64_t q0, cudaStream_t st) {
    if (row_hi <= row_lo) return 0;
    const MInfo mi = make_info(nbins, lmax);
    const size_t smem = sizeof(float) * kRows * RL;
    if (cudaFuncSetAttribute(k_vgemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return -1;
    const int64_t nb = (row_hi - row_lo + kRows - 1) / kRows;
    k_vgemm<<<(unsigned)nb, kVThreads, smem, st>>>(A, RLP, RL, nullptr, row_lo, row_hi, Mr,
                                                          adjoint_m_floats(nbins, lmax), mi, lmax, V, dw, plist, orig,
                                                          q0);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

namespace {
int vgemm_df(const float* A, int RLP, int RL, const int4* blks, int64_t nb, int64_t row_lo, int64_t row_hi,
             const float2* Mr, const float* norm, int nbins, int lmax, float2* V, cudaStream_t st) {
    const MInfo mi = make_info(nbins, lmax);
    const size_t smem = sizeof(float) * ((kRows + 4) * (size_t)RL + 2 * (size_t)(lmax + 1) * nbins * kRows);
    if (cudaFuncSetAttribute(k_vgemm_df, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return -1;
    k_vgemm_df<<<(unsigned)nb, kVThreads, smem, st>>>(A, RLP, RL, blks, row_lo, row_hi, Mr, norm,
                                                      adjoint_m_floats(nbins, lmax), mi, nbins, lmax, V);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}
}  // namespace

int launch_vgemm_blocks_df(const float* A, int RLP, int RL, const int4* blks, int nblks, const float2* Mr,
                           const float* norm, int nbins, int lmax, float2* V, cudaStream_t st) {
    if (nblks <= 0) return 0;
    return vgemm_df(A, RLP, RL, blks, nblks, 0, 0, Mr, norm, nbins, lmax, V, st);
}

int launch_vgemm_rows_df(const float* A, int RLP, int RL, int64_t row_lo, int64_t row_hi, const float2* Mr,
                         const float* norm, int nbins, int lmax, float2* V, cudaStream_t st) {
    const int64_t rows = row_hi - row_lo;
    if (rows <= 0) return 0;
    return vgemm_df(A, RLP, RL, nullptr, (rows + kRows - 1) / kRows, row_lo, row_hi, Mr, norm, nbins, lmax, V, st);
}

}  // namespace g3
