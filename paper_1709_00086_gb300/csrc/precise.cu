// Pair-stage kernels for multipoles that are differentiated: the forward
// multipoles a_lm of Sec. 3.1 and the adjoint pair pass, both in double-float
// arithmetic (an FP32 head plus an FP32 tail: about 44 significant bits per operation; the
// biased sums below are good to 2^-38 - 2^-45 of their largest terms) over the same
// per-bin pair lists as the FP32 kernels of pairlist.cu.
//
// Why: in the Chebyshev form Y_lm = K_lm sum_k c_k T_k(z) (x + iy)^m the
// connection coefficients c_k are non-negative and large where D_lm(1) is much
// larger than D_lm(z) in the bulk, so any per-pair rounding of the terms
// T_k (x + iy)^m (and of the unit vector they come from) reaches the gradient
// amplified by up to two orders of magnitude.  FP32 evaluation leaves the
// gradient near 1e-6 of its largest component at lmax = 10; carrying every
// per-pair quantity and every sum in double-float, and the conversions in
// FP64, brings it to the 1e-8 level, at a fraction of the cost of FP64, which
// runs at 1/58 of the FP32 rate on this part.
//
//   k_accum_df -- per primary (one warp).  Per chunk of 32 list entries each
//                 lane evaluates one pair: the separation from the primary's
//                 image (FP32 head + tail of the FP64 image, so the difference
//                 is exact), r^2, 1/r by one Newton step from rsqrt, the unit
//                 vector, T_k(z) and w (x + iy)^m, all in double-float.  The m = 0
//                 sums stay with the lane; the rest goes through a shared-memory
//                 record to the lanes that own the sums of each m >= 1 (two k of
//                 one m per lane, several pairs of the chunk side by side where the
//                 sums fit in part of the warp), added with biased heads
//                 (bias_fma).  At the end of a bin the Chebyshev ->
//                 Legendre-form connection (times K_lm, head + tail
//                 coefficients) is applied in double-float; the row of A is
//                 stored at the primary's end.  No FP64 arithmetic (but for the rare
//                 close pair): the FP64 pipe runs at 1/58 of the FP32 rate.  Bound by
//                 issue, with shared memory (records in and out) close behind.  100,000
//                 clustered points, lmax = 6 (7.1e8 pairs): 24.9 ms, against 40 ms with
//                 12 instead of 6 operations per term and one sum pair per lane
//                 (twice the shared-memory bytes per term); 23.5 ms with a fixed bias,
//                 biased m = 0 sums and inexact chunk sums.  Sums in the
//                 registers of the pair's lane alone (no records, a
//                 reduction of every sum per bin) took 23 ms there, but three
//                 times this kernel's time at 55 pairs per bin and lmax = 10.
//   k_adj_df   -- per primary (one warp), one pair per lane: the adjoint
//                 coefficients G_{m,k} = w_i sum_l c^(m)_{l-m,k} K_lm V_lm of
//                 the primary (double-float, from the double-float V = M A,
//                 in shared memory with a bound of each bin's sums), the
//                 primary's weight term Re(A^H V), and per pair
//                 F = sum Re(conj(G) T_k (x + iy)^m) with its gradient in
//                 double-float: per m the sums against T_k and T_k' on (Re, Im)
//                 pairs with biased heads, then their products with
//                 (x + iy)^(m-1), whose partial sums as m descends are the x
//                 and y derivatives.  Their tails gather residues of half an ulp of
//                 a head near three times the bin's coefficient norm: a few 2^-44 of the
//                 norm, where the coefficients themselves carry 2^-25 of theirs from the
//                 FP32 rows of A.  Rounded once to FP32 per pair; FP64
//                 atomics for the secondary, a double-float sum for the
//                 primary; its weight term in FP64.  Bound by issue.  100,000
//                 clustered points, lmax = 6: 36.4 ms against 57 with error-free
//                 additions and an FP32 pair per derivative.
// Resident CTAs (registers), 20,000 uniform points, ms at 3 / 4 / 5 / 6 CTAs per SM:
// k_accum_df 0.77 / 0.71 / 0.69 / 0.65 at lmax = 6 and six the best below, 0.80 / 0.74 /
// 0.73 / 0.72 at 7, 1.08 / 0.99 / 1.00 / 0.99 at 8, 1.20 / 1.16 / 1.19 / 1.23 at 10; k_adj_df
// 0.67 / 0.67 / 0.64 / 0.65 at lmax = 4, 0.89 / 0.82 / 0.77 / 0.80 at 5, 1.04 / 0.96 / 0.98 /
// 1.00 at 6, 1.46 / 1.43 / 1.53 / 1.57 at 8, 2.14 / 2.13 / 2.14 / 2.23 at 10.
#include "pair_common.cuh"

namespace g3 {
namespace {

constexpr int kDWarps = 4;
constexpr int kDThreads = kDWarps * 32;
constexpr unsigned kNoPairD = 0xffffffffu;

// ---- double-float arithmetic (error-free transformations) ----------------
// Every operation uses the _rn intrinsics so that the compiler never fuses a
// product into a later addition: the error terms below rely on each rounding.
struct df {
    float h, l;
};

__device__ __forceinline__ df two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}
// |a| >= |b| (or a == 0)
__device__ __forceinline__ df fast_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ df df_add(df a, df b) {
    const df s = two_sum(a.h, b.h);
    return fast_two_sum(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ df df_neg(df a) { return {-a.h, -a.l}; }
__device__ __forceinline__ df df_mul(df a, df b) {
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, e));
    return fast_two_sum(p, e);
}
// product left unnormalised (head, tail with |tail| <~ ulp(head)): for sums
__device__ __forceinline__ df df_mul_u(df a, df b) {
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, e));
    return {p, e};
}
__device__ __forceinline__ df df_mulf(df a, float b) {
    const float p = __fmul_rn(a.h, b);
    float e = __fmaf_rn(a.h, b, -p);
    e = __fmaf_rn(a.l, b, e);
    return fast_two_sum(p, e);
}
// acc += t (t unnormalised): the head's rounding error goes to the tail
__device__ __forceinline__ void df_acc(df& acc, df t) {
    const df s = two_sum(acc.h, t.h);
    acc.l = __fadd_rn(acc.l, __fadd_rn(s.l, t.l));
    acc.h = s.h;
}
__device__ __forceinline__ df df_from(double v) {
    const float h = (float)v;
    return {h, (float)(v - (double)h)};
}
__device__ __forceinline__ double df_to(df a) { return (double)a.h + (double)a.l; }

// (a + ib)(c + id) in double-float
__device__ __forceinline__ void df_cmul(df a, df b, df c, df d, df& re, df& im) {
    re = df_add(df_mul_u(a, c), df_neg(df_mul_u(b, d)));
    im = df_add(df_mul_u(a, d), df_mul_u(b, c));
}

// One coordinate of the separation q - (head + tail): exact up to the tail's
// own rounding (|tail| <= half an ulp of the image), renormalised.
__device__ __forceinline__ df sep(float qh, float ql, float h, float t) {
    const df s = two_sum(qh, -h);
    return two_sum(s.h, __fadd_rn(s.l, __fsub_rn(ql, t)));
}

// Unit vector and 1/r of the separation d (double-float), optionally rotated
// by R (radial line of sight).
__device__ __forceinline__ void unit_df(df dx, df dy, df dz, const df* R, bool radial, df& ux, df& uy, df& uz,
                                        df& rinv) {
    if (radial) {
        const df rx = df_add(df_add(df_mul(R[0], dx), df_mul(R[1], dy)), df_mul(R[2], dz));
        const df ry = df_add(df_add(df_mul(R[3], dx), df_mul(R[4], dy)), df_mul(R[5], dz));
        const df rz = df_add(df_add(df_mul(R[6], dx), df_mul(R[7], dy)), df_mul(R[8], dz));
        dx = rx;
        dy = ry;
        dz = rz;
    }
    const df r2 = df_add(df_add(df_mul(dx, dx), df_mul(dy, dy)), df_mul(dz, dz));
    // y0 ~ r2^(-1/2) (a few ulps); y = y0 + y0 (1 - r2 y0^2) / 2 (Newton), with the
    // residual formed in double-float so that y carries ~44 bits
    const float y0 = rsqrtf(r2.h);
    const float q0 = __fmul_rn(y0, y0);
    const df y2 = {q0, __fmaf_rn(y0, y0, -q0)};
    const df t = df_mul(r2, y2);
    const df e = df_add({1.f, 0.f}, df_neg(t));
    rinv = fast_two_sum(y0, __fmul_rn(__fmul_rn(y0, 0.5f), e.h));
    ux = df_mul(dx, rinv);
    uy = df_mul(dy, rinv);
    uz = df_mul(dz, rinv);
}

// Primary image `code` (position minus the code's box shift, FP64 input used
// when given) as head + tail in shared memory: img[code] head, img[27 + code] tail.
// FP32 input: the position is exact and the shift s (box_h + box_l) is added in
// double-float; FP64 input: formed in FP64.
__device__ __forceinline__ void image_df(float4* img, int code, const float4& P0, const double* pts64, int p,
                                         double boxd, df box) {
    const int sx = code % 3 - 1, sy = (code / 3) % 3 - 1, sz = code / 9 - 1;
    if (!pts64) {
        auto shifted = [&](float v, int sh) {
            return sh == 0 ? df{v, 0.f} : df_add({v, 0.f}, {-(float)sh * box.h, -(float)sh * box.l});
        };
        const df x = shifted(P0.x, sx), y = shifted(P0.y, sy), z = shifted(P0.z, sz);
        img[code] = make_float4(x.h, y.h, z.h, 0.f);
        img[27 + code] = make_float4(x.l, y.l, z.l, 0.f);
        return;
    }
    double x = pts64[3 * (int64_t)p], y = pts64[3 * (int64_t)p + 1], z = pts64[3 * (int64_t)p + 2];
    x -= sx * boxd;
    y -= sy * boxd;
    z -= sz * boxd;
    const float hx = (float)x, hy = (float)y, hz = (float)z;
    img[code] = make_float4(hx, hy, hz, 0.f);
    img[27 + code] = make_float4((float)(x - hx), (float)(y - hy), (float)(z - hz), 0.f);
}

// A secondary's position as head + tail (exact for FP32 input).
__device__ __forceinline__ void load_sec(const ListArgs& a, unsigned e, float4& qv, float3& ql) {
    const unsigned j = e & kIdxMask;
    qv = __ldg(a.pts + j);
    ql = make_float3(0.f, 0.f, 0.f);
    if (a.pts64) {
        const double x = a.pts64[3 * (int64_t)j], y = a.pts64[3 * (int64_t)j + 1], z = a.pts64[3 * (int64_t)j + 2];
        qv.x = (float)x;
        qv.y = (float)y;
        qv.z = (float)z;
        ql = make_float3((float)(x - qv.x), (float)(y - qv.y), (float)(z - qv.z));
    }
}

// The separation of a close pair (close_r2) from the input positions, times the power of
// two `scale`: head and tail leave out the last five bits of FP64 positions, which is all
// of a separation of a few of their ulps.  INLINE: not by a call (k_accum_df, 80 registers
// at lmax = 6: 24.9 ms against 25.2; k_adj_df: 36.5 against 36.4).
template <bool INLINE>
__device__ __forceinline__ void close_df(const ListArgs& a, int p, unsigned e, bool close, df& dx, df& dy, df& dz,
                                         float& scale) {
    scale = 1.f;
    if (close && __fmaf_rn(dx.h, dx.h, __fmaf_rn(dy.h, dy.h, __fmul_rn(dz.h, dz.h))) <= close_r2(a.bins, a.pts64)) {
        double s[4];
        close_sep<INLINE>(a.pts, a.pts64, p, e, a.g.boxd, s);
        dx = df_from(s[0]);
        dy = df_from(s[1]);
        dz = df_from(s[2]);
        scale = (float)s[3];
    }
}

// ---- forward ----------------------------------------------------------------
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
// Biased accumulators.  Two sums at a time (.x and .y), each a head H that carries
// a bias, so that it stays more than twice as large as any term, and a tail: in
// s = fl(H + T C) the difference H - s is then exact (Sterbenz), and one more FMA
// returns what the rounding left.  (H, Lo) += T C with T = (Th, Tl), C = (Ch, Cl)
// takes 6 packed operations instead of the 12 of an error-free addition to a head
// of unknown size.
__device__ __forceinline__ void bias_fma(float2& H, float2& Lo, float2 Th, float2 Tl, float2 Ch, float2 Cl) {
    const float2 s = __ffma2_rn(Th, Ch, H);
    const float2 e = __ffma2_rn(Th, Ch, __fadd2_rn(H, neg2(s)));
    Lo = __ffma2_rn(Th, Cl, __ffma2_rn(Tl, Ch, __fadd2_rn(Lo, e)));
    H = s;
}
// (H, Lo) += T c for a head without a bias (an error-free addition, 11 operations)
__device__ __forceinline__ void df_fma2(float2& H, float2& Lo, float2 Th, float2 Tl, float2 c) {
    const float2 p = __fmul2_rn(Th, c);
    const float2 pe = __ffma2_rn(Th, c, neg2(p));
    const float2 s = __fadd2_rn(H, p), bb = __fadd2_rn(s, neg2(H));
    const float2 er = __fadd2_rn(__fadd2_rn(H, neg2(__fadd2_rn(s, neg2(bb)))), __fadd2_rn(p, neg2(bb)));
    Lo = __ffma2_rn(Tl, c, __fadd2_rn(Lo, __fadd2_rn(er, pe)));
    H = s;
}
// (H, Lo) += C
__device__ __forceinline__ void bias_add(float2& H, float2& Lo, float2 Ch, float2 Cl) {
    const float2 s = __fadd2_rn(H, Ch);
    const float2 e = __fadd2_rn(__fadd2_rn(H, neg2(s)), Ch);
    Lo = __fadd2_rn(Lo, __fadd2_rn(e, Cl));
    H = s;
}

// Forward sums.  The m = 0 sums (reals) stay in the registers of the lane that
// evaluates the pair and are reduced over the warp once per bin.  For m >= 1 the pair goes
// to a record in shared memory,
//   C_m, m = 1..L:      Re.h, Im.h, Re.l, Im.l  of w (x + iy)^m
//   T_k, k = 0..L:      h, l                     (KE values)
// and every lane owns two sums (k0, k0 + 1; k0 even) of one m: one 128-bit load
// gives both T, one the C (LDS returns 128 bytes per cycle whatever is broadcast, so
// bytes per sum count: 16 here, 32 with one sum per lane).  LPG lanes hold all sums;
// where they fit in a half, quarter ... of the warp, G groups share the chunk's pairs.
template <int L>
struct DfRec {
    __host__ __device__ static constexpr int lanes() {
        int n = 0;
        for (int m = 1; m <= L; ++m) n += (L - m + 2) / 2;
        return n;
    }
    __host__ __device__ static constexpr int groups() {
        int g = 1;
        while (g < 16 && lanes() * g * 2 <= 32) g *= 2;
        return g;
    }
    static constexpr int N = lanes();
    static constexpr int G = groups();
    static constexpr int LPG = 32 / G;
    static constexpr int KE = (L + 1) & ~1;
    static constexpr int TB = 4 * L;
    // record stride (floats), an odd number of 16-byte units: conflict-free stores
    static constexpr int RS = ((4 * L + 2 * KE) / 4 % 2) ? 4 * L + 2 * KE : 4 * L + 2 * KE + 4;
    static constexpr int M0 = (L + 2) / 2;  // packed pairs of m = 0
};

__host__ __device__ constexpr size_t accum_df_smem_per_warp(int RL, int RS, int NRP) {
    return (size_t)32 * RS * 4 + 54 * 16 + 9 * 8 + 8 + (size_t)NRP * 8 + (size_t)((RL + 3) & ~3) * 4;
}

template <int L>
__global__ void __launch_bounds__(kDThreads, L <= 6 ? 6 : (L == 7 ? 5 : 4)) k_accum_df(ListArgs a) {
    using R_ = DfRec<L>;
    constexpr int RS = R_::RS, G = R_::G, M0 = R_::M0, KE = R_::KE;
    constexpr int NR = Shape<L>::NR, NRP = Shape<L>::NRP;
    constexpr int kSteps = 32 / G, U = kSteps < 4 ? kSteps : 4;
    extern __shared__ __align__(16) unsigned char draw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned char* base = draw + (size_t)wid * accum_df_smem_per_warp(a.RL, RS, NRP);
    float* rec = reinterpret_cast<float*>(base);                              // [32][RS]
    float4* img = reinterpret_cast<float4*>(base + 32 * RS * 4);              // [54]
    df* Rd = reinterpret_cast<df*>(base + 32 * RS * 4 + 54 * 16);             // [9]
    float2* res = reinterpret_cast<float2*>(base + 32 * RS * 4 + 54 * 16 + 80);  // [NRP] one bin's sums
    float* rowbuf = reinterpret_cast<float*>(base + 32 * RS * 4 + 54 * 16 + 80 + NRP * 8);  // [RL]
    // this lane's order m and first k
    const int grp = lane / R_::LPG;
    int m = 0, k0 = 0;
    {
        int idx = lane % R_::LPG;
        if (idx < R_::N) {
            m = 1;
            while (idx >= (L - m + 2) / 2) {
                idx -= (L - m + 2) / 2;
                ++m;
            }
            k0 = 2 * idx;
        }
    }
    const int offC = m > 0 ? 4 * (m - 1) : 0, offT = R_::TB + 2 * k0;
    const Grid& g = a.g;
    const df boxdf = df_from(g.boxd);  // the box side as head + tail
    const int close_end = close_bins(a.bins, a.pts64);
    const bool radial = g.radial != 0;
    const int qa = a.qrange ? a.qrange[0] : a.qa, qb = a.qrange ? a.qrange[1] : a.qb;
    for (;;) {
        int q = 0;
        if (lane == 0) q = qa + atomicAdd(a.queue, 1);
        q = __shfl_sync(kFull, q, 0);
        if (q >= qb) break;
        const int p = a.plist ? a.plist[q] : q;
        const float4 P0 = a.pts[p];
        if (lane < 27) image_df(img, lane, P0, a.pts64, p, g.boxd, boxdf);
        if (lane < 9) {
            if (radial) {
                double x0 = P0.x, x1 = P0.y, x2 = P0.z;
                if (a.pts64) {
                    x0 = a.pts64[3 * (int64_t)p];
                    x1 = a.pts64[3 * (int64_t)p + 1];
                    x2 = a.pts64[3 * (int64_t)p + 2];
                }
                Rd[lane] = df_from(los_rotation_entry_d(lane, x0, x1, x2, g.boxd));
            } else {
                Rd[lane] = {(lane % 4 == 0) ? 1.f : 0.f, 0.f};
            }
        }
        for (int k = lane; k < a.RL; k += 32) rowbuf[k] = 0.f;
        for (int k = lane; k < NR; k += 32) res[k] = make_float2(0.f, 0.f);
        const int cb = a.base[q] < 0 ? 0 : a.base[q];
        const int nch = a.nchunks[q];
        const int* chunks = a.chunks + (int64_t)cb * 32;
        const int* ordp = a.ord + cb;
        __syncwarp();
        // m = 0: packed (k, k + 1), error-free additions (one per chunk and lane); m >= 1: this
        // lane's sums k0 and k0 + 1 as (Re, Im), biased by 2 + the chunk's terms (each of size
        // <= 1) in Ha .. Lb, and added to SaH .. SbL after every chunk.  The residues that the
        // tail gathers are half an ulp of a head near the bias, so that the bias sets the
        // rounding: emulated with random terms, 2^-45 of the largest |w| (rms) after 4 terms,
        // 2^-42 after 16, 2^-40 after 32, 2^-38 after 200 (error-free heads: 2^-49, 2^-45,
        // 2^-44, 2^-42), where the stored row is rounded to 2^-25 of the entry.
        float2 H0[M0], L0[M0], SaH, SaL, SbH, SbL;
        auto clear = [&]() {
            static_for<0, M0>([&](auto ic) {
                H0[decltype(ic)::value] = L0[decltype(ic)::value] = dup(0.f);
            });
            SaH = SaL = SbH = SbL = dup(0.f);
        };
        clear();
        auto fold1 = [&](float2& SH, float2& SL, float2 H, float2 Lo, float bias) {
            // H = bias + x + xe (a head near 2 has a finer grid than x near -bias)
            const float2 x = __fadd2_rn(H, dup(-bias));
            const float2 xe = __fadd2_rn(H, neg2(__fadd2_rn(x, dup(bias))));
            const float2 s = __fadd2_rn(SH, x), bb = __fadd2_rn(s, neg2(SH));
            const float2 er = __fadd2_rn(__fadd2_rn(SH, neg2(__fadd2_rn(s, neg2(bb)))), __fadd2_rn(x, neg2(bb)));
            SL = __fadd2_rn(SL, __fadd2_rn(__fadd2_rn(er, xe), Lo));
            SH = s;
        };
        // |w| <= cap (a power of two fixed by the first weights of a bin; a larger one
        // flushes the sums): the sums take w / cap
        unsigned cap = 0u;
        bool held = false;  // the sums hold a chunk of this cap
        float inv = 1.f, scale = 1.f;
        // the sums, times cap, into res
        auto flush = [&]() {
            if (m > 0 || G > 1) {
                float h[4] = {SaH.x, SaH.y, SbH.x, SbH.y};
                float l[4] = {SaL.x, SaL.y, SbL.x, SbL.y};
#pragma unroll
                for (int o = 16; o >= R_::LPG; o >>= 1)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float gh = __shfl_xor_sync(kFull, h[i], o), gl = __shfl_xor_sync(kFull, l[i], o);
                        const df t = two_sum(h[i], gh);
                        h[i] = t.h;
                        l[i] = __fadd_rn(__fadd_rn(l[i], gl), t.l);
                    }
                if (m > 0 && grp == 0) {
                    const int s0 = acc_base(L, m) + 2 * k0, n = k0 + 1 <= L - m ? 4 : 2;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (i < n) {
                            const float2 o = res[s0 + i];
                            const df v = df_add({o.x, o.y}, fast_two_sum(h[i] * scale, l[i] * scale));
                            res[s0 + i] = make_float2(v.h, v.l);
                        }
                }
            }
            // m = 0 over the warp by recursive halving
            float h[L + 1], l[L + 1];
            static_for<0, L + 1>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                h[k] = (k & 1) ? H0[k / 2].y : H0[k / 2].x;
                l[k] = (k & 1) ? L0[k / 2].y : L0[k / 2].x;
            });
            int b0 = 0, size = L + 1;
            static_for<0, 5>([&](auto rc) {
                constexpr int r = decltype(rc)::value;
                constexpr int S = bf_size(L + 1, r);
                constexpr int hf = (S + 1) / 2;
                constexpr int o = 16 >> r;
                const bool hi = (lane & o) != 0;
                static_for<0, hf>([&](auto ic) {
                    constexpr int i = decltype(ic)::value;
                    float uh = 0.f, ul = 0.f;
                    if constexpr (i + hf < S) {
                        uh = h[i + hf];
                        ul = l[i + hf];
                    }
                    const float kh = hi ? uh : h[i], kl = hi ? ul : l[i];
                    const float gh = __shfl_xor_sync(kFull, hi ? h[i] : uh, o);
                    const float gl = __shfl_xor_sync(kFull, hi ? l[i] : ul, o);
                    const df t = two_sum(kh, gh);
                    h[i] = t.h;
                    l[i] = __fadd_rn(__fadd_rn(kl, gl), t.l);
                });
                if (hi) {
                    b0 += hf;
                    size -= hf;
                } else {
                    size = size < hf ? size : hf;
                }
            });
            if (size > 0) {  // one slot per lane after five halvings of at most 11
                const float2 o = res[b0];
                const df v = df_add({o.x, o.y}, fast_two_sum(h[0] * scale, l[0] * scale));
                res[b0] = make_float2(v.h, v.l);
            }
            clear();
            held = false;
        };
        // list words three chunks ahead, entries two, points one
        auto word = [&](int i) { return (unsigned)__ldg(ordp + (i < nch ? i : nch - 1)); };
        auto entry = [&](unsigned o) { return (unsigned)__ldg(chunks + (int64_t)(o & 0x3ffffffu) * 32 + lane); };
        unsigned e = kNoPairD, en = kNoPairD, o0 = 0u, o1 = 0u, o2 = 0u;
        float4 qv = make_float4(0.f, 0.f, 0.f, 0.f);
        float3 ql = make_float3(0.f, 0.f, 0.f);
        if (nch > 0) {
            o0 = word(0);
            o1 = word(1);
            o2 = word(2);
            e = entry(o0);
            en = entry(o1);
            if (e != kNoPairD) load_sec(a, e, qv, ql);
        }
        for (int i = 0; i < nch; ++i) {
            float4 qn = make_float4(0.f, 0.f, 0.f, 0.f);
            float3 ln = make_float3(0.f, 0.f, 0.f);
            if (en != kNoPairD) load_sec(a, en, qn, ln);
            const unsigned en2 = entry(o2), o3 = word(i + 3);
            const bool v = e != kNoPairD;
            const unsigned wm = __reduce_max_sync(kFull, v ? __float_as_uint(fabsf(qv.w)) : 0u);
            const int nv = __popc(__ballot_sync(kFull, v));  // the chunk's pairs, its first lanes
            if (wm > cap) {
                if (held) flush();
                const unsigned ex = min((wm >> 23) + 1u, 253u);
                cap = ex << 23;
                scale = __uint_as_float(cap);
                inv = __uint_as_float((254u - ex) << 23);
            }
            held = true;
            {
                // this lane's pair -> its record; a padding lane takes a unit separation
                // and weight 0
                const int code = (int)min(e >> kIdxBits, 26u);
                const float4 hh = img[code], tt = img[27 + code];
                df dx = sep(qv.x, ql.x, hh.x, tt.x), dy = sep(qv.y, ql.y, hh.y, tt.y),
                   dz = sep(qv.z, ql.z, hh.z, tt.z);
                float scale1;
                if (v) {
                    close_df<true>(a, p, e, (int)(o0 >> 26) < close_end, dx, dy, dz, scale1);
                } else {
                    dx = {1.f, 0.f};
                    dy = dz = {0.f, 0.f};
                }
                df ux, uy, uz, rinv;
                unit_df(dx, dy, dz, Rd, radial, ux, uy, uz, rinv);
                const float w = v ? qv.w * inv : 0.f;
                float4* my = reinterpret_cast<float4*>(rec + lane * RS);
                df T[2 * M0];
                T[0] = {1.f, 0.f};
                T[1] = uz;
                const df z2 = {2.f * uz.h, 2.f * uz.l};
                static_for<2, 2 * M0>([&](auto kc) {
                    constexpr int k = decltype(kc)::value;
                    if constexpr (k <= L)
                        T[k] = df_add(df_mul(z2, T[k - 1]), df_neg(T[k - 2]));
                    else
                        T[k] = {0.f, 0.f};
                });
                static_for<0, M0>([&](auto ic) {
                    constexpr int k = 2 * decltype(ic)::value;
                    df_fma2(H0[k / 2], L0[k / 2], make_float2(T[k].h, T[k + 1].h), make_float2(T[k].l, T[k + 1].l),
                            dup(w));
                    if constexpr (k < KE) my[(R_::TB + 2 * k) / 4] = make_float4(T[k].h, T[k].l, T[k + 1].h, T[k + 1].l);
                });
                if constexpr (L >= 1) {
                    df cr = df_mulf(ux, w), ci = df_mulf(uy, w);
                    static_for<1, L + 1>([&](auto mc) {
                        constexpr int mm = decltype(mc)::value;
                        my[mm - 1] = make_float4(cr.h, ci.h, cr.l, ci.l);
                        if constexpr (mm < L) {
                            df nr, ni;
                            df_cmul(cr, ci, ux, uy, nr, ni);
                            cr = nr;
                            ci = ni;
                        }
                    });
                }
            }
            if constexpr (L >= 1) {
                __syncwarp();
                // the chunk's pairs into this lane's two sums, G pairs per step (the
                // records past the last pair hold weight 0)
                const float* rt = rec + grp * RS;
                const int steps = (nv + G - 1) / G;
                const float bias = (float)(steps + 2);
                float2 Ha = dup(bias), Hb = Ha, La = dup(0.f), Lb = La;
                for (int t = 0; t < steps; t += U, rt += U * G * RS) {
                    float4 T4[U], C4[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        C4[u] = *reinterpret_cast<const float4*>(rt + u * G * RS + offC);
                        T4[u] = *reinterpret_cast<const float4*>(rt + u * G * RS + offT);
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const float2 Ch = make_float2(C4[u].x, C4[u].y), Cl = make_float2(C4[u].z, C4[u].w);
                        bias_fma(Ha, La, dup(T4[u].x), dup(T4[u].y), Ch, Cl);
                        bias_fma(Hb, Lb, dup(T4[u].z), dup(T4[u].w), Ch, Cl);
                    }
                }
                fold1(SaH, SaL, Ha, La, bias);
                fold1(SbH, SbL, Hb, Lb, bias);
                __syncwarp();
            }
            if (i + 1 == nch || (o0 ^ o1) >> 26) {  // the bin's last chunk: its columns of the row
                flush();
                cap = 0u;
                __syncwarp();
                const int b = (int)(o0 >> 26);
                for (int sl = lane; sl < NR; sl += 32) {
                    const int col = __ldg(&a.slotconv[sl].x) + b;
                    const int4 cv = __ldg(a.colconv + col);
                    const float2* cf = a.colcoefdf + cv.w;
                    const float2* rs = res + (cv.x - b * NRP);
                    df v2 = {0.f, 0.f};
                    for (int k = 0; k < cv.z; ++k) {
                        const float2 c = __ldg(cf + k), r = rs[cv.y * k];
                        v2 = df_add(v2, df_mul({c.x, c.y}, {r.x, r.y}));
                    }
                    rowbuf[col] = __fadd_rn(v2.h, v2.l);
                }
                __syncwarp();
                for (int k = lane; k < NR; k += 32) res[k] = make_float2(0.f, 0.f);
                __syncwarp();
            }
            e = en;
            qv = qn;
            ql = ln;
            en = en2;
            o0 = o1;
            o1 = o2;
            o2 = o3;
        }
        __syncwarp();
        const int row = a.chunked ? q - a.q0 : a.orig[p];
        float* Arow = a.A + (int64_t)row * a.RLP;
        for (int col = lane; col < a.RL; col += 32) Arow[col] = rowbuf[col];
        if (lane == 0) a.wrow[row] = P0.w;
        __syncwarp();
    }
}

// ---- adjoint ----------------------------------------------------------------
// Coefficients of one bin in shared memory (floats): for m >= 1 the pair (m, k) as
// Re.h, Im.h, Re.l, Im.l at 4 (cidx(m) + k), so that one broadcast load gives both
// operands of a packed operation; then G_{0,k} as h, l.
template <int L>
struct AdjG {
    static constexpr int NC = L * (L + 1) / 2;
    static constexpr int Z = 4 * NC;
    static constexpr int N = (Z + 2 * (L + 1) + 3) & ~3;  // floats per bin
    __host__ __device__ static constexpr int cidx(int m) { return (m - 1) * (L + 1) - (m - 1) * m / 2; }
};
__host__ __device__ constexpr size_t adj_df_smem_per_warp(int B, int N) {
    return (size_t)B * N * 4 + 54 * 16 + (size_t)((B + 1) & ~1) * 8;
}
// the value of a biased sum as head (exact) and tail
__device__ __forceinline__ float2 unbias(float2 H, float b) { return __fadd2_rn(H, dup(-b)); }

// f2d_exact without a branch: subnormal inputs give zero (V has no tail there).
__device__ __forceinline__ double f2d_sel(float x) {
    const unsigned u = __float_as_uint(x), e = u & 0x7f800000u;
    unsigned hi = ((u >> 3) & 0x0fffffffu) + ((1023u - 127u) << 20);
    hi = e == 0x7f800000u ? hi | 0x7ff00000u : (e == 0u ? 0u : hi);
    return __hiloint2double((int)(hi | (u & 0x80000000u)), e == 0u ? 0 : (int)(u << 29));
}

template <int L>
__global__ void __launch_bounds__(kDThreads, L <= 5 ? 5 : 4) k_adj_df(ListArgs a) {
    constexpr int NR = Shape<L>::NR;
    using G_ = AdjG<L>;
    extern __shared__ __align__(16) unsigned char draw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int B = a.bins.nbins;
    unsigned char* base = draw + (size_t)wid * adj_df_smem_per_warp(B, G_::N);
    float* G = reinterpret_cast<float*>(base);                                  // [B][N]
    float4* img = reinterpret_cast<float4*>(base + (size_t)B * G_::N * 4);      // [54]
    float2* bias = reinterpret_cast<float2*>(base + (size_t)B * G_::N * 4 + 54 * 16);  // [B]
    const Grid& g = a.g;
    const df boxdf = df_from(g.boxd);  // the box side as head + tail
    const int close_end = close_bins(a.bins, a.pts64);
    const int qa = a.qrange ? a.qrange[0] : a.qa, qb = a.qrange ? a.qrange[1] : a.qb;
    for (;;) {
        int q = 0;
        if (lane == 0) q = qa + atomicAdd(a.queue, 1);
        q = __shfl_sync(kFull, q, 0);
        if (q >= qb) break;
        const int p = a.plist ? a.plist[q] : q;
        const float4 P0 = a.pts[p];
        if (lane < 27) image_df(img, lane, P0, a.pts64, p, g.boxd, boxdf);
        const int row = a.orig[p];
        const float2* Vrow = a.Vdf + (int64_t)(a.chunked ? q - a.q0 : row) * a.RLP;
        for (int b = 0; b < B; ++b) {
            // this bin's coefficients, and bounds of its sums: s1 over |G|, s2 over
            // k^2 |G| (|T_k| <= 1, |T_k'| <= k^2)
            float s1 = 0.f, s2 = 0.f;
            for (int sl = lane; sl < NR; sl += 32) {
                int m = 0, k = sl, part = 0;
                if (sl > L) {
                    int r = sl - (L + 1);
                    m = 1;
                    while (r >= 2 * (L + 1 - m)) {
                        r -= 2 * (L + 1 - m);
                        ++m;
                    }
                    k = r >> 1;
                    part = r & 1;
                }
                const int4 cv = __ldg(a.slotconv + sl);
                df v = {0.f, 0.f};
                for (int t = 0; t < cv.z; ++t) {
                    const float2 c = __ldg(a.slotcoefdf + cv.w + t), x = Vrow[cv.x + b + t * cv.y];
                    v = df_add(v, df_mul({c.x, c.y}, {x.x, x.y}));
                }
                const df gv = df_mulf(v, P0.w);
                float* Gb = G + b * G_::N;
                if (m == 0) {
                    Gb[G_::Z + 2 * k] = gv.h;
                    Gb[G_::Z + 2 * k + 1] = gv.l;
                } else {
                    Gb[4 * (G_::cidx(m) + k) + part] = gv.h;
                    Gb[4 * (G_::cidx(m) + k) + 2 + part] = gv.l;
                }
                s1 += fabsf(gv.h);
                s2 = fmaf((float)(k * k), fabsf(gv.h), s2);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                s1 += __shfl_xor_sync(kFull, s1, o);
                s2 += __shfl_xor_sync(kFull, s2, o);
            }
            // biases: three times the bound keeps every head above twice any term
            if (lane == 0) bias[b] = make_float2(3.f * s1, 3.f * s2);
        }
        // the primary's own weight term of dL/dw: Re(A^H V), the heads of V in FP64 and their
        // tails (at most 2^-24 of them, and known to about 2^-20 of themselves) in FP32
        {
            const float* Arow = a.A + (int64_t)(a.chunked ? q - a.q0 : row) * a.RLP;
            double t = 0.0;
            float tail = 0.f;
            for (int c0 = lane; c0 < a.RL; c0 += 32 * 4) {
                float2 v[4];
                float x[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {  // (loads of four columns in flight)
                    const bool in = c0 + 32 * u < a.RL;
                    v[u] = in ? Vrow[c0 + 32 * u] : make_float2(0.f, 0.f);
                    x[u] = in ? __ldg(Arow + c0 + 32 * u) : 0.f;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    t = fma(f2d_sel(x[u]), f2d_sel(v[u].x), t);
                    tail = fmaf(v[u].y, x[u], tail);
                }
            }
            t += (double)tail;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(kFull, t, o);
            if (lane == 0) atomicAdd(a.dw + row, t);
        }
        const int cb = a.base[q] < 0 ? 0 : a.base[q];
        const int nch = a.nchunks[q];
        const int* chunks = a.chunks + (int64_t)cb * 32;
        const int* ordp = a.ord + cb;
        __syncwarp();
        df pix = {0.f, 0.f}, piy = {0.f, 0.f}, piz = {0.f, 0.f};  // the primary's share (this lane)
        // list words three chunks ahead, entries two, points one
        auto word = [&](int i) { return (unsigned)__ldg(ordp + (i < nch ? i : nch - 1)); };
        auto entry = [&](unsigned o) { return (unsigned)__ldg(chunks + (int64_t)(o & 0x3ffffffu) * 32 + lane); };
        unsigned e = kNoPairD, en = kNoPairD, o0 = 0u, o1 = 0u, o2 = 0u;
        float4 qv = make_float4(0.f, 0.f, 0.f, 0.f);
        float3 ql = make_float3(0.f, 0.f, 0.f);
        if (nch > 0) {
            o0 = word(0);
            o1 = word(1);
            o2 = word(2);
            e = entry(o0);
            en = entry(o1);
            if (e != kNoPairD) load_sec(a, e, qv, ql);
        }
        for (int i = 0; i < nch; ++i) {
            float4 qn = make_float4(0.f, 0.f, 0.f, 0.f);
            float3 ln = make_float3(0.f, 0.f, 0.f);
            if (en != kNoPairD) load_sec(a, en, qn, ln);
            const unsigned en2 = entry(o2), o3 = word(i + 3);
            if (e != kNoPairD) {
                const int b = (int)(o0 >> 26);
                const float* Gb = G + b * G_::N;
                const float B1 = bias[b].x, B2 = bias[b].y, BF = (float)(L > 0 ? L : 1) * B1;
                const int jj = __ldg(a.orig + (e & kIdxMask));
                const int code = (int)(e >> kIdxBits);
                const float4 hh = img[code], tt = img[27 + code];
                df dx = sep(qv.x, ql.x, hh.x, tt.x), dy = sep(qv.y, ql.y, hh.y, tt.y),
                   dz = sep(qv.z, ql.z, hh.z, tt.z);
                float scale;
                close_df<false>(a, p, e, b < close_end, dx, dy, dz, scale);
                df ux, uy, z, rinv;  // (rinv: 1 / (scale r))
                unit_df(dx, dy, dz, nullptr, false, ux, uy, z, rinv);
                // T_k(z) and T_k'(z) = k U_{k-1}(z), heads and tails
                df T[L + 1], D[L + 1];
                T[0] = {1.f, 0.f};
                D[0] = {0.f, 0.f};
                if constexpr (L >= 1) {
                    T[1] = z;
                    D[1] = {1.f, 0.f};
                    const df z2 = {2.f * z.h, 2.f * z.l};
                    df u0 = {1.f, 0.f}, u1 = z2;  // U_0, U_1
                    static_for<2, L + 1>([&](auto kc) {
                        constexpr int k = decltype(kc)::value;
                        T[k] = df_add(df_mul(z2, T[k - 1]), df_neg(T[k - 2]));
                        D[k] = df_mulf(u1, (float)k);
                        if constexpr (k < L) {
                            const df u2 = df_add({2.f * T[k].h, 2.f * T[k].l}, u0);  // U_k = 2 T_k + U_{k-2}
                            u0 = u1;
                            u1 = u2;
                        }
                    });
                }
                // m = 0: (F, Fz) += G_k (T_k, T_k')
                float2 FH = make_float2(B1, B2), FL = dup(0.f);
                static_for<0, L + 1>([&](auto kc) {
                    constexpr int k = decltype(kc)::value;
                    const float2 gk = *reinterpret_cast<const float2*>(Gb + G_::Z + 2 * k);
                    bias_fma(FH, FL, dup(gk.x), dup(gk.y), make_float2(T[k].h, D[k].h), make_float2(T[k].l, D[k].l));
                });
                // powers of u = x + iy
                df pr[L + 1], pi[L + 1];
                pr[0] = {1.f, 0.f};
                pi[0] = {0.f, 0.f};
                if constexpr (L >= 2) {
                    pr[1] = ux;
                    pi[1] = uy;
                    static_for<2, L>([&](auto mc) {
                        constexpr int m = decltype(mc)::value;
                        df_cmul(pr[m - 1], pi[m - 1], ux, uy, pr[m], pi[m]);
                    });
                }
                // With g_m = sum_k G_{m,k} T_k, h_m likewise with T_k', as (Re, Im) pairs, and
                // p = u^{m-1}: conj(g_m) p = a_m - i b_m.  SA sums (a, b), SZ the same of h, and
                // SF the partial sums of SA as m descends, which is sum m (a_m, b_m); so
                //   F  = F_0 + SA.x x + SA.y y,  dF/dx = SF.x, dF/dy = SF.y,
                //   dF/dz = Fz_0 + SZ.x x + SZ.y y.
                float2 SAH = dup(B1), SAL = dup(0.f), SZH = dup(B2), SZL = dup(0.f), SFH = dup(BF), SFL = dup(0.f);
                static_for<0, L>([&](auto jc) {
                    constexpr int m = L - decltype(jc)::value;
                    float2 gH = dup(B1), gL = dup(0.f), hH = dup(B2), hL = dup(0.f);
                    static_for<0, L - m + 1>([&](auto kc) {
                        constexpr int k = decltype(kc)::value;
                        const float4 gg = *reinterpret_cast<const float4*>(Gb + 4 * (G_::cidx(m) + k));
                        const float2 Gh = make_float2(gg.x, gg.y), Gl = make_float2(gg.z, gg.w);
                        if constexpr (k == 0)
                            bias_add(gH, gL, Gh, Gl);
                        else
                            bias_fma(gH, gL, dup(T[k].h), dup(T[k].l), Gh, Gl);
                        if constexpr (k == 1)
                            bias_add(hH, hL, Gh, Gl);
                        else if constexpr (k > 1)
                            bias_fma(hH, hL, dup(D[k].h), dup(D[k].l), Gh, Gl);
                    });
                    const float2 gh = unbias(gH, B1), zh = unbias(hH, B2);
                    if constexpr (m == 1) {  // p = 1
                        bias_add(SAH, SAL, gh, gL);
                        bias_add(SZH, SZL, zh, hL);
                    } else {
                        const float2 prh = dup(pr[m - 1].h), prl = dup(pr[m - 1].l);
                        const float2 pih = dup(pi[m - 1].h), pil = dup(pi[m - 1].l);
                        bias_fma(SAH, SAL, prh, prl, gh, gL);
                        bias_fma(SAH, SAL, pih, pil, make_float2(gh.y, -gh.x), make_float2(gL.y, -gL.x));
                        if constexpr (L - m >= 1) {  // (h_L = 0)
                            bias_fma(SZH, SZL, prh, prl, zh, hL);
                            bias_fma(SZH, SZL, pih, pil, make_float2(zh.y, -zh.x), make_float2(hL.y, -hL.x));
                        }
                    }
                    bias_add(SFH, SFL, unbias(SAH, B1), SAL);
                });
                const float2 sa = unbias(SAH, B1), sz = unbias(SZH, B2), sf = unbias(SFH, BF);
                const df F0 = fast_two_sum(FH.x - B1, FL.x), Fz0 = fast_two_sum(FH.y - B2, FL.y);
                const df ax = {sa.x, SAL.x}, ay = {sa.y, SAL.y}, zx = {sz.x, SZL.x}, zy = {sz.y, SZL.y};
                const df F = df_add(F0, df_add(df_mul_u(ax, ux), df_mul_u(ay, uy)));
                const df Fz = df_add(Fz0, df_add(df_mul_u(zx, ux), df_mul_u(zy, uy)));
                const df Fx = two_sum(sf.x, SFL.x), Fy = two_sum(sf.y, SFL.y);
                // tangential gradient: (2 w_j / r) (grad F - (grad F . u) u), formed in
                // double-float and rounded once: a per-pair relative error of an FP32
                // ulp is not amplified by the sums over pairs
                const df gdr = df_add(df_add(df_mul(Fx, ux), df_mul(Fy, uy)), df_mul(Fz, z));
                const float tx = df_add(Fx, df_neg(df_mul(gdr, ux))).h;
                const float ty = df_add(Fy, df_neg(df_mul(gdr, uy))).h;
                const float tz = df_add(Fz, df_neg(df_mul(gdr, z))).h;
                const float sc = __fmul_rn(2.f * qv.w, scale * __fadd_rn(rinv.h, rinv.l));
                const float gx = __fmul_rn(sc, tx), gy = __fmul_rn(sc, ty), gz3 = __fmul_rn(sc, tz);
                atomicAdd(a.dw + jj, f2d_exact(__fmul_rn(2.f, __fadd_rn(F.h, F.l))));
                atomicAdd(a.dpos + 3 * (int64_t)jj, f2d_exact(gx));
                atomicAdd(a.dpos + 3 * (int64_t)jj + 1, f2d_exact(gy));
                atomicAdd(a.dpos + 3 * (int64_t)jj + 2, f2d_exact(gz3));
                df_acc(pix, {gx, 0.f});
                df_acc(piy, {gy, 0.f});
                df_acc(piz, {gz3, 0.f});
            }
            e = en;
            qv = qn;
            ql = ln;
            en = en2;
            o0 = o1;
            o1 = o2;
            o2 = o3;
        }
        double di0 = -df_to(pix), di1 = -df_to(piy), di2 = -df_to(piz);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            di0 += __shfl_xor_sync(kFull, di0, o);
            di1 += __shfl_xor_sync(kFull, di1, o);
            di2 += __shfl_xor_sync(kFull, di2, o);
        }
        if (lane == 0) {
            atomicAdd(a.dpos + 3 * (int64_t)row, di0);
            atomicAdd(a.dpos + 3 * (int64_t)row + 1, di1);
            atomicAdd(a.dpos + 3 * (int64_t)row + 2, di2);
        }
        __syncwarp();
    }
}

template <class K>
int launch_persistent(K kern, const ListArgs& a, size_t smem, int nsm, cudaStream_t st) {
    if (smem > 227 * 1024) return -1;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return -1;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kDThreads, smem) != cudaSuccess || per_sm < 1)
        return -1;
    int blocks = per_sm * nsm;
    const int need = (a.qb - a.qa + kDWarps - 1) / kDWarps;
    if (!a.qrange && blocks > need) blocks = need > 0 ? need : 1;
    kern<<<blocks, kDThreads, smem, st>>>(a);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <int L>
int launch_accum_df_t(const ListArgs& a, int nsm, cudaStream_t st) {
    return launch_persistent(k_accum_df<L>, a, accum_df_smem_per_warp(a.RL, DfRec<L>::RS, Shape<L>::NRP) * kDWarps,
                             nsm, st);
}
template <int L>
int launch_adj_df_t(const ListArgs& a, int nsm, cudaStream_t st) {
    return launch_persistent(k_adj_df<L>, a, adj_df_smem_per_warp(a.bins.nbins, AdjG<L>::N) * kDWarps, nsm, st);
}

}  // namespace

int launch_accum_df(int lmax, const ListArgs& a, int nsm, cudaStream_t st) {
    if (!a.qrange && a.qb <= a.qa) return 0;
    switch (lmax) {
        case 0: return launch_accum_df_t<0>(a, nsm, st);
        case 1: return launch_accum_df_t<1>(a, nsm, st);
        case 2: return launch_accum_df_t<2>(a, nsm, st);
        case 3: return launch_accum_df_t<3>(a, nsm, st);
        case 4: return launch_accum_df_t<4>(a, nsm, st);
        case 5: return launch_accum_df_t<5>(a, nsm, st);
        case 6: return launch_accum_df_t<6>(a, nsm, st);
        case 7: return launch_accum_df_t<7>(a, nsm, st);
        case 8: return launch_accum_df_t<8>(a, nsm, st);
        case 9: return launch_accum_df_t<9>(a, nsm, st);
        case 10: return launch_accum_df_t<10>(a, nsm, st);
        default: return -1;
    }
}

int launch_adj_df(int lmax, const ListArgs& a, int nsm, cudaStream_t st) {
    if (!a.qrange && a.qb <= a.qa) return 0;
    switch (lmax) {
        case 0: return launch_adj_df_t<0>(a, nsm, st);
        case 1: return launch_adj_df_t<1>(a, nsm, st);
        case 2: return launch_adj_df_t<2>(a, nsm, st);
        case 3: return launch_adj_df_t<3>(a, nsm, st);
        case 4: return launch_adj_df_t<4>(a, nsm, st);
        case 5: return launch_adj_df_t<5>(a, nsm, st);
        case 6: return launch_adj_df_t<6>(a, nsm, st);
        case 7: return launch_adj_df_t<7>(a, nsm, st);
        case 8: return launch_adj_df_t<8>(a, nsm, st);
        case 9: return launch_adj_df_t<9>(a, nsm, st);
        case 10: return launch_adj_df_t<10>(a, nsm, st);
        default: return -1;
    }
}

}  // namespace g3
