// Pair stage: neighbour gather, exact radial binning, line-of-sight rotation,
// spherical harmonics and the per-primary multipoles a_lm(i, b).
//
// Paper: Algorithm 1 (loop over primaries, neighbour search within rmax,
// separations, rotation, radial bin, multipole accumulation), Sec. 3.1
// (a_lm as a sum of Y_lm over the galaxies of a shell), Sec. 3.3.1
// (pre-binning: pairs of one primary are collected per radial bin into
// buckets and a full bucket is accumulated at once) and Sec. 3.3.2 (vectorise
// over pairs, keep per-lane partial sums and reduce them once).
//
// GB300 mapping.  One warp owns one primary at a time (primaries are pulled
// from a device work counter, the analogue of the paper's OpenMP dynamic
// schedule, Sec. 3.3).  Its lanes sweep the candidate secondaries of the
// sphere of radius rmax -- a few dozen contiguous slot ranges of the cell
// list -- 32 at a time, decide each pair's bin exactly, and append accepted
// pairs to one shared-memory bucket per bin (the paper's pre-binning).  When a
// bucket holds 32*kflush pairs, every lane takes kflush pairs of that bin,
// evaluates Y_lm with an FP32 recurrence and accumulates into (lmax+1)^2
// register partials; a 5-round butterfly then reduces the partials across
// the 32 lanes into the warp's shared-memory a_lm(b).  The arithmetic is
// FP32 on the FMA pipe; only the guard-band re-check of a bin edge and the
// separation of pairs within a few FP32 ulps of one another are FP64.
//
// Harmonics.  Y_lm(rhat) = K_lm Dt_lm(z) (x + i y)^m with rhat = (x, y, z),
// Dt_lm the monic polynomial of degree l-m proportional to the m-th
// derivative of the Legendre polynomial P_l, generated by
//      Dt_mm = 1, Dt_{m+1,m} = z,
//      Dt_{l+1,m} = z Dt_lm - (l^2 - m^2) / (4 l^2 - 1) Dt_{l-1,m},
// and K_lm = (-1)^m sqrt((2l+1)/(4 pi) (l-m)!/(l+m)!) (2l)! / (2^l l! (l-m)!)
// the normalisation (applied once per primary when the A row is written).
//
// Exact binning.  The FP32 r^2 of the candidate decides the bin unless it lies
// within a guard band (a bound on the FP32 error of r^2) around an edge; those
// rare pairs are re-decided in FP64 with the reference's exact operation order
// (d = x_j - x_i, minimum image, r2 = (dx*dx + dy*dy) + dz*dz, no FMA).
#include "pair_common.cuh"

#include <cstdio>

namespace g3 {

namespace {
// Per-warp shared-memory layout (bytes), identical on host and device.
struct WarpSmem {
    int cap;       // bucket capacity per bin (entries)
    int off_res;   // float res[nbins][NRP]
    int off_meta;  // int cnt[nbins], head[nbins], tot[nbins]
    int off_pcs;   // int4 pieces[kMaxPieces]
    int off_prim;  // float4 img[27] (primary position minus each image shift), float R[12],
                   // double pos64[4]
    int off_stash; // scan pipeline parked across a flush: float4 q[D][32], int j[D][32], code[D][32]
    int bytes;
};

__host__ __device__ inline WarpSmem warp_smem(int nrp, int nbins, int kflush) {
    WarpSmem s;
    s.cap = 32 * (kflush + kStashDepth);  // a bin can gain 32 per slot between flush checks
    int o = nbins * (s.cap + 1) * 4;
    o = (o + 15) & ~15;
    s.off_res = o;
    o += nbins * nrp * 4;
    s.off_meta = o;
    o += 3 * nbins * 4;
    o = (o + 15) & ~15;
    s.off_pcs = o;
    o += kMaxPieces * 16;
    s.off_prim = o;
    o += 27 * 16 + 12 * 4 + 4 * 8;
    o = (o + 15) & ~15;
    s.off_stash = o;
    o += kStashDepth * 32 * 24;
    s.bytes = (o + 127) & ~127;
    return s;
}

constexpr int kScanDepth = kStashDepth;

// Accumulate navail bucketed pairs of one bin (kflush per lane) and add the
// lane-reduced sums to res_b.  img[code] holds the primary's position minus
// the image shift of the entry's row, R the LOS rotation (radial mode).
// Entries are fetched three pairs ahead so that the gathers overlap the
// harmonic arithmetic.
template <int L>
__device__ __forceinline__ void flush_bin(const float4* __restrict__ pts, const int* bucket_b,
                                          int cap, int navail, int kflush, int head, float* res_b,
                                          const float4* img, const float* R, int radial, int lane,
                                          const PairArgs& a, int p, bool close) {
    constexpr int NR = Shape<L>::NR;
    float acc[NR];
    static_for<0, NR>([&](auto ic) { acc[decltype(ic)::value] = 0.f; });
#define G3_FETCH(t_, q_, e_)                              \
    do {                                                  \
        const int idx_ = (t_) * 32 + lane;                \
        e_ = 13u << kIdxBits;                             \
        q_ = make_float4(1.f, 0.f, 0.f, 0.f);             \
        if ((t_) < kflush && idx_ < navail) {             \
            int pos_ = head + idx_;                       \
            if (pos_ >= cap) pos_ -= cap;                 \
            e_ = (unsigned)bucket_b[pos_];                \
            q_ = __ldg(pts + (e_ & kIdxMask));            \
        }                                                 \
    } while (0)
    float4 q0, q1, q2;
    unsigned e0, e1, e2;
    G3_FETCH(0, q0, e0);
    G3_FETCH(1, q1, e1);
    G3_FETCH(2, q2, e2);
    for (int t = 0; t < kflush; ++t) {
        const float4 q = q0;
        const unsigned e = e0;
        q0 = q1;
        e0 = e1;
        q1 = q2;
        e1 = e2;
        G3_FETCH(t + 3, q2, e2);
        float w = 0.f, dx = 1.f, dy = 0.f, dz = 0.f;
        if (t * 32 + lane < navail) {
            const float4 o = img[e >> kIdxBits];
            dx = q.x - o.x;
            dy = q.y - o.y;
            dz = q.z - o.z;
            w = q.w;
            if (close && fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= close_r2(a.bins, a.pts64)) {
                double s[4];
                close_sep(pts, a.pts64, p, e, a.g.boxd, s);
                dx = (float)s[0];
                dy = (float)s[1];
                dz = (float)s[2];
            }
            if (radial) {
                const float rx = fmaf(R[0], dx, fmaf(R[1], dy, R[2] * dz));
                const float ry = fmaf(R[3], dx, fmaf(R[4], dy, R[5] * dz));
                const float rz = fmaf(R[6], dx, fmaf(R[7], dy, R[8] * dz));
                dx = rx;
                dy = ry;
                dz = rz;
            }
        }
        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        const float rinv = rsqrtf(r2);
        accum_pair<L>(acc, dz * rinv, dx * rinv, dy * rinv, w);
    }
    butterfly_add<L>(acc, lane, res_b);
#undef G3_FETCH
}

// Adjoint of one bucket of navail pairs of one bin.  With H the primary's
// adjoint multipoles for this bin (times K_lm, in the accumulator slot
// layout, broadcast from shared memory), F(d) = sum_lm Re(conj(H_lm)
// Dt_lm(z) (x + iy)^m) and
//      dL/dw_j += 2 F,   dL/dd = 2 w_j grad_d F,
//      dpos_j += dL/dd,  dpos_i -= dL/dd.
// grad_d F = (g - (g.rhat) rhat) / r with g the gradient of F in the
// (x, y, z) = rhat coordinates: dDt/dz by differentiating the recurrence,
// d(x+iy)^m/dx = m (x+iy)^(m-1), d/dy = i m (x+iy)^(m-1).
template <int L>
__device__ __forceinline__ void flush_grad(const float4* __restrict__ pts, const int* __restrict__ orig,
                                           const int* bucket_b, int cap, int navail, int kflush,
                                           int head, const float* Hb, const float4* img, int lane,
                                           double* dw, double* dpos, double (&dpi)[3], const PairArgs& a, int p,
                                           bool close) {
    float pix = 0.f, piy = 0.f, piz = 0.f;
#define G3_FETCH(t_, q_, e_)                              \
    do {                                                  \
        const int idx_ = (t_) * 32 + lane;                \
        e_ = 13u << kIdxBits;                             \
        q_ = make_float4(1.f, 0.f, 0.f, 0.f);             \
        if ((t_) < kflush && idx_ < navail) {             \
            int pos_ = head + idx_;                       \
            if (pos_ >= cap) pos_ -= cap;                 \
            e_ = (unsigned)bucket_b[pos_];                \
            q_ = __ldg(pts + (e_ & kIdxMask));            \
        }                                                 \
    } while (0)
    float4 q0, q1;
    unsigned e0, e1;
    G3_FETCH(0, q0, e0);
    G3_FETCH(1, q1, e1);
    for (int t = 0; t < kflush; ++t) {
        const float4 q = q0;
        const unsigned e = e0;
        q0 = q1;
        e0 = e1;
        G3_FETCH(t + 2, q1, e1);
        if (t * 32 + lane < navail) {
            const float4 o = img[e >> kIdxBits];
            float dx = q.x - o.x, dy = q.y - o.y, dz = q.z - o.z, sep = 1.f;
            const float wj = q.w;
            const int jj = __ldg(orig + (e & kIdxMask));
            if (close && fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= close_r2(a.bins, a.pts64)) {
                double s[4];
                close_sep(pts, a.pts64, p, e, a.g.boxd, s);
                dx = (float)s[0];
                dy = (float)s[1];
                dz = (float)s[2];
                sep = (float)s[3];
            }
            const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            const float rinv = rsqrtf(r2);  // sep / r
            const float z = dz * rinv, ux = dx * rinv, uy = dy * rinv;
            float F, Fz, Fx = 0.f, Fy = 0.f;
            {  // m = 0 (real)
                float A = Hb[0], Ap = 0.f;
                if constexpr (L >= 1) {
                    A = fmaf(Hb[1], z, A);
                    Ap = Hb[1];
                }
                float d0 = 1.f, d1 = z, p0 = 0.f, p1 = 1.f;
                static_for<2, L + 1>([&](auto lc) {
                    constexpr int l = decltype(lc)::value;
                    constexpr float bt = beta_lm(l - 1, 0);
                    const float d2 = fmaf(z, d1, -bt * d0);
                    const float p2 = fmaf(-bt, p0, fmaf(z, p1, d1));
                    A = fmaf(Hb[l], d2, A);
                    Ap = fmaf(Hb[l], p2, Ap);
                    d0 = d1;
                    d1 = d2;
                    p0 = p1;
                    p1 = p2;
                });
                F = A;
                Fz = Ap;
            }
            float ur = 1.f, ui = 0.f;  // (x + iy)^(m-1)
            static_for<1, L + 1>([&](auto mc) {
                constexpr int m = decltype(mc)::value;
                constexpr int b0 = acc_base(L, m);
                const float nr = fmaf(ur, ux, -ui * uy), ni = fmaf(ur, uy, ui * ux);  // (x+iy)^m
                float A = Hb[b0], Bv = Hb[b0 + 1], Ap = 0.f, Bp = 0.f;
                if constexpr (m + 1 <= L) {
                    A = fmaf(Hb[b0 + 2], z, A);
                    Bv = fmaf(Hb[b0 + 3], z, Bv);
                    Ap = Hb[b0 + 2];
                    Bp = Hb[b0 + 3];
                }
                float d0 = 1.f, d1 = z, p0 = 0.f, p1 = 1.f;
                static_for<m + 2, L + 1>([&](auto lc) {
                    constexpr int l = decltype(lc)::value;
                    constexpr float bt = beta_lm(l - 1, m);
                    const float d2 = fmaf(z, d1, -bt * d0);
                    const float p2 = fmaf(-bt, p0, fmaf(z, p1, d1));
                    const float hr = Hb[b0 + 2 * (l - m)], hi = Hb[b0 + 2 * (l - m) + 1];
                    A = fmaf(hr, d2, A);
                    Bv = fmaf(hi, d2, Bv);
                    Ap = fmaf(hr, p2, Ap);
                    Bp = fmaf(hi, p2, Bp);
                    d0 = d1;
                    d1 = d2;
                    p0 = p1;
                    p1 = p2;
                });
                F = fmaf(A, nr, fmaf(Bv, ni, F));
                Fz = fmaf(Ap, nr, fmaf(Bp, ni, Fz));
                Fx = fmaf((float)m, fmaf(A, ur, Bv * ui), Fx);
                Fy = fmaf((float)m, fmaf(Bv, ur, -A * ui), Fy);
                ur = nr;
                ui = ni;
            });
            const float gdr = fmaf(Fx, ux, fmaf(Fy, uy, Fz * z));
            const float sc = 2.f * wj * (sep * rinv);
            const float gx = sc * fmaf(-gdr, ux, Fx), gy = sc * fmaf(-gdr, uy, Fy),
                        gz = sc * fmaf(-gdr, z, Fz);
            atomicAdd(dw + jj, f2d_exact(2.f * F));
            atomicAdd(dpos + 3 * (int64_t)jj, f2d_exact(gx));
            atomicAdd(dpos + 3 * (int64_t)jj + 1, f2d_exact(gy));
            atomicAdd(dpos + 3 * (int64_t)jj + 2, f2d_exact(gz));
            pix -= gx;
            piy -= gy;
            piz -= gz;
        }
    }
#undef G3_FETCH
    dpi[0] += pix;
    dpi[1] += piy;
    dpi[2] += piz;
}

template <int L, int MODE>
__global__ void __launch_bounds__(kPairThreads, 2) k_pair(PairArgs a) {
    constexpr int NRP = Shape<L>::NRP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double s_e2[kMaxBins + 1];
    __shared__ float2 s_dec[kMaxBins];  // (e2f[b] + guard[b], e2f[b+1] - guard[b+1])
    __shared__ float s_guard0;
    __shared__ unsigned char s_tab[kBinTable + 2];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int B = a.bins.nbins;
    for (int k = threadIdx.x; k < kBinTable + 2; k += blockDim.x) s_tab[k] = a.bintab[k];
    for (int k = threadIdx.x; k <= B; k += blockDim.x) {
        s_e2[k] = a.bins.e2[k];
        if (k < B)
            s_dec[k] = make_float2(a.bins.e2f[k] + a.bins.guard[k], a.bins.e2f[k + 1] - a.bins.guard[k + 1]);
    }
    if (threadIdx.x == 0) s_guard0 = a.bins.guard[0];
    __syncthreads();
    const WarpSmem lay = warp_smem(NRP, B, a.kflush);
    unsigned char* base = smem_raw + (size_t)wid * lay.bytes;
    int* bucket = reinterpret_cast<int*>(base);
    float* res = reinterpret_cast<float*>(base + lay.off_res);
    int* cnt = reinterpret_cast<int*>(base + lay.off_meta);
    int* head = cnt + B;
    int* tot = cnt + 2 * B;
    int4* pcs = reinterpret_cast<int4*>(base + lay.off_pcs);
    float4* img = reinterpret_cast<float4*>(base + lay.off_prim);
    float* Rs = reinterpret_cast<float*>(base + lay.off_prim + 27 * 16);
    double* pd = reinterpret_cast<double*>(base + lay.off_prim + 27 * 16 + 12 * 4);
    float4* st_q = reinterpret_cast<float4*>(base + lay.off_stash);
    int* st_j = reinterpret_cast<int*>(base + lay.off_stash + kStashDepth * 32 * 16);
    int* st_c = st_j + kStashDepth * 32;
    const int cap = lay.cap;
    const int bstride = lay.cap + 1;  // bucket stride (odd: spreads bins over banks)
    const int kf = a.kflush;
    const unsigned lt = lanemask_lt();
    const Grid& g = a.g;
    const float Lb = g.box;
    const bool exact_inputs = (a.pts64 == nullptr);
    const float hi_rej = a.bins.hi_rej, lo_rej = a.bins.lo_rej;
    const float rminf = a.bins.rmin, invw = a.bins.invw;
    const int close_end = close_bins(a.bins, a.pts64);

    unsigned long long my_total = 0;  // lane b < B: pairs accepted into bin b
    long long cur_cat = -1;

    for (;;) {
        int q = 0;
        if (lane == 0) q = a.q0 + atomicAdd(a.queue, 1);
        q = __shfl_sync(kFull, q, 0);
        if (q >= a.nprim) break;
        const int p = a.plist ? a.plist[q] : q;
        const long long cat = (long long)(a.key[p] / (unsigned long long)g.cells_per_cat);
        if (cat != cur_cat) {
            if (cur_cat >= 0 && lane < B && my_total)
                atomicAdd(&a.counts[cur_cat * B + lane], my_total);
            my_total = 0;
            cur_cat = cat;
        }
        const long long kbase = cat * g.cells_per_cat;
        Prim P;
        {
            const float4 xi = a.pts[p];
            P.x = xi.x;
            P.y = xi.y;
            P.z = xi.z;
            if (a.pts64) {
                P.x64 = a.pts64[3 * (int64_t)p];
                P.y64 = a.pts64[3 * (int64_t)p + 1];
                P.z64 = a.pts64[3 * (int64_t)p + 2];
            } else {
                P.x64 = xi.x;
                P.y64 = xi.y;
                P.z64 = xi.z;
            }
        }
        if (lane == 0) {
            pd[0] = P.x64;
            pd[1] = P.y64;
            pd[2] = P.z64;
        }
        if (lane < 27) {
            const int sx = lane % 3 - 1, sy = (lane / 3) % 3 - 1, sz = lane / 9 - 1;
            img[lane] = make_float4(P.x - sx * Lb, P.y - sy * Lb, P.z - sz * Lb, 0.f);
        }
        if (lane < 9)
            Rs[lane] = g.radial ? los_rotation_entry(lane, P.x64, P.y64, P.z64, g.boxd)
                                : ((lane % 4 == 0) ? 1.f : 0.f);
        for (int k = lane; k < B; k += 32) {
            cnt[k] = 0;
            head[k] = 0;
            tot[k] = 0;
        }
        double dpi[3] = {0.0, 0.0, 0.0};  // adjoint: primary-side position gradient
        if constexpr (MODE == 0) {
            for (int k = lane; k < B * NRP; k += 32) res[k] = 0.f;
        } else {
            // adjoint multipoles H = w_i K_lm (M A_i), in the accumulator layout
            const float wi = a.pts[p].w;
            const float* Vrow = a.V + (int64_t)a.orig[p] * a.RLP;
            for (int col = lane; col < a.RL; col += 32) res[a.colmap[col]] = wi * a.colscale[col] * Vrow[col];
        }
        __syncwarp();

        int cxyz[3];
        {
            const float xs[3] = {P.x, P.y, P.z};
            for (int d = 0; d < 3; ++d) {
                int cc = (int)(xs[d] * g.inv_cell);
                cxyz[d] = cc < 0 ? 0 : (cc >= g.nc ? g.nc - 1 : cc);
            }
        }
        const int K = g.reach, W = 2 * K + 1, nrows = W * W;
        const float slack = a.bins.slack, rmax2 = a.bins.rmax2f;

        // ---- candidate stream: pieces of up to 32 rows at a time; an
        // iteration covers up to 32 consecutive slots of one piece.
        int rb = 0, npcs = 0, pi = 0, poff = 0;
        auto build_batch = [&]() {
            // up to three pieces per row (x images -L, 0, +L), kept in registers
            int4 pm = make_int4(0, 0, 0, 0), p0 = pm, pp = pm;
            const int r = rb + lane;
            if (r < nrows)
                row_pieces(r, W, K, cxyz[1], cxyz[2], img[13], g, slack, rmax2, kbase, a.cstart, pm,
                           p0, pp);
            const int npc = (pm.y > pm.x) + (p0.y > p0.x) + (pp.y > pp.x);
            int incl = npc;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += y;
            }
            npcs = __shfl_sync(kFull, incl, 31);
            __syncwarp();
            int k = incl - npc;
            if (pm.y > pm.x) pcs[k++] = pm;
            if (p0.y > p0.x) pcs[k++] = p0;
            if (pp.y > pp.x) pcs[k++] = pp;
            __syncwarp();
            pi = 0;
            poff = 0;
            rb += 32;
        };
        // issue one iteration: returns false once the stream is exhausted
        auto issue = [&](float4& qv, int& jv, int& codev) -> bool {
            while (pi >= npcs && rb < nrows) build_batch();
            if (pi >= npcs) {
                jv = -1;
                codev = 13;
                return false;
            }
            const int4 pc = pcs[pi];
            const int jj = pc.x + poff + lane;
            codev = pc.z;
            jv = jj < pc.y ? jj : -1;
            if (jv >= 0) qv = __ldg(a.pts + jv);
            poff += 32;
            if (pc.x + poff >= pc.y) {
                ++pi;
                poff = 0;
            }
            return true;
        };
        float4 sq[kScanDepth];
        int sj[kScanDepth], sc[kScanDepth];
        unsigned live = 0;  // bit s: slot s holds an issued iteration
#pragma unroll
        for (int s = 0; s < kScanDepth; ++s) {
            sq[s] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (issue(sq[s], sj[s], sc[s])) live |= 1u << s;
        }

        const float tscale = a.bin_tscale;
        for (;;) {
            int fb = -1, fn = 0;
            {
                const int myc = lane < B ? cnt[lane] : 0;
                const unsigned fm = __ballot_sync(kFull, myc >= 32 * kf);
                if (fm) {
                    fb = __ffs(fm) - 1;
                    fn = 32 * kf;
                }
            }
            if (fb < 0 && live) {
                // ---- scan: decide the bins of all pending iterations (independent
                // chains), refill them, then append; the flush check comes next
                int binv[kScanDepth], jv[kScanDepth], cv[kScanDepth];
#pragma unroll
                for (int s = 0; s < kScanDepth; ++s) {
                    const int j = sj[s];
                    const int code = sc[s];
                    const float4 qq = sq[s];
                    const bool on = (live >> s) & 1u;
                    if (on && !issue(sq[s], sj[s], sc[s])) live &= ~(1u << s);
                    int bin = -1;
                    if (on && j >= 0) {
                        const float4 o = img[code];
                        const float dx = qq.x - o.x;
                        const float dy = qq.y - o.y;
                        const float dz = qq.z - o.z;
                        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                        if (!(r2 < hi_rej)) {
                            bin = -1;
                        } else {
                            int ti = (int)(r2 * tscale);
                            ti = ti > kBinTable + 1 ? kBinTable + 1 : ti;
                            const int tv = s_tab[ti];
                            if (tv < kTabReject) {
                                bin = tv;
                            } else if (tv == kTabReject) {
                                bin = -1;
                            } else if (r2 < lo_rej) {
                                bin = -1;
                            } else if (!(r2 > s_guard0)) {
                                bin = (exact_inputs && code == 13 && r2 == 0.f) ? -1 : -2;
                            } else {
                                const float rr = r2 * rsqrtf(r2);
                                int bb = (int)((rr - rminf) * invw);
                                bb = bb < 0 ? 0 : (bb >= B ? B - 1 : bb);
                                const float2 iv = s_dec[bb];
                                bin = (r2 > iv.x && r2 < iv.y) ? bb : -2;
                            }
                            if (bin == -2)
                                bin = exact_bin(a.pts, a.pts64, j, pd[0], pd[1], pd[2], code % 3 - 1,
                                                (code / 3) % 3 - 1, code / 9 - 1, g.boxd, g.periodic,
                                                s_e2, B);
                        }
                    }
                    binv[s] = bin;
                    jv[s] = j;
                    cv[s] = code;
                }
#pragma unroll
                for (int s = 0; s < kScanDepth; ++s) {
                    const int bin = binv[s];
                    // append to the bin's bucket (warp-aggregated per bin)
                    const unsigned peers = __match_any_sync(kFull, bin);
                    const int leader = __ffs(peers) - 1;
                    int pos = 0;
                    if (lane == leader && bin >= 0) {
                        const int c = cnt[bin];
                        const int np = __popc(peers);
                        pos = head[bin] + c;
                        cnt[bin] = c + np;
                    }
                    pos = __shfl_sync(kFull, pos, leader);
                    if (bin >= 0) {
                        pos += __popc(peers & lt);
                        if (pos >= cap) pos -= cap;
                        bucket[bin * bstride + pos] = (int)((unsigned)jv[s] | ((unsigned)cv[s] << kIdxBits));
                    }
                    __syncwarp();
                }
                continue;
            }
            if (fb < 0) {  // stream exhausted: flush the partial buckets one by one
                const int myc = lane < B ? cnt[lane] : 0;
                const unsigned nz = __ballot_sync(kFull, myc > 0);
                if (!nz) break;
                fb = __ffs(nz) - 1;
                fn = cnt[fb];
            }
            const int kk = (fn + 31) >> 5;
            // park the scan pipeline in shared memory so that only the
            // accumulators are live in registers during the flush
#pragma unroll
            for (int s = 0; s < kScanDepth; ++s) {
                st_q[s * 32 + lane] = sq[s];
                st_j[s * 32 + lane] = sj[s];
                st_c[s * 32 + lane] = sc[s];
            }
            __syncwarp();
            if constexpr (MODE == 0)
                flush_bin<L>(a.pts, bucket + fb * bstride, cap, fn, kk, head[fb], res + fb * NRP, img,
                             Rs, g.radial, lane, a, p, fb < close_end);
            else
                flush_grad<L>(a.pts, a.orig, bucket + fb * bstride, cap, fn, kk, head[fb],
                              res + fb * NRP, img, lane, a.dw, a.dpos, dpi, a, p, fb < close_end);
            __syncwarp();
#pragma unroll
            for (int s = 0; s < kScanDepth; ++s) {
                sq[s] = st_q[s * 32 + lane];
                sj[s] = st_j[s * 32 + lane];
                sc[s] = st_c[s * 32 + lane];
            }
            __syncwarp();
            if (lane == 0) {
                int nh = head[fb] + fn;
                if (nh >= cap) nh -= cap;
                head[fb] = nh;
                cnt[fb] -= fn;
                tot[fb] += fn;
            }
            __syncwarp();
        }
        // ---- A row (normalised) or the primary's adjoint, counts
        // A row: original index, or the position inside this chunk of primaries
        const int row = a.chunked ? q - a.q0 : a.orig[p];
        if (MODE == 0 && lane == 0) a.wrow[row] = a.pts[p].w;
        if constexpr (MODE == 0) {
            float* Arow = a.A + (int64_t)row * a.RLP;
            for (int col = lane; col < a.RL; col += 32) Arow[col] = res[a.colmap[col]] * a.colscale[col];
        } else {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                double v = dpi[k];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
                if (lane == 0) atomicAdd(a.dpos + 3 * (int64_t)row + k, v);
            }
        }
        if (lane < B) my_total += (unsigned long long)tot[lane];
        __syncwarp();
    }
    if (cur_cat >= 0 && lane < B && my_total) atomicAdd(&a.counts[cur_cat * B + lane], my_total);
}

template <int L, int MODE>
int launch_mode(const PairArgs& a, int nsm, cudaStream_t st) {
    const WarpSmem lay = warp_smem(Shape<L>::NRP, a.bins.nbins, a.kflush);
    const size_t smem = (size_t)lay.bytes * kPairWarps;
    cudaError_t e = cudaFuncSetAttribute(k_pair<L, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return -1;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_pair<L, MODE>, kPairThreads, smem);
    if (e != cudaSuccess || per_sm < 1) return -1;
    int blocks = per_sm * nsm;
    const int need = (a.nprim + kPairWarps - 1) / kPairWarps;
    if (blocks > need) blocks = need > 0 ? need : 1;
    k_pair<L, MODE><<<blocks, kPairThreads, smem, st>>>(a);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <int L>
int launch_one(const PairArgs& a, int nsm, cudaStream_t st, int mode) {
    return mode == 0 ? launch_mode<L, 0>(a, nsm, st) : launch_mode<L, 1>(a, nsm, st);
}

}  // namespace

size_t pair_smem_per_warp(int lmax, int nbins, int kflush) {
    const int nr = (lmax + 1) * (lmax + 1);
    return (size_t)warp_smem(((nr + 31) / 32) * 32, nbins, kflush).bytes;
}

int pair_nrp(int lmax) {
    const int nr = (lmax + 1) * (lmax + 1);
    return ((nr + 31) / 32) * 32;
}

int launch_pair(int lmax, const PairArgs& a, int nsm, cudaStream_t st, int mode) {
    switch (lmax) {
        case 0: return launch_one<0>(a, nsm, st, mode);
        case 1: return launch_one<1>(a, nsm, st, mode);
        case 2: return launch_one<2>(a, nsm, st, mode);
        case 3: return launch_one<3>(a, nsm, st, mode);
        case 4: return launch_one<4>(a, nsm, st, mode);
        case 5: return launch_one<5>(a, nsm, st, mode);
        case 6: return launch_one<6>(a, nsm, st, mode);
        case 7: return launch_one<7>(a, nsm, st, mode);
        case 8: return launch_one<8>(a, nsm, st, mode);
        case 9: return launch_one<9>(a, nsm, st, mode);
        case 10: return launch_one<10>(a, nsm, st, mode);
        default: return -1;
    }
}

}  // namespace g3
