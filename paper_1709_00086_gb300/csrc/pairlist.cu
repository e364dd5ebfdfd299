// Pair stage split in three kernels (forward): count, scan, accumulate.
//
// Paper: Algorithm 1 and Sec. 3.1 (neighbours within rmax, radial bin,
// rotation, harmonics, multipoles per shell), Sec. 3.3.1 (pre-binning: pairs
// of one primary collected per radial bin before their multipoles are
// computed) and Sec. 3.3.2 (one reduction of the per-lane partials per
// primary and bin instead of one per pair group).
//
//   k_count  -- per primary, the number of candidate secondaries in the
//               sphere's cell rows: at most ceil(candidates/32) + B chunks.
//               One pass over the list pool if it holds the total (k_scan
//               takes its chunks from a counter), else the host places every
//               primary's chunks and cuts the range into passes.
//   k_scan   -- per primary (one warp), streams the candidates of 32 cell rows
//               at a time, slot range by slot range, decides each pair's bin
//               exactly and places the accepted pairs into per-bin chunks of
//               32 (tagged with the bin) of this primary, straight from the
//               candidates' lanes or, where fewer than half of them are
//               pairs, gathered in groups of 32 first.  For a plain forward
//               a chunk holds 32 direction records (unit vector and weight, 512
//               bytes), for the calls that differentiate 32 list entries (slot
//               and image, 128 bytes).
//   k_accum_dir -- plain forwards: per primary (one warp), walks its chunks bin
//               by bin: each lane takes one record of a chunk, adds its
//               harmonics (Chebyshev form, pair_common.cuh) to (lmax+1)^2
//               register partials, and one warp butterfly per (primary, bin)
//               reduces them; the normalised row of multipoles goes to A.
//   k_accum  -- the same from list entries (gather, separation, direction per
//               pair): forwards to be differentiated in FP32, and plain ones
//               whose list budget is too small for records.
//
// Compared with the fused kernel (pair.cu, G3PCF_OPT_PAIR_KERNELS = 1, kept as
// a cross-check), the accumulation runs without the scan's state in registers
// and reduces across lanes once per bin instead of once per bucket.  Plain,
// batched and graph-captured forwards, and the adjoint pair pass (k_adj), all
// walk these lists.
#include "pair_common.cuh"

namespace g3 {

namespace {

constexpr int kLWarps = 4;
constexpr int kLThreads = kLWarps * 32;
constexpr int kChunk = 32;      // pairs per list chunk
// Candidate sub-iterations per trip in k_scan, staged or not, and its stage (pairs)
constexpr int kTripStaged = 4, kTripDirect = 3;
constexpr int kStage = (kTripStaged + 1) * kChunk;
constexpr int kScanWarps = 8;  // warps per CTA of k_scan, kScanCtas CTAs per SM
constexpr int kScanThreads = kScanWarps * 32;
constexpr int kScanCtas = 4;
constexpr unsigned kNoPair = 0xffffffffu;  // padding entry of a list chunk (image code 31 is unused)

// Per-warp shared memory of k_scan: img[27] float4, pd[4] double, pcs[kMaxPieces]
// int2 (the slot ranges of a row batch: first | image code << 27, end), the compaction
// stage if staged (kStage accepted pairs: separation and weight, or list entry, and bin),
// per bin the last written list slot and the chunk count, R[9] float.
template <bool DIR, bool STAGED>
struct ScanSmem {
    static constexpr int N = STAGED ? kStage : 1;
    using Item = typename std::conditional<DIR, float4, int>::type;
    float4 img[27];
    int2 pcs[kMaxPieces];
    Item stage[N];
    int sbin[N];
    int bst[64];  // (63: lanes without a bin)
    int bnbc[32];
    double pd[4];
    float R[12];
};

// Direction record of one accepted pair in radial mode: the unit vector (z, x, y)
// of the separation rotated to the primary's line of sight, and the weight.
__device__ __forceinline__ float4 pair_record(const float4& d, const float* R) {
    const float dx = fmaf(R[0], d.x, fmaf(R[1], d.y, R[2] * d.z));
    const float dy = fmaf(R[3], d.x, fmaf(R[4], d.y, R[5] * d.z));
    const float dz = fmaf(R[6], d.x, fmaf(R[7], d.y, R[8] * d.z));
    const float rinv = rsqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
    return make_float4(dz * rinv, dx * rinv, dy * rinv, d.w);
}
// Head (nearest FP32 values) of image `code` of the primary; see set_image.
__device__ __forceinline__ float4 image_head(int code, const float4& P0, const double* pts64, int p, double boxd) {
    const int sx = code % 3 - 1, sy = (code / 3) % 3 - 1, sz = code / 9 - 1;
    double x = P0.x, y = P0.y, z = P0.z;
    if (pts64) {
        x = pts64[3 * (int64_t)p];
        y = pts64[3 * (int64_t)p + 1];
        z = pts64[3 * (int64_t)p + 2];
    }
    return make_float4((float)(x - sx * boxd), (float)(y - sy * boxd), (float)(z - sz * boxd), 0.f);
}

// Catalog of sorted slot p (cell keys stay below 2^31).
__device__ __forceinline__ long long catalog_of(const ListArgs& a, int p) {
    return a.ncat == 1 ? 0 : (long long)(a.key[p] / (unsigned)a.g.cells_per_cat);
}

// lpp (a power of two) lanes per primary, so that a launch has enough threads
// whatever the number of primaries and of rows: one warp per primary left 23 of 32
// lanes idle at 9 rows (120,000 primaries: 83 us).
constexpr int kCountThreads = 256;
__global__ void __launch_bounds__(kCountThreads) k_count(ListArgs a, int lpp) {
    __shared__ unsigned long long s_cand, s_total;
    __shared__ int s_most;
    if (threadIdx.x == 0) {
        s_cand = s_total = 0;
        s_most = 0;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    const int per = 32 / lpp, sub = lane & (lpp - 1);
    const Grid& g = a.g;
    const int K = g.reach, W = 2 * K + 1, nrows = W * W;
    unsigned long long cand = 0, total = 0;
    int most = 0;
    for (int q0 = a.qa + gw * per; q0 < a.qb; q0 += nw * per) {
        const int q = q0 + lane / lpp;
        long long sum = 0;
        if (q < a.qb) {
            const int p = a.plist ? a.plist[q] : q;
            const float4 P0 = a.pts[p];
            const long long kbase = catalog_of(a, p) * g.cells_per_cat;
            const int cy = cell_of(P0.y, g), cz = cell_of(P0.z, g);
            for (int r = sub; r < nrows; r += lpp) {
                int4 pm, p0, pp;
                row_pieces(r, W, K, cy, cz, P0, g, a.bins.slack, a.bins.rmax2f, kbase, a.cstart, pm, p0, pp);
                sum += max(pm.y - pm.x, 0) + max(p0.y - p0.x, 0) + max(pp.y - pp.x, 0);
            }
        }
        for (int o = lpp >> 1; o > 0; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
        if (q < a.qb && sub == 0) {
            const int need = (int)((sum + kChunk - 1) / kChunk) + a.bins.nbins;
            a.need[q] = need;
            cand += sum;
            total += need;
            most = max(most, need);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        cand += __shfl_xor_sync(kFull, cand, o);
        total += __shfl_xor_sync(kFull, total, o);
    }
    most = __reduce_max_sync(kFull, most);
    if (lane == 0 && most > 0) {
        atomicAdd(&s_cand, cand);
        atomicAdd(&s_total, total);
        atomicMax(&s_most, most);
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_most > 0) {
        atomicAdd(reinterpret_cast<unsigned long long*>(a.status + kCandSlot), s_cand);
        atomicAdd(reinterpret_cast<unsigned long long*>(a.status + kTotalSlot), s_total);
        atomicMax(a.status + kMostSlot, s_most);
    }
}

// k_scan: 116 warp instructions per 32 accepted pairs at 3.7 cells per rmax, and
// every instruction slot counts: logic and selects take two cycles on their pipe,
// match.any 72 beside the other warps' work, so the kernel is bound by issue
// (staged also by the shared-memory pipe, 70% busy), not by DRAM.  The unit vector is formed here because the
// distance test has the separation and 1/r at hand: gathering the point again and
// forming it in the accumulate kernel cost about 100 cycles per chunk there.  The
// bin comes from r = r^2 rsqrt(r^2) by one rounding instead of a table look-up
// (whose bank conflicts cost 3.5 wavefronts per 32 candidates); the 1e-4 of
// the candidates near an edge take the exact rule.  32 warps per SM at 64
// registers: 40 and 48 are 6% and 24% slower.  Staged, two or three loads per trip
// instead of four are 10% and 3% slower; direct (no stage), three and two are the same,
// four spill (3%).  200,000 clustered points (L = 696, 4.0e9 pairs): 16.1 ms writing
// 16 bytes per pair (staged 19.7, which is what the form took that wrote 4 bytes
// and left the direction to the accumulate kernel).
//
// What k_scan writes per pair: a list entry, or for k_accum_dir its direction (in
// radial mode rotated to the primary's line of sight).
constexpr int kEntries = 0, kDirs = 1, kDirsRadial = 2;
constexpr float kRound = 12582912.f;  // 1.5 * 2^23: x + kRound rounds x to the nearest integer
// Predicated shared-memory stores of one staged pair, without a branch.
__device__ __forceinline__ void put_if(bool acc, unsigned at, unsigned bat, int bin, const float4& d) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.s32 p, %0, 0;\n @p st.shared.v4.f32 [%1], {%4, %5, %6, %7};\n"
        " @p st.shared.s32 [%2], %3;\n}\n" ::"r"((int)acc), "r"(at), "r"(bat), "r"(bin), "f"(d.x), "f"(d.y),
        "f"(d.z), "f"(d.w)
        : "memory");
}
__device__ __forceinline__ void put_if(bool acc, unsigned at, unsigned bat, int bin, unsigned e) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.s32 p, %0, 0;\n @p st.shared.u32 [%1], %4;\n"
        " @p st.shared.s32 [%2], %3;\n}\n" ::"r"((int)acc), "r"(at), "r"(bat), "r"(bin), "r"(e)
        : "memory");
}
// MUFU.RSQ alone (subnormal arguments give infinity, which the caller tests).
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// F64: directions of close pairs from FP64 positions (FP32 ones need only a scale, and the
// call behind the FP64 form costs the kernel 5%: 200,000 clustered points 16.9 against
// 16.1 ms; inlined 17.4).
template <int MODE, bool STAGED, bool F64>
__global__ void __launch_bounds__(kScanThreads, kScanCtas) k_scan(ListArgs a) {
    constexpr bool DIR = MODE != kEntries;
    constexpr int kTrip = STAGED ? kTripStaged : kTripDirect;
    using Smem = ScanSmem<DIR, STAGED>;
    extern __shared__ __align__(16) unsigned char ls_raw[];
    __shared__ double s_e2[kMaxBins + 1];
    __shared__ float2 s_dec[kMaxBins];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int B = a.bins.nbins;
    for (int k = threadIdx.x; k <= B; k += blockDim.x) {
        s_e2[k] = a.bins.e2[k];
        if (k < B)
            s_dec[k] = make_float2(a.bins.e2f[k] + a.bins.guard[k], a.bins.e2f[k + 1] - a.bins.guard[k + 1]);
    }
    __syncthreads();
    Smem& S = reinterpret_cast<Smem*>(ls_raw)[wid];
    const unsigned lt = lanemask_lt(), gt = ~lt & ~(1u << lane);
    const Grid& g = a.g;
    const bool exact_inputs = (a.pts64 == nullptr);
    const float invw = a.bins.invw, binc = a.bins.bin_c, lim = a.bins.bin_lim;
    const int K = g.reach, W = 2 * K + 1, nrows = W * W;
    const unsigned stage0 = (unsigned)__cvta_generic_to_shared(S.stage);
    const unsigned bin0 = (unsigned)__cvta_generic_to_shared(S.sbin);
    unsigned long long my_total = 0;
    long long cur_cat = -1;

    const int qa = a.qrange ? a.qrange[0] : a.qa, qb = a.qrange ? a.qrange[1] : a.qb;
    for (;;) {
        int q = 0;
        if (lane == 0) q = qa + atomicAdd(a.queue, 1);
        q = __shfl_sync(kFull, q, 0);
        if (q >= qb) break;
        const int cap_ch = a.need[q];  // chunks reserved for the primary
        int cbase = 0;
        if (a.cursor) {
            if (lane == 0) {
                cbase = atomicAdd(a.cursor, cap_ch);
                if (cbase < 0 || cbase > a.cap - cap_ch) {  // more than the captured pool holds
                    cbase = -1;
                    atomicOr(a.status, kStatusOverflow);
                }
                a.base[q] = cbase;
            }
            cbase = __shfl_sync(kFull, cbase, 0);
        } else {
            cbase = a.base[q];
        }
        if (cbase < 0) {  // no room in the planned passes (flagged by the planner)
            if (lane == 0) a.nchunks[q] = 0;
            continue;
        }
        const int p = a.plist ? a.plist[q] : q;
        const long long cat = catalog_of(a, p);
        if (cat != cur_cat) {
            if (cur_cat >= 0 && lane < B && my_total) atomicAdd(&a.counts[cur_cat * B + lane], my_total);
            my_total = 0;
            cur_cat = cat;
        }
        const long long kbase = cat * g.cells_per_cat;
        const float4 P0 = a.pts[p];
        if (lane < 27) S.img[lane] = image_head(lane, P0, a.pts64, p, g.boxd);
        if (lane < 3) {
            const float pv = lane == 0 ? P0.x : (lane == 1 ? P0.y : P0.z);
            S.pd[lane] = a.pts64 ? a.pts64[3 * (int64_t)p + lane] : (double)pv;
        }
        if constexpr (MODE == kDirsRadial) {
            if (lane < 9) {
                double x0 = P0.x, x1 = P0.y, x2 = P0.z;
                if (a.pts64) {
                    x0 = a.pts64[3 * (int64_t)p];
                    x1 = a.pts64[3 * (int64_t)p + 1];
                    x2 = a.pts64[3 * (int64_t)p + 2];
                }
                S.R[lane] = los_rotation_entry(lane, x0, x1, x2, g.boxd);
            }
        }
        const int cy = cell_of(P0.y, g), cz = cell_of(P0.z, g);
        // this primary's chunks: list entries, or (DIR) one direction per pair
        int* const pool = a.chunks + (int64_t)cbase * kChunk;
        float4* const dpool = a.dirs + (int64_t)cbase * kChunk;
        int* const ptag = a.tag + cbase;
        int* const pord = a.ord + cbase;
        int nch = 0;                   // chunks opened so far (warp-uniform)
        // per bin: the last written slot of the open chunk (chunk * 32 + position;
        // -1, like any full chunk, has position 31) and the chunks opened so far
        S.bst[lane] = S.bst[32 + lane] = -1;
        S.bnbc[lane] = 0;
        __syncwarp();

        // Place one accepted pair per lane (bin 63: none) into the open chunk of
        // its bin, opening a new chunk where a bin's chunk fills (at most one per
        // bin and call).  Lanes of one bin form a group (mine, from match.any: its 72
        // cycles run beside the other warps' instructions); the group's highest
        // lane opens the chunk and leaves the bin's last slot.
        auto place = [&](typename Smem::Item it, int bin, bool v, unsigned mine) {
            const int rank = __popc(mine & lt);
            const int st = S.bst[bin];
            int sl = st + 1 + rank;
            const bool cross = (unsigned)(sl ^ st) >= (unsigned)kChunk;  // past the open chunk
            const bool last = v && (mine & gt) == 0u;
            const bool opens = last && cross;
            const unsigned gm = __ballot_sync(kFull, opens);
            if (gm) {
                // the new chunk of this lane's group: numbered by the groups' highest lanes
                // (mine & gm: the highest lane's bit)
                const int nnew = nch + __popc(gm & ((mine & gm) - 1u));
                if (cross) sl = nnew * kChunk + (sl & (kChunk - 1));
                nch += __popc(gm);
                if (opens) {
                    const int nb = S.bnbc[bin];
                    if (nnew < cap_ch)
                        ptag[nnew] = (nb << 5) | bin;  // (rank among the bin's chunks, bin)
                    else
                        atomicOr(a.status, kStatusOverflow);
                    S.bnbc[bin] = nb + 1;
                }
            }
            if (v && sl < cap_ch * kChunk) {
                if constexpr (MODE == kDirs)
                    dpool[sl] = it;
                else if constexpr (MODE == kDirsRadial)
                    dpool[sl] = pair_record(it, S.R);
                else
                    pool[sl] = it;
            }
            // (every lane has read the bin state: the ballot waited for it)
            if (last) S.bst[bin] = sl;
            __syncwarp();
        };
        int scnt = 0;  // accepted pairs in the stage (warp-uniform)

        // candidates: batches of 32 cell rows -> slot ranges (pieces) -> up to
        // kTrip x 32 slots per trip, all loads of a trip in flight together
        for (int rb = 0; rb < nrows; rb += 32) {
            int4 pm = make_int4(0, 0, 0, 0), p0 = pm, pp = pm;
            const int r = rb + lane;
            if (r < nrows)
                row_pieces(r, W, K, cy, cz, P0, g, a.bins.slack, a.bins.rmax2f, kbase, a.cstart, pm, p0, pp);
            const int npc = (pm.y > pm.x) + (p0.y > p0.x) + (pp.y > pp.x);
            int incl = npc;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += y;
            }
            const int npcs = __shfl_sync(kFull, incl, 31);
            __syncwarp();
            {
                int k = incl - npc;
                if (pm.y > pm.x) S.pcs[k++] = make_int2((int)((unsigned)pm.x | ((unsigned)pm.z << kIdxBits)), pm.y);
                if (p0.y > p0.x) S.pcs[k++] = make_int2((int)((unsigned)p0.x | ((unsigned)p0.z << kIdxBits)), p0.y);
                if (pp.y > pp.x) S.pcs[k++] = make_int2((int)((unsigned)pp.x | ((unsigned)pp.z << kIdxBits)), pp.y);
            }
            __syncwarp();
            for (int pi = 0; pi < npcs; ++pi) {
                const int2 pc = S.pcs[pi];
                const unsigned code = (unsigned)pc.x >> kIdxBits;
                const float4 o = S.img[code];
                for (int j0 = (pc.x & (int)kIdxMask) + lane; j0 < pc.y + lane; j0 += kTrip * kChunk) {
                    // slots past the piece keep a far x (r^2 ~ 1e36: no pair)
                    const float4* src = a.pts + j0;
                    float4 d[kTrip];
#pragma unroll
                    for (int u = 0; u < kTrip; ++u) {
                        d[u] = make_float4(1e18f, 0.f, 0.f, 0.f);
                        if (j0 + u * kChunk < pc.y) d[u] = __ldg(src + u * kChunk);
                    }
                    // bin = round((r - rmin) / width - 1/2); within bin_lim of the bin's
                    // centre (in widths) the FP32 bin is the exact one, else (and where
                    // r is NaN: r^2 is 0 or subnormal) bin_slow decides
                    int bn[kTrip];
                    float rinv[kTrip];
                    bool near[kTrip], any = false;
#pragma unroll
                    for (int u = 0; u < kTrip; ++u) {
                        d[u].x -= o.x;
                        d[u].y -= o.y;
                        d[u].z -= o.z;
                        const float r2 = fmaf(d[u].x, d[u].x, fmaf(d[u].y, d[u].y, d[u].z * d[u].z));
                        rinv[u] = rsqrt_ftz(r2);
                        const float t = fmaf(r2 * rinv[u], invw, binc);
                        const float m = __fadd_rn(t, kRound);
                        bn[u] = __float_as_int(m) - __float_as_int(kRound);
                        near[u] = !(fabsf(__fsub_rn(t, __fsub_rn(m, kRound))) <= lim);
                        any |= near[u];
                    }
                    if (__any_sync(kFull, any)) {
#pragma unroll
                        for (int u = 0; u < kTrip; ++u)
                            if (near[u]) {
                                const float r2 = fmaf(d[u].x, d[u].x, fmaf(d[u].y, d[u].y, d[u].z * d[u].z));
                                float rr = r2;
                                bn[u] = bin_slow(r2, a.bins.lo_rej, a.bins.hi_rej, a.bins.guard[0], s_dec,
                                                 a.bins.rmin, invw, B, exact_inputs, (int)code, a.pts, a.pts64,
                                                 j0 + u * kChunk, S.pd, g.boxd, g.periodic, s_e2);
                                if (DIR && (unsigned)bn[u] < (unsigned)B && r2 <= close_r2(a.bins, a.pts64)) {
                                    if constexpr (F64) {
                                        double s[4];
                                        close_sep(a.pts, a.pts64, S.pd, j0 + u * kChunk, (int)code, g.boxd, s);
                                        d[u] = make_float4((float)s[0], (float)s[1], (float)s[2], d[u].w);
                                    } else {  // exact already
                                        d[u].x *= 0x1p100f;
                                        d[u].y *= 0x1p100f;
                                        d[u].z *= 0x1p100f;
                                    }
                                    rr = fmaf(d[u].x, d[u].x, fmaf(d[u].y, d[u].y, d[u].z * d[u].z));
                                }
                                rinv[u] = rsqrtf(rr);
                            }
                    }
                    if constexpr (!STAGED) {  // place the candidates' lanes as they are
                        unsigned mine[kTrip];
#pragma unroll
                        for (int u = 0; u < kTrip; ++u) {
                            if constexpr (MODE == kDirs)
                                d[u] = make_float4(d[u].z * rinv[u], d[u].x * rinv[u], d[u].y * rinv[u], d[u].w);
                            if ((unsigned)bn[u] >= (unsigned)B) bn[u] = 63;
                            mine[u] = __match_any_sync(kFull, bn[u]);
                        }
#pragma unroll
                        for (int u = 0; u < kTrip; ++u) {
                            if constexpr (DIR)
                                place(d[u], bn[u], bn[u] != 63, mine[u]);
                            else
                                place((unsigned)(j0 + u * kChunk) | (code << kIdxBits), bn[u], bn[u] != 63, mine[u]);
                        }
                        continue;
                    }
#pragma unroll
                    for (int u = 0; u < kTrip; ++u) {
                        // accepted lanes append in lane order
                        const bool acc = (unsigned)bn[u] < (unsigned)B;
                        const unsigned vm = __ballot_sync(kFull, acc);
                        const int at = scnt + __popc(vm & lt);
                        if constexpr (MODE == kDirs)
                            put_if(acc, stage0 + at * 16, bin0 + at * 4, bn[u],
                                   make_float4(d[u].z * rinv[u], d[u].x * rinv[u], d[u].y * rinv[u], d[u].w));
                        else if constexpr (MODE == kDirsRadial)
                            put_if(acc, stage0 + at * 16, bin0 + at * 4, bn[u], d[u]);
                        else
                            put_if(acc, stage0 + at * 4, bin0 + at * 4, bn[u],
                                   (unsigned)(j0 + u * kChunk) | (code << kIdxBits));
                        scnt += __popc(vm);
                    }
                    if (scnt >= kChunk) {
                        __syncwarp();
                        int at = lane;
                        for (; scnt >= kChunk; scnt -= kChunk, at += kChunk) {
                            const int bin = S.sbin[at];
                            place(S.stage[at], bin, true, __match_any_sync(kFull, bin));
                        }
                        // the rest (fewer than 32) to the stage's front
                        const auto it = S.stage[at];
                        const int bin = S.sbin[at];
                        __syncwarp();
                        S.stage[lane] = it;
                        S.sbin[lane] = bin;
                        __syncwarp();
                    }
                }
            }
            __syncwarp();
        }
        if (STAGED && scnt > 0) {  // the last accepted pairs (fewer than 32)
            __syncwarp();
            const int bin = lane < scnt ? S.sbin[lane] : 63;
            place(S.stage[lane], bin, lane < scnt, __match_any_sync(kFull, bin));
        }
        // the bin state back in lane b
        int cfill = kChunk, ccur = 0, nbc = 0;
        if (lane < B) {
            const int st = S.bst[lane];
            cfill = (st & 31) + 1;
            ccur = st >> 5;
            nbc = S.bnbc[lane];
        }
        const unsigned padd = nbc > 0 ? (unsigned)((nbc - 1) * kChunk + cfill) : 0u;  // pairs of bin lane
        // pad the open chunks behind their last entry
        unsigned pmask = __ballot_sync(kFull, lane < B && cfill < kChunk);
        while (pmask) {
            const int b = __ffs(pmask) - 1;
            pmask &= pmask - 1;
            const int c = __shfl_sync(kFull, ccur, b);
            const int f = __shfl_sync(kFull, cfill, b);
            if (lane >= f && c < cap_ch) {
                if constexpr (DIR)
                    dpool[c * kChunk + lane] = make_float4(0.f, 1.f, 0.f, 0.f);  // weight 0
                else
                    pool[c * kChunk + lane] = (int)kNoPair;
            }
        }
        // list the chunks grouped by bin (stable): position = chunks of the
        // lower bins + rank inside the bin
        {
            int off = nbc;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(kFull, off, o);
                if (lane >= o) off += y;
            }
            off -= nbc;
            const int nlist = nch < cap_ch ? nch : cap_ch;
            for (int c0 = 0; c0 < nlist; c0 += 32) {
                const int c = c0 + lane;
                const int t = c < nlist ? ptag[c] : 0;
                const int b = t & 31;
                const int pos = __shfl_sync(kFull, off, b) + (t >> 5);
                if (c < nlist && pos < cap_ch) pord[pos] = c | (b << 26);
            }
        }
        if constexpr (DIR) {  // the tags are read: their first nbins ints take the bins' chunk counts
            __syncwarp();
            if (lane < B) ptag[lane] = nbc;
        }
        if (lane == 0) a.nchunks[q] = nch < cap_ch ? nch : cap_ch;
        my_total += padd;
        __syncwarp();
    }
    if (cur_cat >= 0 && lane < B && my_total) atomicAdd(&a.counts[cur_cat * B + lane], my_total);
}

__global__ void k_plan_init(int* passq, int npass, int qb) {
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p <= npass; p += gridDim.x * blockDim.x) passq[p] = qb;
}

// Exclusive prefix sums of need[qa..qb) in 64 bits (the chunks of a large
// batch exceed 2^31): per-block sums, a scan of those, then the blocks.
constexpr int kScan64 = 1024;
__device__ long long block_scan64(long long v, long long* sh, long long& total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[wid] = x;
    __syncthreads();
    if (wid == 0) {
        long long t = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(kFull, t, o);
            if (lane >= o) t += y;
        }
        sh[lane] = t;
    }
    __syncthreads();
    const long long pre = (wid > 0 ? sh[wid - 1] : 0) + x - v;
    total = sh[(blockDim.x >> 5) - 1];
    __syncthreads();
    return pre;
}
__global__ void k_need_sums(const int* need, int64_t n, long long* bsum) {
    __shared__ long long sh[32];
    const int64_t i = blockIdx.x * (int64_t)kScan64 + threadIdx.x;
    long long tot;
    block_scan64(i < n ? need[i] : 0, sh, tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}
__global__ void k_need_top(long long* bsum, int nb) {
    __shared__ long long sh[32];
    long long carry = 0;
    for (int b0 = 0; b0 < nb; b0 += kScan64) {
        const int i = b0 + threadIdx.x;
        long long tot;
        const long long pre = block_scan64(i < nb ? bsum[i] : 0, sh, tot);
        if (i < nb) bsum[i] = carry + pre;
        carry += tot;
    }
}
__global__ void k_need_final(const int* need, int64_t n, const long long* bsum, long long* out) {
    __shared__ long long sh[32];
    const int64_t i = blockIdx.x * (int64_t)kScan64 + threadIdx.x;
    long long tot;
    const long long pre = block_scan64(i < n ? need[i] : 0, sh, tot);
    if (i < n) out[i] = bsum[blockIdx.x] + pre;
}

__global__ void k_plan(const int* need, const long long* gbase, int qa, int qb, long long stride, int slack,
                       int npass, int* base, int* passq, int* status) {
    for (int q = qa + blockIdx.x * blockDim.x + threadIdx.x; q < qb; q += gridDim.x * blockDim.x) {
        const long long gb = gbase[q - qa];
        const long long pql = gb / stride;
        const int pq = pql < npass ? (int)pql : npass;
        const bool ok = pq < npass && need[q] <= slack;
        base[q] = ok ? (int)(gb - pql * stride) : -1;
        if (!ok) atomicOr(status, kStatusOverflow);
        // first primary of every pass that starts here
        const long long pprevl = q == qa ? -1 : gbase[q - 1 - qa] / stride;
        const int pprev = pprevl < npass ? (int)pprevl : npass;
        for (int pp = pprev + 1; pp <= pq && pp < npass; ++pp) passq[pp] = q;
    }
}

// Asynchronous global -> shared copies (one per lane) and their groups.
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
// 16 bytes, or zeros without reading when !valid
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool valid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int n = valid ? 16 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}
// 16 bytes past L1
__device__ __forceinline__ void cp_async16_cg(void* dst, const void* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Image `code` of the primary (its position minus the code's box shift) as an
// FP32 head img[code] and tail img[27 + code] of the FP64 value (the primary's
// FP64 position when the input is FP64): the separation (q - head) - tail is
// then as exact as FP32 allows even where the shift is a whole box side.
__device__ __forceinline__ void set_image(float4* img, int code, const float4& P0, const double* pts64, int p,
                                          double boxd) {
    const int sx = code % 3 - 1, sy = (code / 3) % 3 - 1, sz = code / 9 - 1;
    double x = P0.x, y = P0.y, z = P0.z;
    if (pts64) {
        x = pts64[3 * (int64_t)p];
        y = pts64[3 * (int64_t)p + 1];
        z = pts64[3 * (int64_t)p + 2];
    }
    x -= sx * boxd;
    y -= sy * boxd;
    z -= sz * boxd;
    const float hx = (float)x, hy = (float)y, hz = (float)z;
    img[code] = make_float4(hx, hy, hz, 0.f);
    img[27 + code] = make_float4((float)(x - hx), (float)(y - hy), (float)(z - hz), 0.f);
}

// Separation of one list entry from the primary (image img[code]), rotated
// to the primary's line of sight in radial mode, as a unit vector and weight.
template <bool EXACT>
__device__ __forceinline__ void pair_dir(const ListArgs& a, int p, bool close, const float4& q, unsigned e,
                                         const float4* img, const float* R, int radial, float& z, float& ux,
                                         float& uy, float& w) {
    float dx = 1.f, dy = 0.f, dz = 0.f;
    w = 0.f;
    if (e != kNoPair) {
        const float4 o = img[e >> kIdxBits];
        dx = q.x - o.x;
        dy = q.y - o.y;
        dz = q.z - o.z;
        if constexpr (EXACT) {  // the tail of the image (nonzero across a box face)
            const float4 ol = img[27 + (e >> kIdxBits)];
            dx -= ol.x;
            dy -= ol.y;
            dz -= ol.z;
        }
        if (close && fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= close_r2(a.bins, a.pts64)) {
            double s[4];
            close_sep(a.pts, a.pts64, p, e, a.g.boxd, s);
            dx = (float)s[0];
            dy = (float)s[1];
            dz = (float)s[2];
        }
        w = q.w;
        if (radial) {
            const float rx = fmaf(R[0], dx, fmaf(R[1], dy, R[2] * dz));
            const float ry = fmaf(R[3], dx, fmaf(R[4], dy, R[5] * dz));
            const float rz = fmaf(R[6], dx, fmaf(R[7], dy, R[8] * dz));
            dx = rx;
            dy = ry;
            dz = rz;
        }
    }
    const float rinv = rsqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
    z = dz * rinv;
    ux = dx * rinv;
    uy = dy * rinv;
}

// Reduce the Chebyshev-form partials over the warp into res_b (accumulator
// slot layout: m = 0 slot k; m >= 1 slot acc_base(m) + 2k + part).
template <int L>
__device__ __forceinline__ void reduce_cheb(float (&acc0)[L + 1], float2 (&accc)[Cheb<L>::NC > 0 ? Cheb<L>::NC : 1],
                                            int lane, float* res_b) {
    constexpr int NR = Shape<L>::NR;
    float acc[NR];  // the (Re, Im) pairs first, then m = 0 (see emit_row)
    static_for<0, Cheb<L>::NC>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        acc[2 * i] = accc[i].x;
        acc[2 * i + 1] = accc[i].y;
    });
    static_for<0, L + 1>([&](auto kc) {
        constexpr int k = decltype(kc)::value;
        acc[2 * Cheb<L>::NC + k] = acc0[k];
    });
    butterfly_add<L>(acc, lane, res_b);
}

// Per-warp shared memory of k_accum / k_adj: img[27] float4 and its low parts
// imglo[27] float4 (below), R[16] float, point ring [kPtRing][32] float4, entry
// ring [kEntRing][32] uint, res[B][res_stride(NRP)] float.
constexpr int kImgBytes = 2 * 27 * 16;
constexpr int kEntRing = 8;
constexpr int kPtRing = 4;
__host__ __device__ constexpr size_t accum_smem_per_warp(int B, int NRP) {
    return (((size_t)B * res_stride(NRP) * 4 + 15) & ~(size_t)15) + kImgBytes + 64 + kEntRing * 32 * 4 + kPtRing * 32 * 16;
}

// The row of A of one primary from the per-bin Chebyshev sums res (Legendre-form
// connection times K_lm), and, when asked for, the tensor-core operands: sqrt(w)
// times the row split into bf16 hi and lo (the operations of the contraction's
// converter warps) at the row's padded position inside its catalog.  One table
// entry per complex column: Re and Im share the coefficients, their sums are one
// 8-byte load.  Two entries per lane, chains unrolled: the warp runs this tail with
// fewer FMA warps beside it, so its latency counts.  20,000 primaries at B = lmax =
// 10: the kernel takes 298 us, 320 with a chain per real column.  Out of line, so
// that the register allocation of the pair loop does not see it.
template <int L>
__device__ __noinline__ void emit_row(const ListArgs& a, const float* res, int row, int p, float w, int lane) {
    constexpr int NT = L / 2 + 1, U = 2;
    float* Arow = a.A + (int64_t)row * a.RLP;
    __nv_bfloat16 *Bh = nullptr, *Bl = nullptr;
    if (a.bop) {
        const int4 bc = __ldg(a.bcat + (a.nbcat == 1 ? 0 : (int)(a.key[p] / (unsigned long long)a.g.cells_per_cat)));
        Bh = a.bop + ((int64_t)bc.x + (row - bc.y)) * 2 * a.bop_pitch;
        Bl = Bh + a.bop_pitch;
    }
    const bool fp32 = !a.bop || !a.skip_a;
    const float sw = sqrtf(w);
    auto put = [&](int col, int opcol, float v) {
        if (fp32) Arow[col] = v;
        if (Bh) {
            const float y = __fmul_rn(v, sw);
            const __nv_bfloat16 h = __float2bfloat16_rn(y);
            Bh[opcol] = h;
            Bl[opcol] = __float2bfloat16_rn(__fsub_rn(y, __bfloat162float(h)));
        }
    };
    const int ne = a.nrowconv;
    for (int e0 = lane; e0 < ne; e0 += 32 * U) {
        int4 t[U];
        float2 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            t[u] = e0 + 32 * u < ne ? __ldg(a.rowconv + e0 + 32 * u) : make_int4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float4* cf = reinterpret_cast<const float4*>(a.rowcoef + 8 * t[u].y);
            const float4 c0 = __ldg(cf);
            float4 c1 = c0;
            if constexpr (NT > 4) c1 = __ldg(cf + 1);
            const float2* r = reinterpret_cast<const float2*>(res + (t[u].x & 0xffff));
            const int n = (t[u].x >> 16) & 0xff, step = t[u].x >> 24;
            v[u] = make_float2(0.f, 0.f);
            static_for<0, NT>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                const float4& c4 = k < 4 ? c0 : c1;
                const float c = (k & 3) == 0 ? c4.x : (k & 3) == 1 ? c4.y : (k & 3) == 2 ? c4.z : c4.w;
                if (k < n) v[u] = __ffma2_rn(make_float2(c, c), r[k * step], v[u]);
            });
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int K = t[u].z >> 16, col = t[u].z & 0xffff, oc = t[u].w;
            if (e0 + 32 * u < ne) {
                if (K > 0) {  // m >= 1: Re, and Im K columns behind it
                    put(col, oc, v[u].x);
                    put(col + K, oc + K, v[u].y);
                } else {  // m = 0: the sums of an even and an odd T_k share a word pair
                    put(col, oc, K < 0 ? v[u].y : v[u].x);
                }
            }
        }
    }
}

// Resident CTAs: three without a bound leave the call behind pair_dir's close pairs more
// registers than the sums need (30,000 uniform points, lmax = 6: 0.367 ms, 0.314 with four;
// 0.181 and 0.167 with six at lmax = 2).
template <int L, bool EXACT>
__global__ void __launch_bounds__(kLThreads, L <= 2 ? 6 : (L <= 4 ? 5 : (L <= 6 ? 4 : 3))) k_accum(ListArgs a) {
    constexpr int NRP = Shape<L>::NRP, RS = res_stride(NRP);
    extern __shared__ __align__(16) unsigned char la_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int B = a.bins.nbins;
    unsigned char* base = la_raw + (size_t)wid * accum_smem_per_warp(B, NRP);
    float4* img = reinterpret_cast<float4*>(base);
    float* Rs = reinterpret_cast<float*>(base + kImgBytes);
    float4* pring = reinterpret_cast<float4*>(base + kImgBytes + 64);
    unsigned* ering = reinterpret_cast<unsigned*>(base + kImgBytes + 64 + kPtRing * 32 * 16);
    float* res = reinterpret_cast<float*>(base + kImgBytes + 64 + kPtRing * 32 * 16 + kEntRing * 32 * 4);
    const Grid& g = a.g;
    const int close_end = close_bins(a.bins, a.pts64);
    const int qa = a.qrange ? a.qrange[0] : a.qa, qb = a.qrange ? a.qrange[1] : a.qb;
    for (;;) {
        int q = 0;
        if (lane == 0) q = qa + atomicAdd(a.queue, 1);
        q = __shfl_sync(kFull, q, 0);
        if (q >= qb) break;
        const int p = a.plist ? a.plist[q] : q;
        const float4 P0 = a.pts[p];
        if (lane < 27) set_image(img, lane, P0, a.pts64, p, g.boxd);
        if (lane < 9) {
            double x0 = P0.x, x1 = P0.y, x2 = P0.z;
            if (a.pts64) {
                x0 = a.pts64[3 * (int64_t)p];
                x1 = a.pts64[3 * (int64_t)p + 1];
                x2 = a.pts64[3 * (int64_t)p + 2];
            }
            Rs[lane] = g.radial ? los_rotation_entry(lane, x0, x1, x2, g.boxd)
                                : ((lane % 4 == 0) ? 1.f : 0.f);
        }
        const int cb = a.base[q] < 0 ? 0 : a.base[q];
        const int nch = a.nchunks[q];
        const int* chunks = a.chunks + (int64_t)cb * kChunk;
        const int* ordp = a.ord + cb;
        for (int k = lane; k < B * RS; k += 32) res[k] = 0.f;
        __syncwarp();
        if (nch > 0) {
            // List slot i = chunk (low 26 bits) | bin << 26.  Copies in flight
            // (cp.async groups): entries up to slot i+4, points up to slot i+2.
            auto ent_async = [&](int i, unsigned o) {
                cp_async4(ering + (i & (kEntRing - 1)) * 32 + lane,
                          chunks + (int64_t)(o & 0x3ffffffu) * kChunk + lane);
            };
            auto pt_async = [&](int i) {
                const unsigned e = ering[(i & (kEntRing - 1)) * 32 + lane];
                const bool v = e != kNoPair;
                cp_async16(pring + (i & (kPtRing - 1)) * 32 + lane, a.pts + (v ? (e & kIdxMask) : 0u), v);
            };
            auto slot = [&](int i) -> unsigned { return i < nch ? (unsigned)__ldg(ordp + i) : 0u; };
            unsigned o0 = slot(0), o1 = slot(1), o2 = slot(2), o3 = slot(3);
            ent_async(0, o0);
            if (nch > 1) ent_async(1, o1);
            cp_async_commit();
            cp_async_wait<0>();
            pt_async(0);
            if (nch > 2) ent_async(2, o2);
            cp_async_commit();
            if (nch > 1) pt_async(1);
            if (nch > 3) ent_async(3, o3);
            cp_async_commit();
            // slot words of i .. i+3 in registers, i+4 .. i+6 loading
            unsigned s4 = slot(4), s5 = slot(5), s6 = slot(6);
            unsigned sA = o0, sB = o1, sC = o2, sD = o3;
            constexpr int NC = Cheb<L>::NC > 0 ? Cheb<L>::NC : 1;
            float acc0[L + 1];
            float2 accc[NC];
            auto clear = [&]() {
                static_for<0, L + 1>([&](auto kc) { acc0[decltype(kc)::value] = 0.f; });
                static_for<0, NC>([&](auto ic) { accc[decltype(ic)::value] = make_float2(0.f, 0.f); });
            };
            clear();
            int curb = (int)(sA >> 26);
            for (int i = 0; i < nch; ++i) {
                cp_async_wait<1>();  // entries of i+2 and points of i have landed
                if (i + 2 < nch) pt_async(i + 2);
                if (i + 4 < nch) ent_async(i + 4, s4);
                cp_async_commit();
                const unsigned s7 = slot(i + 7);
                const int bA = (int)(sA >> 26);
                if (bA != curb) {  // the bin changes: reduce the partials of the last one
                    reduce_cheb<L>(acc0, accc, lane, res + curb * RS);
                    clear();
                    curb = bA;
                }
                {
                    const unsigned e = ering[(i & (kEntRing - 1)) * 32 + lane];
                    const float4 qv = pring[(i & (kPtRing - 1)) * 32 + lane];
                    float z, ux, uy, w;
                    pair_dir<EXACT>(a, p, bA < close_end, qv, e, img, Rs, g.radial, z, ux, uy, w);
                    accum_pair_cheb<L>(acc0, accc, z, ux, uy, w);
                }
                sA = sB;
                sB = sC;
                sC = sD;
                sD = s4;
                s4 = s5;
                s5 = s6;
                s6 = s7;
            }
            cp_async_wait<0>();
            reduce_cheb<L>(acc0, accc, lane, res + curb * RS);
        }
        __syncwarp();
        const int row = a.chunked ? q - a.q0 : a.orig[p];
        emit_row<L>(a, res, row, p, P0.w, lane);
        if (lane == 0) a.wrow[row] = P0.w;
        __syncwarp();
    }
}

// The accumulate kernel of plain forwards: the lists hold direction records
// (k_scan), so a chunk costs one 16-byte copy and one shared-memory load per lane
// and the harmonics.  Bound by issue: at lmax = 10 a chunk's 55 packed FMAs take
// two issue cycles each, the recurrences of T_k and (x + iy)^m about 65 more, the
// list walk about 30; the loop body without any load measures 208 cycles per chunk
// and SM quarter, the kernel 226 (the form that gathers points from list entries:
// 310).  200,000 clustered points (L = 696, 4.0e9 pairs, lmax = 10): 24.5 ms
// against 33.8.  The list words of 32 chunks are held one per lane and read by
// shuffle (a load per chunk: 0.7 ms more).  20,000 uniform points (67 pairs per
// bin): 298 us, of which the butterflies are 86 and the rows of A 70.
constexpr int kDirRing = 8;
__host__ __device__ constexpr size_t accum_dir_smem_per_warp(int B, int NRP) {
    return (((size_t)B * res_stride(NRP) * 4 + 15) & ~(size_t)15) + kDirRing * 32 * 16;
}
template <int L>
__global__ void __launch_bounds__(kLThreads, 3) k_accum_dir(ListArgs a) {
    constexpr int NRP = Shape<L>::NRP, RS = res_stride(NRP);
    extern __shared__ __align__(16) unsigned char la_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int B = a.bins.nbins;
    unsigned char* base = la_raw + (size_t)wid * accum_dir_smem_per_warp(B, NRP);
    float4* ring = reinterpret_cast<float4*>(base) + lane;
    float* res = reinterpret_cast<float*>(base + kDirRing * 32 * 16);
    const int qa = a.qrange ? a.qrange[0] : a.qa, qb = a.qrange ? a.qrange[1] : a.qb;
    for (;;) {
        int q = 0;
        if (lane == 0) q = qa + atomicAdd(a.queue, 1);
        q = __shfl_sync(kFull, q, 0);
        if (q >= qb) break;
        const int p = a.plist ? a.plist[q] : q;
        const float w0 = a.pts[p].w;
        const int cb = a.base[q] < 0 ? 0 : a.base[q];
        const int nch = a.nchunks[q];
        const int nbc = nch > 0 && lane < B ? a.tag[cb + lane] : 0;  // chunks of bin lane
        const float4* recs = a.dirs + (int64_t)cb * kChunk + lane;
        const int* ordp = a.ord + cb;
        for (int k = lane; k < B * RS; k += 32) res[k] = 0.f;
        __syncwarp();
        if (nch > 0) {
            // every lane copies and reads its own record: the ring needs no barrier
            auto copy = [&](int i, unsigned o) {
                cp_async16_cg(ring + (i & (kDirRing - 1)) * 32, recs + (o & 0x3ffffffu) * kChunk);
            };
            auto slot = [&](int i) -> unsigned { return i < nch ? (unsigned)__ldg(ordp + i) : 0u; };
#pragma unroll
            for (int k = 0; k < kDirRing - 1; ++k) {
                if (k < nch) copy(k, slot(k));
                cp_async_commit();
            }
            // list words: 32 chunks' in the lanes, the next 32 loading
            unsigned ow = slot(lane), ow2 = slot(32 + lane);
            constexpr int NC = Cheb<L>::NC > 0 ? Cheb<L>::NC : 1;
            int i = 0;
            for (int b = 0; b < B; ++b) {
                const int end = i + __shfl_sync(kFull, nbc, b);
                if (end == i) continue;
                float acc0[L + 1];
                float2 accc[NC];
                static_for<0, L + 1>([&](auto kc) { acc0[decltype(kc)::value] = 0.f; });
                static_for<0, NC>([&](auto ic) { accc[decltype(ic)::value] = make_float2(0.f, 0.f); });
                for (; i < end; ++i) {
                    cp_async_wait<kDirRing - 2>();  // the records of chunk i have landed
                    const float4 v = ring[(i & (kDirRing - 1)) * 32];
                    const int ic = i + kDirRing - 1;
                    if ((ic & 31) == 0) {
                        ow = ow2;
                        ow2 = slot(ic + 32 + lane);
                    }
                    const unsigned o = __shfl_sync(kFull, ow, ic & 31);
                    if (ic < nch) copy(ic, o);
                    cp_async_commit();
                    accum_pair_cheb<L>(acc0, accc, v.x, v.y, v.z, v.w);
                }
                reduce_cheb<L>(acc0, accc, lane, res + b * RS);
            }
            cp_async_wait<0>();
        }
        __syncwarp();
        const int row = a.chunked ? q - a.q0 : a.orig[p];
        emit_row<L>(a, res, row, p, w0, lane);
        if (lane == 0) a.wrow[row] = w0;
        __syncwarp();
    }
}

// Adjoint pair pass over the pair lists (the derivative of Sec. 3.1's a_lm
// with the pair set and bins held fixed).  Per primary i and bin b the adjoint
// multipoles H_lm = w_i K_lm V_i (V = M A, slot layout) are carried to the
// Chebyshev form, G_{m,k} = sum_l c^(m)_{l-m,k} H_lm (the transpose of the
// forward's connection), so that for a pair with unit separation (x, y, z)
//     F = sum_{m,k} Re(conj(G_{m,k}) T_k(z) (x + iy)^m)
// with dF/dz through T_k' = k U_{k-1} and dF/dx, dF/dy through (x + iy)^m.
// Secondary j receives dL/dw_j += 2F and dL/dpos_j += g, primary i gets -g,
// g = (2 w_j / r)(grad F - (grad F . d) d) (FP64 atomics; the primary's share
// is summed per lane and reduced once).
template <int L>
__global__ void __launch_bounds__(kLThreads) k_adj(ListArgs a) {
    constexpr int NR = Shape<L>::NR, NRP = Shape<L>::NRP;
    extern __shared__ __align__(16) unsigned char la_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int B = a.bins.nbins;
    unsigned char* base = la_raw + (size_t)wid * accum_smem_per_warp(B, NRP);
    float4* img = reinterpret_cast<float4*>(base);
    float4* pring = reinterpret_cast<float4*>(base + kImgBytes + 64);
    unsigned* ering = reinterpret_cast<unsigned*>(base + kImgBytes + 64 + kPtRing * 32 * 16);
    float* G = reinterpret_cast<float*>(base + kImgBytes + 64 + kPtRing * 32 * 16 + kEntRing * 32 * 4);
    const Grid& g = a.g;
    const int close_end = close_bins(a.bins, a.pts64);
    const int qa = a.qrange ? a.qrange[0] : a.qa, qb = a.qrange ? a.qrange[1] : a.qb;
    for (;;) {
        int q = 0;
        if (lane == 0) q = qa + atomicAdd(a.queue, 1);
        q = __shfl_sync(kFull, q, 0);
        if (q >= qb) break;
        const int p = a.plist ? a.plist[q] : q;
        const float4 P0 = a.pts[p];
        if (lane < 27) set_image(img, lane, P0, a.pts64, p, g.boxd);
        const int row = a.orig[p];
        const float* Vrow = a.V + (int64_t)(a.chunked ? q - a.q0 : row) * a.RLP;
        for (int idx = lane; idx < B * NR; idx += 32) {
            const int b = idx / NR, sl = idx - b * NR;
            const int4 cv = __ldg(a.slotconv + sl);
            float v = 0.f;
            for (int t = 0; t < cv.z; ++t) v = fmaf(__ldg(a.slotcoef + cv.w + t), __ldg(Vrow + cv.x + b + t * cv.y), v);
            G[b * NRP + sl] = P0.w * v;
        }
        const int cb = a.base[q] < 0 ? 0 : a.base[q];
        const int nch = a.nchunks[q];
        const int* chunks = a.chunks + (int64_t)cb * kChunk;
        const int* ordp = a.ord + cb;
        __syncwarp();
        double di0 = 0.0, di1 = 0.0, di2 = 0.0;  // -dL/dpos_i, this lane's share
        if (nch > 0) {
            auto ent_async = [&](int i, unsigned o) {
                cp_async4(ering + (i & (kEntRing - 1)) * 32 + lane,
                          chunks + (int64_t)(o & 0x3ffffffu) * kChunk + lane);
            };
            auto pt_async = [&](int i) {
                const unsigned e = ering[(i & (kEntRing - 1)) * 32 + lane];
                const bool v = e != kNoPair;
                cp_async16(pring + (i & (kPtRing - 1)) * 32 + lane, a.pts + (v ? (e & kIdxMask) : 0u), v);
            };
            auto slot = [&](int i) -> unsigned { return i < nch ? (unsigned)__ldg(ordp + i) : 0u; };
            unsigned o0 = slot(0), o1 = slot(1), o2 = slot(2), o3 = slot(3);
            ent_async(0, o0);
            if (nch > 1) ent_async(1, o1);
            cp_async_commit();
            cp_async_wait<0>();
            pt_async(0);
            if (nch > 2) ent_async(2, o2);
            cp_async_commit();
            if (nch > 1) pt_async(1);
            if (nch > 3) ent_async(3, o3);
            cp_async_commit();
            unsigned s4 = slot(4), s5 = slot(5), s6 = slot(6);
            unsigned sA = o0, sB = o1, sC = o2, sD = o3;
            float pix = 0.f, piy = 0.f, piz = 0.f;
            int curb = (int)(sA >> 26);
            for (int i = 0; i < nch; ++i) {
                cp_async_wait<1>();
                if (i + 2 < nch) pt_async(i + 2);
                if (i + 4 < nch) ent_async(i + 4, s4);
                cp_async_commit();
                const unsigned s7 = slot(i + 7);
                const int bA = (int)(sA >> 26);
                if (bA != curb) {
                    di0 -= pix;
                    di1 -= piy;
                    di2 -= piz;
                    pix = piy = piz = 0.f;
                    curb = bA;
                }
                const unsigned e = ering[(i & (kEntRing - 1)) * 32 + lane];
                if (e != kNoPair) {
                    const float4 qv = pring[(i & (kPtRing - 1)) * 32 + lane];
                    const float4 o = img[e >> kIdxBits], ol = img[27 + (e >> kIdxBits)];
                    const int jj = __ldg(a.orig + (e & kIdxMask));
                    float dx = (qv.x - o.x) - ol.x, dy = (qv.y - o.y) - ol.y, dz = (qv.z - o.z) - ol.z, sep = 1.f;
                    if (bA < close_end && fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= close_r2(a.bins, a.pts64)) {
                        double s[4];
                        close_sep(a.pts, a.pts64, p, e, g.boxd, s);
                        dx = (float)s[0];
                        dy = (float)s[1];
                        dz = (float)s[2];
                        sep = (float)s[3];
                    }
                    const float rinv = rsqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));  // sep / r
                    const float z = dz * rinv, ux = dx * rinv, uy = dy * rinv;
                    const float* Gb = G + bA * NRP;
                    // T_k(z) and T_k'(z) = k U_{k-1}(z)
                    float T[L + 1], D[L + 1];
                    T[0] = 1.f;
                    D[0] = 0.f;
                    if constexpr (L >= 1) {
                        T[1] = z;
                        D[1] = 1.f;
                        const float z2 = z + z;
                        float u0 = 1.f, u1 = z2;  // U_0, U_1
                        static_for<2, L + 1>([&](auto kc) {
                            constexpr int k = decltype(kc)::value;
                            T[k] = fmaf(z2, T[k - 1], -T[k - 2]);
                            D[k] = (float)k * u1;  // k U_{k-1}
                            const float u2 = fmaf(z2, u1, -u0);
                            u0 = u1;
                            u1 = u2;
                        });
                    }
                    float F = 0.f, Fz = 0.f, Fx = 0.f, Fy = 0.f;
                    static_for<0, L + 1>([&](auto kc) {
                        constexpr int k = decltype(kc)::value;
                        const float gk = Gb[k];
                        F = fmaf(gk, T[k], F);
                        Fz = fmaf(gk, D[k], Fz);
                    });
                    float pr = 1.f, pim = 0.f;  // (x + iy)^(m-1)
                    static_for<1, L + 1>([&](auto mc) {
                        constexpr int m = decltype(mc)::value;
                        constexpr int b0 = acc_base(L, m);
                        float2 gm = make_float2(0.f, 0.f), gz = make_float2(0.f, 0.f);
                        static_for<0, L - m + 1>([&](auto kc) {
                            constexpr int k = decltype(kc)::value;
                            const float2 gg = *reinterpret_cast<const float2*>(Gb + b0 + 2 * k);
                            gm = __ffma2_rn(make_float2(T[k], T[k]), gg, gm);
                            gz = __ffma2_rn(make_float2(D[k], D[k]), gg, gz);
                        });
                        const float ur = fmaf(pr, ux, -pim * uy), ui = fmaf(pr, uy, pim * ux);  // (x+iy)^m
                        F = fmaf(gm.x, ur, fmaf(gm.y, ui, F));
                        Fz = fmaf(gz.x, ur, fmaf(gz.y, ui, Fz));
                        Fx = fmaf((float)m, fmaf(gm.x, pr, gm.y * pim), Fx);
                        Fy = fmaf((float)m, fmaf(gm.y, pr, -gm.x * pim), Fy);
                        pr = ur;
                        pim = ui;
                    });
                    const float gdr = fmaf(Fx, ux, fmaf(Fy, uy, Fz * z));
                    const float sc = 2.f * qv.w * (sep * rinv);
                    const float gx = sc * fmaf(-gdr, ux, Fx), gy = sc * fmaf(-gdr, uy, Fy),
                                gz3 = sc * fmaf(-gdr, z, Fz);
                    atomicAdd(a.dw + jj, f2d_exact(2.f * F));
                    atomicAdd(a.dpos + 3 * (int64_t)jj, f2d_exact(gx));
                    atomicAdd(a.dpos + 3 * (int64_t)jj + 1, f2d_exact(gy));
                    atomicAdd(a.dpos + 3 * (int64_t)jj + 2, f2d_exact(gz3));
                    pix += gx;
                    piy += gy;
                    piz += gz3;
                }
                sA = sB;
                sB = sC;
                sC = sD;
                sD = s4;
                s4 = s5;
                s5 = s6;
                s6 = s7;
            }
            cp_async_wait<0>();
            di0 -= pix;
            di1 -= piy;
            di2 -= piz;
        }
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

template <int L>
int launch_adj_t(const ListArgs& a, int nsm, cudaStream_t st) {
    const size_t smem = accum_smem_per_warp(a.bins.nbins, Shape<L>::NRP) * kLWarps;
    if (cudaFuncSetAttribute(k_adj<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return -1;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_adj<L>, kLThreads, smem) != cudaSuccess ||
        per_sm < 1)
        return -1;
    int blocks = per_sm * nsm;
    const int need = (a.qb - a.qa + kLWarps - 1) / kLWarps;
    if (!a.qrange && blocks > need) blocks = need > 0 ? need : 1;
    k_adj<L><<<blocks, kLThreads, smem, st>>>(a);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <int L, bool EXACT>
int launch_accum_e(const ListArgs& a, int nsm, cudaStream_t st) {
    const size_t smem = accum_smem_per_warp(a.bins.nbins, Shape<L>::NRP) * kLWarps;
    if (cudaFuncSetAttribute(k_accum<L, EXACT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
        cudaSuccess)
        return -1;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_accum<L, EXACT>, kLThreads, smem) !=
            cudaSuccess ||
        per_sm < 1)
        return -1;
    int blocks = per_sm * nsm;
    const int need = (a.qb - a.qa + kLWarps - 1) / kLWarps;
    if (!a.qrange && blocks > need) blocks = need > 0 ? need : 1;
    k_accum<L, EXACT><<<blocks, kLThreads, smem, st>>>(a);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <int L>
int launch_accum_dir_t(const ListArgs& a, int nsm, cudaStream_t st) {
    const size_t smem = accum_dir_smem_per_warp(a.bins.nbins, Shape<L>::NRP) * kLWarps;
    if (cudaFuncSetAttribute(k_accum_dir<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return -1;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_accum_dir<L>, kLThreads, smem) != cudaSuccess ||
        per_sm < 1)
        return -1;
    int blocks = per_sm * nsm;
    const int need = (a.qb - a.qa + kLWarps - 1) / kLWarps;
    if (!a.qrange && blocks > need) blocks = need > 0 ? need : 1;
    k_accum_dir<L><<<blocks, kLThreads, smem, st>>>(a);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <int L>
int launch_accum_t(const ListArgs& a, int nsm, cudaStream_t st) {
    if (a.dirs) return launch_accum_dir_t<L>(a, nsm, st);
    return a.exact_img ? launch_accum_e<L, true>(a, nsm, st) : launch_accum_e<L, false>(a, nsm, st);
}

template <int MODE, bool STAGED, bool F64>
int launch_scan_s(const ListArgs& a, int nsm, cudaStream_t st) {
    const size_t smem = sizeof(ScanSmem<MODE != kEntries, STAGED>) * kScanWarps;
    auto* k = k_scan<MODE, STAGED, F64>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return -1;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kScanThreads, smem) != cudaSuccess || per_sm < 1)
        return -1;
    int blocks = per_sm * nsm;
    const int need = (a.qb - a.qa + kScanWarps - 1) / kScanWarps;
    if (!a.qrange && blocks > need) blocks = need;
    k<<<blocks, kScanThreads, smem, st>>>(a);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}
// Above 1.5 cells per rmax about half of the candidates or more are pairs, and they
// are placed from the candidates' lanes; below, the accepted ones are gathered in
// groups of 32 first.  200,000 clustered points, scan direct / staged: 34.1 / 32.1 ms
// at 0.86 cells (27% pairs), 21.0 / 22.5 at 1.72 (47%), 16.8 / 19.7 at 3.74 (68%).
template <int MODE, bool F64>
int launch_scan_k(const ListArgs& a, int nsm, cudaStream_t st) {
    return a.bins.rmaxf * a.g.inv_cell < 1.5f ? launch_scan_s<MODE, true, F64>(a, nsm, st)
                                              : launch_scan_s<MODE, false, F64>(a, nsm, st);
}
template <bool F64>
int launch_scan_d(const ListArgs& a, int nsm, cudaStream_t st) {
    return a.g.radial ? launch_scan_k<kDirsRadial, F64>(a, nsm, st) : launch_scan_k<kDirs, F64>(a, nsm, st);
}

}  // namespace

int launch_count(const ListArgs& a, int nsm, cudaStream_t st) {
    if (a.qb <= a.qa) return 0;
    // lanes per primary: at least about 1,000 threads per SM
    const int rows = (2 * a.g.reach + 1) * (2 * a.g.reach + 1);
    int lpp = 1;
    while (lpp < 32 && lpp < rows && (int64_t)(a.qb - a.qa) * lpp < (int64_t)nsm * 1024) lpp *= 2;
    int64_t blocks = ((int64_t)(a.qb - a.qa) * lpp + kCountThreads - 1) / kCountThreads;
    if (blocks > nsm * 4) blocks = nsm * 4;  // (three atomics per block)
    k_count<<<(unsigned)blocks, kCountThreads, 0, st>>>(a, lpp);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_scan(const ListArgs& a, int nsm, cudaStream_t st) {
    if (!a.qrange && a.qb <= a.qa) return 0;
    if (!a.dirs) return launch_scan_k<kEntries, false>(a, nsm, st);
    return a.pts64 ? launch_scan_d<true>(a, nsm, st) : launch_scan_d<false>(a, nsm, st);
}

size_t plan_scan_tmp_bytes(int64_t n) { return 8 * (size_t)((n + kScan64 - 1) / kScan64 + 1); }

int launch_plan(const int* need, long long* gbase, long long* tmp, int qa, int qb, long long stride, int slack,
                int npass, int* base, int* passq, int* status, cudaStream_t st) {
    const int64_t n = (int64_t)qb - qa;
    if (n > 0) {
        const int nb = (int)((n + kScan64 - 1) / kScan64);
        k_need_sums<<<nb, kScan64, 0, st>>>(need + qa, n, tmp);
        k_need_top<<<1, kScan64, 0, st>>>(tmp, nb);
        k_need_final<<<nb, kScan64, 0, st>>>(need + qa, n, tmp, gbase);
    }
    k_plan_init<<<1, 256, 0, st>>>(passq, npass, qb);
    if (qb > qa) {
        int blocks = (qb - qa + 255) / 256;
        if (blocks > 4096) blocks = 4096;
        k_plan<<<blocks, 256, 0, st>>>(need, gbase, qa, qb, stride, slack, npass, base, passq, status);
    }
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_adj(int lmax, const ListArgs& a, int nsm, cudaStream_t st) {
    if (!a.qrange && a.qb <= a.qa) return 0;
    if (a.precise) return launch_adj_df(lmax, a, nsm, st);
    switch (lmax) {
        case 0: return launch_adj_t<0>(a, nsm, st);
        case 1: return launch_adj_t<1>(a, nsm, st);
        case 2: return launch_adj_t<2>(a, nsm, st);
        case 3: return launch_adj_t<3>(a, nsm, st);
        case 4: return launch_adj_t<4>(a, nsm, st);
        case 5: return launch_adj_t<5>(a, nsm, st);
        case 6: return launch_adj_t<6>(a, nsm, st);
        case 7: return launch_adj_t<7>(a, nsm, st);
        case 8: return launch_adj_t<8>(a, nsm, st);
        case 9: return launch_adj_t<9>(a, nsm, st);
        case 10: return launch_adj_t<10>(a, nsm, st);
        default: return -1;
    }
}

int launch_accum(int lmax, const ListArgs& a, int nsm, cudaStream_t st) {
    if (!a.qrange && a.qb <= a.qa) return 0;
    if (a.precise) return launch_accum_df(lmax, a, nsm, st);
    switch (lmax) {
        case 0: return launch_accum_t<0>(a, nsm, st);
        case 1: return launch_accum_t<1>(a, nsm, st);
        case 2: return launch_accum_t<2>(a, nsm, st);
        case 3: return launch_accum_t<3>(a, nsm, st);
        case 4: return launch_accum_t<4>(a, nsm, st);
        case 5: return launch_accum_t<5>(a, nsm, st);
        case 6: return launch_accum_t<6>(a, nsm, st);
        case 7: return launch_accum_t<7>(a, nsm, st);
        case 8: return launch_accum_t<8>(a, nsm, st);
        case 9: return launch_accum_t<9>(a, nsm, st);
        case 10: return launch_accum_t<10>(a, nsm, st);
        default: return -1;
    }
}

}  // namespace g3
