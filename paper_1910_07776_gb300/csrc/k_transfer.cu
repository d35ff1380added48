// Table 2 transfer (Sec. 5): the fits of each problem's training group of runs (one block per
// problem and optimization), then the predictions for its test program, ranking and scoring
// (one block per problem).
#include <float.h>

#include "rank_row.cuh"

namespace {

// ====================================================================== transfer (Table 2)
// A problem q trains on a group of runs: every before/after pair of every run, run by run in
// ascending before slot, a pair never spanning two runs.  The group's versions form one list
// of N (rs_group_layout); KA[q] is their Gram, Kx[q][t][u] the block between test row t and
// version u (dot products; squared distances for IBK).
// Ridge: the bordered dual system of each optimization, M = KA(pairs) + lambda I = L D L^T,
// then b and alpha as in the batched solvers, and the prediction b + sum_a alpha_a Kx[t][u_a].
// IBK: the mean label of the kIbkK pairs nearest to t.  Candidates: outside t's mask (all six
// with RS_RANK_ALL) and inside opt_mask; ranking, threshold, top-k and scoring as in the rank
// pass with the test program's own times.
constexpr int kTrPairs = RS_MAXPAIRS * RS_MAXRUNS;   // pairs of one fit
constexpr int kTrRows = RS_MAXV * RS_MAXRUNS;        // versions of one group
constexpr int kTrThreads = 128;
constexpr int kTrCoef = kTrPairs + 1;                // b, alpha[kTrPairs] per fit in the workspace

// The training group of a problem in shared memory: its versions' masks and log times, and
// the slot of each mask within each run (-1 if absent).
struct GroupSmem {
    double lt[kTrRows];
    uint8_t msk[kTrRows];
    int8_t slot[RS_MAXRUNS][RS_MAXV];
};

__device__ void load_group(GroupSmem& G, const int64_t* __restrict__ a_row, const uint8_t* __restrict__ a_masks,
                           const double* __restrict__ a_lt, int64_t g0, const int (&start)[RS_MAXRUNS + 1], int N) {
    for (int e = threadIdx.x; e < RS_MAXRUNS * RS_MAXV; e += blockDim.x) G.slot[e / RS_MAXV][e % RS_MAXV] = -1;
    for (int u = threadIdx.x; u < N; u += blockDim.x) {
        int r = 0;
        while (u >= start[r + 1]) ++r;
        const int64_t row = a_row[g0 + r] + (u - start[r]);
        G.msk[u] = a_masks[row] & 63;
        G.lt[u] = a_lt[row];
    }
    __syncthreads();
    for (int u = threadIdx.x; u < N; u += blockDim.x) {
        int r = 0;
        while (u >= start[r + 1]) ++r;
        G.slot[r][G.msk[u]] = (int8_t)(u - start[r]);
    }
    __syncthreads();
}

// The pairs of optimization j (one warp, 32 of the group's versions at a time): group version of
// each before side, and labels, run by run in ascending slot order.  Returns their number; more than
// kTrPairs (only possible with repeated masks) is reported.
__device__ int build_pairs(const GroupSmem& G, int j, int R, int N, const int (&start)[RS_MAXRUNS + 1], uint16_t* pu,
                           double* yl, int* dstatus, int q) {
    const int lane = threadIdx.x & 31;
    int np = 0;
    for (int u0 = 0; u0 < N; u0 += 32) {
        const int u = u0 + lane;
        int r = 0, w = -1;
        if (u < N) {
            while (u >= start[r + 1]) ++r;
            const int m = G.msk[u];
            w = (m >> j) & 1 ? -1 : G.slot[r][m | (1 << j)];
        }
        const unsigned b = __ballot_sync(0xffffffffu, w >= 0);
        const int at = np + __popc(b & ((1u << lane) - 1u));
        if (w >= 0) {
            if (at < kTrPairs) {
                pu[at] = (uint16_t)u;
                yl[at] = G.lt[u] - G.lt[start[r] + w];
            } else {
                rs_dev_flag(dstatus, RS_EDATA, q);
            }
        }
        np += __popc(b);
    }
    return np < kTrPairs ? np : kTrPairs;
}

struct M5Tree;

struct TransferArgs {
    const int64_t* group_off;
    int max_runs, stat_stride;
    int64_t n_runs;
    const int64_t* a_row;
    const int32_t* a_fw;
    const uint8_t* a_masks;
    const double* a_lt;
    const int64_t* b_row;
    const int32_t* b_fw;
    const uint8_t* b_masks;
    const double* b_lt;
    const double* KA;
    const double* Kx;
    int ld;
    double lambda;
    double* coef;                        // [Q][6][kTrCoef] ridge fits (written by the fit kernel)
    uint8_t* fst;                        // [Q][6] their status
    double* pred;                        // [Q][64][6] predictions (transfer_predict_kernel)
    int ibk, opt_mask, rank_all;
    int m5p;                             // the M5P model tree instead of ridge
    M5Tree* trees;                       // [Q][6] M5P trees
    const double* ZA;                    // standardized training group rows (M5P fits)
    const int64_t* a_xo;
    const double* ZB;                    // standardized test rows (M5P predictions)
    const int64_t* b_xo;
    uint8_t* fit_status;
    RankPassArgs r;                      // k, ktau, flags (without RS_RANK_ALL), outputs, counters
};

// Reciprocal of a nonzero finite double of either sign (rcp_newton on its magnitude).
__device__ __forceinline__ double rcp_newton_any(double d) {
    return d < 0.0 ? -rcp_newton(-d) : rcp_newton(d);
}

// One block per (problem, optimization): the ridge fit of that optimization's pairs.  The
// factor lives in shared memory (the lower triangle, packed: five blocks of 96 pairs an SM where a
// full square left room for two); right-looking LDL^T whose
// trailing update of each step is spread over all threads (16 row groups x 8 column lanes); the FP64
// pipe bounds it (540 fits of 96 pairs 374 -> 276 us, of which 200 are its instructions; two columns a
// step, with half the barriers, 273),
// reciprocal pivots from rcp_newton kept for the solves, then the two forward solves and the
// back solve of the bordered system, one thread per row.
__global__ void __launch_bounds__(kTrThreads)
transfer_fit_kernel(const TransferArgs a, int nmax) {
    extern __shared__ __align__(16) double fsm[];
    __shared__ GroupSmem G;
    __shared__ uint16_t pu[kTrPairs];
    __shared__ double yl[kTrPairs];
    __shared__ int np_s;
    __shared__ double bval;
    __shared__ double red[8];
    const int q = blockIdx.x, j = blockIdx.y, tid = threadIdx.x;
    auto tri = [](int i) { return i * (i + 1) / 2; };         // row i of the packed lower triangle
    double* M = fsm;
    double* col = M + tri(nmax);
    double* lrow = col + nmax;
    double* ty = lrow + nmax;
    double* t1 = ty + nmax;
    double* dinv = t1 + nmax;
    int start[RS_MAXRUNS + 1], F = 0;
    const int N = rs_group_layout(q, a.group_off, a.max_runs, a.n_runs, a.a_row, a.a_fw, a.b_fw, a.stat_stride, start, F);
    if (N < 0 || N > a.ld) return;                 // reported by the predict / rank kernel
    const int64_t g0 = a.group_off[q];
    const int R = (int)(a.group_off[q + 1] - g0);
    load_group(G, a.a_row, a.a_masks, a.a_lt, g0, start, N);
    if (tid < 32) {
        const int np = build_pairs(G, j, R, N, start, pu, yl, nullptr, q);
        if (tid == 0) np_s = np;
    }
    __syncthreads();
    const int n = np_s;
    double* out = a.coef + ((int64_t)q * RS_NOPT + j) * kTrCoef;
    uint8_t* st_out = a.fst + (int64_t)q * RS_NOPT + j;
    if (n == 0 || n > nmax) {                      // n > nmax: more pairs than the hint allowed
        if (tid == 0) *st_out = n == 0 ? RS_FIT_EMPTY : RS_FIT_NOTPD;
        return;
    }
    if (n == 1) {                                  // one pair: alpha = 0, b = its label
        if (tid == 0) {
            out[0] = yl[0];
            out[1] = 0.0;
            *st_out = finite_bits(yl[0]) ? RS_FIT_OK : RS_FIT_NONFINITE;
        }
        return;
    }
    const double* KAq = a.KA + (int64_t)q * a.ld * a.ld;
    for (int e = tid; e < n * n; e += kTrThreads) {
        const int i = e / n, c = e - i * n;
        if (c <= i) M[tri(i) + c] = __ldg(KAq + (int64_t)pu[i] * a.ld + pu[c]) + (i == c ? a.lambda : 0.0);
    }
    __syncthreads();
    const int ty8 = tid >> 3, tx8 = tid & 7;
    int st = RS_FIT_OK;
    for (int k = 0; k < n; ++k) {
        const double d = M[tri(k) + k];
        if (!pos_finite(d)) {                      // every thread read the same pivot
            st = RS_FIT_NOTPD;
            break;
        }
        const double di = rcp_newton(d);
        if (tid == 0) dinv[k] = di;
        for (int i = k + 1 + tid; i < n; i += kTrThreads) {
            const double c = M[tri(i) + k];
            col[i] = c;
            lrow[i] = c * di;
            M[tri(i) + k] = c * di;
        }
        __syncthreads();
        for (int i = k + 1 + ty8; i < n; i += 16) {
            const double l = lrow[i];
            for (int c = k + 1 + tx8; c <= i; c += 8) M[tri(i) + c] = fma(-l, col[c], M[tri(i) + c]);
        }
        __syncthreads();
    }
    if (st == RS_FIT_OK) {
        if (tid < n) {                             // L t = rhs, two right-hand sides
            ty[tid] = yl[tid];
            t1[tid] = 1.0;
        }
        __syncthreads();
        for (int k = 0; k < n - 1; ++k) {
            if (tid > k && tid < n) {
                const double l = M[tri(tid) + k];
                ty[tid] = fma(-l, ty[k], ty[tid]);
                t1[tid] = fma(-l, t1[k], t1[tid]);
            }
            __syncthreads();
        }
        // num = t_1^T D^-1 t_y, den = t_1^T D^-1 t_1: per-thread terms, warp trees, then the
        // four warps' sums in order
        double pn = 0.0, pd = 0.0;
        if (tid < n) {
            const double sc = t1[tid] * dinv[tid];
            pn = sc * ty[tid];
            pd = sc * t1[tid];
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) {
            pn += __shfl_xor_sync(0xffffffffu, pn, o);
            pd += __shfl_xor_sync(0xffffffffu, pd, o);
        }
        if ((tid & 31) == 0) {
            red[tid >> 5] = pn;
            red[4 + (tid >> 5)] = pd;
        }
        __syncthreads();
        if (tid == 0) bval = ((red[0] + red[1]) + (red[2] + red[3])) * rcp_newton_any(((red[4] + red[5]) + (red[6] + red[7])));
        __syncthreads();
        const double b = bval;
        if (tid < n) ty[tid] = fma(-b, t1[tid], ty[tid]) * dinv[tid];
        __syncthreads();
        for (int k = n - 1; k > 0; --k) {          // L^T alpha = D^-1 (t_y - b t_1)
            if (tid < k) ty[tid] = fma(-M[tri(k) + tid], ty[k], ty[tid]);
            __syncthreads();
        }
        bool fin = true;
        if (tid < n) {
            out[1 + tid] = ty[tid];
            fin = finite_bits(ty[tid]);
        }
        if (tid == 0) out[0] = b;
        st = __syncthreads_and(fin) && finite_bits(b) ? RS_FIT_OK : RS_FIT_NONFINITE;
    }
    if (tid == 0) *st_out = (uint8_t)st;
}

// ====================================================================== M5P (Sec. 3.4)
// The model tree of each (problem, optimization), after the M5' description: grow by the
// standard deviation reduction (SDR), a linear model at every node on the attributes tested
// in its subtree as pruned so far (children are modelled and pruned first), simplified by
// greedy elimination, bottom-up pruning by estimated error, and smoothing on the way up at
// prediction time (k = 15).
//
// One block per fit.  What decides the tree is computed with the reference's own roundings (label
// sums in order, SDRs by IEEE division and square root), but only where it can matter: an SDR takes
// over a hundred FP64 instructions of 64 cycles each, and a node has up to 127 F candidate splits.  So
// every candidate is first bounded in FP32 (prefix sums by shuffles, an explicit error bound), and
// only those whose interval reaches the best one are evaluated exactly; a single survivor needs no
// evaluation.  The tree grows a level at a time: the (node, attribute) scans and partitions of a
// whole level are dealt to the eight warps, five block barriers a level instead of seven a node.
// Greedy elimination keeps the inverse H of the normal equations, the residuals and T = C H (C the
// centred attributes): dropping attribute d changes every residual by (w_d / H_dd) T_ad, so all the
// drop-one errors of a round cost m ns operations, and the round's winner is taken out by rank-one
// updates of H, w and T; the model that stays is solved again from scratch.  Not where attributes nearly
// make up one another (an entry G_kk H_kk, the variance inflation, beyond 2^kM5Inflated), nor where taking d
// out shrinks a diagonal entry of H by more than 2^kM5Shrink since H was last formed: what such updates
// leave of large entries is rounding, so the attributes that stay are solved from their own normal
// equations at once, and the elimination goes on from there.  With pairs of attributes 1e-5 of a deviation
// apart the updates alone chose wrong drops in 25 of 60 models, this form, as an inverse a round, in none.
// (Before: one thread per
// attribute walking every candidate's SDR, an inverse per round and every drop-one model applied to
// every instance, all serial over the nodes.)  Small nodes' models take one warp each.
// 36 problems x 3 runs x 37 attributes (96 instances a fit): 5532 -> 1351 us.
constexpr int kM5MaxN = kTrPairs;                 // instances of one fit
constexpr int kM5MaxNodes = 2 * kM5MaxN - 1;
constexpr int kM5MaxTerms = 64;
constexpr int kM5MaxFeat = 256;
constexpr int kM5Threads = 256;
constexpr int kM5Warps = kM5Threads / 32;
constexpr int kM5WarpTerms = 16, kM5WarpN = 32;   // models up to this size take one warp
constexpr int kM5WarpLd = kM5WarpTerms + 1;
constexpr int kM5WarpBuf = kM5WarpTerms * kM5WarpLd + kM5WarpN * kM5WarpLd +
                           (kM5WarpN * kM5WarpLd + 1) / 2;                   // H, C, T (FP32)
constexpr int kM5Surv = 1024;                     // candidate splits listed for exact evaluation, per level
constexpr double kM5SdFrac = 0.05, kM5Smooth = 15.0, kM5Ridge = 1e-8;
constexpr int kM5Shrink = 6;                      // bits that rank-one updates may take off an entry H_kk
constexpr int kM5Inflated = 16;                   // G_kk H_kk beyond 2^this: no rank-one updates

struct M5Tree {
    int n_nodes;
    int count[kM5MaxNodes];
    int nterm[kM5MaxNodes];
    int16_t attr[kM5MaxNodes], left[kM5MaxNodes], right[kM5MaxNodes], parent[kM5MaxNodes];
    double thr[kM5MaxNodes], b[kM5MaxNodes];
    int16_t term_attr[kM5MaxNodes][kM5MaxTerms];
    double term_w[kM5MaxNodes][kM5MaxTerms];
};

// Per group of threads (a warp, or the block): the vectors of one node's model.
template <int N>
struct M5Vec {
    double colk[N], rowk[N], zbar[N], r[N], w[N], wt[N], fac[N];
    int g0[N], h0[N];                             // G_kk and H_kk when H was last formed (high words)
    float fac32[N], rowk32[N], t32[N], e32[N];    // bounds of |T_ak|, and of the error of T in FP32
    int16_t cand[N];
    uint8_t sel[N];
    double e_cur, b;
    unsigned long long reach;                     // attributes whose drop may be the best
};

struct M5Smem {
    double y[kM5MaxN], y2[kM5MaxN];               // labels and their rounded squares
    const double* zp[kM5MaxN];                    // each instance's standardized row
    float yf[kM5MaxN];                            // labels less the root's mean, in FP32
    double thr[kM5MaxNodes], est[kM5MaxNodes];
    unsigned long long tested[kM5MaxNodes][kM5MaxFeat / 64];
    int16_t attr[kM5MaxNodes], left[kM5MaxNodes], right[kM5MaxNodes], parent[kM5MaxNodes];
    uint8_t lo[kM5MaxNodes], hi[kM5MaxNodes];
    uint8_t ids[kM5MaxN], side[kM5MaxN];
    int level[kM5MaxN + 2];                       // first node of each level
    int nn, nsurv;
    double sd_root;
    // the level's nodes (at most kM5MaxN / 2 that split), by node - first of the level
    float mean[kM5MaxN], tot[kM5MaxN], tot2[kM5MaxN], amax2[kM5MaxN], sda[kM5MaxN], ymax[kM5MaxN];
    float mean0;                                  // magnitude of the root's mean
    unsigned best_hi[kM5MaxN];                    // smallest upper bound of Q, as FP32 bits
    unsigned long long best_red[kM5MaxN];         // largest exact SDR, as FP64 bits
    unsigned best_key[kM5MaxN];                   // attribute << 8 | count of the chosen split
    int cnt[kM5MaxN];                             // survivors; -1: a leaf, -2: by the exact scan
    double s1[kM5MaxN], s2[kM5MaxN];              // exact label sums, in instance order
    unsigned surv[kM5Surv];                       // node << 16 | attribute << 8 | count
    float ql[kM5Surv];                            // their lower bounds of Q
    double red[kM5Surv];                          // their SDRs
    double rcp[kM5MaxN + 1];                      // 1 / c, rounded
    float errp[2][kM5Warps][kM5MaxTerms];
    double sump[kM5Warps];
    float res32[kM5Warps * 32];
    union {
        M5Vec<kM5MaxTerms> blk;
        M5Vec<kM5WarpTerms> wv[kM5Warps];
    } v;
};

// a / c rounded to nearest, y = 1 / c rounded to nearest: q = a y is within a unit of the quotient,
// its residual a - q c is exact in an FMA, and q + r y rounds to the quotient (P. Markstein,
// "Computation of elementary functions on the IBM RISC System/6000 processor", IBM J. Res. Dev. 34,
// 1990).  Three FP64 instructions; magnitudes whose residual could underflow, infinities and NaN take
// the division.
__device__ __forceinline__ double m5_div(double a, double c, double y) {
    const int ex = (__double2hiint(a) >> 20) & 0x7ff;
    if ((unsigned)(ex - 200) > 1600u && a != 0.0) return __ddiv_rn(a, c);
    const double q = __dmul_rn(a, y);
    return __fma_rn(__fma_rn(-q, c, a), y, q);
}

// The standard deviation from a count, sum and sum of squares: sqrt(max(0, (s2 - s1 s1 / c) / c)),
// with one rounding per operation (the reference's arithmetic).
__device__ __noinline__ double m5_sd(int c, double y, double s1, double s2) {
    const double cd = (double)c;
    const double v = m5_div(__dsub_rn(s2, m5_div(__dmul_rn(s1, s1), cd, y)), cd, y);
    return __dsqrt_rn(v > 0.0 ? v : 0.0);
}

__device__ __forceinline__ double m5_warp_sum(double x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Bounds of Q = sqrt(c l2 - l1^2) + sqrt((m - c) r2 - r1^2) (SDR = sd - Q / m) from FP32 prefix
// sums.  Each radicand's error is below 1e-5 n^2 A^2 for n labels of magnitude at most A: labels
// rounded to FP32 and shifted (1.8e-7 A each), sums by at most 12 additions (7e-7 each way), products.
// The exact evaluation works on the labels themselves, of magnitude up to Y: its own rounding, up to
// 6 c m^2 2^-53 Y^2 in a radicand, counts as well, as 6e-7 Y^2 in a2 (a2 = A^2 + 6e-7 Y^2; c >= 2, m <= 128).
__device__ __forceinline__ void m5_bounds(int c, int m, float l1, float l2, float t1, float t2, float a2, float& lo,
                                          float& hi) {
    const float cl = (float)c, cr = (float)(m - c);
    const float r1 = t1 - l1, r2 = t2 - l2;
    const float L = cl * l2 - l1 * l1, R = cr * r2 - r1 * r1;
    const float dl = 1e-5f * a2 * cl * cl, dr = 1e-5f * a2 * cr * cr;
    hi = (sqrtf(fmaxf(L, 0.f) + dl) + sqrtf(fmaxf(R, 0.f) + dr)) * 1.00001f;
    lo = (sqrtf(fmaxf(L - dl, 0.f)) + sqrtf(fmaxf(R - dr, 0.f))) * 0.99999f;
}

// A segment of W lanes (W = 32, or at least m) scans attribute f of a node (instances lo .. lo + m,
// level slot q; f < 0: no attribute for this segment): lowers the node's best upper bound of Q and
// lists the candidates whose lower bound reaches it as it then stands.
__device__ __forceinline__ void m5_scan(M5Smem& S, const uint8_t* srt, const uint8_t* rk, int f, int lo, int m, int q,
                                        int W) {
    const int lane = threadIdx.x & 31, sl = lane & (W - 1);
    const float mean = S.mean[q], t1 = S.tot[q], t2 = S.tot2[q], a2 = S.amax2[q];
    float c1 = 0.f, c2 = 0.f;
    for (int base = 0; base < m; base += W) {
        const int e = base + sl;
        const bool in = e < m && f >= 0;
        const int id = in ? srt[lo + e] : 0;
        const int nx = in && e + 1 < m ? srt[lo + e + 1] : id;
        const float v = in ? S.yf[id] - mean : 0.f;
        float s = v, w = v * v;
        for (int o = 1; o < W; o <<= 1) {
            const float a = __shfl_up_sync(0xffffffffu, s, o, W), b = __shfl_up_sync(0xffffffffu, w, o, W);
            if (sl >= o) {
                s += a;
                w += b;
            }
        }
        s += c1;
        w += c2;
        c1 = __shfl_sync(0xffffffffu, s, 31);      // (carried on for W = 32 only)
        c2 = __shfl_sync(0xffffffffu, w, 31);
        const int c = e + 1;
        float ql = 0.f, qh = __int_as_float(0x7f800000);
        const bool can = in && c >= 2 && m - c >= 2 && rk[nx] != rk[id];
        if (can) m5_bounds(c, m, s, w, t1, t2, a2, ql, qh);
        const unsigned low = __reduce_min_sync(0xffffffffu, __float_as_uint(qh));
        unsigned lim = 0;
        if (lane == 0) lim = low < 0x7f800000u ? atomicMin(&S.best_hi[q], low) : 0u;
        lim = __shfl_sync(0xffffffffu, lim, 0);
        if (can && ql <= __uint_as_float(lim < low ? lim : low)) {
            const int k = atomicAdd(&S.nsurv, 1);
            if (k < kM5Surv) {
                S.surv[k] = (unsigned)q << 16 | (unsigned)f << 8 | (unsigned)c;
                S.ql[k] = ql;
            }
        }
    }
}

// Every candidate of attribute f by the reference's arithmetic, one thread (labels that are not
// finite, or more survivors than fit): the best SDR > 0 of the attribute goes to best / key.
__device__ __noinline__ void m5_exact_scan(const M5Smem& S, const uint8_t* o, const uint8_t* rk, int f, int lo, int m,
                                           int q, double sd, double& best, unsigned& key) {
    double l1 = 0.0, l2 = 0.0;
    for (int c = 1; c < m; ++c) {
        const int ia = o[lo + c - 1], ib = o[lo + c];
        l1 = __dadd_rn(l1, S.y[ia]);
        l2 = __dadd_rn(l2, S.y2[ia]);
        if (rk[ia] == rk[ib] || c < 2 || m - c < 2) continue;
        const double sdl = m5_sd(c, S.rcp[c], l1, l2);
        const double sdr = m5_sd(m - c, S.rcp[m - c], __dsub_rn(S.s1[q], l1), __dsub_rn(S.s2[q], l2));
        const double red = __dsub_rn(sd, m5_div(__dadd_rn(__dmul_rn((double)c, sdl), __dmul_rn((double)(m - c), sdr)),
                                                (double)m, S.rcp[m]));
        if (red > best) {
            best = red;
            key = (unsigned)f << 8 | (unsigned)c;
        }
    }
}

// A group of threads working on one node's model: a warp, or the whole block.
template <bool WARP>
struct M5Group {
    static constexpr int kNT = WARP ? 32 : kM5Threads;
    static __device__ __forceinline__ int tid() { return WARP ? (int)(threadIdx.x & 31) : (int)threadIdx.x; }
    static __device__ __forceinline__ void sync() {
        if (WARP) __syncwarp();
        else __syncthreads();
    }
    static __device__ __forceinline__ bool any(bool x) {      // (also a barrier)
        if (!WARP) return __syncthreads_or(x) != 0;
        __syncwarp();
        return __any_sync(0xffffffffu, x) != 0;
    }
};

// In-place inverse of the nb x nb leading block of M (row stride ld) by Gauss-Jordan elimination
// without pivoting (the systems are symmetric positive definite).
template <bool WARP, class Vec>
__device__ void m5_invert(Vec& V, double* M, int ld, int nb) {
    using Gp = M5Group<WARP>;
    const int tid = Gp::tid();
    for (int k = 0; k < nb; ++k) {
        const double piv = rcp_newton_any(M[k * ld + k]);
        for (int i = tid; i < nb; i += Gp::kNT) {
            V.colk[i] = M[i * ld + k];
            V.rowk[i] = M[k * ld + i] * piv;
        }
        Gp::sync();
        for (int e = tid; e < nb * nb; e += Gp::kNT) {
            const int i = e / nb, j = e - i * nb;
            if (i == k && j == k) M[k * ld + k] = piv;
            else if (i == k) M[k * ld + j] = V.rowk[j];
            else if (j == k) M[i * ld + k] = -V.colk[i] * piv;
            else M[i * ld + j] = fma(-V.colk[i], V.rowk[j], M[i * ld + j]);
        }
        Gp::sync();
    }
}

// Estimated error of the node's model (V.b, V.w on V.sel) over its instances: mean |y - prediction|
// (m + v) / (m - v), v = terms + 1; DBL_MAX when m <= v.  One warp.
template <class Vec>
__device__ double m5_warp_err(const M5Smem& S, const Vec& V, int lo, int m, int nsel) {
    const int lane = threadIdx.x & 31;
    double acc = 0.0;
    for (int a = lane; a < m; a += 32) {
        const int i = S.ids[lo + a];
        const double* z = S.zp[i];
        double p = V.b;
        for (int q = 0; q < nsel; ++q) p = fma(V.w[q], __ldg(z + V.cand[V.sel[q]]), p);
        acc += fabs(S.y[i] - p);
    }
    acc = m5_warp_sum(acc);
    const int v = nsel + 1;
    if (m <= v) return DBL_MAX;
    return acc / m * ((double)(m + v) / (double)(m - v));
}

// H = inverse of the normal equations of V.sel[0 .. ns), w = H r, the intercept and e_cur.
template <bool WARP, class Vec>
__device__ void m5_solve(M5Smem& S, Vec& V, const double* C, double* H, int ld, int ns, int lo, int m, double ybar) {
    using Gp = M5Group<WARP>;
    const int tid = Gp::tid();
    for (int e = tid; e < ns * (ns + 1) / 2; e += Gp::kNT) {
        int f = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
        while (f * (f + 1) / 2 > e) --f;
        while ((f + 1) * (f + 2) / 2 <= e) ++f;
        const int g = e - f * (f + 1) / 2, cf = V.sel[f], cg = V.sel[g];
        double s = 0.0;
        for (int a = 0; a < m; ++a) s = fma(C[a * ld + cf], C[a * ld + cg], s);
        if (f == g) {
            s += kM5Ridge;
            V.g0[f] = __double2hiint(s);
        }
        H[f * ld + g] = s;
        H[g * ld + f] = s;
    }
    Gp::sync();
    m5_invert<WARP>(V, H, ld, ns);
    for (int i = tid; i < ns; i += Gp::kNT) {
        double s = 0.0;
        for (int k = 0; k < ns; ++k) s = fma(H[i * ld + k], V.r[V.sel[k]], s);
        V.w[i] = s;
    }
    Gp::sync();
    if (tid == 0) {
        double b = ybar;
        for (int i = 0; i < ns; ++i) b -= V.w[i] * V.zbar[V.sel[i]];
        V.b = b;
    }
    Gp::sync();
    if (WARP || threadIdx.x < 32) {
        const double e = m5_warp_err(S, V, lo, m, ns);
        if (tid == 0) V.e_cur = e;
    }
    Gp::sync();
}

// The estimated error of a node's model on attribute f (f < 0: none, the label mean) with the reference's
// operations in its order (instances ascending: an inner node's lie by its children), one rounding each.
// One thread.
__device__ __noinline__ double m5_exact_err(const M5Smem& S, int f, int lo, int m) {
    const double md = (double)m;
    unsigned long long in[kM5MaxN / 64] = {};
    for (int a = 0; a < m; ++a) {
        const int i = S.ids[lo + a];
#pragma unroll
        for (int w = 0; w < kM5MaxN / 64; ++w)
            if (i >> 6 == w) in[w] |= 1ull << (i & 63);
    }
    auto each = [&](auto&& take) {
#pragma unroll
        for (int w = 0; w < kM5MaxN / 64; ++w)
            for (unsigned long long x = in[w]; x; x &= x - 1) {
                const int i = 64 * w + __ffsll((long long)x) - 1;
                take(S.y[i], f >= 0 ? __ldg(S.zp[i] + f) : 0.0);
            }
    };
    double b = 0.0, w = 0.0;
    each([&](double y, double) { b = __dadd_rn(b, y); });
    b = __ddiv_rn(b, md);
    if (f >= 0) {
        double zbar = 0.0, g = 0.0, r = 0.0;
        each([&](double, double z) { zbar = __dadd_rn(zbar, z); });
        zbar = __ddiv_rn(zbar, md);
        each([&](double y, double z) {
            const double c = __dsub_rn(z, zbar);
            g = __dadd_rn(g, __dmul_rn(c, c));
            r = __dadd_rn(r, __dmul_rn(c, __dsub_rn(y, b)));
        });
        const double l = __dsqrt_rn(__dadd_rn(g, kM5Ridge));
        w = __ddiv_rn(__ddiv_rn(r, l), l);
        b = __dsub_rn(b, __dmul_rn(w, zbar));
    }
    const int v = f >= 0 ? 2 : 1;
    if (m <= v) return DBL_MAX;
    double e = 0.0;
    each([&](double y, double z) { e = __dadd_rn(e, fabs(__dsub_rn(y, f >= 0 ? __dadd_rn(b, __dmul_rn(w, z)) : b))); });
    return __dmul_rn(__ddiv_rn(e, md), __ddiv_rn((double)(m + v), (double)(m - v)));
}

// The model of internal node t on the attributes tested below it (the lowest kM5MaxTerms of them),
// greedily simplified, and the pruning decision.  H: tmax x ld; C, T32: m x ld.
template <bool WARP, class Vec>
__device__ __noinline__ void m5_model(M5Smem& S, Vec& V, M5Tree* T, int t, int F, double* H, double* C, float* T32, int ld) {
    using Gp = M5Group<WARP>;
    const int tid = Gp::tid(), lane = threadIdx.x & 31;
    const int wp = WARP ? 0 : (int)(threadIdx.x >> 5), nw = WARP ? 1 : kM5Warps;
    const int lo = S.lo[t], m = S.hi[t] - S.lo[t];
    // candidates: the attributes tested in the subtree, ascending
    int nc = 0;
    for (int w = 0; w < kM5MaxFeat / 64; ++w) {
        const unsigned long long bits = S.tested[t][w];
        for (int f = tid; f < 64; f += Gp::kNT)
            if ((bits >> f) & 1ull) {
                const int pos = nc + __popcll(bits & ((1ull << f) - 1ull));
                if (pos < kM5MaxTerms) V.cand[pos] = (int16_t)(64 * w + f);
            }
        nc += __popcll(bits);
    }
    nc = nc < kM5MaxTerms ? nc : kM5MaxTerms;
    double ybar = 0.0;
    for (int a = lane; a < m; a += 32) ybar += S.y[S.ids[lo + a]];
    ybar = m5_warp_sum(ybar) / m;
    Gp::sync();
    for (int e = tid; e < m * nc; e += Gp::kNT) {
        const int a = e / nc, k = e - a * nc;
        C[a * ld + k] = __ldg(S.zp[S.ids[lo + a]] + V.cand[k]);
    }
    Gp::sync();
    for (int k = wp; k < nc; k += nw) {            // a warp centres a column
        double s = 0.0, d = 0.0;
        for (int a = lane; a < m; a += 32) s += C[a * ld + k];
        s = m5_warp_sum(s) / m;
        for (int a = lane; a < m; a += 32) {
            const double c = C[a * ld + k] - s;
            C[a * ld + k] = c;
            d = fma(c, S.y[S.ids[lo + a]] - ybar, d);
        }
        d = m5_warp_sum(d);
        if (lane == 0) {
            V.zbar[k] = s;
            V.r[k] = d;
            V.sel[k] = (uint8_t)k;
        }
    }
    Gp::sync();
    m5_solve<WARP>(S, V, C, H, ld, nc, lo, m, ybar);
    unsigned long long alive = nc >= 64 ? ~0ull : (1ull << nc) - 1ull;
    int ns = nc;
    bool dropped = false;
    if (nc > 0 && m > nc) {                        // else no model with one attribute fewer has an estimate
        const int row = WARP ? lane : (int)threadIdx.x;
        float* res32 = S.res32 + (WARP ? 32 * (int)(threadIdx.x >> 5) : 0);
        double res = 0.0;
        bool formed = true;                        // H, w are those of the nc attributes' normal equations
        bool ill = false;                          // an attribute that the others nearly make up
        for (;;) {
            if (formed) {
                // residuals (lane = instance, kept by the warp that owns its 32 instances) and T = C H in FP32
                formed = false;
                if (row < m) {
                    double p = ybar;
                    for (int i = 0; i < nc; ++i) p = fma(C[row * ld + i], V.w[i], p);
                    res = S.y[S.ids[lo + row]] - p;
                    res32[row] = (float)res;
                }
                for (int e = tid; e < m * nc; e += Gp::kNT) {
                    const int a = e / nc, k = e - a * nc;
                    double s = 0.0;
                    for (int i = 0; i < nc; ++i) s = fma(C[a * ld + i], H[i * ld + k], s);
                    T32[a * ld + k] = (float)s;
                }
                // column k of T has the norm sqrt(H_kk) at most, and no update makes it longer
                ill = false;
                for (int k = tid; k < nc; k += Gp::kNT) {
                    V.h0[k] = __double2hiint(H[k * ld + k]);
                    ill = ill || (V.g0[k] >> 20) + (V.h0[k] >> 20) > 2 * 1023 + kM5Inflated;
                    V.t32[k] = 1.01f * sqrtf(fabsf((float)H[k * ld + k]));
                    V.e32[k] = 6e-8f * V.t32[k];
                }
                ill = Gp::any(ill);
            }
            // w_d / H_dd, then sum_a |res_a + fac_d T_ad| of every attribute still there, in FP32: off by
            // less than 1e-4 of the sizes of its terms, and by what T has lost in the updates
            for (int d = tid; d < nc; d += Gp::kNT) {
                V.fac[d] = (alive >> d) & 1ull ? V.w[d] * rcp_newton_any(H[d * ld + d]) : 0.0;
                V.fac32[d] = (float)V.fac[d];
            }
            Gp::sync();
            if constexpr (!WARP) {                 // lanes = attributes, warps = instances
                float s[2] = {0.f, 0.f}, z[2] = {0.f, 0.f};
                for (int a = wp; a < m; a += nw) {
                    const float ra = res32[a];
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        if (lane + 32 * h < nc) {
                            const float x = V.fac32[lane + 32 * h] * T32[a * ld + lane + 32 * h];
                            s[h] += fabsf(ra + x);
                            z[h] += fabsf(ra) + fabsf(x);
                        }
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    S.errp[0][wp][lane + 32 * h] = s[h];
                    S.errp[1][wp][lane + 32 * h] = z[h];
                }
                __syncthreads();
            }
            if (WARP || wp == 0) {
                float lo32[2] = {0.f, 0.f}, best = __int_as_float(0x7f800000);
                bool on[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int d = lane + 32 * h;
                    on[h] = d < nc && ((alive >> d) & 1ull);
                    if (WARP && h == 1) continue;
                    float s = 0.f, z = 0.f;
                    if (on[h]) {
                        if constexpr (WARP) {
                            for (int a = 0; a < m; ++a) {
                                const float ra = res32[a], x = V.fac32[d] * T32[a * ld + d];
                                s += fabsf(ra + x);
                                z += fabsf(ra) + fabsf(x);
                            }
                        } else {
#pragma unroll
                            for (int w = 0; w < kM5Warps; ++w) {
                                s += S.errp[0][w][d];
                                z += S.errp[1][w][d];
                            }
                        }
                        const float off = 1e-4f * z + 1.01f * (float)m * fabsf(V.fac32[d]) * V.e32[d];
                        lo32[h] = s - off;
                        best = fminf(best, s + off);
                        on[h] = s < 1e30f;         // (not for an estimate that is not finite)
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) best = fminf(best, __shfl_xor_sync(0xffffffffu, best, o));
                const unsigned b0 = __ballot_sync(0xffffffffu, on[0] && !(lo32[0] > best));
                const unsigned b1 = __ballot_sync(0xffffffffu, on[1] && !(lo32[1] > best));
                if (tid == 0) V.reach = (unsigned long long)b1 << 32 | b0;
            }
            Gp::sync();
            // the drops that may be the best, in FP64 from C (nearly always one): the lowest error
            // wins, ties to the lower attribute
            double be = DBL_MAX, bres = 0.0;
            int drop = -1;
            for (unsigned long long rc = V.reach; rc; rc &= rc - 1) {
                const int d = __ffsll((long long)rc) - 1;
                const double fd = V.fac[d];
                for (int i = tid; i < nc; i += Gp::kNT)
                    V.wt[i] = i != d && ((alive >> i) & 1ull) ? fma(-H[i * ld + d], fd, V.w[i]) : 0.0;
                Gp::sync();
                double rn = 0.0;
                if (row < m) {
                    double p = ybar;
                    for (int i = 0; i < nc; ++i) p = fma(C[row * ld + i], V.wt[i], p);
                    rn = S.y[S.ids[lo + row]] - p;
                }
                double e;
                if constexpr (WARP) {
                    e = m5_warp_sum(fabs(rn));
                } else {
                    if (32 * wp < m) {
                        const double x = m5_warp_sum(fabs(rn));
                        if (lane == 0) S.sump[wp] = x;
                    }
                    __syncthreads();
                    e = 0.0;
                    for (int w = 0; 32 * w < m; ++w) e += S.sump[w];
                }
                if (e < be) {                      // (the same in every thread)
                    be = e;
                    drop = d;
                    bres = rn;
                }
                Gp::sync();
            }
            // estimate with ns - 1 terms (v = ns)
            const double est = drop < 0 ? DBL_MAX : be * S.rcp[m] * ((double)(m + ns) * rcp_newton((double)(m - ns)));
            if (m <= ns || drop < 0 || !(est <= V.e_cur)) break;
            const int d = drop;
            dropped = true;
            --ns;
            alive &= ~(1ull << d);
            if (ns == 0) break;
            // take d out: w and the residuals as just computed, H -= H_d H_d^T / H_dd, T -= T_d H_d^T / H_dd
            const double fd = V.fac[d], hi = rcp_newton_any(H[d * ld + d]);
            for (int i = tid; i < nc; i += Gp::kNT) {
                V.colk[i] = H[i * ld + d];
                V.rowk[i] = H[i * ld + d] * hi;
                V.rowk32[i] = (float)V.rowk[i];
                if (i != d) V.e32[i] += fabsf(V.rowk32[i]) * V.e32[d] + 1.3e-7f * V.t32[i];
                V.w[i] = i != d && ((alive >> i) & 1ull) ? fma(-H[i * ld + d], fd, V.w[i]) : 0.0;
            }
            res = bres;
            if (row < m) res32[row] = (float)res;
            Gp::sync();
            if (tid == 0) V.e_cur = est;           // (every thread has compared with it)
            bool lost = ill;                       // or an entry H_ii of which too little is left
            for (int e = tid; e < nc * nc; e += Gp::kNT) {
                const int i = e / nc, j = e - i * nc;
                if (i == d || j == d) continue;
                const double h = fma(-V.colk[i], V.rowk[j], H[i * ld + j]);
                H[i * ld + j] = h;
                if (i == j && ((alive >> i) & 1ull)) lost = lost || __double2hiint(h) + (kM5Shrink << 20) < V.h0[i];
            }
            for (int e = tid; e < m * nc; e += Gp::kNT) {
                const int a = e / nc, k = e - a * nc;
                if (k != d) T32[a * ld + k] = fmaf(-T32[a * ld + d], V.rowk32[k], T32[a * ld + k]);
            }
            if (Gp::any(lost)) {
                // C and the attributes' lists without the dropped columns (a thread a row, ascending), and
                // the model of those that stay
                const int at = tid < nc && ((alive >> tid) & 1ull) ? __popcll(alive & ((1ull << tid) - 1ull)) : -1;
                const int16_t cand = at >= 0 ? V.cand[tid] : (int16_t)0;
                const double zbar = at >= 0 ? V.zbar[tid] : 0.0, r = at >= 0 ? V.r[tid] : 0.0;
                Gp::sync();
                if (at >= 0) {
                    V.cand[at] = cand;
                    V.zbar[at] = zbar;
                    V.r[at] = r;
                    V.sel[at] = (uint8_t)at;
                }
                if (row < m) {
                    int k = 0;
                    for (unsigned long long x = alive; x; x &= x - 1) C[row * ld + k++] = C[row * ld + __ffsll((long long)x) - 1];
                }
                Gp::sync();
                nc = ns;
                alive = (1ull << nc) - 1ull;       // (nc < kM5MaxTerms: one has gone)
                m5_solve<WARP>(S, V, C, H, ld, nc, lo, m, ybar);
                dropped = false;                   // (solved already)
                formed = true;
            }
        }
        Gp::sync();
    }
    if (dropped) {                                 // the model that stays, from its own normal equations
        if (tid < nc && ((alive >> tid) & 1ull)) V.sel[__popcll(alive & ((1ull << tid) - 1ull))] = (uint8_t)tid;
        Gp::sync();
        m5_solve<WARP>(S, V, C, H, ld, ns, lo, m, ybar);
    }
    // the node's model and the pruning decision
    for (int k = tid; k < ns; k += Gp::kNT) {
        T->term_attr[t][k] = V.cand[V.sel[k]];
        T->term_w[t][k] = V.w[k];
    }
    if (tid == 0) {
        T->nterm[t] = ns;
        T->b[t] = V.b;
        T->count[t] = m;
        double e = V.e_cur;
        const int l = S.left[t], r = S.right[t];
        const int ml = S.hi[l] - S.lo[l], mr = S.hi[r] - S.lo[r];
        const double keep = __ddiv_rn(__dadd_rn(__dmul_rn((double)ml, S.est[l]), __dmul_rn((double)mr, S.est[r])), (double)m);
        // A split into halves of two instances and a line through their means have the same estimated error
        // (as have halves of any size on a two-valued attribute), so that their roundings decide: the
        // reference's
        if (ns <= 1 && fabs(e - keep) <= 1e-9 * keep) e = m5_exact_err(S, ns ? V.cand[V.sel[0]] : -1, lo, m);
        if (!(e <= keep)) {
            S.est[t] = keep;
        } else {                                   // a leaf: its parent's candidates get no test
            S.attr[t] = -1;                        // from here down
            S.est[t] = e;
            for (int k = 0; k < kM5MaxFeat / 64; ++k) S.tested[t][k] = 0;
        }
    }
    Gp::sync();
}

// Dynamic shared memory behind M5Smem: while growing, per attribute the instances in (value, index)
// order and each instance's rank among the attribute's distinct values; then the models' matrices.
__host__ __device__ __forceinline__ size_t m5_dyn_bytes(int F) {
    const int nmax = kM5MaxN;
    const size_t grow = 2 * (size_t)F * nmax;
    const int tm = F < kM5MaxTerms ? F : kM5MaxTerms, ld = tm | 1;
    const size_t blk = ((size_t)tm * ld + (size_t)nmax * ld) * sizeof(double) + (size_t)nmax * ld * sizeof(float);
    const size_t wrp = (size_t)kM5Warps * kM5WarpBuf * sizeof(double);
    const size_t mo = blk > wrp ? blk : wrp;
    return grow > mo ? grow : mo;
}

__global__ void __launch_bounds__(kM5Threads)
m5p_fit_kernel(const TransferArgs a, int fmax) {
    constexpr int nmax = kM5MaxN;
    extern __shared__ __align__(16) unsigned char m5sm[];
    M5Smem& S = *reinterpret_cast<M5Smem*>(m5sm);
    unsigned char* dyn = m5sm + ((sizeof(M5Smem) + 15) & ~(size_t)15);
    __shared__ GroupSmem G;
    __shared__ uint16_t pu[kTrPairs];
    __shared__ double yl[kTrPairs];
    __shared__ int np_s;
    const int q = blockIdx.x, j = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int start[RS_MAXRUNS + 1], F = 0;
    const int N = rs_group_layout(q, a.group_off, a.max_runs, a.n_runs, a.a_row, a.a_fw, a.b_fw, a.stat_stride, start, F);
    if (N < 0 || N > a.ld || F > kM5MaxFeat || F > fmax) return;   // reported by the predict / rank kernel
    const int64_t g0 = a.group_off[q];
    const int R = (int)(a.group_off[q + 1] - g0);
    load_group(G, a.a_row, a.a_masks, a.a_lt, g0, start, N);
    if (warp == 0) {
        const int np = build_pairs(G, j, R, N, start, pu, yl, nullptr, q);
        if (lane == 0) np_s = np;
    }
    __syncthreads();
    const int n = np_s;
    M5Tree* T = a.trees + ((int64_t)q * RS_NOPT + j);
    uint8_t* st_out = a.fst + (int64_t)q * RS_NOPT + j;
    if (n == 0) {
        if (tid == 0) *st_out = RS_FIT_EMPTY;
        return;
    }
    uint8_t* srt = dyn;                                           // [F][nmax]
    uint8_t* rk = dyn + (size_t)fmax * nmax;                      // [F][nmax]
    for (int c = tid; c <= kM5MaxN; c += kM5Threads) S.rcp[c] = __drcp_rn((double)(c ? c : 1));
    for (int i = tid; i < n; i += kM5Threads) {
        const int u = pu[i];
        int r = 0;
        while (u >= start[r + 1]) ++r;
        S.zp[i] = a.ZA + a.a_xo[g0 + r] + (int64_t)(u - start[r]) * F;
        S.y[i] = yl[i];
        S.y2[i] = __dmul_rn(yl[i], yl[i]);
        S.ids[i] = (uint8_t)i;
    }
    __syncthreads();
    // presort, a warp per attribute: an instance's place is the number before it by (value, index),
    // its rank the number of smaller values (a label of its group of equals); integer order keys
    for (int f = warp; f < F; f += kM5Warps) {
        long long key[kM5MaxN / 32];
        int pos[kM5MaxN / 32], less[kM5MaxN / 32];
#pragma unroll
        for (int x = 0; x < kM5MaxN / 32; ++x) {
            const int i = lane + 32 * x;
            key[x] = i < n ? okey(__ldg(S.zp[i] + f)) : 0x7fffffffffffffffll;
            pos[x] = less[x] = 0;
        }
#pragma unroll
        for (int x = 0; x < kM5MaxN / 32; ++x)
            for (int s = 0; s < 32 && 32 * x + s < n; ++s) {
                const long long k = __shfl_sync(0xffffffffu, key[x], s);
                const int i = 32 * x + s;
#pragma unroll
                for (int z = 0; z < kM5MaxN / 32; ++z) {
                    less[z] += k < key[z];
                    pos[z] += k < key[z] || (k == key[z] && i < lane + 32 * z);
                }
            }
#pragma unroll
        for (int x = 0; x < kM5MaxN / 32; ++x) {
            const int i = lane + 32 * x;
            if (i < n) {
                srt[f * nmax + pos[x]] = (uint8_t)i;
                rk[f * nmax + i] = (uint8_t)less[x];
            }
        }
    }
    if (warp == 0) {                               // the root's exact sums: lane 0 s1, lane 1 s2, one chain
        double s = 0.0;
        for (int i = 0; i < n; ++i) s = __dadd_rn(s, lane == 1 ? S.y2[i] : S.y[i]);
        const double s1 = __shfl_sync(0xffffffffu, s, 0), s2 = __shfl_sync(0xffffffffu, s, 1);
        const double sd = m5_sd(n, __drcp_rn((double)n), s1, s2);
        if (lane == 0) {
            S.sd_root = sd;
            S.nn = 1;
            S.level[0] = 0;
            S.level[1] = 1;
            S.lo[0] = 0;
            S.hi[0] = (uint8_t)n;
            S.parent[0] = -1;
        }
        const double mean = s1 / n;
        if (lane == 0) S.mean0 = fabsf((float)mean);
        for (int i = lane; i < n; i += 32) S.yf[i] = (float)(S.y[i] - mean);
    }
    __syncthreads();
    // ---- grow, level by level (children get larger numbers than their parents)
    int depth = 0;
    for (;; ++depth) {
        const int n0 = S.level[depth], nl = S.level[depth + 1] - n0;
        if (tid == 0) S.nsurv = 0;
        // per node: FP32 statistics, and leaves by size or deviation (near the line, or with labels
        // that FP32 does not hold: by the exact deviation)
        for (int k = warp; k < nl; k += kM5Warps) {
            const int t = n0 + k, lo = S.lo[t], m = S.hi[t] - lo;
            float s = 0.f, am = 0.f;
            for (int e = lane; e < m; e += 32) {
                const float v = S.yf[S.ids[lo + e]];
                s += v;
                am = fmaxf(am, fabsf(v));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                s += __shfl_xor_sync(0xffffffffu, s, o);
                am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
            }
            const float mean = s / (float)m;
            float t1 = 0.f, t2 = 0.f;
            for (int e = lane; e < m; e += 32) {
                const float v = S.yf[S.ids[lo + e]] - mean;
                t1 += v;
                t2 = fmaf(v, v, t2);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                t1 += __shfl_xor_sync(0xffffffffu, t1, o);
                t2 += __shfl_xor_sync(0xffffffffu, t2, o);
            }
            // the exact label sums in instance order: lane 0 s1, lane 1 s2
            double xs = 0.0;
            bool leaf = m < 4;
            const float sda = sqrtf(t2 / (float)m), lim = (float)(kM5SdFrac * S.sd_root);
            const bool fp32 = t2 < 1e30f && am < 1e15f && lim > 1e-15f;
            // (the exact deviation's rounding: below sqrt(4e-14) of the labels' magnitude)
            const float ymax = am + 1.001f * S.mean0, slack = 1e-3f * lim + 4e-6f * am + 3e-7f * ymax;
            if (!leaf && fp32 && sda < lim - slack) leaf = true;
            int cnt = leaf ? -1 : 0;
            if (!leaf) {
                for (int e = 0; e < m; ++e) {
                    const int i = S.ids[lo + e];
                    xs = __dadd_rn(xs, lane == 1 ? S.y2[i] : S.y[i]);
                }
                const double s1 = __shfl_sync(0xffffffffu, xs, 0), s2 = __shfl_sync(0xffffffffu, xs, 1);
                if (!fp32 || sda <= lim + slack) {
                    if (m5_sd(m, S.rcp[m], s1, s2) <= __dmul_rn(kM5SdFrac, S.sd_root)) cnt = -1;
                    else if (!fp32) cnt = -2;
                }
                if (lane == 0) {
                    S.s1[k] = s1;
                    S.s2[k] = s2;
                }
            }
            if (lane == 0) {
                S.attr[t] = -1;
                S.cnt[k] = cnt;
                S.mean[k] = mean;
                S.tot[k] = t1;
                S.tot2[k] = t2;
                S.amax2[k] = am * am + 6e-7f * ymax * ymax;
                S.ymax[k] = ymax;
                S.sda[k] = sda;
                S.best_hi[k] = 0x7f800000u;
                S.best_red[k] = 0ull;
                S.best_key[k] = 0xffffffffu;
            }
        }
        __syncthreads();
        // the attributes' scans of every splitting node, dealt to the warps; a warp takes several
        // attributes of a node that has few instances
        int x0 = 0;
        for (int k = 0; k < nl; ++k) {
            if (S.cnt[k] < 0) continue;
            const int lo = S.lo[n0 + k], m = S.hi[n0 + k] - lo;
            const int W = m <= 8 ? 8 : m <= 16 ? 16 : 32, per = 32 / W, nt = (F + per - 1) / per;
            for (int x = (warp - x0) & (kM5Warps - 1); x < nt; x += kM5Warps) {
                const int f = x * per + lane / W;
                m5_scan(S, srt + (f < F ? f : 0) * nmax, rk + (f < F ? f : 0) * nmax, f < F ? f : -1, lo, m, k, W);
            }
            x0 = (x0 + nt) & (kM5Warps - 1);       // the next node's first task to the next warp
        }
        __syncthreads();
        const bool over = S.nsurv > kM5Surv;       // then every node of the level by the exact scan
        // of those listed early, the ones that still reach the final bound; how many a node has
        for (int x = tid; x < (over ? 0 : S.nsurv); x += kM5Threads) {
            const unsigned k = S.surv[x] >> 16;
            if (S.ql[x] <= __uint_as_float(S.best_hi[k])) atomicAdd(&S.cnt[k], 1);
            else S.surv[x] = 0xffffffffu;
        }
        __syncthreads();
        const int nsv = over ? 0 : S.nsurv;
        // exact SDRs of the survivors, two threads each (left and right); a node's only survivor
        // whose SDR is positive beyond doubt needs none
        for (int x = tid >> 1; x < ((nsv + kM5Threads / 2 - 1) & ~(kM5Threads / 2 - 1)); x += kM5Threads / 2) {
            const unsigned sv = x < nsv && S.surv[x] != 0xffffffffu ? S.surv[x] : 0u;
            const bool here = x < nsv && S.surv[x] != 0xffffffffu;
            const int k = (int)(sv >> 16), f = (int)(sv >> 8) & 0xff, c = (int)(sv & 0xff);
            const int t = n0 + k, lo = S.lo[t], m = S.hi[t] - lo;
            const bool sure = here && S.cnt[k] == 1 && __uint_as_float(S.best_hi[k]) < 0.999f * (float)m * S.sda[k] - (float)m * (1e-5f * sqrtf(S.amax2[k]) + 3e-7f * S.ymax[k]);
            const bool work = here && !sure;
            double sdx = 0.0;
            if (work) {
                const uint8_t* o = srt + f * nmax + lo;
                double l1 = 0.0, l2 = 0.0;
                for (int e = 0; e < c; ++e) {
                    l1 = __dadd_rn(l1, S.y[o[e]]);
                    l2 = __dadd_rn(l2, S.y2[o[e]]);
                }
                if (tid & 1) {
                    l1 = __dsub_rn(S.s1[k], l1);
                    l2 = __dsub_rn(S.s2[k], l2);
                }
                const int cc = (tid & 1) ? m - c : c;
                sdx = __dmul_rn((double)cc, m5_sd(cc, S.rcp[cc], l1, l2));
            }
            const double other = __shfl_xor_sync(0xffffffffu, sdx, 1);
            if (here && !(tid & 1)) {
                double red = 1.0;
                if (work)
                    red = __dsub_rn(m5_sd(m, S.rcp[m], S.s1[k], S.s2[k]), m5_div(__dadd_rn(sdx, other), (double)m, S.rcp[m]));
                S.red[x] = red;
                if (red > 0.0) atomicMax(&S.best_red[k], (unsigned long long)__double_as_longlong(red));
            }
        }
        // nodes for the exact scan: one thread per attribute
        for (int k = 0; k < nl; ++k) {
            const int c = S.cnt[k];
            if (c != -2 && !(over && c >= 0)) continue;      // (uniform)
            const int t = n0 + k, lo = S.lo[t], m = S.hi[t] - lo;
            const double sd = m5_sd(m, S.rcp[m], S.s1[k], S.s2[k]);
            double best = 0.0;
            unsigned key = 0xffffffffu;
            for (int f = tid; f < F; f += kM5Threads)
                m5_exact_scan(S, srt + f * nmax, rk + f * nmax, f, lo, m, k, sd, best, key);
            if (best > 0.0) atomicMax(&S.best_red[k], (unsigned long long)__double_as_longlong(best));
            __syncthreads();
            if (best > 0.0 && (unsigned long long)__double_as_longlong(best) == S.best_red[k]) atomicMin(&S.best_key[k], key);
            __syncthreads();
        }
        __syncthreads();
        // ties: the lowest attribute, then the lowest count
        for (int x = tid; x < nsv; x += kM5Threads) {
            if (S.surv[x] == 0xffffffffu) continue;
            const int k = (int)(S.surv[x] >> 16);
            const double red = S.red[x];
            if (red > 0.0 && (unsigned long long)__double_as_longlong(red) == S.best_red[k])
                atomicMin(&S.best_key[k], S.surv[x] & 0xffffu);
        }
        __syncthreads();
        // thresholds, sides and the number of instances going left, a warp per splitting node
        for (int k = warp; k < nl; k += kM5Warps) {
            const unsigned key = S.best_key[k];
            if (key == 0xffffffffu) {
                if (lane == 0) S.cnt[k] = -1;
                continue;
            }
            const int t = n0 + k, lo = S.lo[t], m = S.hi[t] - lo, f = (int)(key >> 8), c = (int)(key & 0xff);
            const uint8_t* o = srt + f * nmax + lo;
            const double thr = __dmul_rn(__dadd_rn(__ldg(S.zp[o[c - 1]] + f), __ldg(S.zp[o[c]] + f)), 0.5);
            int left = 0;
            for (int e0 = 0; e0 < m; e0 += 32) {
                const int e = e0 + lane;
                const int i = e < m ? S.ids[lo + e] : 0;
                const bool lf = e < m && __ldg(S.zp[i] + f) <= thr;
                if (e < m) S.side[i] = lf ? 0 : 1;
                left += __popc(__ballot_sync(0xffffffffu, lf));
            }
            // (two neighbouring doubles may have the upper one as their rounded mean: a side without
            // instances is no split)
            if (lane == 0) {
                const bool two = left > 0 && left < m;
                S.attr[t] = two ? (int16_t)f : (int16_t)-1;
                S.thr[t] = thr;
                S.cnt[k] = two ? left : -1;
            }
        }
        __syncthreads();
        if (tid == 0) {
            int nn = S.nn;
            for (int k = 0; k < nl; ++k) {
                if (S.cnt[k] < 0) continue;
                const int t = n0 + k;
                S.left[t] = (int16_t)nn;
                S.right[t] = (int16_t)(nn + 1);
                S.parent[nn] = S.parent[nn + 1] = (int16_t)t;
                S.lo[nn] = S.lo[t];
                S.hi[nn] = S.lo[nn + 1] = (uint8_t)(S.lo[t] + S.cnt[k]);
                S.hi[nn + 1] = S.hi[t];
                nn += 2;
            }
            S.nn = nn;
            S.level[depth + 2] = nn;
        }
        // stable partition of each splitting node's range of every attribute's list and of the
        // instance list, a warp per list
        for (int x = warp; x < nl * (F + 1); x += kM5Warps) {
            const int k = x / (F + 1), f = x - k * (F + 1);
            if (S.cnt[k] < 0) continue;
            const int t = n0 + k, lo = S.lo[t], m = S.hi[t] - lo;
            uint8_t* o = (f < F ? srt + f * nmax : S.ids) + lo;
            int id[kM5MaxN / 32], at[kM5MaxN / 32], l = 0, r = S.cnt[k];
#pragma unroll
            for (int z = 0; z < kM5MaxN / 32; ++z) {
                const int e = 32 * z + lane;
                id[z] = e < m ? o[e] : -1;
                const bool lf = e < m && S.side[id[z]] == 0, rt = e < m && !lf;
                const unsigned bl = __ballot_sync(0xffffffffu, lf), br = __ballot_sync(0xffffffffu, rt);
                at[z] = lf ? l + __popc(bl & ((1u << lane) - 1u)) : r + __popc(br & ((1u << lane) - 1u));
                l += __popc(bl);
                r += __popc(br);
            }
            __syncwarp();
#pragma unroll
            for (int z = 0; z < kM5MaxN / 32; ++z)
                if (id[z] >= 0) o[at[z]] = (uint8_t)id[z];
        }
        __syncthreads();
        if (S.level[depth + 2] == S.level[depth + 1]) break;
    }
    // ---- models and pruning.  Leaves (the label mean) first, a warp each; then the internal nodes
    // level by level from the deepest, small ones a warp each, the others by the block
    const int nn = S.nn;
    for (int t = warp; t < nn; t += kM5Warps) {
        if (S.attr[t] >= 0) continue;
        const int lo = S.lo[t], m = S.hi[t] - lo;
        double s = 0.0, e = 0.0;                   // (in instance order, by every lane: as the reference)
        for (int x = 0; x < m; ++x) s = __dadd_rn(s, S.y[S.ids[lo + x]]);
        s = __ddiv_rn(s, (double)m);
        for (int x = 0; x < m; ++x) e = __dadd_rn(e, fabs(__dsub_rn(S.y[S.ids[lo + x]], s)));
        if (lane == 0) {
            T->nterm[t] = 0;
            T->b[t] = s;
            T->count[t] = m;
            S.est[t] = m <= 1 ? DBL_MAX : __dmul_rn(__ddiv_rn(e, (double)m), __ddiv_rn((double)(m + 1), (double)(m - 1)));
            for (int k = 0; k < kM5MaxFeat / 64; ++k) S.tested[t][k] = 0;
        }
    }
    const int tm = fmax < kM5MaxTerms ? fmax : kM5MaxTerms, ld = tm | 1;
    double* buf = reinterpret_cast<double*>(dyn);
    __syncthreads();
    for (int dp = depth; dp >= 0; --dp) {
        const int n0 = S.level[dp], n1 = S.level[dp + 1];
        for (int t = n0 + tid; t < n1; t += kM5Threads)      // (the children's are final)
            if (S.attr[t] >= 0)
                for (int k = 0; k < kM5MaxFeat / 64; ++k)
                    S.tested[t][k] = S.tested[S.left[t]][k] | S.tested[S.right[t]][k] |
                                     (S.attr[t] / 64 == k ? 1ull << (S.attr[t] % 64) : 0ull);
        __syncthreads();
        // which nodes of the level a warp can take (decided before any of them is pruned)
        for (int t = n0 + tid; t < n1; t += kM5Threads) {
            int nc = 0;
            for (int k = 0; k < kM5MaxFeat / 64; ++k) nc += __popcll(S.tested[t][k]);
            S.cnt[t - n0] = S.attr[t] < 0 ? 0 : (nc <= kM5WarpTerms && S.hi[t] - S.lo[t] <= kM5WarpN ? 1 : 2);
        }
        __syncthreads();
        int turn = 0;
        for (int t = n0; t < n1; ++t)
            if (S.cnt[t - n0] == 1 && (turn++ & (kM5Warps - 1)) == warp) {
                double* wb = buf + warp * kM5WarpBuf;
                m5_model<true>(S, S.v.wv[warp], T, t, F, wb, wb + kM5WarpTerms * kM5WarpLd,
                               reinterpret_cast<float*>(wb + (kM5WarpTerms + kM5WarpN) * kM5WarpLd), kM5WarpLd);
            }
        __syncthreads();
        for (int t = n0; t < n1; ++t)
            if (S.cnt[t - n0] == 2) m5_model<false>(S, S.v.blk, T, t, F, buf, buf + tm * ld,
                                                            reinterpret_cast<float*>(buf + (tm + nmax) * ld), ld);
        __syncthreads();
    }
    for (int t = tid; t < nn; t += kM5Threads) {
        T->attr[t] = S.attr[t];
        T->thr[t] = S.thr[t];
        T->left[t] = S.left[t];
        T->right[t] = S.right[t];
        T->parent[t] = S.parent[t];
    }
    if (tid == 0) {
        T->n_nodes = nn;
        *st_out = RS_FIT_OK;
    }
}

// The M5P prediction for one test vector: the leaf's model, then smoothing with every
// ancestor's model on the way up, p = (n_c p + k q) / (n_c + k).
__device__ double m5_predict(const M5Tree* __restrict__ T, const double* __restrict__ z) {
    auto model = [&](int t) {
        double p = T->b[t];
        for (int k = 0; k < T->nterm[t]; ++k) p = fma(T->term_w[t][k], __ldg(z + T->term_attr[t][k]), p);
        return p;
    };
    int t = 0;
    while (T->attr[t] >= 0) t = __ldg(z + T->attr[t]) <= T->thr[t] ? T->left[t] : T->right[t];
    double p = model(t);
    while (T->parent[t] >= 0) {
        const int u = T->parent[t];
        const double nc = (double)T->count[t];
        p = (nc * p + kM5Smooth * model(u)) / (nc + kM5Smooth);
        t = u;
    }
    return p;
}

// ibk_nearest_mean for a list of n > kIbkK pairs (n up to kTrPairs): the chosen labels are
// summed in ascending pair index.
__device__ __forceinline__ double ibk_nearest_mean_n(int n, const double* __restrict__ Dt, const uint16_t* pu,
                                                     const double* yl) {
    unsigned long long kd[kIbkK];
    int kq[kIbkK];
#pragma unroll
    for (int i = 0; i < kIbkK; ++i) {
        kd[i] = ~0ull;
        kq[i] = 0;
    }
    for (int q = 0; q < n; ++q) ibk_insert(kd, kq, (unsigned long long)__double_as_longlong(__ldg(Dt + pu[q])), q);
    for (int i = 1; i < kIbkK; ++i)          // indices ascending
        for (int m = i; m > 0 && kq[m - 1] > kq[m]; --m) {
            const int x = kq[m];
            kq[m] = kq[m - 1];
            kq[m - 1] = x;
        }
    double sum = 0.0;
    for (int i = 0; i < kIbkK; ++i) sum += yl[kq[i]];
    return sum / (double)kIbkK;
}

// The predictions of one (problem, optimization) for every candidate version of its test program, by
// the fit of transfer_fit_kernel (four lanes a version), the neighbour list of IBK or the M5P tree
// (one lane a version), into pred [Q][64][6] for transfer_rank_kernel.  One block per problem used to
// walk the six optimizations in turn (101 us at 90 problems of 96 pairs; the two kernels: 27 us).
template <int SUB>
__global__ void __launch_bounds__(RS_MAXV * SUB)
transfer_predict_kernel(const TransferArgs a) {
    __shared__ GroupSmem G;
    __shared__ uint16_t pu[kTrPairs];
    __shared__ double yl[kTrPairs];
    __shared__ int np_s;
    const int q = blockIdx.x, j = blockIdx.y, tid = threadIdx.x;
    int start[RS_MAXRUNS + 1], F = 0;
    const int N = rs_group_layout(q, a.group_off, a.max_runs, a.n_runs, a.a_row, a.a_fw, a.b_fw, a.stat_stride, start, F);
    const int64_t rb = a.b_row[q];
    const int VB = (int)(a.b_row[q + 1] - rb);
    if (N < 0 || N > a.ld || VB < 1 || VB > RS_MAXV) return;       // reported by transfer_rank_kernel
    const int64_t g0 = a.group_off[q];
    load_group(G, a.a_row, a.a_masks, a.a_lt, g0, start, N);
    if (tid < 32) {
        const int np = build_pairs(G, j, (int)(a.group_off[q + 1] - g0), N, start, pu, yl, a.r.dstatus, q);
        if (tid == 0) np_s = np;
    }
    __syncthreads();
    const int n = np_s;
    uint8_t* st = a.fst + (int64_t)q * RS_NOPT + j;
    if (a.ibk) {
        if (tid == 0) *st = n > 0 ? RS_FIT_OK : RS_FIT_EMPTY;
        if (n == 0) return;
    } else if (*st != RS_FIT_OK) {
        return;
    }
    const int t = tid / SUB, sub = tid % SUB;
    const bool cand = t < VB && ((a.opt_mask >> j) & 1) && (a.rank_all || !((a.b_masks[rb + (t < VB ? t : 0)] >> j) & 1));
    const double* Kt = a.Kx + ((int64_t)q * RS_MAXV + t) * a.ld;
    double yh = 0.0;
    if (SUB == 1) {
        if (!cand) return;
        if (a.m5p) {
            yh = m5_predict(a.trees + ((int64_t)q * RS_NOPT + j), a.ZB + a.b_xo[q] + (int64_t)t * F);
        } else if (n <= kIbkK) {
            for (int i = 0; i < n; ++i) yh += yl[i];
            yh /= (double)n;
        } else {
            yh = ibk_nearest_mean_n(n, Kt, pu, yl);
        }
    } else {
        const double* cf = a.coef + ((int64_t)q * RS_NOPT + j) * kTrCoef;
        if (cand && n > 1)
            for (int i = sub; i < n; i += SUB) yh = fma(cf[1 + i], __ldg(Kt + pu[i]), yh);
#pragma unroll
        for (int o = 1; o < SUB; o <<= 1) yh += __shfl_xor_sync(0xffffffffu, yh, o);
        if (!cand || sub) return;
        yh += cf[0];
    }
    a.pred[((int64_t)q * RS_MAXV + t) * RS_NOPT + j] = yh;
}

// One block per problem, one thread per version t of the test program: its predictions through
// rank_row, the problem's fit statuses and the counters.
__global__ void __launch_bounds__(RS_MAXV)
transfer_rank_kernel(const TransferArgs a) {
    __shared__ double lt_b[RS_MAXV];
    __shared__ uint8_t msk_b[RS_MAXV];
    __shared__ int8_t slot_b[RS_MAXV];
    const int q = blockIdx.x, tid = threadIdx.x;
    int start[RS_MAXRUNS + 1], F = 0;
    const int N = rs_group_layout(q, a.group_off, a.max_runs, a.n_runs, a.a_row, a.a_fw, a.b_fw, a.stat_stride, start, F);
    const int64_t rb = a.b_row[q];
    const int VB = (int)(a.b_row[q + 1] - rb);
    if (N < 0 || N > a.ld || VB < 1 || VB > RS_MAXV) {
        if (tid == 0) rs_dev_flag(a.r.dstatus, RS_EDATA, q);
        return;
    }
    slot_b[tid] = -1;
    __syncthreads();
    if (tid < VB) {
        msk_b[tid] = a.b_masks[rb + tid] & 63;
        lt_b[tid] = a.b_lt[rb + tid];
        slot_b[msk_b[tid]] = (int8_t)tid;
    }
    __syncthreads();
    const uint8_t* fst = a.fst + (int64_t)q * RS_NOPT;
    RankTally c;
    const int t = tid;
    if (t < VB) {
        const int mt = msk_b[t];
        const uint32_t info = row_summary(t, VB, msk_b, lt_b, slot_b);
        const int candm = (a.rank_all ? 63 : (~mt & 63)) & a.opt_mask;
        int okm = 0;
#pragma unroll
        for (int j = 0; j < RS_NOPT; ++j) okm |= (fst[j] == RS_FIT_OK) << j;
        const double* pr = a.pred + ((int64_t)q * RS_MAXV + t) * RS_NOPT;
        double pred[RS_NOPT];
#pragma unroll
        for (int j = 0; j < RS_NOPT; ++j) pred[j] = ((candm & okm) >> j) & 1 ? pr[j] : 0.0;
        // rank_row's candidates are the optimizations outside the version-mask field: put the
        // excluded ones there (t's own unless all six are ranked, and those outside opt_mask);
        // the fits that are not OK go in the empty-fit field
        const int mfield = ((a.rank_all ? 0 : mt) | ~a.opt_mask) & 63;
        const unsigned long long info64 = (unsigned long long)info | ((unsigned long long)mfield << 30) |
                                          ((unsigned long long)(~okm & 63) << 36);
        rank_row(a.r, rb + t, info64, pred, c);
    }
    if (tid < RS_NOPT) {
        const int st = fst[tid];
        if (a.fit_status) a.fit_status[(int64_t)q * RS_NOPT + tid] = (uint8_t)st;
        if (a.r.counters && st >= 0 && st <= RS_FIT_NONFINITE) atomicAdd(a.r.counters + 9 + st, 1ull);
    }
    if (a.r.counters) {
        const uint32_t vals[10] = {c.rows, c.pred, c.scored, c.sign, c.rec, c.reck, c.rech, c.t1, c.t1h, c.inv};
        const int slot[10] = {0, 1, 2, 3, 4, 5, 6, 7, 8, 13};
#pragma unroll
        for (int i = 0; i < 10; ++i) {
            const uint32_t v = __reduce_add_sync(0xffffffffu, vals[i]);
            if ((tid & 31) == 0 && v) atomicAdd(a.r.counters + slot[i], (unsigned long long)v);
        }
    }
}

__global__ void iota64_kernel(int64_t* out, int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = i;
}

}  // namespace

cudaError_t rs_launch_iota64(int64_t* out, int64_t n, cudaStream_t st) {
    if (n > 0) iota64_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(out, n);
    return cudaGetLastError();
}

size_t rs_m5p_tree_bytes() { return sizeof(M5Tree); }
int rs_m5p_max_feat() { return kM5MaxFeat; }

size_t rs_transfer_fit_bytes(int64_t Q) {
    return (size_t)Q * RS_NOPT * kTrCoef * sizeof(double) + (size_t)Q * RS_NOPT;
}

cudaError_t rs_launch_transfer(const rs_transfer_args& t, cudaStream_t st) {
    TransferArgs a{};
    a.group_off = t.group_off;
    a.max_runs = t.max_runs;
    a.stat_stride = t.stat_stride;
    a.n_runs = t.n_runs;
    a.a_row = t.a_row_offsets;
    a.a_fw = t.a_feat_width;
    a.a_masks = t.a_masks;
    a.a_lt = t.a_log_time;
    a.b_row = t.b_row_offsets;
    a.b_fw = t.b_feat_width;
    a.b_masks = t.b_masks;
    a.b_lt = t.b_log_time;
    a.KA = t.KA;
    a.Kx = t.Kx;
    a.ld = t.ld;
    a.lambda = t.lambda;
    a.coef = t.fit_ws;
    a.fst = reinterpret_cast<uint8_t*>(t.fit_ws + (size_t)t.Q * RS_NOPT * kTrCoef);
    a.ibk = t.ibk;
    a.opt_mask = t.opt_mask & 63;
    a.rank_all = (t.flags & RS_RANK_ALL) != 0;
    a.fit_status = t.fit_status;
    a.m5p = t.m5p;
    a.trees = reinterpret_cast<M5Tree*>(t.m5_ws);
    a.ZA = t.ZA;
    a.a_xo = t.a_x_offsets;
    a.ZB = t.ZB;
    a.pred = const_cast<double*>(t.KA);  // the group's Gram (at least 64 x 64 doubles a problem) is no
                                         // longer read once the fits are made, nor at all without ridge
    a.b_xo = t.b_x_offsets;
    a.r = RankPassArgs{nullptr, 0, nullptr, 0, 0, nullptr, t.dstatus, t.k, okey_host(t.log_tau),
                       t.flags & ~RS_RANK_ALL, t.rec_code, t.rec_pred, t.pred_all, t.counters};
    cudaError_t e = cudaSuccess;
    if (t.m5p) {
        const size_t msmem = ((sizeof(M5Smem) + 15) & ~(size_t)15) + m5_dyn_bytes(t.stat_stride);
        e = cudaFuncSetAttribute(m5p_fit_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)msmem);
        if (e != cudaSuccess) return e;
        m5p_fit_kernel<<<dim3((unsigned)t.Q, RS_NOPT), kM5Threads, msmem, st>>>(a, t.stat_stride);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    } else if (!t.ibk) {
        const int nmax = RS_MAXPAIRS * t.max_runs;
        const size_t fsmem = ((size_t)nmax * (nmax + 1) / 2 + 5 * (size_t)nmax) * sizeof(double);
        e = cudaFuncSetAttribute(transfer_fit_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fsmem);
        if (e != cudaSuccess) return e;
        transfer_fit_kernel<<<dim3((unsigned)t.Q, RS_NOPT), kTrThreads, fsmem, st>>>(a, nmax);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    const dim3 grid((unsigned)t.Q, RS_NOPT);
    if (t.ibk || t.m5p) transfer_predict_kernel<1><<<grid, RS_MAXV, 0, st>>>(a);
    else transfer_predict_kernel<4><<<grid, RS_MAXV * 4, 0, st>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    transfer_rank_kernel<<<(unsigned)t.Q, RS_MAXV, 0, st>>>(a);
    return cudaGetLastError();
}
