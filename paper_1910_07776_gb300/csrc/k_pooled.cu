// k_pooled.cu -- pooled ridge fits in primal form (A3 + A4): one model per optimization j
// trained on the before/after pairs (Sec. 3.3) of MANY programs at once, the training set of a
// tool that has seen many codes (Sec. 5's transfer between codes, at scale).  With n pairs
// far more numerous than the F features, the primal normal equations are the small system:
//     G_j = sum_a c_a c_a^T + lambda I,   r_j = sum_a c_a (y_a - ybar_j),   c_a = z_a - zbar_j,
//     G_j beta_j = r_j,   b_j = ybar_j - zbar_j . beta_j      (the intercept unpenalised).
// The Gram X^T W X (W selecting the pairs of optimization j, centred) is the dense contraction:
// it runs on the tcgen05 tensor cores as one batched GEMM over j, with the BF16 hi/lo split of
// the centred rows (c = hi + lo; G ~ hi hi^T + hi lo^T + lo hi^T, K = 3 n), the operands
// staged feature-major by a transpose kernel and fed by TMA.  The FP64 Cholesky factorisation
// of G_j follows, and (RS_REFINE_X) one step of iterative refinement whose residual
// r_j - lambda beta - sum_a c_a (c_a . beta) is taken exactly in FP64 through the rows.
// Predictions: b_j + z_t . beta_j for every version t of a batch, ranked and scored by
// rank_row (Sec. 2 tier 3).
#include "rank_row.cuh"
#include "tc_gemm.cuh"

namespace {

constexpr int kPoolMaxPairs = 65536;   // pairs per optimization (all programs together)

struct PoolArgs {
    int P, F;
    const int64_t* row_off;
    const int32_t* fw;
    const int64_t* x_off;
    const double* Z;
    const uint8_t* masks;
    const double* lt;
    const uint8_t* use;          // nullable: programs that train
    int* counts;                 // [6][P]
    int64_t* offs;               // [6][P + 1]
    int64_t* zoff;               // [6][NP]: offset in Z of the before version's features
    double* y;                   // [6][NP]: log speedup of the pair
    int NP;                      // pairs capacity per optimization
    double* zbar;                // [6][F]
    double* ybar;                // [6]
    double* G;                   // [6][F][F]
    double* r;                   // [6][F]
    double* s;                   // [6][NP]: c_a . beta during refinement
    double* coef;                // [6][F + 1]: b, beta
    uint8_t* status;             // [6]
    double lambda;
    int* dstatus;
};

// Per program (block of 64 threads, thread = version slot): the number of pairs of each j.
__global__ void __launch_bounds__(RS_MAXV) pooled_count_kernel(PoolArgs a) {
    __shared__ int8_t slot_of[64];
    __shared__ int cnt[RS_NOPT];
    const int p = blockIdx.x, v = threadIdx.x;
    const int64_t r0 = a.row_off[p];
    const int V = (int)(a.row_off[p + 1] - r0);
    slot_of[v] = -1;
    if (v < RS_NOPT) cnt[v] = 0;
    __syncthreads();
    const bool want = !a.use || a.use[p];
    const bool valid = V >= 1 && V <= RS_MAXV && a.fw[p] == a.F;
    if (want && !valid && v == 0) rs_dev_flag(a.dstatus, RS_EDATA, p);   // skipped, reported
    const bool use = want && valid;
    const int m = use && v < V ? (a.masks[r0 + v] & 63) : 0;
    if (use && v < V) slot_of[m] = (int8_t)v;
    __syncthreads();
    if (use && v < V)
        for (int j = 0; j < RS_NOPT; ++j)
            if (!((m >> j) & 1) && slot_of[m | (1 << j)] >= 0) atomicAdd(&cnt[j], 1);
    __syncthreads();
    if (v < RS_NOPT) a.counts[v * a.P + p] = use ? cnt[v] : 0;
}

// Per j (one block): exclusive prefix of the per-program counts.
__global__ void __launch_bounds__(1024) pooled_scan_kernel(PoolArgs a) {
    __shared__ long long wsum[32];
    const int j = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int chunk = (a.P + 1023) / 1024;
    const int p0 = tid * chunk, p1 = p0 + chunk < a.P ? p0 + chunk : a.P;
    long long s = 0;
    for (int p = p0; p < p1; ++p) s += a.counts[j * a.P + p];
    long long incl = s;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        long long w = wsum[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, w, d);
            if (lane >= d) w += y;
        }
        wsum[lane] = w;
    }
    __syncthreads();
    long long off = incl - s + (warp > 0 ? wsum[warp - 1] : 0ll);
    int64_t* o = a.offs + (int64_t)j * (a.P + 1);
    for (int p = p0; p < p1; ++p) {
        o[p] = off;
        off += a.counts[j * a.P + p];
    }
    if (tid == 1023) o[a.P] = off;
}

// Per program: its pairs of each j, in ascending order of the before slot, after the pairs of
// the programs before it.
__global__ void __launch_bounds__(RS_MAXV) pooled_fill_kernel(PoolArgs a) {
    __shared__ int8_t slot_of[64];
    __shared__ int wcnt[RS_NOPT][2];
    const int p = blockIdx.x, v = threadIdx.x, lane = v & 31, warp = v >> 5;
    const int64_t r0 = a.row_off[p];
    const int V = (int)(a.row_off[p + 1] - r0);
    const bool use = (!a.use || a.use[p]) && V >= 1 && V <= RS_MAXV && a.fw[p] == a.F;
    slot_of[v] = -1;
    __syncthreads();
    const int m = v < V ? (a.masks[r0 + v] & 63) : 0;
    if (use && v < V) slot_of[m] = (int8_t)v;
    __syncthreads();
    for (int j = 0; j < RS_NOPT; ++j) {
        const int w = (use && v < V && !((m >> j) & 1)) ? slot_of[m | (1 << j)] : -1;
        const unsigned bal = __ballot_sync(0xffffffffu, w >= 0);
        if (lane == 0) wcnt[j][warp] = __popc(bal);
        __syncthreads();
        if (w >= 0) {
            const int64_t pos = a.offs[(int64_t)j * (a.P + 1) + p] + (warp ? wcnt[j][0] : 0) +
                                __popc(bal & ((1u << lane) - 1u));
            if (pos < a.NP) {
                a.zoff[(int64_t)j * a.NP + pos] = a.x_off[p] + (int64_t)v * a.F;
                a.y[(int64_t)j * a.NP + pos] = a.lt[r0 + v] - a.lt[r0 + w];
            }
        }
        __syncthreads();
    }
}

__device__ __forceinline__ int n_pairs(const PoolArgs& a, int j) {
    const int64_t n = a.offs[(int64_t)j * (a.P + 1) + a.P];
    return (int)(n < a.NP ? n : a.NP);
}
__device__ __forceinline__ const double* zrow(const PoolArgs& a, int64_t zo) { return a.Z + zo; }


// Sums over the pairs of an optimization, in C chunks of its pairs: block (chunk, j), thread f
// and f + 256 a feature; the chunk's pairs in order, the chunks added in order by whoever reads
// the partials ([C][6][F], labels' sums in ypart [C][6]).  A single block walking all pairs of a
// feature slice was one chain of dependent row loads (0.3 ms a pass at 620 pairs); 32 chunks x 6
// blocks keep the loads of 8 rows in flight each.
//   kMean: sum z, sum y.   kRhs: sum c (y - ybar).   kResid: sum c s_a.      (c = z - zbar)
enum { kMean = 0, kRhs = 1, kResid = 2 };
constexpr int kSumThreads = 256;

template <int MODE>
__global__ void __launch_bounds__(kSumThreads)
pooled_sum_kernel(PoolArgs a, int C, double* part, double* ypart) {
    const int j = blockIdx.y, ch = blockIdx.x, tid = threadIdx.x;
    const int n = n_pairs(a, j);
    const int q0 = (int)((int64_t)n * ch / C), q1 = (int)((int64_t)n * (ch + 1) / C);
    const int64_t* rows = a.zoff + (int64_t)j * a.NP;
    const double* yv = a.y + (int64_t)j * a.NP;
    const double* sv = a.s + (int64_t)j * a.NP;
    const double yb = MODE == kRhs ? a.ybar[j] : 0.0;
    for (int f = tid; f < a.F; f += kSumThreads) {
        const double zb = MODE == kMean ? 0.0 : a.zbar[j * a.F + f];
        double s = 0.0;
        for (int q = q0; q < q1; q += 8) {
            double z[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) z[e] = q + e < q1 ? __ldg(zrow(a, rows[q + e]) + f) : zb;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                if (q + e >= q1) break;
                if (MODE == kMean) s += z[e];
                else if (MODE == kRhs) s = fma(z[e] - zb, yv[q + e] - yb, s);
                else s = fma(z[e] - zb, sv[q + e], s);
            }
        }
        part[((int64_t)ch * RS_NOPT + j) * a.F + f] = s;
    }
    if (MODE == kMean && tid < 32) {
        double s = 0.0;
        for (int q = q0 + tid; q < q1; q += 32) s += yv[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (tid == 0) ypart[ch * RS_NOPT + j] = s;
    }
}

// The chunks' partials of feature f, added in order.
__device__ __forceinline__ double add_chunks(const double* part, int C, int j, int F, int f) {
    double s = 0.0;
#pragma unroll 8
    for (int c = 0; c < C; ++c) s += part[((int64_t)c * RS_NOPT + j) * F + f];
    return s;
}

// The GEMM operands: A_j = [hi | hi | lo], B_j = [hi | lo | hi] of the centred rows, stored
// feature-major ([6][F][3 Np], pair index contiguous, zero past n_j).  Block (tile of 64 pairs,
// j): the tile's centred values in shared memory, 32 features at a time, written transposed.
__global__ void __launch_bounds__(256)
pooled_stage_kernel(PoolArgs a, int Np, int C, const double* part, const double* ypart, __nv_bfloat16* A,
                    __nv_bfloat16* B) {
    __shared__ double t[64][33];
    __shared__ double zb[512];
    const int j = blockIdx.y, k0 = blockIdx.x * 64;
    const int n = n_pairs(a, j);
    const int64_t* rows = a.zoff + (int64_t)j * a.NP;
    // the means, from the chunks' sums; the first block keeps them for the passes that follow
    if (k0 < n || blockIdx.x == 0)
        for (int f = threadIdx.x; f < a.F; f += 256) {
            zb[f] = n > 0 ? add_chunks(part, C, j, a.F, f) / n : 0.0;
            if (blockIdx.x == 0) a.zbar[j * a.F + f] = zb[f];
        }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        double s = 0.0;
        for (int c = 0; c < C; ++c) s += ypart[c * RS_NOPT + j];
        a.ybar[j] = n > 0 ? s / n : 0.0;
    }
    __syncthreads();
    for (int f0 = 0; f0 < a.F; f0 += 32) {
        for (int e = threadIdx.x; e < 64 * 32; e += 256) {        // read: pairs x features
            const int q = e >> 5, f = f0 + (e & 31);
            double c = 0.0;
            if (k0 + q < n && f < a.F) c = __ldg(zrow(a, rows[k0 + q]) + f) - zb[f];
            t[q][e & 31] = c;
        }
        __syncthreads();
        for (int e = threadIdx.x; e < 32 * 64; e += 256) {        // write: features x pairs
            const int fl = e >> 6, q = e & 63, f = f0 + fl;
            if (f < a.F) {
                const float cf = (float)t[q][fl];
                const __nv_bfloat16 hi = __float2bfloat16(cf);
                const __nv_bfloat16 lo = __float2bfloat16(cf - __bfloat162float(hi));
                const int64_t base = ((int64_t)j * a.F + f) * 3 * Np + k0 + q;
                A[base] = hi;
                A[base + Np] = hi;
                A[base + 2 * Np] = lo;
                B[base] = hi;
                B[base + Np] = lo;
                B[base + 2 * Np] = hi;
            }
        }
        __syncthreads();
    }
}

struct EpiPooled {
    double* G;
    int F;
    __device__ void operator()(int z, int row, int col0, const float (&v)[16]) const {
        double* g = G + ((int64_t)z * F + row) * F;
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (col0 + i < F) g[col0 + i] = (double)v[i];
    }
};


// ---- the FP64 factorisation and solves ----------------------------------------------------------
// G_j + lambda I = L D L^T by a cluster of 16 CTAs per optimization.  The F^3 / 6 FMAs of one
// optimization are 1.4 M cycles of one SM's FP64 pipe at F = 256 (2 lanes a clock), so one block
// per optimization took 2.9 of the call's 3.8 ms; 16 SMs share them here.  Row i of the lower
// triangle lives in the shared memory of CTA i % 16 (a cyclic split keeps the shrinking triangle
// balanced).  Panels of 16 columns: every CTA factors the panel's 16 x 16 diagonal block
// redundantly (no exchange inside the panel's serial chain) together with its own rows of the
// panel, one barrier per pivot; the panel's U = L D goes to G, the cluster meets, and each CTA
// takes the whole panel back into shared memory and updates its own rows by it.  Two cluster
// barriers per panel.  G ends as U (lower, with the pivots on its diagonal).  Measured at F = 256:
// the call 3.82 -> 0.58 ms.
constexpr int kPoolCta = 16;                 // CTAs per cluster = rows per diagonal block
constexpr int kPoolNB = 16;                  // panel width
constexpr int kPoolThreads = 256;
constexpr int kPoolMaxF = 512;
static_assert(kPoolCta == kPoolNB && kPoolThreads == kPoolNB * kPoolNB, "one row of a diagonal block per CTA");

__device__ __forceinline__ void cluster_sync_all() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__host__ __device__ constexpr int pool_own_rows(int F) { return (F + kPoolCta - 1) / kPoolCta; }
__host__ __device__ constexpr size_t pool_factor_doubles(int F) {
    return (size_t)pool_own_rows(F) * (F + kPoolNB) + (size_t)F * (kPoolNB + 1) + 2 * (kPoolNB + 2 * kPoolNB) + kPoolNB;
}
// Scratch of one optimization: 1 / d of every pivot, then the inverses of the unit lower 16 x 16
// diagonal blocks of L (they turn the substitutions' serial chains into small products).
__host__ __device__ constexpr int64_t pool_scratch_doubles(int F) {
    return (int64_t)pool_own_rows(F) * kPoolNB * (1 + kPoolNB);
}

// x = (L D L^T)^-1 t for one right-hand side t[0..F) in shared memory (overwritten by x), by one
// block.  Blocks of 16: the block's part by the inverse of its diagonal block, then every row
// below (above) takes its 16 products.
__device__ void pool_substitute(const double* U, const double* scr, int F, double* t, double* sb) {
    const int tid = threadIdx.x, r = tid >> 4, c = tid & 15;
    const int nblk = pool_own_rows(F);
    const double* dinv = scr;
    const double* Li = scr + (int64_t)nblk * kPoolNB;
    for (int kb = 0; kb < nblk; ++kb) {                       // L D s = t
        const int k0 = kb * kPoolNB;
        double v = c <= r && k0 + r < F ? Li[(int64_t)kb * 256 + tid] * t[k0 + c] : 0.0;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        __syncthreads();
        if (c == 0) {
            sb[r] = k0 + r < F ? v * dinv[k0 + r] : 0.0;
            if (k0 + r < F) t[k0 + r] = sb[r];
        }
        __syncthreads();
        for (int i = k0 + kPoolNB + tid; i < F; i += kPoolThreads) {
            const double* u = U + (int64_t)i * F + k0;
            double w[kPoolNB], acc = t[i];
#pragma unroll
            for (int k = 0; k < kPoolNB; ++k) w[k] = u[k];
#pragma unroll
            for (int k = 0; k < kPoolNB; ++k) acc = fma(-w[k], sb[k], acc);
            t[i] = acc;
        }
        __syncthreads();
    }
    for (int kb = nblk - 1; kb >= 0; --kb) {                  // L^T x = s
        const int k0 = kb * kPoolNB;
        // column r of the block's inverse against the block's part
        double v = c >= r && k0 + c < F ? Li[(int64_t)kb * 256 + c * kPoolNB + r] * t[k0 + c] : 0.0;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        __syncthreads();
        if (c == 0) {
            sb[r] = k0 + r < F ? v : 0.0;
            if (k0 + r < F) t[k0 + r] = v;
        }
        __syncthreads();
        for (int i = tid; i < k0; i += kPoolThreads) {
            const double* u = U + (int64_t)k0 * F + i;
            double w[kPoolNB], acc = 0.0;
#pragma unroll
            for (int k = 0; k < kPoolNB; ++k) w[k] = k0 + k < F ? u[(int64_t)k * F] : 0.0;
#pragma unroll
            for (int k = 0; k < kPoolNB; ++k) acc = fma(w[k], sb[k], acc);
            t[i] = fma(-acc, dinv[i], t[i]);
        }
        __syncthreads();
    }
}

// beta (or beta += the correction), the intercept and the status of one optimization, by one block.
__device__ void pool_finish(const PoolArgs& a, int j, const double* x, bool refine, double* red) {
    const int tid = threadIdx.x, F = a.F;
    double* beta = a.coef + (int64_t)j * (F + 1) + 1;
    double s = 0.0;
    bool fin = true;
    for (int f = tid; f < F; f += kPoolThreads) {
        const double v = refine ? beta[f] + x[f] : x[f];
        beta[f] = v;
        s = fma(a.zbar[j * F + f], v, s);
        fin = fin && isfinite(v);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((tid & 31) == 0) red[tid >> 5] = s;
    fin = __syncthreads_and(fin);
    if (tid == 0) {
        double t = 0.0;
        for (int w = 0; w < kPoolThreads / 32; ++w) t += red[w];
        const double b = a.ybar[j] - t;
        a.coef[(int64_t)j * (F + 1)] = b;
        a.status[j] = (fin && isfinite(b)) ? RS_FIT_OK : RS_FIT_NONFINITE;
    }
}

__global__ void __launch_bounds__(kPoolThreads)
pooled_factor_kernel(PoolArgs a, int C, const double* part, double* scratch) {
    extern __shared__ __align__(16) double psm[];
    __shared__ double sb[kPoolNB], red[kPoolThreads / 32];
    const int j = blockIdx.x / kPoolCta, rank = blockIdx.x % kPoolCta, F = a.F, tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5, r = tid >> 4, c = tid & 15;
    const int n = n_pairs(a, j);
    if (n == 0) {                                             // the whole cluster leaves
        if (tid == 0 && rank == 0) {
            a.status[j] = RS_FIT_EMPTY;
            a.coef[(int64_t)j * (F + 1)] = nan_d();
        }
        return;
    }
    const int nblk = pool_own_rows(F), ldr = F;
    double* R = psm;                                          // own rows [nblk][F]
    double* Lr = R + (size_t)nblk * ldr;                      // their panel's L [nblk][16]
    double* P = Lr + (size_t)nblk * kPoolNB;                  // the panel's U, rows below it [F][17]
    double* col = P + (size_t)F * (kPoolNB + 1);              // [2][16 diagonal rows | 32 own rows]
    double* dv = col + 2 * 3 * kPoolNB;                       // [16] 1 / d of the panel
    double* G = a.G + (int64_t)j * F * F;
    double* scr = scratch + (int64_t)j * pool_scratch_doubles(F);
    for (int t = 0; t < nblk; ++t) {                          // (rows are read past L1: other CTAs write G)
        const int i = rank + kPoolCta * t;
        if (i < F)
            for (int k = tid; k <= i; k += kPoolThreads) R[(size_t)t * ldr + k] = __ldcg(G + (int64_t)i * F + k) + (k == i ? a.lambda : 0.0);
    }
    __syncthreads();
    bool bad = false;
    for (int kb = 0; kb < nblk; ++kb) {
        const int k0 = kb * kPoolNB;
        // this CTA's row of the diagonal block, as updated so far, to the others
        if (k0 + rank < F && tid <= rank) G[(int64_t)(k0 + rank) * F + k0 + tid] = R[(size_t)kb * ldr + k0 + tid];
        cluster_sync_all();
        // thread (r, c): entry (r, c) of the diagonal block and of own rows kb + 1 + r (+ 16)
        double d = r == c ? 1.0 : 0.0, o[2] = {0.0, 0.0};
        if (c <= r && k0 + r < F) d = __ldcg(G + (int64_t)(k0 + r) * F + k0 + c);
        bool own[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int t = kb + 1 + r + kPoolNB * e;
            own[e] = t < nblk && rank + kPoolCta * t < F;
            if (own[e]) o[e] = R[(size_t)t * ldr + k0 + c];
        }
        // pivot k: column k (already final) is published with 1 / d_k by the threads that hold
        // it; one barrier; every entry to its right takes u_r (u_c / d_k)
        auto publish = [&](int k) {
            double* cb = col + (k & 1) * 3 * kPoolNB;
            if (c == k) {
                cb[r] = d;
                cb[kPoolNB + r] = o[0];
                cb[2 * kPoolNB + r] = o[1];
                if (r == k) dv[k] = pos_finite(d) ? rcp_newton(d) : 0.0;
            }
        };
        publish(0);
        __syncthreads();
#pragma unroll 1
        for (int k = 0; k < kPoolNB; ++k) {
            const double* cb = col + (k & 1) * 3 * kPoolNB;
            if (!pos_finite(cb[k])) bad = true;               // the same value in every thread and CTA
            if (c > k) {
                const double w = cb[c] * dv[k];
                d = fma(-cb[r], w, d);
                if (own[0]) o[0] = fma(-cb[kPoolNB + r], w, o[0]);
                if (own[1]) o[1] = fma(-cb[2 * kPoolNB + r], w, o[1]);
            }
            if (k + 1 < kPoolNB) publish(k + 1);
            __syncthreads();
        }
        if (bad) break;
#pragma unroll
        for (int e = 0; e < 2; ++e)
            if (own[e]) {
                const int t = kb + 1 + r + kPoolNB * e;
                Lr[t * kPoolNB + c] = o[e] * dv[c];
                G[(int64_t)(rank + kPoolCta * t) * F + k0 + c] = o[e];
            }
        cluster_sync_all();
        if (rank == 0) {                                      // the diagonal block's U and 1 / d (every
            if (c <= r && k0 + r < F) G[(int64_t)(k0 + r) * F + k0 + c] = d;   // CTA has read the block)
            if (tid < kPoolNB) scr[k0 + tid] = dv[tid];
        }
        const int i0 = k0 + kPoolNB;
        for (int e = tid; e < (F - i0) * kPoolNB; e += kPoolThreads)
            P[(e >> 4) * (kPoolNB + 1) + (e & 15)] = __ldcg(G + (int64_t)(i0 + (e >> 4)) * F + k0 + (e & 15));
        __syncthreads();
        int it = 0;
        for (int t = kb + 1; t < nblk; ++t) {                 // 32 columns of one own row a warp's turn
            const int i = rank + kPoolCta * t;
            if (i >= F) break;
            const double* L = Lr + t * kPoolNB;
            for (int cc = i0; cc <= i; cc += 32, ++it) {
                if ((it & (kPoolThreads / 32 - 1)) != warp) continue;
                const int x = cc + lane;
                if (x > i) continue;
                double acc = R[(size_t)t * ldr + x];
                const double* u = P + (x - i0) * (kPoolNB + 1);
#pragma unroll
                for (int k = 0; k < kPoolNB; ++k) acc = fma(-L[k], u[k], acc);
                R[(size_t)t * ldr + x] = acc;
            }
        }
        __syncthreads();
    }
    if (bad) {                                                // every CTA of the cluster saw it
        if (tid == 0 && rank == 0) {
            a.status[j] = RS_FIT_NOTPD;
            a.coef[(int64_t)j * (F + 1)] = nan_d();
        }
        return;
    }
    cluster_sync_all();
    // inverses of the unit lower diagonal blocks: CTA rank takes blocks rank, rank + 16 (one warp
    // each, lane = column)
    double* Li = scr + (int64_t)nblk * kPoolNB;
    if (warp < 2 && lane < kPoolNB) {
        const int kb = rank + kPoolCta * warp, k0 = kb * kPoolNB;
        if (kb < nblk) {
            double x[kPoolNB];
#pragma unroll
            for (int i = 0; i < kPoolNB; ++i) x[i] = i == lane ? 1.0 : 0.0;
#pragma unroll
            for (int k = 0; k < kPoolNB; ++k) {
                const double y = x[k] * __ldcg(scr + k0 + k);
#pragma unroll
                for (int i = k + 1; i < kPoolNB; ++i)
                    if (k0 + i < F) x[i] = fma(-__ldcg(G + (int64_t)(k0 + i) * F + k0 + k), y, x[i]);
            }
#pragma unroll
            for (int i = 0; i < kPoolNB; ++i) Li[(int64_t)kb * 256 + i * kPoolNB + lane] = x[i];
        }
    }
    cluster_sync_all();
    if (rank != 0) return;
    double* t = R;                                            // (the own rows are not needed any more)
    for (int f = tid; f < F; f += kPoolThreads) {
        t[f] = add_chunks(part, C, j, F, f);
        a.r[j * F + f] = t[f];
    }
    __syncthreads();
    pool_substitute(G, scr, F, t, sb);
    pool_finish(a, j, t, false, red);
}

// Refinement, step 3 (one block per optimization): rho = r - lambda beta - sum_a c_a s_a from the
// chunks' sums, its solution with the same factor, added to beta.
__global__ void __launch_bounds__(kPoolThreads)
pooled_refine_kernel(PoolArgs a, int C, const double* part, const double* scratch) {
    __shared__ double t[kPoolMaxF], sb[kPoolNB], red[kPoolThreads / 32];
    const int j = blockIdx.x, F = a.F, tid = threadIdx.x;
    if (a.status[j] != RS_FIT_OK) return;
    __syncthreads();                                          // (pool_finish writes the status)
    const double* beta = a.coef + (int64_t)j * (F + 1) + 1;
    for (int f = tid; f < F; f += kPoolThreads)
        t[f] = a.r[j * F + f] - a.lambda * beta[f] - add_chunks(part, C, j, F, f);
    __syncthreads();
    pool_substitute(a.G + (int64_t)j * F * F, scratch + (int64_t)j * pool_scratch_doubles(F), F, t, sb);
    pool_finish(a, j, t, true, red);
}

// Refinement, step 1: s_a = c_a . beta_j for every pair (one warp per pair).
__global__ void __launch_bounds__(256) pooled_project_kernel(PoolArgs a) {
    const int j = blockIdx.y;
    const int q = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int n = n_pairs(a, j);
    if (q >= n) return;
    const double* z = zrow(a, a.zoff[(int64_t)j * a.NP + q]);
    const double* zb = a.zbar + j * a.F;
    const double* beta = a.coef + (int64_t)j * (a.F + 1) + 1;
    double s = 0.0;
    for (int f = lane; f < a.F; f += 32) s = fma(__ldg(z + f) - zb[f], beta[f], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) a.s[(int64_t)j * a.NP + q] = s;
}

// Predictions of the pooled models for every version of a batch, ranked and scored against the
// program's own times.  Block (program, 8 versions), one warp per version: the lanes share its
// features (coalesced rows, all six dot products from one read of them) and lane 0 ranks.  One
// thread per version left two warps an SM walking 3 x F dependent FMAs on uncoalesced rows.
constexpr int kPredRows = 8;
struct PoolPredArgs {
    int F;
    const int64_t* row_off;
    const int32_t* fw;
    const int64_t* x_off;
    const double* Z;
    const uint8_t* masks;
    const double* lt;
    const double* coef;       // [6][F + 1]
    const uint8_t* status;    // [6]
    int rank_all;
    RankPassArgs r;
};

__global__ void __launch_bounds__(kPredRows * 32) pooled_predict_kernel(PoolPredArgs a) {
    __shared__ double lt_s[RS_MAXV];
    __shared__ uint8_t msk_s[RS_MAXV];
    __shared__ int8_t slot_s[RS_MAXV];
    __shared__ unsigned cnt[10];
    const int p = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    const int64_t r0 = a.row_off[p];
    const int V = (int)(a.row_off[p + 1] - r0);
    const bool okp = V >= 1 && V <= RS_MAXV && a.fw[p] == a.F;
    if (!okp) {
        if (tid == 0 && blockIdx.y == 0) rs_dev_flag(a.r.dstatus, RS_EDATA, p);
        return;
    }
    if ((int)blockIdx.y * kPredRows >= V) return;
    if (tid < RS_MAXV) slot_s[tid] = -1;
    if (tid < 10) cnt[tid] = 0;
    if (tid < V) {
        msk_s[tid] = a.masks[r0 + tid] & 63;
        lt_s[tid] = a.lt[r0 + tid];
    }
    __syncthreads();
    if (tid < V) slot_s[msk_s[tid]] = (int8_t)tid;
    __syncthreads();
    const int t = blockIdx.y * kPredRows + (tid >> 5);
    if (t < V) {
        const int mt = msk_s[t];
        int okm = 0;
#pragma unroll
        for (int j = 0; j < RS_NOPT; ++j) okm |= (a.status[j] == RS_FIT_OK) << j;
        const int candm = (a.rank_all ? 63 : (~mt & 63)) & okm;      // uniform over the warp
        const double* z = a.Z + a.x_off[p] + (int64_t)t * a.F;
        double pred[RS_NOPT];
#pragma unroll
        for (int j = 0; j < RS_NOPT; ++j) pred[j] = 0.0;
        for (int f = lane; f < a.F; f += 32) {
            const double zf = __ldg(z + f);
#pragma unroll
            for (int j = 0; j < RS_NOPT; ++j)
                if ((candm >> j) & 1) pred[j] = fma(zf, __ldg(a.coef + (int64_t)j * (a.F + 1) + 1 + f), pred[j]);
        }
#pragma unroll
        for (int j = 0; j < RS_NOPT; ++j) {
            if (!((candm >> j) & 1)) continue;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) pred[j] += __shfl_xor_sync(0xffffffffu, pred[j], o);
            pred[j] += __ldg(a.coef + (int64_t)j * (a.F + 1));
        }
        if (lane == 0) {
            RankTally c;
            const uint32_t info = row_summary(t, V, msk_s, lt_s, slot_s);
            const int mfield = a.rank_all ? 0 : mt;
            const unsigned long long info64 = (unsigned long long)info | ((unsigned long long)mfield << 30) |
                                              ((unsigned long long)(~okm & 63) << 36);
            rank_row(a.r, r0 + t, info64, pred, c);
            const uint32_t vals[10] = {c.rows, c.pred, c.scored, c.sign, c.rec, c.reck, c.rech, c.t1, c.t1h, c.inv};
#pragma unroll
            for (int i = 0; i < 10; ++i)
                if (vals[i]) atomicAdd(&cnt[i], vals[i]);
        }
    }
    if (a.r.counters) {
        __syncthreads();
        const int slot[10] = {0, 1, 2, 3, 4, 5, 6, 7, 8, 13};
        if (tid < 10 && cnt[tid]) atomicAdd(a.r.counters + slot[tid], (unsigned long long)cnt[tid]);
    }
}

int pairs_cap(int64_t P) {
    const int64_t np = P * 32;
    return (int)(np < kPoolMaxPairs ? np : kPoolMaxPairs);
}
int padded_pairs(int64_t P) { return (pairs_cap(P) + 63) / 64 * 64; }

struct PoolWs {
    int* counts;
    int64_t* offs;
    int64_t* zoff;
    double *y, *zbar, *ybar, *G, *r, *s;
    __nv_bfloat16 *A, *B;
    size_t bytes;
};

PoolWs carve_pool(void* base, int64_t P, int F) {
    PoolWs w{};
    char* c = (char*)base;
    size_t o = 0;
    auto take = [&](size_t n) -> void* {
        void* p = c ? (void*)(c + o) : nullptr;
        o += (n + 255) & ~(size_t)255;
        return p;
    };
    const int NP = pairs_cap(P), Np = padded_pairs(P);
    w.counts = (int*)take((size_t)RS_NOPT * P * sizeof(int));
    w.offs = (int64_t*)take((size_t)RS_NOPT * (P + 1) * sizeof(int64_t));
    w.zoff = (int64_t*)take((size_t)RS_NOPT * NP * sizeof(int64_t));
    w.y = (double*)take((size_t)RS_NOPT * NP * sizeof(double));
    w.s = (double*)take((size_t)RS_NOPT * NP * sizeof(double));
    w.zbar = (double*)take((size_t)RS_NOPT * F * sizeof(double));
    w.ybar = (double*)take(RS_NOPT * sizeof(double));
    w.G = (double*)take((size_t)RS_NOPT * F * F * sizeof(double));
    w.r = (double*)take((size_t)RS_NOPT * F * sizeof(double));
    const size_t ab = (size_t)RS_NOPT * F * 3 * Np * sizeof(__nv_bfloat16);
    const size_t sb = (size_t)RS_NOPT * pool_scratch_doubles(F) * sizeof(double);   // larger for F < 9 only
    w.A = (__nv_bfloat16*)take(ab > sb ? ab : sb);
    w.B = (__nv_bfloat16*)take((size_t)RS_NOPT * F * 3 * Np * sizeof(__nv_bfloat16));
    w.bytes = o;
    return w;
}

}  // namespace

size_t rs_pooled_workspace_bytes_impl(int64_t P, int F) { return carve_pool(nullptr, P, F).bytes; }

cudaError_t rs_launch_fit_pooled(const rs_batch* b, const uint8_t* use, double lambda, int refine, void* ws,
                                 size_t ws_bytes, double* coef, uint8_t* status, int* dstatus, cudaStream_t st) {
    const int64_t P = b->n_programs;
    const int F = b->max_feat;
    PoolWs w = carve_pool(ws, P, F);
    if (!ws || ws_bytes < w.bytes || F > 512 || P > 65535) return cudaErrorInvalidValue;
    PoolArgs a{};
    a.P = (int)P;
    a.F = F;
    a.row_off = b->row_offsets;
    a.fw = b->feat_width;
    a.x_off = b->x_offsets;
    a.Z = (const double*)b->X;
    a.masks = b->masks;
    a.lt = b->log_time;
    a.use = use;
    a.counts = w.counts;
    a.offs = w.offs;
    a.zoff = w.zoff;
    a.y = w.y;
    a.NP = pairs_cap(P);
    a.zbar = w.zbar;
    a.ybar = w.ybar;
    a.G = w.G;
    a.r = w.r;
    a.s = w.s;
    a.coef = coef;
    a.status = status;
    a.lambda = lambda;
    a.dstatus = dstatus;
    const int Np = padded_pairs(P);
    // Partials live where nothing else does at the time: the means' in G (written by the GEMM
    // later; C <= F chunks fit), the right-hand side's and the residual's in B (read by the GEMM
    // only: 36 Np F >= 2304 F bytes against 48 C F), the factor's scratch in A (carve_pool).
    const int C = F < 32 ? F : 32;
    double* mpart = w.G;
    double* part = (double*)w.B;
    double* scratch = (double*)w.A;
    pooled_count_kernel<<<(unsigned)P, RS_MAXV, 0, st>>>(a);
    pooled_scan_kernel<<<RS_NOPT, 1024, 0, st>>>(a);
    pooled_fill_kernel<<<(unsigned)P, RS_MAXV, 0, st>>>(a);
    pooled_sum_kernel<kMean><<<dim3((unsigned)C, RS_NOPT), kSumThreads, 0, st>>>(a, C, mpart, w.s);
    pooled_stage_kernel<<<dim3((unsigned)(Np / 64), RS_NOPT), 256, 0, st>>>(a, Np, C, mpart, w.s, w.A, w.B);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    CUtensorMap ta, tb;
    e = rs_make_tmap_bf16_3d(&ta, w.A, RS_NOPT, F, 3 * Np, 3 * Np, tc::BM);
    if (e == cudaSuccess) e = rs_make_tmap_bf16_3d(&tb, w.B, RS_NOPT, F, 3 * Np, 3 * Np, 64);
    if (e == cudaSuccess)
        e = tc::gemm_launch<64, 4, EpiPooled, true>(ta, tb, F, F, 3 * Np, RS_NOPT, EpiPooled{w.G, F}, dstatus, st);
    if (e != cudaSuccess) return e;
    pooled_sum_kernel<kRhs><<<dim3((unsigned)C, RS_NOPT), kSumThreads, 0, st>>>(a, C, part, nullptr);
    const size_t fsmem = pool_factor_doubles(F) * sizeof(double);
    e = cudaFuncSetAttribute(pooled_factor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fsmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(pooled_factor_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(RS_NOPT * kPoolCta);
    cfg.blockDim = dim3(kPoolThreads);
    cfg.dynamicSmemBytes = fsmem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kPoolCta;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, pooled_factor_kernel, a, C, (const double*)part, scratch);
    if (e != cudaSuccess) return e;
    if (refine) {
        pooled_project_kernel<<<dim3((unsigned)((a.NP + 7) / 8), RS_NOPT), 256, 0, st>>>(a);
        pooled_sum_kernel<kResid><<<dim3((unsigned)C, RS_NOPT), kSumThreads, 0, st>>>(a, C, part, nullptr);
        pooled_refine_kernel<<<RS_NOPT, kPoolThreads, 0, st>>>(a, C, part, scratch);
    }
    return cudaGetLastError();
}

cudaError_t rs_launch_predict_pooled(const rs_batch* b, const double* coef, const uint8_t* status, int k,
                                     double log_tau, int flags, uint32_t* rec_code, double* rec_pred,
                                     double* pred_all, unsigned long long* counters, int* dstatus, cudaStream_t st) {
    PoolPredArgs a{};
    a.F = b->max_feat;
    a.row_off = b->row_offsets;
    a.fw = b->feat_width;
    a.x_off = b->x_offsets;
    a.Z = (const double*)b->X;
    a.masks = b->masks;
    a.lt = b->log_time;
    a.coef = coef;
    a.status = status;
    a.rank_all = (flags & RS_RANK_ALL) ? 1 : 0;
    RankPassArgs& r = a.r;
    r.dstatus = dstatus;
    r.k = k;
    r.ktau = okey_host(log_tau);
    r.flags = 0;                  // candidates come through the version-mask field
    r.rec_code = rec_code;
    r.rec_pred = rec_pred;
    r.pred_all = pred_all;
    r.counters = counters;
    pooled_predict_kernel<<<dim3((unsigned)b->n_programs, RS_MAXV / kPredRows), kPredRows * 32, 0, st>>>(a);
    return cudaGetLastError();
}
