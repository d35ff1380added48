// K1: feature vectors (Sec. 2: counters normalised by the cycle count), followed by the
// library's log / per-program z-score reading.  One read of X, one write of Z.
//
// This part's FP64 pipe takes 64 cycles for a warp instruction, its integer multiplier 2 to 4, so
// the logarithms, their mean and the centring run in 64-bit fixed point (53 fraction bits, |log q|
// < 1024) and FP64 is left with two instructions per element: the square that the deviation sums
// and the product that scales it.  log(x / c) is log x - log c, the second taken once per version.
// 256 programs x 64 versions x 1024 FP64 counters: 562 -> 149 us (the two passes over
// memory alone take 40 us); 64 programs x 40 x 256 FP32: 41 -> 16 us.
#include "mbar.cuh"
#include "rank_row.cuh"
#include "rs_internal.cuh"
#include "rs_log_table.h"

namespace {

constexpr long long kClampBits = 0x39b4484bfeebc2a0ll;   // bit pattern of 1e-30
constexpr long long kInfBits = 0x7ff0000000000000ll;
constexpr long long kFixInf = 0x7fffffffffffffffll;       // log of +inf
constexpr long long kFixNone = -0x7fffffffffffffffll - 1; // a cycle count outside the fast range

// log q in units of 2^-53 for the bit pattern of a positive, normal, finite q = 2^e m, m in
// [1, 2).  After P. T. P. Tang's table-driven method (ACM TOMS 16(4), 1990), in integers: the top
// eight fraction bits of m pick an 11-bit c with m c / 2^11 = 1 + r, |r| < 1.26 2^-9, so r is exact
// in 63 fraction bits; log q = e ln2 - log(c / 2^11) + r - r^2/2 + r^3/3 - r^4/4 + r^5/5 - r^6/6.
// r^2 comes from r's 39-bit and 24-bit halves (78 fraction bits), r^3/3 from 31-bit pieces, the
// terms from r^4 on (below 2^-36) in FP32 with the 2^23-offset conversion; ln2 and the logarithms
// have 63 fraction bits.  Against an 80-bit logarithm over 8e7 arguments (exponents -511 .. 510,
// and q within 2^-50 .. 1 of 1): error at most 0.625 units of 2^-53, rms 0.27 (the FP64 form it
// replaces: 2.4 units of 2^-53 max(1, |log q|), rms 0.52, and 9 FP64 instructions).
__device__ __forceinline__ long long fix_log(unsigned hi, unsigned lo, const long long* tl, const uint16_t* tc) {
    const int e = (int)(hi >> 20) - 1023;
    const unsigned mh = (hi & 0xfffffu) | 0x100000u;
    const int i = (int)(mh >> 12) & 0xff;
    const unsigned c = tc[i];
    const long long r = (long long)(((unsigned long long)(mh * c - 0x80000000u) << 32) + (unsigned long long)lo * c);
    const int rh = (int)((r + (1 << 23)) >> 24);                       // 39 fraction bits
    const int rl = (int)(r - ((long long)rh << 24));
    const long long r2 = (long long)rh * rh + (((long long)rh * rl) >> 23);        // 78
    const int r23 = (int)(((long long)(int)(r2 >> 30) * 0x55555555) >> 31);        // r^2 / 3: 49
    const long long t3 = (long long)r23 * rh;                          // 88
    const float rf = (float)rh * 0x1p-39f, q = rf * rf;
    const float t = fmaf(q * q * 0x1p58f, fmaf(q, -1.0f / 6.0f, fmaf(rf, 0.2f, -0.25f)), 12582912.0f);
    const int ti = __float_as_int(t) - 0x4B400000;                     // 58
    const long long s = tl[i] + r - (r2 >> 16) + (t3 >> 25) + ((long long)ti << 5);
    return ((long long)e * kFixLn2Hi << 22) + (((long long)e * kFixLn2Lo + s + 512) >> 10);
}

// The value 2^-53 v as a double, rounded to nearest, by integer operations.
__device__ __forceinline__ double fix_double(long long v) {
    const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    if (a == 0) return 0.0;
    const int lz = __clzll((long long)a);
    const unsigned long long m = a << lz;
    const unsigned long long b = ((unsigned long long)(1023 - 53 + 63 - 1 - lz) << 52) + (m >> 11) + ((m >> 10) & 1ull);
    return __longlong_as_double((long long)(b | ((unsigned long long)v & 0x8000000000000000ull)));
}

__device__ __forceinline__ long long fix_log(double q, const long long* tl, const uint16_t* tc) {
    const long long b = __double_as_longlong(q);
    return fix_log((unsigned)(b >> 32), (unsigned)b, tl, tc);
}

// log(max(q, 1e-30)) with the branches of the plain definition: above the clamp and finite -> its
// logarithm (subnormal q never reach it); +inf -> +inf; q <= 1e-30 or NaN -> log(1e-30).
__device__ __forceinline__ long long fix_log_clamped(double q, const long long* tl, const uint16_t* tc) {
    const long long b = __double_as_longlong(q);
    if (b > kClampBits && b < kInfBits) return fix_log(q, tl, tc);
    return b == kInfBits ? kFixInf : kFixClamp;
}

// A version's cycle count: its logarithm, or kFixNone unless it is positive with an exponent in
// -511 .. 511 (then the difference of two logarithms of that range fits the fixed point).
__device__ __forceinline__ bool fast_hi(unsigned hi) { return hi - (512u << 20) < (1023u << 20); }
__device__ __forceinline__ long long cycle_log(double c, const long long* tl, const uint16_t* tc) {
    return fast_hi((unsigned)__double2hiint(c)) ? fix_log(c, tl, tc) : kFixNone;
}

// log(max(x / c, 1e-30)) of an element; lc = cycle_log(c).  Any value outside the fast range (zeros,
// subnormals, negatives, infinities, NaN, extreme exponents) takes the plain definition's division.
__device__ __forceinline__ long long elem_log(double x, bool cyc, double c, long long lc, const long long* tl,
                                              const uint16_t* tc) {
    const unsigned hi = (unsigned)__double2hiint(x);
    if (!fast_hi(hi) || (cyc && lc == kFixNone)) {
        if ((hi << 1 | (unsigned)__double2loint(x)) == 0u) return kFixClamp;      // 0 (by any c: no more, or NaN)
        return fix_log_clamped(cyc ? x * (1.0 / c) : x, tl, tc);
    }
    const long long l = fix_log(hi, (unsigned)__double2loint(x), tl, tc) - (cyc ? lc : 0ll);
    return l > kFixClamp ? l : kFixClamp;
}
__device__ __forceinline__ long long elem_log(float x, bool cyc, double c, long long lc, const long long* tl,
                                              const uint16_t* tc) {
    const unsigned u = __float_as_uint(x);
    if (u - (1u << 23) >= (254u << 23) || (cyc && lc == kFixNone)) {   // not a positive normal number
        if (u << 1 == 0u) return kFixClamp;
        return fix_log_clamped(cyc ? (double)x * (1.0 / c) : (double)x, tl, tc);
    }
    const long long l = fix_log((u >> 3) + (896u << 20), u << 29, tl, tc) - (cyc ? lc : 0ll);
    return l > kFixClamp ? l : kFixClamp;
}

__device__ __forceinline__ void load_log_tables(long long* tl, uint16_t* tc, int threads) {
    for (int t = threadIdx.x; t < 256; t += threads) {
        tl[t] = kFixLogTab[t];
        tc[t] = kFixRcpTab[t];
    }
}

constexpr int kThreads = 256;

// The mean of n logarithms from the sums of their halves (v >> 24 and v & 0xffffff), rounded to
// the fixed point.
__device__ __forceinline__ long long fix_mean(long long hs, long long ls, int n) {
    const long long q = hs / n;
    const long long rem = ((hs - q * n) << 24) + ls;
    return (q << 24) + (rem + (rem >= 0 ? n / 2 : -(n / 2))) / n;
}

// What the two kernels below do once a thread holds its ROWS logarithms of feature fl (rows r0,
// r0 + GROUPS, ..., those below n; r0 = g, the thread's row group): the mean and the deviation over the
// n rows of the block's feature, then the centred values (as doubles) and 1 / sigma (0: a constant or
// non-finite feature).
// PAIR (16 groups, two a warp): r0 = pair_row(g), and the squares are added in the order of eight groups,
// so that a program's outputs do not depend on the form that the rest of its batch asks for (one chain of
// eight rows in two lanes, but half the sums to add at the end).
template <int FEAT, int ROWS>
struct StdSmem {
    static constexpr int kGroups = kThreads / FEAT;
    long long ph[kGroups][FEAT], mean[FEAT];
    double pq[kGroups][FEAT], rs[FEAT];
    unsigned pl[kGroups][FEAT];
    int inf[FEAT];
    long long tl[256];
    uint16_t tc[256];
};

__device__ __forceinline__ int pair_row(int g) { return (g >> 1) + 8 * (g & 1); }

template <int FEAT, int ROWS, bool PAIR = false>
__device__ __forceinline__ double centre(StdSmem<FEAT, ROWS>& S, const long long (&l)[ROWS], double (&d)[ROWS], int n,
                                         bool active, double* mu, double* sigma) {
    constexpr int G = kThreads / FEAT, kSums = PAIR ? G / 2 : G;
    const int fl = threadIdx.x % FEAT, g = threadIdx.x / FEAT, r0 = PAIR ? pair_row(g) : g;
    long long hs = 0;
    unsigned ls = 0;
#pragma unroll
    for (int q = 0; q < ROWS; ++q)
        if (active && r0 + G * q < n) {
            if (l[q] == kFixInf) S.inf[fl] = 1;
            hs += l[q] >> 24;
            ls += (unsigned)l[q] & 0xffffffu;
        }
    S.ph[g][fl] = hs;
    S.pl[g][fl] = ls;
    __syncthreads();
    if (threadIdx.x < FEAT) {
        hs = 0;
        long long lt = 0;
#pragma unroll
        for (int q = 0; q < G; ++q) {
            hs += S.ph[q][fl];
            lt += S.pl[q][fl];
        }
        S.mean[fl] = fix_mean(hs, lt, n);
    }
    __syncthreads();
    const long long m = S.mean[fl];
    double q2 = 0.0;
#pragma unroll
    for (int q = 0; q < ROWS; ++q) {
        d[q] = 0.0;
        if (active && r0 + G * q < n) {
            d[q] = fix_double(l[q] - m);
            if constexpr (!PAIR) q2 = fma(d[q], d[q], q2);
        }
    }
    if constexpr (PAIR) {                      // rows g / 2, g / 2 + 8, ... of both lanes, in order
#pragma unroll
        for (int q = 0; q < ROWS; ++q) {
            const double e = __shfl_xor_sync(0xffffffffu, d[q], 16);
            const double a = g & 1 ? e : d[q], b = g & 1 ? d[q] : e;
            q2 = fma(b, b, fma(a, a, q2));
        }
    }
    S.pq[g][fl] = q2;
    __syncthreads();
    if (threadIdx.x < FEAT) {
        double t = 0.0;
#pragma unroll
        for (int q = 0; q < kSums; ++q) t += S.pq[q * (G / kSums)][fl];
        t = t * rcp_newton((double)n);
        const bool inf = S.inf[fl] != 0;
        const bool ok = !inf && t > 1e-24;                   // sigma > 1e-12
        const double r = ok ? rsqrt_newton(t) : 0.0;
        S.rs[fl] = r;
        if (active && mu) *mu = inf ? __longlong_as_double(kInfBits) : fix_double(m);
        if (active && sigma) *sigma = inf ? nan_d() : sqrt(t);
    }
    __syncthreads();
    return S.rs[fl];
}

// Block = (program, FEAT-feature slice); thread (g, f) takes rows g, g + GROUPS, ... of feature f
// and keeps them in registers.  A half-warp's or a warp's lanes read consecutive features.  32
// features (8 rows a thread) halve the narrow per-feature work of the statistics per element and
// are taken once the grid fills the chip (256 programs x 1024 features: 149 us against 177 with 16;
// 64 x 256: 15.9 against 17.9); 16 (4 rows a thread) leave the shorter chain for few programs (2
// programs x 96 features: 8.4 us against 9.9 with 32).
template <typename T, int FEAT>
__global__ void __launch_bounds__(kThreads)
standardize_kernel(int P, const int64_t* __restrict__ row_off, const int32_t* __restrict__ fw,
                   const int64_t* __restrict__ xo, const int64_t* __restrict__ fo,
                   const T* __restrict__ X, const double* __restrict__ cycles,
                   double* __restrict__ Z, double* __restrict__ mu, double* __restrict__ sigma,
                   int* dstatus) {
    constexpr int G = kThreads / FEAT, ROWS = RS_MAXV / G;
    constexpr bool PAIR = G == 16;
    static_assert(G == 8 || G == 16, "the squares are added as by eight groups");
    __shared__ StdSmem<FEAT, ROWS> S;
    __shared__ double cyc_s[RS_MAXV];
    __shared__ long long lc_s[RS_MAXV];
    const int p = blockIdx.x;
    const int64_t r0 = row_off[p];
    const int V = (int)(row_off[p + 1] - r0);
    const int F = fw[p];
    const int fl = threadIdx.x % FEAT, g = PAIR ? pair_row(threadIdx.x / FEAT) : threadIdx.x / FEAT;
    const int f = blockIdx.y * FEAT + fl;
    if (blockIdx.y * FEAT >= F) return;
    if (V < 1 || V > RS_MAXV) {
        if (threadIdx.x == 0 && blockIdx.y == 0) rs_dev_flag(dstatus, RS_EDATA, p);
        return;
    }
    const int64_t base = xo[p];
    const bool active = f < F;
    T x[ROWS];
#pragma unroll
    for (int q = 0; q < ROWS; ++q) x[q] = active && g + G * q < V ? X[base + (int64_t)(g + G * q) * F + f] : (T)1;
    load_log_tables(S.tl, S.tc, kThreads);
    if (threadIdx.x < FEAT) S.inf[threadIdx.x] = 0;
    __syncthreads();
    if (cycles && threadIdx.x < V) {
        const double c = cycles[r0 + threadIdx.x];
        cyc_s[threadIdx.x] = c;
        lc_s[threadIdx.x] = cycle_log(c, S.tl, S.tc);
    }
    __syncthreads();
    long long l[ROWS];
#pragma unroll
    for (int q = 0; q < ROWS; ++q) {
        const int r = g + G * q;
        l[q] = r < V ? elem_log(x[q], cycles != nullptr, cyc_s[r], lc_s[r], S.tl, S.tc) : 0;
    }
    double d[ROWS];
    const double rs = centre<FEAT, ROWS, PAIR>(S, l, d, V, active, mu && active ? mu + fo[p] + f : nullptr,
                             sigma && active ? sigma + fo[p] + f : nullptr);
    if (!active) return;
#pragma unroll
    for (int q = 0; q < ROWS; ++q)
        if (g + G * q < V) Z[base + (int64_t)(g + G * q) * F + f] = rs > 0.0 ? d[q] * rs : 0.0;
}

// Standardization of the training side of a transfer (Table 2): problem q trains on the runs
// group_off[q] .. group_off[q+1]-1 (each laid out like one program: at most 64 versions, all
// with the width F of the problem's test program), standardized together -- mu, sigma over
// the vectors of all of them -- into Z in X's layout; mu, sigma at q * stat_stride + f.
// Block = (problem, 16-feature slice), as standardize_kernel with up to kGroupRows rows.
constexpr int kGroupRows = RS_MAXV * RS_MAXRUNS;
constexpr int kFeat = 16;                    // features per block
constexpr int kGroups = kThreads / kFeat;    // row groups per block

template <typename T, int RUNS>
__global__ void __launch_bounds__(kThreads)
group_standardize_kernel(const int64_t* __restrict__ group_off, int max_runs, int64_t n_runs,
                         const int64_t* __restrict__ row_off,
                         const int32_t* __restrict__ fw, const int64_t* __restrict__ xo,
                         const T* __restrict__ X, const double* __restrict__ cycles,
                         const int32_t* __restrict__ fw_test, int stat_stride, double* __restrict__ Z,
                         double* __restrict__ mu, double* __restrict__ sigma, int* dstatus) {
    constexpr int ROWS = RS_MAXV * RUNS / kGroups;           // RUNS >= max_runs
    __shared__ StdSmem<kFeat, ROWS> S;
    __shared__ double cyc_s[RS_MAXV * RUNS];
    __shared__ long long lc_s[RS_MAXV * RUNS];
    __shared__ int64_t rowx[RS_MAXV * RUNS];
    const int q = blockIdx.x;
    int start[RS_MAXRUNS + 1], F = 0;
    const int N = rs_group_layout(q, group_off, max_runs, n_runs, row_off, fw, fw_test, stat_stride, start, F);
    if (N < 0) {
        if (threadIdx.x == 0 && blockIdx.y == 0) rs_dev_flag(dstatus, RS_EDATA, q);
        return;
    }
    if (blockIdx.y * kFeat >= F) return;
    const int fl = threadIdx.x % kFeat, g = threadIdx.x / kFeat;
    const int f = blockIdx.y * kFeat + fl;
    const bool active = f < F;
    const int64_t g0 = group_off[q];
    load_log_tables(S.tl, S.tc, kThreads);
    if (threadIdx.x < kFeat) S.inf[threadIdx.x] = 0;
    __syncthreads();
    for (int u = threadIdx.x; u < N; u += kThreads) {
        int r = 0;
        while (u >= start[r + 1]) ++r;
        const int v = u - start[r];
        rowx[u] = xo[g0 + r] + (int64_t)v * F;
        if (cycles) {
            cyc_s[u] = cycles[row_off[g0 + r] + v];
            lc_s[u] = cycle_log(cyc_s[u], S.tl, S.tc);
        }
    }
    __syncthreads();
    T x[ROWS];
#pragma unroll
    for (int e = 0; e < ROWS; ++e) x[e] = active && g + kGroups * e < N ? X[rowx[g + kGroups * e] + f] : (T)1;
    long long l[ROWS];
#pragma unroll
    for (int e = 0; e < ROWS; ++e) {
        const int u = g + kGroups * e;
        l[e] = u < N ? elem_log(x[e], cycles != nullptr, cyc_s[u], lc_s[u], S.tl, S.tc) : 0;
    }
    double d[ROWS];
    const double rs = centre(S, l, d, N, active, mu + (int64_t)q * stat_stride + f, sigma + (int64_t)q * stat_stride + f);
    if (!active) return;
#pragma unroll
    for (int e = 0; e < ROWS; ++e) {
        const int u = g + kGroups * e;
        if (u < N) Z[rowx[u] + f] = rs > 0.0 ? d[e] * rs : 0.0;
    }
}

// The test side: program q standardized with its training group's statistics (at
// q * stat_stride + f): z = (log max(x / c, 1e-30) - mu) / sigma, or 0 where sigma <= 1e-12.
template <typename T>
__global__ void __launch_bounds__(kThreads)
standardize_apply_kernel(const int64_t* __restrict__ row_off, const int32_t* __restrict__ fw,
                         const int64_t* __restrict__ xo, const T* __restrict__ X,
                         const double* __restrict__ cycles, const double* __restrict__ mu,
                         const double* __restrict__ sigma, int stat_stride, double* __restrict__ Z) {
    __shared__ double cyc_s[RS_MAXV];
    __shared__ long long lc_s[RS_MAXV], tl[256];
    __shared__ uint16_t tc[256];
    __shared__ double rs_s[kFeat];
    __shared__ long long mf_s[kFeat];
    const int p = blockIdx.x;
    const int64_t r0 = row_off[p];
    const int V = (int)(row_off[p + 1] - r0);
    const int F = fw[p];
    const int fl = threadIdx.x % kFeat, g = threadIdx.x / kFeat;
    const int f = blockIdx.y * kFeat + fl;
    // a bad program was reported by group_standardize_kernel
    if (blockIdx.y * kFeat >= F || V < 1 || V > RS_MAXV || F > stat_stride) return;
    load_log_tables(tl, tc, kThreads);
    if (threadIdx.x < kFeat && f < F) {      // the feature's statistics: 1 / sigma, mu in fixed point
        const double sd = sigma[(int64_t)p * stat_stride + f];
        const bool ok = sd > 1e-12;          // (not for the NaN of a feature with an infinite value)
        rs_s[threadIdx.x] = ok ? 1.0 / sd : 0.0;
        mf_s[threadIdx.x] = ok ? __double2ll_rn(mu[(int64_t)p * stat_stride + f] * 9007199254740992.0) : 0;
    }
    __syncthreads();
    if (cycles && threadIdx.x < V) {
        cyc_s[threadIdx.x] = cycles[r0 + threadIdx.x];
        lc_s[threadIdx.x] = cycle_log(cyc_s[threadIdx.x], tl, tc);
    }
    __syncthreads();
    if (f >= F) return;
    const double rs = rs_s[fl];
    const long long m = mf_s[fl];
    const int64_t base = xo[p];
#pragma unroll
    for (int q = 0; q < RS_MAXV / kGroups; ++q) {
        const int r = g + kGroups * q;
        if (r >= V) break;
        const long long l = elem_log(X[base + (int64_t)r * F + f], cycles != nullptr, cyc_s[r], lc_s[r], tl, tc);
        const double d = l == kFixInf ? __longlong_as_double(kInfBits) : fix_double(l - m);
        Z[base + (int64_t)r * F + f] = rs > 0.0 ? d * rs : 0.0;
    }
}

template <typename T>
void launch_group(int runs, dim3 grid, cudaStream_t st, const int64_t* group_off, const rs_batch* train,
                  const rs_batch* test, int max_runs, int stat_stride, double* ZA, double* mu, double* sigma,
                  int* dstatus) {
    auto go = [&](auto kern) {
        kern<<<grid, kThreads, 0, st>>>(group_off, max_runs, train->n_programs, train->row_offsets, train->feat_width,
                                        train->x_offsets, (const T*)train->X, train->cycles, test->feat_width,
                                        stat_stride, ZA, mu, sigma, dstatus);
    };
    if (runs <= 1) go(group_standardize_kernel<T, 1>);
    else if (runs <= 2) go(group_standardize_kernel<T, 2>);
    else go(group_standardize_kernel<T, RS_MAXRUNS>);
}

template <typename T, int FEAT>
void launch_standardize(const rs_batch* b, double* Z, double* mu, double* sigma, int* dstatus, cudaStream_t st) {
    dim3 grid((unsigned)b->n_programs, (unsigned)((b->max_feat + FEAT - 1) / FEAT));
    standardize_kernel<T, FEAT><<<grid, kThreads, 0, st>>>(b->n_programs, b->row_offsets, b->feat_width, b->x_offsets,
                                                           b->feat_offsets, (const T*)b->X, b->cycles, Z, mu, sigma,
                                                           dstatus);
}

}  // namespace

cudaError_t rs_launch_transfer_standardize(const rs_batch* train, const rs_batch* test, const int64_t* group_off,
                                           int max_runs, int stat_stride, double* ZA, double* ZB, double* mu,
                                           double* sigma, int* dstatus, cudaStream_t st) {
    const int Q = test->n_programs;
    dim3 ga((unsigned)Q, (unsigned)((stat_stride + kFeat - 1) / kFeat));
    if (train->dtype == RS_F32)
        launch_group<float>(max_runs, ga, st, group_off, train, test, max_runs, stat_stride, ZA, mu, sigma, dstatus);
    else
        launch_group<double>(max_runs, ga, st, group_off, train, test, max_runs, stat_stride, ZA, mu, sigma, dstatus);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    dim3 gb((unsigned)Q, (unsigned)((test->max_feat + kFeat - 1) / kFeat));
    if (test->dtype == RS_F32)
        standardize_apply_kernel<float><<<gb, kThreads, 0, st>>>(test->row_offsets, test->feat_width, test->x_offsets,
                                                                 (const float*)test->X, test->cycles, mu, sigma,
                                                                 stat_stride, ZB);
    else
        standardize_apply_kernel<double><<<gb, kThreads, 0, st>>>(test->row_offsets, test->feat_width,
                                                                  test->x_offsets, (const double*)test->X,
                                                                  test->cycles, mu, sigma, stat_stride, ZB);
    return cudaGetLastError();
}

cudaError_t rs_launch_standardize(const rs_batch* b, double* Z, double* mu, double* sigma,
                                  int* dstatus, cudaStream_t st) {
    // 32-feature blocks once they give every SM two blocks
    const bool wide = (int64_t)b->n_programs * ((b->max_feat + 31) / 32) >= 304;
    if (b->dtype == RS_F32) {
        if (wide) launch_standardize<float, 32>(b, Z, mu, sigma, dstatus, st);
        else launch_standardize<float, 16>(b, Z, mu, sigma, dstatus, st);
    } else {
        if (wide) launch_standardize<double, 32>(b, Z, mu, sigma, dstatus, st);
        else launch_standardize<double, 16>(b, Z, mu, sigma, dstatus, st);
    }
    return cudaGetLastError();
}
