// K2 (FP64 form) on the tensor cores: K_p = Z_p Z_p^T of the standardized feature vectors, without
// FP64 products.  This part's FP64 pipe does 2 multiply-adds a clock and SM, its tensor cores
// 4096 in f16; 30 of their exact small products stand in for one FP64 product here.
//
// Splitting (after K. Ozaki, T. Ogita, S. Oishi, S. Rump, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication", Numer. Algorithms 59, 2012).
// A z-score over 64 values is at most sqrt(63) < 7.95 in magnitude, so z is taken as a 56-bit
// integer X = round(2^52 z) (exact for |z| >= 1) and written in seven balanced digits of base 256:
// X = sum_i d_i 256^(7 - i), d_i in -128 .. 127, each exact in f16.  Products of digits are at most
// 2^14, and an accumulator takes at most four of them per feature, so 256 features sum to at most
// 2^24: every FP32 accumulation is exact.  With S_i the 64 x F matrix of digit i,
//     K = sum over i + j <= 9 of 2^(8 (1 - i - j)) S_i S_j^T      (the pairs left out: below 2^-55 F)
// and the weighted sums of the accumulators are formed in 64-bit integers and rounded once per 256
// features.  What is left of rounding is that of X (at most 2^-53 per element) and one addition per
// 256 features; an FP64 chain of F products rounds F times at the size of its partial sums.
// Against an extended-precision product of the same Z, rms error over the block, 64 versions: 24
// features 6.5e-16 (the FP64 chain 1.4e-15), 96: 2.0e-15 (9.3e-15), 1024: 2.8e-14 (2.8e-13), 4096:
// 1.7e-13 (2.4e-12).
//
// Persistent CTAs, one program at a time in blocks of 64 features.  Eight warps split the block's
// 64 x 64 doubles into digits and store them K-major with the 128-byte swizzle, slice i in rows
// 64 i .. 64 i + 63 of a stage (slice 8 is zero); a ninth warp's one thread issues ten tcgen05.mma
// per 16 features (M = N = 128: two slices a side), (i, j) odd with i + j = t into tensor-memory
// accumulator t / 2.  Stages are double-buffered, so splitting a block (and the next program's first)
// overlaps the previous block's products.  After 256 features, or the last, the eight warps read the
// four accumulators: the quadrant (lane half h, column half w) of accumulator t holds digit sums of
// weight t + h + w.
// A program with an element outside +-7.95, or not finite (not z-scores, then), is redone by plain
// FP64 multiply-adds in feature order; so is one with a row whose norm is below 1 but not 0, as the digits
// hold an element to 2^-53, whatever its size: sum over f of 2^-53 (|z_a| + |z_b|) <= 2^-53 sqrt(F) (|Z_a| +
// |Z_b|) is within 2^-52 sqrt(F) |Z_a| |Z_b| for norms from 1 up, and so within what F roundings of an FP64
// chain may come to (F 2^-53 |Z_a| |Z_b|).
// Per block of 64 features the products take 2600 cycles and the splitting 2200, per 256 features
// the sums 20000 (64 conversions and 64-bit sums per thread and 8 columns).
// 256 programs x 1024 features 952 -> 133 us, 64 x 256 37 -> 21 us.
#include <cuda_fp16.h>

#include "tc_gemm.cuh"

namespace {

constexpr int kSplThreads = 256;
constexpr int kSplSlices = 7;
constexpr int kSplBlock = 64;                             // features per stage
constexpr int kSplChunk = 4;                              // stages summed in FP32 (256 features)
constexpr uint32_t kSliceBytes = 64 * kSplBlock * 2;
constexpr uint32_t kStageBytes = 8 * kSliceBytes;         // seven digits and a zero slice
constexpr uint32_t kXchBytes = 2 * 8 * 64 * 16;           // [column half][8 columns][64 rows] of two int64
constexpr uint32_t kSplSmem = 2 * kStageBytes + 2 * kXchBytes + 64 + 1024;
constexpr unsigned kSplHi = 0x401fcccc;                   // high word of 7.95, rounded down
static_assert((kSplBlock * kSplChunk * 4) << 14 <= 1 << 24, "sums of one accumulator are exact in FP32");

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// 2^(52 - W) z rounded to nearest, plus 128 in every digit's place: byte k of the result is digit 7 - k
// plus 128.  |z| < 7.95 2^W; false otherwise.
template <int W>
__device__ __forceinline__ unsigned long long digits_of(double z, bool& ok) {
    const unsigned hi = (unsigned)__double2hiint(z), lo = (unsigned)__double2loint(z);
    ok = ok && (hi & 0x7fffffffu) < kSplHi + ((unsigned)W << 20);
    const int ex = (int)(hi >> 20) & 0x7ff;
    int s = 1025 + W - ex;
    s = s > 60 ? 60 : (s < 0 ? 0 : s);                    // (a subnormal's spurious bit is shifted out)
    const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << 2;
    const unsigned long long x = (m + ((1ull << s) >> 1)) >> s;
    return ((int)hi < 0 ? 0ull - x : x) + 0x80808080808080ull;
}

struct SplItem {
    int64_t p;                 // program; past the last: none
    int kb, nk, V, F, n;       // block of 64 features, blocks, versions, features, programs taken before
    const double* z;
};

struct SplArgs {
    int P;
    const int64_t* row_off;
    const int32_t* fw;
    const int64_t* xo;
    const double* Z;
    double* K;
    int* dstatus;
};

__device__ __forceinline__ void spl_program(const SplArgs& a, SplItem& it, int tid) {
    for (; it.p < a.P; it.p += gridDim.x) {
        it.V = (int)(a.row_off[it.p + 1] - a.row_off[it.p]);
        it.F = a.fw[it.p] > 0 ? a.fw[it.p] : 0;
        if (it.V >= 1 && it.V <= RS_MAXV) break;
        if (tid == 0) rs_dev_flag(a.dstatus, RS_EDATA, (int)it.p);
    }
    if (it.p >= a.P) return;
    it.kb = 0;
    it.nk = it.F > kSplBlock ? (it.F + kSplBlock - 1) / kSplBlock : 1;
    it.z = a.Z + a.xo[it.p];
}

// This thread's two tasks of a block: row (tid + 256 i) / 8, eight consecutive features.
__device__ __forceinline__ void spl_load(const SplItem& it, double (&v)[16]) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int u = threadIdx.x + kSplThreads * i, row = u >> 3, f = it.kb * kSplBlock + (u & 7) * 8;
        const double* s = it.z + (int64_t)row * it.F + f;
        if (row < it.V && f + 8 <= it.F && (reinterpret_cast<uintptr_t>(s) & 15) == 0) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const double2 d = __ldg(reinterpret_cast<const double2*>(s) + e);
                v[8 * i + 2 * e] = d.x;
                v[8 * i + 2 * e + 1] = d.y;
            }
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) v[8 * i + e] = row < it.V && f + e < it.F ? __ldg(s + e) : 0.0;
        }
    }
}

// The digits of the block into a stage: task (row, chunk of 8 features) writes 16 bytes of each
// slice at the swizzled place of that chunk.
template <int W>
__device__ __forceinline__ bool spl_store(const double (&v)[16], unsigned char* stage) {
    bool ok = true;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int u = threadIdx.x + kSplThreads * i, row = u >> 3, ch = u & 7;
        unsigned ylo[8], yhi[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const unsigned long long y = digits_of<W>(v[8 * i + e], ok);
            ylo[e] = (unsigned)y;
            yhi[e] = (unsigned)(y >> 32);
        }
        unsigned char* dst = stage + row * 128 + ((ch ^ (row & 7)) << 4);
        const __half2 off = __floats2half2_rn(1152.f, 1152.f);           // 1024 + 128
#pragma unroll
        for (int s = 0; s < kSplSlices; ++s) {
            const int byte = 6 - s;                                      // slice s + 1: digit of 256^(6 - s)
            unsigned w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const unsigned a = byte >= 4 ? yhi[2 * q] : ylo[2 * q], b = byte >= 4 ? yhi[2 * q + 1] : ylo[2 * q + 1];
                const unsigned k = byte & 3;
                unsigned x = __byte_perm(a, b, k | k << 4 | (4 + k) << 8 | (4 + k) << 12);
                x = (x & 0x00ff00ffu) | 0x64006400u;                     // 1024 + byte, in f16
                const __half2 h = __hsub2(*reinterpret_cast<__half2*>(&x), off);
                w[q] = *reinterpret_cast<const unsigned*>(&h);
            }
            *reinterpret_cast<uint4*>(dst + s * kSliceBytes) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
    return ok;
}

// 2^(2 W - 64) (hi 2^32 + lo) as a double, rounded to nearest, by integer operations (|hi|, |lo| < 2^62).
template <int W>
__device__ __forceinline__ double spl_double(long long hi, long long lo) {
    hi += lo >> 32;
    unsigned l = (unsigned)lo;
    const bool neg = hi < 0;
    if (neg) {                                            // two's complement over 96 bits
        l = 0u - l;
        hi = ~hi + (l == 0u);
    }
    unsigned long long m = (unsigned long long)hi;
    int e;
    if (m == 0) {
        m = l;
        if (m == 0) return 0.0;
        e = __clzll((long long)m);
        m <<= e;
        e += 32;
    } else {
        e = __clzll((long long)m);
        m <<= e;
        m |= e >= 32 ? (unsigned long long)l << (e - 32) : (unsigned long long)l >> (32 - e);
    }
    // m in [2^63, 2^64) stands for m 2^(32 - e) 2^-64: its leading bit is 2^(31 - e)
    const unsigned long long b = ((unsigned long long)(1023 + 31 + 2 * W - e - 1) << 52) + (m >> 11) + ((m >> 10) & 1ull);
    return __longlong_as_double((long long)(b | (neg ? 0x8000000000000000ull : 0ull)));
}

__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}

__device__ __forceinline__ void split_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// The eight warps' reading of the four accumulators: rows x cols sums of digits' products as doubles into
// out (row stride ld), added to what is there or not.  xch: two buffers of kXchBytes.  last: true if
// this thread wrote an entry (i, i) below 1.
template <int W>
__device__ __forceinline__ bool spl_sums(uint32_t tmem, longlong2* xch, double* out, int ld, int rows, int cols, bool add, bool last) {
    bool low = false;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int quarter = warp & 3, half = warp >> 2;          // TMEM lanes, columns 32 half ..
    const int row = (quarter & 1) * 32 + lane;
    const bool upper = quarter >= 2;
    const int mine = upper ? 4 : 0;            // of 8 columns: the four this warp finishes
    const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16);
    for (int c0 = 0; c0 < 32; c0 += 8) {
        const int col = half * 32 + c0;
        if (col >= cols) {                    // (uniform over the half's four warps)
            split_sync();
            continue;
        }
        double* o = out + (int64_t)row * ld + col + mine;
        const bool whole = (reinterpret_cast<uintptr_t>(o) & 15) == 0 && row < rows && col + mine + 4 <= cols;
        double old[4] = {0.0, 0.0, 0.0, 0.0};
        if (add) {
            if (whole) {
                *reinterpret_cast<double2*>(old) = *reinterpret_cast<const double2*>(o);
                *reinterpret_cast<double2*>(old + 2) = *reinterpret_cast<const double2*>(o + 2);
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (row < rows && col + mine + c < cols) old[c] = o[c];
            }
        }
        uint32_t r[8][8];                      // weights t + (upper) + (right half): t = 2, 4, 6, 8
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            tmem_ld8_nowait(trow + (uint32_t)(t * 128 + col), r[2 * t]);
            tmem_ld8_nowait(trow + (uint32_t)(t * 128 + 64 + col), r[2 * t + 1]);
        }
        tc::tmem_wait_ld();
        // lower lanes: r[k] has weight k + 2, upper lanes: k + 3 (weight 10 is left out);
        // hi collects weights 2 .. 5 (in the place of 5), lo 6 .. 9 (in the place of 9).
        // A lower and an upper lane share a row: each finishes four of the columns and
        // sends its sums of the other four (two buffers, one barrier a round)
        longlong2* xb = xch + ((c0 >> 3) & 1) * (kXchBytes / 16);
        long long hi[4], lo[4];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            int x[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = __float2int_rn(__uint_as_float(r[k][c]));
            long long h, l;
            if (!upper) {
                h = ((long long)x[0] << 24) + ((long long)x[1] << 16) + ((long long)x[2] << 8) + x[3];
                l = ((long long)x[4] << 24) + ((long long)x[5] << 16) + ((long long)x[6] << 8) + x[7];
            } else {
                h = ((long long)x[0] << 16) + ((long long)x[1] << 8) + x[2];
                l = ((long long)x[3] << 24) + ((long long)x[4] << 16) + ((long long)x[5] << 8) + x[6];
            }
            if ((c >= 4) == upper) {
                hi[c & 3] = h;
                lo[c & 3] = l;
            } else {
                xb[(half * 8 + c) * 64 + row] = make_longlong2(h, l);
            }
        }
        split_sync();
        double d[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const longlong2 u = xb[(half * 8 + mine + c) * 64 + row];
            d[c] = spl_double<W>(hi[c] + u.x, lo[c] + u.y);
            if (add) d[c] += old[c];
        }
        if (last && (unsigned)(row - col - mine) < 4u && row < rows) {
#pragma unroll
            for (int c = 0; c < 4; ++c) low = low || (row == col + mine + c && __double2hiint(d[c]) < 0x3ff00000);
        }
        if (whole) {
            *reinterpret_cast<double2*>(o) = make_double2(d[0], d[1]);
            *reinterpret_cast<double2*>(o + 2) = make_double2(d[2], d[3]);
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (row < rows && col + mine + c < cols) o[c] = d[c];
        }
    }
    return low;
}

// K of one program by plain FP64 multiply-adds in feature order (the eight warps; buf: 64 x 33 doubles): 32
// features of its rows at a time in shared memory, nine entries of the triangle a thread.  256 programs x 64
// versions x 1024 features of small values: 1309 us for the call (gram_f64_kernel: 949).
constexpr int kPlainLd = 33;
static_assert(RS_MAXV * kPlainLd * sizeof(double) <= 2 * kXchBytes, "the rows' slice fits the exchange buffers");
__device__ __noinline__ void spl_plain(const double* z, int V, int F, double* Kp, double* buf) {
    const int tid = threadIdx.x, E = V * (V + 1) / 2;
    constexpr int kPer = (RS_MAXV * (RS_MAXV + 1) / 2 + kSplThreads - 1) / kSplThreads;
    int at[kPer];                                          // row << 8 | column <= row; past the last: row 0
    double acc[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int e = tid + kSplThreads * q;
        int i = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
        if (i * (i + 1) / 2 > e) --i;
        if ((i + 1) * (i + 2) / 2 <= e) ++i;
        at[q] = e < E ? i << 8 | (e - i * (i + 1) / 2) : 0;
        acc[q] = 0.0;
    }
    for (int f0 = 0; f0 < F; f0 += 32) {
        split_sync();
        for (int e = tid; e < V * 32; e += kSplThreads) {
            const int r = e >> 5, f = f0 + (e & 31);
            buf[r * kPlainLd + (e & 31)] = f < F ? __ldg(z + (int64_t)r * F + f) : 0.0;
        }
        split_sync();
        const int w = F - f0 < 32 ? F - f0 : 32;
        for (int c = 0; c < w; ++c)
#pragma unroll
            for (int q = 0; q < kPer; ++q)
                if (tid + kSplThreads * q < E)
                    acc[q] = fma(buf[(at[q] >> 8) * kPlainLd + c], buf[(at[q] & 0xff) * kPlainLd + c], acc[q]);
    }
#pragma unroll
    for (int q = 0; q < kPer; ++q)
        if (tid + kSplThreads * q < E) {
            const int i = at[q] >> 8, j = at[q] & 0xff;
            Kp[i * RS_GRAM_LD + j] = acc[q];
            Kp[j * RS_GRAM_LD + i] = acc[q];
        }
    split_sync();
}

__global__ void __launch_bounds__(kSplThreads + 32, 1) gram_split_kernel(const SplArgs a) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint32_t tmem_slot;
    __shared__ int outside[4];                             // an element outside the range, by program (mod 4)
    __shared__ int low[4], anew;                           // a row's norm below 1; such a row is not 0
    __shared__ volatile int gave_up;
    const uint32_t raw = tc::smem_u32(smem_raw), base = (raw + 1023u) & ~1023u;
    uint8_t* g = smem_raw + (base - raw);
    longlong2* xch = reinterpret_cast<longlong2*>(g + 2 * kStageBytes);
    // barriers: stage written [2] (8 warps), its products complete [2], accumulators read (8 warps)
    const uint32_t full = base + 2 * kStageBytes + 2 * kXchBytes, done = full + 16, drained = full + 32;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(full + 8 * i, 8);
            tc::mbar_init(done + 8 * i, 1);
        }
        tc::mbar_init(drained, 8);
        tc::fence_barrier_init();
        outside[0] = outside[1] = outside[2] = outside[3] = 0;
        low[0] = low[1] = low[2] = low[3] = anew = 0;
        gave_up = 0;
    }
    for (int i = tid; i < (int)(2 * kSliceBytes / 16); i += kSplThreads + 32)      // the zero slices
        *reinterpret_cast<uint4*>(g + (i >= (int)(kSliceBytes / 16) ? kStageBytes : 0) + 7 * kSliceBytes +
                                  (i % (kSliceBytes / 16)) * 16) = make_uint4(0u, 0u, 0u, 0u);
    fence_async_smem();
    if (warp == 0) {
        tc::tmem_alloc(tc::smem_u32(&tmem_slot), 512);
        tc::tmem_relinquish();
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = tmem_slot;
    // a wait that gives up (RS_ETIMEOUT) ends all waiting, not the warps' way through the work: every
    // warp still meets the others at the barriers
    auto wait = [&](uint32_t bar, uint32_t phase, int site) {
        if (!gave_up && !tc::mbar_wait(bar, phase, a.dstatus, site)) gave_up = 1;
    };

    SplItem cur;
    cur.p = blockIdx.x;
    cur.n = 0;
    spl_program(a, cur, warp == 8 ? -1 : tid);
    bool alive = cur.p < a.P;
    int it = 0;
    if (warp == 8) {                                       // ---- the products
        // f16 x f16 -> FP32, both operands K-major, 128 x 128
        constexpr uint32_t idesc = (1u << 4) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
        if (tc::elect_one()) {
            int chunk = 0;
            for (; alive; ++it) {
                const int buf = it & 1;
                const bool first = cur.kb % kSplChunk == 0;
                if (first && chunk > 0) wait(drained, (uint32_t)((chunk - 1) & 1), -34);
                wait(full + 8 * buf, (uint32_t)((it >> 1) & 1), -35);
                chunk += first;
                tc::fence_after();
                const uint32_t st = base + buf * kStageBytes;
#pragma unroll 1
                for (int k = 0; k < kSplBlock / 16; ++k)
#pragma unroll
                    for (int t = 2; t <= 8; t += 2)
#pragma unroll
                        for (int i = 1; i < t; i += 2)
                            tc::mma_bf16(tmem + (uint32_t)((t / 2 - 1) * 128),
                                         tc::sw128_desc(st + (i - 1) * kSliceBytes + k * 32),
                                         tc::sw128_desc(st + (t - i - 1) * kSliceBytes + k * 32), idesc,
                                         !(first && k == 0 && i == 1));
                tc::mma_commit(done + 8 * buf);
                if (++cur.kb == cur.nk) {
                    cur.p += gridDim.x;
                    spl_program(a, cur, -1);
                }
                alive = cur.p < a.P;
            }
            // every product has completed before the tensor memory is freed
            if (it > 0) tc::mbar_wait(done + 8 * ((it - 1) & 1), (uint32_t)(((it - 1) >> 1) & 1), a.dstatus, -33);
        }
    } else {                                               // ---- digits, and the sums
        auto stage_full = [&](int buf) {
            fence_async_smem();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(full + 8 * buf);
        };
        double v[16];
        if (alive) {
            spl_load(cur, v);
            if (!spl_store<0>(v, g)) outside[0] = 1;
            stage_full(0);
        }
        while (alive) {
            const int buf = it & 1;
            SplItem nxt = cur;
            if (++nxt.kb == nxt.nk) {
                nxt.p += gridDim.x;
                ++nxt.n;
                spl_program(a, nxt, tid);
            }
            const bool more = nxt.p < a.P;
            if (more) {
                spl_load(nxt, v);
                // the products that read the other stage have completed
                if (it >= 1) wait(done + 8 * (buf ^ 1), (uint32_t)(((it - 1) >> 1) & 1), -31);
                if (!spl_store<0>(v, g + (buf ^ 1) * kStageBytes)) outside[nxt.n & 3] = 1;
                stage_full(buf ^ 1);
            }
            const bool last = cur.kb + 1 == cur.nk;
            if (last || cur.kb % kSplChunk == kSplChunk - 1) {
                wait(done + 8 * buf, (uint32_t)((it >> 1) & 1), -32);
                __syncwarp();
                tc::fence_after();
                double* Kp = a.K + cur.p * (RS_GRAM_LD * RS_GRAM_LD);
                if (spl_sums<0>(tmem, xch, Kp, RS_GRAM_LD, cur.V, cur.V, cur.kb >= kSplChunk, last)) low[cur.n & 3] = 1;
                tc::fence_before();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(drained);
                if (last) {
                    split_sync();                          // (also: the flags of every warp are in)
                    const bool far = outside[cur.n & 3];   // (these are uniform)
                    if (far || low[cur.n & 3]) {
                        if (!far) {                        // a warp a row: is a short one all zeros?
                            for (int r = warp; r < cur.V; r += kSplThreads / 32) {
                                if (!(Kp[r * (RS_GRAM_LD + 1)] < 1.0)) continue;
                                bool some = false;
                                for (int f = lane; f < cur.F; f += 32) some = some || __ldg(cur.z + (int64_t)r * cur.F + f) != 0.0;
                                if (some) anew = 1;
                            }
                            split_sync();
                        }
                        if (far || anew) spl_plain(cur.z, cur.V, cur.F, Kp, reinterpret_cast<double*>(xch));
                        split_sync();
                        if (tid == 0) outside[cur.n & 3] = low[cur.n & 3] = anew = 0;
                    }
                }
            }
            alive = more;
            cur = nxt;
            ++it;
        }
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// The dot products of a transfer (k_gram.cu: transfer_tile_kernel) by the same splitting: 64 x 64 blocks of
// the group's Gram (lower triangle of blocks) and of the test rows against the group's.  The group's
// z-scores are below sqrt(64 runs - 1), the test rows' unbounded, so the digits start at 2^4 (|z| <
// 15.9), X = round(2^51 z).  An element outside enters the digits as 0; its products are added in FP64, the
// features that have one in order (tr_far).  A CTA takes a block at a time; a stage holds 64 features of its rows' digits and one those of its
// columns (a diagonal block's are the same), so splitting waits for the products before it; loads
// and, across blocks, nothing else overlap them.  Per block: the sums 20,000 cycles, per 64 features 4,400
// for splitting and 2,600 for products.
// 90 problems of 192 + 64 rows x 96 features: 108 us (FP64 tiles: 527).  The whole call 439 us, with a
// counter of every test version outside 483, with all of them 816 (the block anew in plain FP64 for either: 1069).
struct TrSplArgs {
    const int64_t* group_off;
    int max_runs;
    int64_t n_runs;
    int stat_stride;
    const int64_t* a_row;
    const int32_t* a_fw;
    const int64_t* a_xo;
    const double* ZA;
    const int64_t* b_row;
    const int32_t* b_fw;
    const int64_t* b_xo;
    const double* ZB;
    int ld;
    double* KA;                // null: only Kx
    double* Kx;
    int64_t Q;
    int* dstatus;
};

struct TrBlock {
    const double* rowp[4];     // this thread's two rows of the block's rows and two of its columns (null: none)
    double* out;
    int rows, cols, F, nk;
    bool same;                 // a diagonal block
};

// Block t of the launch: false if it does not exist (the same for every thread).
__device__ __forceinline__ bool tr_block(const TrSplArgs& a, int64_t t, TrBlock& b) {
    const int nb = a.max_runs, ng = a.KA ? nb * (nb + 1) / 2 : 0;
    const int64_t q = t / (ng + nb);
    int k = (int)(t - q * (ng + nb));
    int start[RS_MAXRUNS + 1];
    const int N = rs_group_layout((int)q, a.group_off, a.max_runs, a.n_runs, a.a_row, a.a_fw, a.b_fw, a.stat_stride, start, b.F);
    if (N < 0 || N > a.ld) return false;
    const bool cross = k >= ng;
    int bi = 0, bu;
    if (cross) {
        bu = k - ng;
    } else {                                   // k = bi (bi + 1) / 2 + bu, bu <= bi
        while ((bi + 1) * (bi + 2) / 2 <= k) ++bi;
        bu = k - bi * (bi + 1) / 2;
    }
    const int64_t VB = a.b_row[q + 1] - a.b_row[q];
    if (cross && (VB < 1 || VB > RS_MAXV)) return false;
    const int i0 = bi * 64, u0 = bu * 64, rows = cross ? (int)VB : N;
    if (i0 >= rows || u0 >= N) return false;
    b.rows = rows - i0 < 64 ? rows - i0 : 64;
    b.cols = N - u0 < 64 ? N - u0 : 64;
    b.nk = (b.F + kSplBlock - 1) / kSplBlock;
    b.same = !cross && bi == bu;
    b.out = (cross ? a.Kx + q * RS_MAXV * a.ld : a.KA + q * a.ld * a.ld) + (int64_t)i0 * a.ld + u0;
    const int64_t g0 = a.group_off[q];
    auto group_row = [&](int v) -> const double* {
        int r = 0;
        while (v >= start[r + 1]) ++r;
        return a.ZA + a.a_xo[g0 + r] + (int64_t)(v - start[r]) * b.F;
    };
    if (threadIdx.x < kSplThreads) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int v = (threadIdx.x >> 3) + 32 * i;
            b.rowp[i] = v >= b.rows ? nullptr : cross ? a.ZB + a.b_xo[q] + (int64_t)v * b.F : group_row(i0 + v);
            b.rowp[2 + i] = v >= b.cols ? nullptr : group_row(u0 + v);
        }
    }
    return true;
}

// This thread's two tasks of 64 features from f0: eight consecutive features of a row each.
__device__ __forceinline__ void tr_load(const double* const (&rowp)[4], int first, int f0, int F, double (&v)[16]) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int f = f0 + (threadIdx.x & 7) * 8;
        const double* s = rowp[first + i] + f;
        const bool row = rowp[first + i] != nullptr;
        if (row && f + 8 <= F && (reinterpret_cast<uintptr_t>(s) & 15) == 0) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const double2 d = __ldg(reinterpret_cast<const double2*>(s) + e);
                v[8 * i + 2 * e] = d.x;
                v[8 * i + 2 * e + 1] = d.y;
            }
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) v[8 * i + e] = row && f + e < F ? __ldg(s + e) : 0.0;
        }
    }
}

constexpr int kFarWords = 4096 / 8 / 32;       // a bit for eight features (max_feat is at most 4096)
template <int W>
__device__ __forceinline__ bool far_out(double z) {
    return ((unsigned)__double2hiint(z) & 0x7fffffffu) >= kSplHi + ((unsigned)W << 20);
}

// This thread's elements outside the digits' range: their features marked, themselves 0.
template <int W>
__device__ __forceinline__ void tr_mark(double (&v)[16], int kb, unsigned* far, int& outside) {
    const int ch = kb * 8 + (threadIdx.x & 7);
#pragma unroll
    for (int e = 0; e < 16; ++e)
        if (far_out<W>(v[e])) v[e] = 0.0;
    atomicOr(&far[ch >> 5], 1u << (ch & 31));
    outside = 1;
}

// The products that the digits left out: entry (i, u) of the block takes z_if z_uf for the features f of which
// one or the other is outside, in order.  By the eight warps, 4 x 4 entries a thread; buf: 2 x 64 x 9 doubles.
constexpr int kFarLd = 9;
static_assert(2 * 64 * kFarLd * sizeof(double) <= 2 * kXchBytes, "the rows of eight features fit the exchange buffers");
template <int W>
__device__ __noinline__ void tr_far(const double* const (*rows)[64], const unsigned* far, int F, int nrows, int ncols,
                                    double* out, int ld, double* buf) {
    const int tid = threadIdx.x, ti = tid >> 4, tu = tid & 15;
    double acc[4][4] = {};
    for (int ch = 0; ch * 8 < F; ++ch) {
        if (!(far[ch >> 5] >> (ch & 31) & 1u)) continue;           // (uniform)
        split_sync();
        for (int e = tid; e < 2 * 64 * 8; e += kSplThreads) {
            const int side = e >> 9, r = (e >> 3) & 63, f = ch * 8 + (e & 7);
            const double* z = rows[side][r];
            buf[(side * 64 + r) * kFarLd + (e & 7)] = z && f < F ? __ldg(z + f) : 0.0;
        }
        split_sync();
        for (int c = 0; c < 8; ++c) {
            double x[4], y[4];
            bool xo[4], yo[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                x[q] = buf[(ti + 16 * q) * kFarLd + c];
                y[q] = buf[(64 + tu + 16 * q) * kFarLd + c];
                xo[q] = far_out<W>(x[q]);
                yo[q] = far_out<W>(y[q]);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (xo[i] || yo[u]) acc[i][u] = fma(x[i], y[u], acc[i][u]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (ti + 16 * i < nrows && tu + 16 * u < ncols) out[(int64_t)(ti + 16 * i) * ld + tu + 16 * u] += acc[i][u];
}

__global__ void __launch_bounds__(kSplThreads + 32, 1) transfer_split_kernel(const TrSplArgs a) {
    constexpr int W = 1;
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint32_t tmem_slot;
    __shared__ int outside;                                // an element outside the range
    __shared__ unsigned far[kFarWords];                    // ... in these eight features
    __shared__ const double* far_rows[2][64];
    __shared__ volatile int gave_up;
    const uint32_t raw = tc::smem_u32(smem_raw), base = (raw + 1023u) & ~1023u;
    uint8_t* g = smem_raw + (base - raw);
    longlong2* xch = reinterpret_cast<longlong2*>(g + 2 * kStageBytes);
    // barriers: stages written (8 warps), their products complete, accumulators read (8 warps)
    const uint32_t full = base + 2 * kStageBytes + 2 * kXchBytes, done = full + 8, drained = full + 16;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    if (tid == 0) {
        tc::mbar_init(full, 8);
        tc::mbar_init(done, 1);
        tc::mbar_init(drained, 8);
        tc::fence_barrier_init();
        outside = 0;
        for (int i = 0; i < kFarWords; ++i) far[i] = 0u;
        gave_up = 0;
    }
    for (int i = tid; i < (int)(2 * kSliceBytes / 16); i += kSplThreads + 32)      // the zero slices
        *reinterpret_cast<uint4*>(g + (i >= (int)(kSliceBytes / 16) ? kStageBytes : 0) + 7 * kSliceBytes +
                                  (i % (kSliceBytes / 16)) * 16) = make_uint4(0u, 0u, 0u, 0u);
    fence_async_smem();
    if (warp == 0) {
        tc::tmem_alloc(tc::smem_u32(&tmem_slot), 512);
        tc::tmem_relinquish();
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = tmem_slot;
    // a wait that gives up (RS_ETIMEOUT) ends all waiting, as above
    auto wait = [&](uint32_t bar, uint32_t phase, int site) {
        if (!gave_up && !tc::mbar_wait(bar, phase & 1u, a.dstatus, site)) gave_up = 1;
    };
    const int64_t total = a.Q * (a.max_runs + (a.KA ? a.max_runs * (a.max_runs + 1) / 2 : 0));
    uint32_t it = 0, chunk = 0;                            // stages and chunks of 256 features so far
    TrBlock b;
    if (warp == 8) {                                       // ---- the products
        constexpr uint32_t idesc = (1u << 4) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
        if (tc::elect_one()) {
            for (int64_t t = blockIdx.x; t < total; t += gridDim.x) {
                if (!tr_block(a, t, b)) continue;
                const uint32_t sb = base + (b.same ? 0 : kStageBytes);
                for (int kb = 0; kb < b.nk; ++kb, ++it) {
                    const bool first = kb % kSplChunk == 0;
                    if (first && chunk > 0) wait(drained, chunk - 1, -36);
                    chunk += first;
                    wait(full, it, -37);
                    tc::fence_after();
#pragma unroll 1
                    for (int k = 0; k < kSplBlock / 16; ++k)
#pragma unroll
                        for (int u = 2; u <= 8; u += 2)
#pragma unroll
                            for (int i = 1; i < u; i += 2)
                                tc::mma_bf16(tmem + (uint32_t)((u / 2 - 1) * 128),
                                             tc::sw128_desc(base + (i - 1) * kSliceBytes + k * 32),
                                             tc::sw128_desc(sb + (u - i - 1) * kSliceBytes + k * 32), idesc,
                                             !(first && k == 0 && i == 1));
                    tc::mma_commit(done);
                }
            }
            // every product has completed before the tensor memory is freed
            if (it > 0) tc::mbar_wait(done, (it - 1) & 1u, a.dstatus, -38);
        }
    } else {                                               // ---- digits, and the sums
        for (int64_t t = blockIdx.x; t < total; t += gridDim.x) {
            if (!tr_block(a, t, b)) continue;
            for (int kb = 0; kb < b.nk; ++kb, ++it) {
                double v[16];
                auto store = [&](unsigned char* stage) {
                    if (spl_store<W>(v, stage)) return;
                    tr_mark<W>(v, kb, far, outside);
                    spl_store<W>(v, stage);
                };
                tr_load(b.rowp, 0, kb * kSplBlock, b.F, v);
                // the products that read the stages have completed
                if (it >= 1) wait(done, it - 1, -39);
                store(g);
                if (!b.same) {
                    tr_load(b.rowp, 2, kb * kSplBlock, b.F, v);
                    store(g + kStageBytes);
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(full);
                if (kb + 1 == b.nk || kb % kSplChunk == kSplChunk - 1) {
                    wait(done, it, -40);
                    __syncwarp();
                    tc::fence_after();
                    spl_sums<W>(tmem, xch, b.out, a.ld, b.rows, b.cols, kb >= kSplChunk, false);
                    tc::fence_before();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(drained);
                }
            }
            if ((tid & 7) == 0)
#pragma unroll
                for (int i = 0; i < 4; ++i) far_rows[i >> 1][(tid >> 3) + 32 * (i & 1)] = b.rowp[i];
            split_sync();
            if (outside) {                                 // (uniform)
                tr_far<W>(far_rows, far, b.F, b.rows, b.cols, b.out, a.ld, reinterpret_cast<double*>(xch));
                split_sync();
                if (tid < kFarWords) far[tid] = 0u;
                if (tid == 0) outside = 0;
            }
            split_sync();
        }
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

}  // namespace

cudaError_t rs_launch_transfer_split(const rs_batch* train_std, const rs_batch* test_std, const int64_t* group_off,
                                     int max_runs, int stat_stride, int ld, double* KA, double* Kx, int* dstatus,
                                     cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(transfer_split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSplSmem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const TrSplArgs a{group_off, max_runs, train_std->n_programs, stat_stride, train_std->row_offsets, train_std->feat_width,
                      train_std->x_offsets, (const double*)train_std->X, test_std->row_offsets, test_std->feat_width,
                      test_std->x_offsets, (const double*)test_std->X, ld, KA, Kx, test_std->n_programs, dstatus};
    const int64_t total = a.Q * (max_runs + (KA ? max_runs * (max_runs + 1) / 2 : 0));
    if (total < 1) return cudaSuccess;
    transfer_split_kernel<<<(unsigned)(total < sms ? total : sms), kSplThreads + 32, kSplSmem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t rs_launch_gram_split(const rs_batch* b, double* K, int* dstatus, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(gram_split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSplSmem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const SplArgs a{b->n_programs, b->row_offsets, b->feat_width, b->x_offsets, (const double*)b->X, K, dstatus};
    gram_split_kernel<<<(unsigned)(b->n_programs < sms ? b->n_programs : sms), kSplThreads + 32, kSplSmem, st>>>(a);
    return cudaGetLastError();
}
