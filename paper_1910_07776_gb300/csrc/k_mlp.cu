// K5-K8: the learned surrogate.  An MLP 256 -> 512 -> 512 -> 6 (GELU) maps a standardized
// feature vector straight to the six predicted log speedups (a learned stand-in for the
// tier-2 predictor of Sec. 2).  BF16 weights and activations on the tcgen05 tensor cores,
// FP32 accumulation; FP32 master weights with AdamW.
//
// One training step (a fixed sequence, captured once in a CUDA graph and replayed):
//   stage    rows of X (double) -> BF16 X_s [B][256]; labels -> Y_s  (within the step before's update)
//   fwd 1,2  U = X W^T + b (FP32, kept for the backward pass), H = gelu(U) (BF16)
//   fwd 3    out = H2 W3^T + b3; residual; loss; dO = 2 (out - y) / (6B) (BF16)
//   dgrad    dU2 = (dO W3) * gelu'(U2);  dU1 = (dU2 W2) * gelu'(U1)   (BF16)
//   wgrad    dW3 = dO^T H2, dW2 = dU2^T H1, dW1 = dU1^T X_s  (FP32 partials over row ranges, one launch)
//   update   gradients (partials added and bias columns summed in a fixed order), AdamW, BF16 weights
// The tensor cores take an operand with either its K or its rows contiguous, so the weight gradients
// read the activations, and the data gradients the weights, as they lie: nothing is transposed.
// A step of 8,192 rows: 175 -> 61 us (before: 16 launches, with transposed copies of every operand
// written 2 bytes at a time, the sums over rows in three kernels of 11 us each, one atomic addition to
// the loss a row).
#include <math.h>
#include <string.h>

#include <vector>

#include "tc_gemm.cuh"

namespace {

constexpr int kIn = 256, kHid = 512, kOut = 6, kOutP = 16;   // output rows padded to 16

// ---- blob layout (float offsets) --------------------------------------------------------------
struct Blob {
    static constexpr int64_t nW1 = (int64_t)kHid * kIn, nb1 = kHid, nW2 = (int64_t)kHid * kHid, nb2 = kHid;
    static constexpr int64_t nW3 = (int64_t)kOutP * kHid, nb3 = kOutP;
    static constexpr int64_t nP = nW1 + nb1 + nW2 + nb2 + nW3 + nb3;      // one parameter set
    static constexpr int64_t oW1 = 0, ob1 = oW1 + nW1, oW2 = ob1 + nb1, ob2 = oW2 + nW2, oW3 = ob2 + nb2,
                             ob3 = oW3 + nW3;
    // master | m | v | grad  (FP32), then BF16 copies, then feature stats, then counters
    static constexpr int64_t oM = nP, oV = 2 * nP, oG = 3 * nP;
    static constexpr int64_t oBf = 4 * nP;                                 // in floats
    // BF16 region (in bf16 elements from oBf*2 bytes): W1, W2, W3p; the rest is kept so that saved blobs
    // stay readable (it held transposes of W2 and W3)
    static constexpr int64_t bW1 = 0, bW2 = bW1 + nW1, bW3 = bW2 + nW2, bW2t = bW3 + nW3,
                             bW3t = bW2t + nW2, bEnd = bW3t + (int64_t)kHid * kOutP;
    static constexpr int64_t oStats = oBf + (bEnd + 1) / 2 + 64;           // mean[256], std[256]
    static constexpr int64_t oCount = oStats + 2 * kIn;                    // int step, int t
    static constexpr int64_t nFloats = oCount + 64;
};

// GELU in its tanh form (Hendrycks and Gimpel 2016): gelu(u) = u (1 + tanh(c (u + a u^3))) / 2,
// c = sqrt(2 / pi), a = 0.044715, with the hardware tanh (tanh.approx.f32, relative error
// about 2^-11, below the BF16 rounding of the activations): eight FP32 instructions and one
// special-function instruction, so the epilogue stays near the tensor cores' pace.
constexpr float kGeluC = 0.7978845608028654f;
constexpr float kGeluA = 0.044715f;
__device__ __forceinline__ float tanh_hw(float x) {
    float y;
    asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// d/du: (1 + t) / 2 + u (1 - t^2) c (1 + 3 a u^2) / 2
__device__ __forceinline__ float gelu_grad_f(float u) {
    const float u2 = u * u;
    const float t = tanh_hw(kGeluC * fmaf(kGeluA * u2, u, u));
    return 0.5f * (1.0f + t) + 0.5f * u * (1.0f - t * t) * kGeluC * fmaf(3.0f * kGeluA, u2, 1.0f);
}

// ---- epilogues ---------------------------------------------------------------------------------
// Two FP32 operations in one instruction, each rounded as by itself.
__device__ __forceinline__ unsigned long long pk2(float a, float b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void un2(unsigned long long v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// gelu of two values as a BF16 pair.
__device__ __forceinline__ unsigned gelu2(unsigned long long u) {
    const unsigned long long x = mul2(pk2(kGeluC, kGeluC), fma2(mul2(mul2(pk2(kGeluA, kGeluA), u), u), u, u));
    float x0, x1, y0, y1;
    un2(x, x0, x1);
    const unsigned long long y = mul2(mul2(pk2(0.5f, 0.5f), u), add2(pk2(1.0f, 1.0f), pk2(tanh_hw(x0), tanh_hw(x1))));
    un2(y, y0, y1);
    const __nv_bfloat162 h = __floats2bfloat162_rn(y0, y1);
    return *reinterpret_cast<const unsigned*>(&h);
}
// 32 bytes in one store: a whole sector of L2 (16-byte halves of it cost a tag each).
__device__ __forceinline__ void st32(void* p, const unsigned (&h)[8]) {
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 ::"l"(p), "r"(h[0]), "r"(h[1]), "r"(h[2]), "r"(h[3]), "r"(h[4]), "r"(h[5]), "r"(h[6]), "r"(h[7])
                 : "memory");
}
struct EpiHidden {           // U = acc + b (FP32, [unit][B]: a warp's rows side by side); H = gelu(U) (BF16)
    const float* bias;
    float* U;
    __nv_bfloat16* H;
    int64_t ldu;             // rows of the batch
    __device__ void operator()(int row, int col0, const float (&v)[16]) const {
        unsigned h[8];
        const float4* b4 = reinterpret_cast<const float4*>(bias + col0);
        const float4 bias4[4] = {b4[0], b4[1], b4[2], b4[3]};      // (before the stores; the step before may
        float* d = U + (int64_t)col0 * ldu + row;                   // still be writing: no read-only loads)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 b = bias4[q];
            const unsigned long long u0 = add2(pk2(v[4 * q], v[4 * q + 1]), pk2(b.x, b.y));
            const unsigned long long u1 = add2(pk2(v[4 * q + 2], v[4 * q + 3]), pk2(b.z, b.w));
            float x, y;
            un2(u0, x, y);
            d[(int64_t)(4 * q) * ldu] = x;
            d[(int64_t)(4 * q + 1) * ldu] = y;
            un2(u1, x, y);
            d[(int64_t)(4 * q + 2) * ldu] = x;
            d[(int64_t)(4 * q + 3) * ldu] = y;
            h[2 * q] = gelu2(u0);
            h[2 * q + 1] = gelu2(u1);
        }
        st32(H + (int64_t)row * kHid + col0, h);
    }
};

struct EpiInfer {            // inference: out = acc + b3 and its ranking
    const float* bias;
    float* pred;             // nullable: [B][6]
    const uint8_t* masks;    // the settings of the rows already enabled (null: none)
    int flags;
    int k;
    float log_tau;
    uint32_t* rec_code;      // [B], nullable: no ranking
    double* rec_pred;        // [B][k]
    __device__ void rank_row(int64_t row, const float (&o)[16]) const {
        const int cand = (flags & RS_RANK_ALL) || !masks ? 63 : (~masks[row] & 63);
        int above = 0, bm[kOut];
#pragma unroll
        for (int j = 0; j < kOut; ++j) {
            bm[j] = 0;
            above |= (((cand >> j) & 1) && o[j] >= log_tau) << j;
        }
#pragma unroll
        for (int i = 0; i < kOut; ++i)
#pragma unroll
            for (int j = i + 1; j < kOut; ++j) {
                if (o[i] >= o[j]) bm[j] |= 1 << i;
                else bm[i] |= 1 << j;
            }
        uint32_t code = 0x0FFFFFF0u;
        int c = 0;
        double rp[kOut];
#pragma unroll
        for (int x = 0; x < kOut; ++x) rp[x] = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll
        for (int j = 0; j < kOut; ++j) {
            const int pos = __popc(bm[j] & above);
            if (((above >> j) & 1) && pos < k) {
                code = (code & ~(0xFu << (4 + 4 * pos))) | ((uint32_t)j << (4 + 4 * pos));
#pragma unroll
                for (int x = 0; x < kOut; ++x)
                    if (x == pos) rp[x] = o[j];
                ++c;
            }
        }
        rec_code[row] = (code & ~0xFu) | (uint32_t)c;
        if (rec_pred)
#pragma unroll
            for (int x = 0; x < kOut; ++x)
                if (x < k) rec_pred[(int64_t)row * k + x] = rp[x];
    }
    __device__ void operator()(int64_t row, const float (&v)[16]) const {
        float o[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) o[i] = v[i] + bias[i];
        if (rec_code) rank_row(row, o);
        if (pred)
#pragma unroll
            for (int i = 0; i < kOut; ++i) pred[row * kOut + i] = o[i];
    }
};

struct EpiLoss {             // training: out = acc + b3; dO = scale (out - y) and the loss
    static constexpr bool kWarp = true;
    const float* bias;
    const float* Y;          // [B][16]
    __nv_bfloat16* dO;       // [B][16]
    float* part;             // [B / 32]: the minibatch MSE's sums over 32 rows
    float scale;
    __device__ void operator()(int row, bool in, int col0, const float (&v)[16]) const {
        if (col0 != 0) return;
        float l = 0.f;
        unsigned h[8] = {};
        if (in) {
            float g[kOut];
#pragma unroll
            for (int i = 0; i < kOut; ++i) {
                const float r = v[i] + bias[i] - Y[(int64_t)row * kOutP + i];
                l += 0.5f * scale * r * r;          // r^2 / (6 B)
                g[i] = scale * r;
            }
#pragma unroll
            for (int i = 0; i < kOut / 2; ++i) {
                const __nv_bfloat162 p = __floats2bfloat162_rn(g[2 * i], g[2 * i + 1]);
                h[i] = *reinterpret_cast<const unsigned*>(&p);
            }
            st32(dO + (int64_t)row * kOutP, h);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if ((threadIdx.x & 31) == 0) part[row >> 5] = l;
    }
};

struct EpiGeluGrad {         // dU = acc * gelu'(U) (BF16)
    const float* U;          // [unit][B]
    __nv_bfloat16* dU;
    int64_t ldu;
    struct Fetched { float u[16]; };
    __device__ Fetched fetch(int row, bool in, int col0) const {
        const float* u = U + (int64_t)col0 * ldu + row;
        Fetched f;
#pragma unroll
        for (int i = 0; i < 16; ++i) f.u[i] = in ? u[(int64_t)i * ldu] : 0.f;
        return f;
    }
    __device__ void operator()(int row, int col0, const float (&v)[16], const Fetched& f) const {
        unsigned h[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const __nv_bfloat162 p = __floats2bfloat162_rn(v[2 * i] * gelu_grad_f(f.u[2 * i]),
                                                           v[2 * i + 1] * gelu_grad_f(f.u[2 * i + 1]));
            h[i] = *reinterpret_cast<const unsigned*>(&p);
        }
        st32(dU + (int64_t)row * kHid + col0, h);
    }
};

// Pipeline depth of the persistent GEMM (one CTA per SM): four 32 KB stages (BN = 128).
constexpr int kStages = 4;

// The three weight gradients as one problem: each D = A^T B over a range of the batch's rows, A and B
// row-major, D's partial sums (one per range) in FP32.  28 tiles of 128 x 128 a range.  Four further
// warps a CTA start the bias gradients: a column of dU in 32 chains, chain l the rows l, l + 32, ... in
// order, two columns a lane (in the update kernel the chains took 20 us, the weights beside them 10).
constexpr int kWgradExtra = 4;
struct Wgrad {
    float* d[3];             // of W1, W2, W3; range z at + z * zstride
    int64_t zstride;
    int slices, rows;        // ranges, rows of each
    const __nv_bfloat16* du[3];      // dU1, dU2 [B][512], dO [B][16]
    float* chain[3];         // [min(B, 32)][512], the same, [min(B, 32)][16]
    int B;
    int* counters;           // minibatch, Adam's step, and at 8 the call's: counted here
    int64_t steps_per_epoch;
};
struct WgradProb {
    static constexpr bool kAmn = true, kBmn = true;
    struct Tile { int w, m0, n0, z, N, nk; };
    const CUtensorMap *dU1, *X, *dU2, *H1, *dO, *H2;
    const Wgrad& g;
    __device__ long long tiles() const { return 28ll * g.slices; }
    __device__ Tile tile(long long t) const {
        const int z = (int)(t / 28), j = (int)(t % 28), nk = (g.rows + 63) / 64;
        if (j < 16) return Tile{1, (j >> 2) * 128, (j & 3) * 128, z, kHid, nk};
        if (j < 24) return Tile{0, ((j - 16) >> 1) * 128, (j & 1) * 128, z, kIn, nk};
        return Tile{2, 0, (j - 24) * 128, z, kHid, nk};
    }
    __device__ void load(const Tile& t, int kb, uint32_t sa, uint32_t sb, uint32_t bar) const {
        const int y = t.z * g.rows + kb * 64;
        const CUtensorMap *a = t.w == 0 ? dU1 : t.w == 1 ? dU2 : dO, *b = t.w == 0 ? X : t.w == 1 ? H1 : H2;
        tc::tma_load_2d(sa, a, bar, t.m0, y);
        tc::tma_load_2d(sa + 8192, a, bar, t.m0 + 64, y);            // (dO: beyond its 16 columns, zeros)
        tc::tma_load_2d(sb, b, bar, t.n0, y);
        tc::tma_load_2d(sb + 8192, b, bar, t.n0 + 64, y);
    }
    using Fetched = tc::Nothing;
    __device__ Fetched fetch(const Tile&, int, int) const { return Fetched{}; }
    __device__ void extra(int warp, int lane) const {
        const int chains = g.B < 32 ? g.B : 32;
        if (blockIdx.x == 0 && warp == 0 && lane == 0) {
            g.counters[0] = (int)((g.counters[0] + 1) % g.steps_per_epoch);
            g.counters[1] += 1;
            g.counters[8] += 1;
        }
        for (int w = blockIdx.x + gridDim.x * warp; w < 17 * chains; w += gridDim.x * kWgradExtra) {
            const int l = w / 17, j = w % 17;              // 64 columns of dU1, of dU2; dO's 16
            if (j == 16 && lane >= kOutP / 2) continue;
            const int ld = j == 16 ? kOutP : kHid, c = (j & 7) * 64 * (j < 16) + 2 * lane;
            const __nv_bfloat16* src = (j < 8 ? g.du[0] : j < 16 ? g.du[1] : g.du[2]) + c;
            float s0 = 0.f, s1 = 0.f;
#pragma unroll 32
            for (int r = l; r < g.B; r += 32) {
                const unsigned p = *reinterpret_cast<const unsigned*>(src + (int64_t)r * ld);
                s0 += __uint_as_float(p << 16);
                s1 += __uint_as_float(p & 0xffff0000u);
            }
            float* d = (j < 8 ? g.chain[0] : j < 16 ? g.chain[1] : g.chain[2]) + l * ld + c;
            *reinterpret_cast<float2*>(d) = make_float2(s0, s1);
        }
    }
    __device__ void emit(const Tile& t, int row, int col0, const float (&v)[16], const Fetched&) const {
        if (t.w == 2 && row >= kOutP) return;
        float* d = (t.w == 0 ? g.d[0] : t.w == 1 ? g.d[1] : g.d[2]) + t.z * g.zstride + (int64_t)row * t.N + col0;
        unsigned h[2][8];
#pragma unroll
        for (int i = 0; i < 16; ++i) h[i >> 3][i & 7] = __float_as_uint(v[i]);
        st32(d, h[0]);
        st32(d + 8, h[1]);
    }
};
constexpr int kWgradThreads = tc::kGemmThreads<128> + 32 * kWgradExtra;
__global__ void __launch_bounds__(kWgradThreads, 1)
wgrad_kernel(const __grid_constant__ CUtensorMap dU1, const __grid_constant__ CUtensorMap X,
             const __grid_constant__ CUtensorMap dU2, const __grid_constant__ CUtensorMap H1,
             const __grid_constant__ CUtensorMap dO, const __grid_constant__ CUtensorMap H2,
             const __grid_constant__ Wgrad g, int* err) {
    const WgradProb p{&dU1, &X, &dU2, &H1, &dO, &H2, g};
    tc::gemm_core<128, kStages>(p, err);
}

// The function attributes of every product of a training step, set before a graph capture.
template <int BN, class Epi, bool BMN = false>
cudaError_t gemm_attr() {
    return cudaFuncSetAttribute(tc::gemm_kernel<BN, kStages, Epi, false, BMN>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, tc::Layout<BN, kStages>::kBytes);
}
cudaError_t all_attrs() {
    cudaError_t e = gemm_attr<128, EpiHidden>();
    if (e == cudaSuccess) e = gemm_attr<32, EpiLoss>();
    if (e == cudaSuccess) e = gemm_attr<128, EpiGeluGrad, true>();
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::Layout<128, kStages>::kBytes);
    return e;
}

template <int BN, bool BMN = false, class Epi>
cudaError_t gemm(const CUtensorMap& ta, const CUtensorMap& tb, int M, int N, int K, const Epi& epi, int* err,
                 cudaStream_t st) {
    return tc::gemm_launch<BN, kStages, Epi, false, BMN>(ta, tb, M, N, K, 1, epi, err, st);
}

// ---- small kernels -----------------------------------------------------------------------------
// A double as the nearest float (ties to even), by integer operations in the normal float range: a
// conversion instruction takes the narrow FP64 pipe.
__device__ __forceinline__ float f32_of(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    if ((hi & 0x7fffffffu) - (898u << 20) >= (252u << 20)) return (float)x;
    const unsigned l = lo + 0x0fffffffu + ((lo >> 29) & 1u), h = hi + (l < lo);
    return __uint_as_float(((__funnelshift_l(l, h, 3) - (896u << 23)) & 0x7fffffffu) | (hi & 0x80000000u));
}
// Stage a minibatch, a warp a row (eight a block): rows (q B + i) mod n of X (double [n][256]) -> BF16 X_s,
// labels (double [n][6], NaN treated as 0 with zero weight) -> Y_s [B][16].  q is read from the device
// counter, so that the same launch serves every step of a graph.
struct Stage {
    const double* X;
    const double* Y;
    int64_t n;
    int B;
    const int* counters;
    __nv_bfloat16* Xs;
    float* Ys;
    int blocks() const { return (B + 7) / 8; }
    __device__ void operator()(int block) const {
        const int lane = threadIdx.x & 31, i = block * 8 + (threadIdx.x >> 5);      // batch row
        if (i >= B) return;
        const int64_t src = ((int64_t)counters[0] * B + i) % n;
        double x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = X[src * kIn + 32 * e + lane];
        double y = 0.0;
        if (lane < kOut) y = Y[src * kOut + lane];
#pragma unroll
        for (int e = 0; e < 8; ++e) Xs[(int64_t)i * kIn + 32 * e + lane] = __float2bfloat16(f32_of(x[e]));
        if (lane < kOutP) Ys[(int64_t)i * kOutP + lane] = isfinite(y) ? (float)y : 0.f;
    }
};
__global__ void __launch_bounds__(256)
stage_kernel(const __grid_constant__ Stage s) {
    s(blockIdx.x);
}

#include "k_mlp_infer.cuh"

// BF16 copies of the master weights: W1, W2, W3 (padded rows).
__global__ void __launch_bounds__(256)
sync_bf16_kernel(const float* __restrict__ P, __nv_bfloat16* bf) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < Blob::nW1) bf[Blob::bW1 + i] = __float2bfloat16(P[Blob::oW1 + i]);
    if (i < Blob::nW2) bf[Blob::bW2 + i] = __float2bfloat16(P[Blob::oW2 + i]);
    if (i < Blob::nW3)                                      // rows >= 6 stay zero
        bf[Blob::bW3 + i] = __float2bfloat16(i < (int64_t)kOut * kHid ? P[Blob::oW3 + i] : 0.f);
}

// The step's last kernel: gradients from their partial sums (range 0 first, a fixed order, so that every
// step and every graph replay adds the same numbers the same way), AdamW over every parameter (padded
// output rows keep zero gradient and stay zero), the BF16 weights and the loss; and beside these, as they
// share nothing, the next minibatch's staging (the call's last step stages one that a later call stages
// again).  The first kBBlocks blocks take 16 columns each of [b1 | b2 | b3], adding their chains as a
// tree; kWBlocks four weights a thread; the others stage.
constexpr int kWBlocks = (int)((Blob::nW1 + Blob::nW2 + Blob::nW3) / 4 + 255) / 256, kBBlocks = 2 * kHid / 16 + 1;
struct Update {
    float* blob;
    __nv_bfloat16* bf;
    const float* w[3];       // partial sums of dW1, dW2, dW3, ranges zstride apart
    int64_t zstride;
    int slices;
    const float* chain[3];   // of the columns of dU1, dU2 and dO
    int B;
    const float* loss_part;  // [rows of 32]
    float lr, wd;
    const int* counters;
    float* loss_curve;
    Stage next;
};
__device__ __forceinline__ float adamw(const Update& a, float p, float g, float& m, float& v, float c1, float c2) {
    constexpr float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    m = b1 * m + (1.f - b1) * g;
    v = b2 * v + (1.f - b2) * g * g;
    const float mh = m / c1;
    const float vh = v / c2;
    return p - a.lr * (mh / (sqrtf(vh) + eps) + a.wd * p);
}
__global__ void __launch_bounds__(256)
update_kernel(const __grid_constant__ Update a) {
    __shared__ float corr[2], red[32][17];
    const int tid = threadIdx.x;
    tc::let_successor();
    tc::after_predecessor();
    if ((int)blockIdx.x >= kBBlocks + kWBlocks) {
        a.next(blockIdx.x - kBBlocks - kWBlocks);
        return;
    }
    if (tid < 2) corr[tid] = 1.f - powf(tid ? 0.999f : 0.9f, (float)a.counters[1]);
    if ((int)blockIdx.x >= kBBlocks) {
        const int64_t i = ((int64_t)(blockIdx.x - kBBlocks) * 256 + tid) * 4;
        const int k = i < Blob::nW1 ? 0 : i < Blob::nW1 + Blob::nW2 ? 1 : 2;
        const int64_t j = i - (k == 0 ? 0 : k == 1 ? Blob::nW1 : Blob::nW1 + Blob::nW2);      // within its matrix
        const bool in = i < Blob::nW1 + Blob::nW2 + Blob::nW3;
        const int64_t o = (k == 0 ? Blob::oW1 : k == 1 ? Blob::oW2 : Blob::oW3) + j;
        float4* P = reinterpret_cast<float4*>(a.blob + o);
        float4 *M = P + Blob::oM / 4, *V = P + Blob::oV / 4, *G = P + Blob::oG / 4;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f), q = s, m = s, v = s;
        if (in) {
            q = *P;
            m = *M;
            v = *V;
            const float* src = (k == 0 ? a.w[0] : k == 1 ? a.w[1] : a.w[2]) + j;
#pragma unroll 16
            for (int z = 0; z < a.slices; ++z) {
                const float4 p = *reinterpret_cast<const float4*>(src + z * a.zstride);
                s.x += p.x;
                s.y += p.y;
                s.z += p.z;
                s.w += p.w;
            }
        }
        __syncthreads();
        if (in) {
            q.x = adamw(a, q.x, s.x, m.x, v.x, corr[0], corr[1]);
            q.y = adamw(a, q.y, s.y, m.y, v.y, corr[0], corr[1]);
            q.z = adamw(a, q.z, s.z, m.z, v.z, corr[0], corr[1]);
            q.w = adamw(a, q.w, s.w, m.w, v.w, corr[0], corr[1]);
            *P = q;
            *M = m;
            *V = v;
            *G = s;
            if (k == 2 && j >= (int64_t)kOut * kHid) q = make_float4(0.f, 0.f, 0.f, 0.f);
            const __nv_bfloat162 h[2] = {__floats2bfloat162_rn(q.x, q.y), __floats2bfloat162_rn(q.z, q.w)};
            __nv_bfloat16* d = a.bf + (k == 0 ? Blob::bW1 : k == 1 ? Blob::bW2 : Blob::bW3) + j;
            *reinterpret_cast<uint2*>(d) = *reinterpret_cast<const uint2*>(h);
        }
        return;
    }
    const int q = blockIdx.x, k = q < kHid / 16 ? 0 : q < 2 * kHid / 16 ? 1 : 2, ld = k == 2 ? kOutP : kHid;
    const int c0 = k == 2 ? 0 : (q - k * (kHid / 16)) * 16;
    const float* src = (k == 0 ? a.chain[0] : k == 1 ? a.chain[1] : a.chain[2]) + c0 + 2 * (tid & 7);
    float2 s = make_float2(0.f, 0.f);
    if ((tid >> 3) < a.B) s = *reinterpret_cast<const float2*>(src + (tid >> 3) * ld);
    red[tid >> 3][2 * (tid & 7)] = s.x;
    red[tid >> 3][2 * (tid & 7) + 1] = s.y;
    __syncthreads();
    const int lane = tid & 31;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = c0 + 2 * (tid >> 5) + h;
        float g = red[lane][c - c0];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
        if (lane == 0) {
            if (k == 2 && c >= kOut) g = 0.f;
            float* P = a.blob + (k == 0 ? Blob::ob1 : k == 1 ? Blob::ob2 : Blob::ob3) + c;
            *P = adamw(a, *P, g, P[Blob::oM], P[Blob::oV], corr[0], corr[1]);
            P[Blob::oG] = g;
        }
    }
    if (k == 2) {
        float l = 0.f;
        for (int r = tid; r * 32 < a.B; r += 256) l += a.loss_part[r];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        __syncthreads();
        if (lane == 0) red[0][tid >> 5] = l;
        __syncthreads();
        if (tid == 0 && a.loss_curve) {
            for (int w = 1; w < 8; ++w) l += red[0][w];
            a.loss_curve[a.counters[8]] = l;
        }
    }
}

// A call continues from the blob's counters (a restored checkpoint resumes the same sequence
// of minibatches and Adam steps); the minibatch position wraps into this call's rows.
__global__ void wrap_counters_kernel(int* counters, int64_t steps_per_epoch) {
    int64_t q = counters[0] % steps_per_epoch;
    if (q < 0) q += steps_per_epoch;                         // (a blob not zeroed by its owner)
    counters[0] = (int)q;
    if (counters[1] < 0) counters[1] = 0;
    counters[8] = -1;                                        // this call's step
}

// Feature mean / std over the training rows (for the out-of-distribution score): each
// block sums a strided set of rows with one thread per feature (coalesced), then adds its
// partial sums into acc[2][256] (double); feature_stats_finish turns them into mean / std.
__global__ void __launch_bounds__(kIn)
feature_stats_kernel(const double* __restrict__ X, int64_t n, double* acc) {
    const int f = threadIdx.x;
    double s = 0.0, q = 0.0;
    for (int64_t r = blockIdx.x; r < n; r += gridDim.x) {
        const double x = X[r * kIn + f];
        s += x;
        q += x * x;
    }
    atomicAdd(acc + f, s);
    atomicAdd(acc + kIn + f, q);
}
__global__ void feature_stats_finish(const double* acc, int64_t n, float* mean, float* sd) {
    const int f = threadIdx.x;
    const double m = acc[f] / n;
    mean[f] = (float)m;
    sd[f] = (float)sqrt(fmax(acc[kIn + f] / n - m * m, 0.0));
}

// ---- training workspace --------------------------------------------------------------------------
struct TrainWs {
    __nv_bfloat16 *Xs, *H1, *H2, *dO, *dU2, *dU1;
    float *Ys, *U1, *U2;
    double* stats_acc;
    float* part;              // split-K partials of the weight gradients (slices > 1)
    float* loss_part;         // sums over 32 rows
    float* chain[3];          // bias gradients' chains: [min(B, 32)][512] where U1 and U2 were (read
                              // before), [32][16]
    int slices;
    size_t bytes;
};

// K ranges of the weight-gradient products (K = the minibatch rows): the largest power of two
// up to 16 that leaves at least 256 rows per range in whole 64-row blocks.  A few output tiles
// then spread over up to 16x as many CTAs.
int wgrad_slices(int B) {
    int s = 1;
    while (s < 16 && B % (64 * 2 * s) == 0 && B / (2 * s) >= 256) s *= 2;
    return s;
}

size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

TrainWs carve_train(void* base, int B) {
    TrainWs w{};
    char* c = (char*)base;
    size_t o = 0;
    auto take = [&](size_t b) { char* p = c ? c + o : nullptr; o += a256(b); return p; };
    const size_t bf = sizeof(__nv_bfloat16);
    w.Xs = (__nv_bfloat16*)take((size_t)B * kIn * bf);
    w.H1 = (__nv_bfloat16*)take((size_t)B * kHid * bf);
    w.H2 = (__nv_bfloat16*)take((size_t)B * kHid * bf);
    w.dO = (__nv_bfloat16*)take((size_t)B * kOutP * bf);
    w.dU2 = (__nv_bfloat16*)take((size_t)B * kHid * bf);
    w.dU1 = (__nv_bfloat16*)take((size_t)B * kHid * bf);
    w.Ys = (float*)take((size_t)B * kOutP * sizeof(float));
    w.U1 = (float*)take((size_t)B * kHid * sizeof(float));
    w.U2 = (float*)take((size_t)B * kHid * sizeof(float));
    w.stats_acc = (double*)take(2 * kIn * sizeof(double));
    w.chain[0] = w.U1;
    w.chain[1] = w.U2;
    w.chain[2] = (float*)take(32 * kOutP * sizeof(float));
    w.loss_part = (float*)take((size_t)((B + 127) / 128 * 4) * sizeof(float));
    w.slices = wgrad_slices(B);
    w.part = w.slices > 1 ? (float*)take((size_t)w.slices * (Blob::nW1 + Blob::nW2 + Blob::nW3) * sizeof(float))
                          : nullptr;
    w.bytes = o;
    return w;
}

struct Maps {
    CUtensorMap Xs, W1, H1, W2, H2, W3, dO, dU2;             // K-major operands
    CUtensorMap tW3, tW2, tdO, tH2, tdU2, tH1, tdU1, tX;     // the same matrices by boxes of 64 rows
};

cudaError_t make_maps(Maps& m, const TrainWs& w, const __nv_bfloat16* bf, int B) {
    cudaError_t e = cudaSuccess;
    auto mk = [&](CUtensorMap* t, const void* p, int64_t rows, int64_t cols, int box) {
        if (e == cudaSuccess) e = rs_make_tmap_bf16(t, p, rows, cols, cols, box);
    };
    mk(&m.Xs, w.Xs, B, kIn, 128);
    mk(&m.W1, bf + Blob::bW1, kHid, kIn, 128);
    mk(&m.H1, w.H1, B, kHid, 128);
    mk(&m.W2, bf + Blob::bW2, kHid, kHid, 128);
    mk(&m.H2, w.H2, B, kHid, 128);
    mk(&m.W3, bf + Blob::bW3, kOutP, kHid, 32);
    mk(&m.dO, w.dO, B, kOutP, 128);
    mk(&m.dU2, w.dU2, B, kHid, 128);
    mk(&m.tW3, bf + Blob::bW3, kOutP, kHid, 64);
    mk(&m.tW2, bf + Blob::bW2, kHid, kHid, 64);
    mk(&m.tdO, w.dO, B, kOutP, 64);
    mk(&m.tH2, w.H2, B, kHid, 64);
    mk(&m.tdU2, w.dU2, B, kHid, 64);
    mk(&m.tH1, w.H1, B, kHid, 64);
    mk(&m.tdU1, w.dU1, B, kHid, 64);
    mk(&m.tX, w.Xs, B, kIn, 64);
    return e;
}

// Forward + backward for the staged minibatch: the weight gradients' partial sums (straight into the
// blob's gradients when the rows are one range).
cudaError_t step_body(float* blob, const TrainWs& w, const Maps& m, int B, int* counters, int64_t spe, int* err,
                      cudaStream_t st) {
    float* G = blob + Blob::oG;
    const float* P = blob;
    const float sc = 2.0f / (6.0f * (float)B);
    cudaError_t e = gemm<128>(m.Xs, m.W1, B, kHid, kIn, EpiHidden{P + Blob::ob1, w.U1, w.H1, B}, err, st);
    if (e == cudaSuccess)
        e = gemm<128>(m.H1, m.W2, B, kHid, kHid, EpiHidden{P + Blob::ob2, w.U2, w.H2, B}, err, st);
    if (e == cudaSuccess)
        e = gemm<32>(m.H2, m.W3, B, kOutP, kHid, EpiLoss{P + Blob::ob3, w.Ys, w.dO, w.loss_part, sc}, err, st);
    if (e == cudaSuccess)      // dU2 = (dO W3) * gelu'(U2)
        e = gemm<128, true>(m.dO, m.tW3, B, kHid, kOutP, EpiGeluGrad{w.U2, w.dU2, B}, err, st);
    if (e == cudaSuccess)      // dU1 = (dU2 W2) * gelu'(U1)
        e = gemm<128, true>(m.dU2, m.tW2, B, kHid, kHid, EpiGeluGrad{w.U1, w.dU1, B}, err, st);
    if (e != cudaSuccess) return e;
    Wgrad g{};
    g.d[0] = w.slices > 1 ? w.part : G + Blob::oW1;
    g.d[1] = w.slices > 1 ? w.part + Blob::nW1 : G + Blob::oW2;
    g.d[2] = w.slices > 1 ? w.part + Blob::nW1 + Blob::nW2 : G + Blob::oW3;
    g.zstride = Blob::nW1 + Blob::nW2 + Blob::nW3;
    g.slices = w.slices;
    g.rows = B / w.slices;
    g.du[0] = w.dU1;
    g.du[1] = w.dU2;
    g.du[2] = w.dO;
    for (int k = 0; k < 3; ++k) g.chain[k] = w.chain[k];
    g.B = B;
    g.counters = counters;
    g.steps_per_epoch = spe;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int tiles = 28 * w.slices;
    return tc::launch_after(wgrad_kernel, tiles < sms ? tiles : sms, kWgradThreads, tc::Layout<128, kStages>::kBytes, st,
                            m.tdU1, m.tX, m.tdU2, m.tH1, m.tdO, m.tH2, g, err);
}

}  // namespace

size_t rs_surrogate_blob_floats() { return (size_t)Blob::nFloats; }
size_t rs_surrogate_train_ws_bytes(int B) { return carve_train(nullptr, B).bytes; }
size_t rs_surrogate_infer_ws_bytes(int64_t chunk) {
    return a256((size_t)chunk * kIn * 2) + 2 * a256((size_t)chunk * kHid * 2);
}
int64_t rs_surrogate_blob_offset(int which) {
    switch (which) {
        case 0: return Blob::oW1;
        case 1: return Blob::ob1;
        case 2: return Blob::oW2;
        case 3: return Blob::ob2;
        case 4: return Blob::oW3;
        case 5: return Blob::ob3;
        case 6: return Blob::oM;
        case 7: return Blob::oV;
        case 8: return Blob::oG;
        case 9: return Blob::oStats;
        case 10: return Blob::oCount;
        default: return -1;
    }
}

// Train for `steps` minibatches of B rows; rows are taken in order (wrapping) from X / Y.
// graph != 0: the step is captured once and replayed.
cudaError_t rs_launch_surrogate_train(float* blob, const double* X, const double* Y, int64_t n, int B,
                                      int64_t steps, float lr, float wd, float* loss_curve, void* ws,
                                      int use_graph, int* err, cudaStream_t st) {
    TrainWs w = carve_train(ws, B);
    __nv_bfloat16* bf = reinterpret_cast<__nv_bfloat16*>(blob + Blob::oBf);
    int* counters = reinterpret_cast<int*>(blob + Blob::oCount);
    Maps m;
    cudaError_t e = make_maps(m, w, bf, B);
    if (e == cudaSuccess) e = all_attrs();
    if (e != cudaSuccess) return e;
    const int64_t spe = n / B > 0 ? n / B : 1;
    // statistics for the OOD score, BF16 copies of the initial weights, the counters' position
    e = cudaMemsetAsync(w.stats_acc, 0, 2 * kIn * sizeof(double), st);
    if (e != cudaSuccess) return e;
    feature_stats_kernel<<<(unsigned)(n < 1024 ? n : 1024), kIn, 0, st>>>(X, n, w.stats_acc);
    feature_stats_finish<<<1, kIn, 0, st>>>(w.stats_acc, n, blob + Blob::oStats, blob + Blob::oStats + kIn);
    sync_bf16_kernel<<<(unsigned)((Blob::nW2 + 255) / 256), 256, 0, st>>>(blob, bf);
    wrap_counters_kernel<<<1, 1, 0, st>>>(counters, spe);
    const Stage stage{X, Y, n, B, counters, w.Xs, w.Ys};
    stage_kernel<<<stage.blocks(), 256, 0, st>>>(stage);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const bool split = w.slices > 1;
    const float* G = blob + Blob::oG;
    const Update u{blob, bf,
                   {split ? w.part : G + Blob::oW1, split ? w.part + Blob::nW1 : G + Blob::oW2,
                    split ? w.part + Blob::nW1 + Blob::nW2 : G + Blob::oW3},
                   Blob::nW1 + Blob::nW2 + Blob::nW3, w.slices, {w.chain[0], w.chain[1], w.chain[2]}, B, w.loss_part, lr, wd, counters,
                   loss_curve, stage};
    auto one_step = [&](cudaStream_t q) -> cudaError_t {
        cudaError_t e2 = step_body(blob, w, m, B, counters, spe, err, q);
        if (e2 == cudaSuccess) e2 = tc::launch_after(update_kernel, kBBlocks + kWBlocks + stage.blocks(), 256, 0, q, u);
        return e2;
    };
    if (!use_graph || !loss_curve) {
        for (int64_t s = 0; s < steps && e == cudaSuccess; ++s) e = one_step(st);
        return e;
    }
    cudaStream_t cap;
    e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
    if (e != cudaSuccess) return e;
    cudaGraph_t g = nullptr;
    cudaGraphExec_t ge = nullptr;
    e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        const cudaError_t eb = one_step(cap);
        e = cudaStreamEndCapture(cap, &g);
        if (eb != cudaSuccess) e = eb;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&ge, g, 0);
    cudaEvent_t ev;
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e == cudaSuccess) {
        // order the graph after the setup work on st
        cudaEventRecord(ev, st);
        cudaStreamWaitEvent(cap, ev, 0);
        for (int64_t s = 0; s < steps && e == cudaSuccess; ++s) e = cudaGraphLaunch(ge, cap);
        cudaEventRecord(ev, cap);
        cudaStreamWaitEvent(st, ev, 0);
        cudaEventDestroy(ev);
    }
    if (ge) cudaGraphExecDestroy(ge);
    if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(cap);
    return e;
}

// Forward pass over n rows in chunks: pred [n][6] (FP32); optional OOD score and fallback flags.
cudaError_t rs_launch_surrogate_infer(const float* blob, const double* X, int64_t n, float ood_thr,
                                      float* pred, float* score, uint8_t* fallback, const uint8_t* masks,
                                      int k, double tau, int flags, uint32_t* rec_code, double* rec_pred,
                                      void* ws, int64_t chunk, int* err, cudaStream_t st) {
    const __nv_bfloat16* bf = reinterpret_cast<const __nv_bfloat16*>(blob + Blob::oBf);
    (void)ws;                     // the activations stay on the chip: neither the workspace nor its
    (void)chunk;                  // chunks are needed
    CUtensorMap tW1, tW2, tW3;
    cudaError_t e = rs_make_tmap_bf16(&tW1, bf + Blob::bW1, kHid, kIn, kIn, 64);
    if (e == cudaSuccess) e = rs_make_tmap_bf16(&tW2, bf + Blob::bW2, kHid, kHid, kHid, 64);
    if (e == cudaSuccess) e = rs_make_tmap_bf16(&tW3, bf + Blob::bW3, kOutP, kHid, kHid, kOutP);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(mlp_infer_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kInfSmem);
    int dev = 0, sms = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    InferArgs a{};
    a.X = X;
    a.n = n;
    a.b1 = blob + Blob::ob1;
    a.b2 = blob + Blob::ob2;
    a.mean = score || fallback ? blob + Blob::oStats : nullptr;
    a.sd = blob + Blob::oStats + kIn;
    a.thr = ood_thr;
    a.score = score;
    a.fallback = fallback;
    a.out = EpiInfer{blob + Blob::ob3, pred, masks, flags, k, (float)log(tau), rec_code, rec_pred};
    a.err = err;
    const int64_t tiles = (n + 127) / 128;
    mlp_infer_kernel<<<(unsigned)(tiles < sms ? tiles : sms), kInfThreads, kInfSmem, st>>>(tW1, tW2, tW3, a);
    return cudaGetLastError();
}
