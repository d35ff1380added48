// k_mlp_infer.cuh -- the surrogate's forward pass for inference as one persistent kernel (included by
// k_mlp.cu): double rows in, predictions and rankings out, no activation in memory.
//
// A CTA takes tiles of 128 rows.  X (BF16, 64 KB) and one block of 64 units of H2 at a time (two
// buffers of 16 KB) live in shared memory in the tensor cores' operand layout (K-major, 128-byte
// swizzle); H1 lives in tensor memory, two BF16 a cell, as the A operand of the second layer, which so
// reads only its weights from shared memory.  The weights stream, 784 KB a tile from L2, through a
// ring of seven 64 x 128 tiles (112 KB: the latency of L2 times the rate the products take them).
// Roles, connected by mbarriers:
//   warp 0 (one thread)   weight producer (TMA)
//   warp 1 (one thread)   tcgen05.mma issuer, N = 64: L1 (8 blocks of 64 units, K = 256), L2 (8 blocks,
//                         K = 512), L3 (16 units, K = 64 per block of H2, two blocks behind L2, so that
//                         the next tile's L1 starts before this tile's last epilogues)
//   warps 2 .. 9          epilogues: two warps a tensor-memory lane quarter, 32 columns each: bias,
//                         GELU, BF16, into H1 or H2
//   warps 10 .. 25        staging: the next tile's rows from memory as BF16, kept in registers until L1
//                         has read X, with the out-of-distribution score; and the outputs and ranking
//                         of the tile before (by the epilogue warps these cost 5,000 cycles a tile)
// Tensor memory: H1 256 columns, three accumulators of 64 in rotation (a block's epilogue overlaps the
// next blocks' products), L3's 16.
// What binds: shared memory's 128 bytes a clock (per tile the products read 1.4 MB of operands, TMA
// writes 0.8 MB, X and H2 0.2 MB: 19,000 cycles of the 30,300 a tile takes; the issuing thread is at
// work for 22,700 of them) and the epilogues' tanh (8 cycles a warp, 8,200 a tile) and FP32 (9,200).
// Every product sums in the order of K, as the layer-by-layer kernels did (each its own GEMM through
// memory, 263 us per 131,072 rows: staging 81, layers 70, 84 and 28): the same values bit for bit.
// 1,000,000 rows: 2126 -> 886 us.  On the way: H1 in shared memory and 128-column blocks 1.55 ms; the
// issuing thread chosen by its lane number, which left the products' operands in ordinary registers,
// 1.45 ms where elect_one() gives 0.93; 16 epilogue warps 1.04 to 1.07 ms.
#pragma once

constexpr int kInfEpi = 8, kInfStage = 16;                   // epilogue and staging warps
constexpr int kInfThreads = (2 + kInfEpi + kInfStage) * 32;
constexpr uint32_t kLag = 2;                                 // L3 runs this many blocks behind L2
constexpr int kInfRing = 7;
constexpr uint32_t kXSlot = 16384, kWSlot = 16384;
constexpr uint32_t kOffX = 0, kOffH2 = 4 * kXSlot, kOffW = 6 * kXSlot, kOffStat = kOffW + kInfRing * kWSlot;
constexpr uint32_t kOffBias = kOffStat + 2048, kOffBar = kOffBias + 4096;
constexpr uint32_t kInfSmem = kOffBar + 512;                 // (no static shared memory: 1024-byte aligned)
constexpr uint32_t kTmAcc = 256, kTmD3 = 448;                // tensor-memory columns (H1 from 0)

struct InferArgs {
    const double* X;
    int64_t n;
    const float* b1;
    const float* b2;
    const float* mean;       // null: no score
    const float* sd;
    float thr;
    float* score;
    uint8_t* fallback;
    EpiInfer out;            // rows from 0
    int* err;
};

// A double as a float with its fraction truncated, for the normal float range; `range` collects
// (with max) how far an exponent lies outside it.
__device__ __forceinline__ unsigned trunc_bits(double x, unsigned& range) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned d = (hi & 0x7fffffffu) - (898u << 20);
    range = range > d ? range : d;
    return ((__funnelshift_l(lo, hi, 3) - (896u << 23)) & 0x7fffffffu) | (hi & 0x80000000u);
}

// tcgen05.mma of BF16 tiles whose 128-byte-swizzle descriptors differ only in the start address: the
// issuing thread adds to its low word (one thread issues 416 products a tile).
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return ((saddr & 0x3FFFFu) >> 4) | (1u << 16); }
__device__ __forceinline__ void mma_lo(uint32_t d, uint32_t alo, uint32_t blo, uint32_t idesc, bool accumulate) {
    constexpr uint32_t hi = (1024u >> 4) | (1u << 14) | (2u << 29);
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 x, y;\n\t"
        "mov.b64 x, {%1, %5};\n\tmov.b64 y, {%2, %5};\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %3, p;\n\t}"
        ::"r"(d), "r"(alo), "r"(blo), "r"(idesc), "r"((uint32_t)accumulate), "r"(hi)
        : "memory");
}

// The same with A in tensor memory (two BF16 a cell).
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint32_t blo, uint32_t idesc, bool accumulate) {
    constexpr uint32_t hi = (1024u >> 4) | (1u << 14) | (2u << 29);
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 y;\n\t"
        "mov.b64 y, {%2, %5};\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], y, %3, p;\n\t}"
        ::"r"(d), "r"(a), "r"(blo), "r"(idesc), "r"((uint32_t)accumulate), "r"(hi)
        : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const unsigned (&r)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__global__ void __launch_bounds__(kInfThreads, 1)
mlp_infer_kernel(const __grid_constant__ CUtensorMap tW1, const __grid_constant__ CUtensorMap tW2,
                 const __grid_constant__ CUtensorMap tW3, const InferArgs a) {
    using namespace tc;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* g = smem_raw;
    const uint32_t base = smem_u32(smem_raw), bars = base + kOffBar;
    uint32_t& tmem_slot = *reinterpret_cast<uint32_t*>(g + kOffBar + 496);
    volatile int& gave_up = *reinterpret_cast<volatile int*>(g + kOffBar + 500);
    if (base & 1023u) {                            // (the operand layout needs it; uniform)
        if (threadIdx.x == 0) rs_dev_flag(a.err, RS_ECUDA, -40);
        return;
    }
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    float* stat = reinterpret_cast<float*>(g + kOffStat);
    float* bias_s = reinterpret_cast<float*>(g + kOffBias);
    auto wfull = [&](uint32_t s) { return bars + 8u * s; };                    // kInfRing
    auto wempty = [&](uint32_t s) { return bars + 120u + 8u * s; };            // kInfRing
    auto tfull = [&](uint32_t b) { return bars + 240u + 8u * b; };             // 3
    auto tempty = [&](uint32_t b) { return bars + 264u + 8u * b; };            // 3
    auto h1full = [&](uint32_t b) { return bars + 288u + 8u * b; };            // 8
    auto h2full = [&](uint32_t b) { return bars + 352u + 8u * b; };            // 2
    auto h2done = [&](uint32_t b) { return bars + 368u + 8u * b; };            // 2
    const uint32_t xfull = bars + 384u, xfree = bars + 392u, d3full = bars + 400u, d3empty = bars + 408u;
    if (tid == 0) {
        for (int s = 0; s < kInfRing; ++s) {
            mbar_init(wfull(s), 1);
            mbar_init(wempty(s), 1);
        }
        for (int b = 0; b < 3; ++b) {
            mbar_init(tfull(b), 1);
            mbar_init(tempty(b), kInfEpi);
        }
        for (int b = 0; b < 8; ++b) mbar_init(h1full(b), kInfEpi);
        for (int b = 0; b < 2; ++b) {
            mbar_init(h2full(b), kInfEpi);
            mbar_init(h2done(b), 1);
        }
        mbar_init(xfull, kInfStage);
        mbar_init(xfree, 1);
        mbar_init(d3full, 1);
        mbar_init(d3empty, 4);
        fence_barrier_init();
        gave_up = 0;
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(&tmem_slot), 512);
        tmem_relinquish();
    }
    if (a.mean && tid < kIn) {
        const float d = a.sd[tid];
        stat[tid] = a.mean[tid];
        stat[kIn + tid] = d > 0.f ? 1.0f / d : 0.f;
    }
    for (int i = tid; i < 2 * kHid; i += kInfThreads) bias_s[i] = i < kHid ? a.b1[i] : a.b2[i - kHid];
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = tmem_slot;
    const int64_t tiles = (a.n + 127) / 128;
    // a wait that gives up (RS_ETIMEOUT) ends all waiting; every role still goes through its tiles
    auto wait = [&](uint32_t bar, uint32_t phase, int site) {
        if (mbar_try_wait(bar, phase & 1u)) return;
        if (!gave_up && !mbar_wait(bar, phase & 1u, a.err, site)) gave_up = 1;
    };

    if (warp == 0) {
        if (elect_one()) {                         // ---- weights
            uint32_t s = 0, round = 0;             // the ring's next slot, its times round
            auto next = [&] {
                if (++s == kInfRing) {
                    s = 0;
                    ++round;
                }
            };
            auto load = [&](const CUtensorMap* m, int x, int y) {        // 64 units x 128 of K
                if (round >= 1) wait(wempty(s), round - 1, 41);
                mbar_expect_tx(wfull(s), kWSlot);
                tma_load_2d(base + kOffW + s * kWSlot, m, wfull(s), x, y);
                tma_load_2d(base + kOffW + s * kWSlot + kWSlot / 2, m, wfull(s), x + 64, y);
                next();
            };
            auto load_w3 = [&](int k) {            // 16 units x 64 of K
                if (round >= 1) wait(wempty(s), round - 1, 41);
                mbar_expect_tx(wfull(s), 2048);
                tma_load_2d(base + kOffW + s * kWSlot, &tW3, wfull(s), k * 64, 0);
                next();
            };
            for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
                for (uint32_t blk = 0; blk < 8; ++blk) {
                    for (int kb = 0; kb < 4; kb += 2) load(&tW1, kb * 64, blk * 64);
                    if (blk < kLag && t != blockIdx.x) load_w3(8 - kLag + blk);
                }
                for (uint32_t blk = 0; blk < 8; ++blk) {
                    for (int kb = 0; kb < 8; kb += 2) load(&tW2, kb * 64, blk * 64);
                    if (blk >= kLag) load_w3(blk - kLag);
                }
            }
            for (uint32_t k = 8 - kLag; k < 8; ++k)
                if (blockIdx.x < tiles) load_w3(k);
            // every load has landed (the issuer waits for each, unless a wait gave up)
            for (uint32_t q = 0; q < kInfRing; ++q) {
                const uint32_t n = round + (q < s);
                if (n >= 1) mbar_wait(wfull(q), (n - 1) & 1u, a.err, 43);
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {                         // ---- products
            const uint32_t id64 = idesc_bf16(128, 64), id16 = idesc_bf16(128, 16);
            const uint32_t xl = desc_lo(base + kOffX), h2l = desc_lo(base + kOffH2), wl = desc_lo(base + kOffW);
            uint32_t s = 0, round = 0, acc = 0, it = 0;
            auto next = [&] {
                mma_commit(wempty(s));
                if (++s == kInfRing) {
                    s = 0;
                    ++round;
                }
            };
            auto l3 = [&](uint32_t k, uint32_t t) {    // D3 += H2 block k x W3
                wait(h2full(k & 1), 4 * t + (k >> 1), 45);
                if (k == 0 && t >= 1) wait(d3empty, t - 1, 46);
                wait(wfull(s), round, 44);
                fence_after();
                const uint32_t al = h2l + (k & 1) * (kXSlot >> 4), bl = wl + s * (kWSlot >> 4);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) mma_lo(tmem + kTmD3, al + 2 * kk, bl + 2 * kk, id16, (k | kk) != 0);
                next();
                mma_commit(h2done(k & 1));
                if (k == 7) mma_commit(d3full);
            };
            for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x, ++it) {
                wait(xfull, it, 47);
                for (uint32_t blk = 0; blk < 8; ++blk, ++acc) {
                    const uint32_t b = acc % 3, d = tmem + kTmAcc + b * 64;
                    if (acc >= 3) wait(tempty(b), acc / 3 - 1, 48);
#pragma unroll 1
                    for (int kb = 0; kb < 4; kb += 2) {
                        wait(wfull(s), round, 44);
                        fence_after();
                        const uint32_t al = xl + kb * (kXSlot >> 4), bl = wl + s * (kWSlot >> 4);
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk)
                            mma_lo(d, al + (kk >> 2) * (kXSlot >> 4) + 2 * (kk & 3), bl + (kk >> 2) * (kWSlot >> 5) + 2 * (kk & 3),
                                   id64, (kb | kk) != 0);
                        next();
                    }
                    mma_commit(tfull(b));
                    if (blk < kLag && it >= 1) l3(8 - kLag + blk, it - 1);
                }
                mma_commit(xfree);
                for (uint32_t blk = 0; blk < 8; ++blk, ++acc) {
                    const uint32_t b = acc % 3, d = tmem + kTmAcc + b * 64;
                    wait(tempty(b), acc / 3 - 1, 49);
#pragma unroll 1
                    for (int kb = 0; kb < 8; kb += 2) {
                        if (blk == 0) {
                            wait(h1full(kb), it, 50);
                            wait(h1full(kb + 1), it, 50);
                        }
                        wait(wfull(s), round, 44);
                        fence_after();
                        const uint32_t ta = tmem + kb * 32, bl = wl + s * (kWSlot >> 4);
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk)
                            mma_ts(d, ta + 8 * kk, bl + (kk >> 2) * (kWSlot >> 5) + 2 * (kk & 3), id64, (kb | kk) != 0);
                        next();
                    }
                    mma_commit(tfull(b));
                    if (blk >= kLag) l3(blk - kLag, it);
                }
            }
            for (uint32_t k = 8 - kLag; k < 8; ++k)
                if (it >= 1) l3(k, it - 1);
            // every product has completed before the tensor memory is freed
            if (it > 0) mbar_wait(d3full, (it - 1) & 1u, a.err, 51);
        }
    } else if (warp < 2 + kInfEpi) {               // ---- epilogues
        const int quarter = warp & 3, half = (warp - 2) >> 2, row = quarter * 32 + lane;
        const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16);
        uint32_t acc = 0, it = 0;
        for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x, ++it) {
#pragma unroll 1
            for (int x = 0; x < 16; ++x, ++acc) {
                const uint32_t b = acc % 3, k = x & 7;
                const float4* bias = reinterpret_cast<const float4*>(bias_s + (x < 8 ? 0 : kHid) + k * 64 + half * 32);
                wait(tfull(b), acc / 3, 52);
                __syncwarp();
                fence_after();
                uint32_t r[2][16];
                tmem_ld16_nowait(trow + kTmAcc + b * 64 + half * 32, r[0]);
                tmem_ld16_nowait(trow + kTmAcc + b * 64 + half * 32 + 16, r[1]);
                tmem_wait_ld();
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(tempty(b));
                unsigned h[2][8];                  // 32 columns as BF16 pairs
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float4 bv = bias[c];
                    const int q = c >> 2, j = c & 3;
                    h[q][2 * j] = gelu2(add2(pk2(__uint_as_float(r[q][4 * j]), __uint_as_float(r[q][4 * j + 1])), pk2(bv.x, bv.y)));
                    h[q][2 * j + 1] = gelu2(add2(pk2(__uint_as_float(r[q][4 * j + 2]), __uint_as_float(r[q][4 * j + 3])), pk2(bv.z, bv.w)));
                }
                if (x < 8) {
                    tmem_st8(trow + k * 32 + half * 16, h[0]);
                    tmem_st8(trow + k * 32 + half * 16 + 8, h[1]);
                    tmem_wait_st();
                    fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(h1full(k));
                } else {
                    const uint32_t use = 4 * it + (k >> 1);                  // of this buffer
                    if (use >= 1) {                // L3 has taken the block before
                        wait(h2done(k & 1), use - 1, 53);
                        __syncwarp();
                    }
                    uint8_t* dst = g + kOffH2 + (k & 1) * kXSlot + row * 128;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const unsigned* hc = h[c >> 1] + 4 * (c & 1);
                        *reinterpret_cast<uint4*>(dst + (((4 * half + c) ^ (row & 7)) << 4)) = make_uint4(hc[0], hc[1], hc[2], hc[3]);
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(h2full(k & 1));
                }
            }
        }
    } else {                                       // ---- staging
        const int w = warp - 2 - kInfEpi;          // rows w, w + 16, ... of a tile
        constexpr int kRows = 128 / kInfStage;
        static_assert(kRows == 8, "the sums over a row's lanes below");
        const float4* mu = reinterpret_cast<const float4*>(stat + 8 * lane);
        const float4* si = reinterpret_cast<const float4*>(stat + kIn + 8 * lane);
        // the outputs of a tile's rows: one warp per tensor-memory quarter, in turn; the others wait
        // too, as a parity tells only one phase from the next
        auto outputs = [&](uint32_t it) {
            wait(d3full, it, 54);
            __syncwarp();
            if (((w >> 2) & 3) != (int)(it & 3)) return;
            const int quarter = warp & 3;
            fence_after();
            float v[16];
            tmem_ld16(tmem + ((uint32_t)(quarter * 32) << 16) + kTmD3, v);
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(d3empty);
            const int64_t r = ((int64_t)blockIdx.x + (int64_t)it * gridDim.x) * 128 + quarter * 32 + lane;
            if (r < a.n) a.out(r, v);
        };
        uint32_t it = 0;
        for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x, ++it) {
            uint4 hb[kRows];                       // this lane's 8 values of each row as BF16
            float sc[kRows];
#pragma unroll
            for (int q = 0; q < kRows; ++q) {
                const int64_t r = t * 128 + w + kInfStage * q;
                const double2* src = reinterpret_cast<const double2*>(a.X + r * kIn + 8 * lane);
                double x[8];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const double2 v = r < a.n ? __ldcs(src + e) : make_double2(1.0, 1.0);
                    x[2 * e] = v.x;
                    x[2 * e + 1] = v.y;
                }
                // BF16 rounded to nearest even from the truncated float with a sticky last bit: as
                // from the double itself
                unsigned tb[8], range = 0;
#pragma unroll
                for (int e = 0; e < 8; ++e) tb[e] = trunc_bits(x[e], range);
                if (range < (252u << 20)) {
                    unsigned h[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const unsigned l0 = (unsigned)__double2loint(x[2 * e]) << 3, l1 = (unsigned)__double2loint(x[2 * e + 1]) << 3;
                        const __nv_bfloat162 v = __floats2bfloat162_rn(__uint_as_float(tb[2 * e] | (l0 < 1u ? l0 : 1u)),
                                                                       __uint_as_float(tb[2 * e + 1] | (l1 < 1u ? l1 : 1u)));
                        h[e] = *reinterpret_cast<const unsigned*>(&v);
                    }
                    hb[q] = make_uint4(h[0], h[1], h[2], h[3]);
                } else {                           // zeros, subnormals, infinities, NaN: by conversion
                    alignas(16) __nv_bfloat16 h[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const unsigned d = ((unsigned)__double2hiint(x[e]) & 0x7fffffffu) - (898u << 20);
                        const unsigned l = (unsigned)__double2loint(x[e]) << 3;
                        if (d < (252u << 20)) {
                            h[e] = __float2bfloat16(__uint_as_float(tb[e] | (l < 1u ? l : 1u)));
                        } else {
                            h[e] = __float2bfloat16((float)x[e]);
                            tb[e] = __float_as_uint((float)x[e]);
                        }
                    }
                    hb[q] = *reinterpret_cast<const uint4*>(h);
                }
                if (a.mean) {
                    float s = 0.f;
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const float4 m = mu[e], v = si[e];
                        const float mm[4] = {m.x, m.y, m.z, m.w}, vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int z = 0; z < 4; ++z) {
                            const float d = (__uint_as_float(tb[4 * e + z]) - mm[z]) * vv[z];
                            s = fmaf(d, d, s);
                        }
                    }
                    sc[q] = s;
                }
            }
            if (a.mean) {      // eight rows' sums over the lanes at once: halves of the rows change lanes
                const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
                float s4[4], s2[2];
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    s4[j] = (b4 ? sc[4 + j] : sc[j]) + __shfl_xor_sync(0xffffffffu, b4 ? sc[j] : sc[4 + j], 16);
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    s2[j] = (b3 ? s4[2 + j] : s4[j]) + __shfl_xor_sync(0xffffffffu, b3 ? s4[j] : s4[2 + j], 8);
                float s = (b2 ? s2[1] : s2[0]) + __shfl_xor_sync(0xffffffffu, b2 ? s2[0] : s2[1], 4);
                s += __shfl_xor_sync(0xffffffffu, s, 2);
                s += __shfl_xor_sync(0xffffffffu, s, 1);
                const int64_t r = t * 128 + w + kInfStage * (lane >> 2);
                if ((lane & 3) == 0 && r < a.n) {
                    s /= kIn;
                    if (a.score) a.score[r] = s;
                    if (a.fallback) a.fallback[r] = s > a.thr ? 1 : 0;
                }
            }
            if (it >= 2) outputs(it - 2);
            if (it >= 1) {                         // L1 has read the tile before
                wait(xfree, it - 1, 55);
                __syncwarp();
            }
#pragma unroll
            for (int q = 0; q < kRows; ++q) {
                const int row = w + kInfStage * q;
                *reinterpret_cast<uint4*>(g + kOffX + (lane >> 3) * kXSlot + row * 128 + (((lane & 7) ^ (row & 7)) << 4)) = hb[q];
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(xfull);
        }
        if (it >= 2) outputs(it - 2);
        if (it >= 1) outputs(it - 1);
    }
    fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
}
