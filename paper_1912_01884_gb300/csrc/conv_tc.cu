// 3x3 dilated convolutions of the learned window proposal with 32 input and
// 32 output channels on the fifth-generation tensor cores (tcgen05.mma,
// accumulators in tensor memory): the forward, the data gradient (the forward
// of the flipped and transposed weights) and the weight gradient.  The paper
// has no counterpart: the network is an addition in front of the exact method.
//
// Both kernels walk chains of image rows.  A chain is one 128-pixel column
// segment of one image and the rows of one residue modulo the dilation, y =
// rho, rho + dil, rho + 2 dil, ...: the three row taps of a row are then its
// neighbours in the chain, so every input row is copied to shared memory once
// and serves all nine taps.  The rows of all chains, one after the other, are
// split evenly among the persistent CTAs (RowRange); a CTA's piece of a chain
// costs two extra input rows.
//
// An input row is staged by one TMA copy (pixels [x0 - 8, x0 + 136), zero
// outside the image) in the 64-byte swizzled layout, a pixel's 32 channels per
// 64-byte line; a column tap is the same row from pixel 8 + (kx - 1) dil on.
// (Copies of 16 bytes into the no-swizzle layout, by cp.async or by TMA, reach
// 2.6 TB/s on this GPU, 64-byte lines 4.1 TB/s.)
#include <cuda_bf16.h>

#include <algorithm>

#include "cnn.cuh"

namespace fhtdp {
namespace {

constexpr int kTcC = 32;                 // channels
constexpr int kTcM = 128;                // pixels of a segment
constexpr int kTcHalo = 8;               // largest dilation
constexpr int kTcPix = kTcM + 2 * kTcHalo;             // staged pixels of a row
constexpr int kARow = kTcPix * kTcC * 2;                // bytes of one staged row (9,216)

// Device status of the tensor-core convolutions: FHTDP_ETIMEOUT once a
// bounded wait gave up (read with fhtdp_cnn_status).
__device__ int g_conv_tc_status;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor: start address, leading and stride byte
// offsets, each in 16-byte units; bit 46 is the descriptor version.
//  - no swizzle, K-major ("core matrices" of 8 rows x 16 bytes in 128
//    contiguous bytes): the leading offset is the step between core matrices
//    along K, the stride offset the step along N;
//  - 64-byte swizzle (code 4 at bit 61): rows of 64 bytes, eight to a group;
//    K-major (a row = 32 values of K) the stride offset is the step between
//    groups; MN-major (a row = 32 values of M or N for one k) the stride
//    offset is the step between groups of eight k, the leading offset that
//    between blocks of 32 along M or N.
// The swizzle works on address bits, so that an operand may start at any row.
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr & 0x3ffffu) >> 4) | ((uint64_t)((lbo & 0x3ffffu) >> 4) << 16) |
           ((uint64_t)((sbo & 0x3ffffu) >> 4) << 32) | (1ull << 46);
}
constexpr uint64_t kSwizzle64 = 4ull << 61;

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), bf16
// A and B (bits 7-9 and 10-12 = 1), K-major (bits 15 and 16 for MN-major A
// and B), N >> 3 at bit 17, M >> 4 at bit 24 (M = 128).
__host__ __device__ constexpr uint32_t idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(kTcM >> 4) << 24);
}
constexpr uint32_t kMnMajor = (1u << 15) | (1u << 16);

// One lane of a converged warp.  The MMA warp runs its loop with all lanes
// and issues under this predicate: operands computed by the whole warp stay
// in uniform registers, while a loop of one lane spends about 100 cycles an
// MMA on moving them there.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t ad, uint64_t bd, uint32_t id,
                                         uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(ad), "l"(bd), "r"(id), "r"(acc)
        : "memory");
}
// Arrives on `bar` once every MMA issued so far by this thread is complete.
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            smem_u32(bar))
        : "memory");
}
// 32 columns of this warp's lane quarter.
__device__ __forceinline__ void tmem_ld32(uint32_t addr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
        "%28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t addr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(slot)),
                 "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t addr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols)
                 : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("{ .reg .b64 st; mbarrier.arrive.shared::cta.b64 st, [%0]; }" ::"r"(
                     smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t *bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0;
}
// Bounded parity wait.  After `limit` cycles it records FHTDP_ETIMEOUT and
// raises `gave_up`, at which every other wait of the CTA returns at once: the
// roles then run to their end with undefined results.
__device__ __forceinline__ void mbar_wait(uint64_t *bar, uint32_t parity, long long limit,
                                          volatile int *gave_up) {
    if (mbar_try(bar, parity)) return;
    const long long t0 = clock64();
    while (!mbar_try(bar, parity)) {
        if (*gave_up) return;
        if (clock64() - t0 > limit) {
            *gave_up = 1;
            atomicExch(&g_conv_tc_status, FHTDP_ETIMEOUT);
            return;
        }
    }
}
// The last wait for the MMAs before tensor memory is freed: bounded also
// when an earlier wait gave up.
__device__ __forceinline__ void mbar_drain(uint64_t *bar, uint32_t parity, long long limit) {
    const long long t0 = clock64();
    while (!mbar_try(bar, parity) && clock64() - t0 <= limit) {
    }
}

// A TMA copy of `bytes` bytes announced on `bar` (one arrival).
__device__ __forceinline__ void mbar_expect(uint64_t *bar, uint32_t bytes) {
    asm volatile("{ .reg .b64 st; mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1; }" ::"r"(
                     smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}
// One row from pixel x of row y, image n of a [n][y][x][32 channels] map into
// shared memory; zero outside the image.
__device__ __forceinline__ void tma_row(uint32_t dst, const CUtensorMap *map, int x, int y, int n,
                                        uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
        "l"(map), "r"(0), "r"(x), "r"(y), "r"(n), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void fence_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ---------------------------------------------------------------------------
// Forward: Y(p)[co] = act(sum over taps t and channels ci of X(p + off(t))[ci]
// * W[t][ci][co] + bias[co]).
//
// The MMA's rate for few output channels is set by reading the A operand (128
// pixels x 16 channels) from shared memory, about 64 cycles whatever N is, so
// each A operand serves all three row taps: an input row r is multiplied by
// [W(ky=2) | W(ky=1) | W(ky=0)] (N = 96), whose three blocks of 32 columns are
// the accumulators of the output rows before, at and after r in the chain.
// They are neighbours in a ring of 8 accumulators in tensor memory (a group
// that wraps around takes two MMAs), six MMAs of K = 16 per row instead of 18.
// The sums of one output value run over (ky, kx, ci) in ascending order.
//
// Roles: warps 0-3 and 4-7 read finished accumulators back (bias, ReLU or ReLU
// mask, bf16) and store them, row by row in turn; warp 8 issues the MMAs;
// warp 9 copies input rows into 8 stages.
// Bound by DRAM: an input and an output row of 64 bytes a pixel.
// 32 images of 256 x 256: a launch per output tile with a staged copy per tap
// 193 us, these rows by 16-byte asynchronous copies 73, by TMA 44 (6.1 TB/s);
// data gradient with the ReLU mask 182 + 67 -> 62.
constexpr int kFwStages = 8;
constexpr int kFwSlots = 8;
constexpr unsigned kFwCols = kFwSlots * kTcC;            // 256 columns of tensor memory
constexpr int kFwB = 3 * 4 * 96 * 16;                   // weights, [kx][chunk][96 rows][8]
constexpr int kFwMma = 8;                               // the MMA warp
constexpr int kFwThreads = 10 * 32;
constexpr size_t kFwSmem = 1024 + (size_t)kFwStages * kARow + kFwB;   // stages 1024-byte aligned

// Sixteen channels of a pixel at once (dst 32-byte aligned), or eight.
__device__ __forceinline__ void st_px(__nv_bfloat16 *dst, const uint32_t (&v)[8], bool wide) {
    if (wide) {
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst),
                     "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]),
                     "r"(v[7])
                     : "memory");
    } else {
        ((uint4 *)dst)[0] = make_uint4(v[0], v[1], v[2], v[3]);
        ((uint4 *)dst)[1] = make_uint4(v[4], v[5], v[6], v[7]);
    }
}

template <bool kRelu, bool kMask>
__global__ void __launch_bounds__(kFwThreads, 2) conv3x3_rows_kernel(
    const __grid_constant__ CUtensorMap xmap, int N, int H, int W, int dil,
    const __nv_bfloat16 *__restrict__ Wt, int flip, const float *__restrict__ bias,
    const __nv_bfloat16 *__restrict__ mask, __nv_bfloat16 *__restrict__ Y, int wide,
    long long wait_cycles) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t s_full[kFwStages], s_empty[kFwStages];
    __shared__ __align__(8) uint64_t s_acc[kFwSlots], s_free[kFwSlots];
    __shared__ __align__(16) float s_bias[kTcC];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_gave_up;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // uniform
    const uint32_t a0 = (smem_u32(smem) + 1023) & ~1023u, b0 = a0 + kFwStages * kARow;
    unsigned short *wst = (unsigned short *)(smem + (b0 - smem_u32(smem)));
    if (tid == 0) {
        for (int s = 0; s < kFwStages; ++s) {
            mbar_init(&s_full[s], 1);
            mbar_init(&s_empty[s], 1);
        }
        for (int s = 0; s < kFwSlots; ++s) {
            mbar_init(&s_acc[s], 1);
            mbar_init(&s_free[s], 4);
        }
        s_gave_up = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kFwMma) tmem_alloc(&s_tmem, kFwCols);
    // Weights: row block ky of the B operand holds output channels of row tap
    // 2 - ky; flipped and transposed (W'[t][ci][co] = W[8-t][co][ci]) for the
    // data gradient.
    {
        // 8-byte loads, all of a thread's in flight together; weights that do not
        // begin on 8 bytes (any 2-byte address is taken) one value at a time
        constexpr int kLoads = 9 * kTcC * kTcC / 4, kPer = (kLoads + kFwThreads - 1) / kFwThreads;
        uint2 wv[kPer];
        if ((uintptr_t)Wt % 8 == 0) {
#pragma unroll
            for (int m = 0; m < kPer; ++m)
                if (tid + m * kFwThreads < kLoads)
                    wv[m] = __ldg((const uint2 *)Wt + tid + m * kFwThreads);
        } else {
#pragma unroll
            for (int m = 0; m < kPer; ++m)
                if (tid + m * kFwThreads < kLoads) {
                    const unsigned short *q =
                        (const unsigned short *)Wt + 4 * (tid + m * kFwThreads);
                    wv[m] = make_uint2(__ldg(q) | (uint32_t)__ldg(q + 1) << 16,
                                       __ldg(q + 2) | (uint32_t)__ldg(q + 3) << 16);
                }
        }
#pragma unroll
        for (int m = 0; m < kPer; ++m) {
            if (tid + m * kFwThreads >= kLoads) break;
            const int i = 4 * (tid + m * kFwThreads);
            const int a = (i >> 5) & 31, u = i >> 10, t = flip ? 8 - u : u;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int b = (i & 31) + e, ci = flip ? b : a, co = flip ? a : b;
                const uint32_t w = e < 2 ? wv[m].x : wv[m].y;
                const int row = (2 - t / 3) * kTcC + co;
                wst[((t % 3 * 4 + (ci >> 3)) * 96 + row) * 8 + (ci & 7)] =
                    (unsigned short)(e & 1 ? w >> 16 : w);
            }
        }
    }
    if (tid < kTcC) s_bias[tid] = bias ? bias[tid] : 0.0f;
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem, 0);   // uniform
    RowRange<kTcM> rr(N, H, W, dil);
    if (warp == kFwMma) {
        {
            const bool leader = elect_one();
            uint32_t t = 0, oc = 0;   // input rows taken, output rows begun in earlier pieces
            // Operand descriptors: their address field counts 16 bytes, so a
            // step is one addition.  Product m = column tap m / 2, channels 16
            // (m % 2) on; row block b of the weights = row tap 2 - b.
            const uint64_t a_desc = sdesc(a0, 16, 512) | kSwizzle64;
            const uint64_t b_desc = sdesc(b0, 96 * 16, 128);
            uint64_t a_off[6];
#pragma unroll
            for (int m = 0; m < 6; ++m)
                a_off[m] = (uint64_t)(4 * (kTcHalo + ((m >> 1) - 1) * dil) + 2 * (m & 1));
            auto b_off = [](int m) { return (uint64_t)(((m >> 1) * 4 + (m & 1) * 2) * 96); };
            while (rr.next()) {
                for (int j = 0; j < rr.L + 2; ++j, ++t) {
                    const uint32_t s = t % kFwStages;
                    mbar_wait(&s_full[s], (t / kFwStages) & 1, wait_cycles, &s_gave_up);
                    if (j < rr.L) {   // a new accumulator
                        const uint32_t o = oc + j;
                        if (o >= kFwSlots)
                            mbar_wait(&s_free[o % kFwSlots], (o / kFwSlots - 1) & 1, wait_cycles,
                                      &s_gave_up);
                    }
                    tc_fence_after();
                    // Output rows lo..hi of the piece take products of this
                    // input row; their accumulators are side by side, in two
                    // runs where the ring ends between them.
                    const int lo = max(0, j - 2), hi = min(rr.L - 1, j);
                    const uint64_t arow = a_desc + (uint64_t)((s * kARow) >> 4);
                    const uint32_t slot = (oc + lo) % kFwSlots, blk = lo - (j - 2);
                    const uint32_t room = kFwSlots - slot, d1 = tmem + slot * kTcC;
                    const uint64_t b1 = b_desc + blk * kTcC;
                    // `cnt` accumulators from output row lo on: product m
                    auto product = [&](int m, uint32_t cnt) {
                        const uint32_t c1 = min(cnt, room);
                        mma_bf16(d1, arow + a_off[m], b1 + b_off(m), idesc(kTcC * c1), 1);
                        if (cnt > c1)
                            mma_bf16(tmem, arow + a_off[m], b1 + b_off(m) + c1 * kTcC,
                                     idesc(kTcC * (cnt - c1)), 1);
                    };
                    const uint32_t cnt = hi - lo + 1;
                    if (leader) {
                    if (hi == j) {   // the first product of output row j starts its sum
                        mma_bf16(tmem + ((oc + j) % kFwSlots) * kTcC, arow + a_off[0],
                                 b_desc + b_off(0) + 2 * kTcC, idesc(kTcC), 0);
                        if (cnt > 1) product(0, cnt - 1);
                    } else {
                        product(0, cnt);
                    }
                    if (cnt == 3 && room >= 3) {
#pragma unroll
                        for (int m = 1; m < 6; ++m)
                            mma_bf16(d1, arow + a_off[m], b1 + b_off(m), idesc(3 * kTcC), 1);
                    } else {
#pragma unroll
                        for (int m = 1; m < 6; ++m) product(m, cnt);
                    }
                    mma_commit(&s_empty[s]);
                    if (j >= 2) mma_commit(&s_acc[(oc + j - 2) % kFwSlots]);
                    }
                    __syncwarp();
                }
                oc += rr.L;
            }
            // every MMA is complete before the CTA frees its memory
            if (t) mbar_drain(&s_empty[(t - 1) % kFwStages], ((t - 1) / kFwStages) & 1,
                              4 * wait_cycles);
        }
        __syncwarp();
    } else if (warp < 8) {
        // two groups of four warps take the output rows in turn
        uint32_t oc = 0;
        const uint32_t lanes = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
        while (rr.next()) {
            for (int o = 0; o < rr.L; ++o, ++oc) {
                if ((int)(oc & 1) != (warp >> 2)) continue;
                const uint32_t slot = oc % kFwSlots;
                const int x = rr.x0 + (tid & 127);
                const size_t px = (((size_t)rr.n * H + rr.row(rr.i + o)) * W + x) * kTcC;
                uint4 mv[4];
                if (kMask && x < W) {   // in flight during the wait
#pragma unroll
                    for (int q = 0; q < 4; ++q) mv[q] = __ldg((const uint4 *)(mask + px) + q);
                }
                mbar_wait(&s_acc[slot], (oc / kFwSlots) & 1, wait_cycles, &s_gave_up);
                tc_fence_after();
                __syncwarp();
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    uint32_t r[16];
                    tmem_ld16(lanes + slot * kTcC + 16 * half, r);
                    if (half) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&s_free[slot]);
                    }
                    uint32_t packed[8];
#pragma unroll
                    for (int c = 0; c < 16; c += 2) {
                        float v0 = __uint_as_float(r[c]), v1 = __uint_as_float(r[c + 1]);
                        if (!kMask) {
                            const float2 bv = *(const float2 *)&s_bias[16 * half + c];
                            v0 += bv.x;
                            v1 += bv.y;
                        }
                        if (kRelu) {
                            v0 = fmaxf(v0, 0.0f);
                            v1 = fmaxf(v1, 0.0f);
                        }
                        const __nv_bfloat162 hv = __floats2bfloat162_rn(v0, v1);
                        packed[c / 2] = *(const uint32_t *)&hv;
                    }
                    if (kMask) {
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const uint4 m4 = mv[2 * half + (q >> 2)];
                            const uint32_t mw = (q & 3) == 0   ? m4.x
                                                : (q & 3) == 1 ? m4.y
                                                : (q & 3) == 2 ? m4.z
                                                               : m4.w;
                            const float2 mf = __bfloat1622float2(*(const __nv_bfloat162 *)&mw);
                            if (!(mf.x > 0.0f)) packed[q] &= 0xffff0000u;
                            if (!(mf.y > 0.0f)) packed[q] &= 0x0000ffffu;
                        }
                    }
                    if (x < W) st_px(Y + px + 16 * half, packed, wide);
                }
            }
        }
    } else if (lane == 0) {
        uint32_t t = 0;
        while (rr.next()) {
            for (int j = 0; j < rr.L + 2; ++j, ++t) {
                const uint32_t s = t % kFwStages;
                if (t >= kFwStages)
                    mbar_wait(&s_empty[s], (t / kFwStages - 1) & 1, wait_cycles, &s_gave_up);
                mbar_expect(&s_full[s], kARow);
                tma_row(a0 + s * kARow, &xmap, rr.x0 - kTcHalo, rr.row(rr.i - 1 + j), rr.n,
                        &s_full[s]);
            }
        }
        // every copy has landed before the CTA frees its memory
        for (uint32_t r = t > kFwStages ? t - kFwStages : 0; r < t; ++r)
            mbar_drain(&s_full[r % kFwStages], (r / kFwStages) & 1, 4 * wait_cycles);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kFwMma) {
        tc_fence_after();
        tmem_dealloc(tmem, kFwCols);
    }
}

// ---------------------------------------------------------------------------
// Weight and bias gradients: dW[t][ci][co] += sum over pixels p of X(p +
// off(t))[ci] * dZ(p)[co], db[co] += sum of dZ(p)[co].
//
// As GEMMs with the pixels as K, one per column tap kx, of two output rows at
// a time: A = four neighbouring input rows of the chain (M = 4 rows x 32
// channels), B = the two dZ rows between them (N = 2 x 32), so that six of
// the eight 32 x 32 blocks are row taps of one of the two dZ rows (block
// (a, b) is ky = a - b) and two are not used.  24 MMAs per two rows, each
// reading its A operand (the bound of these MMAs) for 64 columns instead of
// 32.  Both operands are MN-major as they lie in memory (channels
// contiguous).  Input rows are staged in pairs in a ring of three; the pair
// in slot 0 is copied to a fourth slot as well, so that the four rows of a
// step are always side by side.
//
// Roles: warp 4 issues the MMAs, warp 5 copies (a step ahead), warps
// 0-3 add up dZ for db and at the end add the accumulators (192 columns of
// tensor memory, kept over the CTA's whole range) to dW.
// Bound by DRAM: an input and a dZ row of 64 bytes a pixel.
// 32 images of 256 x 256: a staged copy per tap 267 us, rows by 16-byte
// asynchronous copies 120, by TMA 51 (5.3 TB/s).
constexpr int kWgPairs = 3;
constexpr int kWgZRow = kTcM * kTcC * 2;                   // a staged dZ row (8,192)
constexpr int kWgXBytes = (kWgPairs + 1) * 2 * kARow;      // 73,728
constexpr size_t kWgSmem = 1024 + kWgXBytes + 2 * 2 * (size_t)kWgZRow;   // 107,520
constexpr int kWgThreads = 192;
constexpr unsigned kWgCols = 256;               // three 64-column accumulators

__global__ void __launch_bounds__(kWgThreads, 2) conv3x3_wgrad_rows_kernel(
    const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap zmap, int N,
    int H, int W, int dil, float *__restrict__ dW, float *__restrict__ db,
    float *__restrict__ part, int vec, long long wait_cycles) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t s_xfull[kWgPairs], s_xempty[kWgPairs];
    __shared__ __align__(8) uint64_t s_zfull[2], s_zempty[2], s_done;
    __shared__ float s_db[128 * 9];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_gave_up;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // uniform
    const uint32_t x0s = (smem_u32(smem) + 1023) & ~1023u, z0s = x0s + kWgXBytes;
    if (tid == 0) {
        for (int s = 0; s < kWgPairs; ++s) {
            mbar_init(&s_xfull[s], 1);
            mbar_init(&s_xempty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&s_zfull[s], 1);
            mbar_init(&s_zempty[s], 1 + 4);   // the MMAs and warps 0-3
        }
        mbar_init(&s_done, 1);
        s_gave_up = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 4) tmem_alloc(&s_tmem, kWgCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem, 0);   // uniform
    RowRange<kTcM> rr(N, H, W, dil);
    if (warp == 4) {
        {
            const bool leader = elect_one();
            uint32_t pc = 0, q = 0;   // pairs and steps taken in all
            const uint64_t x_desc = sdesc(x0s, kARow, 512) | kSwizzle64;
            const uint64_t z_desc = sdesc(z0s, kWgZRow, 512) | kSwizzle64;
            while (rr.next()) {
                const int steps = (rr.L + 1) / 2;
                mbar_wait(&s_xfull[pc % kWgPairs], (pc / kWgPairs) & 1, wait_cycles, &s_gave_up);
                for (int st = 0; st < steps; ++st, ++q, ++pc) {
                    const uint32_t nx = pc + 1;
                    mbar_wait(&s_xfull[nx % kWgPairs], (nx / kWgPairs) & 1, wait_cycles,
                              &s_gave_up);
                    mbar_wait(&s_zfull[q & 1], (q >> 1) & 1, wait_cycles, &s_gave_up);
                    tc_fence_after();
                    const uint64_t xa = x_desc + (uint64_t)(((pc % kWgPairs) * (2 * kARow)) >> 4);
                    const uint64_t zb = z_desc + (uint64_t)(((q & 1) * (2 * kWgZRow)) >> 4);
                    if (leader) {
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx) {
                        const uint64_t ad = xa + (uint64_t)(4 * (kTcHalo + (kx - 1) * dil));
#pragma unroll
                        for (int j = 0; j < kTcM / 16; ++j)
                            mma_bf16(tmem + 64u * kx, ad + 64 * j, zb + 64 * j,
                                     idesc(64) | kMnMajor, q != 0 || j != 0);
                    }
                    mma_commit(&s_xempty[pc % kWgPairs]);
                    mma_commit(&s_zempty[q & 1]);
                    }
                    __syncwarp();
                }
                if (leader) mma_commit(&s_xempty[pc % kWgPairs]);   // the piece's last pair
                __syncwarp();
                ++pc;
            }
            if (leader) mma_commit(&s_done);
            __syncwarp();
            mbar_drain(&s_done, 0, 4 * wait_cycles);
        }
        __syncwarp();
    } else if (warp < 4) {
        // db: thread = 16-byte place tid & 3 of pixels (tid >> 2) + 32 m, which
        // holds channel chunk (tid & 3) ^ ((pixel >> 1) & 3) of each
        float sum[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        uint32_t q = 0;
        while (rr.next()) {
            const int steps = (rr.L + 1) / 2;
            for (int st = 0; st < steps; ++st, ++q) {
                mbar_wait(&s_zfull[q & 1], (q >> 1) & 1, wait_cycles, &s_gave_up);
                {
                    const unsigned char *z = smem + (z0s - smem_u32(smem)) +
                                             (q & 1) * (2 * kWgZRow) + tid * 16;
#pragma unroll
                    for (int m = 0; m < 8; ++m) {
                        const uint4 v =
                            *(const uint4 *)(z + (m >> 2) * kWgZRow + (m & 3) * 32 * 64);
                        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float2 f = __bfloat1622float2(*(const __nv_bfloat162 *)&w[e]);
                            sum[2 * e] += f.x;
                            sum[2 * e + 1] += f.y;
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&s_zempty[q & 1]);
            }
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) s_db[tid * 9 + e] = sum[e];
    } else if (lane == 0) {
        uint32_t pc = 0, q = 0;
        auto pair = [&](int first) {   // chain rows first, first + 1
            const uint32_t s = pc % kWgPairs;
            if (pc >= kWgPairs)
                mbar_wait(&s_xempty[s], (pc / kWgPairs - 1) & 1, wait_cycles, &s_gave_up);
            const int x = rr.x0 - kTcHalo;
            mbar_expect(&s_xfull[s], (s == 0 ? 4 : 2) * kARow);
            for (int r = 0; r < 2; ++r) {
                const int y = rr.row(first + r);
                tma_row(x0s + (2 * s + r) * kARow, &xmap, x, y, rr.n, &s_xfull[s]);
                if (s == 0)
                    tma_row(x0s + (2 * kWgPairs + r) * kARow, &xmap, x, y, rr.n, &s_xfull[s]);
            }
            ++pc;
        };
        while (rr.next()) {
            const int steps = (rr.L + 1) / 2;
            pair(rr.i - 1);
            for (int st = 0; st < steps; ++st, ++q) {
                pair(rr.i + 1 + 2 * st);
                const uint32_t s = q & 1;
                if (q >= 2) mbar_wait(&s_zempty[s], (q / 2 - 1) & 1, wait_cycles, &s_gave_up);
                mbar_expect(&s_zfull[s], 2 * kWgZRow);
                for (int r = 0; r < 2; ++r) {
                    const bool in = 2 * st + r < rr.L;   // rows of this piece only: else zeros
                    tma_row(z0s + (2 * s + r) * kWgZRow, &zmap, rr.x0,
                            in ? rr.row(rr.i + 2 * st + r) : -1, rr.n, &s_zfull[s]);
                }
            }
        }
        // every copy has landed before the CTA frees its memory
        for (uint32_t r = pc > kWgPairs ? pc - kWgPairs : 0; r < pc; ++r)
            mbar_drain(&s_xfull[r % kWgPairs], (r / kWgPairs) & 1, 4 * wait_cycles);
        for (uint32_t r = q > 2 ? q - 2 : 0; r < q; ++r)
            mbar_drain(&s_zfull[r & 1], (r >> 1) & 1, 4 * wait_cycles);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (!s_gave_up) {
        // The two blocks of each tap (ky = a - b, kx) are added in shared
        // memory (the stages are free now), [tap][ci] rows 33 words apart;
        // lane = input channel of input row a = warp.
        float *sw = (float *)(smem + (x0s - smem_u32(smem)));
        for (int b = 0; b < 2; ++b) {
            if (warp < 4 && warp - b >= 0 && warp - b <= 2)
                for (int kx = 0; kx < 3; ++kx) {
                    uint32_t r[32];
                    tmem_ld32(tmem + ((uint32_t)(32 * warp) << 16) + 64u * kx + 32u * b, r);
                    float *dst = sw + (((warp - b) * 3 + kx) * kTcC + lane) * 33;
#pragma unroll
                    for (int c = 0; c < kTcC; ++c)
                        dst[c] = (b ? dst[c] : 0.0f) + __uint_as_float(r[c]);
                }
            __syncthreads();
        }
        // this CTA's sums: a row of `part`, or added to dW and db
        float *mine = part ? part + (size_t)blockIdx.x * kWgradPart : dW;
        for (int i = tid; i < 9 * kTcC * kTcC / 4; i += kWgThreads) {
            const float *v = sw + (i >> 3) * 33 + (i & 7) * 4;
            float *dst = mine + 4 * i;
            if (part) {
                *(float4 *)dst = make_float4(v[0], v[1], v[2], v[3]);
            } else if (vec) {
                asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(
                                 dst),
                             "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3])
                             : "memory");
            } else {
                for (int e = 0; e < 4; ++e) atomicAdd(dst + e, v[e]);
            }
        }
        if (tid < kTcC && (part || db)) {
            // threads that held chunk tid >> 3 of their pixels
            float sum = 0.0f;
            for (int u = 0; u < 32; ++u)
                sum += s_db[(4 * u + ((tid >> 3) ^ ((u >> 1) & 3))) * 9 + (tid & 7)];
            if (part)
                mine[9 * kTcC * kTcC + tid] = sum;
            else
                atomicAdd(db + tid, sum);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 4) {
        tc_fence_after();
        tmem_dealloc(tmem, kWgCols);
    }
}

// CTAs for `rows` chain rows: two per SM, no more than rows.
unsigned row_grid(long long rows) {
    int sms = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return (unsigned)std::min<long long>(rows, 2LL * (sms > 0 ? sms : 152));
}

constexpr long long kWaitCycles = 4000000000LL;   // about two seconds

// Map of [N][H][W][32] bf16 values, boxes of `pixels` pixels of one row.
bool encode_px_map(CUtensorMap *map, const void *base, int N, int H, int W, int pixels) {
    PFN_cuTensorMapEncodeTiled_v12000 fn = tensor_map_encoder();
    if (!fn || (uintptr_t)base % 16) return false;
    cuuint64_t dims[4] = {kTcC, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)N};
    cuuint64_t strides[3] = {kTcC * 2, (cuuint64_t)W * kTcC * 2, (cuuint64_t)H * W * kTcC * 2};
    cuuint32_t box[4] = {kTcC, (cuuint32_t)pixels, 1, 1}, estr[4] = {1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), dims, strides,
              box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// part (optional): scratch of kWgradParts x kWgradPart floats, 16-byte aligned;
// with it dW and db (contiguous, [9][32][32] then [32]) are written, summed in
// a fixed order.  Without it they are added to, in any order.
int cnn_wgrad_tc(const void *X, int N, int H, int W, int dil, const void *dZ, float *dW,
                 float *db, cudaStream_t stream, float *part) {
    if (dil < 1 || dil > kTcHalo || W < 1 || H < 1 || N < 1)
        return set_error(FHTDP_EINVAL, "conv3x3 wgrad: dilation 1..8 and a non-empty image");
    if (((uintptr_t)X | (uintptr_t)dZ) % 16)
        return set_error(FHTDP_EINVAL, "conv3x3 wgrad: x and dz must be 16-byte aligned");
    // set on every call: the attribute belongs to the current device
    int st = cuda_status(cudaFuncSetAttribute(conv3x3_wgrad_rows_kernel,
                                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)kWgSmem),
                         "cudaFuncSetAttribute");
    if (st) return st;
    CUtensorMap xmap, zmap;
    if (!encode_px_map(&xmap, X, N, H, W, kTcPix) || !encode_px_map(&zmap, dZ, N, H, W, kTcM))
        return set_error(FHTDP_ECUDA, "conv3x3 wgrad: no tensor map of x or dz");
    const long long rows = (long long)N * H * ((W + kTcM - 1) / kTcM);
    unsigned grid = row_grid(rows);
    if (part) grid = std::min<unsigned>(grid, kWgradParts);
    conv3x3_wgrad_rows_kernel<<<grid, kWgThreads, kWgSmem, stream>>>(
        xmap, zmap, N, H, W, dil, dW, db, part, (uintptr_t)dW % 16 == 0, kWaitCycles);
    st = launched("conv3x3_wgrad_rows_kernel");
    if (!st && part) st = cnn_sum_parts(part, (int)grid, kWgradPart, kWgradPart, dW, stream);
    return st;
}

// mask (optional): Y is zeroed where mask is not positive (the ReLU of the
// layer whose output mask is); flip: the weights flipped and transposed.
int cnn_conv3x3_tc(const void *X, int N, int H, int W, int dil, const void *Wt,
                   const float *bias, int relu, void *Y, cudaStream_t stream, bool flip,
                   const void *mask) {
    if (dil < 1 || dil > kTcHalo || W < 1 || H < 1 || N < 1)
        return set_error(FHTDP_EINVAL, "conv3x3: dilation 1..8 and a non-empty image");
    // (x: the tensor map; y and the mask: 16-byte accesses)
    if (((uintptr_t)X | (uintptr_t)Y | (uintptr_t)mask) % 16)
        return set_error(FHTDP_EINVAL, "conv3x3: x and y must be 16-byte aligned");
    auto kern = mask ? conv3x3_rows_kernel<false, true>
                : relu ? conv3x3_rows_kernel<true, false>
                       : conv3x3_rows_kernel<false, false>;
    // set on every call: the attribute belongs to the current device
    int st = cuda_status(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)kFwSmem),
                         "cudaFuncSetAttribute");
    if (st) return st;
    CUtensorMap xmap;
    if (!encode_px_map(&xmap, X, N, H, W, kTcPix))
        return set_error(FHTDP_ECUDA, "conv3x3: no tensor map of x");
    const long long rows = (long long)N * H * ((W + kTcM - 1) / kTcM);
    kern<<<row_grid(rows), kFwThreads, kFwSmem, stream>>>(
        xmap, N, H, W, dil, (const __nv_bfloat16 *)Wt, flip ? 1 : 0, bias,
        (const __nv_bfloat16 *)mask, (__nv_bfloat16 *)Y, (uintptr_t)Y % 32 == 0, kWaitCycles);
    return launched("conv3x3_rows_kernel");
}

int cnn_tc_status(int clear) {
    int v = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_conv_tc_status, sizeof(int));
    if (e != cudaSuccess) return cuda_status(e, "cudaMemcpyFromSymbol");
    if (clear) {
        const int z = 0;
        e = cudaMemcpyToSymbol(g_conv_tc_status, &z, sizeof(int));
        if (e != cudaSuccess) return cuda_status(e, "cudaMemcpyToSymbol");
    }
    return v;
}

}  // namespace fhtdp
