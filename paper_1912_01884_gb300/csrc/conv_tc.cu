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
// Shared memory holds operands in the no-swizzle layout of the MMA: "core
// matrices" of 8 x 16 bytes stored as 128 contiguous bytes.  An input row is
// staged as [channel chunk][pixel][8 channels], pixels [x0 - 8, x0 + 136)
// (zero outside the image); a column tap is the same row from pixel 8 + (kx -
// 1) dil.  The step between channel chunks is 32 bytes more than a multiple
// of 128, so that the copies of four chunks of two pixels (consecutive lanes)
// fall into different banks.
#include <cuda_bf16.h>

#include <algorithm>

#include "cnn.cuh"

namespace fhtdp {
namespace {

constexpr int kTcC = 32;                 // channels
constexpr int kTcM = 128;                // pixels of a segment
constexpr int kTcHalo = 8;               // largest dilation
constexpr int kTcPix = kTcM + 2 * kTcHalo;             // staged pixels of a row
constexpr int kAChunk = kTcPix * 16 + 32;               // step between channel chunks
constexpr int kARow = 4 * kAChunk;                      // bytes of one staged row (9,344)

// Device status of the tensor-core convolutions: FHTDP_ETIMEOUT once a
// bounded wait gave up (read with fhtdp_cnn_status).
__device__ int g_conv_tc_status;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor, no swizzle: start address, leading and
// stride byte offsets of the core matrices, each in 16-byte units; bit 46 is
// the descriptor version.  Without swizzling the leading offset is the step
// between core matrices along K and the stride offset the step along M / N,
// for K-major and MN-major operands alike.
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr & 0x3ffffu) >> 4) | ((uint64_t)((lbo & 0x3ffffu) >> 4) << 16) |
           ((uint64_t)((sbo & 0x3ffffu) >> 4) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), bf16
// A and B (bits 7-9 and 10-12 = 1), K-major (bits 15 and 16 for MN-major A
// and B), N >> 3 at bit 17, M >> 4 at bit 24 (M = 128).
__host__ __device__ constexpr uint32_t idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(kTcM >> 4) << 24);
}
constexpr uint32_t kMnMajor = (1u << 15) | (1u << 16);

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

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool valid) {
    // src-size 0 fills the 16 bytes with zeros
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
                 "r"(valid ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void fence_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// The rows [g, end) of this CTA in the sequence of all chains' rows: image by
// image, segment by segment, residue by residue.  next() gives the piece of
// one chain: rows i .. i + L - 1 of the chain (y = rho + dil * i).
struct RowRange {
    long long g, end;
    int H, dil, segs;
    int n, x0, rho, i, L;
    __device__ RowRange(int N, int H_, int W, int dil_)
        : H(H_), dil(dil_), segs((W + kTcM - 1) / kTcM) {
        const long long total = (long long)N * segs * H;
        g = total * blockIdx.x / gridDim.x;
        end = total * (blockIdx.x + 1) / gridDim.x;
    }
    __device__ bool next() {
        if (g >= end) return false;
        const long long u = g / H;
        int h = (int)(g - u * H);
        n = (int)(u / segs);
        x0 = (int)(u - (long long)n * segs) * kTcM;
        const int base = H / dil, more = H - base * dil;   // `more` residues have one row more
        int len;
        if (h < more * (base + 1)) {
            len = base + 1;
            rho = h / len;
            i = h - rho * len;
        } else {
            h -= more * (base + 1);
            len = base;
            rho = more + h / len;
            i = h % len;
        }
        L = (int)min((long long)(len - i), end - g);
        g += L;
        return true;
    }
    __device__ int row(int j) const { return rho + dil * j; }   // image row of chain row j
};

// One input row y of segment x0 into stage `dst`, by 128 threads t: 16-byte
// copies, zero outside the image.
__device__ __forceinline__ void stage_row(const __nv_bfloat16 *X, int n, int y, int x0, int H,
                                          int W, int t, uint32_t dst) {
    const int c = t & 3;
    const bool in = y >= 0 && y < H;
    const __nv_bfloat16 *row = X + (((size_t)n * H + (in ? y : 0)) * W) * kTcC + 8 * c;
#pragma unroll
    for (int m = 0; m < (4 * kTcPix + 127) / 128; ++m) {
        const int q = (t >> 2) + 32 * m;
        if (q >= kTcPix) break;
        const int xx = x0 - kTcHalo + q;
        const bool ok = in && xx >= 0 && xx < W;
        cp_async16(dst + c * kAChunk + q * 16, ok ? row + (size_t)xx * kTcC : X, ok);
    }
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
// Roles: warps 0-3 read finished accumulators back (bias, ReLU or ReLU mask,
// bf16) and store them; warp 4's first lane issues the MMAs; warps 5-8 copy
// input rows into 8 stages (cp.async), three rows in flight per thread.
// Bound by DRAM: an input and an output row of 64 bytes a pixel.
// 32 images of 256 x 256: FWD_BEFORE -> FWD_AFTER.
constexpr int kFwStages = 8, kFwLag = 3;
constexpr int kFwSlots = 8;
constexpr unsigned kFwCols = kFwSlots * kTcC;            // 256 columns of tensor memory
constexpr int kFwB = 3 * 4 * 96 * 16;                   // weights, [kx][chunk][96 rows][8]
constexpr int kFwThreads = 288;
constexpr size_t kFwSmem = kFwB + (size_t)kFwStages * kARow;

// Thirty-two bytes at once (both pointers 32-byte aligned), or sixteen.
__device__ __forceinline__ void st_px(__nv_bfloat16 *dst, const uint32_t (&v)[16], bool wide) {
    if (wide) {
#pragma unroll
        for (int q = 0; q < 2; ++q)
            asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(
                             dst + 16 * q),
                         "r"(v[8 * q]), "r"(v[8 * q + 1]), "r"(v[8 * q + 2]), "r"(v[8 * q + 3]),
                         "r"(v[8 * q + 4]), "r"(v[8 * q + 5]), "r"(v[8 * q + 6]),
                         "r"(v[8 * q + 7])
                         : "memory");
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            ((uint4 *)dst)[q] = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    }
}

template <bool kRelu, bool kMask>
__global__ void __launch_bounds__(kFwThreads, 2) conv3x3_rows_kernel(
    const __nv_bfloat16 *__restrict__ X, int N, int H, int W, int dil,
    const __nv_bfloat16 *__restrict__ Wt, int flip, const float *__restrict__ bias,
    const __nv_bfloat16 *__restrict__ mask, __nv_bfloat16 *__restrict__ Y, int wide,
    long long wait_cycles) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t s_full[kFwStages], s_empty[kFwStages];
    __shared__ __align__(8) uint64_t s_acc[kFwSlots], s_free[kFwSlots];
    __shared__ __align__(16) float s_bias[kTcC];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_gave_up;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t b0 = smem_u32(smem), a0 = b0 + kFwB;
    if (tid == 0) {
        for (int s = 0; s < kFwStages; ++s) {
            mbar_init(&s_full[s], 128);
            mbar_init(&s_empty[s], 1);
        }
        for (int s = 0; s < kFwSlots; ++s) {
            mbar_init(&s_acc[s], 1);
            mbar_init(&s_free[s], 4);
        }
        s_gave_up = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 4) tmem_alloc(&s_tmem, kFwCols);
    // Weights: row block ky of the B operand holds output channels of row tap
    // 2 - ky; flipped and transposed (W'[t][ci][co] = W[8-t][co][ci]) for the
    // data gradient.
    for (int i = tid; i < 9 * kTcC * kTcC; i += kFwThreads) {
        const int b = i & 31, a = (i >> 5) & 31, u = i >> 10;
        const int t = flip ? 8 - u : u, ci = flip ? b : a, co = flip ? a : b;
        const int row = (2 - t / 3) * kTcC + co;
        ((__nv_bfloat16 *)smem)[((t % 3 * 4 + (ci >> 3)) * 96 + row) * 8 + (ci & 7)] = Wt[i];
    }
    if (tid < kTcC) s_bias[tid] = bias ? bias[tid] : 0.0f;
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    RowRange rr(N, H, W, dil);
    if (warp == 4) {
        if (lane == 0) {
            uint32_t t = 0, oc = 0;   // input rows taken, output rows begun in earlier pieces
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
                    const int lo = max(0, j - 2), hi = min(rr.L - 1, j);
                    const uint32_t arow = a0 + s * kARow;
                    // output rows [from, to] of the piece: accumulators side by
                    // side, unless the ring ends between them
                    auto run = [&](uint32_t ad0, uint32_t bd0, int from, int to, uint32_t acc) {
                        while (from <= to) {
                            const uint32_t slot = (oc + from) % kFwSlots;
                            const int cnt = min(to - from + 1, (int)(kFwSlots - slot));
                            mma_bf16(tmem + slot * kTcC, sdesc(ad0, kAChunk, 128),
                                     sdesc(bd0 + (from - (j - 2)) * kTcC * 16, 96 * 16, 128),
                                     idesc(cnt * kTcC), acc);
                            from += cnt;
                        }
                    };
#pragma unroll 1
                    for (int m = 0; m < 6; ++m) {   // column tap, 16 channels
                        const int kx = m >> 1, c2 = (m & 1) * 2;
                        const uint32_t ad0 =
                            arow + (kTcHalo + (kx - 1) * dil) * 16 + c2 * kAChunk;
                        const uint32_t bd0 = b0 + (kx * 4 + c2) * (96 * 16);
                        if (m == 0 && hi == j) {   // the first product of output row j
                            run(ad0, bd0, j, j, 0);
                            run(ad0, bd0, lo, j - 1, 1);
                        } else {
                            run(ad0, bd0, lo, hi, 1);
                        }
                    }
                    mma_commit(&s_empty[s]);
                    if (j >= 2) mma_commit(&s_acc[(oc + j - 2) % kFwSlots]);
                }
                oc += rr.L;
            }
            // every MMA is complete before the CTA frees its memory
            if (t) mbar_drain(&s_empty[(t - 1) % kFwStages], ((t - 1) / kFwStages) & 1,
                              4 * wait_cycles);
        }
        __syncwarp();
    } else if (warp < 4) {
        uint32_t oc = 0;
        while (rr.next()) {
            for (int o = 0; o < rr.L; ++o, ++oc) {
                const uint32_t slot = oc % kFwSlots;
                const int x = rr.x0 + tid;
                const size_t px = (((size_t)rr.n * H + rr.row(rr.i + o)) * W + x) * kTcC;
                uint4 mv[4];
                if (kMask && x < W) {   // in flight during the wait
#pragma unroll
                    for (int q = 0; q < 4; ++q) mv[q] = __ldg((const uint4 *)(mask + px) + q);
                }
                mbar_wait(&s_acc[slot], (oc / kFwSlots) & 1, wait_cycles, &s_gave_up);
                tc_fence_after();
                uint32_t r[32];
                __syncwarp();
                tmem_ld32(tmem + slot * kTcC + ((uint32_t)(32 * warp) << 16), r);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&s_free[slot]);
                if (x >= W) continue;
                uint32_t packed[16];
#pragma unroll
                for (int c = 0; c < kTcC; c += 4) {
                    const float4 bv = *(const float4 *)&s_bias[c];
                    const float bb[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
                    for (int e = 0; e < 4; e += 2) {
                        float v0 = __uint_as_float(r[c + e]) + bb[e];
                        float v1 = __uint_as_float(r[c + e + 1]) + bb[e + 1];
                        if (kRelu) {
                            v0 = v0 > 0.0f ? v0 : 0.0f;
                            v1 = v1 > 0.0f ? v1 : 0.0f;
                        }
                        const __nv_bfloat162 hv = __floats2bfloat162_rn(v0, v1);
                        packed[(c + e) / 2] = *(const uint32_t *)&hv;
                    }
                }
                if (kMask) {
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        const uint4 m4 = mv[q >> 2];
                        const uint32_t mw = (q & 3) == 0   ? m4.x
                                            : (q & 3) == 1 ? m4.y
                                            : (q & 3) == 2 ? m4.z
                                                           : m4.w;
                        const float2 mf = __bfloat1622float2(*(const __nv_bfloat162 *)&mw);
                        if (!(mf.x > 0.0f)) packed[q] &= 0xffff0000u;
                        if (!(mf.y > 0.0f)) packed[q] &= 0x0000ffffu;
                    }
                }
                st_px(Y + px, packed, wide);
            }
        }
    } else {
        const int lt = tid - 160;
        uint32_t t = 0;
        auto landed = [&](uint32_t row) {
            fence_async_smem();
            mbar_arrive(&s_full[row % kFwStages]);
        };
        while (rr.next()) {
            for (int j = 0; j < rr.L + 2; ++j, ++t) {
                const uint32_t s = t % kFwStages;
                if (t >= kFwStages)
                    mbar_wait(&s_empty[s], (t / kFwStages - 1) & 1, wait_cycles, &s_gave_up);
                stage_row(X, rr.n, rr.row(rr.i - 1 + j), rr.x0, H, W, lt, a0 + s * kARow);
                cp_async_commit();
                if (t >= kFwLag) {
                    cp_async_wait<kFwLag>();
                    landed(t - kFwLag);
                }
            }
        }
        cp_async_wait<0>();
        for (uint32_t r = t > kFwLag ? t - kFwLag : 0; r < t; ++r) landed(r);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 4) {
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
// Roles: warp 4's first lane issues the MMAs, warps 5-8 copy (one step
// ahead), warps 0-3 add up dZ for db and at the end add the accumulators (192
// columns of tensor memory, kept over the CTA's whole range) to dW.
// Bound by DRAM: an input and a dZ row of 64 bytes a pixel.
// 32 images of 256 x 256: WG_BEFORE -> WG_AFTER.
constexpr int kWgPairs = 3;
constexpr int kWgChunk = kTcM * 16 + 32;        // step between channel chunks of dZ
constexpr int kWgZRow = 4 * kWgChunk;
constexpr int kWgXBytes = (kWgPairs + 1) * 2 * kARow;      // 74,752
constexpr size_t kWgSmem = kWgXBytes + 2 * 2 * (size_t)kWgZRow;   // 108,032
constexpr int kWgThreads = 288;
constexpr unsigned kWgCols = 256;               // three 64-column accumulators

// 32 consecutive sums of one warp lane into gradient memory.
__device__ __forceinline__ void add32(float *dst, const uint32_t (&r)[32], bool vec) {
    if (vec) {
#pragma unroll
        for (int c = 0; c < 32; c += 4)
            asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(
                             dst + c),
                         "f"(__uint_as_float(r[c])), "f"(__uint_as_float(r[c + 1])),
                         "f"(__uint_as_float(r[c + 2])), "f"(__uint_as_float(r[c + 3]))
                         : "memory");
    } else {
#pragma unroll
        for (int c = 0; c < 32; ++c) atomicAdd(dst + c, __uint_as_float(r[c]));
    }
}

__global__ void __launch_bounds__(kWgThreads, 2) conv3x3_wgrad_rows_kernel(
    const __nv_bfloat16 *__restrict__ X, int N, int H, int W, int dil,
    const __nv_bfloat16 *__restrict__ dZ, float *__restrict__ dW, float *__restrict__ db, int vec,
    long long wait_cycles) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t s_xfull[kWgPairs], s_xempty[kWgPairs];
    __shared__ __align__(8) uint64_t s_zfull[2], s_zempty[2], s_done;
    __shared__ float s_db[kTcC];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_gave_up;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t x0s = smem_u32(smem), z0s = x0s + kWgXBytes;
    if (tid == 0) {
        for (int s = 0; s < kWgPairs; ++s) {
            mbar_init(&s_xfull[s], 128);
            mbar_init(&s_xempty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&s_zfull[s], 128);
            mbar_init(&s_zempty[s], 1 + 4);   // the MMAs and warps 0-3
        }
        mbar_init(&s_done, 1);
        s_gave_up = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < kTcC) s_db[tid] = 0.0f;
    if (warp == 4) tmem_alloc(&s_tmem, kWgCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    RowRange rr(N, H, W, dil);
    if (warp == 4) {
        if (lane == 0) {
            uint32_t pc = 0, q = 0;   // pairs and steps taken in all
            while (rr.next()) {
                const int steps = (rr.L + 1) / 2;
                mbar_wait(&s_xfull[pc % kWgPairs], (pc / kWgPairs) & 1, wait_cycles, &s_gave_up);
                for (int st = 0; st < steps; ++st, ++q, ++pc) {
                    const uint32_t nx = pc + 1;
                    mbar_wait(&s_xfull[nx % kWgPairs], (nx / kWgPairs) & 1, wait_cycles,
                              &s_gave_up);
                    mbar_wait(&s_zfull[q & 1], (q >> 1) & 1, wait_cycles, &s_gave_up);
                    tc_fence_after();
                    const uint32_t xa = x0s + (pc % kWgPairs) * (2 * kARow);
                    const uint32_t zb = z0s + (q & 1) * (2 * kWgZRow);
#pragma unroll 1
                    for (int kx = 0; kx < 3; ++kx) {
                        const uint32_t abase = xa + (kTcHalo + (kx - 1) * dil) * 16;
#pragma unroll
                        for (int j = 0; j < kTcM / 16; ++j)
                            // MN-major, no swizzle: the leading offset steps
                            // along K (8 pixels), the stride offset along M / N
                            mma_bf16(tmem + 64u * kx, sdesc(abase + j * 256, 128, kAChunk),
                                     sdesc(zb + j * 256, 128, kWgChunk), idesc(64) | kMnMajor,
                                     q != 0 || j != 0);
                    }
                    mma_commit(&s_xempty[pc % kWgPairs]);
                    mma_commit(&s_zempty[q & 1]);
                }
                mma_commit(&s_xempty[pc % kWgPairs]);   // the piece's last pair
                ++pc;
            }
            mma_commit(&s_done);
            mbar_drain(&s_done, 0, 4 * wait_cycles);
        }
        __syncwarp();
    } else if (warp < 4) {
        // db: thread = channel chunk tid & 3 of pixels tid >> 2 + 32 m
        float sum[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        uint32_t q = 0;
        while (rr.next()) {
            const int steps = (rr.L + 1) / 2;
            for (int st = 0; st < steps; ++st, ++q) {
                mbar_wait(&s_zfull[q & 1], (q >> 1) & 1, wait_cycles, &s_gave_up);
                if (db) {
                    const unsigned char *z = smem + kWgXBytes + (q & 1) * (2 * kWgZRow) +
                                             (tid & 3) * kWgChunk + (tid >> 2) * 16;
#pragma unroll
                    for (int m = 0; m < 8; ++m) {
                        const uint4 v =
                            *(const uint4 *)(z + (m >> 2) * kWgZRow + (m & 3) * 32 * 16);
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
        if (db) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                for (int o = 4; o < 32; o <<= 1) sum[e] += __shfl_xor_sync(0xffffffffu, sum[e], o);
                if (lane < 4) atomicAdd(&s_db[8 * lane + e], sum[e]);
            }
        }
    } else {
        const int lt = tid - 160;
        uint32_t pc = 0, q = 0;
        // One step's copies are in flight while the MMAs of the step before
        // run: they are announced (landed) before the next step's begin.
        int pend_x = -1, pend_z = -1;
        auto landed = [&]() {
            if (pend_x < 0 && pend_z < 0) return;
            cp_async_commit();
            cp_async_wait<0>();
            fence_async_smem();
            if (pend_x >= 0) mbar_arrive(&s_xfull[pend_x]);
            if (pend_z >= 0) mbar_arrive(&s_zfull[pend_z]);
            pend_x = pend_z = -1;
        };
        auto pair = [&](int first) {   // chain rows first, first + 1
            const uint32_t s = pc % kWgPairs;
            if (pc >= kWgPairs)
                mbar_wait(&s_xempty[s], (pc / kWgPairs - 1) & 1, wait_cycles, &s_gave_up);
            for (int r = 0; r < 2; ++r) {
                stage_row(X, rr.n, rr.row(first + r), rr.x0, H, W, lt,
                          x0s + (2 * s + r) * kARow);
                if (s == 0)
                    stage_row(X, rr.n, rr.row(first + r), rr.x0, H, W, lt,
                              x0s + (2 * kWgPairs + r) * kARow);
            }
            pend_x = (int)s;
            ++pc;
        };
        while (rr.next()) {
            const int steps = (rr.L + 1) / 2;
            landed();
            pair(rr.i - 1);
            for (int st = 0; st < steps; ++st, ++q) {
                landed();
                pair(rr.i + 1 + 2 * st);
                const uint32_t s = q & 1;
                if (q >= 2) mbar_wait(&s_zempty[s], (q / 2 - 1) & 1, wait_cycles, &s_gave_up);
                const int c = lt & 3;
                for (int r = 0; r < 2; ++r) {
                    const bool in = 2 * st + r < rr.L;   // rows of this piece only
                    const __nv_bfloat16 *row =
                        dZ + ((size_t)rr.n * H + (in ? rr.row(rr.i + 2 * st + r) : 0)) * W * kTcC +
                        8 * c;
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        const int p = (lt >> 2) + 32 * m;
                        const bool ok = in && rr.x0 + p < W;
                        cp_async16(z0s + (2 * s + r) * kWgZRow + c * kWgChunk + p * 16,
                                   ok ? row + (size_t)(rr.x0 + p) * kTcC : dZ, ok);
                    }
                }
                pend_z = (int)s;
            }
        }
        landed();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp < 4 && !s_gave_up) {
        // lane = input channel of input row a = warp; block (kx, b) is tap
        // (ky = a - b, kx)
        for (int kx = 0; kx < 3; ++kx)
            for (int b = 0; b < 2; ++b) {
                const int ky = warp - b;
                if (ky < 0 || ky > 2) continue;
                uint32_t r[32];
                tmem_ld32(tmem + ((uint32_t)(32 * warp) << 16) + 64u * kx + 32u * b, r);
                add32(dW + ((size_t)(ky * 3 + kx) * kTcC + lane) * kTcC, r, vec != 0);
            }
        if (db && tid < kTcC) atomicAdd(db + tid, s_db[tid]);
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

}  // namespace

int cnn_wgrad_tc(const void *X, int N, int H, int W, int dil, const void *dZ, float *dW,
                 float *db, cudaStream_t stream) {
    if (dil < 1 || dil > kTcHalo || W < 1 || H < 1 || N < 1)
        return set_error(FHTDP_EINVAL, "conv3x3 wgrad: dilation 1..8 and a non-empty image");
    // set on every call: the attribute belongs to the current device
    int st = cuda_status(cudaFuncSetAttribute(conv3x3_wgrad_rows_kernel,
                                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)kWgSmem),
                         "cudaFuncSetAttribute");
    if (st) return st;
    const long long rows = (long long)N * H * ((W + kTcM - 1) / kTcM);
    conv3x3_wgrad_rows_kernel<<<row_grid(rows), kWgThreads, kWgSmem, stream>>>(
        (const __nv_bfloat16 *)X, N, H, W, dil, (const __nv_bfloat16 *)dZ, dW, db,
        (uintptr_t)dW % 16 == 0, kWaitCycles);
    return launched("conv3x3_wgrad_rows_kernel");
}

// mask (optional): Y is zeroed where mask is not positive (the ReLU of the
// layer whose output mask is); flip: the weights flipped and transposed.
int cnn_conv3x3_tc(const void *X, int N, int H, int W, int dil, const void *Wt,
                   const float *bias, int relu, void *Y, cudaStream_t stream, bool flip,
                   const void *mask) {
    if (dil < 1 || dil > kTcHalo || W < 1 || H < 1 || N < 1)
        return set_error(FHTDP_EINVAL, "conv3x3: dilation 1..8 and a non-empty image");
    auto kern = mask ? conv3x3_rows_kernel<false, true>
                : relu ? conv3x3_rows_kernel<true, false>
                       : conv3x3_rows_kernel<false, false>;
    // set on every call: the attribute belongs to the current device
    int st = cuda_status(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)kFwSmem),
                         "cudaFuncSetAttribute");
    if (st) return st;
    const long long rows = (long long)N * H * ((W + kTcM - 1) / kTcM);
    kern<<<row_grid(rows), kFwThreads, kFwSmem, stream>>>(
        (const __nv_bfloat16 *)X, N, H, W, dil, (const __nv_bfloat16 *)Wt, flip ? 1 : 0, bias,
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
