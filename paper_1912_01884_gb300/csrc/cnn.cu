// The learned shift-window proposal: a 4-layer, 32-channel CNN on a 4x
// downsampled image that predicts, for every band, which of 32 displacement
// bins the best polyline's link falls in; the DP then searches only a window
// around it (pruned DP, with the full DP as fallback).  The paper has no
// counterpart: it is an addition in front of the exact method.
//
// Layout: activations NHWC bf16 ([N][H][W][C], C = 32; the input has C = 1),
// weights bf16 [tap][ci][co] with tap = ky*3 + kx (layer 1: [16][32], taps
// 9..15 zero), FP32 master weights and FP32 accumulation.  The 3x3 dilated
// convolutions ("same" zero padding) of 32 channels run on tcgen05.mma
// (conv_tc.cu).  The single-channel first layer (9 products a value) is bound
// by its 64 bytes a pixel of output: one warp MMA step in registers forward,
// plain FP32 multiply-adds for its weight gradient.
#include <cuda_bf16.h>

#include <algorithm>

#include "cnn.cuh"

namespace fhtdp {
namespace {

constexpr int kC = 32;        // channels
constexpr int kSeg = 64;      // row widths are multiples of it
constexpr int kMaxDil = 8;

// ---------------------------------------------------------------------------
// Eight bf16 values at p as four words; `wide` when p is 16-byte aligned.
__device__ __forceinline__ uint4 ld8(const __nv_bfloat16 *p, bool wide) {
    if (wide) return __ldg((const uint4 *)p);
    const unsigned short *q = (const unsigned short *)p;
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = __ldg(q + 2 * i) | (uint32_t)__ldg(q + 2 * i + 1) << 16;
    return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ void st8(__nv_bfloat16 *p, const uint32_t (&w)[4], bool wide) {
    if (wide) {
        *(uint4 *)p = make_uint4(w[0], w[1], w[2], w[3]);
    } else {
        unsigned short *q = (unsigned short *)p;
#pragma unroll
        for (int i = 0; i < 8; ++i) q[i] = (unsigned short)(i & 1 ? w[i / 2] >> 16 : w[i / 2]);
    }
}

// 4x4 mean pool of uint8 images, scaled to [0, 1]: [N][H][W] -> [N][H/4][W/4].
// A thread makes V = 4 neighbouring values from four 16-byte loads (rows
// 16-byte aligned, W a multiple of 16), or V = 1 from four 4-byte loads.
template <int V>
__global__ void downsample4_kernel(const uint8_t *__restrict__ img, int H, int W, long long total,
                                   __nv_bfloat16 *__restrict__ out) {
    const int Wv = W / (4 * V);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const long long row = i / Wv;   // output row over all images
        const int xv = (int)(i - row * Wv);
        const uint8_t *p = img + row * 4 * W + (size_t)xv * 4 * V;
        unsigned s[V] = {};
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            uint32_t v[V];
            if constexpr (V == 4) {
                const uint4 q = __ldg((const uint4 *)(p + (size_t)r * W));
                v[0] = q.x;
                v[1] = q.y;
                v[2] = q.z;
                v[3] = q.w;
            } else {
                v[0] = __ldg((const uint32_t *)(p + (size_t)r * W));
            }
#pragma unroll
            for (int k = 0; k < V; ++k) s[k] = __dp4a(v[k], 0x01010101u, s[k]);
        }
        __nv_bfloat16 *dst = out + row * (W / 4) + (size_t)xv * V;
        if constexpr (V == 4) {
            __nv_bfloat162 o[2];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                (k & 1 ? o[k / 2].y : o[k / 2].x) =
                    __float2bfloat16((float)s[k] * (1.0f / (16.0f * 255.0f)));
            *(uint2 *)dst = make_uint2(*(const uint32_t *)&o[0], *(const uint32_t *)&o[1]);
        } else {
            dst[0] = __float2bfloat16((float)s[0] * (1.0f / (16.0f * 255.0f)));
        }
    }
}

// ---------------------------------------------------------------------------
// First layer: Y(p)[co] = act(sum over the nine taps of x(p + off) * w[tap][co]
// + bias[co]), one input channel.  A warp takes 16 pixels of a row and one
// m16n8k16 step per eight output channels: A = pixels x taps (taps 9..15 are
// zero), B = the weights, kept in registers.  Column 2 t + e of step j stands
// for channel 8 t + 2 j + e, so that a thread ends up with eight consecutive
// channels of a pixel and a warp stores 512 contiguous bytes.
template <bool kRelu>
__global__ void __launch_bounds__(256) conv3x3_first_kernel(
    const __nv_bfloat16 *__restrict__ X, int H, int W, int dil, unsigned tiles,
    const __nv_bfloat16 *__restrict__ Wt, const float *__restrict__ bias,
    __nv_bfloat16 *__restrict__ Y, bool wide) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const unsigned short *xs = (const unsigned short *)X, *ws = (const unsigned short *)Wt;
    uint32_t b0[4], b1[4];
    float bs[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int co = 8 * (g >> 1) + 2 * j + (g & 1);
        b0[j] = ws[2 * t * kC + co] | (uint32_t)ws[(2 * t + 1) * kC + co] << 16;
        b1[j] = t == 0 ? ws[8 * kC + co] : 0;
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) bs[c] = bias ? bias[8 * t + c] : 0.0f;
    // the thread's taps: 2 t, 2 t + 1 and (t = 0) 8
    const int dy[3] = {(2 * t / 3 - 1) * dil, ((2 * t + 1) / 3 - 1) * dil, dil};
    const int dx[3] = {(2 * t % 3 - 1) * dil, ((2 * t + 1) % 3 - 1) * dil, dil};
    const unsigned per_row = W / 16, step = gridDim.x * (blockDim.x / 32);
    for (unsigned u = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); u < tiles; u += step) {
        const unsigned r = u / per_row;   // row over all images
        const long long row = r;
        const int x0 = (int)(u - r * per_row) * 16, y = (int)(r % (unsigned)H);
        uint32_t a[4];
#pragma unroll
        for (int hi = 0; hi < 2; ++hi) {   // pixels g and g + 8
            uint32_t v[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int yy = y + dy[k], xx = x0 + g + 8 * hi + dx[k];
                v[k] = (k < 2 || t == 0) && yy >= 0 && yy < H && xx >= 0 && xx < W
                           ? __ldg(xs + (row + dy[k]) * W + xx)
                           : 0;
            }
            a[hi] = v[0] | v[1] << 16;
            a[2 + hi] = v[2];
        }
        uint32_t lo[4], hi[4];   // channels 8 t + 2 j, + 1 of pixels g and g + 8
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float c[4];
            asm volatile(
                "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, "
                "{%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
                : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
                : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0[j]), "r"(b1[j]), "f"(0.0f));
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                c[k] += bs[2 * j + (k & 1)];
                if (kRelu) c[k] = fmaxf(c[k], 0.0f);
            }
            const __nv_bfloat162 l = __floats2bfloat162_rn(c[0], c[1]);
            const __nv_bfloat162 h = __floats2bfloat162_rn(c[2], c[3]);
            lo[j] = *(const uint32_t *)&l;
            hi[j] = *(const uint32_t *)&h;
        }
        __nv_bfloat16 *dst = Y + ((size_t)row * W + x0 + g) * kC + 8 * t;
        st8(dst, lo, wide);
        st8(dst + 8 * kC, hi, wide);
    }
}

// ---------------------------------------------------------------------------
// dZ = dY * (Y > 0) in place (the ReLU of a layer, from its output).
__global__ void relu_backward_kernel(const __nv_bfloat16 *__restrict__ Y,
                                     __nv_bfloat16 *__restrict__ dY, long long count) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
         i += (long long)gridDim.x * blockDim.x)
        if (!(__bfloat162float(Y[i]) > 0.0f)) dY[i] = __float2bfloat16(0.0f);
}

// ---------------------------------------------------------------------------
// Weight and bias gradients of the first layer: dW[tap][co] = sum over pixels
// p of x(p + off(tap)) * dZ(p)[co], db[co] = sum of dZ(p)[co].  A thread takes
// eight channels of one pixel of a 64-pixel segment and goes down a chain of
// rows: its nine inputs are three new ones a row and six kept, its 72 + 8 sums
// stay in registers.  Bound by the loads' latency at 16 warps an SM, so three
// rows of dZ are in flight into a ring in shared memory (a slot belongs to one
// thread: no barrier) and one row of inputs, which L2 holds; at the end the 64
// pixels' sums are added in shared memory in a fixed order.  32 images of
// 256 x 256: WMMA tiles with a copy of the inputs per tap 353 us, one row in
// flight 95 us, this 84 us.
constexpr int kW1Ring = 4;    // slots: a row of dZ read, three in flight
constexpr int kW1Sums = 80;   // 9 taps and the bias, eight channels
constexpr int kW1Part = 17 * kC;   // a row of `part`: 16 tap rows (9..15 zero) and the bias
__global__ void __launch_bounds__(256, 2) wgrad_first_kernel(
    const __nv_bfloat16 *__restrict__ X, int N, int H, int W, int dil,
    const __nv_bfloat16 *__restrict__ dZ, float *__restrict__ dW, float *__restrict__ db,
    float *__restrict__ part, bool wide) {
    __shared__ float red[8][4][kW1Sums + 1];
    __shared__ uint4 ring[kW1Ring][256];
    const int c = threadIdx.x & 3, px = threadIdx.x >> 2;
    const unsigned short *xs = (const unsigned short *)X;
    float acc[kW1Sums];
#pragma unroll
    for (int k = 0; k < kW1Sums; ++k) acc[k] = 0.0f;
    RowRange<kSeg> rr(N, H, W, dil);
    while (rr.next()) {
        const int x = rr.x0 + px;
        const bool in0 = x >= dil, in2 = x + dil < W;
        // the three inputs of chain row j at this pixel (zero outside the image)
        auto inputs = [&](int j, uint32_t (&v)[3]) {
            const int y = rr.row(j);
            const unsigned short *p = xs + ((size_t)rr.n * H + (y >= 0 && y < H ? y : 0)) * W + x;
            const bool in = y >= 0 && y < H;
            v[0] = in && in0 ? __ldg(p - dil) : 0;
            v[1] = in ? __ldg(p) : 0;
            v[2] = in && in2 ? __ldg(p + dil) : 0;
        };
        // dZ of chain row i + o into its slot of this thread's ring
        auto dzs = [&](int o) {
            if (o < rr.L) {
                const __nv_bfloat16 *p =
                    dZ + (((size_t)rr.n * H + rr.row(rr.i + o)) * W + x) * kC + 8 * c;
                uint4 *slot = &ring[o % kW1Ring][threadIdx.x];
                if (wide)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                     (uint32_t)__cvta_generic_to_shared(slot)),
                                 "l"(p)
                                 : "memory");
                else
                    *slot = ld8(p, false);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
#pragma unroll
        for (int o = 0; o < kW1Ring - 1; ++o) dzs(o);
        uint32_t v[3];
        float xf[9];   // rows above, at and below
        auto keep = [&](int at) {
#pragma unroll
            for (int k = 0; k < 3; ++k) xf[3 * at + k] = __uint_as_float(v[k] << 16);
        };
        inputs(rr.i - 1, v);
        keep(1);
        inputs(rr.i, v);
        keep(2);
        inputs(rr.i + 1, v);
        for (int o = 0; o < rr.L; ++o) {
#pragma unroll
            for (int k = 0; k < 6; ++k) xf[k] = xf[k + 3];
            keep(2);
            if (o + 1 < rr.L) inputs(rr.i + o + 2, v);
            asm volatile("cp.async.wait_group %0;" ::"n"(kW1Ring - 2) : "memory");
            const uint4 z = ring[o % kW1Ring][threadIdx.x];
            dzs(o + kW1Ring - 1);   // into the slot that the row before was read from
            const uint32_t zw[4] = {z.x, z.y, z.z, z.w};
            float f[8];
#pragma unroll
            for (int e = 0; e < 8; ++e)
                f[e] = __uint_as_float(e & 1 ? zw[e / 2] & 0xffff0000u : zw[e / 2] << 16);
#pragma unroll
            for (int k = 0; k < 9; ++k)
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[8 * k + e] = __fmaf_rn(xf[k], f[e], acc[8 * k + e]);
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[72 + e] += f[e];
        }
    }
#pragma unroll
    for (int k = 0; k < kW1Sums; ++k) {
        float v = acc[k];
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) < 4) red[threadIdx.x >> 5][c][k] = v;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kW1Part; i += blockDim.x) {
        const int row = i / kC, co = i % kC, k = row < 9 ? row : 9;   // tap, or 9: the bias
        float v = 0.0f;
        if (row < 9 || row == 16)
            for (int w = 0; w < 8; ++w) v += red[w][co >> 3][8 * k + (co & 7)];
        if (part)
            part[(size_t)blockIdx.x * kW1Part + i] = v;
        else if (row < 9)
            atomicAdd(dW + i, v);
        else if (row == 16 && db)
            atomicAdd(db + co, v);
    }
}

// out[i] = sum of part[r][i] over the rows r in a fixed order: 32 consecutive
// values a block, 32 rows at a time.
__global__ void __launch_bounds__(1024) sum_parts_kernel(const float *__restrict__ part, int rows,
                                                         int stride, int count,
                                                         float *__restrict__ out) {
    __shared__ float red[32][33];
    const int lane = threadIdx.x & 31, i = blockIdx.x * 32 + lane, w = threadIdx.x >> 5;
    float v = 0.0f;
    if (i < count) {
#pragma unroll 10
        for (int r = w; r < rows; r += 32) v += part[(size_t)r * stride + i];
    }
    red[w][lane] = v;
    __syncthreads();
    v = red[lane][w];   // value blockIdx.x * 32 + w
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0 && blockIdx.x * 32 + w < count) out[blockIdx.x * 32 + w] = v;
}

// ---------------------------------------------------------------------------
// Band head: for image n and band b (rows [b*rpb, (b+1)*rpb) of the low-res
// logits), pooled[c] = log sum_{rows, cols} exp(logit[c]) (a smooth maximum
// over the band), the softmax cross-entropy of the 32 pooled logits against
// the label bin, its gradient dlogit = (softmax - onehot)[c] *
// exp(logit - pooled[c]) * scale, and the predicted bin.
// The sums run as eight chains a channel (position modulo 8, one warp each),
// a value at a time without branches, the next values' loads in flight.  The
// gradient pass takes 16 bytes a thread; the band comes from L2 then.
__global__ void __launch_bounds__(256) band_head_kernel(const __nv_bfloat16 *__restrict__ L,
                                                        int H, int W, int bands,
                                                        const int32_t *__restrict__ labels,
                                                        float scale,
                                                        __nv_bfloat16 *__restrict__ dL,
                                                        float *__restrict__ loss,
                                                        int32_t *__restrict__ pred,
                                                        float *__restrict__ conf, bool wide) {
    __shared__ float smax[8][kC], ssum[8][kC], pooled[kC], dpool[kC];
    const int n = blockIdx.x / bands, b = blockIdx.x % bands;
    const int rpb = H / bands;
    const int positions = rpb * W;
    const __nv_bfloat16 *band = L + ((size_t)n * H + (size_t)b * rpb) * W * kC;
    {
        const int c = threadIdx.x & 31, part = threadIdx.x >> 5;
        const unsigned short *src = (const unsigned short *)band + c;
        float m = -INFINITY, s = 0.0f;
        auto take = [&](unsigned short bits) {
            const float v = __uint_as_float((uint32_t)bits << 16);
            const bool up = v > m;
            const float e = __expf(up ? m - v : v - m);
            s = up ? s * e + 1.0f : s + e;
            m = up ? v : m;
        };
        constexpr int kB = 16;
        int p = part;
        unsigned short q[kB];
        auto fetch = [&](int from) {
#pragma unroll
            for (int k = 0; k < kB; ++k) q[k] = __ldg(src + (size_t)(from + 8 * k) * kC);
        };
        if (p + 8 * (kB - 1) < positions) fetch(p);
        for (; p + 8 * (kB - 1) < positions; p += 8 * kB) {
            unsigned short cur[kB];
#pragma unroll
            for (int k = 0; k < kB; ++k) cur[k] = q[k];
            if (p + 8 * (2 * kB - 1) < positions) fetch(p + 8 * kB);
#pragma unroll
            for (int k = 0; k < kB; ++k) take(cur[k]);
        }
        for (; p < positions; p += 8) take(__ldg(src + (size_t)p * kC));
        smax[part][c] = m;
        ssum[part][c] = s;
    }
    __syncthreads();
    if (threadIdx.x < kC) {
        const int c = threadIdx.x;
        float M = -INFINITY;
        for (int p = 0; p < 8; ++p) M = fmaxf(M, smax[p][c]);
        float S = 0.0f;
        for (int p = 0; p < 8; ++p) S += ssum[p][c] * __expf(smax[p][c] - M);
        pooled[c] = M + __logf(S);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float M = -INFINITY;
        int arg = 0;
        for (int k = 0; k < kC; ++k)
            if (pooled[k] > M) {
                M = pooled[k];
                arg = k;
            }
        float S = 0.0f;
        for (int k = 0; k < kC; ++k) S += __expf(pooled[k] - M);
        const float lse = M + __logf(S);
        const int lab = labels ? labels[n * bands + b] : -1;
        for (int k = 0; k < kC; ++k) dpool[k] = __expf(pooled[k] - lse) - (k == lab ? 1.0f : 0.0f);
        if (loss && lab >= 0) atomicAdd(loss, (lse - pooled[lab]) * scale);
        if (pred) pred[n * bands + b] = arg;
        if (conf) conf[n * bands + b] = __expf(M - lse);   // softmax probability of the argmax
    }
    __syncthreads();
    if (!dL) return;
    const int c8 = (threadIdx.x & 3) * 8;
    const __nv_bfloat16 *base = band + c8;
    __nv_bfloat16 *dbase = dL + (band - L) + c8;
    float pc[8], g[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        pc[e] = pooled[c8 + e];
        g[e] = dpool[c8 + e] * scale;
    }
#pragma unroll 4
    for (int p = threadIdx.x >> 2; p < positions; p += 64) {
        const uint4 q = ld8(base + (size_t)p * kC, wide);
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e)
            v[e] = __uint_as_float(e & 1 ? w[e / 2] & 0xffff0000u : w[e / 2] << 16);
        uint32_t o[4];
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(g[e] * __expf(v[e] - pc[e]),
                                                           g[e + 1] * __expf(v[e + 1] - pc[e + 1]));
            o[e / 2] = *(const uint32_t *)&h;
        }
        st8(dbase + (size_t)p * kC, o, wide);
    }
}

// ---------------------------------------------------------------------------
// Adam on FP32 master parameters; refreshes the bf16 copy used by the
// forward pass (when `wb` is given).
__global__ void adam_kernel(float *__restrict__ p, float *__restrict__ m, float *__restrict__ v,
                            const float *__restrict__ g, int count, float lr, float b1, float b2,
                            float eps, float c1, float c2, __nv_bfloat16 *__restrict__ wb) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float pi = p[i] - lr * (mi * c1) / (sqrtf(vi * c2) + eps);
        p[i] = pi;
        if (wb) wb[i] = __float2bfloat16(pi);
    }
}

// The same step on up to eight tensors, one block row each.
struct AdamTensors {
    AdamTensor t[8];
};
__global__ void adam_all_kernel(const __grid_constant__ AdamTensors a, float lr, float b1, float b2,
                                float eps, float c1, float c2) {
    const AdamTensor &t = a.t[blockIdx.y];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < t.count; i += gridDim.x * blockDim.x) {
        const float gi = t.g[i];
        const float mi = b1 * t.m[i] + (1.0f - b1) * gi;
        const float vi = b2 * t.v[i] + (1.0f - b2) * gi * gi;
        t.m[i] = mi;
        t.v[i] = vi;
        const float pi = t.p[i] - lr * (mi * c1) / (sqrtf(vi * c2) + eps);
        t.p[i] = pi;
        if (t.wb) ((__nv_bfloat16 *)t.wb)[i] = __float2bfloat16(pi);
    }
}

__global__ void to_bf16_kernel(const float *__restrict__ src, __nv_bfloat16 *__restrict__ dst,
                               int count) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x)
        dst[i] = __float2bfloat16(src[i]);
}

// Displacement windows from the predicted bins: bin c covers d + 64 in
// [4c, 4c + 3]; the window is those 4 values with `margin` more on each side,
// clipped to [-(n-1), n-1].
__global__ void bin_windows_kernel(const int32_t *__restrict__ pred, int count, int n, int margin,
                                   int32_t *__restrict__ win) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        const int lo = 4 * pred[i] - 64 - margin, hi = 4 * pred[i] - 61 + margin;
        win[2 * i] = lo < -(n - 1) ? -(n - 1) : lo;
        win[2 * i + 1] = hi > n - 1 ? n - 1 : hi;
    }
}

// He-normal initial weights (standard deviation sqrt(2 / fan_in)) from a
// counter-based SplitMix64 stream (Steele, Lea, Flood, OOPSLA 2014) and the
// Box-Muller transform; zero where `zero_from` <= row (padding taps).
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__global__ void he_init_kernel(float *__restrict__ w, int rows, int cols, int zero_from, float std,
                               unsigned long long seed) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < rows * cols;
         i += gridDim.x * blockDim.x) {
        const unsigned long long r1 = splitmix64(seed ^ (2ull * (unsigned long long)i));
        const unsigned long long r2 = splitmix64(seed ^ (2ull * (unsigned long long)i + 1ull));
        const float u1 = ((float)(r1 >> 40) + 0.5f) * (1.0f / 16777216.0f);
        const float u2 = (float)(r2 >> 40) * (1.0f / 16777216.0f);
        const float z = sqrtf(-2.0f * logf(u1)) * cosf(6.283185307179586f * u2);
        w[i] = (i / cols) >= zero_from ? 0.0f : std * z;
    }
}

int grid_1d(long long count, int block) {
    long long g = (count + block - 1) / block;
    return (int)(g < 1 ? 1 : (g > 152 * 32 ? 152 * 32 : g));
}

}  // namespace

bool cnn_shape_ok(int H, int W, int dil) {
    return H >= 1 && W >= kSeg && W % kSeg == 0 && dil >= 1 && dil <= kMaxDil;
}

int cnn_downsample4(const uint8_t *img, int N, int H, int W, void *out, cudaStream_t stream) {
    const bool wide = W % 16 == 0 && (uintptr_t)img % 16 == 0 && (uintptr_t)out % 8 == 0;
    const long long total = (long long)N * (H / 4) * (W / (wide ? 16 : 4));
    if (wide)
        downsample4_kernel<4><<<grid_1d(total, 256), 256, 0, stream>>>(img, H, W, total,
                                                                     (__nv_bfloat16 *)out);
    else
        downsample4_kernel<1><<<grid_1d(total, 256), 256, 0, stream>>>(img, H, W, total,
                                                                     (__nv_bfloat16 *)out);
    return launched("downsample4_kernel");
}

int cnn_conv3x3(const void *X, int cin, int N, int H, int W, int dil, const void *Wt,
                const float *bias, int relu, void *Y, cudaStream_t stream) {
    if (cin == kC) return cnn_conv3x3_tc(X, N, H, W, dil, Wt, bias, relu, Y, stream);
    // (a GPU's memory holds fewer than 2^31 tiles' outputs of 1 KB)
    const long long tiles = (long long)N * H * (W / 16);
    const int grid = (int)std::min<long long>((tiles + 7) / 8, 152 * 8);
    auto kern = relu ? conv3x3_first_kernel<true> : conv3x3_first_kernel<false>;
    kern<<<grid, 256, 0, stream>>>((const __nv_bfloat16 *)X, H, W, dil, (unsigned)tiles,
                                   (const __nv_bfloat16 *)Wt, bias, (__nv_bfloat16 *)Y,
                                   (uintptr_t)Y % 16 == 0);
    return launched("conv3x3_first_kernel");
}

int cnn_relu_backward(const void *Y, void *dY, long long count, cudaStream_t stream) {
    relu_backward_kernel<<<grid_1d(count, 256), 256, 0, stream>>>(
        (const __nv_bfloat16 *)Y, (__nv_bfloat16 *)dY, count);
    return launched("relu_backward_kernel");
}

int cnn_wgrad(const void *X, int cin, int N, int H, int W, int dil, const void *dZ, float *dW,
              float *db, cudaStream_t stream, float *part) {
    if (cin == kC) return cnn_wgrad_tc(X, N, H, W, dil, dZ, dW, db, stream, part);
    const int grid = (int)std::min<long long>((long long)N * H * (W / kSeg), kWgradParts);
    wgrad_first_kernel<<<grid, 256, 0, stream>>>((const __nv_bfloat16 *)X, N, H, W, dil,
                                                 (const __nv_bfloat16 *)dZ, dW, db, part,
                                                 (uintptr_t)dZ % 16 == 0);
    int st = launched("wgrad_first_kernel");
    if (!st && part) st = cnn_sum_parts(part, grid, kW1Part, kW1Part, dW, stream);
    return st;
}

int cnn_sum_parts(const float *part, int rows, int stride, int count, float *out,
                  cudaStream_t stream) {
    sum_parts_kernel<<<(count + 31) / 32, 1024, 0, stream>>>(part, rows, stride, count, out);
    return launched("sum_parts_kernel");
}

int cnn_band_head(const void *L, int N, int H, int W, int bands, const int32_t *labels,
                  float scale, void *dL, float *loss, int32_t *pred, cudaStream_t stream,
                  float *conf) {
    const bool wide = ((uintptr_t)L | (uintptr_t)dL) % 16 == 0;
    band_head_kernel<<<N * bands, 256, 0, stream>>>((const __nv_bfloat16 *)L, H, W, bands, labels,
                                                     scale, (__nv_bfloat16 *)dL, loss, pred, conf,
                                                     wide);
    return launched("band_head_kernel");
}

int cnn_adam(float *p, float *m, float *v, const float *g, int count, float lr, float b1,
             float b2, float eps, int t, void *wb, cudaStream_t stream) {
    const float c1 = 1.0f / (1.0f - powf(b1, (float)t)), c2 = 1.0f / (1.0f - powf(b2, (float)t));
    adam_kernel<<<grid_1d(count, 256), 256, 0, stream>>>(p, m, v, g, count, lr, b1, b2, eps, c1,
                                                        c2, (__nv_bfloat16 *)wb);
    return launched("adam_kernel");
}

int cnn_adam_all(const AdamTensor *t, int tensors, float lr, float b1, float b2, float eps, int step,
                 cudaStream_t stream) {
    const float c1 = 1.0f / (1.0f - powf(b1, (float)step));
    const float c2 = 1.0f / (1.0f - powf(b2, (float)step));
    AdamTensors a{};
    int most = 1;
    if (tensors < 1 || tensors > 8) return set_error(FHTDP_EINVAL, "adam: 1..8 tensors");
    for (int i = 0; i < tensors; ++i) {
        a.t[i] = t[i];
        most = std::max(most, t[i].count);
    }
    adam_all_kernel<<<dim3(grid_1d(most, 256), tensors), 256, 0, stream>>>(a, lr, b1, b2, eps, c1,
                                                                           c2);
    return launched("adam_all_kernel");
}

int cnn_bin_windows(const int32_t *pred, int count, int n, int margin, int32_t *win,
                    cudaStream_t stream) {
    bin_windows_kernel<<<grid_1d(count, 256), 256, 0, stream>>>(pred, count, n, margin, win);
    return launched("bin_windows_kernel");
}

int cnn_he_init(float *w, int rows, int cols, int zero_from, float std, unsigned long long seed,
                cudaStream_t stream) {
    he_init_kernel<<<grid_1d((long long)rows * cols, 256), 256, 0, stream>>>(w, rows, cols,
                                                                           zero_from, std, seed);
    return launched("he_init_kernel");
}

int cnn_to_bf16(const float *src, void *dst, int count, cudaStream_t stream) {
    to_bf16_kernel<<<grid_1d(count, 256), 256, 0, stream>>>(src, (__nv_bfloat16 *)dst, count);
    return launched("to_bf16_kernel");
}

}  // namespace fhtdp
