// Passes over whole images beside the band FHT of chain.cu: the last dyadic
// level of 256-row bands, the row smoothing and the transpose.
//
// Sec. 2.1 (refs [10], [34]): the Hough image of a band is built bottom-up
// over sub-bands of 1, 2, 4, ..., n rows.  Merging the top half A and the
// bottom half B of a sub-band of m rows gives, for every shift s in [0, m),
//   out(x, s) = A(x, s>>1) + B(x +/- ceil(s/2), s>>1)      (columns mod W)
// with "+" for lines moving right and "-" for lines moving left.  The sum
// tree is therefore fixed (top half + bottom half at every level), which
// makes the float path reproducible bit for bit.
//
// Layout: [band][sign][row][x], x fastest; at the level of m-row sub-bands,
// row j*m + s holds shift s of sub-band j, so the last level (m = n, one
// sub-band) is the [k][2][n][W] Hough layout.
#include "common.cuh"

namespace fhtdp {
namespace {

__device__ __forceinline__ int wrap(int x, int W) {
    return x >= W ? x - W : (x < 0 ? x + W : x);
}

// The last level (sub-bands of n rows from those of n/2): a block writes one
// output row, columns [0, wout), reading columns modulo W.
template <typename Acc>
__global__ void fht_last_kernel(const Acc *__restrict__ src, Shape s, int wout,
                                Acc *__restrict__ dst, int pitch) {
    const int r = blockIdx.x;   // [band][sign][shift]
    const int sh = r % s.n, bs = r / s.n;
    const int move = sh - (sh >> 1);            // ceil(sh / 2)
    const Acc *ra = src + ((size_t)bs * s.n + (sh >> 1)) * pitch;
    const Acc *rb = ra + (size_t)(s.n >> 1) * pitch;
    Acc *out = dst + (size_t)r * pitch;
#pragma unroll 4
    for (int x = threadIdx.x; x < wout; x += blockDim.x)
        out[x] = ra[x] + rb[wrap(bs & 1 ? x - move : x + move, s.W)];
}

// Binomial weights C(2r, r + t), |t| <= r, by value.
struct GaussWeights {
    int32_t c[2 * kMaxGaussR + 1];
};

GaussWeights binomial_weights(int r) {
    GaussWeights g{};
    g.c[0] = 1;
    for (int j = 1; j <= 2 * r; ++j)   // row 2r of Pascal's triangle
        g.c[j] = (int32_t)((int64_t)g.c[j - 1] * (2 * r - j + 1) / j);
    return g;
}

// Main problem, step 1 (Sec. 2.3): every row convolved with the discrete
// Gaussian of half-width r, the unnormalised binomial weights (integer
// arithmetic for integer images, so the sums are exact; float images with each
// product weight * pixel rounded and added in the order t = -r .. r to an
// accumulator starting at 0); pixels outside the row count as zero: a zero
// product leaves an integer or float sum unchanged (a float sum that starts at
// +0 never holds -0).

// r <= 4: a thread makes four neighbouring outputs from the twelve pixels
// around them, read as three groups of four (through L1); bound by DRAM.
// 2048 x 2048 uint8, r = 2: one output a thread 23.5 us, this 7.3 us.
template <typename In, typename Acc, int R>
__global__ void __launch_bounds__(256) gauss_rows4_kernel(const In *__restrict__ img, int pitch,
                                                          int w, int quads, unsigned total,
                                                          bool aligned, bool wide, GaussWeights g,
                                                          Acc *__restrict__ out) {
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const unsigned y = i / quads;
    const int x = 4 * (int)(i - y * quads);
    const In *row = img + (size_t)y * pitch;
    Acc p[12];   // pixels x - 4 .. x + 7
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int c = x - 4 + 4 * k;
        if (aligned && c >= 0 && c + 4 <= w) {
            if constexpr (sizeof(In) == 1) {
                const uint32_t v = __ldg((const uint32_t *)(row + c));
#pragma unroll
                for (int e = 0; e < 4; ++e) p[4 * k + e] = (Acc)((v >> (8 * e)) & 255u);
            } else {
                struct alignas(16) Four {
                    In v[4];
                };
                const Four v = *(const Four *)(row + c);
#pragma unroll
                for (int e = 0; e < 4; ++e) p[4 * k + e] = (Acc)v.v[e];
            }
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                p[4 * k + e] = c + e >= 0 && c + e < w ? (Acc)row[c + e] : Acc(0);
        }
    }
    Acc o[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        Acc acc = 0;
#pragma unroll
        for (int t = 0; t <= 2 * R; ++t) acc += (Acc)g.c[t] * p[4 + e - R + t];
        o[e] = acc;
    }
    Acc *dst = out + (size_t)y * w + x;
    if (wide) {
        struct alignas(16) Four {
            Acc v[4];
        };
        *(Four *)dst = Four{{o[0], o[1], o[2], o[3]}};
    } else {
        for (int e = 0; e < 4 && x + e < w; ++e) dst[e] = o[e];
    }
}

constexpr int kGaussSeg = 1024;   // output columns per block (4 per thread)

// Any r: a block stages one row segment and its 2r-pixel halo in shared memory
// and writes kGaussSeg outputs of the dense [h][w] result.
template <typename In, typename Acc>
__global__ void gauss_rows_kernel(const In *__restrict__ img, int pitch, int w, int r,
                                  GaussWeights g, Acc *__restrict__ out) {
    __shared__ Acc seg[kGaussSeg + 2 * kMaxGaussR];
    const int y = blockIdx.x;
    const int x0 = blockIdx.y * kGaussSeg;
    const In *row = img + (size_t)y * pitch;
    for (int i = threadIdx.x; i < kGaussSeg + 2 * r; i += blockDim.x) {
        const int c = x0 - r + i;
        seg[i] = (c >= 0 && c < w) ? (Acc)row[c] : Acc(0);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kGaussSeg; i += blockDim.x) {
        const int x = x0 + i;
        if (x >= w) break;
        Acc acc = 0;
        for (int t = 0; t <= 2 * r; ++t) acc += (Acc)g.c[t] * seg[i + t];
        out[(size_t)y * w + x] = acc;
    }
}

}  // namespace

template <typename In, typename Acc>
int launch_gauss_rows(const In *img, int pitch, int h, int w, int r, Acc *out,
                      cudaStream_t stream) {
    const GaussWeights g = binomial_weights(r);
    const long long quads = (w + 3) / 4, total = quads * h;
    if (r <= 4 && total < (1LL << 31)) {
        const bool aligned = (uintptr_t)img % (4 * sizeof(In)) == 0 && pitch % 4 == 0;
        const bool wide = (uintptr_t)out % 16 == 0 && w % 4 == 0;
        auto kern = r == 0   ? gauss_rows4_kernel<In, Acc, 0>
                    : r == 1 ? gauss_rows4_kernel<In, Acc, 1>
                    : r == 2 ? gauss_rows4_kernel<In, Acc, 2>
                    : r == 3 ? gauss_rows4_kernel<In, Acc, 3>
                             : gauss_rows4_kernel<In, Acc, 4>;
        kern<<<(unsigned)((total + 255) / 256), 256, 0, stream>>>(
            img, pitch, w, (int)quads, (unsigned)total, aligned, wide, g, out);
        return launched("gauss_rows4_kernel");
    }
    dim3 grid((unsigned)h, (unsigned)((w + kGaussSeg - 1) / kGaussSeg));   // rows in x: h <= 2^20
    gauss_rows_kernel<In, Acc><<<grid, 256, 0, stream>>>(img, pitch, w, r, g, out);
    return launched("gauss_rows_kernel");
}

template int launch_gauss_rows<uint8_t, int32_t>(const uint8_t *, int, int, int, int, int32_t *,
                                                 cudaStream_t);
template int launch_gauss_rows<int32_t, int32_t>(const int32_t *, int, int, int, int, int32_t *,
                                                 cudaStream_t);
template int launch_gauss_rows<float, float>(const float *, int, int, int, int, float *,
                                             cudaStream_t);

template <typename Acc>
int launch_fht_last(const Acc *src, const Shape &s, int wout, Acc *dst, int opitch,
                    cudaStream_t stream) {
    fht_last_kernel<Acc><<<(unsigned)(s.k * 2 * s.n), 256, 0, stream>>>(src, s, wout, dst, opitch);
    return launched("fht_last_kernel");
}

template int launch_fht_last<int32_t>(const int32_t *, const Shape &, int, int32_t *, int,
                                      cudaStream_t);
template int launch_fht_last<float>(const float *, const Shape &, int, float *, int, cudaStream_t);

}  // namespace fhtdp

namespace fhtdp {
namespace {
// Mostly horizontal curves (Sec. 3, Fig. 7) are the mostly vertical curves of
// the transposed image: dst[x][y] = src[y][x], through a 32 x 32 shared tile
// so that both the reads and the writes are row segments.
template <typename T>
__global__ void transpose_kernel(const T *__restrict__ src, int h, int w, int pitch,
                                 T *__restrict__ dst, int dpitch) {
    __shared__ T tile[32][33];
    const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 32;
    for (int dy = threadIdx.y; dy < 32; dy += blockDim.y) {
        const int y = y0 + dy, x = x0 + threadIdx.x;
        if (y < h && x < w) tile[dy][threadIdx.x] = src[(size_t)y * pitch + x];
    }
    __syncthreads();
    for (int dx = threadIdx.y; dx < 32; dx += blockDim.y) {
        const int x = x0 + dx, y = y0 + threadIdx.x;
        if (x < w && y < h) dst[(size_t)x * dpitch + y] = tile[threadIdx.x][dx];
    }
}
// The uint8 transpose with 4-byte words: 64 x 64 byte tiles and 16 x 16
// threads; a thread loads one word of each of four tile rows and stores one
// word (four source rows of one column) of each of four output rows.  Needs
// both base addresses and both pitches 4-byte aligned; ragged edges go byte
// by byte.
__global__ void transpose_u8x4_kernel(const uint8_t *__restrict__ src, int h, int w, int pitch,
                                      uint8_t *__restrict__ dst, int dpitch) {
    __shared__ __align__(4) uint8_t tile[64][68];
    const int x0 = blockIdx.x * 64, y0 = blockIdx.y * 64;
    const int tx = threadIdx.x, ty = threadIdx.y;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int y = y0 + ty + 16 * i, x = x0 + 4 * tx;
        uint32_t v = 0;
        if (y < h) {
            const uint8_t *p = src + (size_t)y * pitch + x;
            if (x + 3 < w) {
                v = *(const uint32_t *)p;
            } else {
                for (int b = 0; b < 4; ++b)
                    if (x + b < w) v |= (uint32_t)p[b] << (8 * b);
            }
        }
        *(uint32_t *)&tile[ty + 16 * i][4 * tx] = v;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int c = ty + 16 * i, x = x0 + c, y = y0 + 4 * tx;
        if (x >= w || y >= h) continue;
        const uint32_t v = (uint32_t)tile[4 * tx][c] | (uint32_t)tile[4 * tx + 1][c] << 8 |
                           (uint32_t)tile[4 * tx + 2][c] << 16 |
                           (uint32_t)tile[4 * tx + 3][c] << 24;
        uint8_t *q = dst + (size_t)x * dpitch + y;
        if (y + 3 < h) {
            *(uint32_t *)q = v;
        } else {
            for (int b = 0; b < 4 && y + b < h; ++b) q[b] = (uint8_t)(v >> (8 * b));
        }
    }
}
}  // namespace

template <typename T>
int launch_transpose(const T *src, int h, int w, int pitch, T *dst, int dpitch,
                     cudaStream_t stream) {
    if (sizeof(T) == 1 && ((uintptr_t)src & 3) == 0 && ((uintptr_t)dst & 3) == 0 &&
        pitch % 4 == 0 && dpitch % 4 == 0) {
        dim3 grid((unsigned)((w + 63) / 64), (unsigned)((h + 63) / 64));   // h, w <= 2^20
        transpose_u8x4_kernel<<<grid, dim3(16, 16), 0, stream>>>(
            (const uint8_t *)src, h, w, pitch, (uint8_t *)dst, dpitch);
        return launched("transpose_u8x4_kernel");
    }
    dim3 grid((unsigned)((w + 31) / 32), (unsigned)((h + 31) / 32));   // h, w <= 2^20
    transpose_kernel<T><<<grid, dim3(32, 8), 0, stream>>>(src, h, w, pitch, dst, dpitch);
    return launched("transpose_kernel");
}

template int launch_transpose<uint8_t>(const uint8_t *, int, int, int, uint8_t *, int,
                                       cudaStream_t);
template int launch_transpose<int32_t>(const int32_t *, int, int, int, int32_t *, int,
                                       cudaStream_t);
template int launch_transpose<float>(const float *, int, int, int, float *, int, cudaStream_t);

}  // namespace fhtdp
