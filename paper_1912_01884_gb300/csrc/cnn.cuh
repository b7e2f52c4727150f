// Kernels of the learned window proposal (cnn.cu).
#pragma once

#include "common.cuh"

namespace fhtdp {

bool cnn_shape_ok(int H, int W, int dil);
int cnn_downsample4(const uint8_t *img, int N, int H, int W, void *out, cudaStream_t stream);
int cnn_conv3x3(const void *X, int cin, int N, int H, int W, int dil, const void *Wt,
                const float *bias, int relu, void *Y, cudaStream_t stream);
int cnn_relu_backward(const void *Y, void *dY, long long count, cudaStream_t stream);
int cnn_wgrad(const void *X, int cin, int N, int H, int W, int dil, const void *dZ, float *dW,
              float *db, cudaStream_t stream, float *part = nullptr);
// Scratch of a weight gradient that is summed in a fixed order: one row per
// CTA of the 288 x 32 weight and 32 bias sums.
constexpr int kWgradParts = 304, kWgradPart = 9 * 32 * 32 + 32;
// out[i] = part[0][i] + part[1][i] + ... (rows of `stride` floats), i < count.
int cnn_sum_parts(const float *part, int rows, int stride, int count, float *out,
                  cudaStream_t stream);
// One Adam step on several parameter tensors in one launch.
struct AdamTensor {
    float *p, *m, *v;
    const float *g;
    void *wb;   // bf16 copy, or null
    int count;
};
int cnn_adam_all(const AdamTensor *t, int tensors, float lr, float b1, float b2, float eps, int step,
                 cudaStream_t stream);
int cnn_band_head(const void *L, int N, int H, int W, int bands, const int32_t *labels,
                  float scale, void *dL, float *loss, int32_t *pred, cudaStream_t stream,
                  float *conf = nullptr);
int cnn_he_init(float *w, int rows, int cols, int zero_from, float std, unsigned long long seed,
                cudaStream_t stream);
int cnn_adam(float *p, float *m, float *v, const float *g, int count, float lr, float b1,
             float b2, float eps, int t, void *wb, cudaStream_t stream);
int cnn_to_bf16(const float *src, void *dst, int count, cudaStream_t stream);
// A chain of image rows: one column segment of kSegment pixels of one image and
// the rows of one residue modulo the dilation, whose row taps are neighbours in
// the chain.  The rows [g, end) of this CTA in the sequence of all chains' rows: image by
// image, segment by segment, residue by residue.  next() gives the piece of
// one chain: rows i .. i + L - 1 of the chain (y = rho + dil * i).
template <int kSegment>
struct RowRange {
    long long g, end;
    int H, dil, segs;
    int n, x0, rho, i, L;
    __device__ RowRange(int N, int H_, int W, int dil_)
        : H(H_), dil(dil_), segs((W + kSegment - 1) / kSegment) {
        const long long total = (long long)N * segs * H;
        g = total * blockIdx.x / gridDim.x;
        end = total * (blockIdx.x + 1) / gridDim.x;
    }
    __device__ bool next() {
        if (g >= end) return false;
        const long long u = g / H;
        int h = (int)(g - u * H);
        n = (int)(u / segs);
        x0 = (int)(u - (long long)n * segs) * kSegment;
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

// The 32-channel layers on tcgen05 (conv_tc.cu); cnn_tc_status reads (and
// with `clear` resets) their device status, synchronising.
int cnn_conv3x3_tc(const void *X, int N, int H, int W, int dil, const void *Wt,
                   const float *bias, int relu, void *Y, cudaStream_t stream, bool flip = false,
                   const void *mask = nullptr);
int cnn_wgrad_tc(const void *X, int N, int H, int W, int dil, const void *dZ, float *dW,
                 float *db, cudaStream_t stream, float *part = nullptr);
int cnn_tc_status(int clear);
int cnn_bin_windows(const int32_t *pred, int count, int n, int margin, int32_t *win,
                    cudaStream_t stream);

}  // namespace fhtdp
