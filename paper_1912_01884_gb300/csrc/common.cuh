// Shared definitions of the CUDA sources (not part of the public ABI).
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include "fhtdp.h"

namespace fhtdp {

// Sentinel of a dead DP state: no admissible polyline continues from it.
// It never takes part in an addition.
template <typename T>
struct Dead;
template <>
struct Dead<int32_t> {
    __host__ __device__ static constexpr int32_t value() { return INT32_MIN; }
};
template <>
struct Dead<float> {
    __device__ static float value() { return __int_as_float(0xff800000u); }
};

// Shape of one image's problem.
struct Shape {
    int h, w, k, n, W, D;  // D = 2n - 1 displacement values
    int log2n;
    // Vertex domain [0, vw) of the band chain and the read-back: w, or W when
    // vertices may lie in the zero padding right of the image (Sec. 2.2).
    int vw;
};

// The continuation window of every displacement: entry d + n - 1 holds the
// range [lo, hi] of next displacements e admissible after d.  The bend-angle
// windows of Sec. 2.3 (Fig. 5, Eqs. 6-7: |atan(e/n) - atan(d/n)| <= gamma)
// and the integer bend limit |e - d| <= B are both such tables.  Passed to
// kernels by value.
constexpr int kMaxD = 511;
struct WindowTable {
    int16_t lo[kMaxD], hi[kMaxD];
    int n;
};
// Fills *t for bands of n rows; false if gamma is negative or not finite.
bool make_angle_table(int n, double gamma, WindowTable *t);

// Largest half-width of the row smoothing (binomial weights up to C(24, 12)).
constexpr int kMaxGaussR = 12;

// Host helpers (api.cu).
int set_error(int code, const char *fmt, ...);
// Clears the calling thread's last error message (every entry point starts so).
void clear_error();
// Checks a launch and counts it (fhtdp_launch_count).
int launched(const char *what);
int cuda_status(cudaError_t err, const char *what);
bool make_shape(int h, int w, int k, Shape *out);
// cuTensorMapEncodeTiled through the runtime's driver entry point (no
// link-time dependency on the driver library); null if there is none.
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder();

// Kernels launched by the API layer.
//
// The Hough rows of an image (chain.cu): columns [0, wout) of [k][2][n] rows
// `opitch` values apart; tmp (the same size) for 256-row bands only.
template <typename In, typename Acc>
int launch_band_fht(const In *img, long long pitch, const Shape &s, int wout, Acc *hough, Acc *tmp,
                    int opitch, cudaStream_t stream);
// The last level of 256-row bands, from the level of their 128-row halves
// (fht_stages.cu).
template <typename Acc>
int launch_fht_last(const Acc *src, const Shape &s, int wout, Acc *dst, int opitch,
                    cudaStream_t stream);
// A point P = (xp, j*n) on the upper border of band j (j = k: the bottom
// border) that the polyline must pass (Subproblems 2-3): the DP treats every
// state whose vertex on that border is not xp as dead.
struct PointMask {
    int j, xp;
};
// The DP in place over Hough rows s.W apart, one launch per band, with the bend
// limit B or (t non-null) a window table.
template <typename Acc>
int launch_dp_window(Acc *hv, const Shape &s, int B, const WindowTable *t, cudaStream_t stream);
template <typename Acc>
int launch_backtrack(const Acc *V, const Shape &s, int B, const WindowTable *t, int32_t *x_out,
                     int32_t *d_out, Acc *score_out, cudaStream_t stream);

// The main problem (Sec. 2.3), step 1: row smoothing into a dense [h][w] image
// (int32 for integer images, float for float ones).
template <typename In, typename Acc>
int launch_gauss_rows(const In *img, int pitch, int h, int w, int r, Acc *out,
                      cudaStream_t stream);
size_t angle_workspace_bytes(const Shape &s);
size_t through_workspace_bytes(const Shape &s);
// The method with vertices anywhere in [0, W) (s.vw = W).
int detect_padded(const void *img, int dtype, int pitch, const Shape &s, int B, int32_t *x_out,
                  int32_t *d_out, void *score_out, void *ws, bool tight, cudaStream_t stream);
// Two different extreme polylines: the optimum and the best one whose top
// vertex is at least sep columns from the optimum's (outputs [2][...]).
int detect_two(const void *img, int dtype, int pitch, const Shape &s, int B, int sep,
               int32_t *x_out, int32_t *d_out, void *score_out, void *ws, bool tight,
               cudaStream_t stream);
// dst[x][y] = src[y][x] (Sec. 3, Fig. 7: mostly horizontal curves).
template <typename T>
int launch_transpose(const T *src, int h, int w, int pitch, T *dst, int dpitch,
                     cudaStream_t stream);

}  // namespace fhtdp
