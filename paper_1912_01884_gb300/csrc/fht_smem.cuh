// Band FHT of one column tile in shared memory (Sec. 2.1), for the kernels
// that store the Hough rows (chain.cu).
//
// F holds m rows of `pitch` words; after the level of 2^l-row sub-bands, row
// j * 2^l + brev(s) holds shift s of sub-band j.  The first two levels are done
// in registers straight from the image (sub-bands of at least 4 rows, chain.cu);
// the rest in shared memory, two levels a pass where possible, in place: a warp
// owns a set of rows and sweeps their columns left to right, and column u is
// only read by columns <= u.  The last level hands its values to `out(s, u,
// four words)` instead of storing them.  Every value is (top half) + (bottom
// half), level by level, so float sums are those of the recursion.
//
// uint8 images keep both slope halves in one 32-bit word, the "+" value of
// column u in the low 16 bits and the "-" value of the mirrored strip (column
// T - 1 - u) in the high ones: sums of at most 128 pixels fit, and one addition
// serves both.
#pragma once

#include "common.cuh"

namespace fhtdp {

template <typename W>
__device__ __forceinline__ W word_from(uint32_t b);
template <>
__device__ __forceinline__ uint32_t word_from<uint32_t>(uint32_t b) { return b; }
template <>
__device__ __forceinline__ int32_t word_from<int32_t>(uint32_t b) { return (int32_t)b; }
template <>
__device__ __forceinline__ float word_from<float>(uint32_t b) { return __uint_as_float(b); }
__device__ __forceinline__ uint32_t word_bits(uint32_t v) { return v; }
__device__ __forceinline__ uint32_t word_bits(int32_t v) { return (uint32_t)v; }
__device__ __forceinline__ uint32_t word_bits(float v) { return __float_as_uint(v); }

__device__ __forceinline__ int bit_reverse(int r, int bits) {
    return bits ? (int)(__brev((unsigned)r) >> (32 - bits)) : 0;
}

template <typename W>
__device__ __forceinline__ void unpack4(const uint4 &q, W *v) {
    v[0] = word_from<W>(q.x);
    v[1] = word_from<W>(q.y);
    v[2] = word_from<W>(q.z);
    v[3] = word_from<W>(q.w);
}
template <typename W>
__device__ __forceinline__ uint4 pack4(const W *v) {
    return make_uint4(word_bits(v[0]), word_bits(v[1]), word_bits(v[2]), word_bits(v[3]));
}

// One level: rows A (shift q of the upper half) and B (the lower half) give
// shifts 2q and 2q + 1.  Q is q modulo 4.
template <typename W, int Q>
__device__ __forceinline__ void fht_pair(const uint4 &a4, const uint4 *b4, uint4 *o) {
    W a[4], b[8], x[4], y[4];
    unpack4(a4, a);
    unpack4(b4[0], b);
    unpack4(b4[1], b + 4);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        x[t] = a[t] + b[Q + t];
        y[t] = a[t] + b[Q + t + 1];
    }
    o[0] = pack4(x);
    o[1] = pack4(y);
}

// Two levels: rows J0..J3 at shift q give shifts 4q .. 4q + 3,
//   [J0(u) + J1(u + q + (r >> 1))] + [J2(u + 2q + ((r + 1) >> 1)) + J3(u + 3q + r)],
// r = 0..3.  Q is q modulo 4.
template <typename W, int Q>
__device__ __forceinline__ void fht_quad(const uint4 &j0, const uint4 *j1, const uint4 *j2,
                                         const uint4 *j3, uint4 *o) {
    constexpr int O2 = (2 * Q) & 3, O3 = (3 * Q) & 3;
    W a[4], b1[8], b2[8], b3[12], r[4][4];
    unpack4(j0, a);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        unpack4(j1[k], b1 + 4 * k);
        unpack4(j2[k], b2 + 4 * k);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) unpack4(j3[k], b3 + 4 * k);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const W a0 = a[t] + b1[Q + t], a1 = a[t] + b1[Q + t + 1];
        r[0][t] = a0 + (b2[O2 + t] + b3[O3 + t]);
        r[1][t] = a0 + (b2[O2 + t + 1] + b3[O3 + t + 1]);
        r[2][t] = a1 + (b2[O2 + t + 1] + b3[O3 + t + 2]);
        r[3][t] = a1 + (b2[O2 + t + 2] + b3[O3 + t + 3]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) o[k] = pack4(r[k]);
}

// The last level, l (sub-bands of 2^(l-1) rows merged), into `out`.  T output
// columns, m rows, NT threads; no barrier.
template <typename W, int NT, typename Out>
__device__ void fht_level(const W *F, int pitch, int m, int l, int T, Out out) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int half = 1 << (l - 1), width = T + m - 2 * half;
    for (int p = warp; p < m / 2; p += NT / 32) {
        const int j = p >> (l - 1), r = p & (half - 1);
        const int q = bit_reverse(r, l - 1);
        const W *A = F + (size_t)(2 * j * half + r) * pitch, *B = A + (size_t)half * pitch;
        const W *Bq = B + (q & ~3);
        for (int u0 = 0; u0 < width; u0 += 128) {
            const int u = u0 + 4 * lane;
            if (u < width) {
                uint4 o[2];
                const uint4 a4 = *(const uint4 *)&A[u];
                const uint4 b4[2] = {*(const uint4 *)&Bq[u], *(const uint4 *)&Bq[u + 4]};
                switch (q & 3) {   // warp-uniform
                    case 0: fht_pair<W, 0>(a4, b4, o); break;
                    case 1: fht_pair<W, 1>(a4, b4, o); break;
                    case 2: fht_pair<W, 2>(a4, b4, o); break;
                    default: fht_pair<W, 3>(a4, b4, o); break;
                }
                out(2 * q, u, o[0]);
                out(2 * q + 1, u, o[1]);
            }
        }
    }
}

// Levels l + 1 and l + 2 (sub-bands of 2^l rows merged into 4 * 2^l) in place, or
// into `out` (kOut, the last ones).
template <typename W, int NT, bool kOut, typename Out>
__device__ void fht_two_levels(W *F, int pitch, int m, int l, int T, Out out) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = 1 << l, width = T + m - 4 * sub;
    for (int p = warp; p < m / 4; p += NT / 32) {
        const int g = p >> l, r = p & (sub - 1);
        const int q = bit_reverse(r, l);
        W *J[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) J[t] = F + (size_t)((4 * g + t) * sub + r) * pitch;
        const W *B1 = J[1] + (q & ~3), *B2 = J[2] + ((2 * q) & ~3), *B3 = J[3] + ((3 * q) & ~3);
        for (int u0 = 0; u0 < width; u0 += 128) {
            const int u = u0 + 4 * lane;
            const bool live = u < width;
            uint4 o[4];
            if (live) {
                const uint4 j0 = *(const uint4 *)&J[0][u];
                const uint4 j1[2] = {*(const uint4 *)&B1[u], *(const uint4 *)&B1[u + 4]};
                const uint4 j2[2] = {*(const uint4 *)&B2[u], *(const uint4 *)&B2[u + 4]};
                const uint4 j3[3] = {*(const uint4 *)&B3[u], *(const uint4 *)&B3[u + 4],
                                     *(const uint4 *)&B3[u + 8]};
                switch (q & 3) {   // warp-uniform
                    case 0: fht_quad<W, 0>(j0, j1, j2, j3, o); break;
                    case 1: fht_quad<W, 1>(j0, j1, j2, j3, o); break;
                    case 2: fht_quad<W, 2>(j0, j1, j2, j3, o); break;
                    default: fht_quad<W, 3>(j0, j1, j2, j3, o); break;
                }
            }
            if (kOut) {
                if (live) {
#pragma unroll
                    for (int t = 0; t < 4; ++t) out(4 * q + t, u, o[t]);
                }
                continue;
            }
            __syncwarp();
            if (live) {   // shift 4q + t to the row of J_{brev2(t)}
                *(uint4 *)&J[0][u] = o[0];
                *(uint4 *)&J[2][u] = o[1];
                *(uint4 *)&J[1][u] = o[2];
                *(uint4 *)&J[3][u] = o[3];
            }
            __syncwarp();
        }
    }
}

// Pitch of F for a tile of T columns: a multiple of 4 words, and reads past
// the last level's columns stay inside the row's pad.
__host__ __device__ inline int fht_pitch(int m, int T) { return (T + m + 16 + 3) & ~3; }

}  // namespace fhtdp
