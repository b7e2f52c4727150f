// Band FHTs in one pass over the image, and the DP as a chain of column tiles
// over the stored Hough rows: the path of single images, of the queries, of
// int32 and float batches and of the calls that run one step of the method.
//
// One image gives the fused engine (engine.cu) few tiles per band level, and
// the levels depend on each other: 16 of 152 SMs work on a level of a 2048 x
// 2048 image, about 15.6 us each.  Here the FHTs, which depend on nothing, run
// first over the whole chip, and the DP items that remain are small: a tile of
// 2048 / n columns (16 for bands of 128 rows), so that a level spreads over the
// chip and the chain advances at the latency of one exchange through L2.
// Bound by that latency, about 5 us a level (poll, V_{b+1} from L2, windows in
// shared memory, store, release).  One call on 2048 x 2048 uint8, n = 128, B =
// 16: engine 249 us, chain 108 (FHT 26); 8192 x 8192 float, 64 bands: 1842 ->
// 974; two polylines 281 -> 124; 24 ragged int32 images in a batch 1406 -> 625.
// Wide uint8 images run on the engine (detect_one).
#include <algorithm>
#include <atomic>
#include <climits>
#include <new>
#include <type_traits>
#include <vector>

#include "chain.cuh"
#include "fht_smem.cuh"

namespace fhtdp {
namespace {

// A load or store under a predicate: a condition in C++ costs a branch each,
// more than the rest of an element's work.
__device__ __forceinline__ uint32_t ld_nc_if(const void *p, bool ok) {   // through L1
    uint32_t v = 0;
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n @p ld.global.nc.b32 %0, [%1];\n}\n"
                 : "+r"(v)
                 : "l"(p), "r"((uint32_t)ok));
    return v;
}
__device__ __forceinline__ uint32_t ld_if_bits(const void *p, bool ok, uint32_t other) {
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n @p ld.global.cg.b32 %0, [%1];\n}\n"
                 : "+r"(other)
                 : "l"(p), "r"((uint32_t)ok));
    return other;
}
template <typename Acc>
__device__ __forceinline__ Acc ld_if(const Acc *p, bool ok, Acc other) {
    return word_from<Acc>(ld_if_bits(p, ok, word_bits(other)));
}
template <typename Acc>
__device__ __forceinline__ void st_if(Acc *p, bool ok, Acc v) {
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n @p st.global.b32 [%0], %1;\n}\n" ::"l"(
                     p),
                 "r"(word_bits(v)), "r"((uint32_t)ok)
                 : "memory");
}

// ---------------------------------------------------------------------------
// Band FHT (Sec. 2.1): a block takes T columns of one sub-band of m <= 128
// rows, builds the first two levels in registers from the image, merges the
// rest in shared memory and writes the rows of both slope signs.  int32 and
// float images run the signs one after the other, the "-" sign on the mirrored
// strip; uint8 images both at once (fht_smem.cuh).  Bound by shared memory
// (about 28 bytes a word and sign) and the stores of the rows.
// 2048 x 2048 uint8, n = 128, a call of fhtdp_fht_bands: four passes over the whole
// arrays 93 us, this 31 (the kernel 26).  Three register levels and 768 threads
// took a quarter more.
constexpr int kFhtNT = 1024;

template <typename In, typename Acc>
struct BandFht {
    static constexpr bool kPacked = sizeof(In) == 1;
    using Wd = typename std::conditional<kPacked, uint32_t, Acc>::type;
    const FhtImg &im;
    const In *base;     // first row of the sub-band
    int x0;
    bool aligned;       // rows can be read four pixels at a time

    // Pixel c of a row of the cyclic band: zero left of the image (the "-"
    // strip never needs the columns it would wrap to: they are padding).
    __device__ Acc px(const In *row, int c) const {
        if (c >= im.W) c -= im.W;
        return c >= 0 && c < im.w ? (Acc)row[c] : Acc(0);
    }
    // Pixels c .. c + 3, c a multiple of 4; kInside: all in the image and
    // aligned.  Elsewhere a predicated load (one launch of one image waits for
    // its edge blocks), or four in unaligned rows and where the four straddle
    // the image's edge; columns past W wrap around (bands of 1 or 2 rows: also
    // in the four that straddle the edge).
    __device__ bool inside4(int c) const { return aligned && c >= 0 && c + 4 <= im.w; }
    template <bool kInside>
    __device__ uint32_t quad8(const In *row, int c) const {
        if (kInside) return __ldg((const uint32_t *)(row + c));
        const bool ok = inside4(c);
        uint32_t v = ld_nc_if(row + c, ok);
        if (c + 3 >= im.W) {
            for (int j = 0; j < 4; ++j) v |= (uint32_t)(uint8_t)px(row, c + j) << (8 * j);
        } else if (!ok && c >= 0 && c < im.w) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                uint32_t b = 0;
                asm volatile(
                    "{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n @p ld.global.nc.u8 %0, [%1];\n}\n"
                    : "+r"(b)
                    : "l"(row + c + j), "r"((uint32_t)(c + j < im.w)));
                v |= b << (8 * j);
            }
        }
        return v;
    }
    template <bool kInside>
    __device__ void quad32(const In *row, int c, Acc *v) const {
        if (kInside) {
            unpack4(__ldg((const uint4 *)(row + c)), v);
            return;
        }
        const bool ok = inside4(c);
        uint4 q = make_uint4(0, 0, 0, 0);
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.u32 p, %5, 0;\n"
            " @p ld.global.nc.v4.b32 {%0, %1, %2, %3}, [%4];\n}\n"
            : "+r"(q.x), "+r"(q.y), "+r"(q.z), "+r"(q.w)
            : "l"(row + c), "r"((uint32_t)ok));
        unpack4(q, v);
        if (c + 3 >= im.W) {
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = px(row, c + j);
        } else if (!ok && c >= 0 && c < im.w) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                v[j] = word_from<Acc>(ld_nc_if(row + c + j, c + j < im.w));
        }
    }
    // Words u .. u + N - 1 (u a multiple of 4) of sub-band row y; kSign 1: of
    // the mirrored strip (packed words hold both).
    template <bool kInside, int kSign, int N>
    __device__ void words(int y, int u, Wd (&P)[N]) const {
        constexpr int NW = (N + 3) / 4;
        const In *row = base + (size_t)y * im.pitch;
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            const int cp = x0 + u + 4 * k, cm = x0 + im.T - 4 - u - 4 * k;
            if constexpr (kPacked) {
                const uint32_t a = quad8<kInside>(row, cp), b = quad8<kInside>(row, cm);
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (4 * k + t < N)
                        P[4 * k + t] = __byte_perm(a, b, t | (7 - t) << 8) & 0x00ff00ffu;
            } else {
                Acc q[4];
                quad32<kInside>(row, kSign == 0 ? cp : cm, q);
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (4 * k + t < N) P[4 * k + t] = q[kSign == 0 ? t : 3 - t];
            }
        }
    }
    // Levels 1 and 2 in registers: a task is four rows and four words.
    template <bool kInside, int kSign>
    __device__ void first_levels(Wd *F, int pitch) const {
        const int C4 = (im.T + im.m - 4 + 3) / 4, tasks = (im.m / 4) * C4;
        for (int t = threadIdx.x; t < tasks; t += kFhtNT) {
            const int g = t / C4, u = 4 * (t - g * C4), y0 = 4 * g;
            Wd B[2][6];   // the lower pair's shifts 0 and 1
            {
                Wd p[6], q[7];
                words<kInside, kSign>(y0 + 2, u, p);
                words<kInside, kSign>(y0 + 3, u, q);
#pragma unroll
                for (int j = 0; j < 6; ++j) {
                    B[0][j] = p[j] + q[j];
                    B[1][j] = p[j] + q[j + 1];
                }
            }
            Wd p[4], q[5], o[4][4];
            words<kInside, kSign>(y0, u, p);
            words<kInside, kSign>(y0 + 1, u, q);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const Wd a0 = p[j] + q[j], a1 = p[j] + q[j + 1];
                o[0][j] = a0 + B[0][j];
                o[1][j] = a0 + B[0][j + 1];
                o[2][j] = a1 + B[1][j + 1];
                o[3][j] = a1 + B[1][j + 2];
            }
            Wd *row = F + (size_t)y0 * pitch + u;   // shift s to row brev2(s)
            *(uint4 *)row = pack4(o[0]);
            *(uint4 *)(row + 2 * pitch) = pack4(o[1]);
            *(uint4 *)(row + pitch) = pack4(o[2]);
            *(uint4 *)(row + 3 * pitch) = pack4(o[3]);
        }
    }
    // The strip's 128-byte lines requested into L2 at once: the register levels
    // would wait for DRAM task by task.
    __device__ void prefetch() const {
        const int lo = max(x0 - (im.m - 1), 0), hi = min(x0 + im.T + im.m - 1, im.w);
        if (lo >= hi) return;
        const int lines = ((hi - lo) * (int)sizeof(In) + 127) / 128 + 1;
        for (int i = threadIdx.x; i < im.m * lines; i += kFhtNT) {
            const int y = i / lines;
            const uintptr_t a = (uintptr_t)(base + (size_t)y * im.pitch + lo);
            const uintptr_t end = (uintptr_t)(base + (size_t)y * im.pitch + hi);
            const uintptr_t line = (a & ~(uintptr_t)127) + (uintptr_t)(i - y * lines) * 128;
            if (line < end) asm volatile("prefetch.global.L2 [%0];" ::"l"(line));
        }
    }
};

// kSplit: a block makes one slope sign, two blocks a tile (int32 and float).
template <typename In, typename Acc, bool kSplit>
__global__ void __launch_bounds__(kFhtNT, 1) fht_band_kernel(const __grid_constant__ FhtImg one,
                                                             const FhtImg *__restrict__ many,
                                                             int count) {
    extern __shared__ __align__(16) unsigned char smem[];
    using Tile = BandFht<In, Acc>;
    using Wd = typename Tile::Wd;
    int i = 0;
    if (many) {   // the last image that starts at or before this block
        int hi = count - 1;
        while (i < hi) {
            const int mid = (i + hi + 1) / 2;
            if (many[mid].item0 <= (int)blockIdx.x) i = mid;
            else hi = mid - 1;
        }
    }
    const FhtImg &im = many ? many[i] : one;
    const int item = (blockIdx.x - (many ? im.item0 : 0)) >> (kSplit ? 1 : 0);
    const int sub = item / im.tiles, T = im.T, x0 = (item - sub * im.tiles) * T;
    const int m = im.m, pitch = fht_pitch(m, T), per_band = im.n / m;
    const int band = sub / per_band, j = sub - band * per_band;
    Acc *rows = (Acc *)im.out + ((size_t)band * 2 * im.n + j * m) * im.opitch;
    const bool vec = im.opitch % 4 == 0 && (uintptr_t)im.out % 16 == 0;
    Wd *F = (Wd *)smem;
    const Tile t{im, (const In *)im.img + (size_t)sub * m * im.pitch, x0,
                 (uintptr_t)im.img % (4 * sizeof(In)) == 0 && im.pitch % 4 == 0};
    t.prefetch();
    // every column that a task reads (the widest: u + 8 past the strip's words)
    const bool inside = t.aligned && x0 >= m + 8 && x0 + T + m + 8 <= im.w;
    // four values of shift s, columns x .. x + 3
    auto store = [&](int sign, int s, int x, const Acc *v) {
        Acc *dst = rows + ((size_t)sign * im.n + s) * im.opitch + x;
        if (vec && x + 4 <= im.wout) {
            *(uint4 *)dst = pack4(v);
        } else {
            for (int e = 0; e < 4; ++e)
                if (x + e < im.wout) dst[e] = v[e];
        }
    };
    for (int sign = kSplit ? blockIdx.x & 1 : 0; sign < (Tile::kPacked ? 1 : 2); ++sign) {
        auto out = [&](int s, int u, const uint4 &q) {
            Acc v[4];
            if constexpr (Tile::kPacked) {
                const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = (Acc)(w[e] & 0xffffu);
                store(0, s, x0 + u, v);
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = (Acc)(w[3 - e] >> 16);
                store(1, s, x0 + T - 4 - u, v);
            } else {
                unpack4(q, v);
                if (sign == 0) {
                    store(0, s, x0 + u, v);
                } else {
                    const Acc r[4] = {v[3], v[2], v[1], v[0]};
                    store(1, s, x0 + T - 4 - u, r);
                }
            }
        };
        int l = 0;   // levels merged
        if (m >= 4) {
            if (inside) {
                if (Tile::kPacked || sign == 0) t.template first_levels<true, 0>(F, pitch);
                else t.template first_levels<true, 1>(F, pitch);
            } else {
                if (Tile::kPacked || sign == 0) t.template first_levels<false, 0>(F, pitch);
                else t.template first_levels<false, 1>(F, pitch);
            }
            l = 2;
        } else {
            const int G = (T + m + 3) / 4;
            for (int idx = threadIdx.x; idx < m * G; idx += kFhtNT) {
                const int y = idx / G, u = 4 * (idx - y * G);
                Wd v[4];
                if (sign == 0) t.template words<false, 0>(y, u, v);
                else t.template words<false, 1>(y, u, v);
                *(uint4 *)&F[(size_t)y * pitch + u] = pack4(v);
            }
        }
        __syncthreads();
        if (l == im.log2m)   // bands of 1 or 4 rows: every level done
            for (int idx = threadIdx.x; idx < m * (T / 4); idx += kFhtNT) {
                const int s = idx / (T / 4), u = 4 * (idx % (T / 4));
                out(s, u, *(const uint4 *)&F[(size_t)bit_reverse(s, l) * pitch + u]);
            }
        while (l < im.log2m) {
            const int left = im.log2m - l;
            if (left > 2) {
                fht_two_levels<Wd, kFhtNT, false>(F, pitch, m, l, T, out);
                l += 2;
            } else if (left == 2) {
                fht_two_levels<Wd, kFhtNT, true>(F, pitch, m, l, T, out);
                l += 2;
            } else {
                fht_level<Wd, kFhtNT>(F, pitch, m, l + 1, T, out);
                l += 1;
            }
            __syncthreads();
        }
        if (kSplit) break;
        __syncthreads();   // F is rewritten for the other sign
    }
}

// Bands of at most 16 rows: a strip of so few rows leaves most of a block of
// fht_band_kernel idle, so a thread takes one column of one band here and adds
// up its sums of both signs in registers, straight from the image (L1 serves the
// overlapping reads).  Bound by the stores of the rows (1 to 4 rows: 4 TB/s and
// more) and from there on by the loads' issue.  2048 x 2048 uint8, n = 1, 2, 4, 8,
// 16: a pass a level 17, 15, 33, 40, 58 us; fht_band_kernel 261, 232, 89, 62, 50;
// this 13, 10, 10, 13, 23.  8192 x 8192 float, n = 8: 620, 1362, 143.  (32 rows
// would need some 270 registers; fht_band_kernel takes 29 us for 2048 x 2048 uint8.)
constexpr int kShortRows = 16;
template <typename In, typename Acc, int kSign, bool kInside>
struct ShortBand {
    const In *base;      // first row of the band
    long long pitch;
    int x, w, W;
    // Column x + j (sign "-": x - j) of a row of the cyclic band.
    __device__ Acc px(const In *row, int j) const {
        int c = kSign == 0 ? x + j : x - j;
        if (!kInside) {
            if (c >= W) c -= W;
            if (c < 0 || c >= w) return Acc(0);   // (left of the image: padding)
        }
        return (Acc)__ldg(row + c);
    }
    // Shifts 0 .. R - 1 of the R rows from row y, words 0 .. M - 1.
    template <int R, int M>
    __device__ void sums(int y, Acc (&o)[R][M]) const {
        if constexpr (R == 1) {
            const In *row = base + y * pitch;
#pragma unroll
            for (int j = 0; j < M; ++j) o[0][j] = px(row, j);
        } else {
            Acc a[R / 2][M], b[R / 2][M + R / 2];
            sums<R / 2, M>(y, a);
            sums<R / 2, M + R / 2>(y + R / 2, b);
#pragma unroll
            for (int s = 0; s < R; ++s)
#pragma unroll
                for (int j = 0; j < M; ++j) o[s][j] = a[s / 2][j] + b[s / 2][j + (s + 1) / 2];
        }
    }
};

// A block: blockDim.x columns of blockDim.y bands.
template <typename In, typename Acc, int N>
__global__ void __launch_bounds__(256) fht_short_kernel(const __grid_constant__ FhtImg im) {
    const int tile = blockIdx.x % im.tiles, x0 = tile * blockDim.x, x = x0 + threadIdx.x;
    const int band = blockIdx.x / im.tiles * blockDim.y + threadIdx.y;
    if (band >= im.subs || x >= im.wout) return;
    const In *base = (const In *)im.img + (size_t)band * N * im.pitch;
    Acc *out = (Acc *)im.out + (size_t)band * 2 * N * im.opitch + x;
    const bool inside = x0 >= N && x0 + (int)blockDim.x + N <= im.w;
    auto one_sign = [&](auto rows, int sign) {
        Acc o[N][1];
        rows.template sums<N, 1>(0, o);
#pragma unroll
        for (int s = 0; s < N; ++s) out[(size_t)(sign * N + s) * im.opitch] = o[s][0];
    };
    if (inside) {
        one_sign(ShortBand<In, Acc, 0, true>{base, im.pitch, x, im.w, im.W}, 0);
        one_sign(ShortBand<In, Acc, 1, true>{base, im.pitch, x, im.w, im.W}, 1);
    } else {
        one_sign(ShortBand<In, Acc, 0, false>{base, im.pitch, x, im.w, im.W}, 0);
        one_sign(ShortBand<In, Acc, 1, false>{base, im.pitch, x, im.w, im.W}, 1);
    }
}

// ---------------------------------------------------------------------------
// The DP chain (Sec. 2.2-2.3, Eqs. 3-4).  An item is one band b and `cols`
// continuation columns xn: with V_{b+1}(xn, e) of all displacements e in
// shared memory, it answers M(xn, d) = max of V_{b+1}(xn, e) over the window
// of d, and adds it in place to the states that end in its columns,
// V_b(xn - d, d) = H_b(xn - d, d) + M(xn, d): every state has one owner.  Items
// come from a queue, band level by band level; an item waits for the tiles of
// band b + 1 within n - 1 columns of its own (bounded acquire spins), so the
// queue cannot deadlock: every item waits only for earlier ones, and a block
// holds at most the item in work and the next one.
//
// A thread owns one column and runs of 8 displacements; its Hough values are
// loaded before the wait.  The window maxima are van Herk / Gil-Werman with the
// runs as blocks: of its run of V_{b+1} a thread stores the maxima from every
// value to the run's end (S) and from its start to every value (P), and a window
// [a, z] is the largest of S(a), P(z) and the runs between (S of their first
// values): two shared-memory reads an output and a few a run, whatever the
// window's length, for the bend limit and for tables alike.  Windows that may
// lie inside one run (shorter than 9) scan the values themselves.  States whose link leaves [0, vw), or that
// the point mask excludes, are never stored as dead: every reader knows them by
// their place (alive()).  Band 0 folds the lexicographic argmax; the last of
// its tiles reads the polyline back (Eq. 5).
// Bound by latency: one flag and one load round trip through L2 per band level.
constexpr int kDpNT = 512;
constexpr int kDpPerSm = 2;     // blocks an SM: all its registers at 64 a thread
constexpr int kRun = 8;         // displacements of a thread's run
// Bend limits up to this read past the range unchecked: 2048 x 2048 uint8, n = 64,
// B = 20, 32: 156 and 161 us the call, clipped 175 and 172 (n = 128, B = 32: 103,
// 108).  B = 40 would still gain, 174 -> 162 us (n = 128: 109 -> 105), for twice the
// dead rows in shared memory.
constexpr int kPadB = 32;
constexpr int kMinLen = kRun + 1;   // windows from this length on span two runs

struct ChainItem {
    int image, band, tile, pad;
};

struct ChainArgs {
    ChainImg one;
    const ChainImg *many;      // several images (device), or null
    const ChainItem *order;    // their queue
    int items;
    ChainCtl *ctl;
    int *report;         // where a wait that gave up is noted as well (or null)
    long long wait_cycles;
    int skip_band, skip_tile;  // test hook: this tile of the first image never publishes
    int band;                  // >= 0: one launch per band (no queue, no flags)
    int store0;                // band 0's values are stored (needed after the run)
    // With use_table the window of d is [tab.lo, tab.hi] instead of |e - d| <= B;
    // minlen: the shortest of them.
    int use_table, minlen;
    WindowTable tab;
};

__device__ __forceinline__ void gave_up(const ChainArgs &a) {
    atomicExch(&a.ctl->status, FHTDP_ETIMEOUT);
    if (a.report) atomicExch(a.report, FHTDP_ETIMEOUT);
}

// The flags are polled with relaxed loads, one fence after the last; a poll
// reads nothing else (another load would double its round trip).
__device__ __forceinline__ int ld_relaxed(const int *p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ void st_rel(int *p, int v) {
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

template <typename Acc>
__device__ __forceinline__ Acc vmax(Acc a, Acc b) {
    return a > b ? a : b;
}
template <>
__device__ __forceinline__ float vmax(float a, float b) {
    return fmaxf(a, b);
}

// Order-preserving 32-bit image of a value (negative zero counts as zero).
__device__ __forceinline__ uint32_t vord(int32_t v) { return (uint32_t)v ^ 0x80000000u; }
__device__ __forceinline__ uint32_t vord(float f) {
    const uint32_t b = __float_as_uint(f == 0.0f ? 0.0f : f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
template <typename Acc>
__device__ __forceinline__ Acc vfrom(uint32_t o);
template <>
__device__ __forceinline__ int32_t vfrom<int32_t>(uint32_t o) {
    return (int32_t)(o ^ 0x80000000u);
}
template <>
__device__ __forceinline__ float vfrom<float>(uint32_t o) {
    return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}
__device__ __forceinline__ int32_t ld_cg(const int32_t *p) { return __ldcg(p); }
__device__ __forceinline__ float ld_cg(const float *p) { return __ldcg(p); }

// State (x, e) of band b: both vertices inside and not excluded by the point.
__device__ __forceinline__ bool alive(const ChainImg &im, int b, int x, int e) {
    const int y = x + e;
    if (x < 0 || x >= im.vw || y < 0 || y >= im.vw) return false;
    return im.mask1 != b + 1 || (im.mask_end ? y : x) == im.mask_x;
}
template <typename Acc>
__device__ __forceinline__ Acc *band_rows(const ChainImg &im, int b) {
    return (Acc *)im.hv + (size_t)b * 2 * im.n * im.pitch;
}
// Place of state (x, d) in its band; d = 0 is stored in both halves, and the
// chain uses the copy in the "-" half.
__device__ __forceinline__ int state_at(const ChainImg &im, int x, int d) {
    return (d <= 0 ? im.n - d : d) * im.pitch + x;
}

// One warp: the polyline from the argmax key (Eq. 5); every band's window is
// scanned by the lanes, the smallest displacement of the largest value kept.
// kCaller: a caller's array, whose d = 0 is read in the "+" half.
// Key 0 (no admissible polyline): x = -1 everywhere and a dead score.
template <typename Acc, bool kCaller = false>
__device__ void chain_readback(const ChainImg &im, const ChainArgs &args, unsigned long long key,
                               int32_t *x_out, int32_t *d_out, Acc *score_out) {
    const int lane = threadIdx.x & 31, n = im.n, D = 2 * n - 1;
    if (key == 0) {
        if (lane == 0) *score_out = Dead<Acc>::value();
        for (int i = lane; i <= im.k; i += 32) x_out[i] = -1;
        for (int i = lane; i < im.k; i += 32) d_out[i] = 0;
        return;
    }
    const unsigned lin = 0xffffffffu - (unsigned)(key & 0xffffffffu);
    int x = (int)(lin / D), d = (int)(lin % D) - (n - 1);
    if (lane == 0) {
        x_out[0] = x;
        d_out[0] = d;
        *score_out = vfrom<Acc>((uint32_t)(key >> 32));
    }
    for (int i = 1; i < im.k; ++i) {
        x += d;
        const int lo = args.use_table ? args.tab.lo[d + n - 1] : max(d - im.B, -(n - 1));
        const int hi = args.use_table ? args.tab.hi[d + n - 1] : min(d + im.B, n - 1);
        const Acc *V = band_rows<Acc>(im, i);
        unsigned best = 0;     // order image of the value (0: none)
        unsigned be = INT_MAX; // its displacement index
        auto value = [&](int e) -> Acc {
            const int at = kCaller && e == 0 ? x : state_at(im, x, e);
            return ld_if(V + at, e <= hi && alive(im, i, x, e), Dead<Acc>::value());
        };
        for (int e0 = lo + lane; e0 <= hi; e0 += 128) {   // four loads in flight
            Acc v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = value(e0 + 32 * j);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                // (NaN, whose comparisons are false, counts as dead)
                const unsigned o = v[j] > Dead<Acc>::value() ? vord(v[j]) : 0;
                if (o > best) {
                    best = o;
                    be = e0 + 32 * j + n - 1;
                }
            }
        }
        const unsigned top = __reduce_max_sync(0xffffffffu, best);
        unsigned at = __reduce_min_sync(0xffffffffu, best == top && top ? be : INT_MAX);
        if (at >= (unsigned)D) {
            if (std::is_same<Acc, float>::value) {   // nothing but NaN: the first one
                be = INT_MAX;
#pragma unroll 1
                for (int e = lo + lane; e <= hi; e += 32) {
                    const Acc v = value(e);
                    if (v != v) be = min(be, (unsigned)(e + n - 1));
                }
                at = __reduce_min_sync(0xffffffffu, be);
            }
            if (at >= (unsigned)D) {   // only with inconsistent values (a wait gave up)
                if (lane == 0 && args.ctl) gave_up(args);
                return;
            }
        }
        d = (int)at - (n - 1);
        if (lane == 0) {
            x_out[i] = x;
            d_out[i] = d;
        }
    }
    if (lane == 0) x_out[im.k] = x + d;
}

// Words between the rows of V: with 16 columns a warp holds two runs, eight
// rows apart, and 18 words put them into different banks.
__host__ __device__ constexpr int row_words(int cols) { return cols == 16 ? 18 : cols; }

// How an image's windows are answered: by scanning the values, from S and P with
// dead rows around the range (bend limits up to kPadB), or from S and P with the
// windows clipped to the range (tables, longer limits): each by itself, or with
// the runs that eight neighbours share taken once, which pays from kSharedLen on
// (bends of 0.17 rad, 2048 x 2048, n = 128: 40 and more, by itself 114.7 us the
// call, shared 113.3; 19 bands of 64 rows, 1400 columns: 20 and more, 103, 108).
enum { kScan, kPadded, kClipped, kShared };
constexpr int kSharedLen = 32;
__host__ __device__ constexpr int window_mode(int use_table, int minlen, int B) {
    if (use_table) return minlen >= kSharedLen ? kShared : minlen >= kMinLen ? kClipped : kScan;
    return 2 * B + 1 < kMinLen ? kScan : B <= kPadB ? kPadded : kShared;
}
// Dead rows above and below the range, whole runs.
__host__ __device__ constexpr int window_pad(int mode, int use_table, int B) {
    if (mode == kScan && !use_table) return kRun;
    return mode == kPadded ? (B + kRun - 1) / kRun * kRun : 0;
}
__host__ __device__ constexpr int range_rows(int n) {
    return (2 * n - 1 + kRun - 1) / kRun * kRun;
}

// kC: the image's tile width, or 0 to take it from the image (a batch of several
// widths: five copies of the code for one kernel spill).  kLong: the code of
// kShared and of scanned tables alone, in a kernel of its own (beside the other
// modes' it cost those 0.2 us a band level: 2048 x 2048 uint8, n = 128, 105.6 ->
// 108.6 us the call); without it kShared runs as kClipped.
template <typename Acc, int kC, bool kLong>
__device__ void chain_item(const ChainImg &im, int band, int tile, unsigned char *smem,
                           const ChainArgs &args) {
    const int C = kC ? kC : im.cols, lg = 31 - __clz(C);
    const int Q = kDpNT >> lg, R = row_words(C);
    const int n = im.n, D = 2 * n - 1, lo = -(n - 1), hi = n - 1, xn0 = tile * C;
    const int u = threadIdx.x & (C - 1), q = threadIdx.x >> lg, xn = xn0 + u;
    const bool last = band == im.k - 1;   // (only one-band images: V = H)
    const int B = im.B, asked = window_mode(args.use_table, args.minlen, B);
    const int mode = kLong ? asked : min(asked, (int)kClipped);
    const int pad = window_pad(mode, args.use_table, B), rows = range_rows(n);
    const Acc dead = Dead<Acc>::value();
    // S (or the values), then P: row e - lo + pad of displacement e
    Acc *S = (Acc *)smem, *P = S + (rows + 2 * pad) * R;
    const Acc *Vb = last ? nullptr : band_rows<Acc>(im, band + 1);
    Acc *Hb = band_rows<Acc>(im, band);
    // A run of kRun displacements lies in one half (bands of at least kRun
    // rows), so its states are a fixed step apart: along a column for V, along a
    // diagonal (fixed end column) for H.  Live states of an unmasked band: both
    // vertices inside.
    const bool in = xn < im.vw, whole = n >= kRun;
    const bool mask_h = im.mask1 == band + 1, mask_v = im.mask1 == band + 2;
    const bool inner = whole && xn0 >= n && xn0 + C + n <= im.vw;   // every state is inside
    // this thread's Hough values (first run), in flight during the wait
    Acc h[kRun];
    auto load_h = [&](int c0) {
        if (inner && !mask_h) {
            // (the last run's eighth row is a row of this band that is not used)
            const int step = c0 <= 0 ? -(im.pitch + 1) : im.pitch - 1;
            const Acc *p = Hb + state_at(im, xn - c0, c0);
#pragma unroll
            for (int i = 0; i < kRun; ++i) h[i] = ld_cg(p + i * step);
        } else if (whole && !mask_h) {
            const int step = c0 <= 0 ? -(im.pitch + 1) : im.pitch - 1;
            const Acc *p = Hb + state_at(im, xn - c0, c0);
#pragma unroll
            for (int i = 0; i < kRun; ++i) {
                const bool ok = in && (unsigned)(xn - c0 - i) < (unsigned)im.vw && c0 + i <= hi;
                h[i] = ld_if(p + i * step, ok, Acc(0));
            }
        } else {
#pragma unroll
            for (int i = 0; i < kRun; ++i) {
                const int d = c0 + i;
                h[i] = d <= hi && alive(im, band, xn - d, d)
                           ? ld_cg(Hb + state_at(im, xn - d, d))
                           : Acc(0);
            }
        }
    };
    load_h(lo + kRun * q);
    for (int i = threadIdx.x; i < 2 * pad * C; i += kDpNT) {
        const int r = i >> lg, at = (r < pad ? r : r + rows) * R + (i & (C - 1));
        S[at] = dead;
        if (mode == kPadded) P[at] = dead;
    }
    if (args.band >= 0) {
        // one launch per band: this one began while the band below still ran
        asm volatile("griddepcontrol.wait;" ::: "memory");
    } else if (!last && threadIdx.x < 32) {
        bool ok = true;
        // bands below k - 1 are items; band k - 1 is complete (unless the test
        // hook holds a tile of it back)
        if (band + 1 < im.k - 1 || args.skip_band == band + 1) {
            const int t0 = max(xn0 - (n - 1), 0) >> lg;
            const int t1 = min(xn0 + C - 1 + n - 1, im.vw - 1) >> lg;
            for (int t = t0 + (int)threadIdx.x; t <= t1 && ok; t += 32) {
                if (band + 1 == im.k - 1 && t != args.skip_tile) continue;
                const int *flag = im.flags + (size_t)(band + 1) * im.tiles + t;
                const long long begin = clock64();
                while (ld_relaxed(flag) == 0) {
                    const long long spent = clock64() - begin;
                    if (spent < 20000) continue;   // (about 10 us)
                    if (ld_relaxed(&args.ctl->status) != FHTDP_OK || spent > args.wait_cycles) {
                        ok = false;
                        break;
                    }
                    __nanosleep(100);
                }
            }
            fence_gpu();
        }
        if (!__all_sync(0xffffffffu, ok) && threadIdx.x == 0)
            gave_up(args);
    }
    if (!last) {
        __syncthreads();
        // V_{b+1} of these columns; the thread's own rows
        for (int c0 = lo + kRun * q; c0 <= hi; c0 += kRun * Q) {
            Acc v[kRun];
            if (inner && !mask_v) {
                const int step = c0 <= 0 ? -im.pitch : im.pitch;
                const Acc *p = Vb + state_at(im, xn, c0);
#pragma unroll
                for (int i = 0; i < kRun; ++i) v[i] = ld_cg(p + i * step);
            } else if (whole && !mask_v) {
                const int step = c0 <= 0 ? -im.pitch : im.pitch;
                const Acc *p = Vb + state_at(im, xn, c0);
#pragma unroll
                for (int i = 0; i < kRun; ++i) {
                    const bool ok =
                        in && (unsigned)(xn + c0 + i) < (unsigned)im.vw && c0 + i <= hi;
                    v[i] = ld_if(p + i * step, ok, dead);
                }
            } else {
#pragma unroll
                for (int i = 0; i < kRun; ++i) {
                    const int e = c0 + i;
                    v[i] = e <= hi && alive(im, band + 1, xn, e) ? ld_cg(Vb + state_at(im, xn, e))
                                                                 : dead;
                }
            }
            if (c0 + kRun - 1 > hi)   // the last run is short
#pragma unroll
                for (int i = 0; i < kRun; ++i)
                    if (c0 + i > hi) v[i] = dead;
            Acc *s = S + (c0 - lo + pad) * R + u, *p = P + (c0 - lo + pad) * R + u;
            if (mode == kScan) {
#pragma unroll
                for (int i = 0; i < kRun; ++i) s[i * R] = v[i];
            } else {
                Acc run = v[0];
                p[0] = run;
#pragma unroll
                for (int i = 1; i < kRun; ++i) p[i * R] = run = vmax(run, v[i]);
                run = v[kRun - 1];
                s[(kRun - 1) * R] = run;
#pragma unroll
                for (int i = kRun - 2; i >= 0; --i) s[i * R] = run = vmax(run, v[i]);
            }
        }
        __syncthreads();
    }
    const Acc *Su = S + u, *Pu = P + u;
    unsigned long long best = 0;
    for (int c0 = lo + kRun * q; c0 <= hi; c0 += kRun * Q) {
        if (c0 != lo + kRun * q) load_h(c0);
        Acc M[kRun];
        const int r0 = c0 - lo + pad;   // the run's first row
        auto run_of = [&](int j) -> Acc { return Su[j * kRun * R]; };   // maximum of run j
        if (last) {
        } else if (mode == kPadded && !kLong) {
            // windows [r - B, r + B]: their first run is j0 or, from row 8 - ol
            // on, j0 + 1; their last one z0 or, from row 8 - oz on, z0 + 1
            const int j0 = (r0 - B) >> 3, z0 = (r0 + B) >> 3;
            const int ol = (r0 - B) & 7, oz = (r0 + B) & 7;
            Acc mid = dead;   // runs j0 + 2 .. z0 - 1
#pragma unroll 1
            for (int j = j0 + 2; j < z0; ++j) mid = vmax(mid, run_of(j));
            const Acc x = run_of(j0 + 1), y = run_of(z0);
            const Acc m00 = j0 + 1 < z0 ? vmax(mid, x) : dead;
            const Acc m01 = j0 + 1 < z0 ? vmax(vmax(mid, x), y) : y;
            const Acc m11 = j0 + 1 < z0 ? vmax(mid, y) : dead;
            const Acc *a = Su + (r0 - B) * R, *z = Pu + (r0 + B) * R;
#pragma unroll
            for (int i = 0; i < kRun; ++i) {
                const bool la = i + ol >= kRun, lz = i + oz >= kRun;
                const Acc between = la ? (lz ? m11 : mid) : (lz ? m01 : m00);
                M[i] = vmax(vmax(a[i * R], z[i * R]), between);
            }
        } else if (kLong && mode == kShared) {
            // Both ends of a window grow with the displacement, so the runs between
            // the last window's first one (ja) and the first window's last one (jz)
            // lie inside all eight: their maximum once.  Each window adds its own
            // few at both ends.  polyline_dp of 2048 x 2048, unrestricted, n = 128:
            // every window's runs by itself 155 us, this 99 (n = 256: 190, 88).
            auto first = [&](int c) -> int {
                return (args.use_table ? args.tab.lo[c - lo] : max(c - B, lo)) - lo;
            };
            auto final = [&](int c) -> int {
                return (args.use_table ? args.tab.hi[c - lo] : min(c + B, hi)) - lo;
            };
            const int ja = first(min(c0 + kRun - 1, hi)) >> 3, jz = final(c0) >> 3;
            Acc mid = dead;
#pragma unroll 1
            for (int j = ja + 1; j < jz; j += 4) {   // four loads in flight
                const int e = jz - 1;
                const Acc x0 = run_of(j), x1 = run_of(min(j + 1, e));
                const Acc x2 = run_of(min(j + 2, e)), x3 = run_of(min(j + 3, e));
                mid = vmax(vmax(mid, vmax(x0, x1)), vmax(x2, x3));
            }
#pragma unroll
            for (int i = 0; i < kRun; ++i) {
                const int c = min(c0 + i, hi), a = first(c), z = final(c), e = z >> 3;
                Acc m = vmax(vmax(Su[a * R], Pu[z * R]), mid);
#pragma unroll 1
                for (int j = (a >> 3) + 1; j <= min(ja, e - 1); ++j) m = vmax(m, run_of(j));
#pragma unroll 1
                for (int j = max(jz, ja + 1); j < e; ++j) m = vmax(m, run_of(j));
                M[i] = m;
            }
        } else if (!kLong && mode == kClipped) {
#pragma unroll
            for (int i = 0; i < kRun; ++i) {
                const int c = min(c0 + i, hi);
                const int a = (args.use_table ? args.tab.lo[c - lo] : max(c - B, lo)) - lo;
                const int z = (args.use_table ? args.tab.hi[c - lo] : min(c + B, hi)) - lo;
                Acc m = vmax(Su[a * R], Pu[z * R]);
                const int e = (z >> 3) - 1;   // the last run inside
#pragma unroll 1
                for (int j = (a >> 3) + 1; j <= e; j += 4) {   // four loads in flight
                    const Acc x0 = run_of(j), x1 = run_of(min(j + 1, e));
                    const Acc x2 = run_of(min(j + 2, e)), x3 = run_of(min(j + 3, e));
                    m = vmax(vmax(m, vmax(x0, x1)), vmax(x2, x3));
                }
                M[i] = m;
            }
        } else if (kLong) {
            // short windows, value by value: four of each of two outputs in flight (a
            // window that has ended repeats its last value).  polyline_dp_angle of
            // 2048 x 2048, n = 32, 0.05 rad: one output's four 286 us, this 270.
#pragma unroll
            for (int i = 0; i < kRun; i += 2) {
                const int c = min(c0 + i, hi), d = min(c0 + i + 1, hi);
                const int a = args.tab.lo[c - lo] - lo, z = args.tab.hi[c - lo] - lo;
                const int f = args.tab.lo[d - lo] - lo, g = args.tab.hi[d - lo] - lo;
                const int most = max(z - a, g - f);
                Acc m = dead, o = dead;
#pragma unroll 1
                for (int t = 0; t <= most; t += 4) {
                    const Acc x0 = Su[min(a + t, z) * R], x1 = Su[min(a + t + 1, z) * R];
                    const Acc x2 = Su[min(a + t + 2, z) * R], x3 = Su[min(a + t + 3, z) * R];
                    const Acc y0 = Su[min(f + t, g) * R], y1 = Su[min(f + t + 1, g) * R];
                    const Acc y2 = Su[min(f + t + 2, g) * R], y3 = Su[min(f + t + 3, g) * R];
                    m = vmax(vmax(m, vmax(x0, x1)), vmax(x2, x3));
                    o = vmax(vmax(o, vmax(y0, y1)), vmax(y2, y3));
                }
                M[i] = m;
                M[i + 1] = o;
            }
        } else {
            // B <= 3: the run and three values either side, widened B times
            Acc w[kRun + 6];
#pragma unroll
            for (int i = 0; i < kRun + 6; ++i) w[i] = Su[(r0 - 3 + i) * R];
#pragma unroll
            for (int t = 1; t <= 3; ++t)
                if (B >= t) {
                    Acc before = w[t - 1];
#pragma unroll
                    for (int i = t; i < kRun + 6 - t; ++i) {
                        const Acc here = w[i];
                        w[i] = vmax(vmax(before, here), w[i + 1]);
                        before = here;
                    }
                }
#pragma unroll
            for (int i = 0; i < kRun; ++i) M[i] = w[i + 3];
        }
        if (inner && !mask_h && band != 0 && args.band < 0) {
            const int step = c0 <= 0 ? -(im.pitch + 1) : im.pitch - 1;
            Acc *p = Hb + state_at(im, xn - c0, c0);
#pragma unroll
            for (int i = 0; i + 1 < kRun; ++i) p[i * step] = M[i] == dead ? dead : h[i] + M[i];
            if (c0 + kRun - 1 <= hi)
                p[(kRun - 1) * step] =
                    M[kRun - 1] == dead ? dead : h[kRun - 1] + M[kRun - 1];
            continue;
        }
        if (whole && !mask_h && band != 0 && args.band < 0) {
            const int step = c0 <= 0 ? -(im.pitch + 1) : im.pitch - 1;
            Acc *p = Hb + state_at(im, xn - c0, c0);
#pragma unroll
            for (int i = 0; i < kRun; ++i)
                st_if(p + i * step,
                      in && (unsigned)(xn - c0 - i) < (unsigned)im.vw && c0 + i <= hi,
                      M[i] == dead ? dead : h[i] + M[i]);
            continue;
        }
#pragma unroll
        for (int i = 0; i < kRun; ++i) {
            const int d = c0 + i, x = xn - d;
            if (d > hi || !alive(im, band, x, d)) continue;
            const Acc v = last ? h[i] : M[i] == dead ? dead : h[i] + M[i];
            if (band != 0 || args.store0) {
                Hb[state_at(im, x, d)] = v;
                if (args.band >= 0 && d == 0) Hb[x] = v;   // both copies of d = 0
            }
            if (band == 0 && v != dead) {
                const unsigned long long k = ((unsigned long long)vord(v) << 32) |
                                             (0xffffffffu - (unsigned)(x * D + d + n - 1));
                best = best > k ? best : k;
            }
        }
    }
    if (band == 0 && args.band < 0) {
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long other = __shfl_xor_sync(0xffffffffu, best, o);
            best = best > other ? best : other;
        }
        if ((threadIdx.x & 31) == 0 && best) atomicMax(im.key, best);
        __syncthreads();
        if (threadIdx.x < 32) {
            int finished = 0;
            if (threadIdx.x == 0) {
                __threadfence();
                finished = atomicAdd(im.done, 1) == im.tiles - 1;
            }
            if (__shfl_sync(0xffffffffu, finished, 0)) {
                __threadfence();
                unsigned long long key = 0;
                if (threadIdx.x == 0) key = atomicAdd(im.key, 0ull);
                key = __shfl_sync(0xffffffffu, key, 0);
                chain_readback<Acc>(im, args, key, im.x_out, im.d_out, (Acc *)im.score_out);
            }
        }
    } else if (args.band < 0) {
        __syncthreads();
        if (threadIdx.x == 0) {
            const ChainImg &first = args.many ? args.many[0] : args.one;
            if (!(band == args.skip_band && tile == args.skip_tile && im.flags == first.flags)) {
                st_rel(im.flags + (size_t)band * im.tiles + tile, 1);
            }
        }
    }
    __syncthreads();   // shared memory is rewritten by the next item
}

// kC: the tile width when all images share it, or 0.
template <typename Acc, int kC, bool kLong>
__global__ void __launch_bounds__(kDpNT, kDpPerSm) dp_chain_kernel(const __grid_constant__ ChainArgs args) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_next;
    auto item = [&](const ChainImg &im, int band, int tile) {
        chain_item<Acc, kC, kLong>(im, band, tile, smem, args);
    };
    if (args.band >= 0) {
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        item(args.one, args.band, blockIdx.x);
        return;
    }
    if (threadIdx.x == 0) s_next = atomicAdd(&args.ctl->queue, 1);
    __syncthreads();
    int cur = s_next;
    while (cur < args.items) {
        __syncthreads();
        // the next item, taken while this one is in work
        if (threadIdx.x == kDpNT - 1) s_next = atomicAdd(&args.ctl->queue, 1);
        if (args.many) {
            const ChainItem it = args.order[cur];
            item(args.many[it.image], it.band, it.tile);
        } else {
            const int lv = cur / args.one.tiles;
            item(args.one, max(args.one.k - 2 - lv, 0), cur - lv * args.one.tiles);
        }
        cur = s_next;   // chain_item ends with a barrier
    }
}

// fhtdp_polyline_dp stores dead states: every state of every band whose link
// leaves [0, vw), and the padding columns.  Its input's d = 0 is the row of the
// "+" half; the chain works on the one of the "-" half, which further blocks
// (kDeadCols columns of a band each) make equal to it.
constexpr int kDeadNT = 128, kDeadCols = 8 * kDeadNT;
template <typename Acc>
__global__ void __launch_bounds__(kDeadNT) dp_dead_kernel(Acc *hv, Shape s) {
    const int row = blockIdx.x;   // [k][2][n]
    if (row >= s.k * 2 * s.n) {
        const int chunks = (s.vw + kDeadCols - 1) / kDeadCols, i = row - s.k * 2 * s.n;
        const int band = i / chunks, x0 = (i - band * chunks) * kDeadCols + threadIdx.x;
        const Acc *plus = hv + (size_t)band * 2 * s.n * s.W;
        Acc *minus = hv + ((size_t)band * 2 + 1) * s.n * s.W, v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e)
            v[e] = ld_if(plus + x0 + e * kDeadNT, x0 + e * kDeadNT < s.vw, Acc(0));
#pragma unroll
        for (int e = 0; e < 8; ++e)
            st_if(minus + x0 + e * kDeadNT, x0 + e * kDeadNT < s.vw, v[e]);
        return;
    }
    const int r = row % (2 * s.n), d = r < s.n ? r : s.n - r;
    Acc *v = hv + (size_t)row * s.W;
    const int from = max(0, -d), to = min(s.vw, s.vw - d);   // live columns
    for (int x = threadIdx.x; x < from; x += blockDim.x) v[x] = Dead<Acc>::value();
    for (int x = max(to, from) + threadIdx.x; x < s.W; x += blockDim.x) v[x] = Dead<Acc>::value();
}

// The second of two different extreme polylines: the argmax of V_0 over the
// columns at least sep from the optimum's top vertex (nothing when there is no
// optimum), then its read-back by the last block.
template <typename Acc>
__global__ void __launch_bounds__(256) second_kernel(const __grid_constant__ ChainArgs args,
                                                     int sep, unsigned long long *key2,
                                                     int *done2, int32_t *x_out, int32_t *d_out,
                                                     Acc *score_out) {
    const ChainImg &im = args.one;
    const int D = 2 * im.n - 1;
    const unsigned long long k1 = *im.key;
    const int x0 = (int)((0xffffffffu - (unsigned)(k1 & 0xffffffffu)) / D);
    const Acc *V = band_rows<Acc>(im, 0);
    unsigned long long best = 0;
    if (k1 != 0)
        for (int e = blockIdx.x; e < D; e += gridDim.x) {
            const int d = e - (im.n - 1);
#pragma unroll 4
            for (int x = threadIdx.x; x < im.vw; x += blockDim.x) {
                if (abs(x - x0) < sep || !alive(im, 0, x, d)) continue;
                const Acc v = ld_cg(V + state_at(im, x, d));
                if (v == Dead<Acc>::value()) continue;
                const unsigned long long k = ((unsigned long long)vord(v) << 32) |
                                             (0xffffffffu - (unsigned)(x * D + e));
                best = best > k ? best : k;
            }
        }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long other = __shfl_xor_sync(0xffffffffu, best, o);
        best = best > other ? best : other;
    }
    if ((threadIdx.x & 31) == 0 && best) atomicMax(key2, best);
    __syncthreads();
    if (threadIdx.x >= 32) return;
    int finished = 0;
    if (threadIdx.x == 0) {
        __threadfence();
        finished = atomicAdd(done2, 1) == (int)gridDim.x - 1;
    }
    if (!__shfl_sync(0xffffffffu, finished, 0)) return;
    __threadfence();
    unsigned long long key = 0;
    if (threadIdx.x == 0) key = atomicAdd(key2, 0ull);
    key = __shfl_sync(0xffffffffu, key, 0);
    chain_readback<Acc>(im, args, key, x_out, d_out, score_out);
}

// fhtdp_backtrack has no workspace: one cluster of eight blocks finds the
// argmax of V_0 (its dead states hold dead values), folded through distributed
// shared memory, and its first warp reads the polyline back.
constexpr int kBtBlocks = 8, kBtNT = 1024;
template <typename Acc>
__global__ void __cluster_dims__(kBtBlocks, 1, 1) __launch_bounds__(kBtNT)
    backtrack_kernel(const __grid_constant__ ChainArgs args) {
    __shared__ unsigned long long s_warp[kBtNT / 32], s_block[kBtBlocks];
    const ChainImg &im = args.one;
    const int D = 2 * im.n - 1;
    // (the cluster barriers: every block runs before its shared memory is
    // written from another, and the blocks' maxima are there before they are read)
    auto cluster_sync = [] {
        asm volatile("barrier.cluster.arrive;\n barrier.cluster.wait;" ::: "memory");
    };
    cluster_sync();
    const Acc *V = band_rows<Acc>(im, 0);
    Acc top = Dead<Acc>::value();   // largest value, and the smallest index that holds it
    unsigned at = 0xffffffffu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // A warp takes a row, or a part of one where the rows are fewer than the warps,
    // with eight loads in flight.  300,000 columns, n = 2: a warp a row 1443 us
    // (int32; float 436), this 17; n = 16: 1486, 106; 100,000 columns, n = 128:
    // 1101, 323.
    constexpr int kWarps = kBtBlocks * kBtNT / 32, kFlight = 8;
    const int parts = max(kWarps / D, 1), len = (im.vw + parts - 1) / parts;
    for (int u = blockIdx.x * (kBtNT / 32) + warp; u < D * parts; u += kWarps) {
        const int e = u / parts, from = (u - e * parts) * len, to = min(from + len, im.vw);
        const int d = e - (im.n - 1);
        const Acc *row = V + (size_t)(d < 0 ? im.n - d : d) * im.pitch;
        for (int x0 = from + lane; x0 < to; x0 += 32 * kFlight) {
            Acc v[kFlight];
#pragma unroll
            for (int i = 0; i < kFlight; ++i)
                v[i] = ld_if(row + x0 + 32 * i, x0 + 32 * i < to, Dead<Acc>::value());
#pragma unroll
            for (int i = 0; i < kFlight; ++i) {   // (NaN loses every comparison)
                const unsigned k = (unsigned)((x0 + 32 * i) * D + e);
                if (v[i] > top || (v[i] == top && k < at)) {
                    top = v[i];
                    at = k;
                }
            }
        }
    }
    unsigned long long best = 0;
    if (top != Dead<Acc>::value())
        best = ((unsigned long long)vord(top) << 32) | (0xffffffffu - at);
    auto warp_max = [](unsigned long long k) {
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long other = __shfl_xor_sync(0xffffffffu, k, o);
            k = k > other ? k : other;
        }
        return k;
    };
    best = warp_max(best);
    if (lane == 0) s_warp[warp] = best;
    __syncthreads();
    if (warp == 0) {
        best = warp_max(s_warp[lane]);
        if (lane == 0) {
            uint32_t slot;
            asm volatile("mapa.shared::cluster.u32 %0, %1, 0;"
                         : "=r"(slot)
                         : "r"((uint32_t)__cvta_generic_to_shared(&s_block[blockIdx.x])));
            asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(slot), "l"(best) : "memory");
        }
    }
    __syncthreads();
    cluster_sync();
    if (blockIdx.x == 0 && warp == 0)
        chain_readback<Acc, true>(im, args, warp_max(lane < kBtBlocks ? s_block[lane] : 0ull),
                                  im.x_out, im.d_out, (Acc *)im.score_out);
}

// ---------------------------------------------------------------------------
// Host side.
int device_sms() {
    static std::atomic<int> cached[64];
    int dev = 0;
    cudaGetDevice(&dev);
    const bool known = dev >= 0 && dev < 64;
    int v = known ? cached[dev].load(std::memory_order_relaxed) : 0;
    if (v > 0) return v;
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    if (v < 1) v = 152;
    if (known) cached[dev].store(v, std::memory_order_relaxed);
    return v;
}

// Columns of a DP item: 2048 / n, so that 512 threads cover its displacements
// in runs of 8.
constexpr int chain_cols(int n) { return n >= 128 ? 16 : n <= 8 ? 256 : 2048 / n; }

size_t up256(size_t v) { return (v + 255) & ~(size_t)255; }

thread_local int g_skip_band = -1, g_skip_tile = -1;
thread_local long long g_skip_wait = 0;

void take_injection(ChainArgs &a) {
    a.wait_cycles = 4000000000LL;   // about two seconds
    a.skip_band = a.skip_tile = -1;
    if (g_skip_band >= 0) {
        a.skip_band = g_skip_band;
        a.skip_tile = g_skip_tile;
        a.wait_cycles = g_skip_wait;
    }
    g_skip_band = g_skip_tile = -1;
}

void chain_table(ChainArgs &a, const WindowTable &t) {
    a.use_table = 1;
    a.tab = t;
    a.minlen = 2 * t.n - 1;
    for (int i = 0; i < 2 * t.n - 1; ++i) {
        const int len = t.hi[i] - t.lo[i] + 1;
        a.minlen = len < a.minlen ? len : a.minlen;
    }
}

// Shared memory of an item of bands of n rows.
constexpr size_t item_bytes(int n, int cols, int use_table, int minlen, int B) {
    const int pad = window_pad(window_mode(use_table, minlen, B), use_table, B);
    return (size_t)(range_rows(n) + 2 * pad) * row_words(cols) * 4 * 2;
}
size_t item_smem(const ChainArgs &a, const ChainImg &im) {
    return item_bytes(im.n, im.cols, a.use_table, a.minlen, im.B);
}

// The dynamic shared memory that every launch allows its kernel: the largest
// that any image asks for.  The limit belongs to the kernel, not to a launch:
// were it set to a launch's own size, a host thread with a smaller image could
// lower it between another thread's call and launch, which is then refused.
// (What a block occupies is the launch's own size.)
constexpr int kFhtSmemMax = 226 * 1024, kDpSmemMax = 96 * 1024;
constexpr size_t most_item_bytes() {
    size_t most = 0;
    for (int n = 1; n <= 256; n *= 2)
        for (int B = 0; B <= 2 * n - 2; ++B)
            for (int table = 0; table < 2; ++table) {
                const size_t v = item_bytes(n, chain_cols(n), table, B + 1, B);
                most = v > most ? v : most;
            }
    return most;
}
static_assert(most_item_bytes() <= kDpSmemMax, "every item fits the limit");
template <typename Kernel>
int allow_smem(Kernel kern, int bytes) {
    return cuda_status(
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes),
        "cudaFuncSetAttribute");
}

// Blocks for one image whose band levels have t tiles.  A level can only use t,
// and blocks that wait for the next one slow those that share their SM: t of
// them, while there is an SM for each two (up to 2 t: the second takes the next
// level's item and loads its Hough values early), and beyond one an SM a
// multiple of half the SMs, so that the SMs are loaded evenly.  The whole chip (304)
// against this rule, whole calls: 2048 x 2048 uint8, n = 128 (t = 128) 130 ->
// 110 us and, from eight streams at once, 155 -> 91 us an image with the bend
// angle; float, n = 128, t = 188: 172 -> 160, t = 282: 392 -> 351 (282 x 32 bands);
// uint8, n = 64, t = 63: 193 -> 168 (t blocks: 173); n = 16, t = 4: 278 -> 270
// (t blocks: 339).
int one_image_blocks(int t) {
    const int sms = device_sms();
    if (2 * t <= sms) return 2 * t;
    if (t <= sms) return t;
    const int half = sms > 1 ? sms / 2 : 1;
    return t / half * half;
}

template <typename Acc, int kC, bool kLong>
int launch_chain(const ChainArgs &a, size_t smem, int blocks, bool dependent, cudaStream_t stream) {
    auto kern = dp_chain_kernel<Acc, kC, kLong>;
    int st = dependent ? FHTDP_OK : allow_smem(kern, kDpSmemMax);   // once a call
    if (st) return st;
    if (a.band < 0) {
        if (a.one.tiles) blocks = std::min(blocks, one_image_blocks(a.one.tiles));
        blocks = std::min(blocks, kDpPerSm * device_sms());
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kDpNT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = dependent ? 1 : 0;
    st = cuda_status(cudaLaunchKernelEx(&cfg, kern, a), "dp_chain_kernel");
    if (st) return st;
    return launched("dp_chain_kernel");
}
template <typename Acc, bool kLong>
int launch_chain_cols(const ChainArgs &a, int cols, size_t smem, int blocks, bool dependent,
                      cudaStream_t stream) {
    switch (cols) {
        case 0: return launch_chain<Acc, 0, kLong>(a, smem, blocks, dependent, stream);
        case 16: return launch_chain<Acc, 16, kLong>(a, smem, blocks, dependent, stream);
        case 32: return launch_chain<Acc, 32, kLong>(a, smem, blocks, dependent, stream);
        case 64: return launch_chain<Acc, 64, kLong>(a, smem, blocks, dependent, stream);
        case 128: return launch_chain<Acc, 128, kLong>(a, smem, blocks, dependent, stream);
        default: return launch_chain<Acc, 256, kLong>(a, smem, blocks, dependent, stream);
    }
}
// Whether kLong's kernel runs an image's windows.
bool long_windows(const ChainArgs &a, const ChainImg &im) {
    const int mode = window_mode(a.use_table, a.minlen, im.B);
    return mode == kShared || (a.use_table && mode == kScan);
}
template <typename Acc>
int launch_chain_cols(const ChainArgs &a, bool longw, int cols, size_t smem, int blocks,
                      bool dependent, cudaStream_t stream) {
    return longw ? launch_chain_cols<Acc, true>(a, cols, smem, blocks, dependent, stream)
                 : launch_chain_cols<Acc, false>(a, cols, smem, blocks, dependent, stream);
}

size_t fht_smem_bytes(int m, int T) { return (size_t)m * fht_pitch(m, T) * 4; }

// Columns of an FHT block: a block's time grows as T + 0.8 m (the passes sweep
// T + m - 4, T + m - 16, ... columns), one fits an SM (1,024 threads of 64
// registers), and the SM with the most blocks decides, so the T (a multiple of
// 16, at most 256) of the least product.  2048 x 2048 uint8, n = 128: T = 64, 128,
// 192, 256 took 46, 34, 44, 33 us (31 now); 1024 x 512, n = 64: T = 32, 64, 128, 256 17,
// 11.5, 15, 21; 512 x 2016, n = 32: T = 112, 240 15.8, 10.2; 8192 x 8192, n = 128:
// T = 128, 192, 256 296, 272, 243.  (Those registers are a few
// too few: 32 to 64 bytes a thread spill.)
int fht_columns(int m, int wout, int subs) {
    const int sms = device_sms();
    int best = 16;
    double least = 1e30;
    for (int T = 256; T >= 16; T -= 16) {
        if (fht_smem_bytes(m, T) > kFhtSmemMax) continue;
        const long long blocks = (long long)((wout + T - 1) / T) * subs;
        const double cost = (blocks + sms - 1) / sms * (T + 0.8 * m);   // on the busiest SM
        if (cost < least) {
            least = cost;
            best = T;
        }
    }
    return best;
}

FhtImg fht_img(const void *img, long long pitch, const Shape &s, int wout, void *out, int opitch) {
    FhtImg f{};
    f.img = img;
    f.pitch = pitch;
    f.w = s.w;
    f.W = s.W;
    f.wout = wout;
    f.n = s.n;
    f.m = s.n < 128 ? s.n : 128;
    while ((1 << f.log2m) < f.m) ++f.log2m;
    f.out = out;
    f.opitch = opitch;
    f.subs = s.h / f.m;
    return f;
}
void set_columns(FhtImg &f, int T) {
    f.T = T;
    f.tiles = (f.wout + T - 1) / T;
}

template <typename In, typename Acc>
int launch_fht_short(FhtImg f, cudaStream_t stream) {
    int bx = 32;   // columns of a block; narrow images: several bands
    while (bx < 256 && bx < f.wout) bx *= 2;
    set_columns(f, bx);
    const int by = 256 / bx;
    const unsigned grid = (unsigned)f.tiles * (unsigned)((f.subs + by - 1) / by);
    auto kern = f.m == 1   ? fht_short_kernel<In, Acc, 1>
                : f.m == 2 ? fht_short_kernel<In, Acc, 2>
                : f.m == 4 ? fht_short_kernel<In, Acc, 4>
                : f.m == 8 ? fht_short_kernel<In, Acc, 8>
                           : fht_short_kernel<In, Acc, 16>;
    kern<<<grid, dim3(bx, by), 0, stream>>>(f);
    return launched("fht_short_kernel");
}

template <typename In, typename Acc>
int launch_fht_img(FhtImg f, cudaStream_t stream) {
    if (f.m <= kShortRows) return launch_fht_short<In, Acc>(f, stream);
    set_columns(f, fht_columns(f.m, f.wout, f.subs));
    const long long blocks = (long long)f.tiles * f.subs;
    const size_t smem = fht_smem_bytes(f.m, f.T);
    auto kern = fht_band_kernel<In, Acc, false>;
    unsigned grid = (unsigned)blocks;
    if constexpr (sizeof(In) > 1) {
        // a block a sign while there is an SM for each (256 x 256 float, n = 128:
        // 20.8 -> 14.6 us; the passes over whole arrays took 16.7)
        if (2 * blocks <= device_sms()) {
            kern = fht_band_kernel<In, Acc, true>;
            grid *= 2;
        }
    }
    int st = allow_smem(kern, kFhtSmemMax);
    if (st) return st;
    kern<<<grid, kFhtNT, smem, stream>>>(f, nullptr, 1);
    return launched("fht_band_kernel");
}

}  // namespace

// The Hough rows of an image, columns [0, wout) of rows `opitch` apart, into
// hough; tmp (the same size) is needed for 256-row bands only, whose last level
// is a pass of its own.
template <typename In, typename Acc>
int launch_band_fht(const In *img, long long pitch, const Shape &s, int wout, Acc *hough, Acc *tmp,
                    int opitch, cudaStream_t stream) {
    Acc *first = s.n > 128 ? tmp : hough;
    // the last level reads columns modulo W
    int st = launch_fht_img<In, Acc>(fht_img(img, pitch, s, s.n > 128 ? s.W : wout, first, opitch),
                                     stream);
    if (!st && s.n > 128) st = launch_fht_last<Acc>(tmp, s, wout, hough, opitch, stream);
    return st;
}
template int launch_band_fht<uint8_t, int32_t>(const uint8_t *, long long, const Shape &, int,
                                               int32_t *, int32_t *, int, cudaStream_t);
template int launch_band_fht<int32_t, int32_t>(const int32_t *, long long, const Shape &, int,
                                               int32_t *, int32_t *, int, cudaStream_t);
template int launch_band_fht<float, float>(const float *, long long, const Shape &, int, float *,
                                           float *, int, cudaStream_t);

template <typename Acc>
int launch_dp_window(Acc *hv, const Shape &s, int B, const WindowTable *t, cudaStream_t stream) {
    const int copies = s.k * ((s.vw + kDeadCols - 1) / kDeadCols);
    dp_dead_kernel<Acc><<<(unsigned)(s.k * 2 * s.n + copies), kDeadNT, 0, stream>>>(hv, s);
    int st = launched("dp_dead_kernel");
    ChainArgs a{};
    a.one.hv = hv;
    a.one.n = s.n;
    a.one.k = s.k;
    a.one.vw = s.vw;
    a.one.pitch = s.W;
    a.one.B = B < 2 * s.n - 2 ? B : 2 * s.n - 2;
    a.one.cols = chain_cols(s.n);
    a.one.tiles = (s.vw + a.one.cols - 1) / a.one.cols;
    a.skip_band = a.skip_tile = -1;
    a.store0 = 1;
    if (t) chain_table(a, *t);
    const size_t smem = item_smem(a, a.one);
    for (int b = s.k - 2; b >= 0 && !st; --b) {
        a.band = b;
        st = launch_chain_cols<Acc>(a, long_windows(a, a.one), a.one.cols, smem, a.one.tiles,
                                    b != s.k - 2, stream);
    }
    return st;
}
template int launch_dp_window<int32_t>(int32_t *, const Shape &, int, const WindowTable *,
                                       cudaStream_t);
template int launch_dp_window<float>(float *, const Shape &, int, const WindowTable *,
                                     cudaStream_t);

template <typename Acc>
int launch_backtrack(const Acc *V, const Shape &s, int B, const WindowTable *t, int32_t *x_out,
                     int32_t *d_out, Acc *score_out, cudaStream_t stream) {
    ChainArgs a{};
    a.one.hv = const_cast<Acc *>(V);
    a.one.n = s.n;
    a.one.k = s.k;
    a.one.vw = s.vw;
    a.one.pitch = s.W;
    a.one.B = B < 2 * s.n - 2 ? B : 2 * s.n - 2;
    a.one.x_out = x_out;
    a.one.d_out = d_out;
    a.one.score_out = score_out;
    if (t) chain_table(a, *t);
    backtrack_kernel<Acc><<<kBtBlocks, kBtNT, 0, stream>>>(a);
    return launched("backtrack_kernel");
}
template int launch_backtrack<int32_t>(const int32_t *, const Shape &, int, const WindowTable *,
                                       int32_t *, int32_t *, int32_t *, cudaStream_t);
template int launch_backtrack<float>(const float *, const Shape &, int, const WindowTable *,
                                     int32_t *, int32_t *, float *, cudaStream_t);

void chain_inject(int band, int tile, long long wait_cycles) {
    g_skip_band = band;
    g_skip_tile = tile;
    g_skip_wait = wait_cycles;
}

ChainLayout chain_layout(const Shape &s, bool smooth, bool tight) {
    ChainLayout L{};
    L.cols = chain_cols(s.n);
    L.tiles = (s.vw + L.cols - 1) / L.cols;
    // rows a multiple of 128 bytes apart; those of 256-row bands hold the cyclic
    // width.  Tight: no padding, the keys in the head, and with 256-row bands the
    // flags in `second`, which the FHT leaves free: no more than the method's own
    // two arrays, which every call accepted before its rows were padded.
    L.pitch = s.n > 128 ? s.W : s.vw;
    if (!tight) L.pitch = (L.pitch + 31) & ~31;
    auto up = [tight](size_t v) { return tight ? (v + 15) & ~(size_t)15 : up256(v); };
    size_t o = sizeof(ChainCtl);
    L.key = tight ? o - 64 : o;   // key, done; key, done of the second polyline
    if (!tight) o += 256;
    L.late = tight && s.n > 128;
    L.flag_bytes = (size_t)s.k * L.tiles * 4;
    L.flags = o;
    if (!L.late) o = up(o + L.flag_bytes);
    L.zero = o;
    const size_t rows = up((size_t)s.k * 2 * s.n * L.pitch * 4);
    L.rows = o;
    o += rows;
    L.second = o;
    if (L.late) L.flags = o;
    if (s.n > 128) o += rows;
    else if (smooth) o = up(o + (size_t)s.h * s.w * 4);
    L.total = o;
    return L;
}

namespace {
template <typename In, typename Acc>
int chain_detect_t(const In *img, int pitch, const Shape &s, const ChainQuery &q, int32_t *x_out,
                   int32_t *d_out, Acc *score_out, char *ws, cudaStream_t stream) {
    const ChainLayout L = chain_layout(s, q.r > 0, q.tight);
    int st = cuda_status(cudaMemsetAsync(ws, 0, L.zero, stream), "cudaMemsetAsync");
    Acc *rows = (Acc *)(ws + L.rows), *second = (Acc *)(ws + L.second);
    if (st) return st;
    if (q.r > 0) {
        // the smoothed image: where the rows will be (256-row bands, whose
        // first pass writes `second`), else in `second`
        Acc *smooth = s.n > 128 ? rows : second;
        st = launch_gauss_rows<In, Acc>(img, pitch, s.h, s.w, q.r, smooth, stream);
        if (!st)
            st = launch_band_fht<Acc, Acc>(smooth, s.w, s, s.vw, rows, second, L.pitch, stream);
    } else {
        st = launch_band_fht<In, Acc>(img, pitch, s, s.vw, rows, second, L.pitch, stream);
    }
    if (!st && L.late)
        st = cuda_status(cudaMemsetAsync(ws + L.flags, 0, L.flag_bytes, stream), "cudaMemsetAsync");
    if (st) return st;
    ChainArgs a{};
    ChainImg &im = a.one;
    im.hv = rows;
    im.n = s.n;
    im.k = s.k;
    im.vw = s.vw;
    im.pitch = L.pitch;
    im.B = q.B < 2 * s.n - 2 ? q.B : 2 * s.n - 2;
    im.cols = L.cols;
    im.tiles = L.tiles;
    im.flags = (int *)(ws + L.flags);
    im.key = (unsigned long long *)(ws + L.key);
    im.done = (int *)(ws + L.key + 8);
    im.x_out = x_out;
    im.d_out = d_out;
    im.score_out = score_out;
    if (q.point) {
        im.mask1 = (q.point->j < s.k ? q.point->j : s.k - 1) + 1;
        im.mask_x = q.point->xp;
        im.mask_end = q.point->j == s.k ? 1 : 0;
    }
    a.items = L.tiles * (s.k > 1 ? s.k - 1 : 1);
    a.ctl = (ChainCtl *)ws;
    a.report = q.report;
    take_injection(a);
    a.band = -1;
    a.store0 = q.sep > 0;
    if (q.table) chain_table(a, *q.table);
    st = launch_chain_cols<Acc>(a, long_windows(a, im), im.cols, item_smem(a, im), a.items, false,
                                stream);
    if (!st && q.sep > 0) {
        const int D = 2 * s.n - 1;
        second_kernel<Acc><<<D, 256, 0, stream>>>(
            a, q.sep, (unsigned long long *)(ws + L.key + 16), (int *)(ws + L.key + 24),
            x_out + s.k + 1, d_out + s.k, score_out + 1);
        st = launched("second_kernel");
    }
    return st;
}
}  // namespace

// ---------------------------------------------------------------------------
// Batches.  Workspace: [head][flags, key and done of every image][FHT table]
// [image table][queue][rows of every image]; the first two parts are cleared by
// every run.
struct ChainBatch {
    int dtype;
    std::vector<ChainImage> images;
    std::vector<FhtImg> fht;         // as uploaded
    std::vector<ChainImg> imgs;
    std::vector<ChainItem> order;
    std::vector<size_t> flags, keys, rows;   // offsets
    size_t zero = 0, fht_off = 0, img_off = 0, order_off = 0, total = 0, fht_smem = 0;
    int fht_blocks = 0, cols = 0;    // cols 0: several tile widths
};

ChainBatch *chain_batch_create(const std::vector<ChainImage> &images, int dtype) {
    ChainBatch *b = new (std::nothrow) ChainBatch();
    if (!b) return nullptr;
    b->dtype = dtype;
    b->images = images;
    size_t o = sizeof(ChainCtl);
    struct Level {
        double when;
        int image, lv;
    };
    std::vector<Level> levels;
    for (const ChainImage &c : images) {
        const int i = (int)b->imgs.size();
        ChainImg im{};
        im.n = c.s.n;
        im.k = c.s.k;
        im.vw = c.s.vw;
        im.pitch = (c.s.vw + 31) & ~31;
        im.B = c.B < 2 * c.s.n - 2 ? c.B : 2 * c.s.n - 2;
        im.cols = chain_cols(c.s.n);
        im.tiles = (c.s.vw + im.cols - 1) / im.cols;
        im.x_out = c.x_out;
        im.d_out = c.d_out;
        im.score_out = c.score_out;
        b->cols = i == 0 ? im.cols : b->cols == im.cols ? im.cols : 0;
        b->keys.push_back(o);
        o += 16;
        b->flags.push_back(o);
        o = (o + (size_t)im.k * im.tiles * 4 + 15) & ~(size_t)15;
        FhtImg f = fht_img(c.img, c.pitch, c.s, c.s.vw, nullptr, im.pitch);
        set_columns(f, std::min(256, (c.s.vw + 15) & ~15));   // the least work a column
        f.item0 = b->fht_blocks;
        b->fht_blocks += f.tiles * f.subs;
        b->fht_smem = std::max(b->fht_smem, fht_smem_bytes(f.m, f.T));
        b->imgs.push_back(im);
        b->fht.push_back(f);
        const int L = std::max(im.k - 1, 1);
        for (int lv = 0; lv < L; ++lv) levels.push_back(Level{(lv + 0.5) / L, i, lv});
    }
    // Queue: every image's band levels in proportion to their number, so that
    // all chains begin and end together and each level's wait is covered by the
    // other images' items.
    std::stable_sort(levels.begin(), levels.end(),
                     [](const Level &x, const Level &y) { return x.when < y.when; });
    for (const Level &l : levels) {
        const ChainImg &im = b->imgs[l.image];
        for (int t = 0; t < im.tiles; ++t)
            b->order.push_back(ChainItem{l.image, std::max(im.k - 2 - l.lv, 0), t, 0});
    }
    b->zero = o = up256(o);
    b->fht_off = o;
    o = up256(o + b->fht.size() * sizeof(FhtImg));
    b->img_off = o;
    o = up256(o + b->imgs.size() * sizeof(ChainImg));
    b->order_off = o;
    o = up256(o + b->order.size() * sizeof(ChainItem));
    for (const ChainImg &im : b->imgs) {
        b->rows.push_back(o);
        o = up256(o + (size_t)im.k * 2 * im.n * im.pitch * 4);
    }
    b->total = o;
    return b;
}
void chain_batch_destroy(ChainBatch *b) { delete b; }
size_t chain_batch_bytes(const ChainBatch *b) { return b->total; }
long long chain_batch_items(const ChainBatch *b) { return (long long)b->order.size(); }
long long chain_batch_width(const ChainBatch *b) {
    long long tiles = 0;
    for (const ChainImg &im : b->imgs) tiles += im.tiles;
    return tiles;
}
int chain_batch_tile(const ChainBatch *b, int n) {
    for (const ChainImg &im : b->imgs)
        if (im.n == n) return im.cols;
    return 0;
}

int chain_batch_upload(ChainBatch *b, void *ws, cudaStream_t stream) {
    char *W = (char *)ws;
    for (size_t i = 0; i < b->imgs.size(); ++i) {
        b->fht[i].out = b->imgs[i].hv = W + b->rows[i];
        b->imgs[i].flags = (int *)(W + b->flags[i]);
        b->imgs[i].key = (unsigned long long *)(W + b->keys[i]);
        b->imgs[i].done = (int *)(W + b->keys[i] + 8);
    }
    auto put = [&](size_t off, const void *src, size_t bytes) {
        return cuda_status(cudaMemcpyAsync(W + off, src, bytes, cudaMemcpyHostToDevice, stream),
                           "cudaMemcpyAsync");
    };
    int st = put(b->fht_off, b->fht.data(), b->fht.size() * sizeof(FhtImg));
    if (!st) st = put(b->img_off, b->imgs.data(), b->imgs.size() * sizeof(ChainImg));
    if (!st) st = put(b->order_off, b->order.data(), b->order.size() * sizeof(ChainItem));
    return st;
}

namespace {
template <typename Acc>
int chain_batch_run_t(const ChainBatch *b, char *ws, const WindowTable *t, cudaStream_t stream) {
    int st = allow_smem(fht_band_kernel<Acc, Acc, false>, kFhtSmemMax);
    if (st) return st;
    fht_band_kernel<Acc, Acc, false><<<(unsigned)b->fht_blocks, kFhtNT, b->fht_smem, stream>>>(
        b->fht[0], (const FhtImg *)(ws + b->fht_off), (int)b->fht.size());
    st = launched("fht_band_kernel");
    if (st) return st;
    ChainArgs a{};
    a.many = (const ChainImg *)(ws + b->img_off);
    a.order = (const ChainItem *)(ws + b->order_off);
    a.items = (int)b->order.size();
    a.ctl = (ChainCtl *)ws;
    take_injection(a);
    a.band = -1;
    if (t) chain_table(a, *t);
    size_t smem = 0;
    bool longw = true;   // all images alike
    for (const ChainImg &im : b->imgs) {
        smem = std::max(smem, item_smem(a, im));
        longw = longw && long_windows(a, im);
    }
    return launch_chain_cols<Acc>(a, longw, b->cols, smem, a.items, false, stream);
}
}  // namespace

int chain_batch_clear(const ChainBatch *b, void *ws, cudaStream_t stream) {
    return cuda_status(cudaMemsetAsync(ws, 0, b->zero, stream), "cudaMemsetAsync");
}

int chain_batch_run(const ChainBatch *b, void *ws, const WindowTable *t, cudaStream_t stream) {
    return b->dtype == FHTDP_F32 ? chain_batch_run_t<float>(b, (char *)ws, t, stream)
                                 : chain_batch_run_t<int32_t>(b, (char *)ws, t, stream);
}

int chain_detect(const void *img, int dtype, int pitch, const Shape &s, const ChainQuery &q,
                 int32_t *x_out, int32_t *d_out, void *score_out, void *ws, cudaStream_t stream) {
    if (dtype == FHTDP_U8)
        return chain_detect_t<uint8_t, int32_t>((const uint8_t *)img, pitch, s, q, x_out, d_out,
                                                (int32_t *)score_out, (char *)ws, stream);
    if (dtype == FHTDP_I32)
        return chain_detect_t<int32_t, int32_t>((const int32_t *)img, pitch, s, q, x_out, d_out,
                                                (int32_t *)score_out, (char *)ws, stream);
    return chain_detect_t<float, float>((const float *)img, pitch, s, q, x_out, d_out,
                                        (float *)score_out, (char *)ws, stream);
}

}  // namespace fhtdp
