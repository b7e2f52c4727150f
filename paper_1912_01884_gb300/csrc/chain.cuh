// Band FHT in one pass and the DP chain over stored Hough rows (chain.cu).
#pragma once

#include <vector>

#include "common.cuh"

namespace fhtdp {

// Head of a workspace that the chain runs on; the first word after `queue` is
// the status that fhtdp_workspace_status reads.
struct ChainCtl {
    int queue, status;
    int pad[62];   // (the last 64 bytes: the keys of a tight layout)
};

// One image: its Hough rows / DP values and its outputs.
struct ChainImg {
    void *hv;                  // [k][2][n][pitch] 4-byte values
    int n, k, vw, pitch, B;    // vertices in [0, vw); B the bend limit (clamped to 2n - 2)
    int cols, tiles;           // columns of a tile, tiles of a band
    int *flags;                // [k][tiles] publication flags (null: bands run one launch each)
    unsigned long long *key;   // argmax of V_0
    int *done;                 // band-0 tiles finished
    int32_t *x_out, *d_out;
    void *score_out;
    // Subproblems 2-3: with mask1 > 0 the states of band mask1 - 1 whose vertex
    // on the point's border (mask_end: the link's end, else its start) is not
    // column mask_x are dead.
    int mask1, mask_x, mask_end;
};

// One image's Hough rows: bands of n rows of img into out, columns [0, wout).
struct FhtImg {
    const void *img;
    long long pitch;
    int w, W, wout;      // image width, cyclic width w + n, columns to write
    int n, m, log2m;     // band height; sub-bands of m = min(n, 128) rows are merged
    void *out;           // [k][2][n][opitch], row j * m + s for sub-band j, shift s
    int opitch, T, tiles, subs;   // T columns a block (a multiple of 16)
    int item0;           // first block of this image in a launch of several
};

// Workspace of a single-image run: [head][key, done][flags][rows][second].
struct ChainLayout {
    size_t key, flags, rows, second, zero, total, flag_bytes;
    int pitch, cols, tiles;
    bool late;   // the flags lie in `second` and are cleared after the FHT
};
// smooth: the image is smoothed first (angle queries, r > 0).  tight: the least
// workspace that is accepted.
ChainLayout chain_layout(const Shape &s, bool smooth, bool tight = false);

struct ChainQuery {
    int B = 0;                          // bend limit
    const WindowTable *table = nullptr; // or window table
    const PointMask *point = nullptr;
    int r = 0;                          // smoothing half-width
    int sep = 0;                        // > 0: also the second polyline
    bool tight = false;                 // the layout of chain_layout(.., tight)
    int *report = nullptr;              // a second place for the run's status
};
// FHT (after smoothing), DP and read-back of one image on workspace ws of at
// least chain_layout().total bytes.
int chain_detect(const void *img, int dtype, int pitch, const Shape &s, const ChainQuery &q,
                 int32_t *x_out, int32_t *d_out, void *score_out, void *ws, cudaStream_t stream);

// A batch of int32 or float images (bands of at most 128 rows): all their
// FHTs in one launch, all their DP items in one more.
struct ChainImage {
    const void *img;
    long long pitch;
    Shape s;
    int B;
    int32_t *x_out, *d_out;
    void *score_out;
};
struct ChainBatch;
ChainBatch *chain_batch_create(const std::vector<ChainImage> &images, int dtype);
void chain_batch_destroy(ChainBatch *b);
size_t chain_batch_bytes(const ChainBatch *b);
long long chain_batch_items(const ChainBatch *b);
// The tiles of a band level over all images, and the columns of the DP items of
// band height n (0: no such image).
long long chain_batch_width(const ChainBatch *b);
int chain_batch_tile(const ChainBatch *b, int n);
// The batch's tables for workspace ws (from host memory held by the batch).
int chain_batch_upload(ChainBatch *b, void *ws, cudaStream_t stream);
// A run: the clearing of its head, then the launches.  t (optional): bend-angle
// windows for all images (one band height).
int chain_batch_clear(const ChainBatch *b, void *ws, cudaStream_t stream);
int chain_batch_run(const ChainBatch *b, void *ws, const WindowTable *t, cudaStream_t stream);

// The next chain run of this thread never publishes tile `tile` of band
// `band`, and its waits give up after `wait_cycles` (band < 0: none).
void chain_inject(int band, int tile, long long wait_cycles);

}  // namespace fhtdp
