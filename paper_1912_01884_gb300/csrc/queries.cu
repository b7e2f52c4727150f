// Queries on one image, host side only.
//
// Subproblems 2-3 (Sec. 2.2-2.3): the extreme polyline through a given point
// P on a band border.
// The paper builds the part below P by the DP over bands j..k-1 and the part
// above P by the same DP on bands 0..j-1 flipped about Ox.  Here one DP runs
// over all bands and treats every state of P's band whose vertex on P's
// border is not xp as dead, so the optimum over V_0 is the best polyline
// through P with the bend limit at every vertex, P included, and the usual
// read-back (Eq. 5) returns it.
#include "chain.cuh"

namespace fhtdp {

// Through-point, padded and two-polyline queries share the size: vertices in
// [0, w) or in [0, W).
size_t through_workspace_bytes(const Shape &s) {
    Shape padded = s;
    padded.vw = s.W;
    const size_t a = chain_layout(s, false).total, b = chain_layout(padded, false).total;
    return a > b ? a : b;
}

// Vertices anywhere in the zero-padded band width (Sec. 2.2: Hough columns
// up to w + h/k - 1).  The cyclic FHT never wraps for a link with both ends
// in [0, W), so its values are the plain sums with zeros right of the image;
// the DP and the read-back run over the vertex domain s.vw = W.
int detect_padded(const void *img, int dtype, int pitch, const Shape &s, int B, int32_t *x_out,
                  int32_t *d_out, void *score_out, void *ws, bool tight, cudaStream_t stream) {
    ChainQuery q;
    q.tight = tight;
    q.B = B;
    return chain_detect(img, dtype, pitch, s, q, x_out, d_out, score_out, ws, stream);
}

// Two different extreme polylines (Sec. 3, Figs. 6d and 7a; the paper gives
// no rule): the optimum, then the best polyline whose top vertex lies at
// least sep columns from the optimum's, both read back from the same V.
int detect_two(const void *img, int dtype, int pitch, const Shape &s, int B, int sep,
               int32_t *x_out, int32_t *d_out, void *score_out, void *ws, bool tight,
               cudaStream_t stream) {
    ChainQuery q;
    q.tight = tight;
    q.B = B;
    q.sep = sep;
    return chain_detect(img, dtype, pitch, s, q, x_out, d_out, score_out, ws, stream);
}

}  // namespace fhtdp
