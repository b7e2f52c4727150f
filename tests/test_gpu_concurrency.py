"""Calls of different sizes beside each other: from two host threads, and in one
CUDA graph.  Results are the oracle's, so a launch that another call's sizes
disturbed shows up as a status or as a wrong polyline."""
import threading

import numpy as np
import pytest

import oracle
from helpers import to_device

pytestmark = pytest.mark.gpu


def _img(h, w, dtype, seed):
    rng = np.random.default_rng(seed)
    if dtype == "f32":
        return np.abs(rng.standard_normal((h, w))).astype(np.float32)
    return rng.integers(0, 256, (h, w)).astype(np.uint8 if dtype == "u8" else np.int32)


# (h, w, k, B): the largest and the smallest shared memory of the FHT and of the
# DP with the same code (16 columns an item: bands of 128 and 256 rows).
_SIZES = {"large": (256, 300, 2, 24), "small": (256, 40, 1, 0), "long": (512, 130, 2, 200),
          "short": (16, 64, 4, 1)}


def _detect(img, k, B):
    return oracle.detect_f32(img, k, B) if img.dtype == np.float32 else oracle.detect(img, k, B)


@pytest.mark.parametrize("dtype", ["u8", "i32", "f32"])
@pytest.mark.parametrize("pair", [("large", "small"), ("long", "large"), ("large", "short")])
def test_two_threads_with_different_sizes(lib, dtype, pair):
    import torch
    jobs, errors = [], []
    for name in pair:
        h, w, k, B = _SIZES[name]
        img = _img(h, w, dtype, len(name))
        jobs.append((to_device(img), k, B, _detect(img, k, B), torch.cuda.Stream()))
    torch.cuda.synchronize()
    start = threading.Barrier(2)

    def work(img, k, B, want, stream):
        try:
            start.wait(60)
            with torch.cuda.stream(stream):
                for r in range(300):
                    got = lib.detect_polyline(img, k, B, stream=stream)
                    H = lib.fht_bands(img, k, stream=stream)
                    if r % 50 == 0:
                        x, d, s = (t.cpu().numpy() for t in got)
                        assert list(x) == list(want[0]) and list(d) == list(want[1])
                        assert s[0] == s.dtype.type(want[2])
                del H
            stream.synchronize()
        except Exception as e:   # noqa: BLE001 (handed to the test's thread)
            errors.append(e)

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


@pytest.mark.parametrize("dtype", ["u8", "f32"])
def test_one_graph_holds_calls_of_two_sizes(lib, dtype):
    """detect_polyline of a large and of a small image, and the layer calls (the
    DP's launches depend on each other programmatically), captured in one
    graph that is replayed after the inputs changed."""
    import torch
    sizes = [_SIZES["large"], _SIZES["small"], _SIZES["long"]]
    first = [to_device(_img(h, w, dtype, 3)) for h, w, _, _ in sizes]

    def calls():
        out = []
        for img, (h, w, k, B) in zip(first, sizes):
            out.append(lib.detect_polyline(img, k, B))
            V = lib.polyline_dp(lib.fht_bands(img, k), h, w, k, B)
            out.append(lib.backtrack(V, h, w, k, B))
        return out

    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        calls()
    side.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = calls()
    for seed in (11, 12):
        want = []
        for img, (h, w, k, B) in zip(first, sizes):
            new = _img(h, w, dtype, seed)
            img.copy_(torch.from_numpy(new))
            want += 2 * [_detect(new, k, B)]
        graph.replay()
        torch.cuda.synchronize()
        for (x, d, s), (xo, do, so) in zip(out, want):
            assert x.tolist() == list(xo) and d.tolist() == list(do)
            assert s.cpu().numpy()[0] == s.cpu().numpy().dtype.type(so)
