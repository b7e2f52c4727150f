"""Single uint8 images on both sides of the rule that sends them to the engine or
to the chain (one band, wide images, bend limits, rows that TMA cannot copy):
every route returns the oracle's polyline."""
import numpy as np
import pytest

import oracle
from helpers import to_device

pytestmark = pytest.mark.gpu


def _img(h, w, seed):
    return np.random.default_rng(seed).integers(0, 256, (h, w)).astype(np.uint8)


def _same(got, want):
    x, d, s = (t.cpu().numpy() for t in got)
    assert list(x) == list(want[0]) and list(d) == list(want[1]) and s[0] == want[2]


# (n, k, w): the widths at which the rule changes, one column less, odd ones.
_SHAPES = [(1, 1, 700), (2, 1, 3), (8, 1, 65535), (8, 1, 65536), (16, 1, 2048), (32, 1, 37),
           (64, 1, 320), (64, 1, 321), (128, 1, 320), (128, 1, 321), (256, 1, 320), (256, 1, 321),
           (32, 2, 10239), (32, 2, 10240), (32, 3, 19456), (64, 2, 14336), (64, 4, 24575),
           (64, 4, 24576), (128, 2, 6656), (128, 3, 9217), (128, 2, 13313), (256, 2, 3072),
           (256, 2, 3073), (256, 4, 7168)]


@pytest.mark.parametrize("n,k,w", _SHAPES)
def test_detect_on_both_sides_of_the_rule(lib, n, k, w):
    img = _img(n * k, w, n + k + w)
    dev = to_device(img)
    for B in (4, 5, 16) if n < 256 else (4, 16, 33):
        _same(lib.detect_polyline(dev, k, B), oracle.detect(img, k, B))


@pytest.mark.parametrize("n,k,w", [s for s in _SHAPES if s[1] > 1])
def test_through_a_point_on_both_sides_of_the_rule(lib, n, k, w):
    img = _img(n * k, w, n + k + w + 1)
    dev = to_device(img)
    for j, xp in ((0, w // 2), (1, w - 1), (k, 0)):
        _same(lib.detect_through_point(dev, k, 16, j, xp), oracle.detect_through(img, k, 16, j, xp))


def test_rows_of_a_wider_array_and_the_route_by_alignment(lib):
    """The same wide image at every byte offset: TMA rows, and rows that go the
    other way."""
    import torch
    img = _img(256, 6700, 5)
    want = oracle.detect(img, 2, 16)
    for off in (0, 1, 8, 16):
        wide = torch.zeros((256, 6752), dtype=torch.uint8, device="cuda")
        wide[:, off:off + 6700] = to_device(img)
        _same(lib.detect_polyline(wide[:, off:off + 6700], 2, 16), want)
