"""The row-chain convolutions and the first layer at their edges: fewer rows
than the dilation, pieces of one row, odd pieces (a step of the weight gradient
with one row), rows that end inside a segment, more rows than CTAs, unaligned
buffers.  Tolerances as for the other layers: bf16 outputs within two roundings
(2^-7 of the value, and of the largest term for sums near zero), FP32 gradients
within 1e-3 of the value and 1e-2."""
import ctypes

import numpy as np
import pytest

from oracle import cnn_ref

pytestmark = pytest.mark.gpu


def _bf16(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(torch.bfloat16)


def _np(t):
    return t.float().cpu().numpy().astype(np.float64)


def _stream():
    import torch
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


def _close(got, want):
    assert np.all(np.abs(got - want) <= 2.0 ** -7 * np.abs(want) + 3e-2)


@pytest.mark.parametrize("N,H,W,dil", [(1, 1, 64, 1), (1, 3, 64, 8), (2, 8, 128, 8), (1, 40, 192, 4),
                                       (3, 33, 320, 3), (2, 200, 128, 1), (1, 129, 64, 2)])
def test_row_chains_match_reference(lib, N, H, W, dil):
    import torch
    L = lib.lib()
    rng = np.random.default_rng(N + H + W + dil)
    x, dz = _bf16(rng.standard_normal((N, H, W, 32))), _bf16(rng.standard_normal((N, H, W, 32)) * 0.5)
    w, b = _bf16(rng.standard_normal((288, 32)) * 0.1), rng.standard_normal(32).astype(np.float32)
    xd, dzd, wd, bd = x.cuda(), dz.cuda(), w.cuda(), torch.from_numpy(b).cuda()
    y, dx = torch.empty_like(xd), torch.empty_like(xd)
    wf = torch.empty(9216, dtype=torch.bfloat16, device="cuda")
    dw, db = torch.zeros(288, 32, device="cuda"), torch.zeros(32, device="cuda")
    assert L.fhtdp_cnn_status(1) == 0
    assert L.fhtdp_cnn_conv3x3(xd.data_ptr(), 32, N, H, W, dil, wd.data_ptr(), bd.data_ptr(), 1,
                               y.data_ptr(), _stream()) == 0
    assert L.fhtdp_cnn_conv3x3_dgrad(dzd.data_ptr(), N, H, W, dil, wd.data_ptr(), wf.data_ptr(),
                                     dx.data_ptr(), _stream()) == 0
    assert L.fhtdp_cnn_conv3x3_wgrad(xd.data_ptr(), 32, N, H, W, dil, dzd.data_ptr(), dw.data_ptr(),
                                     db.data_ptr(), _stream()) == 0
    assert L.fhtdp_cnn_status(0) == 0
    w64 = _np(w).reshape(9, 32, 32)
    _close(_np(y), np.maximum(cnn_ref.conv3x3(_np(x), w64, b.astype(np.float64), dil), 0))
    _close(_np(dx), cnn_ref.conv3x3_dgrad(_np(dz), w64, dil))
    rw, rb = cnn_ref.conv3x3_wgrad(_np(x), _np(dz), dil)
    assert np.allclose(dw.cpu().numpy().reshape(9, 32, 32), rw, rtol=1e-3, atol=1e-2)
    assert np.allclose(db.cpu().numpy(), rb, rtol=1e-3, atol=1e-2)


@pytest.mark.parametrize("N,H,W,dil,shift", [(1, 1, 64, 1, 0), (2, 9, 128, 8, 1), (1, 70, 64, 3, 0)])
def test_first_layer_and_head_on_any_alignment(lib, N, H, W, dil, shift):
    """`shift` bf16 values between the buffers and a 16-byte boundary."""
    import torch
    L = lib.lib()
    rng = np.random.default_rng(H + dil)

    def place(a):
        flat = torch.zeros(a.numel() + 8, dtype=torch.bfloat16, device="cuda")
        view = flat[shift:shift + a.numel()].view(a.shape)
        view.copy_(a)
        return view

    x = _bf16(rng.standard_normal((N, H, W, 1)))
    w = np.zeros((16, 32))
    w[:9] = rng.standard_normal((9, 32)) * 0.3
    wb, dz = _bf16(w), _bf16(rng.standard_normal((N, H, W, 32)))
    xd, wd, dzd, y = place(x), place(wb), place(dz), place(torch.zeros_like(dz))
    dw, db = torch.zeros(16, 32, device="cuda"), torch.zeros(32, device="cuda")
    assert L.fhtdp_cnn_conv3x3(xd.data_ptr(), 1, N, H, W, dil, wd.data_ptr(), None, 0, y.data_ptr(),
                               _stream()) == 0
    assert L.fhtdp_cnn_conv3x3_wgrad(xd.data_ptr(), 1, N, H, W, dil, dzd.data_ptr(), dw.data_ptr(),
                                     db.data_ptr(), _stream()) == 0
    _close(_np(y), cnn_ref.conv3x3(_np(x), _np(wb)[:9].reshape(9, 1, 32), np.zeros(32), dil))
    rw, rb = cnn_ref.conv3x3_wgrad(_np(x), _np(dz), dil)
    assert np.allclose(dw.cpu().numpy()[:9], rw[:, 0], rtol=1e-3, atol=1e-2)
    assert np.all(dw.cpu().numpy()[9:] == 0) and np.allclose(db.cpu().numpy(), rb, rtol=1e-3, atol=1e-2)
    # the head: one band of H rows
    labels = rng.integers(0, 32, (N, 1)).astype(np.int32)
    dl, loss = place(torch.zeros_like(dz)), torch.zeros(1, device="cuda")
    pred = torch.zeros(N, dtype=torch.int32, device="cuda")
    lab = torch.from_numpy(labels).cuda()
    assert L.fhtdp_cnn_band_head(dzd.data_ptr(), N, H, W, 1, lab.data_ptr(), 1.0 / N, dl.data_ptr(),
                                 loss.data_ptr(), pred.data_ptr(), _stream()) == 0
    _, rl, rdz, rpred = cnn_ref.band_head(_np(dz), 1, labels)
    assert np.array_equal(pred.cpu().numpy(), np.asarray(rpred).reshape(-1))
    assert abs(float(loss) - rl) <= 1e-4 * abs(rl)
    assert np.all(np.abs(_np(dl) - rdz) <= 2.0 ** -7 * np.abs(rdz) + 1e-6)


# Weights at any 2-byte address (a view into a flat parameter buffer), `shift`
# bf16 values past a 16-byte boundary: the same sums, so the same bits.
@pytest.mark.parametrize("shift", [1, 2, 3, 4, 6, 7])
def test_row_chains_take_weights_at_any_address(lib, shift):
    import torch
    L = lib.lib()
    N, H, W, dil = 1, 9, 128, 2
    rng = np.random.default_rng(shift)
    x, w = _bf16(rng.standard_normal((N, H, W, 32))).cuda(), _bf16(rng.standard_normal(9216) * 0.1)
    b = torch.from_numpy(rng.standard_normal(32).astype(np.float32)).cuda()
    flat = torch.zeros(9216 + 8, dtype=torch.bfloat16, device="cuda")
    wf = torch.empty(9216, dtype=torch.bfloat16, device="cuda")
    got = []
    for at in (0, shift):
        wd = flat[at:at + 9216]
        wd.copy_(w)
        y, dx = torch.empty_like(x), torch.empty_like(x)
        assert L.fhtdp_cnn_conv3x3(x.data_ptr(), 32, N, H, W, dil, wd.data_ptr(), b.data_ptr(), 1,
                                   y.data_ptr(), _stream()) == 0
        assert L.fhtdp_cnn_conv3x3_dgrad(x.data_ptr(), N, H, W, dil, wd.data_ptr(), wf.data_ptr(),
                                         dx.data_ptr(), _stream()) == 0
        got.append((y.view(torch.int16).cpu(), dx.view(torch.int16).cpu()))
    w64 = _np(w).reshape(9, 32, 32)
    _close(_np(got[0][0].view(torch.bfloat16)),
           np.maximum(cnn_ref.conv3x3(_np(x), w64, _np(b), dil), 0))
    for p, q in zip(*got):
        assert torch.equal(p, q)
