"""Exact 3x3 convolutions of stride 2 on the tensor cores at the edges of their tiles: forward with residual and statistics,
data gradient with a gated residual; against the oracle (operands and results in bfloat16: one unit of the largest element is
4e-3, a sum taken in another order moves a result by one)."""
import numpy as np
import pytest
import torch

from oracle import layers as L

pytestmark = pytest.mark.gpu

# (N, H, W, Ci, Co): one output pixel, rows that fill no tile, several images or row groups per tile, channel counts of less than
# a chunk or of no whole number of chunks, several column tiles, the longest rows (128; 254 for the channels of the halo kernel)
SHAPES = [(1, 2, 2, 16, 32), (5, 6, 10, 16, 32), (5, 12, 12, 24, 40), (130, 14, 14, 32, 64), (2, 34, 20, 64, 128), (7, 8, 8, 256, 512),
          (2, 32, 32, 160, 320), (1, 4, 128, 64, 64), (33, 4, 4, 48, 96), (2, 6, 200, 16, 32),
          (1, 4, 254, 16, 32)]


def _mk(shape, seed, scale=1.0):
    t = (torch.from_numpy(np.random.default_rng(seed).standard_normal(shape).astype(np.float32)) * scale).cuda().bfloat16()
    return t, t.float().cpu().numpy().astype(np.float64)


def _close(got, want, bar=1e-2):
    got = got.float().cpu().numpy().astype(np.float64)
    assert np.abs(got - want).max() <= bar * max(np.abs(want).max(), 1e-30)


@pytest.mark.parametrize("share", [1, 4])
@pytest.mark.parametrize("shape", SHAPES)
def test_stride_2(shape, share):
    from paper_1906_09108_b200 import binding as B
    ops = B.ConvOps(B.FDG_BF16_TC)
    n, h, w, ci, co = shape
    s = B.fdg_conv_shape(n, h, w, ci, co, 3, 2, 1)
    assert ops.path(s, 0) and ops.path(s, 1)
    wt, wo = _mk((co, 3, 3, ci), 1, (2.0 / (9 * ci)) ** 0.5)
    (x, xo), (res, reso), (gate, gateo) = (_mk((n, h, w, ci), k) for k in (2, 3, 4))
    (dy, dyo), (resy, resyo) = (_mk((n, h // 2, w // 2, co), k) for k in (5, 6))
    want = L.conv2d_forward(xo, wo, 2, 1)
    _close(ops.forward(s, x, wt, share=share), want)
    _close(ops.forward(s, x, wt, res=resy, share=share), want + resyo)
    y, part = ops.forward(s, x, wt, share=share, reduce=True)
    _close(y, want)
    assert part.shape[0] > 0
    ys = y.float().cpu().numpy().astype(np.float64).reshape(-1, co)
    tot = part.double().sum(dim=0).cpu().numpy()
    # fp32 sums of at most a few thousand values per thread and row of sums
    assert np.abs(tot[:co] - ys.sum(0)).max() <= 1e-5 * np.abs(ys).sum(0).max()
    assert np.abs(tot[co:] - (ys ** 2).sum(0)).max() <= 1e-5 * (ys ** 2).sum(0).max()
    wf = ops.flip_weights(s, wt)
    dxo, _ = L.conv2d_backward(dyo, xo, wo, 2, 1)
    _close(ops.dgrad(s, dy, wt, wf, share=share), dxo)
    _close(ops.dgrad(s, dy, wt, wf, res=res, res_mask=gate, share=share), dxo + reso * (gateo > 0))
    assert not ops.timed_out()


@pytest.mark.parametrize("shape, spread", [((4, 2, 66, 8, 16), False), ((4, 4, 66, 48, 24), False), ((8, 8, 8, 16, 32), True), ((8, 8, 12, 24, 40), True)])
def test_dy_is_spread_only_for_a_weight_gradient_that_reads_it(shape, spread):
    """Rows of more than 64 pixels outside the halo-tile kernel's channels: the weight gradient runs on the CUDA cores, from dy
    itself, and the scratch for the spread-out copy is left alone; elsewhere it holds dy at the even pixels of zeros."""
    import ctypes as C
    from paper_1906_09108_b200 import binding as B
    ops = B.ConvOps(B.FDG_BF16_TC)
    n, h, w, ci, co = shape
    s = B.fdg_conv_shape(n, h, w, ci, co, 3, 2, 1)
    assert ops.path(s, 1) and bool(ops.path(s, 2)) == spread
    (x, xo), (dy, dyo) = _mk((n, h, w, ci), 1), _mk((n, h // 2, w // 2, co), 2)
    room = C.c_size_t()
    assert ops.lib.fdg_conv_wgrad_scratch_bytes(B.FDG_BF16_TC, C.byref(s), C.byref(room)) == B.FDG_OK
    scratch, dw = torch.empty(room.value, dtype=torch.uint8, device="cuda"), torch.empty((co, 3, 3, ci), device="cuda")
    ex = B.fdg_conv_extra()
    up = torch.full((n, h, w, co), 7.0, dtype=torch.bfloat16, device="cuda")
    ex.dy_spread = up.data_ptr()
    assert ops.lib.fdg_conv_wgrad(B.FDG_BF16_TC, C.byref(s), x.data_ptr(), dy.data_ptr(), dw.data_ptr(), scratch.data_ptr(), room.value,
                                  C.byref(ex), ops.status.data_ptr(), torch.cuda.current_stream().cuda_stream) == B.FDG_OK
    want = torch.full_like(up, 7.0)
    if spread:
        want.zero_()
        want[:, ::2, ::2] = dy
    assert torch.equal(up, want)
    dwo = L.conv2d_backward(dyo, xo, np.zeros((co, 3, 3, ci)), 2, 1)[1]
    _close(dw, dwo, 1e-3)
    assert not ops.timed_out()
