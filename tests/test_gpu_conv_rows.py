"""The grouped-pixel convolutions at sizes where their tiles, groups and image loops have edges: forward with residual and
statistics, data gradient with a gated residual and the sums of the batch-norm backward pass."""
import numpy as np
import pytest
import torch

from oracle import layers as L

pytestmark = pytest.mark.gpu

# (N, H, W, C, share): odd heights, widths of a few groups or one, more images than a CTA takes at once, single images
SHAPES = [(5, 28, 28, 16, 1), (3, 17, 24, 16, 4), (1, 1, 4, 16, 1), (130, 12, 12, 16, 2), (7, 5, 40, 32, 4),
          (9, 14, 14, 32, 1), (1, 3, 2, 32, 1), (131, 7, 7, 64, 2), (3, 20, 9, 64, 4), (2, 40, 40, 16, 1)]


def _mk(shape, seed, scale=1.0):
    t = (torch.from_numpy(np.random.default_rng(seed).standard_normal(shape).astype(np.float32)) * scale).cuda().bfloat16()
    return t, t.float().cpu().numpy().astype(np.float64)


def _close(got, want, bar):
    got = got.float().cpu().numpy().astype(np.float64)
    assert np.abs(got - want).max() <= bar * max(np.abs(want).max(), 1e-30)


@pytest.mark.parametrize("shape", SHAPES)
def test_grouped_pixel_convolutions(shape):
    from paper_1906_09108_b200 import binding as B
    ops, ew = B.ConvOps(B.FDG_BF16_TC), B.EwOps(B.FDG_BF16_TC)
    n, h, w, c, share = shape
    s = B.fdg_conv_shape(n, h, w, c, c, 3, 1, 1)
    assert ops.path(s, 0) and ops.path(s, 1)
    wt, wo = _mk((c, 3, 3, c), 1, (2.0 / (9 * c)) ** 0.5)
    (x, xo), (res, reso), (gate, gateo), (dy, dyo), (nm, nmo), (nx, nxo) = (_mk((n, h, w, c), k) for k in range(2, 8))
    want = L.conv2d_forward(xo, wo, 1, 1)
    _close(ops.forward(s, x, wt, share=share), want, 1e-2)
    y, part = ops.forward(s, x, wt, res=res, share=share, reduce=True)
    _close(y, want + reso, 1e-2)
    ys = y.float().cpu().numpy().astype(np.float64).reshape(-1, c)
    tot = part.double().sum(dim=0).cpu().numpy()
    for got, ref in ((tot[:c], ys.sum(0)), (tot[c:], (ys * ys).sum(0))):
        assert np.abs(got - ref).max() <= 1e-4 * (ys * ys).sum(0).max()
    stats = ew.bn_stats(nx)
    dx, part = ops.dgrad(s, dy, wt, ops.flip_weights(s, wt), res=res, res_mask=gate, share=share, next_bn=(nm, nx, stats))
    _close(dx, L.conv2d_backward(dyo, xo, wo, 1, 1)[0] + reso * (gateo > 0), 1e-2)
    dz = (dx.float().cpu().numpy() * (nmo > 0)).reshape(-1, c).astype(np.float64)
    st = stats.double().cpu().numpy().reshape(-1)
    dzx = dz * ((nxo.reshape(-1, c) - st[:c]) * st[c:2 * c])
    tot = part.double().sum(dim=0).cpu().numpy()
    assert np.abs(tot[:c] - dz.sum(0)).max() <= 1e-4 * np.abs(dz).sum(0).max()
    assert np.abs(tot[c:] - dzx.sum(0)).max() <= 1e-4 * np.abs(dzx).sum(0).max()
    assert not ops.timed_out()
