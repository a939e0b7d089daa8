"""The register-tiled CUDA-core convolutions on shapes where their tiling can go wrong -- row segments, row tiles, channel
chunks and channel blocks that are not full, several images per tile -- in both storage types, against the oracle's
convolution with the bars of test_gpu_conv_ops.py; and the sums they form for the batch norm that follows."""
import numpy as np
import pytest
import torch

from tests.test_gpu_conv_ops import _run

pytestmark = pytest.mark.gpu

# (N, H, W, Ci, Co, R, stride, pad)
SHAPES = [(2, 33, 30, 3, 16, 3, 1, 1),       # the stem: three channels; odd height, a last segment of two pixels
          (3, 7, 7, 20, 36, 3, 1, 1),        # channel counts that fill neither a chunk nor a thread column of 8
          (2, 9, 64, 4, 68, 3, 1, 1),        # two channel blocks, the widest rows
          (5, 4, 6, 17, 66, 3, 1, 1),        # odd channel counts
          (300, 4, 4, 12, 20, 3, 1, 1),      # several images per tile
          (160, 16, 16, 16, 32, 3, 1, 1),    # 8 channels per thread
          (2, 64, 64, 4, 4, 3, 2, 1),        # stride 2: rows of a tile bounded by shared memory
          (3, 14, 14, 36, 40, 3, 2, 1),
          (2, 10, 12, 40, 72, 1, 1, 0), (3, 12, 10, 36, 68, 1, 2, 0),
          # weight gradients whose rows leave shared memory for fewer row groups than the block has threads for
          (2, 64, 64, 4, 32, 1, 1, 0), (2, 64, 64, 8, 32, 1, 1, 0), (2, 56, 56, 24, 4, 3, 2, 1), (2, 64, 64, 32, 8, 1, 2, 0),
          (3, 13, 63, 8, 32, 1, 1, 0),
          # images of one row: more of them would fill the block than shared memory holds with their border rows
          (2368, 1, 64, 4, 4, 3, 1, 1)]


@pytest.mark.parametrize("shape", SHAPES)
def test_direct_conv_fp32(shape):
    _run("fp32", shape, False)


@pytest.mark.parametrize("shape", [s for s in SHAPES if s[3] % 8 or s[4] % 8])
def test_direct_conv_bf16(shape):
    _run("bf16", shape, False)


@pytest.mark.parametrize("shape", [(4, 32, 30, 3, 16), (200, 9, 7, 3, 64), (2, 12, 20, 5, 128)])
def test_statistics_rows_of_the_stem(shape):
    """The rows of (sum y, sum y^2) add up to those of the stored output; at most 256 rows."""
    from paper_1906_09108_b200 import binding as B
    n, h, w, ci, co = shape
    ops = B.ConvOps(B.FDG_BF16_TC)
    s = B.fdg_conv_shape(n, h, w, ci, co, 3, 1, 1)
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((n, h, w, ci), device="cuda", generator=g).to(ops.dtype)
    wt = torch.randn((co, 3, 3, ci), device="cuda", generator=g).to(ops.dtype)
    y, rows = ops.forward(s, x, wt, reduce=True)
    assert 0 < rows.shape[0] <= B.FDG_CONV_PARTIAL_ROWS
    got = rows.double().sum(0).cpu().numpy()
    yd = y.double().reshape(-1, co)
    want = torch.cat([yd.sum(0), (yd * yd).sum(0)]).cpu().numpy()
    scale = np.concatenate([yd.abs().sum(0).cpu().numpy(), want[co:]])
    assert np.max(np.abs(got - want) / scale) < 1e-5


@pytest.mark.parametrize("shape", [(1, 16, 16, 3, 16, 3, 1, 1),       # a row per group of threads: the groups' sums
                                   (1, 12, 12, 36, 36, 3, 1, 1),      # four rows per group: a thread's own sums
                                   (1, 16, 16, 16, 24, 1, 2, 0)])     # a projection
def test_bf16_weight_gradients_add_rows_in_64_bits(shape):
    """A large row, small ones, and the large one's negative (one block takes the image): the small rows are what is left,
    to the last bit.  Sums of rows in fp32 lose all of them (2^30 has steps of 128)."""
    from oracle import layers as L
    from paper_1906_09108_b200 import binding as B
    n, h, w, ci, co, r, st, pad = shape
    ops = B.ConvOps(B.FDG_BF16_TC)
    s = B.fdg_conv_shape(n, h, w, ci, co, r, st, pad)
    p, q = ops.out_hw(s)
    x, dy = np.ones((n, h, w, ci)), np.ones((n, p, q, co))
    dy[:, 0] = dy[:, -1] = 0
    dy[:, 0, q // 2], dy[:, -1, q // 2] = 2.0 ** 30, -2.0 ** 30
    want = L.conv2d_backward(dy, x, np.zeros((co, r, r, ci)), st, pad)[1]
    got = ops.wgrad(s, torch.from_numpy(x).cuda().to(ops.dtype), torch.from_numpy(dy).cuda().to(ops.dtype)).cpu().numpy()
    assert np.array_equal(got, want.astype(np.float32))
    assert np.abs(want).min() < 2.0 ** 10


def test_context_of_64x64_images_fp32():
    """A network whose projection's weight gradient (1x1, 64x64, 8 -> 32 channels) asks for rows of 19 KB: a whole
    iteration through the context, to the bar of the fp32 mode."""
    from tests.fdg_pair import run_pair
    arch = dict(family="resnet6n2", blocks=(1, 1), widths=(32, 32), stem_width=8, in_h=64, in_w=64, in_c=3, num_classes=10, batch=3)
    res = run_pair(arch, 1, (), 2, lr=0.01, seed=1)
    assert max(res["grads"], res["params"], res["loss"]) <= 1e-4, res["grads_by_step"]
