"""bf16 convolutions on image sizes, batches and channel counts that fill no tile of the tensor-core kernels: the three
operators against the oracle's convolution, with the bars of test_gpu_conv_ops.py."""
import pytest

from tests.test_gpu_conv_ops import _run

pytestmark = pytest.mark.gpu

# (N, H, W, Ci, Co, R, stride, pad)
RAGGED = [(3, 24, 24, 128, 128, 3, 1, 1),     # five groups of 5 rows per image, the last with 4; 32-pixel slab rows
          (5, 12, 12, 128, 256, 3, 1, 1),     # two groups of 6 rows; 16-pixel slab rows of which 12 count
          (7, 6, 6, 256, 256, 3, 1, 1),       # three images per tile, a last tile of one; 8-pixel slab rows of which 6 count
          (5, 3, 3, 64, 128, 3, 1, 1),        # fourteen images per tile, fewer in the batch
          (97, 4, 4, 256, 128, 3, 1, 1),      # odd batch on tiles of eight images
          (3, 12, 12, 128, 256, 3, 2, 1), (5, 24, 24, 64, 128, 1, 2, 0), (7, 12, 12, 128, 256, 1, 2, 0),
          (3, 40, 40, 48, 48, 3, 1, 1),       # 48-pixel slab rows: three steps per slab; 48 of 64 channels
          (2, 5, 64, 40, 72, 3, 1, 1),        # rows of 64 pixels, odd height, channel counts that are no multiple of 16
          (3, 28, 28, 24, 24, 3, 1, 1), (9, 14, 14, 24, 48, 3, 2, 1), (6, 28, 28, 24, 48, 1, 2, 0),
          (8, 16, 16, 8, 8, 3, 1, 1), (8, 16, 16, 8, 16, 3, 2, 1), (8, 16, 16, 8, 16, 1, 2, 0),
          (3, 16, 16, 80, 112, 3, 1, 1),      # patch kernel with a last chunk of 16 channels
          (2, 16, 16, 288, 576, 3, 1, 1),     # column tiles and channel chunks that are no power of two
          (4, 8, 8, 576, 296, 3, 1, 1)]       # a last column tile that is not full


@pytest.mark.parametrize("shape", RAGGED)
def test_conv_ops_bf16_ragged_shapes(shape):
    _run("bf16", shape, True)
