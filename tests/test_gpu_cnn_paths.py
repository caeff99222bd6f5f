"""The convolution kernels of the paper's map sizes (28 x 28 inputs) at other channel counts and
minibatches: odd counts (a pair and a group of four output channels with an idle place), one
channel, more than a block's threads, odd minibatches (a block with one of its two samples), few
samples and more than SMs, and channel counts whose staging does not fit, which take the general kernels."""
import pytest

import test_gpu_cnn
from test_gpu_cnn import _setup  # noqa: F401  (the module fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,b,G", [
    ((28, 1, 1, 3, 2, 2), 1, 1),
    ((28, 3, 5, 12, 9, 4), 3, 2),
    ((28, 7, 2, 8, 8, 3), 2, 3),
    ((28, 13, 21, 16, 12, 10), 5, 2),          # 273 channel pairs, 78 kernel-row groups
    ((28, 30, 6, 8, 8, 5), 3, 2),
    ((28, 30, 40, 8, 8, 3), 1, 2),             # 134 KB of padded weights
    ((28, 69, 17, 8, 8, 3), 1, 1),             # past 200 KB: the general kernels
    # more samples than SMs, so two and three per block, the last block of a worker with one
    ((28, 3, 5, 12, 9, 4), 79, 2),
    ((28, 11, 6, 8, 8, 3), 51, 3),
])
def test_gradients_at_other_channel_counts(shape, b, G):
    test_gpu_cnn.test_gradients_match_the_oracle(shape, b, G)
