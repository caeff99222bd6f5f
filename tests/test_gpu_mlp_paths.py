"""The CUDA-core products at the sizes where their tiles, splits and routes change.

The gradients are compared with the oracle at the bars of test_gpu_mlp.  The bar of the fp32
cases is the 1e-5 of that file: sums of K products in fp32, one rounding of 6e-8 each, grow
as sqrt(K) at random, 2e-6 for the K = 1,000 of the longest.
"""
import numpy as np
import pytest
import torch

from paper_1805_08469_gb300 import gem, sim, synth, synth_gpu

from test_gpu_mlp import _gradient_parity, _setup  # noqa: F401  (_setup is the module's fixture)

pytestmark = pytest.mark.gpu


# Minibatches around a tile of 32 and 64 rows; layers whose rows are not 16-byte aligned (odd
# widths), narrower than a k-tile and with a remainder; K long enough for a split, with a last
# part that is short, and one class.
@pytest.mark.parametrize("dims,b,workers", [
    ([13, 7, 3], 1, [0]),
    ([784, 64, 10], 32, [2, 0]),
    ([131, 33, 5], 31, [1]),
    ([300, 65, 10], 33, [0, 1, 2]),
    ([785, 63, 61, 2], 64, [0]),
    ([256, 128, 129, 10], 65, [2, 1]),
    ([1000, 20, 10], 127, [1, 0]),
    ([516, 96, 16], 128, [0, 2]),
    ([400, 50, 10], 130, [0]),                 # a batch past the split's limit
])
def test_small_products_match_oracle(dims, b, workers):
    _gradient_parity(dims, b, sim.GEM_MLP_FP32, 1e-5, 1e-5, 3, workers)


# 40 million FMAs per product: 33.6 million per worker here
@pytest.mark.parametrize("workers", [[0], [0, 1], [2, 1, 0]])
def test_both_sides_of_the_small_product_rule(workers):
    _gradient_parity([512, 512, 10], 128, sim.GEM_MLP_FP32, 1e-5, 1e-5, 3, workers)


# TF32 products that the tensor cores do not take: fewer than 32 rows or a K below 32, and those
# of small networks
@pytest.mark.parametrize("dims,b", [([784, 64, 10], 8), ([100, 31, 10], 31), ([96, 40, 16], 64),
                                    ([300, 130, 65, 10], 130), ([516, 384, 10], 128)])
def test_tf32_small_products_match_oracle(dims, b):
    _gradient_parity(dims, b, sim.GEM_MLP_TF32, 1e-4, 1e-2, 3, [1, 0])


def test_tf32_tiles_96_wide():
    """13 workers of 1,000 columns: 143 tiles 96-wide, the last one of a row 40 columns, on K with
    a remainder (the bars of the wide layers in test_gpu_mlp)."""
    _gradient_parity([100, 1000, 516, 10], 128, sim.GEM_MLP_TF32, 3e-4, 1e-2, 13, list(range(13)))
