"""The CUDA-core products at the sizes where their tiles, splits and routes change.

The gradients are compared with the oracle at the bars of test_gpu_mlp.  The bar of the fp32
cases is the 1e-5 of that file: sums of K products in fp32, one rounding of 6e-8 each, grow
as sqrt(K) at random, 2e-6 for the K = 1,000 of the longest.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1805_08469_gb300 import gem, sim, synth, synth_gpu

from test_gpu_mlp import _gradient_parity, _setup, rel_l2, theta0_with_biases  # noqa: F401  (_setup is the module's fixture)

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


# TF32 products that the tensor cores do not take: fewer than 32 rows or a K below 32
@pytest.mark.parametrize("dims,b", [([784, 64, 10], 8), ([100, 31, 10], 31), ([96, 40, 16], 64)])
def test_tf32_small_products_match_oracle(dims, b):
    _gradient_parity(dims, b, sim.GEM_MLP_TF32, 1e-4, 1e-2, 3, [1, 0])


@pytest.mark.parametrize("layout", ["rows", "spaced", "reversed", "scattered", "one"])
def test_gradients_are_the_same_wherever_the_caller_wants_them(layout):
    """Equally spaced rows are written in place, others through a copy: the same values, and
    nothing outside the P floats of a row."""
    dims, b, seed = [40, 37, 10], 20, 5
    P = synth.mlp_param_count(dims)
    workers = [2, 0, 1] if layout != "one" else [1]
    ld = (P + 3) // 4 * 4 + (64 if layout == "spaced" else 0)
    X = torch.empty((300, dims[0]), device="cuda")
    y = torch.empty(300, dtype=torch.int32, device="cuda")
    synth_gpu.data(seed, X, y, 10)
    rows = np.random.default_rng(1).integers(0, 300, (len(workers), b)).astype(np.int32)
    buf = torch.full((8, ld), -7.0, device="cuda")
    at = {"rows": [0, 1, 2], "spaced": [1, 3, 5], "reversed": [2, 1, 0], "scattered": [0, 5, 3], "one": [4]}[layout]
    with gem.Gem(P, 3, 0.01, 0.9, 1e-8) as G:
        G.set_theta(synth_gpu.xavier(seed, dims, torch.empty(P, device="cuda")))
        M = sim.gem_mlp_create(G.h, dims, b)
        sim.gem_mlp_set_data(M, X, y)
        apart = [torch.empty(P, device="cuda") for _ in range(2 * len(workers))][::2]
        sim.gem_mlp_grad(M, workers, rows, [buf[i, :P] for i in at])
        for k, w in enumerate(workers):        # one worker at a time
            sim.gem_mlp_grad(M, [w], rows[k:k + 1], [apart[k]])
        sim.gem_mlp_status(M)
        sim.gem_mlp_destroy(M)
    for k, i in enumerate(at):
        assert torch.allclose(buf[i, :P], apart[k], rtol=0, atol=1e-6 * float(apart[k].abs().max()))
    mask = torch.ones_like(buf, dtype=torch.bool)
    for i in at:
        mask[i, :P] = False
    assert bool((buf[mask] == -7.0).all())


def test_tf32_tiles_96_wide():
    """13 workers of 1,000 columns: 143 tiles 96-wide, the last one of a row 40 columns, on K with
    a remainder (the bars of the wide layers in test_gpu_mlp)."""
    _gradient_parity([100, 1000, 516, 10], 128, sim.GEM_MLP_TF32, 3e-4, 1e-2, 13, list(range(13)))


# A network without a hidden layer: its first product is also the logits.  The rows of a minibatch
# are in random order with repeats, and with 3 rows the data set is shorter than the minibatch.
@pytest.mark.parametrize("dims", [[784, 10], [37, 3], [40, 37, 10]])
@pytest.mark.parametrize("precision", [sim.GEM_MLP_FP32, sim.GEM_MLP_TF32])
@pytest.mark.parametrize("b,rows", [(1, 500), (33, 500), (128, 500), (33, 3)])
def test_minibatch_rows_of_every_entry_point(dims, precision, b, rows):
    """gem_mlp_grad, gem_mlp_grad_static and gem_mlp_run read the rows that they are given.  The
    bars are those of test_gpu_mlp: 1e-5 for fp32 products and, with TF32 operands, 1e-2
    where the delta is rounded, 1e-4 for the loss; theta 1e-4 and 2e-3."""
    seed, n, T = 11, 3, 7
    tf32 = precision == sim.GEM_MLP_TF32
    bar, deep = (1e-4, 1e-2) if tf32 else (1e-5, 1e-5)
    P = synth.mlp_param_count(dims)
    rng = np.random.default_rng(rows + b)
    X = rng.standard_normal((rows, dims[0])).astype(np.float32)
    y = rng.integers(0, dims[-1], rows).astype(np.int32)
    order = rng.integers(0, n, T).astype(np.int32)
    batches = rng.integers(0, rows, (T, b)).astype(np.int32)
    theta0 = theta0_with_biases(seed, dims)
    Xd, yd, td = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), torch.from_numpy(theta0).cuda()
    got = [torch.empty((P + 3) // 4 * 4, device="cuda")[:P] for _ in range(2 * n)]
    losses = torch.empty(2 * n, device="cuda")
    run_losses = torch.empty(T, device="cuda")
    with gem.Gem(P, n, 0.01, 0.9, 1e-8) as G:
        G.set_theta(td)
        M = sim.gem_mlp_create(G.h, dims, b, precision)
        try:
            sim.gem_mlp_set_data(M, Xd, yd)
            sim.gem_mlp_grad(M, list(range(n)), batches[:n], got[:n], losses)
            G.sync()
            for k in range(n):
                sim.gem_mlp_grad_static(dims, b, precision, td, Xd, yd, batches[k], got[n + k], losses[n + k:])
            torch.cuda.synchronize()
            sim.gem_mlp_run(M, order, batches, run_losses)
            G.sync()
            theta = G.theta().cpu().numpy()
            sim.gem_mlp_status(M)
        finally:
            sim.gem_mlp_destroy(M)
    for k in range(2 * n):
        r = batches[k % n]
        loss, g = oracle.mlp_loss_grad(dims, theta0.astype(np.float64), X[r], y[r], tf32=tf32)
        assert rel_l2(got[k].cpu().numpy(), g) < deep, k
        assert abs(float(losses[k]) - loss) <= bar * abs(loss) + 1e-6, k
    th, m, s = theta0.copy(), np.zeros((n, P), np.float32), np.tile(theta0, (n, 1))
    _r, ref = oracle.mlp_sim_run(dims, th, m, s, order, X, y, batches, eta=0.01, mu=0.9, eps=1e-8, tf32=tf32,
                                 want_losses=True)
    assert rel_l2(theta, th) < (2e-3 if tf32 else 1e-4)
    np.testing.assert_allclose(run_losses.cpu().numpy(), ref, rtol=2e-3 if tf32 else 1e-4)


@pytest.mark.parametrize("dims,G", [([100, 72, 40, 10], 3), ([100, 1000, 516, 10], 2)])
@pytest.mark.parametrize("layout", ["rows", "spaced"])
def test_tf32_gradients_are_the_same_wherever_the_caller_wants_them(dims, G, layout):
    """The tensor cores' weight gradients in the caller's rows directly: the bits of the same call
    with rows in reverse order, which are copied, and nothing outside the P floats of a row."""
    b, seed = 48, 5
    P = synth.mlp_param_count(dims)
    ld = (P + 3) // 4 * 4 + (64 if layout == "spaced" else 0)
    X = torch.empty((300, dims[0]), device="cuda")
    y = torch.empty(300, dtype=torch.int32, device="cuda")
    synth_gpu.data(seed, X, y, 10)
    rows = np.random.default_rng(1).integers(0, 300, (G, b)).astype(np.int32)
    at = list(range(1, G + 1))
    direct = torch.full((G + 2, ld), -7.0, device="cuda")
    copied = torch.full((G + 2, ld), -7.0, device="cuda")
    with gem.Gem(P, G, 0.01, 0.9, 1e-8) as Gh:
        Gh.set_theta(synth_gpu.xavier(seed, dims, torch.empty(P, device="cuda")))
        M = sim.gem_mlp_create(Gh.h, dims, b, sim.GEM_MLP_TF32)
        sim.gem_mlp_set_data(M, X, y)
        sim.gem_mlp_grad(M, list(range(G)), rows, [direct[i, :P] for i in at])
        sim.gem_mlp_grad(M, list(range(G)), rows, [copied[G + 1 - i, :P] for i in at])
        sim.gem_mlp_status(M)
        sim.gem_mlp_destroy(M)
    for i in at:
        assert torch.equal(direct[i, :P], copied[G + 1 - i, :P])
        assert bool((direct[i, :P] != -7.0).all())
    mask = torch.ones_like(direct, dtype=torch.bool)
    mask[1:G + 1, :P] = False
    assert bool((direct[mask] == -7.0).all()) and bool((copied[mask] == -7.0).all())
