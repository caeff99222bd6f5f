"""The commit kernel's quotient, copy ring and slot plan at the sizes where they can go wrong.

The quotients are compared with numpy's IEEE division bit for bit over every significand of the
denominator, which is what the refinement of the reciprocal depends on, and over the
operand ranges on both sides of the kernel's range check: with eps = 1e-18, just above its lower
end, the kernel divides by itself wherever the operands allow it, with 1e-38 by the
intrinsic everywhere.  The batches are compared with single
commits, and those with the oracle by test_gpu_commit.
"""
import numpy as np
import pytest
import torch

from paper_1805_08469_gb300 import gem
from paper_1805_08469_gb300._build import build_library

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    build_library()
    torch.cuda.set_device(0)


def _factors(g, m, s, eta, mu, eps):
    """Factors that one commit at theta = 0 applies, from the kernel and from numpy in fp32."""
    P = g.size
    f32 = np.float32
    with gem.Gem(P, 1, eta, mu, eps) as G:
        gem.gem_load_state(G.h, theta=np.zeros(P, np.float32), m=m[None], s=s[None])
        pi = torch.empty(P, device="cuda")
        G.commit_batch_pi([0], [torch.from_numpy(g).cuda()], [pi])
        G.sync()
        got = pi.cpu().numpy()
    with np.errstate(all="ignore"):
        dt = -(f32(eta) * g)
        energy = np.abs(f32(mu) * m + dt)
        q = (energy - np.abs(f32(0) - s)) / (np.abs(dt) + f32(eps))
        want = np.where(q > 0, q, f32(0))
    return got, want


@pytest.mark.parametrize("eps", [1e-18, 1e-38])
@pytest.mark.parametrize("exponents", [(-1, 1), (-30, 30), (-70, 70), (-126, 126)])
def test_factor_quotients_are_correctly_rounded(exponents, eps):
    """Every significand of the denominator (eta = 1 and, for |g| >= 2^-30, den = |g|), numerators
    and exponents at random; (-70, 70) and (-126, 126) reach past the range check."""
    lo, hi = exponents
    rng = np.random.default_rng(hi)
    P = 1 << 23
    den = np.ldexp((np.arange(P, dtype=np.float64) + P) / P, rng.integers(lo, hi, P)).astype(np.float32)
    num = np.ldexp(1 + rng.random(P), rng.integers(lo, hi, P)).astype(np.float32)
    got, want = _factors(den, num, np.zeros(P, np.float32), 1.0, 0.9375, eps)
    assert np.array_equal(got.view(np.uint32), want.view(np.uint32))


@pytest.mark.parametrize("eps", [1e-18, 1e-38])
@pytest.mark.parametrize("exponent", [-25, 0, 25])
def test_factor_quotients_of_the_largest_significand(exponent, eps):
    """den = 2 - 2^-23 times a power of two, the one denominator whose refined reciprocal may miss
    round to nearest; a numerator that is a power of two then shows it."""
    P = 1 << 23
    den = np.full(P, np.ldexp(2.0 - 2.0 ** -23, exponent), np.float32)
    m = np.ldexp((np.arange(P, dtype=np.float64) + P) / P * 8, exponent).astype(np.float32)
    energy = np.abs(np.float32(0.9375) * m - den)
    assert (np.frexp(energy)[0] == 0.5).any()
    got, want = _factors(den, m, np.zeros(P, np.float32), 1.0, 0.9375, eps)
    assert np.array_equal(got.view(np.uint32), want.view(np.uint32))


def test_factor_quotients_of_special_values():
    """Zeros, subnormals, infinities and NaNs in g, m and s, each with each."""
    v = np.array([0.0, -0.0, 1e-45, -1e-40, 1.2e-38, 1e-20, -3.5, 2.0 ** 61, 3e38, np.inf, -np.inf, np.nan], np.float32)
    g, m, s = (x.ravel().copy() for x in np.meshgrid(v, v, v, indexing="ij"))
    for eps in (1e-8, 1e-16, 1e-30):
        got, want = _factors(g, m, s, 0.5, 0.5, eps)
        assert np.array_equal(got.view(np.uint32), want.view(np.uint32))


# Repeats at every distance from 1 on, more of them open at once than there are slots, in launches
# of 2, 32, 33 and 200 commits and across them; P around a block (128 lanes), an SM's worth of
# blocks, and ragged.
@pytest.mark.parametrize("P", [1, 4, 127, 509, 513, 152 * 32 * 4 + 1, 152 * 128 * 4 + 3, 400_003])
@pytest.mark.parametrize("rule", [0, 1, 2, 3, 5])
def test_batches_equal_single_commits(P, rule):
    rng = np.random.default_rng(P + rule)
    n = 12
    orders = [[3, 3], [0, 1, 0, 1, 2, 2, 2] * 4 + [0, 1, 2, 3], rng.integers(0, n, 33).tolist(),
              list(range(n)) + list(range(n))[::-1] + rng.integers(0, n, 176).tolist()]
    ld = (P + 3) // 4 * 4
    theta0 = torch.from_numpy((0.05 * rng.standard_normal(P)).astype(np.float32)).cuda()
    pool = torch.zeros((16, ld), device="cuda")
    pool[:, :P] = torch.from_numpy((0.1 * rng.standard_normal((16, P))).astype(np.float32)).cuda()
    with gem.Gem(P, n, 0.01, 0.9, 1e-8) as A, gem.Gem(P, n, 0.01, 0.9, 1e-8) as B:
        for G in (A, B):
            G.set_theta(theta0)
            G.set_mode(rule, 1.5)
        k = 0
        for order in orders:
            grads = [pool[(k + i) % 16, :P] for i in range(len(order))]
            k += len(order)
            A.commit_batch(order, grads)
            for w, g in zip(order, grads):
                B.commit(w, g)
        A.sync()
        B.sync()
        assert torch.equal(A.theta(), B.theta())
        for w in range(n):
            assert torch.equal(A.snapshot(w), B.snapshot(w)) and torch.equal(A.moment(w), B.moment(w))


# Gradient rows on 128-byte lines and between them (every row of a launch, or one), and each
# remainder of a ragged row.
@pytest.mark.parametrize("P", [3, 510, 4097, 200_003])
@pytest.mark.parametrize("offsets", [(0,), (4,), (28,), (0, 0, 12)])
@pytest.mark.parametrize("rule", [0, 1, 5])
def test_gradient_rows_at_every_alignment(P, offsets, rule):
    rng = np.random.default_rng(P)
    ld = (P + 31) // 32 * 32 + 32
    pool = torch.zeros((6, ld), device="cuda")
    pool.copy_(torch.from_numpy((0.1 * rng.standard_normal((6, ld))).astype(np.float32)))
    assert pool.data_ptr() % 128 == 0
    rows = [pool[i, o:o + P] for i, o in zip(range(6), offsets * 6)]
    order = [0, 1, 2, 0, 0, 1]
    with gem.Gem(P, 3, 0.01, 0.9, 1e-8) as A, gem.Gem(P, 3, 0.01, 0.9, 1e-8) as B:
        for G in (A, B):
            G.set_theta(torch.from_numpy(rng.standard_normal(P).astype(np.float32)).cuda() if G is A else A.theta().clone())
            G.set_mode(rule, 1.5)
        A.commit_batch(order, rows)
        for w, g in zip(order, rows):
            B.commit(w, g.clone())
        A.sync()
        B.sync()
        assert torch.equal(A.theta(), B.theta())
        for w in range(3):
            assert torch.equal(A.snapshot(w), B.snapshot(w)) and torch.equal(A.moment(w), B.moment(w))


@pytest.mark.parametrize("offset", [0, 4, 28])
@pytest.mark.parametrize("rule", [0, 1, 5])
def test_host_gradient_rows_at_every_alignment(offset, rule):
    """Page-locked gradients on 128-byte lines and between them, read in place: the bits of the
    same batch from device memory."""
    P, n, order = 20_003, 3, [0, 1, 2, 0, 0, 1, 2, 2]
    rng = np.random.default_rng(offset + rule)
    ld = (P + 31) // 32 * 32 + 32
    host = torch.from_numpy((0.1 * rng.standard_normal((len(order), ld))).astype(np.float32)).pin_memory()
    theta0 = torch.from_numpy(rng.standard_normal(P).astype(np.float32)).cuda()
    dev = host.cuda()
    assert host.data_ptr() % 128 == 0 and dev.data_ptr() % 128 == 0
    with gem.Gem(P, n, 0.01, 0.9, 1e-8) as A, gem.Gem(P, n, 0.01, 0.9, 1e-8) as B:
        for G in (A, B):
            G.set_theta(theta0)
            G.set_mode(rule, 1.5)
        A.commit_batch_host(order, [host[k, offset:offset + P] for k in range(len(order))])
        B.commit_batch(order, [dev[k, offset:offset + P].clone() for k in range(len(order))])
        A.sync()
        B.sync()
        assert torch.equal(A.theta(), B.theta())
        for w in range(n):
            assert torch.equal(A.snapshot(w), B.snapshot(w)) and torch.equal(A.moment(w), B.moment(w))
