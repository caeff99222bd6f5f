"""Performance cases: what a program that trains with this library has it do.

A program holds a handle (``gem.Gem``) with the central variable and every worker's moment
and snapshot, and either commits gradients of its own (one by one, or in batches, from device
or page-locked host memory, with or without the scaling factors' medians), or lets the
simulator run its network (the MLPs and the MNIST convolutional network) for the next T
commits of the schedule.  Families:

  single   gem_commit calls, one commit each
  batch    gem_commit_batch under any of the commit rules
  host     gem_commit_batch_host from page-locked memory, then theta read back
  pi       gem_commit_batch_pi_median: the commits, every factor, its medians per segment
  mlp_grad, cnn_grad  gem_mlp_grad, gem_cnn_grad: gradients of a segment's workers
  mlp_run  gem_mlp_run or gem_mlp_run_pi: T commits, forward/backward included
  cnn_run  gem_cnn_run or gem_cnn_run_pi: the same on the convolutional network

A pass of the commit families and of the runs goes on from the state the previous pass left,
as training does.  Hyper-parameters and input distributions are those of the benchmark
(heavy-tailed gradients; teacher-labelled N(0, 1) rows; template images).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1805_08469_gb300 import cnn, gem, sim, synth_gpu

ETA, MU, EPS = 0.01, 0.9, 1e-8
CNN_ETA = 0.05
ROWS = 60000                 # rows of the training sets
DIMS_SMALL, DIMS_LARGE = "784-64-10", "784-1000-1000-10"
RULES = {"gem": 0, "downpour": 1, "adaptive": 2, "kappa_sqrt": 3, "kappa_linear": 4, "momentum": 5}


def listed():
    return [
        # a small model trained by the caller's own loop: one call per gradient, where the
        # latency of a call and a launch is all there is
        dict(name="single_p51k_n4", family="single", P=50890, n=4, K=16),
        # mid-sized flat vector, 100 queued gradients at once (the state is L2-scale)
        dict(name="batch_p1.2m_n20", family="batch", rule="gem", P=1200000, n=20, K=100),
        # the headline: ResNet-50-sized vector, 100 workers, batches of 100 commits
        dict(name="batch_p25m_n100", family="batch", rule="gem", P=25000000, n=100, K=100),
        # a comparison rule on a ragged length, fewer commits than workers
        dict(name="batch_kappa_p3m_n30", family="batch", rule="kappa_linear", P=3000007, n=30, K=24),
        # gradients that arrive in page-locked host memory, theta read back each step
        dict(name="host_p5m_n100", family="host", P=5000000, n=100, K=16),
        # the paper's statistic on a flat vector: factors recorded, medians per tensor
        dict(name="pi_p5m_n30", family="pi", rule="gem", P=5000000, n=30, K=64, nseg=6),
        # gradients of one segment's workers for a caller with its own commit loop
        dict(name="mlp_grad_tf32_l13", family="mlp_grad", dims=DIMS_LARGE, b=128, n=20, L=13, tf32=1),
        # end-to-end training: the small MLP (short kernels, latency), ...
        dict(name="mlp_small_n4", family="mlp_run", dims=DIMS_SMALL, b=32, n=4, T=64, tf32=0, queue=0, pi=0),
        # ... the large one in fp32 under the queue schedule, ...
        dict(name="mlp_fp32_n30", family="mlp_run", dims=DIMS_LARGE, b=128, n=30, T=48, tf32=0, queue=1, pi=0),
        # ... in TF32 with 100 workers,
        dict(name="mlp_tf32_n100", family="mlp_run", dims=DIMS_LARGE, b=128, n=100, T=100, tf32=1, queue=0, pi=0),
        # the MNIST network with 100 workers,
        dict(name="cnn_n100", family="cnn_run", shape="28-10-20-128-64-10", b=64, n=100, T=64, pi=0),
        # and with 30 while following the median factor of each tensor
        dict(name="cnn_pi_n30", family="cnn_run", shape="28-10-20-128-64-10", b=64, n=30, T=32, pi=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _flat(rng, K):
    """P and n of a flat vector whose K commits and n workers fit the largest listed case."""
    while True:
        P, n = _log_int(rng, 1000, 25000000), _log_int(rng, 1, 100)
        if P * K <= 2.5e9 and P * n <= 2.5e9:
            return P, n


def draw(rng):
    family = rng.choice(["single", "batch", "batch", "batch", "host", "pi", "mlp_grad", "mlp_run", "mlp_run",
                         "mlp_run", "cnn_grad", "cnn_run", "cnn_run"])
    if family == "single":
        K = rng.randint(4, 32)
        P, n = _flat(rng, K)
        return dict(family=family, P=P, n=n, K=K)
    if family == "batch":
        K = _log_int(rng, 2, 250)
        P, n = _flat(rng, K)
        rule = rng.choice(["gem", "gem", "gem"] + list(RULES))
        return dict(family=family, rule=rule, P=P, n=n, K=K)
    if family == "host":
        P, n = _log_int(rng, 100000, 10000000), rng.randint(4, 60)
        return dict(family=family, P=P, n=n, K=rng.randint(4, 24))
    if family == "pi":
        K = _log_int(rng, 4, 100)
        P, n = _flat(rng, 4 * K)
        rule = rng.choice(["gem", "gem", "kappa_sqrt"])
        return dict(family=family, rule=rule, P=P, n=n, K=K, nseg=rng.choice([1, 2, 4, 6, 10]))
    if family == "cnn_grad":
        return dict(family=family, shape="28-10-20-128-64-10", b=_log_int(rng, 8, 96), n=24, L=rng.randint(1, 24))
    if family == "cnn_run":
        shape = rng.choice(["28-10-20-128-64-10"] * 3 + ["20-6-12-48-32-10"])
        return dict(family=family, shape=shape, b=_log_int(rng, 8, 96), n=_log_int(rng, 2, 100),
                    T=rng.randint(8, 48), pi=rng.randint(0, 1))
    d0 = rng.choice([784, 784, _log_int(rng, 16, 1000)])
    hidden = [_log_int(rng, 16, 1100) for _ in range(rng.choice([1, 2, 2, 3]))]
    dims = "-".join(str(d) for d in [d0] + hidden + [rng.choice([10, 10, rng.randint(2, 32)])])
    b, tf32 = _log_int(rng, 8, 160), rng.randint(0, 1)
    if family == "mlp_grad":
        return dict(family=family, dims=dims, b=b, n=24, L=rng.randint(1, 24), tf32=tf32)
    return dict(family=family, dims=dims, b=b, n=_log_int(rng, 2, 100), T=rng.randint(8, 48), tf32=tf32,
                queue=rng.randint(0, 1), pi=rng.randint(0, 1))


def _ints(text):
    return [int(x) for x in text.split("-")]


def _mlp_params(dims):
    return sum(o * i + o for i, o in zip(dims, dims[1:]))


def _mlp_tensors(dims):
    """Offsets of [W_1, b_1, W_2, ...] in the flat layout, and P at the end."""
    off = [0]
    for i, o in zip(dims, dims[1:]):
        off += [off[-1] + o * i, off[-1] + o * i + o]
    return off


def _cnn_tensors(shape):
    """Shapes of the ten parameter tensors of the convolutional network, in layout order."""
    H, c1, c2, f1, f2, C = shape
    F = c2 * (((H - 4) // 2 - 4) // 2) ** 2
    return [(c1, 1, 5, 5), (c1,), (c2, c1, 5, 5), (c2,), (f1, F), (f1,), (f2, f1), (f2,), (C, f2), (C,)]


class _State:
    """What the program keeps between calls.  The network is freed with it; the handle with the
    last of its users, since the outputs are views of the handle's memory."""

    net, free_net = 0, None

    def __del__(self):
        if self.net:
            self.free_net(self.net)


class _Borrowed:
    """A handle's device memory as a CUDA array that keeps the handle."""

    def __init__(self, G, ptr, shape):
        self.G = G
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<f4", "data": (ptr, False), "version": 3,
                                         "strides": None}


def _view(G, ptr, *shape):
    return torch.as_tensor(_Borrowed(G, ptr, shape), device="cuda")


_stream = None


def _handle(s, P, n, eta, theta0):
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()      # the program's one stream: its passes follow each other
    s.G = gem.Gem(P, n, eta, MU, EPS, stream=_stream)
    torch.cuda.synchronize()
    s.G.set_theta(theta0)
    s.G.sync()
    s.theta = _view(s.G, gem.gem_theta(s.G.h), P)
    s.m = _view(s.G, gem.gem_moment(s.G.h, 0), n, s.G.stride)
    s.s = _view(s.G, gem.gem_pull(s.G.h, 0), n, s.G.stride)


def _segments(case):
    """Segment offsets of the pi family: tensors of unequal size, the last one short."""
    P, k = case["P"], case["nseg"]
    return [0] + [int(P * (1 - 0.3 ** i)) for i in range(1, k)] + [P]


def _data(seed, d0, classes):
    """Teacher-labelled N(0, 1) rows."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn(ROWS, d0, device="cuda", generator=g)
    y = (X @ torch.randn(d0, classes, device="cuda", generator=g)).argmax(1).to(torch.int32)
    return X, y


def prepare(case, seed):
    s = _State()
    s.case = case
    fam = case["family"]
    rng = np.random.default_rng(seed)
    if fam in ("single", "batch", "host", "pi"):
        P, K = case["P"], case["K"]
        theta0 = synth_gpu.theta0_flat(seed, torch.empty(P, device="cuda"))
        ld = (P + 3) // 4 * 4                       # rows start on 16-byte boundaries
        pool = torch.empty((K, ld), device="cuda")
        synth_gpu.grad_heavytail(seed, 0, pool, P)
        _handle(s, P, case["n"], ETA, theta0)
        s.order = [int(w) for w in sim.gem_schedule_uniform(seed, case["n"], K)[0]]
        s.G.set_mode(RULES[case.get("rule", "gem")], 2.5 if "kappa" in case.get("rule", "") else 1.0)
        s.pool, s.theta0 = pool, theta0
        s.grads = [pool[k, :P] for k in range(K)]
        if fam == "host":
            host = torch.empty((K, ld), pin_memory=True)
            host.copy_(pool)
            s.pool, s.host = None, host
            s.grads = [host[k, :P] for k in range(K)]
            s.out = torch.empty(P, pin_memory=True)
        if fam == "pi":
            s.pi = torch.empty((K, ld), device="cuda")
            s.rows = [s.pi[k, :P] for k in range(K)]
            s.seg = _segments(case)
            s.lo = torch.empty((K, case["nseg"]), device="cuda")
            s.hi = torch.empty_like(s.lo)
        return s
    if fam.startswith("cnn"):
        shape = _ints(case["shape"])
        T, b = case.get("T") or case["L"], case["b"]
        P = cnn.gem_cnn_param_count(shape)
        theta0 = synth_gpu.cnn_theta0(seed, shape, torch.empty(P, device="cuda"))
        s.X = torch.empty((ROWS, shape[0] ** 2), device="cuda")
        s.y = torch.empty(ROWS, dtype=torch.int32, device="cuda")
        synth_gpu.cnn_data(seed, s.X, s.y, shape[5])
        s.drop = synth_gpu.dropout(seed, 0, torch.empty((T, b, shape[2]), device="cuda"))
        _handle(s, P, case["n"], CNN_ETA, theta0)
        s.net, s.free_net = cnn.gem_cnn_create(s.G.h, shape, b), cnn.gem_cnn_destroy
        cnn.gem_cnn_set_data(s.net, s.X, s.y)
        if fam == "cnn_run":
            s.order = sim.gem_schedule_uniform(seed, case["n"], T)[0]
        tensors = 10
    else:
        dims = _ints(case["dims"])
        b = case["b"]
        P = _mlp_params(dims)
        theta0 = synth_gpu.xavier(seed, dims, torch.empty(P, device="cuda"))
        s.X, s.y = _data(seed, dims[0], dims[-1])
        _handle(s, P, case["n"], ETA, theta0)
        s.net = sim.gem_mlp_create(s.G.h, dims, b, case["tf32"])
        s.free_net = sim.gem_mlp_destroy
        sim.gem_mlp_set_data(s.net, s.X, s.y)
        tensors = 2 * (len(dims) - 1)
        T = case.get("T") or case["L"]
        if fam == "mlp_run":
            schedule = sim.gem_schedule_queue if case["queue"] else sim.gem_schedule_uniform
            s.order = schedule(seed, case["n"], T)[0]
    if fam.endswith("grad"):
        # snapshots of workers in mid-training: each a little off the others
        g = torch.Generator(device="cuda").manual_seed(seed + 1)
        snaps = theta0 + 0.005 * torch.randn(case["n"], P, device="cuda", generator=g)
        torch.cuda.synchronize()
        gem.gem_load_state(s.G.h, s=snaps)
        s.G.sync()
        s.workers = rng.permutation(case["n"])[:T].astype(np.int32)
        s.g = torch.zeros((T, (P + 3) // 4 * 4), device="cuda")
        torch.cuda.synchronize()
        s.grads = [s.g[k, :P] for k in range(T)]
    s.theta0 = theta0
    s.batch_rows = rng.integers(0, ROWS, (T, b)).astype(np.int32)
    s.losses = torch.empty(T, device="cuda")
    if case.get("pi"):
        s.lo = torch.empty((T, tensors), device="cuda")
        s.hi = torch.empty_like(s.lo)
    return s


def run(s):
    case = s.case
    fam = case["family"]
    if fam == "single":
        for w, g in zip(s.order, s.grads):
            s.G.commit(w, g)
    elif fam == "batch":
        s.G.commit_batch(s.order, s.grads)
    elif fam == "host":
        s.G.commit_batch_host(s.order, s.grads)
        gem.gem_read_theta(s.G.h, s.out)
        return {"theta": s.theta, "m": s.m, "s": s.s, "out": s.out}
    elif fam == "pi":
        s.G.commit_batch_pi_median(s.order, s.grads, s.rows, s.seg, s.lo, s.hi)
        return {"theta": s.theta, "m": s.m, "s": s.s, "pi": s.pi[:, :case["P"]], "lo": s.lo, "hi": s.hi}
    elif fam == "mlp_grad":
        sim.gem_mlp_grad(s.net, s.workers, s.batch_rows, s.grads, s.losses)
        return {"grads": s.g, "losses": s.losses}
    elif fam == "cnn_grad":
        cnn.gem_cnn_grad(s.net, s.workers, s.batch_rows, s.drop, s.grads, s.losses)
        return {"grads": s.g, "losses": s.losses}
    elif fam == "mlp_run":
        if case["pi"]:
            sim.gem_mlp_run_pi(s.net, s.order, s.batch_rows, s.lo, s.hi, s.losses)
        else:
            sim.gem_mlp_run(s.net, s.order, s.batch_rows, s.losses)
    else:
        if case["pi"]:
            cnn.gem_cnn_run_pi(s.net, s.order, s.batch_rows, s.drop, s.lo, s.hi, s.losses)
        else:
            cnn.gem_cnn_run(s.net, s.order, s.batch_rows, s.drop, s.losses)
    out = {"theta": s.theta, "m": s.m, "s": s.s}
    if fam in ("mlp_run", "cnn_run"):
        out["losses"] = s.losses
        if case["pi"]:
            out.update(lo=s.lo, hi=s.hi)
    return out


def _distinct(n, T):
    """Expected number of distinct workers in T uniform draws of n."""
    return n * (1 - (1 - 1 / n) ** T)


def work(case):
    fam = case["family"]
    if fam in ("single", "batch", "host", "pi"):
        P, n, K = case["P"], case["n"], case["K"]
        d = _distinct(n, K)
        rule = case.get("rule", "gem")
        state = {"downpour": 4, "adaptive": 4, "momentum": 12}.get(rule, 16)   # m, s read and written
        b = P * (4 * K + 8 + state * d) + (4 * P if fam == "host" else 0) + (4 * P * K if fam == "pi" else 0)
        return {"bytes": b, "flops": 12 * P * K}
    b = case["b"]
    if fam.startswith("cnn"):
        H, c1, c2, f1, f2, C = _ints(case["shape"])
        P1 = (H - 4) // 2
        H2 = P1 - 4
        F = c2 * (H2 // 2) ** 2
        P = sum(math.prod(t) for t in _cnn_tensors(_ints(case["shape"])))
        conv1, conv2 = c1 * 25 * (H - 4) ** 2, c2 * c1 * 25 * H2 ** 2
        # forward, weight gradients, and input gradients down to conv1's output
        macs = 2 * conv1 + 3 * conv2 + 3 * (f1 * F + f2 * f1 + C * f2)
        x_bytes = 4 * H * H
    else:
        dims = _ints(case["dims"])
        P = _mlp_params(dims)
        macs = sum(3 * i * o for i, o in zip(dims, dims[1:])) - dims[0] * dims[1]
        x_bytes = 4 * dims[0]
    if fam.endswith("grad"):
        L = case["L"]
        return {"bytes": L * (8 * P + b * x_bytes), "flops": 2 * L * b * macs}
    T = case["T"]
    d = _distinct(case["n"], T)
    return {"bytes": P * (8 + 16 * d) + T * b * x_bytes, "flops": 2 * T * b * macs}


def tolerance(case):
    fam = case["family"]
    if fam in ("single", "batch", "host", "pi"):
        return "exact"     # gem.h fixes every operation and its order
    if case.get("tf32"):
        # measured against 64 bits: gradients 1.4e-2, moments 1.6e-2, theta 5e-4.  Rounding
        # softmax - onehot to TF32 makes the deeper gradients depend on 1-ulp changes at this level
        return {"rel": 3e-2}
    # fp32: measured against 64 bits: 1e-6 to 1e-5, and moments 1.2e-3 where a ReLU or a pooling
    # window within fp32 rounding of a tie takes the other branch and moves one sample's share
    # of a few gradient elements whole
    return {"rel": 5e-3, "max": 0.9}


# ------------------------------------------------------------------ the same in 64 bits

def _f32(x):
    return float(np.float32(x))


def _commit64(th, m, s, g, eta, rule, tau):
    """One commit in place on 64-bit vectors; returns the factors (None for momentum)."""
    dt = g.double() * -_f32(eta)
    pi = None
    if rule in ("downpour", "adaptive"):
        pi = torch.full_like(th, 1.0 if rule == "downpour" else 1.0 / (tau + 1.0))
        th.addcmul_(pi, dt)
    else:
        m.mul_(_f32(MU)).add_(dt)
        if rule == "momentum":
            th.add_(m)
        else:
            scale = {"kappa_sqrt": math.sqrt(2.5), "kappa_linear": 2.5}.get(rule, 1.0)
            pi = ((m.abs() * scale - (th - s).abs()) / (dt.abs() + _f32(EPS))).clamp_(min=0)
            th.addcmul_(pi, dt)
    s.copy_(th)
    return pi


def _medians(v, seg):
    lo, hi = [], []
    for a, e in zip(seg, seg[1:]):
        x = v[a:e].sort().values
        lo.append(x[(e - a - 1) // 2])
        hi.append(x[(e - a) // 2])
    return torch.stack(lo), torch.stack(hi)


def _padded(rows, stride):
    return torch.nn.functional.pad(rows, (0, stride - rows.shape[1]))


class _Truth:
    """theta, m and s of a handle in 64 bits; the moment and snapshot rows of the strided layout."""

    def __init__(self, s, eta, rule="gem"):
        P, n = s.G.P, s.G.n
        self.th = s.theta0.double()
        self.m = torch.zeros((n, s.G.stride), dtype=torch.float64, device="cuda")
        self.s = torch.zeros_like(self.m)
        self.s[:, :P] = self.th
        self.P, self.eta, self.rule, self.last, self.t = P, eta, rule, [-1] * n, 0

    def snapshot(self, w):
        return self.s[w, :self.P]

    def commit(self, w, g):
        tau = self.t - self.last[w] - 1
        self.last[w], self.t = self.t, self.t + 1
        return _commit64(self.th, self.m[w, :self.P], self.snapshot(w), g, self.eta, self.rule, tau)

    def out(self):
        return {"theta": self.th, "m": self.m, "s": self.s}


def _mlp_grad64(dims, theta, X, y):
    """Mean softmax cross-entropy of the rows and its gradient, in 64 bits."""
    off = _mlp_tensors(dims)
    W = [theta[off[2 * l]:off[2 * l + 1]].view(dims[l + 1], dims[l]) for l in range(len(dims) - 1)]
    A = [X.double()]
    for l, w in enumerate(W):
        z = A[-1] @ w.T + theta[off[2 * l + 1]:off[2 * l + 2]]
        A.append(z.relu() if l + 1 < len(W) else z)
    logp = A[-1].log_softmax(1)
    D = logp.exp()
    i = torch.arange(len(y), device="cuda")
    loss = -logp[i, y.long()].mean()
    D[i, y.long()] -= 1
    D /= len(y)
    g = torch.empty_like(theta)
    for l in reversed(range(len(W))):
        g[off[2 * l]:off[2 * l + 1]] = (D.T @ A[l]).reshape(-1)
        g[off[2 * l + 1]:off[2 * l + 2]] = D.sum(0)
        if l:
            D = (D @ W[l]) * (A[l] > 0)
    return loss, g


def _cnn_grad64(shape, theta, X, y, drop):
    F = torch.nn.functional
    parts, off = [], 0
    for t in _cnn_tensors(shape):
        k = math.prod(t)
        parts.append(theta[off:off + k].view(t).clone().requires_grad_(True))
        off += k
    w1, b1, w2, b2, f1, c1, f2, c2, f3, c3 = parts
    H = shape[0]
    with torch.enable_grad():
        h = F.max_pool2d(F.conv2d(X.double().view(-1, 1, H, H), w1, b1), 2).relu()
        h = F.max_pool2d(F.conv2d(h, w2, b2) * drop.double()[:, :, None, None], 2).relu().flatten(1)
        h = F.linear(F.linear(F.linear(h, f1, c1).relu(), f2, c2).relu(), f3, c3)
        loss = F.cross_entropy(h, y.long())
        grads = torch.autograd.grad(loss, parts)
    return loss.detach(), torch.cat([g.reshape(-1) for g in grads])


def exact(case, seed):
    s = prepare(case, seed)
    torch.cuda.synchronize()
    fam = case["family"]
    rule = case.get("rule", "gem")
    t = _Truth(s, CNN_ETA if fam.startswith("cnn") else ETA, rule)
    if fam in ("single", "batch", "host", "pi"):
        P = case["P"]
        pi, lo, hi = [], [], []
        for w, g in zip(s.order, s.grads):
            f = t.commit(w, g.cuda())
            if fam == "pi":
                a, b = _medians(f, s.seg)
                pi.append(f)
                lo.append(a)
                hi.append(b)
        out = t.out()
        if fam == "host":
            out["out"] = t.th.cpu()
        if fam == "pi":
            out.update(pi=torch.stack(pi), lo=torch.stack(lo), hi=torch.stack(hi))
        return out
    is_cnn = fam.startswith("cnn")
    shape = _ints(case["shape"]) if is_cnn else None
    dims = None if is_cnn else _ints(case["dims"])
    rows = torch.from_numpy(s.batch_rows.astype(np.int64)).cuda()

    def gradient(theta, k):
        r = rows[k]
        if is_cnn:
            return _cnn_grad64(shape, theta, s.X[r], s.y[r], s.drop[k])
        return _mlp_grad64(dims, theta, s.X[r], s.y[r])

    if fam.endswith("grad"):
        snaps = s.s.double()
        got = [gradient(snaps[int(w), :s.G.P], k) for k, w in enumerate(s.workers)]
        g = _padded(torch.stack([x[1] for x in got]), s.g.shape[1])
        return {"grads": g, "losses": torch.stack([x[0] for x in got])}
    # A run takes some 1e5 ReLU and pooling decisions per commit; a few lie within fp32 rounding
    # of a tie, and where one goes the other way theta, the moments and the medians move by 100
    # times the rounding itself and more.  How far a run is from the one in 64 bits says which
    # decisions flipped and not how precise it is (mlp_grad and cnn_grad say that), so of the
    # runs only the losses have a value here.
    losses = []
    for k, w in enumerate(int(x) for x in s.order):
        loss, g = gradient(t.snapshot(w), k)
        t.commit(w, g)
        losses.append(loss)
    return {"theta": None, "m": None, "s": None, "losses": torch.stack(losses),
            **({"lo": None, "hi": None} if case["pi"] else {})}
