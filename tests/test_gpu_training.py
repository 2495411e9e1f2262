"""The network's training step (forward and backward tiles, the summed gradient,
Adam and the BF16 copies, launched as one chain) against its parts.

1. k full-batch epochs in one call give the parameters of k calls of one epoch,
   bit for bit: a one-epoch call starts with a plain launch and ends with a
   synchronisation.
2. Adam in numpy, fed by loss_grad on each minibatch, the last one ragged.
   Both sides' FP32 parameters agree to rounding, so now and then a weight
   falls on the other side of a BF16 boundary and moves the gradients it
   enters by about 2^-9 of one term; Adam turns a gradient's relative change
   into the same share of its step lr, except where the gradient nearly
   vanishes.  So all but 2% of the parameters must agree within 2% of a step;
   with gradients of weights one step old most do not (checked on the CPU)."""
import numpy as np
import pytest

LR, B1, B2, EPS = 0.05, 0.9, 0.999, 1e-8
CASES = [(1000, 384), (515, 512), (700, 128), (257, 257)]   # samples, batch


@pytest.fixture(scope="module")
def L():
    import torch
    assert torch.cuda.is_available()
    from paper_2103_10516_gb300 import build, mlt
    build.build()
    return mlt


def _data(n, seed=1):
    rng = np.random.default_rng(seed)
    x = rng.uniform(-1.0, 1.0, (n, 16)).astype(np.float32)
    return x, np.sin(2.0 * x[:, 0] + x[:, 3] * x[:, 5]).astype(np.float32)


class _Adam:
    def __init__(self, p):
        self.p, self.m, self.v, self.k = p.astype(np.float32), np.zeros(p.size, np.float32), np.zeros(p.size, np.float32), 0

    def step(self, g):
        f = np.float32
        self.k += 1
        self.m = f(B1) * self.m + f(1.0 - B1) * g
        self.v = f(B2) * self.v + f(1.0 - B2) * g * g
        c1, c2 = f(1.0 - B1 ** self.k), f(1.0 - B2 ** self.k)
        self.p = self.p - f(LR) * (self.m / c1) / (np.sqrt(self.v / c2) + f(EPS))


def _numpy_grad(p, x, t):
    """Loss gradient of the 16-128-128-1 ReLU network in FP64."""
    w1, b1, w2 = p[:2048].reshape(128, 16), p[2048:2176], p[2176:18560].reshape(128, 128)
    b2, w3, b3 = p[18560:18688], p[18688:18816], p[18816]
    a1 = x @ w1.T + b1
    h1 = np.maximum(a1, 0)
    a2 = h1 @ w2.T + b2
    h2 = np.maximum(a2, 0)
    dy = 2.0 * (h2 @ w3 + b3 - t) / x.shape[0]
    g2 = dy[:, None] * w3 * (a2 > 0)
    g1 = (g2 @ w2) * (a1 > 0)
    return np.concatenate([(g1.T @ x).ravel(), g1.sum(0), (g2.T @ h1).ravel(), g2.sum(0), dy @ h2, [dy.sum()]])


def _off(p, q):
    return np.mean(np.abs(p - q) > 0.02 * LR)


def _init(rng):
    return np.concatenate([rng.standard_normal(2048) * (2 / 16) ** 0.5, np.zeros(128),
                           rng.standard_normal(16384) * (2 / 128) ** 0.5, np.zeros(128),
                           rng.standard_normal(128) / 128 ** 0.5, [0.0]]).astype(np.float32)


@pytest.mark.parametrize("n,batch", [c for c in CASES if c[0] > c[1]])
def test_stale_weights_show(n, batch):
    x, t = (v.astype(np.float64) for v in _data(n))
    good, stale = _Adam(_init(np.random.default_rng(5))), _Adam(_init(np.random.default_rng(5)))
    old = stale.p
    for b in range(0, n, batch):
        good.step(_numpy_grad(good.p.astype(np.float64), x[b:b + batch], t[b:b + batch]).astype(np.float32))
        now = stale.p
        stale.step(_numpy_grad(old.astype(np.float64), x[b:b + batch], t[b:b + batch]).astype(np.float32))
        old = now
    assert _off(good.p, stale.p) > 0.4


@pytest.mark.gpu
@pytest.mark.parametrize("n", [100, 128, 1000, 2176])
def test_epochs_in_one_call_equal_single_epochs(L, n):
    x, t = _data(n)
    with L.Surrogate(seed=3) as one, L.Surrogate(seed=3) as many:
        last = one.train(x, t, epochs=6, batch=n, lr=LR)
        for _ in range(6):
            each = many.train(x, t, epochs=1, batch=n, lr=LR)
        assert np.array_equal(one.get_params(), many.get_params())
        assert last == each
        assert np.array_equal(one.predict(x), many.predict(x))


@pytest.mark.gpu
@pytest.mark.parametrize("n,batch", CASES)
def test_minibatches_against_numpy_adam(L, n, batch):
    x, t = _data(n)
    with L.Surrogate(seed=3) as net, L.Surrogate(seed=3) as ref:
        adam = _Adam(ref.get_params())
        losses = 0.0
        for b in range(0, n, batch):
            loss, g = ref.loss_grad(x[b:b + batch], t[b:b + batch])
            losses += loss * len(x[b:b + batch])
            adam.step(g)
            ref.set_params(adam.p)
        got = net.train(x, t, epochs=1, batch=batch, lr=LR)
        assert _off(net.get_params(), adam.p) <= 0.02
        # the losses of the steps before the last update: FP32 sums of BF16 products
        assert abs(got - losses / n) <= 0.01 * losses / n
