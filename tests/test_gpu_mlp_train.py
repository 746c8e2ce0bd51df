"""The gradient and training kernels at the edges of their tiles (8, 16 and
32 samples) and of the rules that pick one, against the oracle's FP64
backward and an FP64 Adam.

Gradient: the bound of the existing 1000-sample test (1e-5 of its norm).
Training: a gradient good to 1e-5 moves an Adam step lr m / sqrt(v) of a
typical component by about 1e-5 of lr; components whose gradient is a
hundredth of the typical one by 1e-3 lr.  So the root mean square difference
after k steps stays below 1e-3 k lr (a batch with one sample too many or too
few, or an epoch in another order, moves it by at least lr / batch), and the
losses, smooth in the parameters, below 1e-4 relative.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_2601_03806_gb300 import flbm
    return flbm


@pytest.fixture(scope="module")
def M(oracle_mod):
    from oracle import mlp
    return mlp


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    return torch


def samples(M, n, seed):
    rng = np.random.default_rng(seed)
    theta = (M.init_params(seed) + 0.05 * rng.normal(size=M.NPARAM)).astype(np.float32)
    return theta, rng.normal(size=(n, 28)).astype(np.float32), rng.normal(size=(n, 27)).astype(np.float32)


def mt64(seed):
    """64-bit Mersenne twister (Nishimura 2000), as std::mt19937_64."""
    mask = (1 << 64) - 1
    s = [seed & mask]
    for i in range(1, 312):
        s.append((6364136223846793005 * (s[-1] ^ (s[-1] >> 62)) + i) & mask)
    while True:
        for i in range(312):
            x = (s[i] & 0xFFFFFFFF80000000) | (s[(i + 1) % 312] & 0x7FFFFFFF)
            s[i] = s[(i + 156) % 312] ^ (x >> 1) ^ (0xB5026F5AA96619E9 if x & 1 else 0)
        for x in s:
            x ^= (x >> 29) & 0x5555555555555555
            x ^= (x << 17) & 0x71D67FFFEDA60000
            x ^= (x << 37) & 0xFFF7EEE000000000
            yield x ^ (x >> 43)


# 152 SMs: tiles of 8 up to 1216 samples, of 16 up to 2432, of 32 beyond;
# 9728 samples fill two CTAs per SM, 700,000 more than 64 tiles per CTA
@pytest.mark.parametrize("n", [1, 7, 8, 9, 1216, 1217, 2432, 2433, 2465, 9729, 700001])
def test_gradient_at_tile_edges(F, M, torch_cuda, n):
    theta, x, t = samples(M, n, n)
    X, T = (torch_cuda.from_numpy(a).cuda() for a in (x, t))
    g, loss = F.mlp_grad(theta, X, T)
    go, lo = 0.0, 0.0
    for s in range(0, n, 100000):
        xs, ts = x[s:s + 100000].astype(float), t[s:s + 100000].astype(float)
        go = go + M.backward(theta.astype(float), xs, ts) * (len(xs) / n)
        lo += M.loss(theta.astype(float), xs, ts) * (len(xs) / n)
    assert abs(loss - lo) <= 1e-6 * lo
    assert np.linalg.norm(g - go) <= 1e-5 * np.linalg.norm(go)


def test_gradient_of_a_row_offset_by_one_float(F, M, torch_cuda):
    """Arrays aligned to 4 bytes only."""
    theta, x, t = samples(M, 100, 4)
    bx, bt = (torch_cuda.zeros(a.size + 1, device="cuda") for a in (x, t))
    bx[1:], bt[1:] = (torch_cuda.from_numpy(a).cuda().reshape(-1) for a in (x, t))
    g, _ = F.mlp_grad(theta, bx[1:].view(100, 28), bt[1:].view(100, 27))
    go = M.backward(theta.astype(float), x.astype(float), t.astype(float))
    assert np.linalg.norm(g - go) <= 1e-5 * np.linalg.norm(go)


@pytest.mark.parametrize("n,batch,epochs", [(5, 8, 3), (100, 1, 1), (1000, 96, 1), (5000, 1024, 2), (6000, 1300, 1),
                                            (9000, 4000, 2), (1, 4, 2), (1030, 1, 1)])
def test_training_follows_adam(F, M, torch_cuda, n, batch, epochs):
    theta0, x, t = samples(M, n, 7 * n + batch)
    seed, lr = 11, 1e-3
    X, T = (torch_cuda.from_numpy(a).cuda() for a in (x, t))
    theta, losses = F.mlp_train(theta0, X, T, epochs=epochs, batch=batch, lr=lr, seed=seed)
    rng, p, m1, m2, it, ref = mt64(seed), theta0.astype(float), 0.0, 0.0, 0, []
    b = min(batch, n)
    nb = -(-n // b)
    for _ in range(epochs):
        mult, off = 1, 0
        if n > 1:
            mult = 1 + next(rng) % (n - 1)
            while math.gcd(mult, n) != 1:
                mult = 1 + next(rng) % (n - 1)
            off = next(rng) % n
        order = (np.arange(n) * mult + off) % n
        total = 0.0
        for k in range(nb):
            i = order[k * b:(k + 1) * b]
            xs, ts = x[i].astype(float), t[i].astype(float)
            g = M.backward(p, xs, ts)
            total += M.loss(p, xs, ts) * len(i)
            m1, m2 = 0.9 * m1 + 0.1 * g, 0.999 * m2 + 0.001 * g * g
            rate = lr * (0.05 + 0.475 * (1 + math.cos(math.pi * it / max(epochs * nb - 1, 1))))
            it += 1
            p = p - rate * math.sqrt(1 - 0.999 ** it) / (1 - 0.9 ** it) * m1 / (np.sqrt(m2) + 1e-8)
        ref.append(total / n)
    assert np.sqrt(np.mean((theta - p) ** 2)) <= 1e-3 * it * lr
    assert np.abs(losses - ref).max() <= 1e-4 * max(ref)


def test_a_training_seed_gives_one_result(F, M, torch_cuda):
    theta0, x, t = samples(M, 3000, 2)
    X, T = (torch_cuda.from_numpy(a).cuda() for a in (x, t))
    a, la = F.mlp_train(theta0, X, T, epochs=2, batch=256, lr=1e-2, seed=3)
    b, lb = F.mlp_train(theta0, X, T, epochs=2, batch=256, lr=1e-2, seed=3)
    assert np.array_equal(a, b) and np.array_equal(la, lb)
