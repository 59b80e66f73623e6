"""The cost model's sums have one order (bias first, then the terms as they are
numbered, fused multiply-adds), for every batch size: predictions, loss and
gradients equal those of the same chains on the host, bit for bit.  A unit whose
sum ends within rounding of zero gets its ReLU mask from that order."""
import numpy as np
import pytest

import paper_1609_00061_gb300 as pa

pytestmark = pytest.mark.gpu

F32 = np.float32


@pytest.fixture(scope="module")
def eng():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    e = pa.Engine(0)
    yield e
    e.close()


def fma(a, b, c):
    """Correctly rounded FP32 a b + c: the product is exact in 64 bits, the sum is
    rounded to odd there, so that rounding it to 32 bits rounds once."""
    p, c = a.astype(np.float64) * b.astype(np.float64), c.astype(np.float64)
    s = p + c
    t = s - p
    err = (p - (s - t)) + (c - t)
    even = (s.view(np.int64) & 1) == 0
    s = np.where((err != 0) & even, np.nextafter(s, np.where(err > 0, np.inf, -np.inf)), s)
    return s.astype(F32)


def chain(start, A, B):
    """start[n][m] + sum_k A[n][k] B[m][k], k in order."""
    acc = start.astype(F32)
    for k in range(A.shape[1]):
        acc = fma(np.broadcast_to(A[:, k:k + 1], acc.shape), np.broadcast_to(B[:, k], acc.shape), acc)
    return acc


def reference(p, sizes, X, T):
    Ws, bs, at = [], [], 0
    for ni, no in zip(sizes[:-1], sizes[1:]):
        Ws.append(p[at:at + no * ni].reshape(no, ni))
        bs.append(p[at + no * ni:at + no * (ni + 1)])
        at += no * (ni + 1)
    n, acts = len(X), [X]
    for l, (W, b) in enumerate(zip(Ws, bs)):
        z = chain(np.broadcast_to(b, (n, len(b))), acts[-1], W)
        acts.append(z if l + 1 == len(Ws) else np.where(z < 0, F32(0), z))
    y = acts[-1][:, 0]
    e = y - T
    part = np.zeros(256, F32)
    for k in range(n):
        part[k % 256] += e[k] * e[k]
    w = 128
    while w:
        part[:w] += part[w:2 * w]
        w //= 2
    d = (e / F32(n))[:, None]
    grads = []
    for l in range(len(Ws) - 1, -1, -1):
        gw = chain(np.zeros(Ws[l].shape, F32), np.ascontiguousarray(d.T), np.ascontiguousarray(acts[l].T))
        gb = np.zeros(d.shape[1], F32)
        for r in range(n):
            gb = gb + d[r]
        grads[:0] = [gw.reshape(-1), gb]
        if l:
            below = chain(np.zeros((n, sizes[l]), F32), d, np.ascontiguousarray(Ws[l].T))
            d = np.where(acts[l] > 0, below, F32(0))
    return y, F32(0.5) * part[0] / F32(n), np.concatenate(grads)


@pytest.mark.parametrize("hidden,nlayers,n", [
    (1, 0, 3), (5, 1, 1), (16, 2, 304), (33, 2, 305), (128, 3, 256), (130, 2, 608),
    (129, 1, 700), (260, 2, 37), (8, 8, 1216), (20, 1, 1300), (1024, 1, 9)])
def test_sums_in_order(eng, hidden, nlayers, n):
    import torch
    m = pa.CostModel(eng, hidden=hidden, nlayers=nlayers, seed=1)
    sizes = [pa.N_FEATURES] + [hidden] * nlayers + [1]
    rng = np.random.default_rng(1000 * hidden + 10 * nlayers + n)
    p = rng.normal(size=m.n_params).astype(F32) * F32(0.3)
    X = rng.normal(size=(n, pa.N_FEATURES)).astype(F32)
    T = rng.normal(size=n).astype(F32)
    m.set_params(p)
    y, loss, grads = reference(p, sizes, X, T)
    xd, td = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
    assert np.array_equal(m.forward(xd).cpu().numpy(), y)
    assert F32(m.backward(xd, td)) == loss
    assert np.array_equal(m.get_grads(), grads)
    m.close()


@pytest.mark.parametrize("n", [2, 400, 1000])
def test_mask_of_a_cancelling_sum(eng, n):
    """bias + big - big: the bias is lost in the first addition, the unit is off."""
    import torch
    m = pa.CostModel(eng, hidden=2, nlayers=1, seed=1)
    W = np.zeros((2, pa.N_FEATURES), F32)
    W[:, 0], W[:, 1] = 2.0 ** 26, -2.0 ** 26
    p = np.concatenate([W.reshape(-1), [F32(1), F32(-1)], [F32(3), F32(5)], [F32(7)]]).astype(F32)
    m.set_params(p)
    x = torch.ones(n, pa.N_FEATURES, device="cuda")
    assert torch.equal(m.forward(x), torch.full((n,), 7.0, device="cuda"))
    m.backward(x, torch.zeros(n, device="cuda"))
    g = m.get_grads()
    assert not g[:2 * pa.N_FEATURES + 4].any()  # nothing reaches the units that are off
    m.close()
