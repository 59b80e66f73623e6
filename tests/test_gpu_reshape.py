"""Reshapes into matrix form at the edges of their kernels: permutations whose
last axis is a run of 1, 2, 3 or 4 words, transposes around the 256-value
tiles, reductions over few and many values (by words, by whole rows, and
together with a permutation), through clusters against the oracle."""
import numpy as np
import pytest

import paper_1609_00061_gb300 as pa

from test_gpu_parity import check_same, pack, rand_bits

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    e = pa.Engine(0)
    e.set_path("rowor")
    yield e
    e.close()


CASES = [
    # (X vars, Y vars, keep, res by var)
    ((1, 0), (1, 2), (0, 2), [65, 300, 70]),                 # A transposed
    ((1, 0), (2, 1), (0, 2), [257, 255, 513]),               # both transposed
    ((1, 0, 3), (1, 2), (0, 3, 2), [64, 70, 66, 128]),       # words moved, runs of 2
    ((1, 0, 3), (1, 2), (0, 3, 2), [33, 40, 66, 192]),       # runs of 3
    ((1, 0, 3), (1, 2), (0, 3, 2), [20, 30, 66, 512]),       # runs of 4
    ((0, 4, 1), (1, 2), (0, 2), [50, 64, 70, 1, 300]),       # a private axis in the middle
    ((1, 4, 0), (1, 2), (0, 2), [128, 64, 70, 1, 300]),      # the same, then transposed
    ((1, 0, 4), (1, 2), (0, 2), [128, 96, 70, 1, 300]),      # the packed axis private, transposed
    ((0, 1, 4, 5), (1, 2), (0, 2), [9, 64, 70, 1, 60, 200]),  # two private axes, rows of words
    ((4, 0, 1), (1, 2), (0, 2), [3, 64, 70, 1, 4000]),       # few results, long reduction
    ((4, 1), (1, 2), (2,), [1, 64, 70, 1, 5000]),
    ((0, 1), (2, 0), (1, 2), [300, 520, 290]),
    ((0, 1, 2), (0, 1, 2), (2, 0, 1), [70, 64, 65]),         # Hadamard, permuted
    ((0, 1), (0, 2), (0, 1, 2), [65, 130, 66]),              # outer product per batch value
    ((0, 1), (0, 1), (0,), [500, 1000]),                     # dots of short and long rows
    ((0, 1), (0, 1), (0,), [70, 5000]),
]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("density", [0.004, 0.3])
def test_reshaped_clusters(eng, orc, case, density):
    xv, yv, keep, vres = CASES[case]
    rng = np.random.default_rng(8800 + 10 * case + int(100 * density))
    X = rand_bits(rng, tuple(vres[v] for v in xv), density)
    Y = rand_bits(rng, tuple(vres[v] for v in yv), density)
    want = orc.contract(orc.Arr(X, xv), orc.Arr(Y, yv), keep, vres).data
    got = eng.contract(pack(X, xv), pack(Y, yv), keep)
    eng.sync()
    check_same(got, want, str(CASES[case]))


@pytest.mark.parametrize("vres", [(310, 70, 65), (320, 33, 257), (305, 256, 64), (306, 1, 130),
                                  (40, 300, 800)])
def test_many_transposes(eng, orc, vres):
    """Transposes of more tiles than the GPU takes at once (a 32 x 32 block per
    thread), and of wide tiles: every edge of blocks, words and tiles."""
    rng = np.random.default_rng(8900 + sum(vres))
    X, Y = rand_bits(rng, vres, 0.4), rand_bits(rng, vres, 0.6)
    want = orc.contract(orc.Arr(X, (0, 1, 2)), orc.Arr(Y, (0, 1, 2)), (0, 2, 1), list(vres)).data
    got = eng.contract(pack(X, (0, 1, 2)), pack(Y, (0, 1, 2)), (0, 2, 1))
    eng.sync()
    check_same(got, want, str(vres))


def test_transpose_beyond_32_bit_indexes(eng):
    """An operand of more than 2^31 words, its last axis moved to the front: the
    transpose counts words in 64 bits."""
    import torch
    M, K, N, T = (1 << 15) + 64, 1 << 16, 64, 64
    free, _ = torch.cuda.mem_get_info()
    if free < 80 << 30:
        pytest.skip("needs 80 GB of device memory")
    A = pa.BitArray.empty((0, 1, 3), (M, K, T), 0)
    B = pa.BitArray.empty((1, 2, 3), (K, N, T), 0)
    a, b = A.words.view(M, K), B.words.view(K, N)
    a.zero_()
    b.zero_()
    rng = np.random.default_rng(1)
    m = np.concatenate([[0, M - 1, M - 1, 0], rng.integers(0, M, 400)])
    k = np.concatenate([[0, K - 1, 0, K - 1], rng.integers(0, K, 400)])
    n = rng.integers(0, N, len(m))
    av, bv = {}, {}  # one to three values of the last axis per place
    for i in range(len(m)):
        t = rng.integers(0, T, 3)
        av[m[i], k[i]] = av.get((m[i], k[i]), 0) | (1 << int(t[0])) | (1 << int(t[1]))
        bv[k[i], n[i]] = bv.get((k[i], n[i]), 0) | (1 << int(t[0])) | (1 << int(t[2]))

    def put(dst, values):
        at = torch.tensor(list(values), device="cuda")
        dst[at[:, 0], at[:, 1]] = torch.from_numpy(np.array(list(values.values()), np.uint64).view(np.int64)).cuda()

    put(a, av)
    put(b, bv)
    want = np.zeros((M, N), np.uint64)
    for (mi, ki), x in av.items():
        for (kj, nj), y in bv.items():
            if ki == kj:
                want[mi, nj] |= np.uint64(x & y)
    got = eng.contract(A, B, (0, 2, 3))
    eng.sync()
    assert np.array_equal(got.words.view(M, N).cpu().numpy().view(np.uint64), want)
    assert want.any()
    del A, B, a, b, got
    torch.cuda.empty_cache()
