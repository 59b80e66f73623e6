"""The row-OR at the edges of its dispatch: every tile width, the three ways a
tile is staged (one run of memory, 2-D boxes, 8-byte copies), rows per warp
batch from 1 to 32, K ranges around one and several chunks, lists that overflow
into windows, and problems with few and many CTAs.  Bit for bit against the
oracle's cluster (Eq. GAM)."""
import numpy as np
import pytest

import paper_1609_00061_gb300 as pa

from test_gpu_parity import pack

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


def bits(rng, shape, kind):
    """Runs like a thick curve's ("runs"), scattered bits or nearly full rows."""
    if kind == "runs":
        out = np.zeros(shape, np.uint8).reshape(-1, shape[-1])
        for r in range(out.shape[0]):
            for _ in range(rng.integers(0, 4)):
                s = int(rng.integers(0, shape[-1]))
                out[r, s:s + int(rng.integers(1, 90))] = 1
        return out.reshape(shape)
    return (rng.random(shape) < {"sparse": 0.01, "half": 0.5, "full": 0.999}[kind]).astype(np.uint8)


def check(eng, orc, x, y, xv, yv, keep, res):
    got = eng.contract(pack(x, xv), pack(y, yv), keep)
    want = orc.contract(orc.Arr(x, xv), orc.Arr(y, yv), keep, res).data
    diff = int((got.to_numpy() != want).sum())
    assert diff == 0, f"{diff} of {want.size} pixels differ"
    assert got.padding_clean()


@pytest.mark.parametrize("N", [64, 128, 190, 256, 300, 512, 600, 1024, 1090, 2048, 2100])
@pytest.mark.parametrize("K", [63, 65, 320, 577, 1100])
def test_widths_and_lengths(eng, orc, N, K):
    rng = np.random.default_rng(N * 10000 + K)
    for M, kind in ((3, "half"), (70, "runs"), (523, "sparse")):
        x, y = bits(rng, (M, K), kind), bits(rng, (K, N), "runs")
        check(eng, orc, x, y, (0, 1), (1, 2), (0, 2), [M, K, N])


@pytest.mark.parametrize("K", [2047, 2048, 2049, 2400, 4097, 20000])
@pytest.mark.parametrize("N", [50, 130, 512])
def test_chunked_k(eng, orc, K, N):
    rng = np.random.default_rng(N * 100000 + K)
    for M, kind in ((1, "full"), (40, "half"), (130, "runs")):
        x, y = bits(rng, (M, K), kind), bits(rng, (K, N), "sparse")
        check(eng, orc, x, y, (0, 1), (1, 2), (0, 2), [M, K, N])


@pytest.mark.parametrize("nb,M,K,N", [(9, 33, 65, 64), (200, 20, 96, 130), (170, 64, 512, 512),
                                      (12, 5, 33, 1000), (160, 3, 129, 63)])
def test_shared_batch_axis(eng, orc, nb, M, K, N):
    rng = np.random.default_rng(nb * 1000 + K)
    for kind in ("runs", "half"):
        x, y = bits(rng, (nb, M, K), kind), bits(rng, (nb, K, N), "runs")
        check(eng, orc, x, y, (0, 1, 2), (0, 2, 3), (0, 1, 3), [nb, M, K, N])


# A single cluster whose K range fits one chunk: no second chunk, and so no launch
# that clears the result, even where CTAs are few.  (Next to tiles of 32 words a chunk
# has at most 576 rows.)
@pytest.mark.parametrize("M,K,N,chunks", [(6611, 653, 911, 1), (700, 700, 100, 1), (64, 2048, 64, 1),
                                          (300, 600, 2100, 2)])
def test_single_cluster_has_one_launch(eng, orc, M, K, N, chunks):
    rng = np.random.default_rng(M + K + N)
    x, y = bits(rng, (M, K), "runs"), bits(rng, (K, N), "runs")
    pa.pa_profile_enable(eng.ctx)
    try:
        pa.pa_profile_read(eng.ctx)
        check(eng, orc, x, y, (0, 1), (1, 2), (0, 2), [M, K, N])
        names = pa.pa_profile_read(eng.ctx)
    finally:
        pa.pa_profile_enable(eng.ctx, False)
    names.pop("words_or")  # a counter
    assert sorted(names) == (["rowor_kernel"] if chunks == 1 else ["memset", "rowor_kernel"]), names
