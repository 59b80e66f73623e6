"""The plot kernel's FP32 error bound where it is widest against what the kernel
evaluates.  Every plot equals the oracle's bit for bit (the FP64 decision has no
tolerance)."""
import itertools

import numpy as np
import pytest

import paper_1609_00061_gb300 as pa
from paper_1609_00061_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    e = pa.Engine(0)
    yield e
    e.close()


def check(eng, orc, rel, axes, what):
    got = eng.plot(rel, axes)
    want = orc.plot_relation(rel, axes).data
    diff = int((got.to_numpy() != want).sum())
    assert diff == 0, f"{what}: {diff} of {want.size} pixels differ"
    assert got.padding_clean(), what


# Rows that end inside a word, in plots with more undecided words per block than
# threads take piece by piece: the word's pixels are evaluated about its middle.
@pytest.mark.parametrize("res", [17, 20, 31, 33, 36, 40, 48, 63, 81, 97])
@pytest.mark.parametrize("degree", [3, 6, 8, 12, 16])
def test_partial_words_at_high_degree(eng, orc, res, degree):
    rng = W.SplitMix64(8000 + 32 * res + degree)
    for box, eps in ((3.0, 0.05), (1.0, 0.05), (1.0, 0.01)):
        for one_sided in (False, True):
            axes = [(-box, box, 256), (0.0 if one_sided else -box, box, res)]
            for kind in (W.KIND_EQ, W.KIND_LE, W.KIND_LT):
                rel = W.Relation((0, 1), degree, rng.normal(W.coeff_count(2, degree)), kind, eps)
                check(eng, orc, rel, axes, f"box {box} one-sided {one_sided} kind {kind}")


# The same in pieces of 8 pixels, the last of which ends inside (few rows).
@pytest.mark.parametrize("res", [5, 6, 7, 13, 21, 38, 71])
@pytest.mark.parametrize("degree", [3, 8, 16])
def test_partial_pieces_at_high_degree(eng, orc, res, degree):
    rng = W.SplitMix64(8100 + 32 * res + degree)
    for rows in (3, 24):
        for box in (1.0, 3.0):
            axes = [(-box, box, rows), (-box, box, res)]
            for kind in (W.KIND_EQ, W.KIND_LT):
                rel = W.Relation((0, 1), degree, rng.normal(W.coeff_count(2, degree)), kind, 0.05)
                check(eng, orc, rel, axes, f"rows {rows} box {box} kind {kind}")


def small_box(rng, box, degree, shape, kind, eps):
    """N(0,1) coefficients in units of the box: every monomial counts on it."""
    n = len(shape)
    c = rng.normal(W.coeff_count(n, degree))
    axes = [(-box, box, r) for r in shape]
    return W.Relation(tuple(range(n)), degree, c / box ** total_degrees(n, degree), kind, eps), axes


def total_degrees(n, degree):
    """Total degree of every coefficient (graded order)."""
    out = []
    for d in range(degree + 1):
        out += [d] * (W.coeff_count(n, d) - (W.coeff_count(n, d - 1) if d else 0))
    return np.array(out, dtype=np.float64)


# Coefficients beyond FP32's range on a box so small that f is of order one.
@pytest.mark.parametrize("box,degree", [(1e-10, 4), (1e-12, 3), (1e-20, 2), (1e-3, 16), (1e-40, 1)])
def test_coefficients_beyond_fp32(eng, orc, box, degree):
    rng = W.SplitMix64(8200 + degree)
    for kind in (W.KIND_EQ, W.KIND_LE, W.KIND_LT):
        for shape in ((300, 333), (31, 2000)):
            for eps in (-1.0, 0.01):
                rel, axes = small_box(rng, box, degree, shape, kind, eps)
                check(eng, orc, rel, axes, f"{shape} kind {kind} eps {eps}")
    rel, axes = small_box(rng, box, degree, (17, 19, 70), W.KIND_EQ, -1.0)
    check(eng, orc, rel, axes, "3 ports")


# Large coefficients within FP32's range on small boxes: powers of the pixel width
# and of the coordinates fall below it.
@pytest.mark.parametrize("box,degree", [(1e-9, 4), (1e-6, 5), (1e-2, 16), (0.1, 16), (1e-4, 8),
                                        (1e-1, 12), (1e-7, 3)])
def test_powers_below_fp32(eng, orc, box, degree):
    rng = W.SplitMix64(8300 + degree)
    for kind in (W.KIND_EQ, W.KIND_LE):
        for shape in ((500, 333), (500, 64), (90, 1500)):
            for eps in (-1.0, 0.01, 1e-4):
                rel, axes = small_box(rng, box, degree, shape, kind, eps)
                check(eng, orc, rel, axes, f"{shape} kind {kind} eps {eps}")
    rel, axes = small_box(rng, box, min(degree, 6), (17, 19, 70), W.KIND_EQ, -1.0)
    check(eng, orc, rel, axes, "3 ports")


# Boxes of very different sizes on the ports, coefficients to match; values of f
# far from one; plots in which every pixel, or none, is on.
@pytest.mark.parametrize("boxes", [(1e-12, 1e6), (1e6, 1e-12), (1e15, 1e-15), (1e-3, 3e5, 1e-8), (1e17, 1e17)])
@pytest.mark.parametrize("scale", [1.0, 1e-40, 1e60, 1e-200])
def test_uneven_boxes_and_scales(eng, orc, boxes, scale):
    n, degree = len(boxes), 3
    rng = W.SplitMix64(8400 + int(np.log10(scale)))
    c = rng.normal(W.coeff_count(n, degree)) * scale
    for e in itertools.product(range(degree + 1), repeat=n):
        if sum(e) <= degree:
            c[orc.coeff_index(e, degree)] /= np.prod([b ** float(k) for b, k in zip(boxes, e)])
    shape = (61, 190) if n == 2 else (9, 11, 140)
    axes = [(-b, 0.9 * b, r) for b, r in zip(boxes, shape)]
    for kind in (W.KIND_EQ, W.KIND_LT):
        for eps in (-1.0, 0.0, 0.02 * scale, 1e30 * scale):
            rel = W.Relation(tuple(range(n)), degree, c, kind, eps)
            check(eng, orc, rel, axes, f"kind {kind} eps {eps}")


# FP64 sums that overflow on the way make the pixel's value infinite: off.
def test_fp64_overflow_on_the_way(eng, orc):
    # port 0 innermost: c x0 overflows before the tiny x1 brings it back
    axes = [(1e10, 2e10, 70), (1e-20, 2e-20, 70)]
    c = np.zeros(W.coeff_count(2, 2))
    c[orc.coeff_index((1, 1), 2)] = 1e300
    for kind, eps in ((W.KIND_LE, 1e300), (W.KIND_EQ, 1e300), (W.KIND_LT, 2e290)):
        check(eng, orc, W.Relation((0, 1), 2, c, kind, eps), axes, f"kind {kind}")
