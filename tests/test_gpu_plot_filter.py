"""The plot kernel's FP32 filter where it can go wrong: rows that end inside a
word or an 8-pixel piece, rows longer than one pass of the kernel, many pixels
inside the filter's error bound, boxes far from zero and high degrees.  Every
plot equals the oracle's bit for bit (the FP64 decision has no tolerance)."""
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


def check(eng, orc, rel, axes, what, strict=False):
    got = eng.plot(rel, axes, strict=strict)
    want = orc.plot_relation(rel, axes, strict=strict).data
    diff = int((got.to_numpy() != want).sum())
    assert diff == 0, f"{what}: {diff} of {want.size} pixels differ"
    assert got.padding_clean(), what
    return want


@pytest.mark.parametrize("res", [2, 5, 12, 17, 31, 33, 48, 63, 65, 80, 97, 129, 495])
@pytest.mark.parametrize("degree", [1, 2, 3, 4, 5])
def test_row_ends(eng, orc, res, degree):
    rng = W.SplitMix64(7000 + 16 * res + degree)
    for arity, lead in ((2, [37]), (3, [9, 11])):
        axes = [(-2.0, 1.5, r) for r in lead] + [(-1.25, 2.0, res)]
        for kind in (W.KIND_EQ, W.KIND_LE, W.KIND_LT):
            rel = W.Relation(tuple(range(arity)), degree,
                             rng.normal(W.coeff_count(arity, degree)), kind)
            check(eng, orc, rel, axes, f"arity {arity} kind {kind}")


@pytest.mark.parametrize("shape", [(200001,), (3, 140000), (2, 2, 131072 + 70), (4097, 2)])
def test_long_rows_and_many_rows(eng, orc, shape):
    rng = W.SplitMix64(7100 + shape[-1])
    n = len(shape)
    axes = [(-1.0, 2.0, r) for r in shape]
    for kind in (W.KIND_EQ, W.KIND_LE):
        rel = W.Relation(tuple(range(n)), 3, rng.normal(W.coeff_count(n, 3)), kind)
        check(eng, orc, rel, axes, f"{shape} kind {kind}")


@pytest.mark.parametrize("case", range(6))
def test_pixels_inside_the_bound(eng, orc, case):
    """Thousands of centres with |f| - eps at or near zero."""
    axes = [(0.0, 3.0, 300), (0.0, 3.0, 333)] if case % 2 else [(0.0, 3.0, 300)] * 2
    # f = a x - b y: |f| = eps along whole lines of centres, not representable in FP32
    a, b = (0.1, 0.1) if case < 2 else (0.1, 0.3) if case < 4 else (1e-3, 1e-3)
    eps = 10 * a * 0.01
    for strict in (False, True):
        for kind in (W.KIND_EQ, W.KIND_LE, W.KIND_LT):
            rel = W.Relation((0, 1), 1, [0.0, a, -b], kind, eps)
            check(eng, orc, rel, axes, f"a {a} b {b} strict {strict} kind {kind}", strict)
    rel = W.Relation((0, 1), 3, [0, 0, 0, 0, 0, 0, 1, -3, 3, -1], W.KIND_EQ, 0.0)  # (x - y)^3
    check(eng, orc, rel, axes, "eps 0")
    rel = W.Relation((0, 1), 3, [0, 0, 0, 0, 0, 0, 1, -3, 3, -1], W.KIND_EQ, 1e-9)
    check(eng, orc, rel, axes, "eps 1e-9")


@pytest.mark.parametrize("lo", [100.0, -1000.0, 1e6])
def test_boxes_far_from_zero(eng, orc, lo):
    rng = W.SplitMix64(7200 + int(abs(lo)))
    axes = [(lo, lo + 1.0, 90), (lo - 3.0, lo - 2.5, 150), (lo, lo + 0.25, 100)]
    for vs, degree in (((0, 1), 3), ((1, 0, 2), 2), ((0,), 4)):
        c = rng.normal(W.coeff_count(len(vs), degree))
        # move the solution set into the box: the constant term cancels f at its middle
        mid = [axes[v][0] + 0.5 * (axes[v][1] - axes[v][0]) for v in vs]
        c[0] -= orc.eval_poly(degree, c, mid)
        for eps in (-1.0, 1e-6 * abs(lo) ** (degree - 1)):
            rel = W.Relation(vs, degree, c, W.KIND_EQ, eps)
            check(eng, orc, rel, axes, f"{vs} degree {degree} eps {eps}")


@pytest.mark.parametrize("arity,degree", [(1, 16), (2, 9), (2, 16), (3, 6), (4, 3), (5, 2)])
def test_generic_degrees(eng, orc, arity, degree):
    rng = W.SplitMix64(7300 + 32 * arity + degree)
    res = {1: 3000, 2: 200, 3: 40, 4: 14, 5: 8}[arity]
    axes = [(-1.3 + 0.1 * p, 1.2 + 0.05 * p, res + p) for p in range(arity)]
    for kind in (W.KIND_EQ, W.KIND_LT):
        for eps in (-1.0, 0.01):
            rel = W.Relation(tuple(range(arity)), degree,
                             rng.normal(W.coeff_count(arity, degree)), kind, eps)
            check(eng, orc, rel, axes, f"kind {kind} eps {eps}")
