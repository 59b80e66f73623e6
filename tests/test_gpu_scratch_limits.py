"""Reshapes that reduce an axis and transpose take an intermediate array where
there is memory for it, and do without it where a context's cap or the static
array leaves none: the same bits either way, and nothing refused that fits
without it."""
import numpy as np
import pytest

import paper_1609_00061_gb300 as pa
from paper_1609_00061_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def network(k, m, n):
    """R1(k, p, m), R2(k, n), (m, n) exposed: R1 is reduced over p and transposed."""
    axes = [(-1.0, 1.0, k), (-1.0, 1.0, 2), (-1.0, 1.0, m), (-1.0, 1.0, n)]
    rels = [W.Relation((0, 1, 2), 1, [0.1, 1.0, 0.3, -0.7]), W.Relation((0, 3), 1, [0.05, 1.0, 0.9])]
    return W.System("reduced and transposed", axes, rels, (2, 3))


def solve(engine, sysm):
    out = pa.BitArray.empty(sysm.exposed, [sysm.axes[v][2] for v in sysm.exposed], 0)
    out.words.fill_(-1)
    st = pa.pa_solve_network(engine.ctx, sysm.axes, sysm.rels, sysm.exposed, out)
    engine.sync()
    return out, st


def test_capped_workspace(orc):
    sysm = network(1024, 1000, 300)
    eng = pa.Engine(0)
    eng.set_path("rowor")
    full, st = solve(eng, sysm)
    want = orc.solve(sysm.axes, sysm.rels, sysm.exposed).data
    assert np.array_equal(full.to_numpy(), want)
    eng.close()
    capped = pa.Engine(0, workspace_cap=st["workspace_bytes"] - (64 << 10))
    capped.set_path("rowor")
    for call in range(3):  # planned, kept, replayed
        out, st2 = solve(capped, sysm)
        assert np.array_equal(out.to_numpy(), want), call
        assert st2["workspace_bytes"] < st["workspace_bytes"] - (64 << 10)
    capped.close()


def test_static_array():
    sysm = network(6400, 6528, 64)
    eng = pa.Engine(0)
    eng.set_path("rowor")
    full, st = solve(eng, sysm)
    assert st["workspace_bytes"] > 16 << 20  # with the intermediate
    eng.close()
    out = pa.BitArray.empty(sysm.exposed, [sysm.axes[v][2] for v in sysm.exposed], 0)
    out.words.fill_(-1)
    st2 = pa.pa_solve_network_static(sysm.axes, sysm.rels, sysm.exposed, out)
    assert st2["workspace_bytes"] <= 16 << 20
    assert np.array_equal(out.to_numpy(), full.to_numpy())
