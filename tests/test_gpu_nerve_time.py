"""Nerves of covers with many elements per point end in the time of their pairs.
The limits are several times what the pairs take and a small part of what the
faults named beside them took."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
mg = pytest.importorskip("paper_2011_03209_gb300")

pytestmark = pytest.mark.gpu


def _nerve_ms(X, nint, ov, eps, min_pts):
    m = len(nint)
    Xd = torch.from_numpy(X).to("cuda:0")
    torch.cuda.synchronize()
    prm = mg.params((mg.LENS_COORD,) * m, tuple(range(m)), nint, ov, eps, min_pts, mg.FP32)
    ms = []
    with mg.Context(0) as ctx:
        ctx.set_timing(True)
        for _ in range(4):
            g = mg.mapper_graph(ctx, Xd, prm)
            ms.append(g.stats()["ms_nerve"])
        got = g.numpy()
        lens, _ = g.lens(len(X), m)
    ref = oracle.mapper_graph(X, lens, nint, ov, eps, min_pts)
    for k in ("node_offsets", "node_members", "node_elem", "edges"):
        assert np.array_equal(np.asarray(got[k]), np.asarray(ref[k])), k
    return min(ms), len(got["edges"])


def test_more_edges_than_the_set_holds():
    # 113k edges of 1.6 M pairs: the sort takes 0.6 ms, every pair through the full set 39
    X = np.random.default_rng(5).uniform(-1, 1, (1000, 3)).astype(np.float32)
    ms, edges = _nerve_ms(X, (30, 30), (0.9, 0.9), 0.4, 3)
    assert edges > 32768
    assert ms < 10.0, ms


def test_points_in_many_elements():
    # up to 250 elements a point, 31k pairs each; all of at most 32385 edges. A
    # thread a point took 20 ms and more
    X = np.random.default_rng(6).uniform(-1, 1, (2000, 3)).astype(np.float32)
    ms, edges = _nerve_ms(X, (255,), (0.996,), 0.5, 3)
    assert 20_000 < edges <= 32768
    assert ms < 6.0, ms
