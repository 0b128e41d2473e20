"""Graphs, forests and eccentricities at the edges of the dispatch rules: more
edges than the nerve's hash set holds, more elements than the layout kernels
and the pair search take in one go, enough rows for several hooking rounds, a
queue of tied distances that overflows, values outside the FP32 expansion."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
mg = pytest.importorskip("paper_2011_03209_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = mg.Context(0)
    yield c
    c.close()


def _device(X):
    Xd = torch.from_numpy(np.ascontiguousarray(X)).to("cuda:0")
    torch.cuda.synchronize()
    return Xd


# edges: a point in k elements that is a node of its own in each gives
# k (k - 1) / 2 (13.5k and 101k edges here). elements: 70^2 = 4900, 135^2 =
# 18225. rows: 175k (several hooking rounds)
@pytest.mark.parametrize("n,d,nint,ov,eps,min_pts,prec", [
    (4000, 3, (13, 11), (0.45, 0.45), 1e-6, 1, mg.BF16),         # the hash set
    (30_000, 3, (13, 11), (0.45, 0.45), 1e-6, 1, mg.FP32),       # more edges than it holds
    (6000, 3, (70, 70), (0.3, 0.3), 0.2, 2, mg.BF16),
    (6000, 3, (135, 135), (0.3, 0.3), 0.2, 2, mg.FP32),
    (140_000, 2, (900,), (0.2,), 0.02, 3, mg.BF16),
])
def test_graph_equals_oracle(ctx, n, d, nint, ov, eps, min_pts, prec):
    X = np.random.default_rng(n + len(nint)).uniform(-1, 1, (n, d)).astype(np.float32)
    m = len(nint)
    prm = mg.params((mg.LENS_COORD,) * m, tuple(range(m)), nint, ov, eps, min_pts, prec)
    g = mg.mapper_graph(ctx, _device(X), prm)
    got = g.numpy()
    lens, _ = g.lens(n, m)
    ref = oracle.mapper_graph(X, lens, nint, ov, eps, min_pts)
    for k in ("node_offsets", "node_members", "node_elem", "edges"):
        assert np.array_equal(np.asarray(got[k]), np.asarray(ref[k])), k


@pytest.mark.parametrize("n,d", [(400, 3), (700, 9)])
def test_forest_of_tied_distances(ctx, n, d):
    # every point has all others of its value at distance 0 and its lattice
    # neighbours at 1: far more tied pairs than 8 a row
    X = np.random.default_rng(n).integers(0, 2, (n, d)).astype(np.float32)
    Xd = _device(X)
    lens, _ = mg.mapper_lens(ctx, Xd, (mg.LENS_COORD,), (0,))
    cover = mg.mapper_cover(ctx, lens, (1,), (0.0,))
    got = mg.mapper_single_linkage(ctx, Xd, cover, 1.5).numpy()
    offs, pts = cover.numpy()
    u, v, d2 = oracle.msf(X, pts[offs[0]:offs[1]], 1.5)
    want = sorted(zip(d2.tolist(), u.tolist(), v.tolist()))
    assert sorted(zip(got["d2"].tolist(), got["u"].tolist(), got["v"].tolist())) == want


# scale 2^e: squares that underflow, ordinary ones, squares past FP32; the sum
# of n positive terms of d squares, each rounded a few times in FP64
@pytest.mark.parametrize("e", [-90, 0, 80])
@pytest.mark.parametrize("n,d,pad", [(1, 1, 0), (33, 7, 0), (1001, 32, 3), (515, 64, 0), (2050, 129, 1)])
def test_eccentricity_over_the_range_of_values(ctx, n, d, pad, e):
    rng = np.random.default_rng(n + d)
    A = (rng.standard_normal((n, d + pad)) + rng.uniform(-3, 3, d + pad)).astype(np.float32) * np.float32(2.0 ** e)
    Ad = _device(A)
    f, _ = mg.mapper_lens(ctx, Ad[:, :d], (mg.LENS_ECC,), (0,))
    X = A[:, :d].astype(np.longdouble)
    mu = X.mean(0)
    dev = ((X - mu) ** 2).sum(1)
    want = np.sqrt(dev + dev.mean()).astype(np.float64)
    assert np.allclose(f.cpu().numpy()[:, 0], want, rtol=1e-12, atol=0.0)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("d", [7, 64])
def test_eccentricity_rejects_non_finite_values(ctx, bad, d):
    X = np.random.default_rng(d).standard_normal((500, d)).astype(np.float32)
    X[331, d // 2] = bad
    with pytest.raises(mg.MapperError):
        mg.mapper_lens(ctx, _device(X), (mg.LENS_ECC,), (0,))
