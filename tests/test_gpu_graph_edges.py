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


def _graph(ctx, Xd, nint, ov, eps, min_pts, prec):
    g = mg.mapper_graph(ctx, Xd, mg.params((mg.LENS_COORD,), (0,), (nint,), (ov,), eps, min_pts, prec))
    return g.numpy(), g.stats()


# counts stop at minPts once they are known to reach it; lists hold up to 64
@pytest.mark.parametrize("min_pts", [1, 2, 64, 65, 66, 300])
@pytest.mark.parametrize("tile_n", [128, 256])
def test_core_flags_at_the_limits_of_the_counts(min_pts, tile_n):
    rng = np.random.default_rng(min_pts)
    c = rng.standard_normal((5, 24)) * 4
    X = (c[rng.integers(0, 5, 3000)] + rng.standard_normal((3000, 24)) * rng.choice([0.3, 1.0], (3000, 1))).astype(np.float32)
    with mg.Context(0) as ctx:
        ctx.set_pass1_tile_n(tile_n)
        g = mg.mapper_graph(ctx, _device(X), mg.params((mg.LENS_COORD,), (0,), (3,), (0.3,), 3.5, min_pts, mg.BF16))
        got, core = g.numpy(), g.clusters().numpy(len(g.cover().numpy()[1]))[1]
        lens, _ = g.lens(len(X), 1)
    ref = oracle.mapper_graph(X, lens, (3,), (0.3,), 3.5, min_pts)
    assert np.array_equal(core, ref["core"])
    for k in ("node_offsets", "node_members", "node_elem", "edges"):
        assert np.array_equal(np.asarray(got[k]), np.asarray(ref[k])), k


# every squared distance is an integer and eps^2 is one of them: whole blocks
# of band pairs, and near ties that have to be counted
def test_blocks_of_band_pairs(ctx):
    X = np.random.default_rng(3).integers(0, 2, (2000, 16)).astype(np.float32)
    got, st = _graph(ctx, _device(X), 2, 0.3, 2.0, 40, mg.BF16)
    lens = X[:, :1].astype(np.float64)
    ref = oracle.mapper_graph(X, lens, (2,), (0.3,), 2.0, 40)
    assert st["near_ties"] == ref["near_ties"] > 0
    for k in ("node_offsets", "node_members", "node_elem", "edges"):
        assert np.array_equal(np.asarray(got[k]), np.asarray(ref[k])), k


# columns in K blocks of 64: A's tile kept whole (1 to 3 blocks) or streamed
@pytest.mark.parametrize("d", [40, 64, 100, 192, 250, 257, 400])
@pytest.mark.parametrize("n", [1500, 14_000])
def test_three_products_at_every_depth(d, n):
    rng = np.random.default_rng(d)
    c = rng.standard_normal((12, d)) * 0.6
    X = (c[rng.integers(0, 12, n)] + rng.standard_normal((n, d))).astype(np.float32)
    eps = float(np.sqrt(2.0 * d) * 0.98)
    with mg.Context(0) as ctx:
        Xd = _device(X)
        ref, rs = _graph(ctx, Xd, 2, 0.2, eps, 10, mg.FP32)
        for tile_n in (128, 256):
            ctx.set_pass1_tile_n(tile_n)
            ctx.set_pass1_screen(2)
            got, st = _graph(ctx, Xd, 2, 0.2, eps, 10, mg.BF16)
            assert st["n_core"] == rs["n_core"]
            for k in ref:
                assert np.array_equal(np.asarray(got[k]), np.asarray(ref[k])), (tile_n, k)


# more than 8192 all-in tile pairs, in tiles that are one component and tiles
# that are not
@pytest.mark.parametrize("prec", [mg.FP32, mg.BF16])
def test_many_all_in_pairs(ctx, prec):
    rng = np.random.default_rng(11)
    X = np.concatenate([rng.normal(0, 0.01, (22_000, 4)), rng.normal(0, 0.01, (900, 4)) + 3.0,
                        rng.uniform(-4, 6, (400, 4))]).astype(np.float32)
    X = X[rng.permutation(len(X))]
    prm = mg.params((mg.LENS_COORD,), (0,), (1,), (0.0,), 1.0, 5, prec)
    g = mg.mapper_graph(ctx, _device(X), prm)
    assert g.stats()["tile_pairs_in"] >= 8192
    got = g.numpy()
    ref = oracle.mapper_graph(X, X[:, :1].astype(np.float64), (1,), (0.0,), 1.0, 5)
    for k in ("node_offsets", "node_members", "node_elem", "edges"):
        assert np.array_equal(np.asarray(got[k]), np.asarray(ref[k])), k
