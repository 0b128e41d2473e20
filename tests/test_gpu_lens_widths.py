"""Lens kernels at the widths where their layout changes: the L2 norm's lanes
per row (d = 32, 64, 128, 256), the PCA's column blocks and power iteration
(d = 32 .. 256 on a cluster, more on one CTA), rows that do not fill a warp."""
import math

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


@pytest.mark.parametrize("d", [1, 7, 8, 9, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 600])
@pytest.mark.parametrize("n", [1, 7, 33, 1001])
def test_l2_lens_is_the_exact_norm(ctx, n, d):
    rng = np.random.default_rng(1000 * d + n)
    X = rng.standard_normal((n, d)).astype(np.float32) * np.exp2(rng.integers(-30, 30, (n, d))).astype(np.float32)
    X[rng.random((n, d)) < 0.1] = 0.0
    X[n // 2] *= np.float32(2.0 ** -100)                   # a row of small and subnormal values
    f, _ = mg.mapper_lens(ctx, _device(X), (mg.LENS_L2,), (0,))
    want = [math.sqrt(math.fsum(v * v for v in row)) for row in X.astype(np.float64)]
    assert np.array_equal(f.cpu().numpy()[:, 0], np.array(want))


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("d", [5, 40, 100, 200])
def test_l2_graph_rejects_non_finite_rows(ctx, d, bad):
    X = np.random.default_rng(d).standard_normal((300, d)).astype(np.float32)
    X[137, d - 1] = bad
    with pytest.raises(mg.MapperError):
        mg.mapper_graph(ctx, _device(X), mg.params((mg.LENS_L2,), (0,), (5,), (0.2,), 1.0, 3, mg.BF16))


# the projections are the defining expression in the basis found, bit for bit;
# the basis spans the top axes (1e-6, as the power iteration's tolerance)
@pytest.mark.parametrize("n,d", [(2, 1), (50, 2), (300, 31), (300, 32), (4096, 33), (4097, 64), (2047, 65), (2049, 128),
                                 (5000, 129), (3000, 256), (900, 257)])
def test_pca_widths(ctx, n, d):
    rng = np.random.default_rng(d)
    scale = np.linspace(1.0, 2.0, d) * np.where(np.arange(d) == d // 2, 6.0, 1.0)
    if d > 2:
        scale[0] = 20.0
    X = (rng.standard_normal((n, d)) * scale + rng.uniform(-5, 5, d)).astype(np.float32)
    X[: n // 3, 0] = np.float32(1.5)                       # constant runs
    K = 2 if d > 1 else 1
    prm = mg.params((mg.LENS_PCA,) * K, tuple(range(K)), (3,) * K, (0.1,) * K, 1e-3, 2, mg.FP32)
    g = mg.mapper_graph(ctx, _device(X), prm)
    f, pca = g.lens(n, K)
    mu, axes = pca[:d], pca[d:].reshape(-1, d)
    for k in range(K):
        acc = np.zeros(n)
        for c in range(d):                                  # one rounding per operation, columns in order
            acc = acc + (X[:, c].astype(np.float64) - mu[c]) * axes[k, c]
        assert np.array_equal(f[:, k], acc)
    assert np.allclose(mu, X.astype(np.float64).mean(0), rtol=1e-13, atol=1e-13)
    w, v = np.linalg.eigh(np.cov(X.T.astype(np.float64).reshape(d, n), bias=True).reshape(d, d))
    if n > d and d > 2 and w[-1] > 1.2 * w[-2] and w[-2] > 1.2 * w[-3]:
        for k in range(K):
            assert 1.0 - abs(axes[k] @ v[:, -1 - k]) <= 1e-6
