"""Principal axes up to high ranks: the power iteration's shared memory holds one
row of the columns per axis, and every number of axes launches."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
mg = pytest.importorskip("paper_2011_03209_gb300")

pytestmark = pytest.mark.gpu


# 8 bytes x 128 (256) columns x axes around 48 KB, beside the kernel's other 3 to
# 6 KB; the lower counts first, since a raised limit stays
@pytest.mark.parametrize("d,axes", [(100, (43, 44, 45, 46, 47, 48)), (128, (47,)), (200, (19, 20, 21, 22, 23, 24)),
                                    (256, (23,)), (60, (59,)), (30, (29,))])
def test_high_axes_launch(d, axes):
    n = 700
    rng = np.random.default_rng(d)
    X = (rng.standard_normal((n, d)) * np.linspace(3.0, 1.0, d)).astype(np.float32)
    Xd = torch.from_numpy(X).to("cuda:0")
    torch.cuda.synchronize()
    for k in axes:
        with mg.Context(0) as ctx:
            g = mg.mapper_graph(ctx, Xd, mg.params((mg.LENS_PCA,), (k,), (2,), (0.1,), 1.0, 2, mg.FP32))
            f, pca = g.lens(n, 1)
        mu, ax = pca[:d], pca[d:].reshape(-1, d)
        assert ax.shape[0] == k + 1
        # unit axes, each orthogonal to the earlier ones (1e-6, the iteration's tolerance)
        assert np.allclose(ax @ ax.T, np.eye(k + 1), atol=1e-6)
        acc = np.zeros(n)
        for c in range(d):                                  # one rounding per operation, columns in order
            acc = acc + (X[:, c].astype(np.float64) - mu[c]) * ax[k, c]
        assert np.array_equal(f[:, 0], acc)
