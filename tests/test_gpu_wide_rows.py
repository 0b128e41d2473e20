"""Graphs of rows wide enough that a kernel's shared memory, its own arrays
counted in, passes what a launch gets without asking (1408 to 1536 columns of
the tile-pair classification, 3053 to 3072 of the power iteration on one CTA)."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
mg = pytest.importorskip("paper_2011_03209_gb300")

pytestmark = pytest.mark.gpu


def _device(X):
    Xd = torch.from_numpy(X).to("cuda:0")
    torch.cuda.synchronize()
    return Xd


@pytest.mark.parametrize("d", [1376, 1377, 1408, 1500, 1536, 1537])
@pytest.mark.parametrize("prec", [mg.FP32, mg.BF16])
def test_wide_graph_equals_oracle(d, prec):
    n = 400
    rng = np.random.default_rng(d)
    c = rng.standard_normal((4, d))
    X = (c[rng.integers(0, 4, n)] + 0.1 * rng.standard_normal((n, d))).astype(np.float32)
    eps = 0.1 * float(np.sqrt(2.0 * d))
    with mg.Context(0) as ctx:
        g = mg.mapper_graph(ctx, _device(X), mg.params((mg.LENS_COORD,), (0,), (3,), (0.3,), eps, 3, prec))
        got = g.numpy()
        lens, _ = g.lens(n, 1)
    ref = oracle.mapper_graph(X, lens, (3,), (0.3,), eps, 3)
    for k in ("node_offsets", "node_members", "node_elem", "edges"):
        assert np.array_equal(np.asarray(got[k]), np.asarray(ref[k])), k


@pytest.mark.parametrize("d", [3040, 3060, 3072, 3080])
def test_wide_axes(d):
    rng = np.random.default_rng(d)
    X = rng.standard_normal((200, d)).astype(np.float32)
    X[:, 0] *= 30.0
    with mg.Context(0) as ctx:
        g = mg.mapper_graph(ctx, _device(X), mg.params((mg.LENS_PCA,), (0,), (2,), (0.1,), 1.0, 2, mg.FP32))
        _, pca = g.lens(200, 1)
    assert abs(pca[d]) > 0.9 and abs(np.linalg.norm(pca[d:]) - 1.0) < 1e-12
