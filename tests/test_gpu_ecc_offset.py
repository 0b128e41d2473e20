"""The eccentricity of clouds away from the origin and of few columns: the mean
keeps its 53 bits.

The values lie on a grid on which every column sum is exact in FP64, so the mean
is the one rounding of sum / n on any machine, and the reference takes that mean.
What is left are FP64 roundings (u = 2^-53): one of x - mu and one FMA a column
(q within d + 2 of them, relative), the mean of q over the rows (at most 30 adds
in a chain, a division), their sum and the square root."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
mg = pytest.importorskip("paper_2011_03209_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mean,grid", [(0.0, 2.0 ** -20), (1e3, 2.0 ** -14), (1e4, 2.0 ** -10), (1e6, 2.0 ** -4)])
@pytest.mark.parametrize("d", [1, 4, 33, 64, 256])
def test_eccentricity_keeps_the_mean(d, mean, grid):
    n = 3000
    rng = np.random.default_rng(d)
    X = (np.round((mean + rng.standard_normal((n, d))) / grid) * grid).astype(np.float32)
    mu = X.astype(np.float64).sum(0) / n
    Xd = torch.from_numpy(X).to("cuda:0")
    torch.cuda.synchronize()
    with mg.Context(0) as ctx:
        f, _ = mg.mapper_lens(ctx, Xd, (mg.LENS_ECC,), (0,))
        torch.cuda.synchronize()
        got = f.cpu().numpy()[:, 0]
    q = ((X.astype(np.longdouble) - mu) ** 2).sum(1)
    want = np.sqrt(q + q.mean())
    u = 2.0 ** -53
    tol = ((d + 2) + 30 + 2) / 2 * u + u
    err = np.abs((got - want) / want).max()
    assert err <= tol, (float(err), tol)
