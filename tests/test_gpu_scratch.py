"""Device memory that calls take from the stream-ordered pool, read from the
pool's own counters."""
import ctypes

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
mg = pytest.importorskip("paper_2011_03209_gb300")

pytestmark = pytest.mark.gpu

USED_CURRENT, USED_HIGH = 7, 8                              # CU_MEMPOOL_ATTR_USED_MEM_CURRENT, _HIGH


class Pool:
    """The device's default pool (torch's own tensors are not in it)."""

    def __init__(self):
        torch.cuda.init()
        self.cu = ctypes.CDLL("libcuda.so.1")
        dev, self.pool = ctypes.c_int(), ctypes.c_void_p()
        assert self.cu.cuDeviceGet(ctypes.byref(dev), 0) == 0
        assert self.cu.cuDeviceGetDefaultMemPool(ctypes.byref(self.pool), dev) == 0

    def get(self, attr):
        v = ctypes.c_uint64()
        assert self.cu.cuMemPoolGetAttribute(self.pool, attr, ctypes.byref(v)) == 0
        return v.value

    def peak_of(self, call):
        """The most that `call` holds beyond what is held before it."""
        torch.cuda.synchronize()
        before = self.get(USED_CURRENT)
        zero = ctypes.c_uint64(0)
        assert self.cu.cuMemPoolSetAttribute(self.pool, USED_HIGH, ctypes.byref(zero)) == 0
        out = call()
        torch.cuda.synchronize()
        return self.get(USED_HIGH) - before, out


def _device(X):
    Xd = torch.from_numpy(np.ascontiguousarray(X)).to("cuda:0")
    torch.cuda.synchronize()
    return Xd


def test_principal_axes_keep_no_second_cloud():
    n, d = 600_000, 256
    X = torch.randn((n, d), device="cuda:0", generator=torch.Generator("cuda:0").manual_seed(1))
    X[:, 3] *= 4.0
    pool = Pool()
    with mg.Context(0) as ctx:
        peak, (f, _) = pool.peak_of(lambda: mg.mapper_lens(ctx, X, (mg.LENS_PCA,), (0,)))
        got = f[:, 0].cpu().numpy()
    # 256 MiB of centred rows, 44 MB of partial tiles (the cloud: 614 MB)
    assert peak < 400e6, peak
    # the axis is column 3 but for the sample's correlations with it (4 / sqrt(n) in
    # all, over the eigenvalues' gap of 15: less than 0.03 of the projections' size)
    x3 = X[:, 3].double().cpu().numpy()
    assert np.abs(np.corrcoef(got, x3)[0, 1]) > 0.999


def _forest(budget, X, eps):
    with mg.Context(0, hbm_budget=budget) as ctx:
        Xd = _device(X)
        lens, _ = mg.mapper_lens(ctx, Xd, (mg.LENS_COORD,), (0,))
        cover = mg.mapper_cover(ctx, lens, (4,), (0.2,))
        peak, f = Pool().peak_of(lambda: mg.mapper_single_linkage(ctx, Xd, cover, eps))
        return peak, f.numpy()


# the budgets give the queue a quarter: 4 MB of the 6 to 7 MB that 8 entries a row
# would take, 64 KB, 15 entries, none
@pytest.mark.parametrize("budget", [16 << 20, 256 << 10, 999, 1])
def test_forest_queue_keeps_to_the_budget(budget):
    X = np.random.default_rng(2).standard_normal((40_000, 3)).astype(np.float32)
    free, want = _forest(0, X, 0.08)
    assert len(want["u"]) > 1000
    peak, got = _forest(budget, X, 0.08)
    for k in want:
        assert np.array_equal(got[k], want[k]), k
    queue = 128 * 40_000
    assert peak <= free - (queue - budget / 4) + 4096, (peak, free)


# about 20 nodes, whose edges the list has room for in little space, and about 300
@pytest.mark.parametrize("n,nint", [(500, 8), (3000, 150)])
def test_a_graph_keeps_its_edges_only(n, nint):
    X = np.random.default_rng(3).standard_normal((n, 3)).astype(np.float32)
    prm = mg.params((mg.LENS_COORD,), (0,), (nint,), (0.3,), 0.8, 3, mg.FP32)
    pool = Pool()
    with mg.Context(0) as ctx:
        Xd = _device(X)
        graphs = [mg.mapper_graph(ctx, Xd, prm)]
        torch.cuda.synchronize()
        before = pool.get(USED_CURRENT)
        graphs += [mg.mapper_graph(ctx, Xd, prm) for _ in range(32)]
        torch.cuda.synchronize()
        kept = (pool.get(USED_CURRENT) - before) / 32
        got = graphs[-1].numpy()
        lens, _ = graphs[-1].lens(n, 1)
        del graphs
    assert len(got["edges"]) > 0
    # 1.4 memberships a point of 50 bytes and 16 bytes a point, in some 20 arrays of
    # whole kilobytes; a list of up to 16 KB
    assert kept < 100 * n + (40 << 10), kept
    ref = oracle.mapper_graph(X, lens, (nint,), (0.3,), 0.8, 3)
    assert np.array_equal(got["edges"], ref["edges"])
