"""Covers and balanced covers at the edges of the radix sort's dispatch: one
CTA, a cluster of CTAs, tiles with two launches a digit, tiles with scanned
counts, one digit and several, all against the oracle (equal: integers)."""
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


# p = 0: one membership a point (two on a shared bound), so n is the number of
# keys: 1024 (one CTA) | 131072 (cluster of 8) | 4194304 (512 tiles) | more
@pytest.mark.parametrize("n,intervals,p", [
    (1, (3,), 0.0), (1023, (7,), 0.0), (1024, (256,), 0.0), (1025, (257,), 0.0), (8193, (20,), 0.3),
    (16385, (300,), 0.0), (131071, (50,), 0.0), (131072, (1,), 0.0), (131073, (50,), 0.0), (200_003, (1000,), 0.45),
    (70_001, (31, 37), 0.25), (4_194_000, (9,), 0.0), (4_300_001, (600,), 0.0)])
def test_cover_equals_oracle(ctx, n, intervals, p):
    rng = np.random.default_rng(n)
    f = rng.standard_normal((n, len(intervals)))
    f[: n // 7] = np.sort(f[: n // 7], axis=0)            # runs of equal digits beside random ones
    offs, pts = mg.mapper_cover(ctx, torch.from_numpy(f).to("cuda:0"), intervals, (p,) * len(intervals)).numpy()
    ro, rp = oracle.cover(f, intervals, (p,) * len(intervals))
    assert np.array_equal(offs, ro) and np.array_equal(pts, rp)


@pytest.mark.parametrize("n", [1, 33, 1025, 20_001, 131_073])
def test_balanced_cover_equals_oracle(ctx, n):
    rng = np.random.default_rng(n)
    f = np.round(rng.standard_normal((n, 1)) * 100.0) / 7.0 if n % 2 else rng.standard_normal((n, 1))
    offs, pts = mg.mapper_cover(ctx, torch.from_numpy(f).to("cuda:0"), (17,), (0.3,), balanced=True).numpy()
    ro, rp = oracle.cover(f, (17,), (0.3,), balanced=True)
    assert np.array_equal(offs, ro) and np.array_equal(pts, rp)
