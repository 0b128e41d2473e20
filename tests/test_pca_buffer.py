"""The buffer that mapper_lens hands over for the PCA basis holds what the call
writes: the mean and every axis up to the highest one asked for."""
import ctypes
import types

import numpy as np
import pytest

pytest.importorskip("torch")
mg = pytest.importorskip("paper_2011_03209_gb300")


@pytest.mark.parametrize("axes", [(0,), (1,), (0, 1), (3, 2)])
def test_pca_buffer_holds_mean_and_axes(monkeypatch, axes):
    n, d = 10, 6
    sizes, given = {}, []
    real_empty = np.empty

    def empty(shape, dtype=np.float64):
        a = real_empty(shape, dtype)
        sizes[a.ctypes.data] = a.size
        return a

    def lens_ex(*a):
        given.append(a[-1])
        return 0

    out = types.SimpleNamespace(data_ptr=lambda: 0)
    monkeypatch.setattr(mg, "_torch", lambda: types.SimpleNamespace(empty=lambda *a, **k: out, float64=None))
    monkeypatch.setattr(mg, "_x_args", lambda X: (ctypes.c_void_p(0), n, d, d, None))
    monkeypatch.setattr(np, "empty", empty)
    ctx = types.SimpleNamespace(device=0, h=None, _lib=types.SimpleNamespace(mapper_lens_ex=lens_ex))
    mg.mapper_lens(ctx, None, (mg.LENS_PCA,) * len(axes), axes)
    if given[0] is not None:
        assert sizes[given[0].value] >= d * (2 + max(axes))
