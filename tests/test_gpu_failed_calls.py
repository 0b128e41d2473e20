"""A call that fails after it has queued a read-back leaves none on its way into
the context's page-locked scratch."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
mg = pytest.importorskip("paper_2011_03209_gb300")

pytestmark = pytest.mark.gpu


def test_failed_graph_leaves_no_copy_behind():
    # the radius is refused once the cover (12 M keys to sort) and the copy of its
    # offsets are queued; what is left to wait for afterwards are freed buffers
    n = 4_000_000
    X = torch.rand((n, 2), device="cuda:0", generator=torch.Generator("cuda:0").manual_seed(1))
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    left = []
    with mg.Context(0, stream=stream) as ctx:
        for _ in range(6):
            prm = mg.params((mg.LENS_COORD,), (0,), (500,), (0.66,), -1.0, 3, mg.FP32)
            with pytest.raises(mg.MapperError):
                mg.mapper_graph(ctx, X, prm)
            t = time.perf_counter()
            stream.synchronize()
            left.append((time.perf_counter() - t) * 1e6)
    assert min(left) < 100.0, left
