"""The mean of the pivots is the same bit for bit whether the kernel or the host
forms it: its order of additions, and clouds from host and device memory."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "pivot_mean.h"
#include <cstdio>
#include <cstdlib>
#include <vector>
// argv: K dp; the pivots on stdin, the means on stdout
int main(int, char** argv)
{
    const int K = atoi(argv[1]), dp = atoi(argv[2]);
    std::vector<float> pv((size_t)K * dp), c(dp);
    if (fread(pv.data(), 4, pv.size(), stdin) != pv.size()) return 1;
    mgb::pivot_mean_host(pv.data(), K, dp, c.data());
    fwrite(c.data(), 4, c.size(), stdout);
    return 0;
}
"""


@pytest.mark.parametrize("K,dp", [(1, 32), (7, 32), (8, 64), (9, 32), (100, 96), (256, 160)])
def test_order_of_the_sum(tmp_path, K, dp):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    (tmp_path / "t.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-Wall", "-Werror", "-I",
                    os.path.join(ROOT, "paper_2011_03209_gb300", "csrc"), str(tmp_path / "t.cpp"), "-o",
                    str(tmp_path / "t")], check=True)
    Pv = (np.random.default_rng(K).standard_normal((K, dp)) + 100.0).astype(np.float32)
    out = subprocess.run([str(tmp_path / "t"), str(K), str(dp)], input=Pv.tobytes(), capture_output=True, check=True)
    got = np.frombuffer(out.stdout, dtype=np.float32)
    parts = []
    for w in range(8):
        s = np.zeros(dp, np.float32)
        for row in Pv[w::8]:
            s = s + row
        parts.append(s)
    want = parts[0]
    for s in parts[1:]:
        want = want + s
    assert np.array_equal(got, want / np.float32(K))


@pytest.mark.gpu
def test_host_and_device_clouds_get_one_layout():
    torch = pytest.importorskip("torch")
    mg = pytest.importorskip("paper_2011_03209_gb300")
    # whole numbers far from the origin: many points nearly as close to two pivots
    X = (np.random.default_rng(4).integers(0, 4, (60_000, 8)) + 1000.3).astype(np.float32)
    prm = mg.params((mg.LENS_L2,), (0,), (6,), (0.3,), 1.1, 5, mg.BF16)
    Xd = torch.from_numpy(X).to("cuda:0")
    torch.cuda.synchronize()
    with mg.Context(0) as ctx:
        got = [mg.mapper_graph(ctx, x, prm).stats() for x in (X, Xd)]
    for k in ("tile_pairs_in", "tile_pairs_out", "tile_pairs_tc", "tile_pairs_simt"):
        assert got[0][k] == got[1][k], k
