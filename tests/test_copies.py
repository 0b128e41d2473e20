"""Copying a result's arrays to the caller: every queued copy is waited for,
also when a later one (or the wait) fails. The copies are stand-ins."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "copies.h"
#include <cstdio>
#include <cstdlib>
using mgb::CopyOut;
// argv: the item whose copy fails (-1: none), the wait's status
int main(int argc, char** argv)
{
    const int bad = atoi(argv[1]), wait_status = atoi(argv[2]);
    char a[8], b[8], c[8];
    int queued = 0, waits = 0, queued_at_wait = -1;
    auto queue = [&](const CopyOut&) { return queued++ == bad ? -3 : 0; };
    auto wait = [&]() { ++waits; queued_at_wait = queued; return wait_status; };
    int rc = mgb::copy_all({{a, b, 8}, {nullptr, b, 8}, {b, c, 8}, {c, a, 0}, {c, a, 4}}, queue, wait);
    printf("%d %d %d %d\n", rc, queued, waits, queued_at_wait);
    rc = mgb::copy_all({{nullptr, b, 8}, {c, a, 0}}, queue, wait);
    printf("%d %d\n", rc, waits);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("copies")
    (d / "t.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_2011_03209_gb300", "csrc"),
                    str(d / "t.cpp"), "-o", str(d / "t")], check=True)
    return str(d / "t")


# (item that fails, wait's status) -> status, copies queued, waits, queued before the wait
@pytest.mark.parametrize("bad,wait,want", [(-1, 0, (0, 3, 1, 3)), (0, 0, (-3, 1, 1, 1)), (1, 0, (-3, 2, 1, 2)),
                                           (2, 0, (-3, 3, 1, 3)), (-1, -4, (-4, 3, 1, 3)), (2, -4, (-3, 3, 1, 3))])
def test_queued_copies_are_waited_for(program, bad, wait, want):
    out = subprocess.run([program, str(bad), str(wait)], capture_output=True, text=True, check=True).stdout.split("\n")
    assert tuple(map(int, out[0].split())) == want
    assert out[1] == "0 1"                                  # nothing asked for: no wait


def test_results_are_copied_through_it():
    src = open(os.path.join(ROOT, "paper_2011_03209_gb300", "csrc", "capi.cu")).read()
    for name in ("mapper_cover_copy", "mapper_clusters_copy", "mapper_forest_copy", "mapper_graph_copy", "mapper_graph_lens"):
        body = src[src.index(f"int {name}("):]
        body = body[:body.index("\n}\n")]
        assert "return copies_out(" in body and "cudaMemcpyAsync" not in body, name
