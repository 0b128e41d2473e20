"""A file of shapes timed on an earlier revision of the count pass (a header
without the revision, or with another) is not used, and is replaced."""
import pytest

from paper_2011_03209_gb300 import synth

torch = pytest.importorskip("torch")
mg = pytest.importorskip("paper_2011_03209_gb300")

pytestmark = pytest.mark.gpu


def _run(Xd, w):
    prm = mg.params(w.lens_kind, w.lens_arg, w.n_intervals, w.overlap, w.eps, w.min_pts, mg.BF16)
    with mg.Context(0) as c:
        mg.mapper_graph(c, Xd, prm)


def test_shapes_of_another_revision_are_not_used(tmp_path, monkeypatch):
    path = tmp_path / "tune.txt"
    monkeypatch.setenv("MAPPER_TUNE_CACHE", str(path))
    w = synth.mixture_100k()
    Xd = torch.from_numpy(w.X).to("cuda:0")
    torch.cuda.synchronize()
    _run(Xd, w)
    header, *rows = path.read_text().splitlines()
    keys = [r.split()[0] for r in rows]
    assert keys
    prop = torch.cuda.get_device_properties(0)
    old = f"mapper-tune-v1 {prop.name} sms={prop.multi_processor_count}"
    other = header.replace("count-pass-", "count-pass-9")
    for foreign in (old, other):
        assert foreign != header
        # a key of no call of this test: it would be merged into the file if the file were used
        path.write_text("\n".join([foreign, "12345 128"] + [f"{k} 128" for k in keys]) + "\n")
        _run(Xd, w)
        lines = path.read_text().splitlines()
        assert lines[0] == header and "12345 128" not in lines
    # its own header: kept
    path.write_text("\n".join([header, "12345 128"]) + "\n")
    _run(Xd, w)
    assert "12345 128" in path.read_text().splitlines()
