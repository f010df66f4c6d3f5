"""DRAM bytes in bench.py's roofline entries: those of the captured workload only."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_traffic_is_that_of_the_captured_workload(tmp_path, monkeypatch):
    sys.path.insert(0, ROOT)
    import hashlib

    import bench
    src = os.path.join(ROOT, "paper_1710_06316_gb300", "csrc", "fmm.cu")
    digest = hashlib.sha1(open(src, "rb").read()).hexdigest()[:12]
    (tmp_path / "profiles").mkdir()
    (tmp_path / "profiles" / "ncu_traffic.txt").write_text(
        "# stage bytes digest files workload\np2p 1000 %s fmm.cu 162/500/6/1\nm2l 7 0000 fmm.cu 162/500/6/1\n" % digest)
    os.symlink(os.path.join(ROOT, "paper_1710_06316_gb300"), tmp_path / "paper_1710_06316_gb300")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.ncu_traffic("p2p", "162/500/6/1") == 1000.0
    for other in ("10455600/500/6/1", "162/500/6/0", "162/500/8/1"):
        assert bench.ncu_traffic("p2p", other) is None           # another mesh, precision or order
    assert bench.ncu_traffic("m2l", "162/500/6/1") is None        # sources changed since the capture
