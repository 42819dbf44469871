"""The recorded DRAM traffic of a kernel stays valid while host code changes, and
not when device code does."""
import os
import shutil

import bench


def test_source_hash(tmp_path, monkeypatch):
    sub = os.path.join("paper_2202_01631_gb300", "csrc")
    shutil.copytree(os.path.join(bench.ROOT, sub), tmp_path / sub)
    want = bench.source_hash()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.source_hash() == want
    for name in sorted(os.listdir(tmp_path / sub)):
        device = name.endswith(".cuh") or name.startswith("lbdp_prec_")
        text = (tmp_path / sub / name).read_text()
        (tmp_path / sub / name).write_text(text + "// more\n")
        assert (bench.source_hash() != want) == device, name
        (tmp_path / sub / name).write_text(text)
