"""bench.py's record of captured DRAM traffic belongs to a kernel's whole source, the headers it
includes too, and its kernel names to the shapes that they ran."""
import os
import shutil

import bench


def test_a_changed_header_changes_the_key(tmp_path, monkeypatch):
    rel = "paper_1908_09359_gb300/csrc"
    shutil.copytree(os.path.join(bench.ROOT, rel), tmp_path / rel)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    for t in bench.NCU_TRAFFIC.values():
        before = bench.source_sha(t["source"])
        for header, matters in (("fused_pipe.cuh", True), ("tc_util.cuh", True), ("proposal.cuh", False)):
            p = tmp_path / rel / header
            text = p.read_text()
            p.write_text(text + "// changed\n")
            assert (bench.source_sha(t["source"]) != before) == matters, (t["source"], header)
            p.write_text(text)
        assert bench.source_sha(t["source"]) == before


def test_kernel_names_follow_the_shapes():
    assert bench.fused_kernel("fused4", True) == "env4_pipe_kernel"
    assert "env4_fused_kernel" in bench.fused_kernel("fused4", False)
    assert bench.fused_kernel("fused3", True) == "env3_fused_kernel"
    assert "proj3_tile_kernel" in bench.fused_kernel("fusedP", False)
