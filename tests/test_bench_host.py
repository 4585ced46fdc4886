"""Host logic of bench.py that needs no device."""
import bench


def test_captured_traffic_is_reported_for_the_kernels_it_was_taken_of(tmp_path, monkeypatch):
    """DRAM bytes from a capture belong to the kernels that were captured: comments and layout may change, code may not."""
    csrc, profiles = tmp_path / "paper_2607_19893_b200" / "csrc", tmp_path / "profiles"
    csrc.mkdir(parents=True)
    profiles.mkdir()
    (csrc / "a.cu").write_text("int f() { return 1; }  // one\n")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.dram_traffic_from_profiles("w") is None  # not captured
    capture = profiles / "dram_traffic_view_step_w.txt"
    capture.write_text(f"# a capture\n# sources {bench.kernel_sources_digest()} of it\n# stage bytes\nadam 12\nproject 30\n")
    assert bench.dram_traffic_from_profiles("w") == {"adam": 12.0, "project": 30.0}
    (csrc / "a.cu").write_text("// another word on it\nint f() {\n  return 1;\n}\n")
    assert bench.dram_traffic_from_profiles("w") == {"adam": 12.0, "project": 30.0}
    (csrc / "a.cu").write_text("int f() { return 2; }\n")
    assert bench.dram_traffic_from_profiles("w") is None
    capture.write_text("# a capture of unknown sources\nadam 12\n")
    assert bench.dram_traffic_from_profiles("w") is None
