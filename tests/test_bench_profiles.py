"""bench.py reads DRAM bytes per unit of work from the committed profile
summaries, if they were taken of the present kernel source."""
import os

import pytest

import bench

PROFILES = [("fwd_bf16_connected_52x52.md", "psr_fwd_bf16.cu", "dram bytes per evaluated config-site"),
            ("fwd2d_tc_connected_52x52.md", "psr_fwd2d_tc.cu", "dram bytes per evaluated patch"),
            ("lru_tc_connected_tfim256.md", "psr_lru_tc.cu", "dram bytes per evaluated site"),
            ("scan_52x52_layer.md", "psr_scan.cu", "dram bytes per element")]


@pytest.mark.parametrize("profile,src,key", PROFILES)
def test_a_committed_profile_of_the_present_source_gives_a_number(profile, src, key):
    text = open(os.path.join(bench.ROOT, "profiles", profile)).read()
    present = bench.kernel_hash(src) in text
    assert (bench.profiled_traffic_per_unit(profile, src, key) is not None) == present


@pytest.mark.parametrize("note", ["", " (taken after a change", " of `kernel`"])
def test_notes_after_a_quoted_value_do_not_count(tmp_path, monkeypatch, note):
    (tmp_path / "profiles").mkdir()
    csrc = tmp_path / "paper_2605_13807_gb300" / "csrc"
    csrc.mkdir(parents=True)
    (csrc / "k.cu").write_text("// kernel\n")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    (tmp_path / "profiles" / "p.md").write_text(
        "- kernel source sha256/16: `%s`%s\n- dram bytes per item: `12.5`%s\n" % (bench.kernel_hash("k.cu"), note, note))
    assert bench.profiled_traffic_per_unit("p.md", "k.cu", "dram bytes per item") == 12.5
    (csrc / "k.cu").write_text("// another kernel\n")
    assert bench.profiled_traffic_per_unit("p.md", "k.cu", "dram bytes per item") is None
