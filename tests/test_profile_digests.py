"""The ncu figures that the bench line reports from profiles/ belong to the
kernels in the tree: a change of their code has to come with a new record, and
a change of comments does not void one."""
import glob
import os

import pytest

import bench

PROFILES = sorted(glob.glob(os.path.join(bench.ROOT, "profiles", "*.md")))


def record(path):
    rec = {}
    for line in open(path):
        for key in ("sources_sha256:", "sources:"):
            if line.strip().strip("`").startswith(key):
                rec[key] = line.strip().strip("`")[len(key):].strip()
    return rec


RECORDED = [p for p in PROFILES if "sources_sha256:" in record(p)]


@pytest.mark.parametrize("path", RECORDED, ids=[os.path.basename(p) for p in RECORDED])
def test_recorded_figures_match_the_sources(path):
    rec = record(path)
    assert rec["sources_sha256:"] == bench.kernel_sources_digest(rec.get("sources:", ""))


def test_bench_line_has_its_recorded_figures():
    assert bench.recorded_traffic("traffic_peakmap_n4.md") is not None
    assert bench.recorded_traffic("traffic_correlate_n4.md") is not None
    assert bench.recorded_value("k_peakmap_n4_64x512x512.md", "warp_inst_per_voxel") is not None


def test_digest_counts_code_only():
    src = 'int a = 1;  // one\nconst char* s = "// kept  /* kept */";\nchar q = \'"\'; /* two\n lines */ int b;\n'
    same = "// other words\nint a =\n\n  1;\nconst char* s = \"// kept  /* kept */\"; char q = '\"';\nint b;"
    assert bench.code_text(src) == bench.code_text(same)
    for code in (src.replace("= 1", "= 2"), src.replace("kept  /*", "kept /*"), src.replace("int b", "int c")):
        assert bench.code_text(code) != bench.code_text(src)
