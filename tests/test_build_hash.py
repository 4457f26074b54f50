"""The build's hash of the sources, part of the tuner cache's key: any source counts, nothing else does."""
import importlib
import shutil

build = importlib.import_module("paper_1606_00247_gb300.build")


def test_source_hash_follows_the_sources(tmp_path):
    csrc = tmp_path / "csrc"
    shutil.copytree(build.CSRC, csrc)
    h = build.source_hash(str(csrc))
    assert h == build.source_hash() and 0 <= h < 2**64
    (csrc / "notes.txt").write_text("no source")
    assert build.source_hash(str(csrc)) == h
    for f in ("m2l_tc.cu", "common.cuh"):
        with open(csrc / f, "a") as s:
            s.write("\n")
        assert build.source_hash(str(csrc)) != h
        h = build.source_hash(str(csrc))
