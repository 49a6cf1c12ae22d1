"""The benchmark reports the committed DRAM traffic of the sparse kernel only while
every source that decides it is the one the capture was taken from (host only)."""
import os
import shutil

import pytest

import bench


@pytest.mark.parametrize("changed", [None, *bench.SPARSE_SOURCES])
def test_traffic_follows_every_source(changed, tmp_path, monkeypatch):
    csrc = tmp_path / "paper_2609_27373_gb300" / "csrc"
    csrc.mkdir(parents=True)
    for name in bench.SPARSE_SOURCES:
        shutil.copy(os.path.join(bench.ROOT, "paper_2609_27373_gb300", "csrc", name), csrc / name)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    (tmp_path / "profiles").mkdir()
    (tmp_path / "profiles" / "attn_sparse_4k.md").write_text(
        f"# capture\n\ntraffic_bytes_per_launch: 123\nsource_sha256_16: {bench.sparse_sources_sha()}\n")
    if changed:
        with open(csrc / changed, "a") as f:
            f.write("// changed\n")
    assert bench.sparse_traffic_bytes() == (None if changed else 123)
