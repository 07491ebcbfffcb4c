"""bench.py's lists of the sources a kernel kind is made of: a name that leads to no file is an error of the list and
must not drop out of the hash that keys the committed traffic figures."""
import os

import bench

CSRC = os.path.join(bench.ROOT, "paper_2306_17263_gb300", "csrc")


def test_a_missing_source_changes_the_hash(monkeypatch):
    monkeypatch.setattr(bench, "KIND_SOURCES", {"curl32": ["k_tiled.cu"]})
    h = bench.kernel_sources_hash("curl32")
    monkeypatch.setattr(bench, "KIND_SOURCES", {"curl32": ["k_tiled.cu", "no_such_file.cuh"]})
    assert bench.kernel_sources_hash("curl32") != h


def test_the_lists_name_files_with_their_headers():
    for kind, files in bench.KIND_SOURCES.items():
        for f in files:
            assert os.path.exists(os.path.join(CSRC, f)), (kind, f)
    for kind in ("curl32", "solve32"):  # the launcher and the polynomial the walks take their coefficients from
        assert {"k_pdl.cuh", "k_rec64.cu", "k_rec64.cuh", "k_walk_dev.cuh"} <= set(bench.KIND_SOURCES[kind])
