"""What bench.py reports beside its times: the sources that a profiled figure belongs to."""
import os
import shutil

import pytest

import bench

CSRC = os.path.join("paper_1406_6438_gb300", "csrc")


@pytest.mark.parametrize("kind,header", [(8, "vans_pair.cuh"), (8, "vans_tma.cuh"), (9, "vans_pair.cuh"),
                                         (9, "vans_device.cuh"), (9, "vans_internal.h"), (7, "vans_pipeline.cuh"),
                                         (7, "vans_tma.cuh"), (0, "vans_device.cuh")])
def test_hash_covers_every_header_of_the_kernel(tmp_path, monkeypatch, kind, header):
    """A change of a header that the kernel's arithmetic or layout is in makes a figure
    profiled before it stale."""
    shutil.copytree(os.path.join(bench.ROOT, CSRC), tmp_path / CSRC)
    shutil.copytree(os.path.join(bench.ROOT, "include"), tmp_path / "include")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    before = bench.kernel_hash(kind)
    with open(tmp_path / CSRC / header, "a") as f:
        f.write("\n// another\n")
    assert bench.kernel_hash(kind) != before
