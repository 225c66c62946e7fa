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


def test_roofline_is_that_of_the_bound():
    """Several steps per launch are bound by the FP32 pipe: their fraction is of its rate,
    in TFLOP/s; one step per launch by HBM, in GB/s.  One step of 4096^2 in 200 us,
    four in 400."""
    cells = 4096 * 4096
    r = bench.roofline(7, cells, 200e-6, 1, sms=152)
    assert r["bound"] == "hbm" and r["unit"] == "GB/s" and r["achieved"] == pytest.approx(76 * cells / 200e-6 / 1e9)
    assert r["frac"] == pytest.approx(r["achieved"] / bench.peaks()[0])
    r = bench.roofline(9, cells, 400e-6, 4, sms=152)
    assert r["bound"] == "fp32" and r["unit"] == "TFLOP/s"
    assert r["achieved"] == pytest.approx(bench.FLOPS_PER_CELL * cells / 100e-6 / 1e12)
    assert r["peak"] == pytest.approx(152 * 128 * 2 * 2.07e9 / 1e12, rel=0.02)
    assert r["frac"] == pytest.approx(r["achieved"] / r["peak"]) and 0 < r["frac"] < 1
    assert r["hbm"]["achieved"] == pytest.approx(76 * cells / 400e-6 / 1e9)


@pytest.mark.parametrize("kind,key", [(4, "load_balance"), (9, "single_step_load_balance"), (0, None)])
def test_load_balance_names_the_launch_it_is_of(kind, key):
    """The profile of a batch that runs several steps per launch is of its single-step
    launch, which the timed region does not run."""
    class Batch:
        def profile_step(self):
            return {"efficiency": 0.9}
    got = bench.load_balance(Batch(), kind)
    assert got == ({} if key is None else {key: {"efficiency": 0.9}})
