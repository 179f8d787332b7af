"""A committed traffic figure counts only for the sources it was captured from."""
import os

import pytest

import bench


@pytest.mark.parametrize("key", sorted(bench.PROFILES))
def test_profile_covers_every_source_of_the_captured_launch(key):
    name, files = bench.PROFILES[key]
    assert os.path.exists(os.path.join(bench.ROOT, "profiles", name))
    assert all(os.path.exists(os.path.join(bench.CSRC, f)) for f in files)
    assert {"tma_common.cuh", "static_step.cu"} <= set(files)  # helpers; tile plan and grid
    if key.startswith(("c2", "c3")):
        storage = {"fp32": "f32", "fp16": "f16", "bf16": "bf16"}[key.split("_")[1]]
        plan = "d5" if key.startswith("c2") else "d11"
        assert {"kernels_static.cuh", "static_unit.cuh", "static_%s_%s.cu" % (storage, plan)} <= set(files)


def test_a_changed_source_takes_the_figure_away(tmp_path, monkeypatch):
    for f in os.listdir(bench.CSRC):
        (tmp_path / f).write_bytes(open(os.path.join(bench.CSRC, f), "rb").read())
    monkeypatch.setattr(bench, "CSRC", str(tmp_path))
    for key, (_, files) in bench.PROFILES.items():
        before = bench.kernel_source_hash(files)
        for f in files:
            p = tmp_path / f
            p.write_bytes(p.read_bytes() + b"\n")
            assert bench.kernel_source_hash(files) != before
            before = bench.kernel_source_hash(files)
