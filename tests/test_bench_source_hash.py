"""The hash that ties a recorded DRAM traffic to the kernels it was measured on
covers every source that holds a step kernel."""
import glob
import os
import shutil

import bench


def test_hash_covers_every_step_kernel(tmp_path, monkeypatch):
    src = os.path.join(bench.ROOT, "paper_2312_14789_gb300", "csrc")
    dst = tmp_path / "paper_2312_14789_gb300" / "csrc"
    shutil.copytree(src, dst)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    whole = bench.kernel_source_hash()
    steps = sorted(glob.glob(str(dst / "kernels*.cu"))) + sorted(glob.glob(str(dst / "*.cuh")))
    assert any(f.endswith("kernels_cluster.cu") for f in steps) and len(steps) >= 14
    for f in steps:
        text = open(f).read()
        open(f, "w").write(text + "// changed\n")
        assert bench.kernel_source_hash() != whole, f
        open(f, "w").write(text)
    assert bench.kernel_source_hash() == whole
