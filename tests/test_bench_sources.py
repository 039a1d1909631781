"""bench.py's kernel hashes cover every header that the kernel is made of."""
import os
import shutil

import pytest

CASES = [("single", 2), ("single", 3), ("fused", 2), ("fused", 3), ("resident", 2)]


@pytest.mark.parametrize("path,d", CASES)
def test_kernel_hash_follows_the_kernels_headers(monkeypatch, tmp_path, path, d):
    import bench

    names = [os.path.basename(p) for p in bench._sources(path, d)]
    own = {"single": [], "resident": ["mdf_res2d.cuh", "mdf_fuse2d.cuh"],
           "fused": ["mdf_fuse2d.cuh"] + ["mdf_fuse3d.cuh"] * (d == 3)}[path]
    shared = ["mdf_kernels.cuh", "mdf_lattice.cuh", "mdf_f32x2.cuh", "mdf_f64.cuh", "mdf_pack16.cuh", "mdf_eq.cuh",
              "mdf_aa.cuh", "mdf_vec16p.cuh"]
    assert names == sorted(own + shared)
    # a change of any of them is a change of the hash
    copy = tmp_path / "csrc"
    shutil.copytree(bench.CSRC, copy)
    monkeypatch.setattr(bench, "CSRC", str(copy))
    before = bench._kernel_sha(bench._sources(path, d))
    for name in names:
        text = (copy / name).read_text()
        (copy / name).write_text(text + "// changed\n")
        assert bench._kernel_sha(bench._sources(path, d)) != before
        (copy / name).write_text(text)
    assert bench._kernel_sha(bench._sources(path, d)) == before
