"""The stamped counters of the bench line are void when any file that their
kernels are compiled from has changed (no GPU)."""
import os
import re
import shutil

import pytest

import bench

CSRC = os.path.join(bench.ROOT, "paper_2403_16862_gb300", "csrc")


def _includes(path, seen):
    for name in re.findall(r'^\s*#include\s+"([^"]+)"', open(path).read(), flags=re.M):
        f = os.path.normpath(os.path.join(os.path.dirname(path), name))
        if f not in seen:
            seen.add(f)
            _includes(f, seen)
    return seen


@pytest.mark.parametrize("kernel,unit", [("k_point_grad_hash", "raster_bwd.cu"), ("k_hash_fwd", "hashgrid.cu"),
                                         ("step", "sample.cu"), ("step", "hashgrid.cu"), ("step", "raster_fwd.cu"),
                                         ("step", "raster_fwd_wide.cu"), ("step", "raster_bwd.cu")])
def test_stamp_covers_what_the_kernel_is_compiled_from(tmp_path, monkeypatch, kernel, unit):
    shutil.copytree(CSRC, tmp_path / "paper_2403_16862_gb300" / "csrc")
    shutil.copytree(os.path.join(bench.ROOT, "include"), tmp_path / "include")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    top = str(tmp_path / "paper_2403_16862_gb300" / "csrc" / unit)
    files = _includes(top, {top})
    assert len(files) > 2
    before = bench.source_stamp(kernel)
    for f in files:
        text = open(f).read()
        open(f, "w").write(text + "\n// changed\n")
        assert bench.source_stamp(kernel) != before, f
        open(f, "w").write(text)
    assert bench.source_stamp(kernel) == before
