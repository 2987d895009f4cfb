"""The hash that ties a stored traffic figure to the kernels it was captured on
covers the order of launches of both paths."""
import os
import shutil

import pytest

import bench

API = os.path.join("paper_2412_11809_gb300", "csrc", "tpc_api.cu")


@pytest.mark.parametrize("line", [
    "    launch_features(w, L);\n    launch_outputs(w, L);\n",      # the time-sorted path
    "    launch_gather(w, L);\n",                                    # the general sort
    "    launch_arrival_output(w, L);\n"])                           # the arrival-order path
def test_hash_covers_the_launch_order(line, tmp_path, monkeypatch):
    root = str(tmp_path)
    shutil.copytree(os.path.join(bench.ROOT, "paper_2412_11809_gb300", "csrc"),
                    os.path.join(root, "paper_2412_11809_gb300", "csrc"))
    want = bench.kernel_source_sha()
    monkeypatch.setattr(bench, "ROOT", root)
    assert bench.kernel_source_sha() == want
    path = os.path.join(root, API)
    text = open(path).read()
    assert line in text
    open(path, "w").write(text.replace(line, "", 1))
    assert bench.kernel_source_sha() != want
