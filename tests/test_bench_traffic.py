"""The bench line's recorded DRAM traffic belongs to the source it was captured on:
a figure counts as current only while the files of that precision's kernel are the
ones named in the summary."""
import hashlib
import os
import shutil

import pytest

import bench

FP16 = ("team.cu", "team_map.h", "dense_sched.h", "ptx.cuh")
FP32 = ("dense.cu", "dense_sched.h", "ptx.cuh")


@pytest.fixture
def tree(tmp_path, monkeypatch):
    src = os.path.join(bench.ROOT, "paper_1502_07266_gb300", "csrc")
    dst = tmp_path / "paper_1502_07266_gb300" / "csrc"
    dst.mkdir(parents=True)
    (tmp_path / "profiles").mkdir()
    for f in set(FP16 + FP32):
        shutil.copy(os.path.join(src, f), dst / f)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    return tmp_path


def record(tree, precision, files):
    csrc = tree / "paper_1502_07266_gb300" / "csrc"
    lines = ["precision: " + precision, "schedule: two_front", "b_aux: 2", "dram bytes per full-size launch: 1e9"]
    lines += ["%s sha1: %s" % (f, hashlib.sha1((csrc / f).read_bytes()).hexdigest()) for f in files]
    (tree / "profiles" / "dense_traffic.txt").write_text("\n".join(lines) + "\n")


@pytest.mark.parametrize("precision,files,others", [
    ("split_fp16", FP16, ("dense.cu",)), ("fp16", FP16, ("dense.cu",)), ("fp32", FP32, ("team.cu", "team_map.h"))])
def test_figure_follows_its_kernel(tree, precision, files, others):
    csrc = tree / "paper_1502_07266_gb300" / "csrc"
    for f in others:                                  # another precision's kernel changes: still current
        record(tree, precision, files)
        with open(csrc / f, "a") as h:
            h.write("// changed\n")
        assert bench._dense_traffic(127, precision, "two_front", 2) == 1e9
    for f in files:                                   # its own does: no figure
        record(tree, precision, files)
        assert bench._dense_traffic(127, precision, "two_front", 2) == 1e9
        with open(csrc / f, "a") as h:
            h.write("// changed\n")
        assert bench._dense_traffic(127, precision, "two_front", 2) is None
    record(tree, precision, files)
    assert bench._dense_traffic(127, "fp32" if precision != "fp32" else "fp16", "two_front", 2) is None
