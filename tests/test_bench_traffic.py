"""The benchmark quotes a committed DRAM count of the sweep only while the
sources that hold the sweep are the ones it was captured from."""
import os

import pytest

import bench
from paper_1507_05141_gb300 import inputs

SOURCES = ("shd_sweep.cu", "shd_internal.cuh")


def _tree(tmp_path):
    csrc = tmp_path / "paper_1507_05141_gb300" / "csrc"
    csrc.mkdir(parents=True)
    for f in SOURCES + ("shd_kernels.cu",):
        (csrc / f).write_text("// " + f)
    lines = ["# a capture", "- dram bytes per launch: 123"]
    lines += [f"- {f} sha256: `{bench._sha256(os.path.join(csrc, f))}`" for f in SOURCES + ("shd_kernels.cu",)]
    (tmp_path / "profiles").mkdir()
    (tmp_path / "profiles" / "sweep_jet64_mixed.md").write_text("\n".join(lines) + "\n")
    return csrc


@pytest.mark.parametrize("changed", [None, "shd_sweep.cu", "shd_internal.cuh", "shd_kernels.cu"])
def test_traffic_follows_the_sweep_sources(tmp_path, monkeypatch, changed):
    csrc = _tree(tmp_path)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    spec = inputs.jet(n=4, G=1, L=1)
    spec.grid = (64, 64, 64)
    if changed:
        (csrc / changed).write_text("// another kernel")
    want = None if changed in SOURCES else 123
    assert bench.sweep_traffic("mixed", spec) == want
    spec.grid = (32, 32, 32)
    assert bench.sweep_traffic("mixed", spec) is None
