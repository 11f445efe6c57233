"""The bench line's recorded DRAM traffic counts only for the sources it was
taken with: a change to any file that the fused kernel is compiled from drops
it."""
import os
import shutil

import pytest

import bench
from paper_2606_00724_gb300 import synth

W = synth.WORKLOADS["c3"]


def _tree(tmp_path):
    csrc = tmp_path / "paper_2606_00724_gb300" / "csrc"
    shutil.copytree(os.path.join(bench.ROOT, "paper_2606_00724_gb300", "csrc"), csrc)
    (tmp_path / "profiles").mkdir()
    return csrc


def test_record_of_the_current_sources_counts(tmp_path):
    csrc = _tree(tmp_path)
    rec = tmp_path / "profiles" / "wf_fused_kernel_traffic.md"
    rec.write_text(f"| {W.name} | 1 MB | 2 MB | 3145728 | 3000000 | {bench.fused_source_hash(str(csrc))} |\n")
    assert bench.recorded_traffic(W, str(tmp_path)) == 3145728


@pytest.mark.parametrize("name", bench.FUSED_SOURCES)
def test_changed_source_drops_the_record(tmp_path, name):
    csrc = _tree(tmp_path)
    rec = tmp_path / "profiles" / "wf_fused_kernel_traffic.md"
    rec.write_text(f"| {W.name} | 1 MB | 2 MB | 3145728 | 3000000 | {bench.fused_source_hash(str(csrc))} |\n")
    with open(csrc / name, "a") as f:
        f.write("\n// changed\n")
    assert bench.recorded_traffic(W, str(tmp_path)) is None


def test_every_header_of_the_fused_kernel_is_covered():
    csrc = os.path.join(bench.ROOT, "paper_2606_00724_gb300", "csrc")
    seen, todo = set(), ["wf_fused.cu"]
    while todo:
        f = todo.pop()
        seen.add(f)
        for ln in open(os.path.join(csrc, f)):
            if ln.startswith('#include "'):
                h = ln.split('"')[1]
                if h not in seen and os.path.exists(os.path.join(csrc, h)):
                    todo.append(h)
    assert seen == set(bench.FUSED_SOURCES)
