"""bench.py's DRAM counters belong to all of a kernel's device code: the file
and the headers that hold parts of it; an edit of any turns them into null.
And the names of the kernels that a call ran."""

import os
import shutil

import pytest

import bench

CSRC = os.path.join("paper_2608_03473_gb300", "csrc")


@pytest.mark.parametrize("profile", sorted(bench.PROFILED))
def test_an_edit_of_any_file_of_the_kernel(tmp_path, monkeypatch, profile):
    os.makedirs(tmp_path / "profiles")
    os.makedirs(tmp_path / CSRC)
    for f in bench.PROFILED[profile]:
        shutil.copy(os.path.join(bench.ROOT, CSRC, f), tmp_path / CSRC / f)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    (tmp_path / "profiles" / profile).write_text(f"<!-- traffic some_workload 123 {bench.kernel_hash(profile)} -->\n")
    assert bench.profiled_traffic("some_workload") == 123 and bench.profiled_traffic("another") is None
    for f in bench.PROFILED[profile]:
        text = (tmp_path / CSRC / f).read_text()
        (tmp_path / CSRC / f).write_text(text + "\n// edited\n")
        assert bench.profiled_traffic("some_workload") is None, f
        (tmp_path / CSRC / f).write_text(text)
    assert bench.profiled_traffic("some_workload") == 123


@pytest.mark.parametrize("profile", sorted(bench.PROFILED))
def test_every_header_with_device_code_counts(profile):
    # what the kernel's file includes of this folder, but for host-side declarations
    seen, todo = set(), [bench.PROFILED[profile][0]]
    while todo:
        f = todo.pop()
        if f in seen:
            continue
        seen.add(f)
        for line in open(os.path.join(bench.ROOT, CSRC, f)):
            if line.startswith('#include "') and line.split('"')[1].endswith(".cuh"):
                todo.append(line.split('"')[1])
    assert seen == set(bench.PROFILED[profile])


def test_kernels_run():
    zero = {k: 0 for k in (*bench.ROUTES, "graphs")}
    assert bench.kernels_run(zero, {**zero, "rows": 5}) == "entry-row kernels"
    assert bench.kernels_run(zero, {**zero, "rows": 1, "warps": 1}) == "entry-row kernels, warp-tile kernel"
    assert bench.kernels_run(zero, {**zero, "graphs": 1}) == "none"
