"""The guard on captured DRAM figures in bench.py: a kernel's sources are its file and every header of the
project that it includes, and a change in any of them makes its figures stale."""
import os
import re
import shutil

import pytest

import bench


@pytest.mark.parametrize("kernel", sorted(bench.KERNEL_FILES))
def test_sources_are_closed_under_includes(kernel):
    names = bench.kernel_sources(kernel)
    assert bench.KERNEL_FILES[kernel] in names and len(names) >= 4
    for name in names:
        for inc in re.findall(r'#include "([^"]+)"', open(os.path.join(bench.CSRC, name)).read()):
            assert inc in names or not os.path.exists(os.path.join(bench.CSRC, inc))


@pytest.mark.parametrize("kernel", sorted(bench.KERNEL_FILES))
def test_a_change_in_any_source_changes_the_hash(kernel, tmp_path, monkeypatch):
    before = bench.source_sha(kernel)
    for name in bench.kernel_sources(kernel):
        d = tmp_path / name
        shutil.copytree(bench.CSRC, d)
        monkeypatch.setattr(bench, "CSRC", str(d))
        assert bench.source_sha(kernel) == before
        with open(d / name, "a") as fh:
            fh.write("\n// changed\n")
        assert bench.source_sha(kernel) != before, name
        monkeypatch.undo()


def test_every_captured_figure_names_a_known_kernel():
    assert {k for k, _ in bench.DRAM_BYTES_PER_LAUNCH} <= set(bench.KERNEL_FILES)
