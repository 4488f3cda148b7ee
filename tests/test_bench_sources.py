"""The recorded figures of the pair kernels (executed FLOPs, DRAM bytes) hold for the sources they were taken on:
bench.py must notice a change in any file that those kernels are compiled from."""

import os
import re
import shutil
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402

CSRC = os.path.join(ROOT, "paper_2005_02498_gb300", "csrc")


def included(name, seen=()):
    """Files under csrc/ that `name` includes, itself first."""
    seen = list(seen) + [name]
    for inc in re.findall(r'#include "([^"/]+)"', open(os.path.join(CSRC, name)).read()):
        if inc not in seen:
            seen = included(inc, seen)
    return seen


def test_every_source_of_the_pair_kernels_is_hashed():
    assert set(bench.KERNEL_SOURCES) == set(included("dd_kernels.cu"))


@pytest.mark.parametrize("name", sorted(bench.KERNEL_SOURCES))
def test_a_change_in_any_of_them_is_noticed(name, tmp_path, monkeypatch):
    d = tmp_path / "paper_2005_02498_gb300" / "csrc"
    d.mkdir(parents=True)
    for f in bench.KERNEL_SOURCES:
        shutil.copy(os.path.join(CSRC, f), d / f)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    before = bench.kernel_source_sha()
    with open(d / name, "a") as f:
        f.write("// changed\n")
    assert bench.kernel_source_sha() != before
