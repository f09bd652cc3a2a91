"""The hash that ties the committed traffic figures to the kernels: it changes
with every source that the forward path is built from."""
import os
import re
import shutil

import pytest

import bench
from paper_2209_09671_gb300 import _build

NOT_FORWARD = {"fvm_adjoint.cu", "fvm_measure.cu"}


def _sources():
    """The forward translation units and the headers they include."""
    names = set(_build.SOURCES) - NOT_FORWARD
    for n in sorted(names):
        text = open(os.path.join(_build.CSRC, n)).read()
        names |= {h for h in re.findall(r'#include "(\w+\.\w+)"', text) if h != "fvm_adjoint.h"}
    for h in [n for n in names if not n.endswith(".cu")]:
        text = open(os.path.join(_build.CSRC, h)).read()
        names |= set(re.findall(r'#include "(\w+\.\w+)"', text))
    return sorted(names)


@pytest.mark.parametrize("name", _sources())
def test_hash_follows_the_forward_sources(name, tmp_path, monkeypatch):
    csrc = tmp_path / "paper_2209_09671_gb300" / "csrc"
    shutil.copytree(_build.CSRC, csrc)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    before = bench.source_hash()
    with open(csrc / name, "a") as f:
        f.write("\n")
    assert bench.source_hash() != before
