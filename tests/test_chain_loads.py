"""Kernels launched by launch_pdl can be resident while the kernels before them
still write, so they may not use the non-coherent load path, which is defined
only for data that nobody writes during the kernel's life."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1511_07152_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    return re.sub(r"\s+", " ", text)


def _files():
    return sorted(f for f in os.listdir(CSRC)
                  if f.endswith(".cu") and "launch_pdl(" in _source(f))


def test_chained_kernels_are_found():
    assert {"sepw_bin.cu", "sepw_tiled.cu", "sepw_window.cu"} <= set(_files())


@pytest.mark.parametrize("name", _files() + ["sepw_internal.cuh"])
def test_no_noncoherent_loads(name):
    text = _source(name)
    assert "__ldg(" not in text
    assert ".nc" not in text
    assert not re.search(r"const [\w ]+ ?\* ?__restrict__", text)
