"""Bulk copies reach the issuing CTA only: the library is loaded by one process on each of several GPUs, and
loads that one CTA issues for its whole cluster are kept out of it in every form."""

import pathlib

import pytest

import paper_1310_5954_gb300 as pkg

CSRC = pathlib.Path(pkg.__file__).parent / "csrc"


@pytest.mark.parametrize("path", sorted(p.name for p in CSRC.iterdir() if p.suffix in (".cu", ".cuh", ".cpp", ".hpp")))
def test_no_load_for_the_cluster(path):
    assert "multicast" not in (CSRC / path).read_text()
