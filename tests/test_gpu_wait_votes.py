"""A warp's bounded wait has one answer: lanes poll on their own, and if one runs
out while its neighbours still see the phase complete, none of them may go on
into shuffles or warp-collective tensor-memory instructions without it."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_02328_gb300", "csrc")


@pytest.mark.parametrize("name,wait", [("pairs.cu", "mbar_wait_bounded"), ("tile.cuh", "mbar_wait_bounded")])
def test_ring_kernels_wait_by_the_warp(name, wait):
    src = open(os.path.join(CSRC, name)).read()
    assert not re.search(r"\b%s\(" % wait, src) and "mbar_wait_warp(" in src


@pytest.mark.gpu
def test_a_warp_whose_lanes_disagree_gives_up_together():
    pytest.importorskip("torch")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_02328_gb300 import _lib
    rc, ms = _lib.af_diag_bounded_wait(2, 1 << 16)
    assert rc == _lib.AF_ETIMEOUT and ms < 1000.0
    rc, _ = _lib.af_diag_bounded_wait(1, 1 << 16)  # without lanes that give up the same wait succeeds
    assert rc == _lib.AF_OK
