"""Blocks of one launch that depend on one another: the Cholesky inverse's kernels run to the end whatever order and
however few at a time their blocks are scheduled in.  A block that waited for others of its launch would run into
its time limit on a GPU that another stream keeps busy, so no kernel there reads a clock or spins."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1810_07772_gb300", "csrc")


def test_cholesky_blocks_wait_for_nothing():
    text = re.sub(r"//[^\n]*", "", open(os.path.join(SRC, "k_eps.cu")).read())
    assert "atomicAdd(arrived" in text                  # the hand-over: the last block to arrive goes on
    for wait in ("globaltimer", "clock64", "ld.acquire", "nanosleep", "while (seen", "GW_E_TIMEOUT"):
        assert wait not in text, wait
