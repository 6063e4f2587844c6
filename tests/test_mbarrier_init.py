"""Every kernel that initialises mbarriers synchronises before another thread
can use them: between the end of the initialising branch (``fence_mbar_init``
by one thread) and the first copy, arrival, wait or commit that names a barrier
stands a warp, block or cluster barrier.  ``fence.mbarrier_init`` and proxy
fences order nothing between threads.

Read from the sources, since the hardware shows the missing barrier only when
the compiler leaves the warp diverged.
"""

import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1901_07499_gb300", "csrc")
SYNC = re.compile(r"__syncwarp\(|__syncthreads\w*\(|cluster\.sync\(|\bbar_sync\(|\bnamed_sync\(")
USE = re.compile(r"\b(?:bulk_load|\w*issue\w*|fetch|mbar_expect\w*|mbar_arrive|mbar_wait\w*|"
                 r"wait_slot|umma_commit)\(")


def _text(path):
    with open(path) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


def _after_branch(text, at):
    """Text behind the block that encloses position ``at``."""
    depth = 0
    for i in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth < 0:
            return text[i + 1:]
    raise AssertionError("unbalanced braces")


def _sites():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = _text(path)
        for m in re.finditer(r"\bfence_mbar_init\(\);", text):
            name = re.findall(r"\b(\w+_kernel)\(", text[:m.start()])[-1]
            yield pytest.param(text, m.end(), id="%s:%s" % (os.path.basename(path), name))


@pytest.mark.parametrize("text,at", list(_sites()))
def test_a_barrier_stands_before_the_first_use(text, at):
    rest = _after_branch(text, at)
    sync, use = SYNC.search(rest), USE.search(rest)
    assert sync is not None and use is not None
    assert sync.start() < use.start(), rest[:use.end()][-200:]


def test_the_sites_are_found():
    kernels = {p.id.split(":")[1] for p in _sites()}
    assert {"frame_kernel", "warp_kernel", "pair_kernel", "twin_kernel", "twin_rows_kernel",
            "twinpair_kernel", "dn_conv32_kernel", "dn_xtc_kernel"} <= kernels
