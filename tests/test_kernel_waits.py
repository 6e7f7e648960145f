"""Checks, from the kernels' sources, of ordering and exit rules that no run can be made to break safely:
a missing release or a copy still in flight at a kernel's exit corrupts memory only now and then."""

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_12659_gb300", "csrc")


def _source(*path):
    with open(os.path.join(CSRC, *path)) as f:
        return f.read()


def _sources():
    for d, _, names in os.walk(CSRC):
        for n in names:
            if n.endswith((".cu", ".cuh", ".h")):
                yield os.path.relpath(os.path.join(d, n), CSRC), _source(d, n)


def test_arrivals_on_a_peers_barrier_release_the_reads_before_them():
    # A peer that waits for such an arrival overwrites what the arriving warp has just read.
    found = 0
    for name, text in _sources():
        for arrival in re.findall(r"mbarrier\.arrive\.[\w.:]*shared::cluster\.b64", text):
            found += 1
            assert arrival.startswith("mbarrier.arrive.release.cluster."), f"{name}: {arrival}"
    assert found == 1
