"""Rules of the kernels' synchronisation, checked in their sources: a run that breaks one of them looks right until it does not."""
import os
import re

import pytest

from paper_2601_01712_b200 import build

SOURCES = {os.path.basename(p): open(p).read() for p in build.sources() if p.endswith(".cu")}


@pytest.mark.parametrize("name", [n for n, text in SOURCES.items() if "load_cluster4(tc::" in text])
def test_reads_of_a_peers_shared_memory_are_released_before_it_may_end(name):
    """What follows the last read of a peer's shared memory is an arrival that releases the read: a relaxed one orders nothing, and the
    peer may end while the read is under way."""
    text = SOURCES[name]
    after = text[text.rindex("load_cluster4(tc::"):]
    end = re.search(r"tc::cluster_(sync|wait)\(\)", after)
    assert end, "no cluster barrier behind the reads"
    assert end.group(1) == "sync" or "tc::cluster_arrive_release()" in after[:end.start()]
