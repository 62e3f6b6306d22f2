"""Rules of the kernels' synchronisation, checked in their sources: a run that breaks one of them looks right until it does not."""
import os
import re

import pytest

from paper_2601_01712_b200 import build

SOURCES = {p: open(os.path.join(build.CSRC, p)).read() for p in sorted(os.listdir(build.CSRC)) if p.endswith((".cu", ".cuh"))}


@pytest.mark.parametrize("name", [n for n, text in SOURCES.items() if "load_cluster4(tc::" in text])
def test_reads_of_a_peers_shared_memory_are_released_before_it_may_end(name):
    """What follows the last read of a peer's shared memory is an arrival that releases the read: a relaxed one orders nothing, and the
    peer may end while the read is under way."""
    text = SOURCES[name]
    after = text[text.rindex("load_cluster4(tc::"):]
    end = re.search(r"tc::cluster_(sync|wait)\(\)", after)
    assert end, "no cluster barrier behind the reads"
    assert end.group(1) == "sync" or "tc::cluster_arrive_release()" in after[:end.start()]


@pytest.mark.parametrize("name", [n for n, text in SOURCES.items() if re.search(r"mbar_wait\(|RowStats", text)])
def test_two_warps_that_share_a_barrier_keep_count(name):
    """Every wait gives up after a second.  Two warps that meet at a barrier in a loop must come to it equally often: if one left alone
    after a wait of its own ran out, the other would wait at the barrier for ever.  So a barrier of 64 threads is a vote on which both leave
    (tc::pair_all), or a warp that left early still goes through the meetings it owes."""
    text = SOURCES[name]
    plain = re.findall(r".*bar(?:rier)?(?:\.cta)?\.sync[^;]*\b64\s*;.*", text)
    assert all("auto meet = [&]" in line for line in plain)
    if plain:
        assert len(plain) == 1 and re.search(r"for \(; j < nb; \+\+j\) meet\(\);", text)
