"""Every TMEM allocation of a CTA pair comes after a barrier of the cluster:
one CTA allocating while its peer has not started can leave the peer waiting
in tcgen05.alloc for good.  The only such instruction is in one helper, which
takes the barrier first, in all threads."""

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_08573_gb300", "csrc")


def test_pair_allocation_follows_a_cluster_barrier():
    text = {}
    for f in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, f)) as h:
            text[f] = re.sub(r"//[^\n]*", "", h.read())
    assert [f for f, s in text.items() for _ in re.findall(r"tcgen05\.alloc\.cta_group::2", s)] == ["ff_ptx.cuh"]
    body = re.search(r"void tmem_alloc_pair\([^)]*\) \{(.*?)\n\}", text["ff_ptx.cuh"], re.S).group(1)
    assert re.match(r"\s*cluster_sync\(\);\s*if \(\w+\) \{\s*asm volatile\(\"tcgen05\.alloc", body)
    # and no caller puts it under a condition on the thread
    calls = [(f, line) for f, s in text.items() if f != "ff_ptx.cuh" for line in s.splitlines()
             if "tmem_alloc_pair(" in line]
    assert len(calls) == 3
    for f, line in calls:
        assert re.match(r"\s*ptx::tmem_alloc_pair\(", line), (f, line)
