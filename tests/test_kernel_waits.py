"""What the device code waits with, read from its source: a wait that cannot give up would hold the GPU for good once any other
wait of the CTA has given up and its warps no longer keep step."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2206_08869_b200", "csrc")


def test_nobody_arrives_at_a_named_barrier_without_waiting():
    """Warps that all wait at a named barrier cross it in step, whatever their other waits return. One that only arrives does
    not: two of its arrivals stand for one of another warp, which then waits for an arrival that never comes."""
    crossings = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        with open(path) as f:
            text = f.read()
        assert not re.search(r'"[^"]*\bbar(rier)?(\.cta)?\.arrive\b', text), path
        crossings += len(re.findall(r'"bar\.sync \d+, ', text))
    assert crossings >= 6
