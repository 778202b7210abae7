"""What the device code waits with, read from its source: a wait that cannot give up would hold the GPU for good once any other
wait of the CTA has given up and its warps no longer keep step."""
import glob
import os
import re

import pytest

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


def _ring_states(slots, convs, both_see):
    """Every order in which weight copies can land in a ring that two warps read, chunk by chunk in turn. A barrier's test passes if the
    phase before the current one has the parity that is asked for. Returns (a chunk was multiplied before its copy had landed, somebody
    waits for good)."""
    chunks = [(q, kc) for q, nk in enumerate(convs) for kc in range(nk)]
    first = [sum(convs[:q]) for q in range(len(convs))]
    n = len(chunks)

    def full(state, g):                          # the test of the barrier of chunk g's slot, for its round
        landed = sum(1 for k in range(g % slots, n, slots) if state[3] >> k & 1)
        return landed % 2 != g // slots % 2

    def steps(state):
        at, armed, issued, mask = state
        if issued < n:                           # the loader: the slot's last chunk is done with
            k = issued - slots
            if k < 0 or all(at[w] > k for w in (0, 1) if both_see or w == chunks[k][1] & 1):
                yield at, armed, issued + 1, mask
        for k in range(issued):                  # any copy in flight lands
            if not mask >> k & 1:
                yield at, armed, issued, mask | 1 << k
        for w in (0, 1):
            g = at[w]
            if g == n:
                continue
            q, kc = chunks[g]
            operand = min(at) >= first[q]        # the conv before is complete
            go = tuple(at[v] + (v == w) for v in (0, 1)), tuple(armed[v] and v != w for v in (0, 1)), issued, mask
            if kc & 1 != w:
                if (not both_see or full(state, g)) and (operand or not (kc == 0 and w >= convs[q])):
                    yield go
            elif not armed[w]:                   # the weights are waited for before the operand is
                if full(state, g):
                    yield at, tuple(armed[v] or v == w for v in (0, 1)), issued, mask
            elif operand:
                yield go if mask >> g & 1 else None

    seen, todo, stale, stuck = set(), [((0, 0), (False, False), 0, 0)], False, False
    while todo:
        state = todo.pop()
        if state in seen:
            continue
        seen.add(state)
        after = list(steps(state))
        stale |= None in after
        stuck |= not after and min(state[0]) < n
        todo += [s for s in after if s is not None]
    return stale, stuck


@pytest.mark.parametrize("slots,convs", [(3, (4, 4)), (4, (3, 3, 3)), (3, (1, 3, 4)), (4, (2, 1, 3, 4))])
def test_a_ring_that_changes_hands_is_seen_by_both(slots, convs):
    """Levels of one tile deal a conv's chunks to two warps. Where each tests only its own chunks' slots, a copy that is late is
    taken for the one before the last."""
    assert _ring_states(slots, convs, True) == (False, False)
    if slots == 3 or 3 in convs[:-1]:
        assert _ring_states(slots, convs, False)[0]
    with open(os.path.join(CSRC, "res_flow.cu")) as f:
        text = f.read()
    skipped = re.search(r"if \(one && \(kc & 1\) != which\) \{(.*?)\n      \}", text, re.S).group(1)
    assert "rf_wait(f, &ctl->w_full[slot]" in skipped and "rf_arrive_local(&ctl->w_empty[slot])" in skipped
    assert re.search(r"mbar_init\(ptx::smem_u32\(&ctl\.w_empty\[s\]\), 2\)", text)
