"""The 3D plane pipeline's ring of planes is read across warps, so what orders a refill after the reads is the block's
barrier.  The order of an iteration is read from the kernel's source, and every pair of a read and a refill of one
slot is checked for a barrier between them."""
import os
import re

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1601_08103_gb300", "csrc",
                      "planepipe.cuh")


def _iteration(text):
    """What one iteration does with the ring, in program order."""
    body = text[text.index("auto iteration = ["):]
    body = re.sub(r"//[^\n]*", "", body[:body.index("\n    };")])
    what = {"copy_wait<": "wait", "fetch(free_slot)": "fill", "__syncthreads()": "barrier", "first(r)": "read"}
    found = sorted((body.index(k), v) for k, v in what.items())
    assert all(body.count(k) == 1 for k in what)
    return [v for _, v in found]


def test_a_refill_waits_for_every_warps_reads():
    text = open(SOURCE).read()
    stages = int(re.search(r"kPpStages = (\d+);", text).group(1))
    order = _iteration(text)
    assert "take(lane == 31 ? 1 : 0, lane == 31 ? after : before)" in text  # the read across warps
    # the iterations' events: (event, slot), slots as the kernel turns them
    events, slot, free = [], 0, stages - 1
    for _ in range(4 * stages):
        events += [(e, {"fill": free, "read": slot}.get(e)) for e in order]
        free, slot = slot, (slot + 1) % stages
    for a, (e, s) in enumerate(events):
        for b in range(a + 1, len(events)):
            f, t = events[b]
            between = [x for x, _ in events[a:b]]
            if {e, f} == {"read", "fill"} and s == t:
                # a barrier parts them (a read after a fill also has to wait for the copy)
                assert "barrier" in between, (a, b)
                assert e == "read" or "wait" in between, (a, b)
