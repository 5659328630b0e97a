"""Host code that waits for the device, read as text (no GPU needed)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_16182_gb300", "csrc")


def test_event_times_are_read_after_a_wait_for_the_event():
    """cudaEventElapsedTime answers "not ready" for an event the runtime does
    not yet see as complete, so it is called in one place, behind a wait."""
    hits = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*"))):
        if not path.endswith((".cu", ".cuh", ".h")):
            continue
        text = re.sub(r"//[^\n]*", "", open(path).read())
        hits += [(os.path.basename(path), text[:k.start()]) for k in re.finditer(r"\bcudaEventElapsedTime\(", text)]
    assert [h[0] for h in hits] == ["lpp_engine.cu"]
    before = hits[0][1]
    body = before[before.rindex("float elapsed_ms("):]
    assert re.search(r"cudaEventSynchronize\(b\)", body)
