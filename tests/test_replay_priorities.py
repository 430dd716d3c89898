"""The factorisation runs on a high- and a low-priority stream; a graph forgets the
priorities of its nodes unless it is instantiated to use them.  Nothing but a time
shows it on the device, so the source is checked."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1404_0447_gb300", "csrc",
                   "capi.cu")


def test_replayed_factorisation_keeps_its_priorities():
    text = open(SRC).read()
    assert re.search(r"cudaGraphInstantiate\(&ex, g, priorities \? cudaGraphInstantiateFlagUseNodePriority : 0\)", text)
    call = re.search(r"replay_or_enqueue\(h, &h->fgraph_exec\[bk\], [^,]+, st, (\w+)", text)
    assert call and call.group(1) == "true"
