"""The factorisation and the adjoint run on a high- and a low-priority stream; a graph
forgets the priorities of its nodes unless it is instantiated to use them.  Nothing
but a time shows it on the device, so the source is checked."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1404_0447_gb300", "csrc",
                   "capi.cu")


def test_replayed_two_stream_sequences_keep_their_priorities():
    text = open(SRC).read()
    assert re.search(r"cudaGraphInstantiate\(&ex, g, priorities \? cudaGraphInstantiateFlagUseNodePriority : 0\)", text)
    for name in ("fgraph_exec[bk]", "agraph_exec"):
        call = re.search(r"replay_or_enqueue\(h, &h->" + re.escape(name) + r", [^,]+, st, (\w+)", text)
        assert call and call.group(1) == "true"
