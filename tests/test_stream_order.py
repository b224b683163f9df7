"""The library's copies and fills are ordered on a stream.

A handle runs on its caller's stream, which may be a non-blocking one that
does not wait for the legacy default stream.  A copy from pageable memory on
the legacy stream may return once the data is staged, before it has reached the
device, so nothing would order the handle's kernels after it.  The plain
(stream-less) forms of the runtime's copies and fills go to the legacy stream:
the sources use none of them.
"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_03148_gb300", "csrc")
LEGACY = re.compile(r"\bcuda(?:Memcpy(?:2D|3D|ToSymbol|FromSymbol|Peer)?|Memset(?:2D|3D)?)\s*\(")


def test_copies_and_fills_name_their_stream():
    found = []
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        text = re.sub(r"/\*.*?\*/", lambda m: "\n" * m.group().count("\n"), text, flags=re.S)
        for k, line in enumerate(text.splitlines(), 1):
            if LEGACY.search(line.split("//")[0]):
                found.append(f"{name}:{k}: {line.strip()}")
    assert not found, found
