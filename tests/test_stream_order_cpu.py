"""What the library clears or copies is ordered on the context's stream.

cudaMemset and cudaMemcpy without a stream run on the legacy default stream,
which nothing orders against a caller's non-blocking stream: a counter cleared
there can still be uncleared, or be cleared in the middle, when the kernel that
counts on it runs.  The one place that may use them is sg_init, which waits for
the device before it returns the context."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1410_6685_gb300", "csrc")
UNORDERED = re.compile(r"\bcuda(?:Memset|Memcpy)(?:2D|3D)?\s*\(")


def test_no_unordered_memory_operations():
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*"))):
        with open(path, encoding="utf-8") as f:
            text = f.read()
        init = re.search(r"^sg_status sg_init\(.*?^}", text, re.S | re.M)
        for m in UNORDERED.finditer(text):
            if (init and init.start() <= m.start() < init.end()
                    and "cudaDeviceSynchronize()" in text[m.end():init.end()]):
                continue
            found.append("%s:%d" % (os.path.basename(path), text.count("\n", 0, m.start()) + 1))
    assert found == []
