"""Asynchronous copies and the compiler, by reading the sources: a statement that starts, closes or waits for copies must be
a barrier to the compiler too.  A thread that waits for its own copies reads their words with ordinary loads and no
__syncthreads() between, and without the clobber those loads may be placed above the wait."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1805_10032_b200", "csrc")


def test_copies_and_their_waits_clobber_memory():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.h"))):
        for text in re.findall(r"asm\s*(?:volatile)?\s*\(.*?\);", open(path).read(), re.S):
            if "cp.async" in text:
                seen += 1
                assert "volatile" in text and '"memory"' in text, (os.path.basename(path), text)
    assert seen
