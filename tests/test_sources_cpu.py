"""What can be said of the device code from its sources alone."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1705_04862_b200", "csrc")


def sources():
    return {os.path.basename(p): open(p).read() for p in sorted(glob.glob(os.path.join(CSRC, "*")))}


def test_there_is_one_build():
    """No switch of the preprocessor gives another kernel, or another way to launch one, than the one that is tested."""
    for name, text in sources().items():
        for directive in re.findall(r"^\s*#\s*((?:el)?if.*|ifn?def.*|define.*|undef.*)$", text, re.M):
            assert directive == "ifdef __CUDACC__", (name, directive)      # the host compiler reads the host's part
