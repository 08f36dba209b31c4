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


def test_every_kernel_family_has_a_launch():
    """The names that the profile can report are those of kernels that are there."""
    text = sources()
    families = re.findall(r"KID_\w+", re.search(r"enum KernelId \{(.*?)\};", text["common.cuh"], re.S).group(1))
    names = re.search(r"names\[KID_COUNT\] = \{(.*?)\};", text["common.cuh"], re.S).group(1)
    assert families[-1] == "KID_COUNT" and len(re.findall(r'"\w+"', names)) == len(families) - 1
    elsewhere = "".join(t for name, t in text.items() if name != "common.cuh")
    for kid in families[:-1]:
        assert re.search(r"\b%s\b" % kid, elsewhere), kid
