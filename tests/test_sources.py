"""Rules of the CUDA sources that no run can show reliably: checked by reading them."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_05096_b200", "csrc")


def _code(name):
    """A source file without its comments."""
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def test_no_load_takes_the_read_only_path():
    """Kernels start while the kernel before them still runs and wait inside: nothing they read is read-only for their whole
    life, so no load may go through the read-only path (a line of it may sit in L1 from before)."""
    names = [os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "*.cu*"))]
    assert len(names) >= 9
    for name in names:
        assert not re.search(r"__ldg\s*\(|ld\.global\.nc|\bldg\b", _code(name)), name
