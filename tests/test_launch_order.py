"""What the sources have to keep to so that kernels launched with programmatic stream serialization, each of which may
start while its predecessor runs, stay ordered like a plain stream (the rules stand in tik_ptx.cuh)."""
import glob
import os
import re

from paper_2609_35140_b200 import build


def _sources():
    for path in sorted(glob.glob(os.path.join(build.CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        yield os.path.basename(path), re.sub(r"/\*.*?\*/", "", text, flags=re.S)


def test_no_load_that_may_move_above_the_wait():
    """__restrict__ and read-only loads tell the compiler that an input does not change while the kernel lives."""
    for name, text in _sources():
        assert not re.search(r"__restrict__|\b__ldg\b|ld\.global\.nc", text), name
