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


def _kernels():
    for name, text in _sources():
        for body in text.split("__global__")[1:]:
            head = re.search(r"\b(\w+_kernel)\s*\(", body)
            if head:
                yield name + ": " + head.group(1), body


def test_dependents_are_released_after_the_wait_and_the_tensor_memory():
    """A dependent CTA on the same SM may allocate tensor memory before it waits: were it released while a CTA of this
    grid has yet to allocate, the two could wait for each other for ever."""
    seen = set()
    for name, body in _kernels():
        releases = [m.start() for m in re.finditer(r"\bpdl_launch_dependents\(\)", body)]
        allocs = [m.start() for m in re.finditer(r"\btmem_alloc(?:_pair)?\(", body)]
        assert releases and "pdl_wait()" in body, name
        assert body.index("pdl_wait()") < releases[0], name
        if allocs:
            assert max(allocs) < body.index("__syncthreads()", max(allocs)) < releases[0], name
            seen.add(name.split(": ")[1])
    assert seen == {"attn_kernel", "attn_persist_kernel", "attn_bwd_kernel", "decode2_kernel", "decode_cluster_kernel",
                    "linear_kernel", "linear_unit_kernel", "linear_narrow_kernel", "logprob_kernel"}
