"""What dependent launches rest on (csrc/ptx.cuh, dep_wait): a kernel may start before the kernel
in front of it on the stream has finished, so whatever it reads before the wait has to be complete
when it is launched.  Read from the sources, since running the opposite could leave an array."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2107_12371_gb300", "csrc")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    text = re.sub(r"/\*.*?\*/", " ", text, flags=re.S)
    return re.sub(r"//[^\n]*", " ", text)


def body(text, head):
    """The braces' content of the definition whose text begins with `head`."""
    at = text.index("{", text.index(head))
    depth, i = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[at + 1:i]
        i += 1


def test_a_handles_arrays_are_complete_before_a_product_can_be_launched():
    """build_sell writes the arrays that products read ahead of their wait, and the tuner launches
    products right after it."""
    b = body(source("convert.cu"), "spmv_status_t build_sell(")
    last_kernel = b.rindex("<<<")
    assert "cudaStreamSynchronize(st)" in b[last_kernel:]
    # (an early return behind that kernel, if any, is an error's)
    assert b[last_kernel:].count("return SPMV_OK") == 1
