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


FILES = ["spmv.cu", "spmm.cu", "cg.cu", "cgkern.cuh", "mcg.cu"]  # those with dependent launches


def test_vectors_are_read_behind_the_wait():
    """Vectors may still be written when a dependent launch begins, so nothing there reads them as
    read-only data (whose loads the compiler may also move ahead of the wait), and the loads that
    it could move are volatile."""
    for name in FILES:
        assert not re.search(r"__ldc?g\s*\(|\.nc\b", source(name)), name
    reads = re.findall(r"void ld_x\([^{]*\{[^}]*\}|(?:double|float) ld_(?:x|l2)\([^{]*\{.*?\n\}",
                       source("ptx.cuh"), flags=re.S)
    assert len(reads) >= 8
    for r in reads:
        assert "asm volatile" in r or "= ld_x(p)" in r, r
        assert ".nc" not in r and "asm(" not in r, r


def test_vectors_of_dependent_kernels_are_not_restricted():
    """A restricted pointer's loads may be moved across the wait whatever it clobbers."""
    kernels = 0
    for name in FILES:
        text = source(name)
        for m in re.finditer(r"__global__", text):
            head = text[m.start():text.index("{", m.start())]
            code = body(text[m.start():], "__global__")
            if "dep_wait" not in code:
                continue
            kernels += 1
            for arg in re.findall(r"__restrict__\s+(\w+)", head):
                assert arg in ("sp", "val"), (name, arg)
    assert kernels >= 12
