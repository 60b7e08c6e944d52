"""Kernels may start while the one before them still writes what they will read, and wait for it at pdl_wait().  In the source
nothing may allow a load above that wait (no GPU needed)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_01798_b200", "csrc")


def _sources():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            yield f, re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())


def test_no_read_only_promise_about_what_other_kernels_write():
    for f, text in _sources():
        assert "__ldg(" not in text, f
        # typed pointers are dereferenced; the gradient's `const void*` is an address for volatile asm loads
        for m in re.finditer(r"const\s+(\w+)\s*\*\s*__restrict__", text):
            assert m.group(1) in ("void", "char"), (f, m.group(0))


def test_every_kernel_waits():
    """In its own body, or in the block function that it hands the wait to (WAIT = true)."""
    kernels = 0
    for f, text in _sources():
        for m in re.finditer(r"__global__[^;{]*?(\w+)\(", text):
            body = text[m.end():text.index("\n}\n", m.end())]
            kernels += 1
            assert "pdl_wait()" in body or re.search(r"lut_block<BITS, true>", body), (f, m.group(1))
    assert kernels >= 10
