"""Kernels that may be launched while their predecessor still runs (those that call grid_wait()) read what it
writes by plain loads only. ld.global.nc, which __ldg and const __restrict__ pointers turn into, is defined for
data that nobody writes while the kernel is alive, and the compiler may move such a load above the wait. Only
the wall tables, written once when a context is created, may be read that way. Checked in the sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_09160_gb300", "csrc")
SOURCES = ("adjoint.cuh", "aux_kernels.cuh", "stream_collide.cuh", "stream_collide_sep.cuh")
TABLES = re.compile(r"__ldg\(a\.(mask|links) \+ ")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _kernels(text):
    """(name, source from __global__ to the end of the body) of every kernel."""
    for m in re.finditer(r"__global__", text):
        head = text.index("{", m.end())
        depth, at = 1, head + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[at], 0)
            at += 1
        yield re.search(r"\b(k_\w+)\(", text[m.start():]).group(1), text[m.start():at]


def test_overlapped_kernels_read_by_plain_loads():
    seen = set()
    for name in SOURCES:
        for kernel, body in _kernels(_code(name)):
            if "grid_wait()" not in body:
                continue
            seen.add(kernel)
            assert "__restrict__" not in body, kernel
            for use in re.findall(r"__ldg\([^;]*", body):
                assert TABLES.match(use), (kernel, use[:60])
    assert seen == {"k_adjoint", "k_phase_advance", "k_phase_forces", "k_stream_collide", "k_stream_collide_sep"}


def test_shared_loads_of_overlapped_kernels_are_plain():
    """The storage codec and the sum over blocks, which those kernels call."""
    assert "__ldg" not in _code("lattice.cuh")
    sums = _code("stream_collide.cuh")
    at = sums.index("void sum_partials")
    assert "__restrict__" not in sums[at:sums.index("{", at)]
