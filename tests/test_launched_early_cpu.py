"""What the kernels that are launched early (set up on SMs that the kernel before has left) have to keep to, read from their
source: a kernel that broke it would hang a GPU, or read what the kernel before has not written yet, once in a long while only."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2012_02030_b200", "csrc")


def _source(path):
    with open(path) as f:
        return re.sub(r"/\*.*?\*/|//[^\n]*", "", f.read(), flags=re.S)


def _block(text, start, brackets="{}"):
    """From `start` to the end of the first bracketed block behind it."""
    depth = 0
    for x in range(text.index(brackets[0], start), len(text)):
        depth += (text[x] == brackets[0]) - (text[x] == brackets[1])
        if depth == 0:
            return text[start:x + 1]
    raise AssertionError("no end")


def _kernels():
    """(name, parameters and body) of every kernel, the helpers that a kernel begins with written out in it."""
    helpers = {}
    for name, file in (("after_previous", "ap_common.cuh"), ("begin_with_tmem", "ap_sm100.cuh")):
        text = _source(os.path.join(CSRC, file))
        m = re.search(r"\b%s\(" % name, text)
        if m:
            helpers[name] = _block(text, text.index("{", m.start()))
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = _source(path)
        for m in re.finditer(r"__global__", text):
            kernel = _block(text, m.start())
            name = re.search(r"(\w+_kernel)\s*\(", kernel).group(1)
            for helper, body in helpers.items():
                kernel = re.sub(r"\b%s\b[^;]*;" % helper, lambda _: body, kernel)
            out.append((os.path.basename(path)[:-3] + ":" + name, kernel))
    return out


KERNELS = dict(_kernels())
EARLY = sorted(k for k, body in KERNELS.items() if "wait_previous()" in body or "griddepcontrol.wait" in body)


def test_kernels_are_found():
    assert len(EARLY) >= 14 and len(KERNELS) > len(EARLY)
    assert sum("tmem_alloc(" in KERNELS[k] for k in EARLY) == 6


@pytest.mark.parametrize("name", [k for k in EARLY if "tmem_alloc(" in KERNELS[k]])
def test_tensor_memory_is_taken_between_the_kernel_before_and_the_kernel_behind(name):
    """An allocation blocks until columns are free.  A block that held some while it waits for the kernel before, or let the kernel
    behind take some before it has its own, would be one of a ring of blocks that wait for one another."""
    body = KERNELS[name]
    assert body.count("tmem_alloc(") == 1
    alloc = body.index("tmem_alloc(")
    assert "wait_previous()" in body[:alloc]
    barrier = re.search(r"__syncthreads\(\)|bar\.sync", body[alloc:])
    allow = body.index("allow_next()")
    assert allow > alloc + barrier.end()


@pytest.mark.parametrize("name", EARLY)
def test_no_parameter_is_declared_read_only(name):
    """The compiler may read through a const __restrict__ parameter as if nobody wrote there while the kernel is resident."""
    parameters = KERNELS[name].split("{", 1)[0]
    assert not re.search(r"const\s+[\w ]+\*\s*__restrict__", parameters)


def test_no_load_takes_its_data_for_read_only():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        assert not re.search(r"\.global\S*\.nc\b|\b__ldg\b", _source(path)), path
