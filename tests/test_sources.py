"""Rules of the CUDA sources that no run can show broken: kernels overlap their launch with the kernel
before them, so what they do ahead of stream_order(), and how they read memory, matters."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1603_05279_b200", "csrc")
SOURCES = {os.path.basename(f): re.sub(r"//[^\n]*|/\*.*?\*/", "", open(f).read(), flags=re.S)
           for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*")))}


def kernels(source):
    """(name, text from the kernel's first line to the next kernel's) of a source."""
    parts = source.split("__global__")[1:]
    return [(re.search(r"(\w+)\s*\(", re.sub(r"__launch_bounds__\([^)]*\)", "", p)).group(1), p) for p in parts]


@pytest.mark.parametrize("name", sorted(SOURCES))
def test_no_load_promises_that_memory_is_constant(name):
    """A read-only load may be moved ahead of stream_order(), to where the kernel before still writes."""
    assert "__ldg(" not in SOURCES[name] and "ld.global.nc" not in SOURCES[name]
    assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", SOURCES[name])


@pytest.mark.parametrize("name", sorted(n for n in SOURCES if "launch_kernel(" in SOURCES[n] and n.endswith(".cu")))
def test_memory_is_not_read_before_the_kernel_in_front_is_done(name):
    for kernel, text in kernels(SOURCES[name]):
        before, wait, _ = text.partition("stream_order();")
        assert wait, "%s: %s does not wait for the kernels before it" % (name, kernel)
        assert not re.search(r"load_global\(|cp\.async|bulk_copy_g2s\(", before[before.index("{"):].split("auto ")[0]), kernel


@pytest.mark.parametrize("name", sorted(n for n in SOURCES if "tcgen05.alloc" in SOURCES[n]))
def test_tensor_memory_is_taken_before_the_next_kernel_may_start(name):
    """stream_order() may let the next kernel start.  A block of it that takes an SM's tensor memory before
    this kernel's block there has would hold it while it waits for this kernel: neither would ever go on."""
    found = [text for _, text in kernels(SOURCES[name]) if "tcgen05.alloc" in text and "stream_order();" in text]
    for text in found:
        before = text.partition("stream_order();")[0]
        assert "__syncthreads();" in before[before.rindex("tcgen05.alloc"):]
    assert found or name == "peaks.cu"               # measures with ordinary launches
