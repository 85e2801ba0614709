"""Rules of the CUDA sources that a compiler does not check.  No GPU is needed."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_03858_b200", "csrc")


def code(path):
    """The source without comments."""
    text = open(path).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", " ", text, flags=re.S)


def test_no_load_takes_the_non_coherent_path():
    # Kernels are launched so that they may start while the kernel before them still writes, and their inputs
    # are what it writes: ld.global.nc, __ldg and const __restrict__ are for memory that nobody writes
    # while the kernel lives.
    files = glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.h"))
    assert files
    for path in files:
        found = re.findall(r"__ldg\b|\bld\.global\.nc\b|__restrict__", code(path))
        assert not found, (os.path.basename(path), found)


def test_every_kernel_with_an_early_launch_waits_for_its_predecessor():
    seen = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        text = code(path)
        for m in re.finditer(r"__global__[^;{]*?\b(\w+_kernel)\([^)]*\)\s*\{(.*?)\n\}", text, flags=re.S):
            name, body = m.groups()
            ordinary = re.search(r"\b" + name + r"(<\w+>)?\s*<<<", text)
            assert ("pdl_wait()" in body) != bool(ordinary), name
            seen += 1
    assert seen >= 10
