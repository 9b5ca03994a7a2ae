"""Alignment of the shared memory that holds the local sweeps' state (rcm_local.cuh), from the sources.

The bitmap at the start of the state is read and written 16 bytes at a time, and dynamic shared memory
begins wherever a kernel's static part ends unless its declaration says otherwise. Nothing at run time
shows a missing attribute until the static part changes size, and a misaligned access would be a fault on
the GPU, so the declarations are checked as text."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1610_08128_gb300", "csrc")
KERNEL_FILES = ("rcm_single_kernels.cuh", "rcm_batch.cu")


def test_dynamic_shared_memory_of_the_engines_is_16_byte_aligned():
    found = 0
    for name in KERNEL_FILES:
        with open(os.path.join(CSRC, name)) as f:
            for line in f:
                code = line.split("//")[0]
                if "extern __shared__" in code:
                    found += 1
                    assert re.search(r"__align__\((16|32|64|128)\)", code), (name, line.strip())
    assert found >= 4  # the grid, component, small and batch kernels


def test_bitmap_words_come_in_whole_16_byte_groups():
    with open(os.path.join(CSRC, "rcm_local.cuh")) as f:
        text = f.read()
    rule = re.search(r"int local_vis_words\(long long n\) \{ return \(int\)\((.*)\); \}", text).group(1)
    for n in (0, 1, 96, 97, 98, 127, 128, 129, 4608, 79872, 1_000_001, 1_458_000):
        words = eval(rule.replace("/", "//"), {"n": n})
        # a bit per vertex from a first word that may start in the middle, then whole groups of four words
        assert words % 4 == 0 and 32 * words >= n + 31
