"""Checks of the kernel sources that need no GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_08637_b200", "csrc")


def test_dynamic_shared_memory_keeps_its_address_space():
    """Every kernel that aligns its dynamic shared memory does so with align_smem: an address rounded through an integer
    loses its address space, and every access becomes a generic one (5 to 10 % of a kernel's time)."""
    aligned = 0
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        for use in re.findall(r"uint8_t\* smem = ([^;]*);", text):
            assert use == "align_smem(smem_raw)", (name, use)
            aligned += 1
    assert aligned >= 4
