"""The tagged exchange of the grid's iteration kernel orders a value and its tag by nothing but their
sharing one 64-bit element of a memory access (narrower elements of a vector access are separate
accesses in no given order): every relaxed access of the kernel's source has 64-bit elements."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2302_14344_gb300",
                   "csrc", "grid_iter.cuh")


def test_value_and_tag_share_a_64_bit_element():
    with open(SRC) as f:
        ops = re.findall(r"(ld|st)\.relaxed\.gpu\.global\.((?:v[24]\.)?[bu]\d+)", f.read())
    assert {o for o, _ in ops} == {"ld", "st"}
    assert all(t.endswith("64") for _, t in ops), ops
