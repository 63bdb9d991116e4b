"""What the CTAs of the persistent kernels exchange must arrive whole.  A value
word and its epoch are one 64-bit element: PTX's memory model makes the elements
of a vector access (and scalar accesses) indivisible, not the vector, so no
exchange access may have 32-bit elements, and every one is a relaxed access at
device scope (a weak one may be torn or kept in a register)."""
import os
import re

from paper_1812_04789_gb300 import build


def test_exchange_accesses_have_64_bit_elements():
    src = open(os.path.join(build.CSRC, "dg_exchange.cuh")).read()
    ops = re.findall(r'"((?:ld|st)\.[a-z0-9_.]+)', src)
    assert ops
    for op in ops:
        assert re.fullmatch(r"(ld|st)\.relaxed\.gpu\.global(\.v2)?\.u64", op), op
