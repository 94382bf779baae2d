"""Two lanes share a translation on the FP64 path: each writes one part (real or imaginary)
of the pair's row in shared memory and both then read both parts.  Only a __syncwarp orders
one lane's writes before the other's reads (votes and shuffles do not); a missing one
seldom shows in the results, so the sources are read."""
import os
import re

import pytest

from paper_2210_07021_gb300 import build

TEXT = open(os.path.join(build.CSRC, "m2l_pair64.cu")).read()


@pytest.mark.parametrize("function", ["k_m2l_pair64", "translate_row64"])
def test_a_warp_synchronisation_orders_the_parts(function):
    body = TEXT[TEXT.index(function + "("):]
    body = re.sub(r"//[^\n]*", "", body[:body.index("\n}\n")])
    written = body.index("row[2 * l + prt] = c[l]")
    read = body.index("const double orr = row[2 * l]")
    assert "__syncwarp(" in body[written:read]
