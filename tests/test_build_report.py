"""What ptxas reported of the convolution, which is written to fit 64 registers (four CTAs per SM): it does not spill."""
import os
import re

import pytest

from paper_2609_23900_b200 import build


def spills(source):
    """Bytes of spill stores and loads of each kernel of a source (mangled names)."""
    path = os.path.join(build.HERE, "build", source + ".ptxas")
    if not os.path.exists(path):
        pytest.skip("the library was not built here")
    return {m[1]: (int(m[2]), int(m[3])) for m in
            re.finditer(r"Compiling entry function '(\w+)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads", open(path).read(), re.S)}


@pytest.mark.parametrize("rows", ["f", "13__nv_bfloat16"])
def test_the_convolution_does_not_spill(rows):
    found = {k: v for k, v in spills("kernels.cu").items() if re.search(rf"11conv_kernelI{rows}Li(4|8|16)E", k)}
    assert len(found) == 6 and all(v == (0, 0) for v in found.values()), found
