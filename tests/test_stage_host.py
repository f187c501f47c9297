"""What the build says of the stage operators' kernels."""
import os
import re

import pytest


@pytest.fixture(scope="module")
def registers():
    """Registers per thread of each instance of the RMSNorm kernel, as (pieces of a row per thread, rows per CTA)."""
    from paper_2608_15943_b200 import build
    log = os.path.join(build.OBJ, "kvp_stage.o.log")
    build.build()
    if not os.path.exists(log):
        pytest.skip("the object was built elsewhere")
    text = open(log).read()
    return {(int(a), int(b)): int(n) for a, b, n in
            re.findall(r"rmsnorm_kernelILi(\d)ELi(\d)E.*?Used (\d+) registers", text, flags=re.S)}


@pytest.mark.parametrize("pieces,rows,ctas", [(1, 1, 5), (1, 2, 5), (2, 1, 3), (2, 2, 3), (3, 1, 4), (4, 1, 3)])
def test_rmsnorm_ctas_fit_an_sm(registers, pieces, rows, ctas):
    """As many CTAs of 256 threads as the launch counts on; rows of more than 4096 elements need four and three of them."""
    assert ctas * 256 * registers[(pieces, rows)] <= 65536
