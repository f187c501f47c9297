"""What the sources and the build say of the kernels."""
import glob
import os
import re
import subprocess
from decimal import Decimal, getcontext
import ctypes as C

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


def test_no_input_is_taken_for_constant():
    """Kernels come up while the ones ahead still write their inputs (programmatic dependent launch), and the element-wise
    operators may work in place: neither allows a pointer that promises nobody else writes, nor a read-only load."""
    from paper_2608_15943_b200 import build
    for path in glob.glob(os.path.join(build.CSRC, "*.cu*")):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        assert not re.search(r"__restrict__|__ldg\b|ld\.global\.nc", code), path


@pytest.mark.parametrize("dh", [8, 64, 128, 192, 256])
@pytest.mark.parametrize("theta", [1.5, 10000.0, 500000.0, 1e6])
def test_rope_frequencies_fill_their_float_pairs(tmp_path, dh, theta):
    """hi + lo against theta^(-2i/dh) in 60 digits: what two floats of 24 bits hold, and no more error than that."""
    from paper_2608_15943_b200 import build
    src = tmp_path / "f.cpp"
    src.write_text('#include "kvp_rope_freq.h"\n'
                   'extern "C" void freqs(double t, int dh, float* out) { kvp::rope_frequencies(t, dh, out, out + 1, 2); }\n')
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I" + build.CSRC, str(src), "-o", str(tmp_path / "f.so")], check=True)
    out = (C.c_float * dh)()
    C.CDLL(str(tmp_path / "f.so")).freqs(C.c_double(theta), dh, out)
    getcontext().prec = 60
    for i in range(dh // 2):
        want = (Decimal(theta).ln() * Decimal(-2 * i) / Decimal(dh)).exp()
        got = Decimal(out[2 * i]) + Decimal(out[2 * i + 1])
        assert abs(got / want - 1) <= Decimal(2) ** -48, i
