"""Kernels that start while the one before them still runs must not read through loads the compiler may move in front of
their wait."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1911_05181_b200", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    text = re.sub(r"/\*.*?\*/", " ", text, flags=re.S)
    return re.sub(r"//[^\n]*", " ", text)


WAIT = r"\bchain_wait(?:_only)?\(\);"
CHAINED = [f for f in sorted(os.listdir(CSRC)) if f.endswith(".cu") and re.search(WAIT, _code(f))]


def test_the_chained_kernels_are_found():
    assert {"reduce.cu", "tc_gemm.cu", "pair_gemm.cu", "bf16_gemm.cu"} <= set(CHAINED)


@pytest.mark.parametrize("name", CHAINED + [f for f in sorted(os.listdir(CSRC)) if f.endswith(".cuh")])
def test_no_read_only_loads(name):
    code = _code(name)
    assert not re.findall(r"\b__ld(?:g|cg|ca|cs|lu|cv)\s*\(|ld\.global\.nc", code)
    assert not re.findall(r"\bconst\s+\w+\s*\*\s*(?:const\s+)?__restrict__", code)


@pytest.mark.parametrize("name", CHAINED)
def test_every_chained_kernel_waits(name):
    # a kernel launched through launch_chained, or with the programmatic attribute, waits for the one before it
    code = _code(name)
    launched = set(re.findall(r"launch_chained\(\s*(\w+_kernel)", code)) | set(re.findall(r"cudaLaunchKernelEx\(&cfg, (\w+_kernel)", code))
    launched |= set(re.findall(r"run\((\w+_kernel)<", code))
    assert launched
    for k in launched:
        at = code.index(k + "(", code.index("__global__"))
        body = code[at:code.find("__global__", at) if code.find("__global__", at) > 0 else len(code)]
        assert re.search(WAIT, body), k
