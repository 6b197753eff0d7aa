"""The fp16-pair kernels move registers between their warps: what the epilogue warps take is what the others give back only
when every variant is compiled with the number of registers the shares were worked out for."""
import os
import re
import subprocess

from paper_1911_05181_b200 import buildlib


def test_pair_kernels_are_compiled_with_the_registers_their_shares_add_up_to(tmp_path):
    src = os.path.join(buildlib.CSRC, "pair_gemm.cu")
    want = int(re.search(r"LAUNCH_REGS = (\d+)", open(src).read()).group(1))
    flags = [f for f in buildlib.NVCC_FLAGS]
    r = subprocess.run([buildlib._nvcc()] + flags + ["-Xptxas", "-v", "-c", src, "-o", str(tmp_path / "pair.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    used = re.findall(r"Compiling entry function '(\w*pair_gemm_kernel\w*)'.*?Used (\d+) registers", r.stderr, flags=re.S)
    assert len(used) == 10                      # five epilogues, by one CTA and by a pair
    assert {int(n) for _, n in used} == {want}, used
    # and the launch refuses a kernel compiled with another number
    assert re.search(r"allow_dynamic_smem\(pair_gemm_kernel<EPI, CG>, SMEM_BUDGET, configured, LAUNCH_REGS\)", open(src).read())
