"""What ptxas reports for the self-attention kernels: their softmax warps hold 32 logits, 16 packed weights and the codes of a
chunk at the register limit of the launch, and a spill there is paid for every score."""
import re
import shutil
import subprocess

import pytest

from paper_2501_04304_b200 import build

NVCC = shutil.which("nvcc") or shutil.which("/usr/local/cuda/bin/nvcc")
# (head size, fixed scale, writes codes, few codes); heads of 160 are left out: they spill 8 bytes where they write codes
VARIANTS = [(d, *v) for d in (40, 64, 80, 128) for v in ((0, 0, 0), (0, 0, 1), (0, 1, 0), (0, 1, 1), (1, 0, 0), (1, 1, 0))]


def _symbol(d, fixed, codes, few):
    return f"_ZN3dgq21self_attn_logq_kernelILi{d}ELb{fixed}ELb{codes}ELb{few}EEEv14CUtensorMap_stS1_S1_NS_12SelfAttnArgsE"


@pytest.mark.skipif(NVCC is None, reason="needs nvcc")
def test_self_attention_does_not_spill(tmp_path):
    flags = [f for f in build.NVCC_FLAGS if f != "-shared"]
    entries = ",".join(f"-e,{_symbol(*v)}" for v in VARIANTS)
    res = subprocess.run([NVCC, *flags, "-Xptxas", "-v," + entries, "-cubin", build.SRC, "-o", str(tmp_path / "k.cubin")],
                         capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-2000:]
    spills = {m[1]: (int(m[2]), int(m[3])) for m in re.finditer(
        r"Function properties for (\S+)\s+\d+ bytes stack frame, (\d+) bytes spill stores, (\d+) bytes spill loads", res.stderr)}
    assert {v: spills[_symbol(*v)] for v in VARIANTS} == {v: (0, 0) for v in VARIANTS}
