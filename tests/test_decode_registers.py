"""The decode attention keeps its running maxima, sums and outputs in registers: no
spills in the tensor-core kernel, which three CTAs an SM leave 168 registers a thread.
Spills cost dense decode 1 to 3%."""
import os
import re
import shutil
import subprocess

import pytest

from paper_2609_13141_gb300 import _build


def test_tensor_core_attention_does_not_spill(tmp_path):
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("no nvcc")
    cmd = [_build._nvcc(), *_build.CFLAGS, "-Xptxas", "-v", "-c", os.path.join(_build.CSRC, "k_decode.cu"), "-o",
           str(tmp_path / "k_decode.o")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    found = re.findall(r"Compiling entry function '(\S*dec_attn_tc_kernel\S*)'.*?(\d+) bytes spill stores, (\d+) bytes "
                       r"spill loads.*?Used (\d+) registers", r.stderr, flags=re.S)
    assert len(found) == 8   # G = 1, 2, 4, 8, SAS and dense lists
    for name, stores, loads, regs in found:
        assert (int(stores), int(loads)) == (0, 0), name
        assert int(regs) <= 168, name
