"""The streaming step kernels against the registers of their launch bounds.

The plain FP32 kernels, alone and in a batch, carry the full-size workloads: a
register spilled inside their march cost the batch a fifth of its rate.  What
the compiler prints for them (-Xptxas -v) has to show no spill."""
import os
import re
import subprocess

import pytest

from paper_2303_14119_gb300 import _build


@pytest.mark.skipif(not os.path.exists(_build.NVCC), reason="no nvcc")
def test_plain_fp32_step_kernels_do_not_spill(tmp_path):
    out = subprocess.run([_build.NVCC, *_build.ARCH, *_build.FLAGS, "-Xptxas", "-v", "-c",
                          os.path.join(_build.CSRC, "fk_stream.cu"), "-o", str(tmp_path / "o.o")],
                         capture_output=True, text=True, check=True).stderr
    spills = {}
    for part in out.split("Compiling entry function")[1:]:
        name = re.search(r"'(\S+)'", part).group(1)
        # template arguments <float, PADDED = false, BGK = false>
        m = re.search(r"(step_stream(?:_batch)?_kernel)IfLb0ELb0E", name)
        if m:
            spills[m.group(1)] = re.search(r"(\d+) bytes spill stores, (\d+) bytes spill loads",
                                           part).groups()
    assert spills == {"step_stream_kernel": ("0", "0"), "step_stream_batch_kernel": ("0", "0")}
