"""The streaming step kernels against the registers of their launch bounds.

The FP32 whole-CTA kernels carry the full-size workloads: a register spilled
inside their march cost a batch a tenth to a fifth of its rate.  What the
compiler prints for them (-Xptxas -v) has to show no spill."""
import os
import re
import subprocess

import pytest

from paper_2303_14119_gb300 import _build


@pytest.fixture(scope="module")
def spills(tmp_path_factory):
    """Spilled bytes (stores, loads) of each step kernel of a whole CTA:
    (kernel, template arguments as mangled)."""
    if not os.path.exists(_build.NVCC):
        pytest.skip("no nvcc")
    obj = str(tmp_path_factory.mktemp("registers") / "o.o")
    out = subprocess.run([_build.NVCC, *_build.ARCH, *_build.FLAGS, "-Xptxas", "-v", "-c",
                          os.path.join(_build.CSRC, "fk_stream.cu"), "-o", obj],
                         capture_output=True, text=True, check=True).stderr
    found = {}
    for part in out.split("Compiling entry function")[1:]:
        name = re.search(r"'(\S+)'", part).group(1)
        m = re.search(r"(step_stream(?:_batch)?_kernel)I([fd]Lb[01]ELb[01])E", name)
        if m:
            s = re.search(r"(\d+) bytes spill stores, (\d+) bytes spill loads", part)
            found[m.groups()] = tuple(map(int, s.groups()))
    return found


@pytest.mark.parametrize("kernel", ["step_stream_kernel", "step_stream_batch_kernel"])
def test_plain_fp32_step_kernels_do_not_spill(spills, kernel):
    assert spills[kernel, "fLb0ELb0"] == (0, 0)


def test_fp32_batch_kernel_with_collisions_does_not_spill(spills):
    """One kernel for rows with padding and without."""
    assert ("step_stream_batch_kernel", "fLb0ELb1") not in spills
    assert spills["step_stream_batch_kernel", "fLb1ELb1"] == (0, 0)
