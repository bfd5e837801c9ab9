"""Registers of the dense composite: its grid is eight 256-thread CTAs per SM, and it is as fast as
the loads of the CTAs that fit there at once."""
import os
import re
import subprocess

import pytest

from paper_2608_27735_gb300 import _build


@pytest.fixture(scope="module")
def registers():
    src = os.path.join(_build.CSRC, "composite.cu")
    r = subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-Xptxas", "-v", "-c", src, "-o", os.devnull],
                       capture_output=True, text=True, check=True)
    out = {}
    for part in r.stderr.split("Compiling entry function")[1:]:
        m = re.search(r"composite_kernelILi(\d)ELb([01])E", part)
        if m:
            out[int(m[1]), m[2] == "1"] = (int(re.search(r"Used (\d+) registers", part)[1]),
                                           int(re.search(r"(\d+) bytes spill loads", part)[1]))
    return out


@pytest.mark.parametrize("pix,f16,ctas", [(1, True, 8), (2, True, 8), (1, False, 8), (2, False, 6)])
def test_dense_composite_fits_its_ctas(registers, pix, f16, ctas):
    """65,536 registers per SM, handed out to a warp in multiples of eight per thread."""
    regs, spilled = registers[pix, f16]
    assert spilled == 0
    assert 65536 // (256 * ((regs + 7) // 8 * 8)) >= ctas
