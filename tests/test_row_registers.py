"""Registers of the general row DFT (csrc/fft.cu, k_fft_rows), as the assembler reports them: 64 a thread at
most, four CTAs of 256 threads on an SM, in float64 too (PIC_DHT_F64_GEMM, lengths that are no power of two)."""
import re
import shutil
import subprocess

import pytest

from paper_1611_05712_gb300 import build as B


def test_four_ctas_on_an_sm(tmp_path):
    if shutil.which("nvcc") is None:
        pytest.skip("nvcc not available")
    src = [s for s in B.sources() if s.endswith("/fft.cu")][0]
    r = subprocess.run(["nvcc", "-c", src, "-o", str(tmp_path / "fft.o"), "-Xptxas", "-v"] + B.ARCH + B.FLAGS,
                       capture_output=True, text=True, check=True)
    name, regs = None, {}
    for line in r.stderr.splitlines():
        m = re.search(r"Compiling entry function '(\S+)'", line)
        if m:
            name = m.group(1)
        m = re.search(r"Used (\d+) registers", line)
        if m and "k_fft_rows" in name:
            regs[name] = int(m.group(1))
    assert sum("IdL" in n for n in regs) == 2   # float64, forward and inverse
    assert max(regs.values()) <= 64, regs
