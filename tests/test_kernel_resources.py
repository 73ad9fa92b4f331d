"""Register counts that a launch depends on, as the compiler reports them
(no GPU): the diagnostics kernel for short rows runs four blocks of 256 threads
on an SM, which 64 registers a thread allow."""
import re
import subprocess

from paper_2203_00879_gb300 import build


def _registers(source, kernel):
    r = subprocess.run([build.NVCC, *build.ARCH, *build.FLAGS, "-Xptxas", "-v", "-c", source, "-o", "/dev/null"],
                       cwd=build.CSRC, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out, name = [], None
    for line in r.stderr.splitlines():
        m = re.search(r"Compiling entry function '(\S+)'", line)
        if m:
            name = m.group(1)
        m = re.search(r"Used (\d+) registers", line)
        if m and name and kernel in name:
            out.append(int(m.group(1)))
    return out


def test_diagnostics_of_short_rows_fit_four_blocks():
    regs = _registers("rk_kernels.cu", "diag_partial_kernel")
    assert regs and min(regs) <= 65536 // (4 * 256), regs
