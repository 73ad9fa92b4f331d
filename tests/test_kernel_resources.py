"""Register counts that a launch depends on, as the compiler reports them
(no GPU): the diagnostics kernel for short rows runs four blocks of 256 threads
on an SM, which 64 registers a thread allow; the FP64 sweeps of a single field
run 36 warps, which 56 allow."""
import functools
import re
import subprocess

from paper_2203_00879_gb300 import build


@functools.lru_cache(None)
def _report(source):
    r = subprocess.run([build.NVCC, *build.ARCH, *build.FLAGS, "-Xptxas", "-v", "-c", source, "-o", "/dev/null"],
                       cwd=build.CSRC, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return r.stderr.splitlines()


def _registers(source, kernel):
    out, name = [], None
    for line in _report(source):
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


def test_fp64_single_field_sweeps_keep_their_warps():
    # line_kernel<double, mode, axis>, modes 0 (first derivative) and 3 (compact second)
    regs = _registers("line_kernels.cu", "line_kernelIdLi0E") + _registers("line_kernels.cu", "line_kernelIdLi3E")
    assert len(regs) == 6 and max(regs) <= 56, regs
