"""What the benchmark says of the kernels, against the sources (CPU): the lists
that tag profiler counters name every file in which a device function that the
kind runs is defined, and a kind counts as many launches as its launcher makes."""
import os
import re

import pytest

from paper_2203_00879_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

USES = {
    "prep": ["prep_kernel", "prep_point", "narrow_f64"],
    "wall_bc": ["wall_kernel", "wall_update", "corner_update"],
    "diagnostics": ["diag_partial_kernel", "diag_final_kernel", "narrow_f64"],
    "sweep_x": ["scan_kernel", "scan_body", "sweep_point"],
    "sweep_y": ["march_kernel", "march_body", "sweep_point"],
    "sweep_z": ["march_kernel", "march_body", "sweep_point"],
    "filter": ["scan_kernel", "scan_body", "march_kernel", "march_body", "line_kernel", "line_body",
               "nohap_solve_column", "filter_update_kernel", "prep_point", "widen_f32"],
    "visc_rk_update": ["visc_rk_kernel", "visc_rk_body", "mixed_update", "widen_f32"],
}


def _defined_in(name):
    # "... void name(" or "... double name(" at the start of a definition
    pat = re.compile(r"^(?:__global__|__device__|static __device__)[^;{]*?\b%s\(" % name, re.M | re.S)
    return [f for f in sorted(os.listdir(build.CSRC)) if f.endswith((".cu", ".cuh"))
            and pat.search(open(os.path.join(build.CSRC, f)).read())]


@pytest.mark.parametrize("kind", sorted(build.KERNEL_FILES))
def test_lists_name_every_source(kind):
    for name in USES[kind]:
        files = _defined_in(name)
        assert files, name
        missing = set(files) - set(build.KERNEL_FILES[kind])
        assert not missing, (kind, name, missing)


def _launches(source, function):
    """Kernel launches that one call of a launcher makes: the branches of an if
    each hold one."""
    text = open(os.path.join(build.CSRC, source)).read()
    body = re.search(r"\n(?:template [^\n]*\n)?cudaError_t %s\(.*?\n}\n" % function, text, re.S).group(0)
    return body.count("<<<") - len(re.findall(r"\n    else\n", body))


def test_launches_per_kind():
    src = open(os.path.join(ROOT, "bench.py")).read()
    per_kind = dict(re.findall(r'"(\w+)": (\d+)', re.search(r"LAUNCHES_PER_KIND = \{(.*?)\}", src, re.S).group(1)))
    assert int(per_kind["wall_bc"]) == _launches("rk_kernels.cu", "launch_wall_bc")
    assert int(per_kind["diagnostics"]) == _launches("rk_kernels.cu", "launch_diagnostics")
    # three sweeps and the update
    assert int(per_kind["filter"]) == 3 + _launches("rk_kernels.cu", "launch_filter_update")
    assert _launches("rk_kernels.cu", "launch_prep") == 1
