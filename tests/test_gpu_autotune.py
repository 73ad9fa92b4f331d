"""Sub-domain length of a mixed-form box that leaves it to the autotuner, on the
axes whose FP32 derivative does not depend on it (x in the Thomas form, every
axis in the banded one): the default, 64 or, in lines of at most 64 points, 32,
in every process -- not whichever of three equal launches a timer saw as the
fastest.  The box shapes are of this test alone (choices are kept per shape)."""
import pytest

import nopcs_synth as S
from gpu_util import binding, stream_ptr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form,axes", [("THOMAS", (0,)), ("BANDED", (0, 1, 2))])
def test_untimed_axes_take_the_default(form, axes):
    N = binding()
    for k in range(6):
        n = (131 + 3 * k, 97 + k, 139 - 2 * k)
        p = S.box_params(n, sub_n=(-1, -1, -1))
        ctx = N.nopcs_init([p], prec=N.NOPCS_MIXED, form=getattr(N, "NOPCS_FORM_" + form), stream=stream_ptr())
        try:
            sub = N.nopcs_box_info(ctx, 0)["sub_n"]
        finally:
            N.nopcs_destroy(ctx)
        assert all(sub[a] == 64 for a in axes), (n, sub)
        assert all(s in (32, 64, 128) for s in sub), (n, sub)


@pytest.mark.parametrize("form", ["AUTO", "THOMAS", "GEMM_3XTF32", "GEMM_BF16X3", "BANDED"])
def test_short_lines_take_32(form):
    N = binding()
    p = S.box_params((64, 45, 37), sub_n=(-1, -1, -1))
    ctx = N.nopcs_init([p], prec=N.NOPCS_MIXED, form=getattr(N, "NOPCS_FORM_" + form), stream=stream_ptr())
    try:
        assert N.nopcs_box_info(ctx, 0)["sub_n"] == [32, 32, 32]
    finally:
        N.nopcs_destroy(ctx)
